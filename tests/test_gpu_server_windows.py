"""GPU parity of a request's window search over more assets than the search's
block has threads (512): requests of one asset, of one block less one, exactly,
and more, and of two blocks and a rest, with events on both ends of the window
and in windows that hold no event but those, against the FP64 CPU oracle on the
events in the window. Both the given cutoff and the one found on the device.
Tolerances of the serving form: max |dR| <= 1e-4, max |dSigma_ij| /
sqrt(V_i V_j) <= 1e-4 with V the realised variances of the window."""
import time

import numpy as np
import pytest

import oracle
from paper_2003_02842_gb300 import synth

pytestmark = pytest.mark.gpu

D = 1030
T0, T1 = 100.0, 900.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.fixture(scope="module")
def served():
    import paper_2003_02842_gb300 as mm
    rng = np.random.default_rng(17)
    off, ts, ps = [0], [], []
    for i in range(D):
        inner = rng.integers(101, 900, size=0 if i % 7 == 3 else 1 + i % 9)
        t = np.unique(np.concatenate([[T0, T1], inner, rng.integers(0, 100, size=i % 4),
                                      rng.integers(901, 1000, size=i % 5)])).astype(np.float64)
        ts.append(t)
        ps.append(np.cumsum(rng.standard_normal(t.size)))
        off.append(off[-1] + t.size)
    day = (np.array(off, dtype=np.int64), np.concatenate(ts), np.concatenate(ps))
    srv = mm.mm_server_create(D=D, N_max=40, max_events=day[0][-1], max_slots=2, tol=1e-6, kernel="es",
                              basis="fejer")
    mm.mm_server_load(srv, *day)
    yield day, srv
    mm.mm_server_destroy(srv)


@pytest.mark.parametrize("N", [0, 24])
@pytest.mark.parametrize("n", [1, 511, 512, 513, D])
def test_windows_of_many_assets(served, n, N):
    import paper_2003_02842_gb300 as mm
    (off, t, p), srv = served
    assets = np.random.default_rng(n).permutation(D)[:n].astype(np.int32)
    tk = mm.mm_server_submit(srv, T0, T1, assets, N=N, sigma=True)
    got, end = [], time.time() + 60.0
    while not got and time.time() < end:
        got += mm.mm_server_poll(srv, wait=0.05)
    c, = got
    assert c["ticket"] == tk and c["status"] == 0
    to, tt, pp = [0], [], []
    for a in assets:
        s = slice(off[a], off[a + 1])
        m = (t[s] >= T0) & (t[s] <= T1)
        tt.append(t[s][m])
        pp.append(p[s][m])
        to.append(to[-1] + int(m.sum()))
    to, V = np.array(to, dtype=np.int64), np.array([np.sum(np.diff(x) ** 2) for x in pp])
    tt, pp = np.concatenate(tt), np.concatenate(pp)
    nyq = oracle.nyquist(to, tt, T0, T1)
    want = N if N else nyq if 1 <= nyq <= 40 else 40  # none, or one above N_max: served at N_max
    assert c["N"] == want
    o = oracle.estimate(to, tt, pp, N=want, basis="fejer", window=(T0, T1))
    assert np.max(np.abs(c["Sigma"].astype(np.float64) - o["Sigma"]) / np.sqrt(np.outer(V, V))) <= 1e-4
    assert np.max(np.abs(c["R"].astype(np.float64) - o["R"])) <= 1e-4
