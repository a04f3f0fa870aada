"""The transform of several short rows per CTA (more rows than SMs): a last CTA
with fewer rows, one row more than the SMs, rows of a few points and of
thousands, plans of radices up to 16 and above (n = 6250); every coefficient
against the oracle's direct sum at the mixed path's tolerance (Eq. (15) <= 1e-5
at tol 1e-6), a single problem and a batch."""
import numpy as np
import pytest

import oracle
from paper_2003_02842_gb300 import synth

from gpu_helpers import rel_l2_rows, run, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("D,N", [(153, 1), (153, 700), (310, 50), (310, 3100), (457, 6), (1000, 333)])
def test_rows_per_cta_match_direct_sum(D, N):
    ev = synth.random_events(400 + N, D=D, n_range=(2, 25), T=900.0)
    out = run(dict(tol=1e-6, kernel="es", basis="dirichlet", prec="bf16x3"), ev, N)
    assert out["status"] == 0 and out["info"]["fft_algo"] == 0
    assert rel_l2_rows(out["F"], oracle.coeffs_F(ev.offsets, ev.t, ev.logp, N)).max() <= 1e-5


def test_batch_rows_per_cta():
    import paper_2003_02842_gb300 as mm
    reps, D, N = 500, 2, 50
    evs = [synth.random_events(r, D=D, n_range=(20, 100), T=100.0 + r) for r in range(reps)]
    ev = synth.concat_events(evs)
    b = mm.mm_batch_create(reps=reps, D=D, N_max=N, max_events=ev.n_events, tol=1e-6)
    off, t, p = to_dev(ev)
    mm.mm_batch_epps(b, off, t, p, [1, 7, N])
    assert mm.mm_batch_sync(b) == 0
    F = mm.mm_batch_coeffs(b).cpu().numpy()
    mm.mm_batch_destroy(b)
    for r in (0, 1, 151, 152, 303, 499):
        ref = oracle.coeffs_F(evs[r].offsets, evs[r].t, evs[r].logp, N)
        assert rel_l2_rows(F[r * D:(r + 1) * D], ref).max() <= 1e-5


@pytest.mark.parametrize("D,N", [(305, 6000), (306, 6000), (456, 6000), (457, 6000), (608, 5000), (609, 4500)])
def test_long_rows_in_several_waves(D, N):
    # both sides of the line between two rows a CTA and a CTA a row
    ev = synth.random_events(600 + D, D=D, n_range=(2, 12), T=900.0)
    out = run(dict(tol=1e-6, kernel="es", basis="dirichlet", prec="bf16x3"), ev, N)
    assert out["status"] == 0 and out["info"]["fft_algo"] == 0 and out["info"]["fft_split"] == 1
    assert rel_l2_rows(out["F"], oracle.coeffs_F(ev.offsets, ev.t, ev.logp, N)).max() <= 1e-5
