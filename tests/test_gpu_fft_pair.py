"""The cluster pair's transform at the edges of its passes and its paired
unpacking: rows of a few points to the largest, plans of two to four passes and
of radices up to 16, 25 and 32 (three kernels), cutoffs that use less than half,
just half and all of a half row's outputs (a cutoff below N_max keeps its own
grid, so N sets the row). Every coefficient against the oracle's direct sum at
the mixed path's tolerance (Eq. (15) <= 1e-5 at tol 1e-6)."""
import pytest

import oracle
from paper_2003_02842_gb300 import synth

from gpu_helpers import rel_l2_rows, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("N", [1, 2, 5, 11, 50, 121, 333, 720, 1561, 2187, 5000, 6250, 8100, 11999, 12150, 13121, 14399])
def test_pair_matches_direct_sum(N):
    ev = synth.random_events(500 + N, D=3, n_range=(10, 300), T=2500.0)
    out = run(dict(tol=1e-6, kernel="es", basis="dirichlet", prec="bf16x3", fft_algo="asset_pair"), ev, N)
    assert out["status"] == 0
    assert out["info"]["fft_algo"] == 1 or out["info"]["fft_split"] == 3
    assert rel_l2_rows(out["F"], oracle.coeffs_F(ev.offsets, ev.t, ev.logp, N)).max() <= 1e-5


@pytest.mark.parametrize("N", [1, 2, 11, 121, 720, 2187, 6250, 6560, 8100, 10124, 12150, 13121, 14399, 14580])
def test_these_lengths_take_the_pair(N):
    # rows of 8 to 30,000 points, odd half rows (6561 and 10,125 points) among them: no
    # fall-back to another transform may pass unseen
    ev = synth.random_events(700 + N, D=2, n_range=(10, 60), T=2500.0)
    out = run(dict(tol=1e-6, kernel="es", basis="dirichlet", prec="bf16x3", fft_algo="asset_pair"), ev, N)
    assert out["status"] == 0 and out["info"]["fft_algo"] == 0 and out["info"]["fft_split"] == 3
    assert rel_l2_rows(out["F"], oracle.coeffs_F(ev.offsets, ev.t, ev.logp, N)).max() <= 1e-5


@pytest.mark.parametrize("D,N", [(77, 6560), (78, 10124), (153, 14399), (160, 1)])
def test_rows_fetched_ahead(D, N):
    # more rows than the 76 pairs that run at once, each of which brings the row 76 on into L2:
    # one, two and many of them, rows whose half is no whole number of 16-byte pieces
    ev = synth.random_events(800 + D, D=D, n_range=(3, 30), T=2500.0)
    out = run(dict(tol=1e-6, kernel="es", basis="dirichlet", prec="bf16x3", fft_algo="asset_pair"), ev, N)
    assert out["status"] == 0 and out["info"]["fft_split"] == 3
    assert rel_l2_rows(out["F"], oracle.coeffs_F(ev.offsets, ev.t, ev.logp, N)).max() <= 1e-5
