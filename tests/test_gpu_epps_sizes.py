"""The cutoff sweep at the sizes where its work items change: sweeps around a
warp's 32 modes, small problems up to and beyond 511 modes and 4 assets (a warp
each, or CTAs), many short segments, one long one, one problem (many CTAs) and
more problems than CTAs; against Eqs. (2), (3) in float64 on the sweep's own
coefficients.

Tolerance relative to sqrt(Sigma_ii Sigma_jj), in units of eps of the working
type: a lane adds at most 16 modes of an item (two roundings each), five
shuffle steps, the items of one segment (256 modes or more each, else 32), and
about ten roundings for products, weights and output (Cauchy-Schwarz bounds the
sum of the terms' absolute values)."""
import numpy as np
import pytest

from paper_2003_02842_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

EPS = {"bf16x3": 2.0**-24, "fp64": 2.0**-53}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec", ["bf16x3", "fp64"])
@pytest.mark.parametrize("basis", ["dirichlet", "fejer"])
@pytest.mark.parametrize("reps,D,cuts", [
    (3, 1, [1]), (5, 2, list(range(1, 33))), (310, 2, [1, 31, 32, 33, 63, 64]), (2, 3, [511]), (2, 3, [5, 512]),
    (4, 4, [2, 3, 5, 100, 333, 510]), (2, 5, list(range(1, 129))), (1, 12, [7, 8, 9, 40, 700, 1500]),
    (306, 10, [1, 2, 3, 64, 600]), (1, 2, [3000])])
def test_sweep_at_item_edges(prec, basis, reps, D, cuts):
    import paper_2003_02842_gb300 as mm
    ev = synth.random_events(300 + D, D=reps * D, n_range=(20, 60), T=500.0)
    off, t, p = to_dev(ev)
    b = mm.mm_batch_create(reps=reps, D=D, N_max=cuts[-1], max_events=ev.n_events,
                           tol=1e-12 if prec == "fp64" else 1e-6, basis=basis, prec=prec)
    for _ in range(2):  # the first call and a graph replay
        S, R = mm.mm_batch_epps(b, off, t, p, cuts)
    assert mm.mm_batch_sync(b) == 0
    F = mm.mm_batch_coeffs(b).cpu().numpy().astype(np.complex128).reshape(reps, D, -1)
    S, R = S.cpu().numpy().astype(np.float64), R.cpu().numpy().astype(np.float64)
    mm.mm_batch_destroy(b)
    k = np.arange(F.shape[2])
    n_items = max(len(k) // 256 + 2, 4)
    tol = (2 * 16 + 5 + n_items + 10) * EPS[prec]
    for j, N in enumerate(cuts):
        w = np.full(N + 1, 1.0 / (2 * N + 1)) if basis == "dirichlet" else (1.0 - k[:N + 1] / N) / (N + 1)
        w = np.where(k[:N + 1] > 0, 2.0, 1.0) * w * (2 * np.pi) ** 2
        ref = np.einsum("rik,rjk,k->rij", F[..., :N + 1], F[..., :N + 1].conj(), w).real
        sd = np.sqrt(np.einsum("rii->ri", ref))
        sc = sd[:, :, None] * sd[:, None, :]
        assert np.max(np.abs(S[:, j] - ref) / sc) <= tol
        assert np.max(np.abs(R[:, j] - ref / sc)) <= 3 * tol
        assert np.all(np.einsum("rii->ri", R[:, j]) == 1.0)
