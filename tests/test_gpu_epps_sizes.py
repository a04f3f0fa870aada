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


@pytest.mark.parametrize("basis", ["dirichlet", "fejer"])
@pytest.mark.parametrize("D,N,chain", [(1, 511, 32), (2, 200, 28), (3, 350, 77), (4, 100, 44), (4, 352, 132)])
def test_both_forms_of_small_problems(basis, D, N, chain):
    # one problem fewer than a warp each is taken for (28 per step of its chain; never beyond
    # 128 steps) and just as many, on the coefficients of one event set
    import torch

    import paper_2003_02842_gb300 as mm
    cuts = sorted({1, 2, 31, 32, 33, N // 2, N - 1, N})
    reps = 28 * chain
    tol = (2 * 16 + 5 + 4 + 10) * EPS["bf16x3"]
    one = synth.random_events(700 + D, D=D, n_range=(20, 40), T=500.0)
    n = one.n_events
    out = []
    for r in (reps - 1, reps):
        off = torch.from_numpy(np.concatenate([one.offsets[:-1] + i * n for i in range(r)] + [[r * n]])).cuda()
        t, p = torch.from_numpy(np.tile(one.t, r)).cuda(), torch.from_numpy(np.tile(one.logp, r)).cuda()
        b = mm.mm_batch_create(reps=r, D=D, N_max=N, max_events=r * n, tol=1e-6, basis=basis)
        S, R = mm.mm_batch_epps(b, off, t, p, cuts)
        assert mm.mm_batch_sync(b) == 0
        F = mm.mm_batch_coeffs(b)[:D].cpu().numpy().astype(np.complex128)
        for x in (S, R):  # every problem is the same
            assert float((x - x[:1]).abs().max()) <= 3 * tol * float(x[0].abs().max())
        out.append((F, S[0].cpu().numpy().astype(np.float64), R[0].cpu().numpy().astype(np.float64)))
        mm.mm_batch_destroy(b)
    k = np.arange(N + 1)
    for F, S, R in out:
        for j, c in enumerate(cuts):
            w = np.full(c + 1, 1.0 / (2 * c + 1)) if basis == "dirichlet" else (1.0 - k[:c + 1] / c) / (c + 1)
            w = np.where(k[:c + 1] > 0, 2.0, 1.0) * w * (2 * np.pi) ** 2
            ref = np.einsum("ik,jk,k->ij", F[:, :c + 1], F[:, :c + 1].conj(), w).real
            sc = np.sqrt(np.outer(np.diag(ref), np.diag(ref)))
            assert np.max(np.abs(S[j] - ref) / sc) <= tol and np.max(np.abs(R[j] - ref / sc)) <= 3 * tol


def test_few_small_problems_are_not_kept_waiting():
    # 32 problems of 4 assets and 511 modes: 15 us of sweep over CTAs, 74 us with a warp each
    import torch

    import paper_2003_02842_gb300 as mm
    R, D, N, n = 32, 4, 511, 600
    ev = synth.random_events(9, D=R * D, n_range=(n, n), T=28800.0)
    x = to_dev(ev)
    b = mm.mm_batch_create(reps=R, D=D, N_max=N, max_events=ev.n_events, tol=1e-6)
    cuts = [1, 100, 300, N]
    S, Rr = mm.mm_batch_epps(b, *x, cuts)
    mm.mm_batch_profile_enable(b, True)
    best = 1e9
    for _ in range(8):
        torch.cuda.synchronize()
        mm.mm_batch_profile_read(b, reset=True)
        mm.mm_batch_epps(b, *x, cuts, sigma=S, R=Rr)
        torch.cuda.synchronize()
        best = min(best, mm.mm_batch_profile_read(b)["gram"][0])
    assert best < 0.035  # ms
    mm.mm_batch_destroy(b)
