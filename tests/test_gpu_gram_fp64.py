"""The FP64 contraction (4 x 4 tiles, modes over the lanes of a warp, chunks
over warps and splits) against numpy in float64 on the same coefficients.

Sizes: assets below, at and beyond a tile edge; modes below, at and beyond a
32-mode chunk, a CTA's eight warps and the split threshold. Tolerance: every
entry is a sum of 2(N + 1) weighted products whose absolute values add up to
at most sqrt(Sigma_ii Sigma_jj) (Cauchy-Schwarz); any order of summation of n
terms is within n 2^-53 of that, each term carries at most four roundings
(two weights, two products), on either side.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("basis", ["dirichlet", "fejer"])
@pytest.mark.parametrize("D,N", [(1, 1), (2, 31), (3, 32), (4, 255), (5, 1023), (2, 40000), (9, 1055), (17, 2500),
                                 (130, 300)])
def test_fp64_contraction_at_tile_and_chunk_edges(D, N, basis):
    import torch
    import paper_2003_02842_gb300 as mm
    rng = np.random.default_rng([D, N])
    F = rng.standard_normal((D, N + 1)) + 1j * rng.standard_normal((D, N + 1))
    F[:, 0] = F[:, 0].real
    plan = mm.mm_plan_create(D=D, N_max=N, tol=1e-12, basis=basis, prec="fp64")
    S, R = mm.mm_corr(plan, torch.from_numpy(F).cuda(), N)
    assert mm.mm_plan_sync(plan) == 0
    S, R = S.cpu().numpy(), R.cpu().numpy()
    mm.mm_destroy(plan)
    k = np.arange(N + 1)
    w = np.full(N + 1, 1.0 / (2 * N + 1)) if basis == "dirichlet" else (1.0 - k / N) / (N + 1)
    w = np.where(k > 0, 2.0, 1.0) * w * (2 * np.pi) ** 2
    A = np.sqrt(w)[:, None] * np.stack([F.real.T, F.imag.T], 0)  # 2 x (N+1) x D
    S_ref = np.einsum("rki,rkj->ij", A, A)
    sd = np.sqrt(np.diag(S_ref))
    bound = 2 * (2 * (N + 1) + 4) * 2.0**-53
    assert np.max(np.abs(S - S_ref) / np.outer(sd, sd)) <= bound
    assert np.array_equal(S, S.T) and np.array_equal(np.diag(R), np.ones(D))
    assert np.max(np.abs(R - S_ref / np.outer(sd, sd))) <= 2 * bound + 8 * 2.0**-53


@pytest.mark.parametrize("basis", ["dirichlet", "fejer"])
@pytest.mark.parametrize("D,N", [(255, 40), (256, 15), (256, 16), (500, 30), (577, 1), (640, 31), (1000, 30), (1000, 63),
                                 (320, 8000), (500, 2000)])
def test_fp64_contraction_of_many_assets(D, N, basis):
    # both forms' tiles (4 x 4 and 64 x 64) around the sizes where one takes over from the
    # other, whole and broken tiles and 16-mode chunks, one split and several. Against
    # numpy by the bound above
    import torch
    import paper_2003_02842_gb300 as mm
    gen = torch.Generator(device="cuda").manual_seed(D + N)
    F = torch.randn((D, N + 1), dtype=torch.complex128, device="cuda", generator=gen)
    F[:, 0] = F[:, 0].real.to(F.dtype)
    plan = mm.mm_plan_create(D=D, N_max=N, tol=1e-12, basis=basis, prec="fp64")
    S, R = mm.mm_corr(plan, F, N)
    assert mm.mm_plan_sync(plan) == 0
    S, R = S.cpu().numpy(), R.cpu().numpy()
    mm.mm_destroy(plan)
    F = F.cpu().numpy()
    k = np.arange(N + 1)
    w = np.full(N + 1, 1.0 / (2 * N + 1)) if basis == "dirichlet" else (1.0 - k / N) / (N + 1)
    w = np.where(k > 0, 2.0, 1.0) * w * (2 * np.pi) ** 2
    A = (np.sqrt(w)[:, None] * np.stack([F.real.T, F.imag.T], 0)).reshape(-1, D)
    S_ref = A.T @ A
    sd = np.sqrt(np.diag(S_ref))
    bound = 2 * (2 * (N + 1) + 4) * 2.0**-53
    assert np.max(np.abs(S - S_ref) / np.outer(sd, sd)) <= bound
    assert np.array_equal(S, S.T) and np.array_equal(np.diag(R), np.ones(D))
    assert np.max(np.abs(R - S_ref / np.outer(sd, sd))) <= 2 * bound + 8 * 2.0**-53


def test_fp64_contraction_takes_the_faster_form():
    # 64 x 64 tiles for many assets and few modes (five to seven times as fast there), 4 x 4
    # for few assets and where whole waves of large tiles would stand half empty
    import torch
    import paper_2003_02842_gb300 as mm
    for D, N, splits in ((1000, 30, 1), (500, 2000, 4), (600, 2000, 1)):
        plan = mm.mm_plan_create(D=D, N_max=N, tol=1e-12, prec="fp64")
        F = torch.randn((D, N + 1), dtype=torch.complex128, device="cuda")
        mm.mm_corr(plan, F, N)
        assert mm.mm_plan_get_info(plan)["gram_splits"] == splits
        S, R = torch.empty((D, D), dtype=torch.float64, device="cuda"), torch.empty((D, D), dtype=torch.float64,
                                                                                  device="cuda")
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            mm.mm_corr(plan, F, N, sigma=S, R=R)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        if (D, N) == (1000, 30):
            assert best < 0.25  # ms: 0.108 with 64 x 64 tiles, 0.579 with 4 x 4
        mm.mm_destroy(plan)
