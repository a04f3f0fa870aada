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
