"""The positive semi-definite repair at the sizes where its layouts change: one
asset, odd and even counts around a warp's lanes (idle round-robin players,
the folded triangle's half-empty middle row), the largest one-CTA matrices and
the first multi-CTA ones. The repaired Sigma is compared with numpy's
eigenvalue clipping of the library's own unrepaired Sigma (float64).

Tolerance: as in test_gpu_pairwise.py, 8 D eps of the matrix's Frobenius norm
(the iteration stops at an off-diagonal norm of 2 D eps and every element
meets about 2 D rotations a sweep), plus the output's own rounding, eps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = {"bf16x3": 2.0**-24, "fp64": 2.0**-53}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec,D", [("bf16x3", d) for d in (1, 2, 3, 31, 33, 64, 65, 129, 158, 159)] +
                         [("fp64", d) for d in (1, 2, 3, 31, 33, 64, 65, 112, 113)])
def test_repair_at_layout_edges(prec, D):
    import torch
    import paper_2003_02842_gb300 as mm
    rng = np.random.default_rng([D, 5])
    N = 300
    cdt = np.complex64 if prec == "bf16x3" else np.complex128
    F = (rng.standard_normal((D, N + 1)) + 1j * rng.standard_normal((D, N + 1))).astype(cdt)
    F[1:] = 0.6 * F[:1] + 0.8 * F[1:]
    Ns = [int(x) for x in rng.integers(1, 40, size=D)]
    Ns[0] = N
    plan = mm.mm_plan_create(D=D, N_max=N, basis="fejer", prec=prec)
    Fd = torch.from_numpy(F).cuda()
    S0, _, c0 = mm.mm_corr_pairwise(plan, Fd, N, Ns, psd_repair=False)
    S1, R1, c1 = mm.mm_corr_pairwise(plan, Fd, N, Ns, psd_repair=True)
    assert mm.mm_plan_sync(plan) == 0
    S0, S1, R1 = (x.cpu().numpy().astype(np.float64) for x in (S0, S1, R1))
    assert int(c0.item()) == 0
    mm.mm_destroy(plan)
    w, V = np.linalg.eigh(S0)
    ref = (V * np.maximum(w, 0.0)) @ V.T
    norm = np.linalg.norm(S0)
    tol = (8 * D + 1) * EPS[prec] * norm
    assert np.linalg.norm(S1 - ref) <= 2 * tol
    assert np.array_equal(S1, S1.T) and np.array_equal(np.diag(R1), np.ones(D))
    # eigenvalues further from zero than the iteration's own error are counted exactly
    assert np.sum(w < -tol) <= int(c1.item()) <= np.sum(w < tol)
