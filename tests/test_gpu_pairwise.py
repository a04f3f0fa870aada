"""GPU parity of the pairwise-cutoff covariance and its nearest positive
semi-definite repair (Sec. 3.1) against the oracle.

Tolerances: Sigma, max |dSigma_ij| / sqrt(Sigma_ii Sigma_jj) <= 1e-4 (mixed)
and 1e-9 (FP64), R <= 1e-4 / 1e-9, as for the common cutoff. The repair maps
a symmetric matrix to its nearest positive semi-definite one, a map that
moves no two inputs further apart in the Frobenius norm than they were: the
repaired matrices may differ by at most twice the input matrices' difference
plus the eigensolver's own rounding, 1e-12 of the norm for the float64
Jacobi iteration (FP64 plans) and 1e-5 for the float32 one (mixed
precisions, whose Sigma is itself correct to about 1e-5 of its scale).
"""
import numpy as np
import pytest

import oracle
from paper_2003_02842_gb300 import synth

from gpu_helpers import sigma_err, to_dev

pytestmark = pytest.mark.gpu

TOL = {"fp64": dict(tol=1e-12, sig=1e-9, R=1e-9, eig=1e-12), "bf16x3": dict(tol=1e-6, sig=1e-4, R=1e-4, eig=1e-5)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


def _case(seed, D=24):
    # per-asset cutoffs from 2 to 119 (fewer distinct values for many assets:
    # the oracle evaluates Algorithm 3 once per distinct pairwise cutoff)
    ev = synth.random_events(80 + seed, D=D, n_range=(30, 300), T=3000.0)
    Ns = np.random.default_rng(seed).integers(2, 120 if D <= 24 else 30, size=D)
    return ev, [int(x) for x in Ns]


def _run(ev, Ns, prec, basis, repair):
    import torch
    import paper_2003_02842_gb300 as mm
    tl = TOL[prec]
    Nc = max(Ns)
    plan = mm.mm_plan_create(D=ev.D, N_max=Nc, max_events=ev.n_events, tol=tl["tol"], kernel="es", basis=basis,
                             prec=prec)
    off, t, p = to_dev(ev)
    F, _ = mm.mm_coeffs(plan, off, t, p, Nc)
    S, R, clipped = mm.mm_corr_pairwise(plan, F, Nc, Ns, psd_repair=repair)
    torch.cuda.synchronize()
    st = mm.mm_plan_sync(plan)
    out = dict(S=S.cpu().numpy().astype(np.float64), R=R.cpu().numpy().astype(np.float64),
               clipped=int(clipped.item()), status=st)
    mm.mm_destroy(plan)
    return out


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
@pytest.mark.parametrize("basis", ["dirichlet", "fejer"])
def test_pairwise_cutoffs_match_oracle(prec, basis):
    ev, Ns = _case(0)
    out = _run(ev, Ns, prec, basis, repair=False)
    S_ref, R_ref = oracle.cov_pairwise_cutoffs(ev.offsets, ev.t, ev.logp, Ns, basis=basis)
    assert out["status"] == 0 and out["clipped"] == 0
    assert sigma_err(out["S"], S_ref) <= TOL[prec]["sig"]
    assert np.max(np.abs(out["R"] - R_ref)) <= TOL[prec]["R"]


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
@pytest.mark.parametrize("basis", ["dirichlet", "fejer"])
@pytest.mark.parametrize("seed,D", [(1, 24), (3, 24), (5, 200), (7, 500)])
def test_psd_repair_matches_oracle(prec, basis, seed, D):
    # D = 24: the one-CTA Jacobi iteration in shared memory; D = 200 and 500
    # (the serving workload's largest request): the iteration over every SM.
    # The iteration stops once the off-diagonal norm is below 2 D eps of the
    # matrix norm (eps of its working type), and every element meets about 2D
    # rotations per sweep, so the decomposition's backward error is of order
    # D eps of the norm: the repaired matrix is held to 8 D eps of the norm
    # (about 1e-4 in float32 at D = 200-500, the mixed path's own Sigma
    # tolerance) beyond twice the input's own distance from the oracle's.
    ev, Ns = _case(seed, D=D)
    raw = _run(ev, Ns, prec, basis, repair=False)
    out = _run(ev, Ns, prec, basis, repair=True)
    S_ref, _ = oracle.cov_pairwise_cutoffs(ev.offsets, ev.t, ev.logp, Ns, basis=basis)
    P_ref, neg = oracle.nearest_psd(S_ref)
    assert neg >= 1  # the pairwise estimate is not positive semi-definite here
    assert out["status"] == 0
    # eigenvalues within the iteration's accuracy of zero may fall either way
    lam = np.linalg.eigvalsh(0.5 * (S_ref + S_ref.T))
    eps_w = 1.1e-16 if prec == "fp64" else 6e-8
    tiny = np.sum(np.abs(lam) <= 4 * D * eps_w * np.abs(lam).max())
    assert abs(out["clipped"] - neg) <= tiny
    d_in = np.linalg.norm(raw["S"] - S_ref)
    tol_eig = max(TOL[prec]["eig"], 8 * D * eps_w)
    assert np.linalg.norm(out["S"] - P_ref) <= 2.0 * d_in + tol_eig * np.linalg.norm(S_ref)
    assert np.linalg.eigvalsh(out["S"]).min() >= -max(1e-5, tol_eig) * np.abs(lam).max()
    assert np.max(np.abs(out["R"] - oracle.corr(P_ref))) <= 10 * max(TOL[prec]["R"], tol_eig)


@pytest.mark.parametrize("basis", ["dirichlet", "fejer"])
def test_equal_cutoffs_reduce_to_common_estimate_and_need_no_repair(basis):
    import torch
    import paper_2003_02842_gb300 as mm
    ev, _ = _case(2, D=10)
    N = 60
    plan = mm.mm_plan_create(D=ev.D, N_max=N, max_events=ev.n_events, tol=1e-6, kernel="es", basis=basis)
    off, t, p = to_dev(ev)
    F, _ = mm.mm_coeffs(plan, off, t, p, N)
    S0, R0 = mm.mm_corr(plan, F, N)
    S1, R1, c1 = mm.mm_corr_pairwise(plan, F, N, [N] * ev.D, psd_repair=True)
    torch.cuda.synchronize()
    assert mm.mm_plan_sync(plan) == 0
    assert int(c1.item()) == 0  # a Gram matrix: nothing to clip
    assert sigma_err(S1.cpu().numpy(), S0.cpu().numpy().astype(np.float64)) <= 2e-5
    assert np.max(np.abs(R1.cpu().numpy() - R0.cpu().numpy())) <= 2e-5
    mm.mm_destroy(plan)


def test_pairwise_rejects_bad_arguments():
    import torch
    import paper_2003_02842_gb300 as mm
    ev, Ns = _case(4, D=6)
    Nc = max(Ns)
    plan = mm.mm_plan_create(D=ev.D, N_max=Nc, max_events=ev.n_events, tol=1e-6, kernel="es", basis="fejer")
    off, t, p = to_dev(ev)
    F, _ = mm.mm_coeffs(plan, off, t, p, Nc)
    for bad in ([0] + Ns[1:], [Nc + 1] + Ns[1:], Ns[:-1]):
        with pytest.raises((mm.MMError, ValueError)):
            mm.mm_corr_pairwise(plan, F, Nc, bad)
    mm.mm_destroy(plan)
    D = 4001  # beyond the repair's limit (its rotation arrays fill 48 KB)
    plan = mm.mm_plan_create(D=D, N_max=8, max_events=0, tol=1e-6, kernel="es")
    F = torch.zeros((D, 9), dtype=torch.complex64, device="cuda")
    F[:, 1] = 1.0
    with pytest.raises(mm.MMError):
        mm.mm_corr_pairwise(plan, F, 8, [8] * D, psd_repair=True)
    S, R, c = mm.mm_corr_pairwise(plan, F, 8, [8] * D)
    torch.cuda.synchronize()
    mm.mm_destroy(plan)


@pytest.mark.parametrize("prec,D,repair", [("bf16x3", 20, 3), ("bf16x3", 159, 1), ("fp64", 20, 3), ("fp64", 113, 1)])
def test_launches_are_counted(prec, D, repair):
    # the pairwise sums and the output, and the repair's kernels: iteration, eigenvectors and
    # product where one CTA iterates, one cooperative kernel beyond that
    import torch

    import paper_2003_02842_gb300 as mm
    plan = mm.mm_plan_create(D=D, N_max=30, tol=1e-6, prec=prec)
    F = torch.randn((D, 31), dtype=torch.complex128 if prec == "fp64" else torch.complex64, device="cuda")
    for psd, want in ((False, 2), (True, 2 + repair)):
        before = mm.mm_plan_get_info(plan)["launches"]
        mm.mm_corr_pairwise(plan, F, 30, [30] * D, psd_repair=psd)
        assert mm.mm_plan_get_info(plan)["launches"] - before == want
    mm.mm_plan_sync(plan)
    mm.mm_destroy(plan)


def test_first_use_that_fails_to_clear_its_counters_is_repeated():
    # The first call runs on a stream whose capture has been invalidated (by a host call that
    # a capture does not allow): its allocations succeed, the clearing of the split sums'
    # arrival counters is refused. The next call, on a working stream, has to clear them (in
    # memory that may hold the 0xff bytes written here) and not to meet the first one's error.
    import ctypes

    import torch

    import paper_2003_02842_gb300 as mm
    D, N = 40, 4000
    gen = torch.Generator(device="cuda").manual_seed(5)
    F = torch.randn((D, N + 1), dtype=torch.complex64, device="cuda", generator=gen)
    Ns = [N - 10 * i for i in range(D)]
    fresh = mm.mm_plan_create(D=D, N_max=N, tol=1e-6)
    S0, R0, _ = mm.mm_corr_pairwise(fresh, F, N, Ns)
    assert mm.mm_plan_sync(fresh) == 0

    plan = mm.mm_plan_create(D=D, N_max=N, tol=1e-6)
    R = torch.full((D, D), 7.0, device="cuda")
    stream = torch.cuda.Stream()
    x = torch.full((256 << 20,), 255, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    del x
    torch.cuda.empty_cache()
    cu = ctypes.CDLL("libcuda.so.1")
    h = ctypes.c_void_p(stream.cuda_stream)
    hN = (ctypes.c_int32 * D)(*Ns)
    assert cu.cuStreamBeginCapture_v2(h, 2) == 0  # relaxed: allocations are allowed
    try:
        assert cu.cuStreamSynchronize(h) != 0  # not allowed: invalidates the capture
        st = mm._lib.load().mm_corr_pairwise(plan.handle, ctypes.c_void_p(F.data_ptr()), N, hN, 0, None,
                                             ctypes.c_void_p(R.data_ptr()), None, h)
    finally:
        graph = ctypes.c_void_p()
        cu.cuStreamEndCapture(h, ctypes.byref(graph))
    assert st != 0
    S1, R1, _ = mm.mm_corr_pairwise(plan, F, N, Ns)
    assert mm.mm_plan_sync(plan) == 0
    assert torch.equal(S0, S1) and torch.equal(R0, R1)
    mm.mm_destroy(plan)
    mm.mm_destroy(fresh)


@pytest.mark.parametrize("prec,D", [("fp64", 120), ("bf16x3", 159), ("bf16x3", 560)])
def test_scratch_of_large_matrices(prec, D):
    # matrix, eigenvectors and estimate (float64 D x D each) and up to 1.4 MB of split sums; no
    # log of rotations (4.6 MB at 120 assets in float64) where the whole GPU iterates, no
    # split sums (2.5 MB at 560 assets) where every tile of pairs has one CTA
    import torch

    import paper_2003_02842_gb300 as mm
    plan = mm.mm_plan_create(D=D, N_max=30, tol=1e-6, prec=prec)
    before = mm.mm_plan_get_info(plan)["workspace_bytes"]
    F = torch.randn((D, 31), dtype=torch.complex128 if prec == "fp64" else torch.complex64, device="cuda")
    mm.mm_corr_pairwise(plan, F, 30, [30] * D, psd_repair=True)
    assert mm.mm_plan_sync(plan) == 0
    assert mm.mm_plan_get_info(plan)["workspace_bytes"] - before < 3 * 8 * D * D + 1500000
    mm.mm_destroy(plan)
