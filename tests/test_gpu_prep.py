"""The records' kernel where its loads and its grid change form: times and prices
that start 8 bytes off a 16-byte boundary, assets shorter than a thread's four
events, a request for some of a server's assets with more events than one pass of
the looped grid takes, and an unsorted time far beyond the window, whose cell does
not fit the fixed-point word. float32 against an FP64 plan (the float32 path's own
rounding at these sizes, at most 1e-6 relative, its parity tests' figure), FP64
against the oracle's direct sum (1e-9: tolerance 1e-12 and the direct sum's own
rounding), a request by the serving form's bounds (1e-4)."""
import numpy as np
import pytest

import oracle
from paper_2003_02842_gb300 import synth

from gpu_helpers import rel_l2_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


def _coeffs(ev, N, prec, tol, shift=0, room=0):
    import torch
    import paper_2003_02842_gb300 as mm

    def dev(a):
        x = torch.zeros(a.size + shift, dtype=torch.from_numpy(a).dtype, device="cuda")
        x[shift:] = torch.from_numpy(a).cuda()
        return x[shift:]

    plan = mm.mm_plan_create(D=ev.D, N_max=N, max_events=ev.n_events + room, tol=tol, kernel="es", prec=prec)
    F, _ = mm.mm_coeffs(plan, torch.from_numpy(ev.offsets).cuda(), dev(ev.t), dev(ev.logp), N)
    assert mm.mm_plan_sync(plan) == 0
    F = F.cpu().numpy().astype(np.complex128)
    mm.mm_destroy(plan)
    return F


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [(2, 7), (1023, 1029), (4000, 5000)])
def test_alignment_and_short_assets(n, shift):
    ev = synth.random_events(n[0], D=9, n_range=n, T=3600.0)
    G = _coeffs(ev, 300, "fp64", 1e-12, shift)
    assert rel_l2_rows(G, oracle.coeffs_F(ev.offsets, ev.t, ev.logp, 300)).max() <= 1e-9
    assert rel_l2_rows(_coeffs(ev, 300, "bf16x3", 1e-6, shift), _coeffs(ev, 300, "fp64", 1e-6, shift)).max() <= 1e-6


def test_request_beyond_one_pass():
    import time
    import paper_2003_02842_gb300 as mm
    n, N = 800_001, 100  # two of three assets: more events than the looped grid takes in a pass
    ev = synth.random_events(3, D=3, n_range=(n, n), T=86400.0)
    srv = mm.mm_server_create(D=3, N_max=N, max_events=ev.n_events, max_slots=1, tol=1e-6, kernel="es", basis="fejer")
    mm.mm_server_load(srv, ev.offsets, ev.t, ev.logp)
    t0, t1 = float(ev.t.min()), float(ev.t.max())
    mm.mm_server_submit(srv, t0, t1, np.array([2, 0], dtype=np.int32), N=N, sigma=True)
    got, end = [], time.time() + 60.0
    while not got and time.time() < end:
        got += mm.mm_server_poll(srv, wait=0.05)
    mm.mm_server_destroy(srv)
    c, = got
    assert c["status"] == 0 and c["N"] == N
    (ta, pa), (tb, pb) = ev.asset(2), ev.asset(0)
    o = oracle.estimate(np.array([0, n, 2 * n]), np.concatenate([ta, tb]), np.concatenate([pa, pb]), N=N,
                        basis="fejer", window=(t0, t1))
    V = np.array([np.sum(np.diff(x) ** 2) for x in (pa, pb)])
    assert np.max(np.abs(c["Sigma"].astype(np.float64) - o["Sigma"]) / np.sqrt(np.outer(V, V))) <= 1e-4
    assert np.max(np.abs(c["R"].astype(np.float64) - o["R"])) <= 1e-4


@pytest.mark.parametrize("prec", ["bf16x3", "fp64"])
@pytest.mark.parametrize("far", [7300.0, 1e9, 1e30])
def test_time_far_beyond_the_window(prec, far):
    import torch
    import paper_2003_02842_gb300 as mm
    ev = synth.random_events(5, D=2, n_range=(500, 500), T=3600.0)
    t = ev.t.copy()
    t[250] = far
    plan = mm.mm_plan_create(D=2, N_max=100, max_events=ev.n_events, kernel="es", prec=prec)
    mm.mm_coeffs(plan, torch.from_numpy(ev.offsets).cuda(), torch.from_numpy(t).cuda(),
                 torch.from_numpy(ev.logp).cuda(), 100)
    assert mm.mm_plan_sync(plan) == 1  # invalid argument, before "unsorted"
    mm.mm_destroy(plan)


def test_float32_offsets_keep_24_significant_bits():
    # One return an asset at cell b + d of 4096 cells of width 1, d in [1/4, 1/2) a multiple of
    # 2^-24, then the same 2^-25 later: the coefficients' phases, -2 pi k (b + d) / 4096, have to
    # turn by 2^-25 of a cell. Rounded to 2^-24 the second set turns by twice that. A tap's
    # float32 rounding moves a single asset by some 1e-7 of a cell, the mean of 4096 by 2.5e-9;
    # the bound is three times that.
    import torch

    import paper_2003_02842_gb300 as mm
    D, N, M = 4096, 1020, 4096.0
    rng = np.random.default_rng(41)
    u = rng.integers(64, 4000, D) + rng.integers(2**22, 2**23, D) * 2.0**-24
    turned = []
    for add in (0.0, 2.0**-25):
        t = np.stack([u + add, np.full(D, M - 1.0)], 1).ravel()
        p = np.tile([0.0, 1.0], D)
        off = np.arange(0, 2 * D + 1, 2, dtype=np.int64)
        plan = mm.mm_plan_create(D=D, N_max=N, max_events=2 * D, tol=1e-6)
        F, _ = mm.mm_coeffs(plan, *[torch.from_numpy(x).cuda() for x in (off, t, p)], N, window=(0.0, M))
        assert mm.mm_plan_sync(plan) == 0 and mm.mm_plan_get_info(plan)["Mr"] == 4096
        mm.mm_destroy(plan)
        k = torch.arange(N + 1, device="cuda", dtype=torch.float64)
        x = torch.from_numpy(u).cuda()
        ref = torch.polar(torch.ones(D, N + 1, device="cuda", dtype=torch.float64),
                          2.0 * np.pi * (torch.frac(x[:, None] * k / M)))
        phase = (F.to(torch.complex128) * ref * 2.0 * np.pi).imag  # -2 pi k (shift) / M
        turned.append(-(phase * k).sum() / (k * k).sum() / D * M / (2.0 * np.pi))
    assert abs(float(turned[1] - turned[0]) - 2.0**-25) <= 2.0**-27
