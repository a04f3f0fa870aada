"""The float32 scatter's choice between one word per cell (sparse tiles) and two
(dense ones), at its edges: stencils' widths holding 20 and 21 records, 1024
and 1025 records in a tile, dense tiles larger than half the shared words, odd
tile sizes, one return dwarfing the others, returns near the ends of the float
range. Against an FP64 plan of the same tolerance, which shares the kernel's
truncation: the float32 path's own rounding is at most 1e-6 relative (its parity
tests bound it by the same figure); and the oracle's direct sum (Eq. (15) <=
1e-5)."""
import numpy as np
import pytest

import oracle
from paper_2003_02842_gb300 import synth

from gpu_helpers import rel_l2_rows, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


def _coeffs(ev, N, kernel, prec, tile=0, tol=1e-6):
    import paper_2003_02842_gb300 as mm
    plan = mm.mm_plan_create(D=ev.D, N_max=N, max_events=ev.n_events, tol=tol, kernel=kernel, prec=prec,
                             spread_tile=tile)
    F, _ = mm.mm_coeffs(plan, *to_dev(ev), N)
    assert mm.mm_plan_sync(plan) == 0
    F = F.cpu().numpy()
    mm.mm_destroy(plan)
    return F.astype(np.complex128)


def _check(ev, N, kernel="es", tile=0, scale=1.0):
    F, G = _coeffs(ev, N, kernel, "bf16x3", tile) / scale, _coeffs(ev, N, kernel, "fp64") / scale
    assert rel_l2_rows(F, G).max() <= 1e-6
    assert rel_l2_rows(F, oracle.coeffs_F(ev.offsets, ev.t, ev.logp, N) / scale).max() <= 1e-5


def _clusters(per, N, seed=0):
    # clusters of `per` records inside a few cells, between empty stretches
    rng = np.random.default_rng([per, N, seed])
    T, cell = 10000.0, 10000.0 / (4 * N + 2)
    t = np.sort(np.concatenate([[0.0, T], (np.arange(20)[:, None] * 500 + 7.3 +
                                           rng.uniform(0, 8 * cell, (20, per))).ravel()]))
    p = 4.6 + np.cumsum(0.01 * rng.standard_normal(len(t)))
    return synth.from_lists([t, t[::2]], [p, p[::2]])


@pytest.mark.parametrize("kernel", ["es", "kb", "gauss"])
@pytest.mark.parametrize("per", [19, 20, 21, 40])
def test_records_per_stencil_width(kernel, per):
    _check(_clusters(per, 900), 900, kernel)


@pytest.mark.parametrize("n", [1024, 1025, 1026, 3000])
@pytest.mark.parametrize("tile", [0, 37, 2047, 4095])
def test_chunk_and_tile_edges(n, tile):
    ev = synth.random_events(n + tile, D=2, n_range=(n, n), T=5000.0)
    _check(ev, 1000, tile=tile)


@pytest.mark.parametrize("N,n", [(1000, 20000), (2100, 60000), (500, 4000)])
def test_dense_tiles_in_parts(N, n):
    ev = synth.random_events(n, D=2, n_range=(n, n), T=28800.0)
    _check(ev, N, tile=4096)
    _check(ev, N)


@pytest.mark.parametrize("scale", [2.0**-100, 2.0**-92, 2.0**-80, 2.0**80])
def test_returns_near_the_float_range(scale):
    ev = synth.random_events(5, D=2, n_range=(300, 600), T=2000.0)
    _check(synth.Events(ev.offsets, ev.t, (ev.logp - 4.6) * scale), 700, scale=scale)


def test_one_return_dwarfs_the_others():
    ev = synth.random_events(6, D=2, n_range=(500, 600), T=2000.0)
    lp = ev.logp.copy()
    lp[100:] += 1.0e4
    _check(synth.Events(ev.offsets, ev.t, lp), 700)


def test_small_returns_beside_a_large_one_keep_their_digits():
    # One return of 1 among 5300 of 2^-32 to 2^-30.4, all of one sign, in one tile of 4096 cells
    # with at most 20 records in any stencil's width. Each is below half the quantum that the
    # large one would set for one word a cell (2^-29); together they are 2.5e-6 of it, 20 times
    # the float32 rounding of the transform of both. What they add to the coefficients is
    # taken against the large return alone.
    n, N = 5300, 1020
    u = (np.arange(n + 1) + 0.25 * np.sin(np.arange(n + 1))) / n
    u[0], u[-1] = 0.0, 1.0
    v = 2.0**-31 * (1.0 + 0.5 * np.cos(6.0 * np.pi * u[:-1]))
    one = np.zeros(n)
    one[n // 3] = 1.0

    def coeffs(r):
        ev = synth.from_lists([u * 1000.0], [np.concatenate([[0.0], np.cumsum(r)])])
        return ev, _coeffs(ev, N, "es", "bf16x3", tile=4096)[0]

    ev, F = coeffs(one + v)
    _, F1 = coeffs(one)
    small = synth.Events(ev.offsets, ev.t, np.concatenate([[0.0], np.cumsum(v)]))
    ref = oracle.coeffs_F(small.offsets, small.t, small.logp, N)[0]
    assert np.abs((F - F1 - ref)[:6]).max() <= 0.3 * abs(ref[0])


@pytest.mark.parametrize("kernel,tol,msp", [("gauss", 1e-8, 9), ("gauss", 1e-11, 12), ("gauss", 1e-12, 13), ("es", 1e-12, 9)])
@pytest.mark.parametrize("n", [300, 9000])
def test_wide_stencils(kernel, tol, msp, n):
    # 18 to 26 taps (24 and 25 on both sides of an instantiation), sparse and dense tiles
    import paper_2003_02842_gb300 as mm
    ev = synth.random_events(n, D=2, n_range=(n, n), T=5000.0)
    plan = mm.mm_plan_create(D=2, N_max=1000, max_events=ev.n_events, tol=tol, kernel=kernel)
    F, _ = mm.mm_coeffs(plan, *to_dev(ev), 1000)
    info = mm.mm_plan_get_info(plan)
    assert mm.mm_plan_sync(plan) == 0 and info["msp"] == msp and info["spread_poly"] == 1
    F = F.cpu().numpy().astype(np.complex128)
    mm.mm_destroy(plan)
    assert rel_l2_rows(F, _coeffs(ev, 1000, kernel, "fp64", tol=tol)).max() <= 1e-6


@pytest.mark.parametrize("tol", [1e-6, 1e-3])
@pytest.mark.parametrize("run", [0.94, 0.9411, 0.9412, 0.9999, 1.0001, 1.88, 1.883])
def test_one_word_filled_to_its_last_bit(run, tol):
    # 30 groups of 20 records within a ten-thousandth of a cell, of one sign: a cell gets the
    # whole sum of a run, `run`, around the powers of two where the word's scale changes
    # (run times 1.0625 below and above one and two); an overflow would turn the sign
    import torch

    import paper_2003_02842_gb300 as mm
    N, T = 1020, 4096.0
    t = (128.0 * np.arange(1, 31)[:, None] + 1e-5 * np.arange(20)[None, :]).ravel()
    p = np.arange(len(t) + 1) * (run / 20)
    off = torch.tensor([0, len(t) + 1]).cuda()
    x = (off, torch.from_numpy(np.append(t, 4090.0)).cuda(), torch.from_numpy(p).cuda())
    F = []
    for prec in ("bf16x3", "fp64"):
        plan = mm.mm_plan_create(D=1, N_max=N, max_events=len(p), tol=tol, prec=prec)
        c, _ = mm.mm_coeffs(plan, *x, N, window=(0.0, T))
        assert mm.mm_plan_sync(plan) == 0 and mm.mm_plan_get_info(plan)["Mr"] == 4096
        F.append(c.cpu().numpy().astype(np.complex128))
        mm.mm_destroy(plan)
    assert rel_l2_rows(F[0], F[1]).max() <= max(1e-6, 0.2 * tol)
