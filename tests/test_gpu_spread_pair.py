"""The FP64 path's float-pair spreading against float64 throughout (the gather
variant) on the same plan otherwise, and against the oracle.

Tolerance between the two: a tap's error is at most 7e-15 of the kernel's peak
and each grid cell's error is then at most that times the returns it gathers;
the transform and deconvolution raise high modes by up to the ratio of the
kernel's transform, about 10 at tol 1e-12. 1e-13 of the coefficients' norm (a
tenth of the tolerance the plan was asked for) covers both."""
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


def _both(ev, N, kernel, tile, tol=1e-12):
    kw = dict(tol=tol, kernel=kernel, basis="dirichlet", prec="fp64", spread_tile=tile)
    out = run(dict(kw, spread_algo="scatter"), ev, N)
    ref = run(dict(kw, spread_algo="gather"), ev, N)
    assert out["status"] == ref["status"]
    return out["F"], ref["F"]


@pytest.mark.parametrize("kernel", ["es", "kb", "gauss"])
@pytest.mark.parametrize("tile,N", [(0, 1), (0, 30), (37, 200), (0, 1023), (0, 5000), (2048, 4096)])
def test_pair_taps_match_float64_taps(kernel, tile, N):
    ev = synth.random_events(60 + N, D=3, n_range=(300, 2500), T=4000.0, grid=4001 if N == 1023 else None)
    F, G = _both(ev, N, kernel, tile)
    assert rel_l2_rows(F, G).max() <= 1e-13


@pytest.mark.parametrize("N", [1, 40, 700])
def test_dense_tiles(N):
    # whole warps of records in one cell, several staged chunks per tile
    ev = synth.random_events(7, D=2, n_range=(30000, 30000), T=28800.0)
    F, G = _both(ev, N, "es", 0)
    assert rel_l2_rows(F, G).max() <= 1e-13
    assert rel_l2_rows(F, oracle.coeffs_F(ev.offsets, ev.t, ev.logp, N)).max() <= 1e-10


@pytest.mark.parametrize("scale", [2.0**-900, 2.0**-300, 2.0**300, 2.0**900])
def test_returns_of_any_magnitude(scale):
    # a power of two scales every step exactly
    ev = synth.random_events(8, D=2, n_range=(50, 400), T=1000.0)
    F0, _ = _both(ev, 100, "es", 0)
    big = synth.Events(ev.offsets, ev.t, (ev.logp - 4.6) * scale)
    one = synth.Events(ev.offsets, ev.t, ev.logp - 4.6)
    F1, _ = _both(one, 100, "es", 0)
    F2, G2 = _both(big, 100, "es", 0)
    assert rel_l2_rows(F2 / scale, F1).max() <= 1e-15 and rel_l2_rows(F1, F0).max() <= 1e-11
    assert rel_l2_rows(F2 / scale, G2 / scale).max() <= 1e-13


def test_tight_tolerances_keep_float64_taps():
    # below the pair taps' range both variants evaluate the kernel in float64
    ev = synth.random_events(9, D=2, n_range=(100, 500), T=1000.0)
    F, G = _both(ev, 300, "es", 0, tol=1e-14)
    assert rel_l2_rows(F, G).max() <= 2e-15


def _coeffs(ev, N, algo, kernel="es", tol=1e-12):
    import paper_2003_02842_gb300 as mm
    plan = mm.mm_plan_create(D=ev.D, N_max=N, max_events=ev.n_events, tol=tol, kernel=kernel, prec="fp64",
                             spread_algo=algo)
    F, _ = mm.mm_coeffs(plan, *to_dev(ev), N)
    mm.mm_plan_sync(plan)
    F = F.cpu().numpy()
    mm.mm_destroy(plan)
    return F


@pytest.mark.parametrize("size", [0.9 * 2.0**1023, 1.2 * 2.0**1023, 1.9 * 2.0**1023])
def test_returns_at_the_top_of_float64(size):
    # four returns of +-size (their exponent's power, 2^1024, is beyond float64 from 2^1023 on);
    # a coefficient is at most 4 size / (2 pi), finite. The oracle works on 2^-1000 of them
    t = np.array([0.0, 130.0, 377.0, 781.5, 1000.0])
    ev = synth.from_lists([t], [0.5 * size * (-1.0) ** np.arange(5)])
    F = _coeffs(ev, 60, "scatter")
    ref = oracle.coeffs_F(ev.offsets, ev.t, ev.logp * 2.0**-1000, 60)
    assert np.isfinite(F).all()
    assert rel_l2_rows(F * 2.0**-1000, ref).max() <= 1e-11


def test_a_return_beyond_float64_gives_nan():
    ev = synth.random_events(11, D=2, n_range=(60, 90), T=1000.0)
    p = ev.logp.copy()
    p[10], p[11] = 1.7e308, -1.7e308  # the first asset's return overflows
    ev = synth.Events(ev.offsets, ev.t, p)
    F, G = _coeffs(ev, 40, "scatter"), _coeffs(ev, 40, "gather")
    assert np.isnan(F[0]).all() and not np.isfinite(G[0]).any()
    assert rel_l2_rows(F[1:], G[1:]).max() <= 1e-13


def test_subnormal_returns():
    # returns below 2^-1022, some 40 bits above float64's last place (2^-1074)
    ev = synth.random_events(12, D=2, n_range=(60, 90), T=1000.0)
    ev = synth.Events(ev.offsets, ev.t, (ev.logp - 4.6) * 2.0**-1024)
    assert np.abs(np.diff(ev.logp)).max() < 2.0**-1022
    F, G = _coeffs(ev, 40, "scatter") * 2.0**1000, _coeffs(ev, 40, "gather") * 2.0**1000
    assert np.linalg.norm(G) > 0 and rel_l2_rows(F, G).max() <= 1e-9


def _mode_errors(ev, N, kernel, tol):
    """|scatter - gather| (float64 throughout) of each mode, rms over the rows, in units of a row's rms."""
    F, G = _coeffs(ev, N, "scatter", kernel, tol), _coeffs(ev, N, "gather", kernel, tol)
    rms = np.sqrt((np.abs(G) ** 2).mean(1, keepdims=True))
    return np.sqrt(((np.abs(F - G) / rms) ** 2).mean(0))


@pytest.mark.parametrize("kernel", ["es", "kb", "gauss"])
@pytest.mark.parametrize("N", [30, 700, 4096, 10124, 20000])
def test_modes_next_to_the_cutoff(kernel, N):
    # The deconvolution raises the pairs' rounding most there; what is promised is half the
    # tolerance, rms over the last fiftieth of the modes, and a tenth of it over a row
    ev = synth.random_events(70 + N, D=6, n_range=(200, 6000), T=28800.0)
    for tol in (1e-10, 1e-12):
        e = _mode_errors(ev, N, kernel, tol)
        assert np.sqrt((e[-max(1, (N + 1) // 50):] ** 2).mean()) <= 0.5 * tol
        assert np.sqrt((e**2).mean()) <= 1e-13


@pytest.mark.parametrize("kernel", ["es", "kb", "gauss"])
@pytest.mark.parametrize("N", [30, 700, 1000, 5000])
def test_pairs_from_a_tolerance_of_1e_12(kernel, N):
    # Two float64 paths that only add in another order agree to some 1e-15 of a row's rms, the
    # pairs differ by 1e-14 and more: which one ran shows on both sides of the line
    ev = synth.random_events(90 + N, D=4, n_range=(200, 3000), T=28800.0)
    rms = {tol: float(np.sqrt((_mode_errors(ev, N, kernel, tol) ** 2).mean())) for tol in (1e-12, 9.9e-13)}
    assert rms[1e-12] > 4e-15 and rms[9.9e-13] < 3e-15


@pytest.mark.parametrize("kernel", ["es", "kb", "gauss"])
def test_a_plan_at_one_cutoff_after_another(kernel):
    # the fit that a plan keeps over cutoffs is the one that each cutoff needs: a new plan's
    # coefficients, bit for bit (integer sums, a transform in a fixed order)
    import paper_2003_02842_gb300 as mm
    ev = synth.random_events(13, D=2, n_range=(100, 900), T=5000.0)
    x = to_dev(ev)
    plan = mm.mm_plan_create(D=2, N_max=3000, max_events=ev.n_events, tol=1e-12, kernel=kernel, prec="fp64")
    for N in (700, 701, 31, 3000, 700, 1024):
        F, _ = mm.mm_coeffs(plan, *x, N)
        assert mm.mm_plan_sync(plan) == 0
        assert np.array_equal(F.cpu().numpy(), _coeffs(ev, N, "scatter", kernel))
    mm.mm_destroy(plan)
