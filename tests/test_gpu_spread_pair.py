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

from gpu_helpers import rel_l2_rows, run

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
