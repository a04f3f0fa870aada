"""The float32 scatter on both sides of the densities where its form changes: half
tiles and the widths-first test from a quarter of a record a cell, runs of records
from one record a cell, assets of unequal density in one plan. Against an FP64 plan
of the same tolerance: the float32 path's own rounding at these sizes is at most
1e-6 relative (its parity tests' figure)."""
import numpy as np
import pytest

from paper_2003_02842_gb300 import synth

from gpu_helpers import rel_l2_rows, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


def _coeffs(ev, N, kernel, prec):
    import paper_2003_02842_gb300 as mm
    plan = mm.mm_plan_create(D=ev.D, N_max=N, max_events=ev.n_events, tol=1e-6, kernel=kernel, prec=prec)
    F, _ = mm.mm_coeffs(plan, *to_dev(ev), N)
    assert mm.mm_plan_sync(plan) == 0
    Mr = mm.mm_plan_get_info(plan)["Mr"]
    F = F.cpu().numpy().astype(np.complex128)
    mm.mm_destroy(plan)
    return F, Mr


@pytest.mark.parametrize("kernel", ["es", "gauss"])
@pytest.mark.parametrize("per_cell", [0.24, 0.26, 0.5, 0.99, 1.01, 1.6])
def test_density_edges(per_cell, kernel):
    N = 1500
    n = int(per_cell * 6144)  # M_r at this cutoff
    ev = synth.random_events(n, D=3, n_range=(n // 2, n + n // 2), T=28800.0)
    (F, Mr), (G, _) = _coeffs(ev, N, kernel, "bf16x3"), _coeffs(ev, N, kernel, "fp64")
    assert Mr == 6144
    assert rel_l2_rows(F, G).max() <= 1e-6
