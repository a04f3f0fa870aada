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


def _busy(t_busy, seed):
    """One asset with events at the times t_busy of [0, 6144] (a cell each at N = 1500) among eleven sparse ones."""
    rng = np.random.default_rng(seed)
    ts = [np.unique(np.concatenate([[0.0, 6144.0], rng.uniform(0, 6144, 200)])) for _ in range(11)]
    ts.insert(4, np.unique(np.concatenate([[0.0, 6144.0], t_busy])))
    return synth.from_lists(ts, [4.6 + np.cumsum(0.01 * rng.standard_normal(len(t))) for t in ts])


@pytest.mark.parametrize("kernel", ["es", "kb", "gauss"])
@pytest.mark.parametrize("where", ["all", "first part", "part edge", "tile edge", "row ends"])
def test_busy_asset_in_a_sparse_plan(where, kernel):
    # a plan of less than a quarter of a record a cell has tiles of 4096 cells; a busy asset's are
    # taken in two parts of 2048, each with the records that reach it: spread over the
    # row, in one part alone, around the edges of parts, tiles and row (its periodic images)
    rng = np.random.default_rng(17)
    at = {"all": (0, 6144), "first part": (100, 1900), "part edge": (2030, 2066), "tile edge": (4080, 4112)}
    if where == "row ends":
        t = np.concatenate([rng.uniform(0, 20, 1200), rng.uniform(6124, 6144, 1200)])
    else:
        t = rng.uniform(*at[where], 12000 if where == "all" else 2500)
    ev = _busy(t, 5)
    (F, Mr), (G, _) = _coeffs(ev, 1500, kernel, "bf16x3"), _coeffs(ev, 1500, kernel, "fp64")
    assert Mr == 6144 and 4 * ev.n_events < Mr * ev.D
    assert rel_l2_rows(F, G).max() <= 1e-6
