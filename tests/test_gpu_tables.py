"""Per-cutoff tables: the mixed-precision plans' deconvolution factors of the
ES kernel come from a Chebyshev series of its transform, the FP64 plans' from
the quadrature itself. Both plans of one tolerance spread with the same kernel
on the same grid, so their coefficients share the kernel's truncation error
and differ by the float32 path's own rounding only: at most 1e-6 relative
(its parity tests bound that rounding by the same figure). A repeated call at
another cutoff rebuilds the tables."""
import numpy as np
import pytest

from paper_2003_02842_gb300 import synth

from gpu_helpers import rel_l2_rows, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


# half-widths M_sp = 3, 5, 7, 9, 14 (the series has 15 to 25 terms; stencils of more than 32 points are refused)
@pytest.mark.parametrize("tol", [0.3, 1e-4, 1e-8, 1e-12, 1e-22])
def test_mixed_tables_follow_the_quadrature(tol):
    import paper_2003_02842_gb300 as mm
    ev = synth.random_events(91, D=3, n_range=(200, 400), T=2000.0)
    off, t, p = to_dev(ev)
    plans = [mm.mm_plan_create(D=ev.D, N_max=3000, max_events=ev.n_events, tol=tol, kernel="es", prec=prec)
             for prec in ("bf16x3", "fp64")]
    for N in (1, 2, 40, 1000, 3000, 999):
        F = [mm.mm_coeffs(plan, off, t, p, N)[0].cpu().numpy() for plan in plans]
        assert [mm.mm_plan_sync(plan) for plan in plans] == [0, 0]
        assert rel_l2_rows(F[0], F[1]).max() <= 1e-6
    for plan in plans:
        mm.mm_destroy(plan)
