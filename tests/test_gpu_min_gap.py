"""The Nyquist cutoff where an asset's gaps are shared by several blocks: sizes
on both sides of a block's 1024 gaps, one to many assets, assets of no and of one
event, the deciding gap at the ends and between two blocks, and the words that
the blocks meet in cleared between calls, a refused one included. The cutoff is
a whole number and equals the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()


def _case(D, n, seed):
    """Asset i: n events (asset 1 none, asset 2 one) with gaps of 16..31 and one of 4 + i % 8."""
    rng = np.random.default_rng(seed)
    off, ts = [0], []
    for i in range(D):
        m = 0 if i == 1 else 1 if i == 2 else n
        g = rng.integers(16, 32, size=max(m - 1, 0)).astype(np.float64)
        if g.size:
            g[min(g.size - 1, (0, g.size - 1, 1022, 1023, 1024)[i % 5])] = 4 + i % 8
        ts.append(np.concatenate([[0.0], np.cumsum(g)])[:m] + (0.0 if i == 0 else 1.0))
        off.append(off[-1] + m)
    return np.array(off, dtype=np.int64), np.concatenate(ts)


@pytest.mark.parametrize("D", [1, 5, 300])
@pytest.mark.parametrize("n", [2, 257, 1024, 1025, 1026, 2050, 9000])
def test_cutoff_equals_oracle(D, n):
    import torch
    import paper_2003_02842_gb300 as mm
    off, t = _case(D, n, 7 * D + n)
    dev = lambda a: torch.from_numpy(a).cuda()
    plan = mm.mm_plan_create(D=D, N_max=8, max_events=int(off[-1]), tol=1e-6, kernel="es", basis="fejer")
    want = oracle.nyquist(off, t, t.min(), t.max())
    assert mm.mm_nyquist(plan, dev(off), dev(t)) == want
    bad = t.copy()
    bad[1] = bad[0]  # a duplicate time: refused, and nothing of it left behind
    with pytest.raises(mm.MMError):
        mm.mm_nyquist(plan, dev(off), dev(bad))
    half = np.floor(t / 2.0)  # halved gaps of at least 2 stay positive
    assert mm.mm_nyquist(plan, dev(off), dev(half)) == oracle.nyquist(off, half, half.min(), half.max())
    mm.mm_destroy(plan)
