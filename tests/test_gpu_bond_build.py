"""Bond lists against the oracle where the bond build splits its work: short rows, rows
of several 32-element chunks, rows longer than the staged 512, caller orders that are not
the internal one, and both filters."""
import numpy as np
import pytest

import oracle
from paper_2506_05362_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [1.05, 1.8, 2.5, 4.2, 6.3])
@pytest.mark.parametrize("filters", ["none", "notch", "sphere", "both"])
def test_bond_lists_match_oracle(cells, filters):
    from paper_2506_05362_gb300 import pd
    sc = S.small_block(nx=13, ny=12, nz=11, jitter=0.0 if cells == 2.5 else 0.02)
    h = sc.h
    sc.horizon = cells * h
    p = np.random.default_rng(3).permutation(sc.n)
    sc.x, sc.vol, sc.grain, sc.v0 = sc.x[p], sc.vol[p], (p % 2 if cells < 2 else 0 * p).astype(np.int32), sc.v0[p]
    f = []
    if filters in ("notch", "both"):  # half of the plane between two layers, and one through a layer of nodes
        f.append((S.FILTER_NOTCH, [0.0, 1.0, 0.0, -5.5 * h, -h, 5.4 * h, -h, 6.0 * h, 5.6 * h, 20 * h, 0.0, 0.0]))
        f.append((S.FILTER_NOTCH, [1.0, 0.0, 0.0, -4.0 * h, 3.9 * h, -h, -h, 4.1 * h, 4.0 * h, 20 * h, 0.0, 0.0]))
    if filters in ("sphere", "both"):
        f.append((S.FILTER_SPHERE, [6.0 * h, 6.0 * h, 5.0 * h, 2.0 * h] + [0.0] * 8))
    sc.filters = f
    ctx = pd.Context.from_scenario(sc, lanes=8)
    ref = oracle.Model.from_scenario(sc)
    rp, col = ctx.bonds()
    assert np.array_equal(rp, ref.rowptr) and np.array_equal(col, ref.col)
    if cells > 6:
        assert np.diff(rp).max() > 512
    ctx.close()
