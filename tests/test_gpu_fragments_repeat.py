"""Fragment labels of the same state, again and again: the threads of a pass over the parents
run in any order, and the labels do not depend on it."""
import numpy as np
import pytest

import oracle
from paper_2506_05362_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(20000, 1, 1), (60, 20, 9)])
def test_labels_are_the_same_every_time(shape):
    from paper_2506_05362_gb300 import pd
    sc = S.small_block(nx=shape[0], ny=shape[1], nz=shape[2], jitter=0.0)
    sc.horizon = 1.5 * sc.h
    p = np.random.default_rng(2).permutation(sc.n)  # caller order far from the internal one
    sc.x, sc.vol, sc.grain, sc.v0 = sc.x[p], sc.vol[p], sc.grain[p], sc.v0[p]
    ctx = pd.Context.from_scenario(sc, lanes=8)
    rowptr, col = ctx.bonds()
    row = np.repeat(np.arange(sc.n), np.diff(rowptr))
    cut = (sc.x[row, 0] < 7.5 * sc.h) != (sc.x[col, 0] < 7.5 * sc.h)  # one crack, two fragments
    broken = cut.astype(np.uint8)
    ctx.set_state(broken=broken)
    want, nf = oracle.fragments(rowptr, col, broken)
    assert nf == 2
    for _ in range(400):
        label, m = ctx.fragments()
        assert m == 2 and np.array_equal(label, want)
    ctx.close()
