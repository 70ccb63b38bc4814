"""Wall reactions summed in parallel over groups, blocks and components: every lane count,
one to six walls, blocks that touch a wall and blocks that do not."""
import numpy as np
import pytest

import oracle
from paper_2506_05362_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


def boxed(nw):
    sc = S.sphere()
    rc = sc.material.contact_radius
    lo, hi = sc.x.min(0), sc.x.max(0)
    sc.walls = []
    for a in range(3):
        for s, q in ((1.0, lo[a] - 0.6 * rc), (-1.0, hi[a] + 0.6 * rc)):
            n, x, v = np.zeros(3), np.zeros(3), np.zeros(3)
            n[a], x[a], v[a] = s, q, 0.5 * s
            sc.walls.append(S.Wall(tuple(n), tuple(x), tuple(v)))
    sc.walls = sc.walls[:nw]
    return sc


@pytest.mark.parametrize("lanes", [4, 8, 16, 32])
@pytest.mark.parametrize("nw", [1, 3, 6])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_reactions_match_the_oracle_and_the_multi_step_kernel(lanes, nw, precision):
    from paper_2506_05362_gb300 import pd
    sc = boxed(nw)
    ref = oracle.Model.from_scenario(sc)
    ref.forces()
    assert np.all(np.abs(ref.react).max(1) > 0)
    areas, out = [1e-6] * nw, []
    for pm in (1, -1):
        ctx = pd.Context.from_scenario(sc, precision=precision, lanes=lanes, tiles=-1, pairs=-1, persistent=pm)
        ctx.forces()
        wf = ctx.bulk_stress(areas)[1]
        # FP64 wall forces on both sides, sums of at most a few thousand terms of one sign
        assert np.abs(wf - ref.react).max() <= 1e-12 * np.abs(ref.react).max()
        ctx.step(0.5 * ctx.stable_dt(), 9)
        out.append([np.asarray(q).copy() for q in ctx.get_state()[:3]] +
                   [ctx.bulk_stress(areas)[1], ctx.bulk_stress_mean(areas)[1], ctx.get_walls()])
        ctx.close()
    for k, (a, b) in enumerate(zip(*out)):
        if k in (3, 4):  # summed over other blocks where the two kernels' grids differ (32 lanes)
            assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
        else:
            assert np.array_equal(a, b)
