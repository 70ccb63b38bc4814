"""A segment whose contact list goes stale is taken up again at the step it stopped in:
the same bits as rebuilding every step (a list's superset does not change any sum)."""
import numpy as np
import pytest

from test_gpu_failures import colliding_pair

pytestmark = pytest.mark.gpu


def run(sc, calls, **kw):
    from paper_2506_05362_gb300 import pd, scenarios as S
    ctx = pd.Context.from_scenario(sc, **kw)
    walls = [S.Wall((0.0, 0.0, 1.0), (0.0, 0.0, float(sc.x[:, 2].min()) - 2e-4), (0.0, 0.0, 20.0))]
    ctx.set_walls(S.walls_array(walls))
    dt = 0.5 * ctx.stable_dt()
    for n in calls:
        ctx.step(dt, n)
    u, v, b, t = ctx.get_state()
    out = [np.asarray(q).copy() for q in (u, v, b, ctx.get_walls())], ctx.step_counters(), t
    ctx.close()
    return out


# rebuild periods beyond what the list lasts, chunks of 1 to 64 steps (the list goes stale in
# the first chunk, a later one, in a chunk's last step), several segments, calls of odd length
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("persistent", [-1, 1])
@pytest.mark.parametrize("chunk,every,calls", [(64, 40, [150]), (7, 6, [33, 40]), (16, 15, [16, 17, 1, 64]),
                                               (64, 64, [65, 2])])
def test_resumed_segment_gives_the_bits_of_a_rebuild_every_step(precision, persistent, chunk, every, calls):
    sc = colliding_pair(speed=12.0)
    kw = dict(precision=precision, persistent=persistent, skin=0.01 * sc.material.contact_radius)
    want, (n0, r0, b0), t0 = run(sc, calls, contact_every=1, **kw)
    got, (n1, r1, b1), t1 = run(sc, calls, contact_every=every, chunk=chunk, **kw)
    assert b0 == 0 and b1 > 0
    assert n0 == n1 == sum(calls)
    assert sum(calls) / every < r1 < r0
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    # the time is summed over segments, whose lengths follow the period: at most 150 roundings
    assert abs(t1 - t0) <= 150 * 2.0 ** -53 * t0
