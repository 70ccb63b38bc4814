"""The multi-step kernel where each step reads what other SMs wrote in the step before:
touching grains with damping and friction, positions that decide contacts, bonds that break
and stay broken.  The same bits as one launch a step."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,lanes", [("mixed", 8), ("mixed", 32), ("fp64", 16)])
@pytest.mark.parametrize("beta,mu", [(0.0, 0.0), (0.4, 0.0), (0.4, 0.3)])
def test_multi_step_kernel_sees_the_step_before(precision, lanes, beta, mu):
    from paper_2506_05362_gb300 import pd, scenarios as S, surrogate
    sc = S.shape_study("sphere", n_side=2, seed=3, gap_cells=-1.45)
    if beta:
        sc.material.beta_d = surrogate.damping_coefficient(sc.material, sc.horizon, float(sc.vol.mean()), beta)
    sc.material.mu = mu
    rng = np.random.default_rng(5)
    # grains thrown at the middle of the box, fast enough to break bonds where they meet
    c = np.stack([sc.x[sc.grain == g].mean(0) for g in range(int(sc.grain.max()) + 1)])
    sc.v0 = -40.0 * ((c - c.mean(0)) / np.linalg.norm(c - c.mean(0), axis=1)[:, None])[sc.grain]
    sc.v0 = sc.v0 + rng.normal(0.0, 0.5, sc.x.shape)
    out = []
    for persistent in (1, -1):
        ctx = pd.Context.from_scenario(sc, precision=precision, lanes=lanes, persistent=persistent)
        ctx.step(0.5 * ctx.stable_dt(), 400)
        u, v, broken, _ = ctx.get_state()
        out.append([np.asarray(q).copy() for q in (u, v, broken)] + [ctx.contacts()])
        ctx.close()
    assert out[1][2].any() and len(out[1][3]) > 0
    for a, b in zip(*out):
        assert np.array_equal(a, b)
