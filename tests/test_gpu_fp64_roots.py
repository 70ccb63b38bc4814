"""Bond lengths of the FP64 path over the whole range of their exponent, zero included: many
grains of two nodes each, the bond of every grain of another length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
H = 1e-3


def pairs(n, G0, break_mode):
    """A context of n two-node grains along y (bond along x), and their reference positions."""
    from paper_2506_05362_gb300 import pd, scenarios as S
    x = np.zeros((2 * n, 3))
    x[1::2, 0] = H
    x[:, 1] = np.repeat(np.arange(n), 2) * 4 * H
    mat = S.Material(E=72e9, rho=2440.0, G0=G0, contact_radius=0.8 * H, break_mode=break_mode)
    ctx = pd.Context(x, np.full(2 * n, H ** 3), np.repeat(np.arange(n, dtype=np.int32), 2), mat, precision="fp64",
                     contact=False, lanes=8)
    ctx.build_bonds(1.5 * H)
    assert ctx.B == 2 * n
    return ctx


def test_lengths_from_2e_minus_140_to_2e_plus_140():
    e = np.linspace(-140.0, 140.0, 1201)
    length = 2.0 * 10.0 ** e * np.random.default_rng(1).uniform(0.5, 1.0, e.size)
    ctx = pairs(e.size, 1e306, 0)  # s0 of some 1e148: nothing breaks
    # the bond of grain g from (H, 0, 0) to length[g] along z
    u = np.zeros((2 * e.size, 3))
    u[1::2, 0] = -H
    u[1::2, 2] = length
    ctx.set_state(u=u)
    F = ctx.forces()
    K = 2.0 * 72e9 / 3.0
    c = 18.0 * K / (np.pi * (1.5 * H) ** 4)
    want = c * ((length - H) / H) * H ** 3  # c s V
    # a root good to an ulp, the roundings of strain and products, and those of c on both sides:
    # some 20 half ulps of the larger of the two lengths the strain compares
    tol = 3e-15 * c * np.maximum(length, H) / H * H ** 3
    assert np.all(np.abs(F[0::2, 2] - want) <= tol)
    assert np.all(np.abs(F[1::2, 2] + want) <= tol)
    assert not F[:, :2].any() and not ctx.get_state()[2].any()
    ctx.close()


@pytest.mark.parametrize("length", [0.0, 5e-324, 1e-200, 1e-155, 1e160, 1e300])
def test_lengths_beyond_the_range_break(length):
    """|s| = 1 of a bond whose ends meet, |s| beyond any s0 of one whose square overflows: both
    break, and the step goes on."""
    ctx = pairs(40, 135.0, 1)
    u = np.zeros((80, 3))
    u[1::2, 0] = -H
    u[1::2, 2] = length
    u[2:, :] = 0.0  # the first grain only
    ctx.set_state(u=u)
    broken = np.asarray(ctx.get_state()[2])
    assert broken[:2].all() and not broken[2:].any()
    assert not ctx.forces().any()
    ctx.step(1e-9, 3)
    assert np.array_equal(ctx.get_state()[0], u)
    ctx.close()


@pytest.mark.parametrize("jitter", [0.0, 0.05])
def test_a_body_at_rest_or_moved_as_a_whole_has_no_force(jitter):
    from paper_2506_05362_gb300 import pd, scenarios as S
    sc = S.small_block(nx=9, ny=8, nz=7, jitter=jitter)
    ctx = pd.Context.from_scenario(sc, precision="fp64")
    assert not ctx.forces().any()
    u = np.zeros(sc.x.shape) + np.array([1.0, -2.0, 0.5]) * sc.h  # the same for every node: no difference at all
    ctx.set_state(u=u)
    assert not ctx.forces().any()
    ctx.close()
