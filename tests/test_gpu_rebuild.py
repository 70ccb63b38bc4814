"""Contact search against brute force, at the sizes where its kernels split the work:
rows per block, rows with more candidates than a thread collects in its first walk, and
lists that outgrow their room."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def brute(x, rc):
    """Ordered pairs (i, j), i != j, with |x_j - x_i| < rc, FP64 in the library's order of operations."""
    d = x[None, :, :] - x[:, None, :]
    d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    hit = d2 < rc * rc
    np.fill_diagonal(hit, False)
    return np.argwhere(hit).astype(np.int32)


@pytest.mark.parametrize("n,box,capacity", [
    (1, 1.0, 0), (2, 0.5, 0), (127, 4.0, 0), (128, 4.0, 0), (129, 4.0, 0), (1300, 9.0, 0),
    (60, 0.9, 0),        # everyone near everyone: rows of up to 59 candidates
    (900, 5.0, 0),       # rows around the 16 a thread collects at first
    (900, 5.0, 64),      # the list outgrows its room and is rebuilt in a larger one
])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_contact_pairs_match_brute_force(n, box, capacity, precision):
    from paper_2506_05362_gb300 import pd, scenarios as S
    rng = np.random.default_rng(n)
    h = 1e-3
    x = rng.uniform(0.0, box * h, (n, 3))
    mat = S.Material(E=72e9, rho=2440.0, G0=135.0, contact_radius=0.8 * h, contact_factor=0.0)
    ctx = pd.Context(x, np.full(n, h ** 3), np.arange(n, dtype=np.int32), mat, precision=precision, lanes=8,
                     cand_capacity=capacity)
    ctx.build_bonds(1e-6 * h)
    got = ctx.contacts()
    assert np.array_equal(got, brute(x, 0.8 * h))
    # the same from a moved state
    u = rng.uniform(-0.5 * h, 0.5 * h, (n, 3))
    ctx.set_state(u=u)
    uu = ctx.get_state()[0]
    assert np.array_equal(ctx.contacts(), brute(x + uu, 0.8 * h))
    ctx.close()
