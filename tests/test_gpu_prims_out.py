"""The primitive output divides as IEEE division does, bit for bit: signed zeros,
quotients near and below the smallest normal number, huge and non-finite values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(512,), (64, 9), (24, 9, 5)])
def test_velocity_is_the_quotient(n):
    import paper_2305_09163_gb300 as mfc
    nd, nn = len(n), n + (1,) * (3 - len(n))
    shape = nn[::-1]
    rng = np.random.default_rng(nd)
    q = np.empty((2 + nd,) + shape)
    q[0] = np.exp2(rng.uniform(-20, 20, shape))
    q[1 + nd] = 1e5
    m = np.exp2(rng.uniform(-1070, 1000, (nd,) + shape)) * rng.choice([-1.0, 1.0], (nd,) + shape)
    flat = m.reshape(-1)
    special = [0.0, -0.0, 5e-324, -5e-324, 2.2250738585072014e-308, -1e-309, 1e-300, 1.7e308, -np.inf, np.inf, np.nan]
    flat[::3][:11 * 12] = np.tile(special, 12)
    q[1:1 + nd] = m
    s = mfc.Solver(nn, (0.0,) * 3, (1.0,) * 3, (1,) * 6, (1.4,), (0.0,))
    s.set_state(torch.from_numpy(np.ascontiguousarray(q)).cuda())
    u = s.get_prims().cpu().numpy()[1:1 + nd]
    s.close()
    with np.errstate(all="ignore"):
        want = m / q[0]
    bad = np.isnan(want)
    assert np.array_equal(np.isnan(u), bad)
    assert np.array_equal(u[~bad].view(np.int64), want[~bad].view(np.int64))
