"""Harvested training samples against the same definitions in numpy float64:
smallest and ragged grids, one to three dimensions and fluids, and values and
epsilons outside the range of the kernel's float-float form.

Tolerance: the stored values are FP32 and at most 8 in magnitude (4.8e-7 of
rounding); the float64 reference subtracts nearly equal values of a stencil that
is at least 1e-7 of its centre (1e-9)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ATOL = 1e-6


def _js(v, eps):
    p = [(2 * v[0] - 7 * v[1] + 11 * v[2]) / 6, (-v[1] + 5 * v[2] + 2 * v[3]) / 6, (2 * v[2] + 5 * v[3] - v[4]) / 6]
    b = [13 / 12 * (v[0] - 2 * v[1] + v[2]) ** 2 + (v[0] - 4 * v[1] + 3 * v[2]) ** 2 / 4,
         13 / 12 * (v[1] - 2 * v[2] + v[3]) ** 2 + (v[1] - v[3]) ** 2 / 4,
         13 / 12 * (v[2] - 2 * v[3] + v[4]) ** 2 + (3 * v[2] - 4 * v[3] + v[4]) ** 2 / 4]
    a = [g / (eps + x) ** 2 for g, x in zip((0.1, 0.6, 0.3), b)]
    return sum(x * y for x, y in zip(a, p)) / sum(a)


def _mix(z):
    u = np.uint64
    z = z + u(0x9E3779B97F4A7C15)
    z = (z ^ (z >> u(30))) * u(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> u(27))) * u(0x94D049BB133111EB)
    return z ^ (z >> u(31))


def _reference(w, n, count, seed, eps, tau):
    u = np.uint64
    nd = 3 if n[2] > 1 else 2 if n[1] > 1 else 1
    nc = [n[a] // 2 if a < nd else 1 for a in range(3)]
    h0 = _mix(u(seed) ^ _mix(np.arange(count, dtype=u)))
    h1 = _mix(h0)
    h2 = _mix(h1)
    h3 = _mix(h2)
    i64 = lambda v: v.astype(np.int64)
    d, side, var = i64(h0 % u(nd)), i64((h0 >> u(20)) & u(1)), i64((h0 >> u(24)) % u(w.shape[0]))
    face = 2 + i64(h1 % np.array([m - 6 for m in nc], dtype=np.int64).astype(u)[d])
    cc = [i64(h2 % u(nc[0])), i64((h2 >> u(21)) % u(nc[1])), i64(h3 % u(nc[2]))]
    stride = [1, n[0], n[0] * n[1]]
    flat, base = w.reshape(-1), var * (n[0] * n[1] * n[2])

    def fetch(along, bits, skip):
        idx = base
        for a in range(nd):
            b = np.where(d < a, (bits >> max(a - 1, 0)) & 1, (bits >> a) & 1) if skip else (bits >> a) & 1
            idx = idx + np.where(d == a, along if skip else 2 * along + b, 2 * cc[a] + b) * stride[a]
        return flat[idx]

    W = [sum(fetch(face - 2 + m, ch, False) for ch in range(2 ** nd)) / 2 ** nd for m in range(6)]
    st = [np.where(side == 0, W[m], W[5 - m]) for m in range(5)]
    tgt = 0.0
    for ch in range(2 ** (nd - 1)):
        f = [fetch(2 * face - 1 + m, ch, True) for m in range(6)]
        tgt = tgt + 0.5 * (_js(f[:5], eps) + _js(f[:0:-1], eps))
    tgt = tgt / 2 ** (nd - 1)
    c = st[2]
    s = np.max([np.abs(v - c) for v in st], axis=0)
    tn = (tgt - c) / (s + 1e-30)
    good = (s > 1e-7 * np.abs(c)) & (s > 1e-300) & (np.abs(tn) <= 8.0)
    s = s + 1e-30
    z = lambda v: np.where(good, v, 0.0)
    x = [z((v - c) / s) for v in st]
    ph = [z((2 * st[0] - 7 * st[1] + 11 * st[2]) / 6 / s - c / s), z((-st[1] + 5 * st[2] + 2 * st[3]) / 6 / s - c / s),
          z((2 * st[2] + 5 * st[3] - st[4]) / 6 / s - c / s)]
    D = [st[k + 1] - st[k] for k in range(4)]
    b = np.array([2.5 * D[1] ** 2 - 2.75 * D[1] * D[0] + D[0] ** 2, D[1] ** 2 + D[2] ** 2 - 1.25 * D[1] * D[2],
                  2.5 * D[2] ** 2 - 2.75 * D[2] * D[3] + D[3] ** 2])
    smooth = good & ~(b.max(0) > tau * (b.min(0) + 1e-6 * s * s))
    return np.stack(x, 1), np.stack(ph, 1), z(tn), smooth.astype(np.float64), z((_js(st, eps) - c) / s)


@pytest.mark.parametrize("n,nf", [((16, 1, 1), 1), ((40, 1, 1), 3), ((16, 16, 1), 2), ((34, 18, 1), 2),
                                  ((16, 16, 16), 2), ((20, 18, 22), 1), ((18, 24, 16), 3)])
@pytest.mark.parametrize("scale,eps", [(1.0, 1e-6), (1e9, 1e-30), (3e17, 1e-6), (1e-19, 1e-6), (1.0, 1e-40)])
def test_harvest_matches_float64(n, nf, scale, eps):
    import paper_2305_09163_gb300 as mfc
    nd = 3 if n[2] > 1 else 2 if n[1] > 1 else 1
    rng = np.random.default_rng(n[0] + nf)
    # a smooth field, noise, and flat blocks whose stencils are stored as zeros
    w = np.cumsum(rng.standard_normal((2 * nf + nd, n[2], n[1], n[0])), axis=3)
    w[:, :, :, : n[0] // 4] = w[:, :1, :1, :1]
    w *= scale
    count = 3001
    out = [torch.empty((count, k) if k > 1 else count, dtype=torch.float32, device="cuda") for k in (5, 3, 1, 1, 1)]
    mfc.mfc_harvest(torch.from_numpy(w).cuda(), n, nf, eps, 100.0, count, 17, *out)
    for got, want in zip(out, _reference(w, n, count, 17, eps, 100.0)):
        assert np.abs(got.cpu().numpy() - want).max() <= ATOL
