"""The discontinuity sensor of a harvested sample switches at its threshold whatever the
size of the stencil: for tau 1e-6 below and above the value at which the float64
definition switches (its own rounding is ~1e-15, the kernel's float-float ~1e-12)."""
import numpy as np
import pytest

from test_gpu_harvest import _reference

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -30, 2.0 ** -50, 2.0 ** -56, 2.0 ** -59, 2.0 ** -70, 2.0 ** 50])
def test_sensor_threshold(scale):
    import paper_2305_09163_gb300 as mfc
    n, nf, eps, count, seed = (64, 1, 1), 1, 1e-6, 400, 3
    rng = np.random.default_rng(1)
    # steps of one to two units with flat runs between: one stencil's indicator is zero
    # there and the threshold rests on the 1e-6 s^2 term
    w = np.cumsum((rng.random((3, 1, 1, 64)) < 0.2) * rng.uniform(1.0, 2.0, (3, 1, 1, 64)), axis=3) * scale
    lo, hi = np.full(count, 1e-3), np.full(count, 1e9)
    for _ in range(90):
        mid = np.sqrt(lo * hi)
        on = _reference(w, n, count, seed, eps, mid)[3] > 0
        lo, hi = np.where(on, lo, mid), np.where(on, mid, hi)
    picks = np.flatnonzero((hi > 1e4) & (hi < 1e8))[:20]
    assert len(picks) == 20
    wd = torch.from_numpy(w).cuda()
    out = [torch.empty((count, k) if k > 1 else count, dtype=torch.float32, device="cuda") for k in (5, 3, 1, 1, 1)]
    for i in picks:
        for factor, want in ((1 - 1e-6, 0.0), (1 + 1e-6, 1.0)):
            mfc.mfc_harvest(wd, n, nf, eps, float(hi[i] * factor), count, seed, *out)
            assert float(out[3][i]) == want, (i, factor)
