"""The FP64 path's range does not depend on the cell size: a state near the top of
the documented range (pressure and velocity 2e17, energy flux ~1e36) in a box of
2^-20 must give the right-hand side of the unit box times 2^20 and the same state
after a step of 2^-20 the length, bit for bit (every factor is a power of two).
The rates of the small box are ~1e43, above the float32 range."""
import numpy as np
import pytest

import oracle
import workloads
from parity_util import rhs_error

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOP, SHRINK = 2e17, 2.0 ** -20


def _prims(n, nf, model):
    w = workloads.random_prims(n, nf, seed=5, water_air=False)
    nd = len(n)
    u, p = w[nf:nf + nd], w[nf + nd]
    u *= TOP / np.abs(u).max()
    p *= TOP / p.max()
    w[:nf] *= 1.0 / TOP
    w = np.ascontiguousarray(w)
    return workloads.six_equation_prims(w, nf, spread=0.0, seed=6) if model == 2 else w


def _solver(n, nf, size, bc, stretched, params):
    import paper_2305_09163_gb300 as mfc
    gam, pin = workloads.fluids(nf, water_air=False)
    nn = tuple(n) + (1,) * (3 - len(n))
    s = mfc.Solver(nn, (0.0,) * 3, (size,) * 3, (bc,) * (2 * len(n)) + (1,) * (6 - 2 * len(n)), gam, pin, **params)
    if stretched:
        for d, m in enumerate(n):
            h = np.random.default_rng(d).uniform(0.5, 2.0, m)
            s.set_grid(d, size * np.concatenate([[0.0], np.cumsum(h)]) / m)
    return s


@pytest.mark.parametrize("n,nf,bc,stretched,params", [
    ((131,), 1, 1, False, {}), ((70,), 2, 0, False, {}), ((37, 29), 2, 2, False, {}), ((21, 19, 17), 2, 1, False, {}),
    ((21, 19, 17), 3, 0, False, {}), ((23, 18), 2, 3, False, {}), ((21, 19, 17), 2, 3, True, {}),
    ((19, 22, 17), 2, 1, False, {"weno_order": 3}), ((19, 22, 17), 2, 1, False, {"model": 1}),
    ((19, 22, 17), 2, 2, False, {"model": 2}), ((19, 22, 17), 2, 2, False, {"yz_kernel": 0}),
    ((19, 22, 17), 2, 3, False, {"yz_kernel": 0, "model": 0})])
def test_rates_scale_with_the_box(n, nf, bc, stretched, params):
    w = torch.from_numpy(_prims(n, nf, params.get("model", 0))).cuda()
    got = []
    for size in (1.0, SHRINK):
        s = _solver(n, nf, size, bc, stretched, params)
        s.set_state_prim(w)
        R = s.rhs()
        dt = s.cfl_dt(0.2)
        s.step(dt)
        got.append((R.cpu().numpy() * size, dt / size, s.get_state().cpu().numpy()))
        s.close()
    assert np.isfinite(got[0][0]).all() and np.isfinite(got[0][2]).all()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


def test_small_box_matches_the_oracle():
    import paper_2305_09163_gb300 as mfc
    n, nf = (33, 31, 29), 2
    gam, pin = workloads.fluids(nf, water_air=False)
    pb = oracle.Problem(n, (0,) * 3, (SHRINK,) * 3, (1,) * 6, gam, pin, fallback=True)
    w = _prims(n, nf, 0)
    q = oracle.cons_from_prims(pb, w)
    R_cpu, fmax, _ = oracle.rhs(pb, q, return_info=True)
    s = _solver(n, nf, SHRINK, 1, False, {})
    s.set_state_prim(torch.from_numpy(w).cuda())
    assert rhs_error(pb, q, s.rhs().cpu().numpy(), R_cpu, fmax).max() <= 1e-11
    out = torch.empty((2 * nf + 3, n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    mfc.mfc_rhs_noalloc(torch.from_numpy(q).cuda(), out, pb.n, pb.lo, pb.hi, pb.bc, gam, pin)
    assert rhs_error(pb, q, out.cpu().numpy(), R_cpu, fmax).max() <= 1e-11
