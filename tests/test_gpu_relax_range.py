"""A phase energy far above the cell's total energy (1e30 in one cell, out of any range
but not out of the state's) ends relaxed like any other: the step leaves a finite state
whose time step is that of the state without it, to the cell's own change, since the
relaxation sets every phase energy from the total one."""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,nf,params", [
    ("fp64", (17, 14, 13), 2, {}), ("fp64", (23, 19), 3, {}), ("fp64", (17, 14, 13), 2, {"fallback": 0}),
    ("fp64", (17, 14, 13), 2, {"weno_order": 3}), ("fp64", (70,), 2, {}), ("mixed", (17, 14, 13), 2, {}),
    ("mixed", (70,), 2, {})])
def test_oversized_phase_energy_is_reset(precision, n, nf, params):
    import paper_2305_09163_gb300 as mfc
    gam, pin = workloads.fluids(nf)
    pb = oracle.Problem(n, (0,) * 3, (1,) * 3, (1,) * 6, gam, pin, fallback=True, model="six")
    w = workloads.six_equation_prims(workloads.random_prims(n, nf, seed=8), nf, spread=0.0, seed=1)
    q0 = np.ascontiguousarray(oracle.cons_from_prims(pb, w))
    cell = tuple(m // 2 for m in reversed(pb.n))
    rows = q0.shape[0]
    # first and last phase (of three, the middle one's 1e30 leaves the cell a sound speed that
    # takes the time step down, as it always did)
    for v in (rows - nf, rows - 1):
        q = q0.copy()
        q[(v,) + cell] = 1e30
        s = mfc.Solver(pb.n, pb.lo, pb.hi, pb.bc, gam, pin, precision=precision, model=2, **params)
        s.set_state(torch.from_numpy(q).cuda())
        dt = s.cfl_dt(0.3)   # takes no phase energy
        s.step(1e-9)
        assert s.cfl_dt(0.3) > 0.5 * dt
        assert torch.isfinite(s.get_state()).all()
        s.close()
