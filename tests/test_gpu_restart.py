"""A run continued from a saved state is the uninterrupted run, bit for bit: the time
step of the saved state, its right-hand side and the states that follow (the last stage
of a step leaves primitives and the CFL rate behind, a restart recovers them from the
state)."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,nf,model,rk,stretched", [
    ((90,), 2, 2, 3, False), ((31, 26), 2, 2, 3, False), ((19, 17, 18), 2, 2, 3, False), ((19, 17, 18), 3, 2, 3, False),
    ((19, 17, 18), 2, 2, 1, False), ((40,), 3, 2, 1, False), ((19, 17, 18), 2, 2, 2, True),
    ((19, 17, 18), 2, 0, 3, False), ((19, 17, 18), 3, 0, 1, True), ((60,), 1, 0, 1, False), ((31, 26), 2, 1, 2, False)])
def test_restart_is_bitwise(precision, n, nf, model, rk, stretched):
    import paper_2305_09163_gb300 as mfc
    gam, pin = workloads.fluids(nf)
    nn = n + (1,) * (3 - len(n))
    w = workloads.random_prims(n, nf, seed=21, noise=0.01)
    if model == 2:
        w = workloads.six_equation_prims(w, nf, spread=0.1, seed=22)

    def solver():
        s = mfc.Solver(nn, (0.0,) * 3, (1.0,) * 3, (1,) * 6, gam, pin, precision=precision, model=model, rk_order=rk)
        if stretched:
            for d, m in enumerate(n):
                s.set_grid(d, np.concatenate([[0.0], np.cumsum(np.random.default_rng(d).uniform(0.8, 1.2, m))]) / m)
        return s

    a = solver()
    a.set_state_prim(torch.from_numpy(np.ascontiguousarray(w)).cuda())
    for _ in range(3):
        a.step(a.cfl_dt(0.2))
        b = solver()
        b.set_state(a.get_state())
        dt = a.cfl_dt(0.2)
        assert b.cfl_dt(0.2) == dt
        assert torch.equal(b.rhs(), a.rhs())
        b.step(dt)
        want = b.get_state()
        b.close()
        c = solver()
        c.set_state(a.get_state())
        a.step(dt)
        assert torch.equal(a.get_state(), want)
        c.step(dt)
        assert torch.equal(c.get_state(), want)
        c.close()
    a.close()
