"""A cell value that is not a number shows in the right-hand side: a NaN or infinite
volume fraction in that cell's volume-fraction row, in the six-equation model also in its
phase-energy rows, where a NaN pressure (total energy) shows too."""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("n,nf,params", [
    ((40,), 2, {}), ((21, 18), 3, {}), ((17, 16, 15), 2, {}), ((17, 16, 15), 3, {}), ((17, 16, 15), 2, {"yz_kernel": 0}),
    ((17, 16, 15), 2, {"weno_order": 3}), ((17, 16, 15), 2, {"model": 1}), ((17, 16, 15), 3, {"model": 2}),
    ((21, 18), 2, {"model": 2}), ((17, 16, 15), 2, {"grid": 1})])
def test_bad_cell_reaches_the_rates(n, nf, params, bad):
    import paper_2305_09163_gb300 as mfc
    params = dict(params)
    stretched = params.pop("grid", 0)
    six = params.get("model") == 2
    nd = len(n)
    gam, pin = workloads.fluids(nf)
    pb = oracle.Problem(n, (0,) * 3, (1,) * 3, (1,) * 6, gam, pin, fallback=True, model="six" if six else "allaire")
    w = workloads.random_prims(n, nf, seed=3)
    if six:
        w = workloads.six_equation_prims(w, nf, spread=0.0, seed=4)
    q = np.ascontiguousarray(oracle.cons_from_prims(pb, w))
    cell = tuple(m // 2 for m in reversed(pb.n))
    ia, ie = nf + nd + 1, nf + nd
    s = mfc.Solver(pb.n, pb.lo, pb.hi, pb.bc, gam, pin, **params)
    if stretched:
        for d, m in enumerate(n):
            s.set_grid(d, np.concatenate([[0.0], np.cumsum(np.random.default_rng(d).uniform(0.5, 2.0, m))]))

    def rates(row):
        qb = q.copy()
        qb[(row,) + cell] = bad
        s.set_state(torch.from_numpy(qb).cuda())
        out = [s.rhs().cpu().numpy()]
        if not params and not stretched:
            r = torch.empty_like(torch.from_numpy(q)).cuda()
            mfc.mfc_rhs_noalloc(torch.from_numpy(qb).cuda(), r, pb.n, pb.lo, pb.hi, pb.bc, gam, pin)
            out.append(r.cpu().numpy())
        return [R[(slice(None),) + cell] for R in out]

    for R in rates(ia):
        assert not np.isfinite(R[ia])
        if six:
            assert not np.isfinite(R[ia + nf - 1:]).any()
    if six:
        for R in rates(ie):
            assert not np.isfinite(R[ia + nf - 1:]).any()
    s.close()
