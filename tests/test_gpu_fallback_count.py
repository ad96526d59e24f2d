"""The counter of first-order faces counts each face once, however the sweeps are split:
equal to the oracle's count, in the forms whose states it shares (a block of cells with a
volume fraction of -0.01, which no rounding decides)."""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _count(n, nf, bc, precision, segment, params):
    import paper_2305_09163_gb300 as mfc
    six = params.get("model") == 2
    gam, pin = workloads.fluids(nf)
    pb = oracle.Problem(n, (0,) * 3, (1,) * 3, (bc,) * (2 * len(n)) + (1,) * (6 - 2 * len(n)), gam, pin, fallback=True,
                        model={0: "allaire", 1: "kapila", 2: "six"}[params.get("model", 0)],
                        weno_order=params.get("weno_order", 5))
    w = workloads.random_prims(n, nf, seed=8, jumps=False, noise=0.0)
    block = tuple(slice(m // 4, m // 4 + (m + 1) // 2) for m in w.shape[1:])
    ia = nf + len(n) + 1
    w[(ia,) + block] = -0.01
    if nf == 3:
        w[(ia + 1,) + block] = 0.5
    if six:
        w = workloads.six_equation_prims(w, nf, spread=0.0, seed=9)
    q = np.ascontiguousarray(oracle.cons_from_prims(pb, np.ascontiguousarray(w)))
    _, _, want = oracle.rhs(pb, q, return_info=True)
    s = mfc.Solver(pb.n, pb.lo, pb.hi, pb.bc, gam, pin, precision=precision, segment=segment, **params)
    s.set_state(torch.from_numpy(q).cuda())
    s.rhs()
    got = s.fallback_count()
    s.close()
    assert want > 0
    return got, want


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("segment", [0, 8, 14, 256])
@pytest.mark.parametrize("n,nf,bc,params", [
    ((300,), 2, 1, {}), ((61, 37), 2, 0, {}), ((33, 21, 19), 2, 1, {}), ((33, 21, 19), 3, 2, {}),
    ((33, 21, 19), 2, 1, {"yz_kernel": 0}), ((33, 21, 19), 2, 0, {"weno_order": 3}), ((33, 21, 19), 2, 1, {"model": 1}),
    ((33, 21, 19), 2, 1, {"model": 2})])
def test_every_face_is_counted_once(n, nf, bc, params, segment, precision):
    got, want = _count(n, nf, bc, precision, segment, params)
    assert got == want


def test_several_chunks_per_share():
    got, want = _count((1015, 763), 2, 1, "fp64", 0, {})
    assert got == want
