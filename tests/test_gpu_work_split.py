"""FP64 right-hand side against the oracle at the sizes where the sweeps' split
into CTAs can go wrong: rows and grids that end exactly at, one before and one
after a CTA's share."""
import pytest

import oracle
import workloads
from parity_util import rhs_error

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_FP64 = 1e-11   # the FP64 path's parity gate (flux scale of each component)


def _check(n, bc=1, nf=2, **params):
    import paper_2305_09163_gb300 as mfc
    gam, pin = workloads.fluids(nf)
    pb = oracle.Problem(n, (0, 0, 0), (1, 1, 1), (bc,) * 6, gam, pin, fallback=True)
    w = workloads.random_prims(n, nf, seed=11)
    q = oracle.cons_from_prims(pb, w)
    R_cpu, fmax, _ = oracle.rhs(pb, q, return_info=True)
    s = mfc.Solver(pb.n, pb.lo, pb.hi, pb.bc, pb.gamma, pb.pi_inf, **params)
    s.set_state_prim(torch.from_numpy(w).cuda())
    R = s.rhs().cpu().numpy()
    s.close()
    assert rhs_error(pb, q, R, R_cpu, fmax).max() <= TOL_FP64


# an x CTA owns 128 k - 2 slots (n + 2 per row): one share exactly, one slot
# over it, shares that cut rows at every column, and (last) k above 1
@pytest.mark.parametrize("n", [(124,), (125,), (250,), (1000,), (40, 3), (61, 7), (5, 200), (1021, 400)])
def test_x_share_edges(n):
    _check(n)


# y/z CTAs take 32 cells of the flat transverse plane and segments of 4 m - 2
# cells: planes of 15, 32, 33 and 31 cells, directions that leave 1, 2 or 3 cells
# to the last segment, 2D rows below, at and above a warp
@pytest.mark.parametrize("n", [(5, 3, 3), (8, 4, 8), (11, 7, 3), (31, 131, 3), (3, 3, 77), (31, 9), (32, 127), (33, 130)])
@pytest.mark.parametrize("bc", [0, 2, 3])
def test_yz_plane_and_segment_edges(n, bc):
    _check(n, bc)
