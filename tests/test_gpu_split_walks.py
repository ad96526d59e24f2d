"""The sweeps where one CTA walks several chunks, in every form: x shares of two and
three chunks that end exactly at, one before and one after a CTA's slots, and y/z
segments of six cells and more with every remainder.  The expected split of each case is
asserted from the restated rules, so that a changed rule cannot empty a case.

x: all rows of the state are the same, so every row's right-hand side is, bit for bit,
that of a three-row grid, wherever the shares cut the rows (the y fluxes of equal rows
cancel exactly).  y/z: a cell's right-hand side does not depend on the segment length, bit
for bit.  Both are also compared with the oracle at one size."""
import numpy as np
import pytest

import oracle
import split_rules
import workloads
from paper_2305_09163_gb300 import learned
from parity_util import rhs_error

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = [("fp64", 1, {}), ("fp64", 3, {}), ("fp64", 2, {"weno_order": 3}), ("fp64", 2, {"model": 1}),
         ("fp64", 2, {"model": 2}), ("fp64", 2, {"stretched": 1}), ("fp64", 2, {"model": 2, "stretched": 1}),
         ("mixed", 2, {}), ("mixed", 2, {"weno_order": 3}), ("mixed", 2, {"model": 2}), ("mixed", 2, {"stretched": 1}),
         ("learned", 2, {})]
IDS = ["-".join([p, str(nf)] + ["%s%s" % kv for kv in o.items()]) for p, nf, o in FORMS]


def _solver(n, precision, nf, options, **more):
    import paper_2305_09163_gb300 as mfc
    gam, pin = workloads.fluids(nf)
    o = {k: v for k, v in options.items() if k != "stretched"}
    nn = tuple(n) + (1,) * (3 - len(n))
    s = mfc.Solver(nn, (0.0,) * 3, (1.0,) * 3, (1,) * 6, gam, pin, precision=precision, **o, **more)
    if options.get("stretched"):
        for d, m in enumerate(n):
            s.set_grid(d, np.concatenate([[0.0], np.cumsum(np.random.default_rng(d).uniform(0.8, 1.25, m))]) / m)
    if precision == "learned":
        s.set_mlp(learned.init_params(3))
    return s


def _prims(n, nf, options):
    w = workloads.random_prims(n, nf, seed=31)
    return workloads.six_equation_prims(w, nf, spread=0.05, seed=32) if options.get("model") == 2 else w


# (row length + 2, rows): k chunks, shares of 254 or 382 slots; last slot at a share's
# end, one after it, one before it
@pytest.mark.parametrize("p,rows,k,over", [(1016, 604, 2, 0), (1017, 763, 2, 1), (1017, 761, 2, 253),
                                           (1146, 803, 3, 0), (383, 2675, 3, 1)])
@pytest.mark.parametrize("precision,nf,options", FORMS[:2], ids=IDS[:2])
def test_x_shares_of_several_chunks(precision, nf, options, p, rows, k, over):
    _x_rows(precision, nf, options, p, rows, k, over)


@pytest.mark.parametrize("precision,nf,options", FORMS[2:], ids=IDS[2:])
def test_x_shares_in_every_form(precision, nf, options):
    _x_rows(precision, nf, options, 1017, 763, 2, 1)


def _x_rows(precision, nf, options, p, rows, k, over):
    nx = p - 2
    assert split_rules.chunks_per_block(p * rows) == k and p * rows % (128 * k - 2) == over
    assert split_rules.chunks_per_block(p * 3) == 1
    row = torch.from_numpy(np.ascontiguousarray(_prims((nx, 3), nf, options)[:, :, :1, :])).cuda()
    out = []
    for ny in (3, rows):
        # the y faces of a stretched grid are those of its own row count; equal rows cancel on any
        s = _solver((nx, ny), precision, nf, options)
        s.set_state_prim(row.expand(-1, -1, ny, -1).contiguous())
        out.append(s.rhs())
        s.close()
    small, large = out
    assert torch.equal(large, small[:, :, :1, :].expand_as(large))


@pytest.mark.parametrize("n,dirs", [((32, 103, 33), (1,)), ((100, 21, 48), (1,)), ((160, 129, 1), (1,)),
                                    ((33, 31, 108), (2,))])
@pytest.mark.parametrize("precision,nf,options", FORMS, ids=IDS)
def test_segments_agree(precision, nf, options, n, dirs):
    n = n[:2] if n[2] == 1 else n
    fp64 = precision == "fp64"
    cells = int(np.prod(n))
    if fp64:
        assert all(split_rules.segment(cells // n[d], n[d], True) >= 6 for d in dirs)
    w = torch.from_numpy(np.ascontiguousarray(_prims(n, nf, options))).cuda()
    ref = None
    lengths = [0, 8, 10, 14, 18, 34, 256] + [n[d] - r for d in dirs for r in (1, 2, 3)]
    for L in lengths:   # 0: the rule's own choice
        if L > 256:
            continue
        s = _solver(n, precision, nf, options, segment=L)
        s.set_state_prim(w)
        R = s.rhs()
        s.step(1e-9)
        q = s.get_state()
        s.close()
        assert torch.isfinite(R).all()
        ref = ref or (R, q)
        assert torch.equal(R, ref[0]) and torch.equal(q, ref[1]), L


@pytest.mark.parametrize("n,nf", [((100, 90, 77), 2), ((1015, 763), 2)])
def test_several_chunks_match_the_oracle(n, nf):
    rows = int(np.prod(n[1:]))
    assert split_rules.chunks_per_block((n[0] + 2) * rows) >= 2
    assert split_rules.segment(n[0] * (rows // n[1]), n[1], True) >= 6
    gam, pin = workloads.fluids(nf)
    pb = oracle.Problem(n, (0,) * 3, (1,) * 3, (1,) * 6, gam, pin, fallback=True)
    w = workloads.random_prims(n, nf, seed=11)
    q = oracle.cons_from_prims(pb, w)
    R_cpu, fmax, _ = oracle.rhs(pb, q, return_info=True)
    s = _solver(n, "fp64", nf, {})
    s.set_state_prim(torch.from_numpy(w).cuda())
    assert rhs_error(pb, q, s.rhs().cpu().numpy(), R_cpu, fmax).max() <= 1e-11
    s.close()
