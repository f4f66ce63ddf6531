"""The largest tiles that gj_op_tune accepts launch: row tiles that fill the shared memory beside
the kernels' static part to the byte, or nearly (P line pairs take (2 P + 1) N complex values), for
products, pair products and the solver; one pair more is refused."""
import numpy as np
import pytest

import synth
from oracle import operator as oop
from tests.gpu_common import TOL, lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)
# precision, padded x, line pairs: 231424, 231424, 231400 and 230384 of 231424 bytes
TILES = [("fp32", 256, 56), ("fp64", 128, 56), ("fp32", 325, 44), ("fp64", 119, 60)]


@pytest.mark.parametrize("prec,npad_x,pairs", TILES)
def test_largest_row_tiles(prec, npad_x, pairs):
    gj = lib()
    g = synth.uniform_grid(9, 8, 9, 8, 3, 40.0)
    A = [oop.dense_matrix(g, oop.GRAVITY), oop.dense_matrix(g, oop.MAGNETIC, MAG)]
    ops = [gj.bttb_setup(g, "gravity", precision=prec, npad=(16, npad_x)),
           gj.bttb_setup(g, "magnetic", MAG, precision=prec, npad=(16, npad_x))]
    rng = np.random.default_rng(3)
    dev = lambda v: [to_dev(x, prec) for x in v]
    m, r = rng.standard_normal((2, g.n)), rng.standard_normal((2, g.s))
    P = gj.solver_params(lam=(2.0, 100.0), kmax=3, stop_on_chi2=False)

    def solve():
        models = dev([np.zeros(g.n)] * 2)
        gj.rrcg_joint_solve(ops, P, dev(r), dev([np.ones(g.s)] * 2), dev([np.ones(g.nz)] * 2), models)
        return [x.cpu().numpy() for x in models]

    want = solve()
    for op in ops:
        op.tune(P_row=pairs)
        with pytest.raises(gj.GJError):
            op.tune(P_row=pairs + 1)
        assert op.tiles()["P_row"] == pairs
    d, a = gj.g_forward_pair(ops, dev(m)), gj.g_adjoint_pair(ops, dev(r))
    for i in range(2):
        for x in (d[i], ops[i].forward(dev(m)[i])):
            assert rel(x.cpu().numpy(), A[i] @ m[i]) <= TOL[prec]
        for x in (a[i], ops[i].adjoint(dev(r)[i])):
            assert rel(x.cpu().numpy(), A[i].T @ r[i]) <= TOL[prec]
    for x, y in zip(solve(), want):
        assert rel(x, y) <= TOL[prec]  # the same transforms, whatever the tile
    for op in ops:
        op.close()


@pytest.mark.parametrize("prec,npad", [("fp64", (45, 66)), ("fp32", (45, 66)), ("fp32", (1024, 66))])
def test_shapes_given_back_to_the_library(prec, npad):
    """After GJ_TUNE_AUTO an operator is what it was before any setting, bit for bit."""
    gj = lib()
    from paper_2112_15562_gb300._lib import GJ_TUNE_AUTO

    g = synth.uniform_grid(30, 22, 30, 22, 12, 40.0)
    ops = [gj.bttb_setup(g, "gravity", precision=prec, npad=npad), gj.bttb_setup(g, "magnetic", MAG, precision=prec, npad=npad)]
    rng = np.random.default_rng(4)
    m = [to_dev(x, prec) for x in rng.standard_normal((2, g.n))]
    r = [to_dev(x, prec) for x in rng.standard_normal((2, g.s))]
    products = lambda: [*gj.g_forward_pair(ops, m), *gj.g_adjoint_pair(ops, r), ops[1].forward(m[1]), ops[0].adjoint(r[0])]
    tiles, want = ops[0].tiles(), products()
    for op in ops:
        op.tune(P_row=3, C_col=1, L_grp=2, radix_order=2)
    assert ops[0].tiles() == {"P_row": 3, "C_col": 1, "L_grp": 2, "radix_order": 2}
    products()
    for op in ops:
        op.tune(P_row=GJ_TUNE_AUTO, C_col=GJ_TUNE_AUTO, L_grp=GJ_TUNE_AUTO, radix_order=0)
    assert ops[0].tiles() == tiles
    for x, y in zip(products(), want):
        assert (x == y).all()
    for op in ops:
        op.close()
