"""The general kernels (any padded size) at the sizes where their plans change: every
codelet radix first, in the middle and last, pruned and unpruned ends (data longer than
half of the padded size), tiles with absent columns, layers and lines, and layer sums
kept on chip or met through memory.  Products against the FP64 dense oracle; pair calls
against single ones."""
import numpy as np
import pytest

import synth
from oracle import operator as oop
from tests.gpu_common import TOL, lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)
# (padded y, padded x): two-stage plans with every radix 2 to 17, three- and four-stage plans,
# lengths of one radix, odd lengths
SIZES = [(15, 16), (17, 18), (20, 21), (22, 24), (25, 26), (27, 28), (30, 32), (33, 34), (35, 36), (39, 40), (42, 44),
         (45, 48), (49, 50), (51, 52), (55, 56), (60, 63), (64, 65), (68, 70), (77, 78), (80, 84), (91, 96), (98, 99),
         (112, 119), (130, 144), (182, 189), (225, 255), (289, 288), (294, 300), (512, 520), (729, 833), (1001, 1024),
         (1190, 1458), (2023, 2048)]


@pytest.fixture(scope="module")
def small():
    g = synth.uniform_grid(8, 7, 8, 7, 3, 50.0)
    return g, oop.dense_matrix(g, oop.MAGNETIC, MAG)


@pytest.mark.parametrize("npad", SIZES, ids=lambda v: f"{v[0]}x{v[1]}")
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_every_radix(small, npad, prec):
    gj = lib()
    g, A = small
    op = gj.bttb_setup(g, "magnetic", MAG, precision=prec, npad=npad)
    rng = np.random.default_rng(3)
    m, r = rng.standard_normal(g.n), rng.standard_normal(g.s)
    for _ in range(2):  # the second pass finds the sums and counters as the first left them
        assert rel(op.forward(to_dev(m, prec)).cpu().numpy(), A @ m) <= TOL[prec]
        assert rel(op.adjoint(to_dev(r, prec)).cpu().numpy(), A.T @ r) <= TOL[prec]
    op.close()


@pytest.mark.parametrize("order", [0, 1, 2])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_data_longer_than_half_the_padded_size(order, prec):
    gj = lib()
    g = synth.uniform_grid(3, 2, 21, 19, 5, 40.0, off_x=9, off_y=8)
    A = oop.dense_matrix(g, oop.GRAVITY)
    rng = np.random.default_rng(4)
    m, r = rng.standard_normal(g.n), rng.standard_normal(g.s)
    for npad in [(20, 23 + 1), (21, 25), (24, 30), (26, 34)]:
        op = gj.bttb_setup(g, "gravity", precision=prec, npad=npad)
        op.tune(radix_order=order)
        assert rel(op.forward(to_dev(m, prec)).cpu().numpy(), A @ m) <= TOL[prec]
        assert rel(op.adjoint(to_dev(r, prec)).cpu().numpy(), A.T @ r) <= TOL[prec]
        op.close()


@pytest.mark.parametrize("shape", [(1, 1, 9), (2, 1, 1), (4, 3, 2), (8, 7, 4), (16, 64, 9)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_pairs_at_every_launch_shape(shape, prec):
    """(line pairs, columns, layers per CTA): ragged last tiles, one to nine layer groups a sum."""
    gj = lib()
    g = synth.uniform_grid(13, 11, 17, 12, 9, 40.0, off_x=2, off_y=1)
    A = [oop.dense_matrix(g, oop.GRAVITY), oop.dense_matrix(g, oop.MAGNETIC, MAG)]
    ops = [gj.bttb_setup(g, "gravity", precision=prec, npad=(30, 35)),
           gj.bttb_setup(g, "magnetic", MAG, precision=prec, npad=(30, 35))]
    for op in ops:
        op.tune(P_row=shape[0], C_col=shape[1], L_grp=shape[2])
    rng = np.random.default_rng(5)
    m, r = [rng.standard_normal(g.n) for _ in range(2)], [rng.standard_normal(g.s) for _ in range(2)]
    for _ in range(2):
        d = gj.g_forward_pair(ops, [to_dev(x, prec) for x in m])
        a = gj.g_adjoint_pair(ops, [to_dev(x, prec) for x in r])
        for i in range(2):
            assert rel(d[i].cpu().numpy(), A[i] @ m[i]) <= TOL[prec]
            assert rel(a[i].cpu().numpy(), A[i].T @ r[i]) <= TOL[prec]
    for op in ops:
        op.close()
