"""The kernels at the edges of their launch rules: Gramian vectors off 16-byte boundaries and at
the ends of blocks and grids, recomputed spectra at even and odd plans and offset windows,
spectra built in several chunks, and the row tiles of the N = 1024 kernels with line pairs that
do and do not straddle layers.  Against the FP64 oracle, with the tolerances of the parity tests."""
import numpy as np
import pytest
import torch

import synth
from oracle import gramian as ogm
from oracle import operator as oop
from tests.gpu_common import TOL, lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [1, 3, 4, 1023, 1029, 304 * 4096 + 5])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_gramian_alignments(prec, n, shift):
    """shift: elements the second vector starts past a 16-byte boundary."""
    gj = lib()
    rng = np.random.default_rng(n)
    m1 = rng.uniform(0, 1, n)
    m2 = 0.1 * m1 + 0.01 * rng.standard_normal(n)
    x1 = to_dev(m1, prec)
    x2 = to_dev(np.concatenate([np.zeros(shift), m2]), prec)[shift:]
    S, l1, l2 = gj.gramian_value_grad(x1, x2)
    only, none1, none2 = gj.gramian_value_grad(x1, x2, want_dirs=False)
    assert none1 is None and none2 is None and only.item() == S.item()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        again, _, _ = gj.gramian_value_grad(x1, x2)
    side.synchronize()
    assert again.item() == S.item()  # the sums' order is fixed
    m1, m2 = x1.double().cpu().numpy(), x2.double().cpu().numpy()
    scale = (m1 @ m1) * (m2 @ m2)
    assert abs(S.item() - ogm.gramian(m1, m2)) <= (1e-12 if prec == "fp64" else 2e-6) * scale
    if n > 1:
        r1, r2 = ogm.ascent_directions(m1, m2)
        vtol = 1e-10 if prec == "fp64" else 1e-4
        assert rel(l1.cpu().numpy(), r1) <= vtol and rel(l2.cpu().numpy(), r2) <= vtol


# (stations x, y, prisms x, y, layers, offsets), padded (y, x): tables even in both offsets
# (equal grids) and not; windows that leave offset 0 out on one side or the other; odd plans;
# one layer; plans whose columns go one line a block
RECOMPUTE = [((6, 5, 6, 5, 4), {}, (11, 13)), ((6, 5, 6, 5, 1), {}, (12, 16)), ((6, 4, 6, 4, 3), {}, (2023, 16)),
             ((7, 6, 4, 3, 3), dict(off_x=9, off_y=8), (0, 0)), ((4, 3, 7, 6, 2), dict(off_x=-5, off_y=-4), (15, 17)),
             ((5, 5, 5, 5, 3), dict(off_x=1), (1190, 18)), ((9, 2, 3, 8, 2), {}, (1024, 21))]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("sizes,offs,npad", RECOMPUTE)
def test_recomputed_spectra(prec, sizes, offs, npad):
    gj = lib()
    g = synth.uniform_grid(*sizes, 40.0, **offs)
    rng = np.random.default_rng(7)
    m, r = rng.standard_normal(g.n), rng.standard_normal(g.s)
    for field, f in (("gravity", oop.GRAVITY), ("magnetic", oop.MAGNETIC)):
        A = oop.dense_matrix(g, f, MAG)
        op = gj.bttb_setup(g, field, MAG if field == "magnetic" else None, precision=prec, npad=npad, recompute=True)
        for _ in range(2):
            assert rel(op.forward(to_dev(m, prec)).cpu().numpy(), A @ m) <= TOL[prec]
            assert rel(op.adjoint(to_dev(r, prec)).cpu().numpy(), A.T @ r) <= TOL[prec]
        op.close()


def test_spectra_built_in_chunks():
    """65 layers at 1024 x 1024 take three chunks of the build (256 MB of row transforms)."""
    gj = lib()
    g = synth.uniform_grid(4, 3, 3, 4, 65, 40.0, dz=15.0)
    rng = np.random.default_rng(8)
    m = rng.standard_normal(g.n)
    for field, f in (("gravity", oop.GRAVITY), ("magnetic", oop.MAGNETIC)):
        op = gj.bttb_setup(g, field, MAG if field == "magnetic" else None, precision="fp32", npad=(1024, 1024))
        assert rel(op.forward(to_dev(m, "fp32")).cpu().numpy(), oop.dense_matrix(g, f, MAG) @ m) <= TOL["fp32"]
        op.close()


@pytest.mark.parametrize("sizes", [(4, 6, 5, 6, 3), (4, 5, 6, 5, 4), (3, 9, 3, 16, 2), (40, 8, 33, 2, 1)])
@pytest.mark.parametrize("npad", [(1024, 1024), (512, 512)])
def test_row_tiles_of_the_warp_kernels(sizes, npad):
    """Lines per layer even (pairs of one 16-byte word) and odd (pairs across layers), full and
    ragged tiles, one line past the last pair; both fields in one launch and one at a time."""
    gj = lib()
    g = synth.uniform_grid(*sizes, 40.0)
    A = [oop.dense_matrix(g, oop.GRAVITY), oop.dense_matrix(g, oop.MAGNETIC, MAG)]
    ops = [gj.bttb_setup(g, "gravity", precision="fp32", npad=npad),
           gj.bttb_setup(g, "magnetic", MAG, precision="fp32", npad=npad)]
    assert all(op.info.fast_path == (2 if npad[0] == 1024 else 1) for op in ops)
    rng = np.random.default_rng(9)
    m = [to_dev(rng.standard_normal(g.n), "fp32") for _ in range(2)]
    r = [to_dev(rng.standard_normal(g.s), "fp32") for _ in range(2)]
    d, a = gj.g_forward_pair(ops, m), gj.g_adjoint_pair(ops, r)
    for i in range(2):
        md, rd = m[i].double().cpu().numpy(), r[i].double().cpu().numpy()
        for x in (d[i], ops[i].forward(m[i])):
            assert rel(x.cpu().numpy(), A[i] @ md) <= TOL["fp32"]
        for x in (a[i], ops[i].adjoint(r[i])):
            assert rel(x.cpu().numpy(), A[i].T @ rd) <= TOL["fp32"]
        ops[i].close()


def test_solver_creation_refuses_a_capturing_stream():
    gj = lib()
    g = synth.uniform_grid(8, 8, 8, 8, 3, 40.0)
    ops = [gj.bttb_setup(g, "gravity", precision="fp64"), gj.bttb_setup(g, "magnetic", MAG, precision="fp64")]
    vec = lambda n: [torch.ones(n, dtype=torch.float64, device="cuda") for _ in range(2)]
    d, sg, w, m = vec(g.s), vec(g.s), vec(g.nz), vec(g.n)
    out = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out.add_(1.0)
        with pytest.raises(gj.GJError):
            gj.Solver(ops, gj.solver_params(kmax=2), d, sg, w, m)
    graph.replay()
    torch.cuda.synchronize()
    assert out.tolist() == [1.0] * 4  # the capture went on
    sv = gj.Solver(ops, gj.solver_params(kmax=2), d, sg, w, m)
    sv.iterate(2)
    assert sv.report()["iterations"] >= 0
    sv.close()
    for op in ops:
        op.close()


def test_refused_host_solve_leaves_nothing_behind():
    """A parameter refused after the inputs were copied in; the next solve is that of a fresh start."""
    gj = lib()
    g = synth.uniform_grid(8, 8, 8, 8, 3, 40.0)
    ops = [gj.bttb_setup(g, "gravity", precision="fp64"), gj.bttb_setup(g, "magnetic", MAG, precision="fp64")]
    rng = np.random.default_rng(11)
    data = [rng.standard_normal(g.s) for _ in range(2)]
    ones = lambda n: [np.ones(n) for _ in range(2)]
    models = []
    for refuse in (False, True):
        if refuse:
            with pytest.raises(gj.GJError):
                gj.rrcg_joint_solve_host(ops, gj.solver_params(kmax=3, lo=(2.0, 0.0), hi=(1.0, 0.1)), data, ones(g.s),
                                         ones(g.nz), [np.zeros(g.n) for _ in range(2)])
        m = [np.zeros(g.n) for _ in range(2)]
        gj.rrcg_joint_solve_host(ops, gj.solver_params(kmax=3), data, ones(g.s), ones(g.nz), m)
        models.append(m)
    for i in range(2):
        assert np.array_equal(models[0][i], models[1][i])
    for op in ops:
        op.close()
