"""1024 x 1024 embeddings of lines longer than the 512 values that the warp-FFT row kernels hold:
more prisms than that along x, more stations, and one value more or less, for single and pair
products and for the solver.  Against the FP64 dense oracle, with the tolerances of the other parity
tests (products 1e-5; Phi of every iteration 1e-4, models 1e-3)."""
import numpy as np
import pytest

import synth
from oracle import operator as oop
from oracle import weights as owt
from oracle.rrcg import RRCGParams, rrcg_joint
from tests.gpu_common import TOL, lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)
# (stations x, y, prisms x, y, layers), offset x
SIZES = [((400, 3, 600, 3, 2), 100), ((600, 2, 400, 3, 2), -100), ((513, 3, 512, 3, 1), 0), ((512, 3, 513, 2, 1), 1),
         ((512, 3, 512, 4, 1), 0)]


@pytest.mark.parametrize("sizes,off", SIZES)
def test_lines_beyond_512_values(sizes, off):
    gj = lib()
    g = synth.uniform_grid(*sizes, 40.0, off_x=off)
    A = [oop.dense_from_table(oop.kernel_table(g, oop.GRAVITY), g), oop.dense_from_table(oop.kernel_table(g, oop.MAGNETIC, MAG), g)]
    ops = [gj.bttb_setup(g, "gravity", precision="fp32", npad=(1024, 1024)),
           gj.bttb_setup(g, "magnetic", MAG, precision="fp32", npad=(1024, 1024))]
    assert all(op.info.fast_path == 2 for op in ops)
    rng = np.random.default_rng(12)
    m = [to_dev(rng.standard_normal(g.n), "fp32") for _ in range(2)]
    r = [to_dev(rng.standard_normal(g.s), "fp32") for _ in range(2)]
    d, a = gj.g_forward_pair(ops, m), gj.g_adjoint_pair(ops, r)
    for i in range(2):
        md, rd = m[i].double().cpu().numpy(), r[i].double().cpu().numpy()
        for x in (d[i], ops[i].forward(m[i])):
            assert rel(x.cpu().numpy(), A[i] @ md) <= TOL["fp32"]
        for x in (a[i], ops[i].adjoint(r[i])):
            assert rel(x.cpu().numpy(), A[i].T @ rd) <= TOL["fp32"]

    noise = synth.standard_normal((2, g.s), 13)
    obs = [owt.noisy_data(A[i] @ synth.uniform_model(g, 0.0, v, 14 + i), 0.01, 0.01, noise[i]) for i, v in enumerate((1.0, 0.1))]
    dob, sig = [o[0] for o in obs], [o[1] for o in obs]
    wdep = [owt.depth_weights(g.z_edges, 2.0), owt.depth_weights(g.z_edges, 3.0)]
    kw = dict(lam=(2.0, 100.0), kmax=4, stop_on_chi2=False)
    ref = rrcg_joint([lambda x, i=i: A[i] @ x for i in range(2)], [lambda y, i=i: A[i].T @ y for i in range(2)], dob, sig,
                     [np.zeros(g.n)] * 2, [np.repeat(w, g.nx * g.ny) for w in wdep], RRCGParams(**kw))
    dev = lambda v: [to_dev(x, "fp32") for x in v]
    model = dev([np.zeros(g.n)] * 2)
    rep = gj.rrcg_joint_solve(ops, gj.solver_params(**kw), dev(dob), dev(sig), dev(wdep), model, history=True)
    for k in range(5):
        for i in range(2):
            assert rep["history"][k]["phi"][i] == pytest.approx(ref.history[k]["phi"][i], rel=1e-4), (k, i)
    for i in range(2):
        assert rel(model[i].cpu().numpy(), ref.m[i]) <= 1e-3
        ops[i].close()
