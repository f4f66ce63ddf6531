"""FP32 joint solves on every kernel family against the FP64 oracle on the same (FP32) inputs, at
the accuracy that single-precision products allow.

The magnetic data are some 200 times the gravity data and the weighted residuals the other way
round, so a complex transform that carries a line of each field rounds the smaller one by the
larger: Phi and the models were then off by up to 8e-6, by a
different amount after any change of rounding.  Tolerances: with eps = 2e-7 for a product of one
field and data of at most 100 standard deviations, the residuals are off by at most
100 eps = 2e-5 of a standard deviation each, at random, which is 2 * 2e-5 / sqrt(s) = 1e-6 of
Phi at s = 1500 data that fit to one standard deviation, and the misfits here are well above that:
5e-7.  The models add the rounding of some ten vector operations an iteration: 1e-6."""
import numpy as np
import pytest

import synth
from oracle import operator as oop
from oracle import weights as owt
from oracle.rrcg import RRCGParams, rrcg_joint
from tests.gpu_common import lib, rel, to_dev

pytestmark = pytest.mark.gpu

KW = dict(p=(1, 1), alpha1=(2e4, 2e4), q=(0.95, 0.95), alpha_min=(5.0, 20.0), lam=(2.0, 100.0), lo=(0.0, 0.0),
          hi=(1.0, 0.1), kmax=20, stop_on_chi2=False)
MAG = synth.Mag(50000.0, 60.0, 10.0)


def single(x):
    return np.asarray(x, dtype=np.float32).astype(np.float64)


@pytest.fixture(scope="module")
def surveys():
    g = synth.uniform_grid(50, 30, 50, 30, 10, 100.0)
    B = [oop.BCCB(oop.kernel_table(g, oop.GRAVITY), g, 60, 100), oop.BCCB(oop.kernel_table(g, oop.MAGNETIC, MAG), g, 60, 100)]
    wdep = [single(owt.depth_weights(g.z_edges, beta)) for beta in (2.0, 3.0)]
    out = []
    for seed in range(10):
        noise = synth.standard_normal((2, g.s), 1000 + seed)
        obs = [owt.noisy_data(B[i].forward(synth.dipping_blocks(g, v, seed)), 0.01, 0.01, noise[i])
               for i, v in enumerate((1.0, 0.1))]
        dob, sig = [single(o[0]) for o in obs], [single(o[1]) for o in obs]
        ref = rrcg_joint([b.forward for b in B], [b.adjoint for b in B], dob, sig, [np.zeros(g.n)] * 2,
                         [np.repeat(w, g.nx * g.ny) for w in wdep], RRCGParams(**KW))
        out.append((dob, sig, ref))
    return g, wdep, out


@pytest.mark.parametrize("npad", [(0, 0), (63, 105), (256, 512), (512, 512), (1024, 108), (1024, 1024)],
                         ids=lambda v: f"{v[0]}x{v[1]}")
def test_fp32_solves_keep_single_precision(surveys, npad):
    gj = lib()
    g, wdep, cases = surveys
    ops = [gj.bttb_setup(g, "gravity", precision="fp32", npad=npad), gj.bttb_setup(g, "magnetic", MAG, precision="fp32", npad=npad)]
    worst = [0.0, 0.0]
    for dob, sig, ref in cases:
        m = [to_dev(np.zeros(g.n), "fp32") for _ in range(2)]
        rep = gj.rrcg_joint_solve(ops, gj.solver_params(**KW), [to_dev(x, "fp32") for x in dob],
                                  [to_dev(x, "fp32") for x in sig], [to_dev(x, "fp32") for x in wdep], m)
        assert rep["iterations"] == 20
        for i in range(2):
            want = ref.history[-1]["phi"][i]
            worst[0] = max(worst[0], abs(rep["phi"][i] - want) / want)
            worst[1] = max(worst[1], rel(m[i].cpu().numpy(), ref.m[i]))
    print(f"\npadded {npad[0]}x{npad[1]}: worst of {len(cases)} solves: Phi {worst[0]:.1e}, models {worst[1]:.1e}")
    assert worst[0] <= 5e-7 and worst[1] <= 1e-6, worst
    for op in ops:
        op.close()


@pytest.mark.parametrize("npad", [(0, 0), (512, 512), (256, 512), (1024, 27), (1024, 1024)],
                         ids=lambda v: f"{v[0]}x{v[1]}")
def test_data_lines_without_a_second_line(npad):
    """An odd number of station rows: the last transform of each field holds one line.  One row
    alone, and more rows than a block takes."""
    gj = lib()
    for sx, sy in ((7, 1), (13, 9), (14, 27)):
        if npad[1] and sx + 12 > npad[1]:
            continue
        g = synth.uniform_grid(sx, sy, 13, sy, 4, 50.0)
        A = [oop.dense_matrix(g, oop.GRAVITY), oop.dense_matrix(g, oop.MAGNETIC, MAG)]
        noise = synth.standard_normal((2, g.s), 5)
        obs = [owt.noisy_data(A[i] @ synth.uniform_model(g, 0.0, v, 6 + i), 0.01, 0.01, noise[i]) for i, v in enumerate((1.0, 0.1))]
        wdep = [owt.depth_weights(g.z_edges, beta) for beta in (2.0, 3.0)]
        kw = dict(KW, kmax=3)
        ref = rrcg_joint([lambda x, i=i: A[i] @ x for i in range(2)], [lambda y, i=i: A[i].T @ y for i in range(2)],
                         [o[0] for o in obs], [o[1] for o in obs], [np.zeros(g.n)] * 2,
                         [np.repeat(w, g.nx * g.ny) for w in wdep], RRCGParams(**kw))
        for prec in ("fp32", "fp64") if npad == (0, 0) else ("fp32",):
            ops = [gj.bttb_setup(g, "gravity", precision=prec, npad=npad), gj.bttb_setup(g, "magnetic", MAG, precision=prec, npad=npad)]
            m = [to_dev(np.zeros(g.n), prec) for _ in range(2)]
            rep = gj.rrcg_joint_solve(ops, gj.solver_params(**kw), *[[to_dev(x, prec) for x in v] for v in
                                                                    ([o[0] for o in obs], [o[1] for o in obs], wdep)], m, history=True)
            tol = 1e-9 if prec == "fp64" else 1e-4  # as in the other parity tests of a solve's history
            for k in range(4):
                for i in range(2):
                    assert rep["history"][k]["phi"][i] == pytest.approx(ref.history[k]["phi"][i], rel=tol), (sx, sy, k, i)
            for i in range(2):
                assert rel(m[i].cpu().numpy(), ref.m[i]) <= (1e-9 if prec == "fp64" else 1e-3)
            for op in ops:
                op.close()
