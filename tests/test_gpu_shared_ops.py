"""Calls on one pair of operators, one after the other in one stream, between the iterations of a
solve: a solver keeps everything that one iteration leaves for the next, so products of its
operators and a second solver on them change nothing.  FP64 agrees to rounding (the sums are
atomic), FP32 to 1e-5, as for the graph and eager forms of a solve."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_common import lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)
PATHS = [("fp64", (0, 0)), ("fp32", (0, 0)), ("fp32", (512, 512)), ("fp32", (256, 512)), ("fp32", (1024, 32)), ("fp32", (1024, 1024))]


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("prec,npad", PATHS, ids=lambda v: v if isinstance(v, str) else f"{v[0]}x{v[1]}")
def test_calls_between_iterations(prec, npad, graph):
    gj = lib()
    g = synth.uniform_grid(16, 13, 16, 13, 6, 50.0)
    ops = [gj.bttb_setup(g, "gravity", precision=prec, npad=npad), gj.bttb_setup(g, "magnetic", MAG, precision=prec, npad=npad)]
    dev = lambda v: [to_dev(x, prec) for x in v]
    P = gj.solver_params(lam=(50.0, 1500.0), kmax=8, stop_on_chi2=False)

    def solver(seed):
        m = [synth.smooth_blocky(g, v, seed + i, n_boxes=2, sigma=2.0) for i, v in enumerate((0.5, 0.05))]
        d = gj.g_forward_pair(ops, dev(m))
        s = [torch.full_like(x, 0.02 * float(x.abs().max())) for x in d]
        models = dev([np.zeros(g.n)] * 2)
        return gj.Solver(ops, P, d, s, dev([np.ones(g.nz)] * 2), models), models

    alone = []
    for seed in (1, 2):
        sv, models = solver(seed)
        sv.iterate(8, use_graph=graph)
        alone.append([x.cpu().numpy() for x in models] + [sv.report()["phi"]])
        sv.close()
    (a, ma), (b, mb) = solver(1), solver(2)
    rng = np.random.default_rng(3)
    x, r = dev(rng.standard_normal((2, g.n))), dev(rng.standard_normal((2, g.s)))
    for k in range(8):
        a.iterate(1, use_graph=graph)
        b.iterate(1, use_graph=graph)
        if k % 2:
            gj.g_adjoint_pair(ops, r)
        else:
            ops[0].forward(x[0])
            ops[1].adjoint(r[1])
            ops[1].forward(x[1])
    tol = 1e-12 if prec == "fp64" else 1e-5
    for sv, models, want in ((a, ma, alone[0]), (b, mb, alone[1])):
        assert sv.report()["iterations"] == 8
        for i in range(2):
            assert rel(models[i].cpu().numpy(), want[i]) <= tol
            assert sv.report()["phi"][i] == pytest.approx(want[2][i], rel=tol)
        sv.close()
    for op in ops:
        op.close()
