"""A solver made after one was refused on a capturing stream is the solver of a fresh start, bit for
bit up to the atomic sums' order, and the pools and operators it shares with the refused one serve it."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_common import lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)


@pytest.mark.parametrize("prec,npad", [("fp64", (0, 0)), ("fp32", (256, 512))])
def test_solve_after_a_refused_creation(prec, npad):
    gj = lib()
    g = synth.uniform_grid(9, 8, 9, 8, 3, 40.0)
    ops = [gj.bttb_setup(g, "gravity", precision=prec, npad=npad), gj.bttb_setup(g, "magnetic", MAG, precision=prec, npad=npad)]
    d = gj.g_forward_pair(ops, [to_dev(synth.uniform_model(g, 0.0, v, 3 + i), prec) for i, v in enumerate((0.5, 0.05))])
    sg = [torch.full_like(x, 0.02 * float(x.abs().max())) for x in d]
    w = [to_dev(np.ones(g.nz), prec) for _ in range(2)]
    P = gj.solver_params(kmax=3, stop_on_chi2=False, lam=(2.0, 100.0))
    out = torch.zeros(4, device="cuda")
    torch.cuda.synchronize()

    def solve():
        m = [to_dev(np.zeros(g.n), prec) for _ in range(2)]
        sv = gj.Solver(ops, P, d, sg, w, m)
        sv.iterate(3)
        rep = sv.report()
        sv.close()
        assert rep["status"] == 0 and rep["iterations"] == 3
        return [x.cpu().numpy() for x in m], rep["phi"]

    want, phi = solve()
    m = [to_dev(np.zeros(g.n), prec) for _ in range(2)]
    torch.cuda.synchronize()
    with torch.cuda.graph(torch.cuda.CUDAGraph()):
        out.add_(1.0)
        with pytest.raises(gj.GJError):
            gj.Solver(ops, P, d, sg, w, m)
    got, phi2 = solve()
    tol = 1e-12 if prec == "fp64" else 1e-5
    for i in range(2):
        assert np.linalg.norm(want[i]) > 0 and rel(got[i], want[i]) <= tol
        assert phi2[i] == pytest.approx(phi[i], rel=tol)
    for op in ops:
        op.close()
