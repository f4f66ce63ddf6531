"""Host threads that each set up operators, solve, step solvers, and take everything down again, on
streams of their own: the results are those of one thread after the other, and no thread's graph
capture is disturbed by another's clean-up.  Products and the Gramian bit for bit, solves to the
rounding of their atomic sums (as for the graph and eager forms)."""
import threading

import pytest
import torch

import synth
from tests.gpu_common import lib

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)
JOBS = [("fp32", (0, 0), (24, 20, 6)), ("fp32", (512, 512), (30, 22, 5)), ("fp32", (256, 512), (26, 18, 7)), ("fp64", (0, 0), (16, 12, 5)),
        ("fp32", (1024, 1024), (20, 14, 3))]


def job(gj, precision, npad, size, seed):
    nx, ny, nz = size
    g = synth.uniform_grid(nx, ny, nx, ny, nz, 50.0)
    ops = [gj.bttb_setup(g, "gravity", precision=precision, npad=npad), gj.bttb_setup(g, "magnetic", MAG, precision=precision, npad=npad)]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    m = [v * torch.rand(g.n, dtype=ops[0].dtype, device="cuda", generator=gen) for v in (0.5, 0.05)]
    d = gj.g_forward_pair(ops, m)
    a = gj.g_adjoint_pair(ops, d)
    S, l1, l2 = gj.gramian_value_grad(m[0], m[1])
    sg = [0.02 * torch.ones_like(x) * x.abs().max() for x in d]
    w = [torch.ones(nz, dtype=ops[0].dtype, device="cuda") for _ in range(2)]
    P = gj.solver_params(kmax=6, stop_on_chi2=False, lam=(2.0, 100.0))
    models = [torch.zeros_like(x) for x in m]
    rep = gj.rrcg_joint_solve(ops, P, d, sg, w, models)
    stepped = [torch.zeros_like(x) for x in m]
    sv = gj.Solver(ops, P, d, sg, w, stepped)
    sv.iterate(3, use_graph=False)
    sv.iterate(3, use_graph=True)
    sv.close()
    for op in ops:
        op.close()
    assert rep["iterations"] == 6
    torch.cuda.current_stream().synchronize()
    return [x.cpu() for x in (*d, *a, S, l1, l2)], [x.cpu() for x in (*models, *stepped)]


def test_threads_with_their_own_operators():
    gj = lib()
    want = [job(gj, *j, seed=i) for i, j in enumerate(JOBS)]
    got, errors = [[] for _ in JOBS], []

    def run(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(4):
                    got[i].append(job(gj, *JOBS[i], seed=i))
        except Exception as exc:
            errors.append((JOBS[i], exc))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(JOBS))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i, (exact, solves) in enumerate(want):
        tol = 1e-12 if JOBS[i][0] == "fp64" else 1e-5
        for e, s in got[i]:
            assert all(torch.equal(x, y) for x, y in zip(e, exact)), JOBS[i]
            assert all(float((x - y).norm()) <= tol * float(y.norm()) for x, y in zip(s, solves)), JOBS[i]
