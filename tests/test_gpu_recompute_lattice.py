"""Recomputed spectra where layers much thicker than the cells are wide take the near field over the
whole grid, so that each layer's lattice is built with the layer: products against the dense oracle
and against stored spectra, repeated, with the tolerances of the parity tests."""
import numpy as np
import pytest

import synth
from oracle import operator as oop
from tests.gpu_common import TOL, lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("sizes,off", [((12, 9, 70, 70, 24), (30, 29)), ((70, 61, 70, 61, 20), (0, 0))])
def test_lattice_of_one_layer_at_a_time(prec, sizes, off):
    gj = lib()
    g = synth.uniform_grid(*sizes, 40.0, dz=400.0, off_x=off[0], off_y=off[1])
    rng = np.random.default_rng(21)
    m, r = rng.standard_normal(g.n), rng.standard_normal(g.s)
    for field, f in (("gravity", oop.GRAVITY), ("magnetic", oop.MAGNETIC)):
        mag = MAG if field == "magnetic" else None
        K = oop.kernel_table(g, f, MAG)
        jy, jx = rng.permutation(g.s)[:20], rng.permutation(g.n)[:40]
        d, a = oop.forward_rows(K, g, m, jy), oop.adjoint_cols(K, g, r, jx)
        ops = [gj.bttb_setup(g, field, mag, precision=prec, recompute=rc) for rc in (True, False)]
        for op in (ops[0], ops[0], ops[1]):
            y, x = op.forward(to_dev(m, prec)).cpu().numpy(), op.adjoint(to_dev(r, prec)).cpu().numpy()
            assert rel(y[jy], d) <= TOL[prec] and rel(x[jx], a) <= TOL[prec]
        for op in ops:
            op.close()
