"""Products in any unit of length: with every length scaled by 2^k the total-field anomaly stays the
same and the vertical gravity scales by 2^k (w / R^3 over a volume), also where a distance's fifth
power is outside FP32.  Both precisions against the unscaled operator, which other tests compare
with the oracle; powers of two change nothing but the corner sums' logarithms near the stations."""
import numpy as np
import pytest

import synth
from tests.gpu_common import TOL, lib, rel, to_dev

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("recompute", [False, True])
def test_scaled_lengths(prec, recompute):
    gj = lib()
    rng = np.random.default_rng(31)
    sizes = (40, 37, 40, 37, 5)
    m, r = rng.uniform(0, 1, 40 * 37 * 5), rng.uniform(0, 1, 40 * 37)
    for field, mag in (("gravity", None), ("magnetic", MAG)):
        want = None
        for k in (0, 24, -40):
            g = synth.uniform_grid(*sizes, 100.0 * 2.0 ** k, dz=60.0 * 2.0 ** k)
            op = gj.bttb_setup(g, field, mag, precision=prec, recompute=recompute)
            f = 2.0 ** -k if field == "gravity" else 1.0
            got = [f * x.double().cpu().numpy() for x in (op.forward(to_dev(m, prec)), op.adjoint(to_dev(r, prec)))]
            op.close()
            want = want or got
            for a, b in zip(got, want):
                assert rel(a, b) <= TOL[prec], (field, k)
