"""FP32 products against FP64 ones on the same inputs: they are not scaled.  Constants that all
round the same way shrink every transform a little, and that gain adds up where other rounding
averages out (-1.1e-7 at N = 256, -1.3e-7 at 512, -1.7e-7 at 1024 with cos(pi/8) and sqrt(1/2) both
rounded down).  Tolerance: the constants as chosen leave 5e-9 a product at these sizes, rounding of
10^4 independent values 2e-9, and the spectra's own rounding (3e-8 each, some ten of them dominant)
1e-8; twice their sum, rounded up: 4e-8.  The error that is left has no such sum: 3e-7."""
import pytest
import torch

import synth
from tests.gpu_common import lib

pytestmark = pytest.mark.gpu

MAG = synth.Mag(50000.0, 60.0, 10.0)


@pytest.mark.parametrize("npad,size", [((256, 256), 128), ((512, 512), 250), ((256, 512), 120), ((1024, 1024), 400),
                                       ((1024, 256), 120)], ids=lambda v: str(v))
def test_products_are_not_scaled(npad, size):
    gj = lib()
    g = synth.uniform_grid(size, size, size, size, 6, 50.0)
    gen = torch.Generator(device="cuda").manual_seed(5)
    for field, mag in (("gravity", None), ("magnetic", MAG)):
        op, ref = gj.bttb_setup(g, field, mag, precision="fp32", npad=npad), gj.bttb_setup(g, field, mag, precision="fp64")
        m, r = torch.randn(g.n, generator=gen, device="cuda"), torch.randn(g.s, generator=gen, device="cuda")
        for y, x in ((op.forward(m), ref.forward(m.double())), (op.adjoint(r), ref.adjoint(r.double()))):
            y = y.double()
            gain = float(y @ x) / float(x @ x) - 1.0
            assert abs(gain) <= 4e-8, (field, gain)
            assert float((y - x).norm() / x.norm()) <= 3e-7
        op.close()
        ref.close()
