"""The Gramian's directions written over its vectors: the same bits as into buffers of their own, for
either order of the two, with 16-byte and single loads, over one block and many, on both entry
points."""
import numpy as np
import pytest
import torch

from tests.gpu_common import lib, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n,shift", [(37, 0), (37, 1), (304 * 4096 * 3 + 7, 0), (304 * 4096 * 3 + 7, 1)])
@pytest.mark.parametrize("swap", [False, True])
@pytest.mark.parametrize("name", ["gj_gramian_value_grad", "gj_gramian_value_grad_noalloc"])
def test_directions_over_the_vectors(prec, n, shift, swap, name):
    lib()
    from paper_2112_15562_gb300 import _lib

    call = getattr(_lib.load(), name)
    code = _lib.GJ_FP64 if prec == "fp64" else _lib.GJ_FP32_MIXED
    rng = np.random.default_rng(n)
    m = [to_dev(rng.uniform(0, 1, n + shift), prec)[shift:] for _ in range(2)]
    st = torch.cuda.current_stream().cuda_stream
    S = torch.zeros(2, dtype=torch.float64, device="cuda")
    out = [torch.empty(n + shift, dtype=m[0].dtype, device="cuda")[shift:] for _ in range(2)]
    assert call(n, code, m[0].data_ptr(), m[1].data_ptr(), S.data_ptr(), out[0].data_ptr(), out[1].data_ptr(), st) == 0
    over = [m[1], m[0]] if swap else m
    assert call(n, code, m[0].data_ptr(), m[1].data_ptr(), S.data_ptr() + 8, over[0].data_ptr(), over[1].data_ptr(), st) == 0
    assert S[0].item() == S[1].item()
    assert torch.equal(over[0], out[0]) and torch.equal(over[1], out[1])
