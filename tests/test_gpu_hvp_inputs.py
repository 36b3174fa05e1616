"""mm_hessian_vec reads device inputs where they are: outputs that coincide with an input, overlap it shifted, or lie
apart all give the product of the inputs as they were at the call, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1405_2728_gb300 import inputs
from gpu_cases import dev, make_pair

pytestmark = pytest.mark.gpu
CELL = (3.90625e-9, 3.90625e-9, 5e-9)


@pytest.mark.parametrize("which", ["m", "v"])
@pytest.mark.parametrize("shift", [0, 2, -2, 64])
def test_output_over_an_input(mmlib, which, shift):
    prob, oprob = make_pair(mmlib, 12, 7, 3, CELL)
    n = 3 * 12 * 7 * 3
    m = inputs.random_unit_m(oprob.shape, 3)
    v = inputs.random_unit_m(oprob.shape, 4)
    v -= np.sum(m * v, axis=0, keepdims=True) * m
    want = torch.empty(m.shape, dtype=torch.float64, device="cuda")
    mmlib.mm_hessian_vec(prob, dev(m), (1e3, 0, 0), dev(v), want)
    buf = torch.zeros(n + 200, dtype=torch.float64, device="cuda")
    src = buf[100:100 + n].view(m.shape)
    out = buf[100 + shift:100 + shift + n].view(m.shape)      # 16-byte aligned
    src.copy_(dev(m if which == "m" else v))
    other = dev(v if which == "m" else m)
    mmlib.mm_hessian_vec(prob, *((src, (1e3, 0, 0), other) if which == "m" else (other, (1e3, 0, 0), src)), out)
    assert torch.equal(out, want)
    host = np.empty(m.shape)
    mmlib.mm_hessian_vec(prob, m, (1e3, 0, 0), v, host)       # host arrays go through the work buffers
    assert np.array_equal(host, want.cpu().numpy())
