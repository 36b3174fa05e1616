"""mm_hessian_vec takes device inputs that do not lie on a boundary of their type: they are copied, not read in place."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1405_2728_gb300 import inputs
from gpu_cases import dev, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,dtype", [("MM_FP64", torch.float64), ("MM_FP32", torch.float32)])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_unaligned_device_inputs(mmlib, prec, dtype, offset):
    prob, oprob = make_pair(mmlib, 12, 7, 3, (3.90625e-9, 3.90625e-9, 5e-9), precision=getattr(mmlib, prec))
    m = dev(inputs.random_unit_m(oprob.shape, 3), dtype)
    v = dev(inputs.random_unit_m(oprob.shape, 4), dtype)
    H = (1e3, 0.0, 0.0)
    want, out = torch.empty_like(m), torch.empty_like(m)
    mmlib.mm_hessian_vec(prob, m, H, v, want)

    def shifted(t):
        raw = t.reshape(-1).view(torch.uint8)
        buf = torch.zeros(raw.numel() + 16, dtype=torch.uint8, device="cuda")
        buf[offset:offset + raw.numel()] = raw
        return buf, ctypes.c_void_p(buf.data_ptr() + offset)

    (mb, mp), (vb, vp) = shifted(m), shifted(v)
    torch.cuda.synchronize()
    h = (ctypes.c_double * 3)(*H)
    for a, b in ((mp, ctypes.c_void_p(v.data_ptr())), (ctypes.c_void_p(m.data_ptr()), vp), (mp, vp)):
        out.zero_()
        torch.cuda.synchronize()
        assert mmlib.lib().mm_hessian_vec(prob.handle, a, h, b, ctypes.c_void_p(out.data_ptr()), None) == mmlib.MM_OK
        assert np.array_equal(out.cpu().numpy(), want.cpu().numpy())
