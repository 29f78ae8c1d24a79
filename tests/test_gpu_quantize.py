"""The quantizer's vector and element paths: lengths around its groups of four
and its block's share, operands off the 16-byte (codes off the 4-byte)
boundary.  Codes and scale equal the definition's bit for bit."""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("xo,yo", [(0, 0), (1, 0), (0, 1), (2, 3)])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 4096, 4099, 152 * 8 * 256 * 16 + 1, 1_000_003])
def test_codes_and_scale(n, xo, yo):
    import torch
    import paper_2305_01024_gb300 as ft
    h = ft.Handle(0)
    x = torch.zeros(n + 8, device="cuda")[xo:xo + n]
    x.copy_(torch.from_numpy(synth.normal((n,), 8100 + n % 1000)))
    x[::7] *= 1e-5  # codes in the subnormal range
    for dtype, y in ((ft.E4M3, torch.zeros(n + 8, dtype=torch.uint8, device="cuda")[yo:yo + n]),
                     (ft.BF16, torch.zeros(n + 8, dtype=torch.bfloat16, device="cuda")[yo:yo + n])):
        s = C.c_float(0.0)
        rc = ft.lib().ftgemm_quantize(h._h, n, C.c_void_p(x.data_ptr()), C.c_void_p(y.data_ptr()), dtype, C.byref(s))
        assert rc == 0, ft.lib().ftgemm_last_error()
        torch.cuda.synchronize()
        if dtype == ft.BF16:
            assert s.value == 1.0 and torch.equal(y, x.to(torch.bfloat16))
            continue
        scale = np.float32(x.abs().max().item()) / np.float32(448.0)
        assert np.float32(s.value) == scale
        want = (x.cpu() / torch.tensor(scale)).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).view(torch.uint8)
        assert torch.equal(y.cpu(), want)
    h.close()
