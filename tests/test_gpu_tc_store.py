"""Stores of the tensor-core epilogue at the edges of its tiles: whole and
ragged column groups, rows on and off 16 bytes, beta, OFF and TILE, single
CTAs and pairs.  Integers below 2^24: C is exact; elements of the buffer
outside C keep their value."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pair", [0, 1])
@pytest.mark.parametrize("level", ["off", "tile"])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (2.0, 0.0), (1.0, -1.0)])
@pytest.mark.parametrize("N,ldc,off", [(252, 252, 0), (253, 256, 0), (504, 504, 1), (505, 505, 0), (520, 524, 4)])
@pytest.mark.parametrize("M", [93, 125, 257])
def test_store_exact(M, N, ldc, off, alpha, beta, level, pair):
    import torch
    import paper_2305_01024_gb300 as ft
    K = 72
    for dt, tt in ((ft.BF16, torch.bfloat16), (ft.E4M3, torch.float8_e4m3fn)):
        k = K if dt == ft.BF16 else 2 * K
        A, B, C0 = synth.integers((M, k), 9100 + M), synth.integers((k, N), 9200 + N), synth.integers((M, N), 9300 + N)
        dA, dB = torch.from_numpy(A).cuda().to(tt), torch.from_numpy(B).cuda().to(tt)
        if dt == ft.E4M3:
            dA, dB = dA.view(torch.uint8), dB.view(torch.uint8)
        flat = torch.full((off + M * ldc + 8,), 7.0, device="cuda")
        C = flat[off:off + M * ldc].view(M, ldc)[:, :N]
        C.copy_(torch.from_numpy(C0))
        h = ft.Handle(0)
        h.set_tc_pair(pair)
        rep = h.gemm(dA, dB, C, alpha=alpha, beta=beta, level=level, dtype=dt)
        h.close()
        want = alpha * (A.astype(np.float64) @ B.astype(np.float64)) + beta * C0
        assert rep.detected == 0
        assert np.array_equal(C.cpu().numpy().astype(np.float64), want)
        C.fill_(7.0)
        assert bool((flat == 7.0).all())
