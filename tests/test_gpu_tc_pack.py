"""Operand layouts of the tensor-core encode pass at the edges of its blocks:
columns around the data tile (252 bf16, 248 e4m3), elements of K around a
k-block (64, 128) and a block's share of them, B on and off the 8-byte
boundary.  Integers: C and the located faults are exact."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [0, 1, 4])
@pytest.mark.parametrize("N", [1, 7, 247, 252, 253, 260, 509])
@pytest.mark.parametrize("M,K", [(3, 8), (124, 56), (126, 72), (130, 264), (251, 1096)])
@pytest.mark.parametrize("dtype", ["bf16", "e4m3"])
def test_tile_level_exact(dtype, M, N, K, off):
    import torch
    import paper_2305_01024_gb300 as ft
    dt = ft.BF16 if dtype == "bf16" else ft.E4M3
    K = K if dtype == "bf16" else K * 2
    A, B = synth.integers((M, K), 8200 + M), synth.integers((K, N), 8300 + N)
    tt = torch.bfloat16 if dtype == "bf16" else torch.float8_e4m3fn
    ldb = N + off
    dA = torch.from_numpy(A).cuda().to(tt)
    wide = torch.zeros(K * ldb + 8, device="cuda").to(tt)
    wide = wide if dtype == "bf16" else wide.view(torch.uint8)
    dB = wide[off:off + K * ldb].view(K, ldb)[:, :N]
    src = torch.from_numpy(B).cuda().to(tt)
    dB.copy_(src if dtype == "bf16" else src.view(torch.uint8))
    if dtype == "e4m3":
        dA = dA.view(torch.uint8)
    C = torch.zeros(M, N, device="cuda")
    h = ft.Handle(0)
    dm, dn = ft.tc_tile(dt, ft.FT_TILE)
    r, c = min(dm - 1, M - 1), (N - 1) % dn
    rep = h.gemm(dA, dB, C, level=ft.FT_TILE, dtype=dt, inject=[(0, (N - 1) // dn, -1, r, c, 2048.0)])
    h.close()
    assert np.array_equal(C.cpu().numpy().astype(np.int64), A.astype(np.int64) @ B.astype(np.int64))
    assert [(x["row"], x["col"], x["kind"], x["delta"]) for x in rep.records] == [(r, N - 1, 0, 2048.0)]
