"""fp32 on the tensor cores where the last wave of 256-column tiles runs as
halves of 128 in a second launch: more tiles than CTA pairs and a short
remainder, with and without a last tile whose second half is outside C.
Integers: C and the located faults are exact."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

WIDE = dict(m_tb=128, n_tb=128, k_tb=32, m_w=64, n_w=64, m_t=16, n_t=8)


@pytest.mark.parametrize("level", ["off", "warp", "block"])
@pytest.mark.parametrize("M,N,K,split", [(2560, 2304, 512, 1), (2500, 2060, 700, 1), (1290, 1925, 2048, 2)])
def test_tail_exact(M, N, K, split, level):
    import torch
    import paper_2305_01024_gb300 as ft
    A, B, C0 = synth.integers((M, K), 7800 + M), synth.integers((K, N), 7900 + N), synth.integers((M, N), 8000 + K)
    tm, tn, ks = -(-M // 128), -(-N // 128), -(-K // 32)
    faults = []
    if level != "off":
        # tiles across both launches, their last rows and columns, every target
        at = [(0, 0), (tm - 1, tn - 1), (tm // 2, tn - 2), (tm - 1, tn - 3), (1, tn - 1), (tm - 3, 2), (tm - 2, tn // 2)]
        for f, (i, j) in enumerate(at):
            faults.append((i, j, (5 * f) % ks, min(127, M - 128 * i - 1), min(127, N - 128 * j - 1), 256.0 * (f + 1),
                           f % 3))
    h = ft.Handle(0)
    h.set_schedule(dict(WIDE, cadence=8, split_k=split))
    C = torch.from_numpy(C0.copy()).cuda()
    rep = h.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, beta=-1.0, level=level, inject=faults)
    h.close()
    assert np.array_equal(C.cpu().numpy().astype(np.int64), A.astype(np.int64) @ B.astype(np.int64) - C0.astype(np.int64))
    want = [(i, j, 128 * i + r if g != 2 else -1, 128 * j + c if g != 1 else -1, 0 if g == 0 else 2)
            for i, j, _, r, c, _, g in faults]
    assert sorted((r["tile_m"], r["tile_n"], r["row"], r["col"], r["kind"]) for r in rep.records) == sorted(want)
