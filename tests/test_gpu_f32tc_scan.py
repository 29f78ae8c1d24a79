"""Long K with few outputs on the tensor cores: units of one warp whose periods
are walked as shares side by side.  Shares that end early, a ragged last unit
and last period, periods of several segments, beta, and units with a scheduled
fault of every target, which one warp walks in order.  Integers: C and the
records are exact."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

UNITS = {"small": (16, 16, 16, 8, 16, 2, 2), "medium": (32, 32, 8, 16, 32, 4, 4)}
FIELDS = ("m_tb", "n_tb", "k_tb", "m_w", "n_w", "m_t", "n_t")


@pytest.mark.parametrize("unit", ["small", "medium"])
@pytest.mark.parametrize("M,N,K,period", [(250, 130, 4096, 256), (256, 256, 4353, 256), (33, 500, 17000, 1024),
                                          (130, 97, 16 * 256 + 1, 128), (257, 255, 12300, 512)])
@pytest.mark.parametrize("faulted", [False, True])
def test_shares_exact(unit, M, N, K, period, faulted):
    import torch
    import paper_2305_01024_gb300 as ft
    s = dict(zip(FIELDS, UNITS[unit]))
    s.update(cadence=period // s["k_tb"], split_k=1)
    t = s["m_tb"]
    A, B, C0 = synth.integers((M, K), 9500 + M), synth.integers((K, N), 9600 + K), synth.integers((M, N), 9700 + N)
    tm, tn, ks = -(-M // t), -(-N // t), -(-K // s["k_tb"])
    faults = []
    if faulted:
        at = [(0, 0, 3), (tm - 1, tn - 1, ks - 1), (tm // 2, tn // 2, ks // 2), (0, tn - 1, ks // 3)]
        for f, (i, j, k) in enumerate(at):
            faults.append((i, j, k, min(t, M - t * i) - 1, min(t, N - t * j) - 1, 512.0 * (f + 1), f % 3))
    h = ft.Handle(0)
    h.set_schedule(s)
    C = torch.from_numpy(C0.copy()).cuda()
    rep = h.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, alpha=1.0, beta=2.0, level="block",
                 inject=faults)
    h.close()
    want = A.astype(np.int64) @ B.astype(np.int64) + 2 * C0.astype(np.int64)
    assert np.array_equal(C.cpu().numpy().astype(np.int64), want)
    rec = [(i, j, t * i + r if g != 2 else -1, t * j + c if g != 1 else -1, 0 if g == 0 else 2)
           for i, j, _, r, c, _, g in faults]
    assert sorted((r["tile_m"], r["tile_n"], r["row"], r["col"], r["kind"]) for r in rep.records) == sorted(rec)
