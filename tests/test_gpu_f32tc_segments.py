"""fp32 on the tensor cores with verification periods that are no multiple of
256: every period is several checksum segments, its last one shorter, in one
pass over K, over splits of K and by segments of K.  Integers: C and the
records are exact."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
TUPLES = {"wide32": (128, 128, 32, 64, 64, 16, 8), "medium": (32, 32, 8, 16, 32, 4, 4), "small": (16, 16, 16, 8, 16, 2, 2)}
FIELDS = ("m_tb", "n_tb", "k_tb", "m_w", "n_w", "m_t", "n_t")


@pytest.mark.parametrize("name,shape,period,split", [
    ("wide32", (640, 512, 1400), 384, 1), ("wide32", (520, 388, 4160), 1056, 2), ("wide32", (300, 516, 9340), 3232, 1),
    ("medium", (200, 130, 9340), 3200, 1), ("medium", (256, 256, 17000), 288, 1), ("small", (256, 250, 20000), 416, 1)])
def test_odd_periods_bit_exact(orc, name, shape, period, split):
    import torch
    import paper_2305_01024_gb300 as ft
    M, N, K = shape
    s = dict(zip(FIELDS, TUPLES[name]))
    s.update(cadence=period // s["k_tb"], split_k=split)
    t, kt = s["m_tb"], s["k_tb"]
    A, B = synth.integers((M, K), 9300 + M), synth.integers((K, N), 9400 + K)
    ks = -(-K // kt)
    p = s["cadence"]
    # the last k-step of a period, the first of the next, the last of all; one on each checksum
    faults = [(0, 0, p - 1, 3, 5, 512.0), (0, 1, p, 7, 2, -256.0), (1, 0, ks - 1, 1, 1, 1024.0),
              (1, 1, p // 2, 2, 3, 128.0, 1), (2, 2, p + 1, 0, 3, 64.0, 2)]
    h = ft.Handle(0)
    h.set_schedule(s)
    C = torch.zeros(M, N, device="cuda")
    rep = h.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, level="block", inject=faults)
    h.close()
    res = orc.gemm_ft(A, B, orc.Schedule(**s, level=3, lam=32.0, u=U), faults=faults)
    assert np.array_equal(C.cpu().numpy().astype(np.int64), A.astype(np.int64) @ B.astype(np.int64))

    def key(r):
        g = r if isinstance(r, dict) else vars(r)
        return (g["tile_m"], g["tile_n"], g["kstep"], g["row"], g["col"], g["kind"], g["delta"])
    assert [key(r) for r in rep.records] == [key(r) for r in res.records]
    assert rep.corrected == 3 and rep.checksum_only == 2
