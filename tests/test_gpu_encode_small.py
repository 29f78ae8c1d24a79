"""The one-launch encode pass of small fp32 problems, at the edges of its blocks
(32 rows of A, 128 columns of B, 256 elements of K a step) and of its range,
with B on and off the 16-byte boundary: integers, C and the records exact."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

SMALL = dict(m_tb=16, n_tb=16, k_tb=16, m_w=8, n_w=16, m_t=2, n_t=2, cadence=16, split_k=1)
TALL = dict(m_tb=32, n_tb=128, k_tb=8, m_w=16, n_w=64, m_t=4, n_t=8, cadence=32, split_k=1)


@pytest.mark.parametrize("K", [1, 31, 255, 256, 257, 700, 1024, 1025])
@pytest.mark.parametrize("M,N", [(31, 127), (32, 128), (33, 129), (5, 3), (100, 260)])
@pytest.mark.parametrize("sched,level", [(SMALL, 3), (SMALL, 2), (TALL, 3), (TALL, 2), (TALL, 1), (SMALL, 0)])
def test_exact(orc, M, N, K, sched, level):
    import torch
    import paper_2305_01024_gb300 as ft
    A, B = synth.integers((M, K), 8400 + K), synth.integers((K, N), 8500 + K)
    ldb = N + (K % 3)  # on and off the boundary
    dB = torch.zeros(K, ldb, device="cuda")[:, :N]
    dB.copy_(torch.from_numpy(B))
    h = ft.Handle(0)
    h.set_schedule(sched)
    C = torch.zeros(M, N, device="cuda")
    faults = [(0, 0, -1, 2, 1, 4096.0)] if level else []
    rep = h.gemm(torch.from_numpy(A).cuda(), dB, C, level=level, inject=faults)
    h.close()
    assert np.array_equal(C.cpu().numpy().astype(np.int64), A.astype(np.int64) @ B.astype(np.int64))
    if not level:
        return
    f = {k: sched[k] for k in ("m_tb", "n_tb", "k_tb", "m_w", "n_w", "m_t", "n_t", "cadence", "split_k")}
    res = orc.gemm_ft(A, B, orc.Schedule(**f, level=level, lam=32.0, u=2.0 ** -24), faults=faults)
    assert [(r["row"], r["col"], r["kind"], r["delta"]) for r in rep.records] == \
        [(r.row, r.col, r.kind, r.delta) for r in res.records]
    for g, o in zip(rep.records, res.records):
        assert g["tau"] == pytest.approx(o.tau, rel=1e-4)
