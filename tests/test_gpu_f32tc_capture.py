"""A captured fp32 tensor-core call: what one replay's operands hold does not
reach the next.  A replay that meets a value outside the planes' range is
computed by the CUDA-core kernel, the one after it by the tensor cores again,
with the bits it had before."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,split", [("off", 1), ("block", 1), ("block", 2)])
def test_replays_do_not_see_each_other(level, split):
    import torch
    import paper_2305_01024_gb300 as ft
    M, N, K = 1024, 1000, 512
    A, B = synth.uniform((M, K), 9801), synth.uniform((K, N), 9802)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    dC, dA2 = torch.zeros(M, N, device="cuda"), torch.from_numpy(A).cuda()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    h = ft.Handle(0, stream=stream)
    h.set_schedule(dict(m_tb=128, n_tb=128, k_tb=16, m_w=64, n_w=64, m_t=16, n_t=8, cadence=16, split_k=split))

    def call(a):
        h.gemm(a, dB, dC, level=level, report=False)
    call(dA)
    torch.cuda.synchronize()
    eager = dC.cpu().numpy()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        call(dA)

    def replay(tiny):
        dA[3, 5] = 2.0 ** -120 if tiny else float(A[3, 5])
        dC.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        return dC.cpu().numpy()
    assert np.array_equal(replay(False), eager)
    stand_by = replay(True)
    rows = np.arange(M) != 3
    assert not np.array_equal(stand_by[rows], eager[rows])  # the other kernel's rounding
    assert np.allclose(stand_by[rows], eager[rows], rtol=0, atol=2 * K * 2.0 ** -24 * K)
    assert np.array_equal(replay(False), eager)
    # nor does an ordinary call of the handle that met such a value
    dA2[7, 9] = 2.0 ** -120
    torch.cuda.synchronize()
    call(dA2)
    torch.cuda.synchronize()
    assert np.array_equal(replay(False), eager)
    assert h.report_fetch().detected == 0
    h.close()
