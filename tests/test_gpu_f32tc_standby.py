"""The CUDA-core stand-by of the fp32 tensor-core route, on each of its ways:
a call with a report (the host looks at the flag), a call without one and a
call over splits of K (kernels that look at it themselves).  One value below
the planes' range, a fault, beta, aligned and unaligned operands; then a call
in range on the same handle.

Tolerances: the worst-case bound 2*K*u*|A||B| of an fp32 product, with one u
of |beta C| and, at the corrected element, its threshold."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
WIDE = dict(m_tb=128, n_tb=128, k_tb=16, m_w=64, n_w=64, m_t=16, n_t=8, cadence=16)


@pytest.mark.parametrize("report,split", [(True, 1), (False, 1), (True, 3), (False, 2)])
@pytest.mark.parametrize("level", ["off", "warp", "block"])
@pytest.mark.parametrize("aligned", [True, False])
def test_value_outside_the_planes(report, split, level, aligned):
    import torch
    import paper_2305_01024_gb300 as ft
    M, N, K = (1024, 896, 1024) if aligned else (1023, 897, 1009)
    A, B, C0 = synth.uniform((M, K), 9901), synth.uniform((K, N), 9902), synth.uniform((M, N), 9903)
    good = A.copy()
    A[5, 7] = 2.0 ** -120
    r, c = 128 + 17, 256 + 40
    faults = None if level == "off" else [(1, 2, 30, 17, 40, 256.0)]
    h = ft.Handle(0)
    h.set_schedule(dict(WIDE, split_k=split))
    dB = torch.from_numpy(B).cuda()

    def call(a):
        dC = torch.from_numpy(C0.copy()).cuda()
        rep = h.gemm(torch.from_numpy(a).cuda(), dB, dC, alpha=0.75, beta=-0.5, level=level, inject=faults, report=report)
        if not report:
            rep = h.report_fetch()
        a, b = a.astype(np.float64), B.astype(np.float64)
        bound = 2 * K * U * 0.75 * (np.abs(a) @ np.abs(b)) + 2 * U * np.abs(C0)
        if faults:
            assert (rep.detected, rep.corrected) == (1, 1)
            assert (rep.records[0]["row"], rep.records[0]["col"]) == (r, c)
            bound[r, c] += 0.75 * rep.records[0]["tau"]
        else:
            assert rep.detected == 0
        C = dC.cpu().numpy()
        assert np.all(np.abs(C - (0.75 * (a @ b) - 0.5 * C0)) <= bound)
        return C
    cores, tensor = call(A), call(good)
    rows = np.arange(M) != 5
    assert not np.array_equal(cores[rows], tensor[rows])  # two kernels, two roundings
    assert np.array_equal(call(A), cores)
    assert np.array_equal(call(good), tensor)
    h.close()


def test_kernel_time_covers_the_stand_by():
    """The statistics' kernel time is that of the kernel that computed C, with
    and without a report; a call counts once."""
    import torch
    import paper_2305_01024_gb300 as ft
    n = 2048
    A, B = torch.rand(n, n, device="cuda"), torch.rand(n, n, device="cuda")
    A[3, 4] = 2.0 ** -120
    C = torch.zeros(n, n, device="cuda")
    h = ft.Handle(0)
    ms = {}
    for report in (True, False):
        h.gemm(A, B, C, level="block", report=report)
        h.enable_timing(True)
        h.stats(reset=True)
        for _ in range(5):
            h.gemm(A, B, C, level="block", report=report)
        st = h.stats(reset=True)
        h.enable_timing(False)
        assert st["timed_launches"] == 5
        ms[report] = st["kernel_ms"]
    h.close()
    assert ms[False] > 0.5 * ms[True]  # (a few us a call, without the stand-by)
