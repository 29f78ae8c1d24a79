"""fp32 calls where the device has no room for the tensor-core route's planes:
they run on the CUDA cores, and the workspace the handle has is left as it is
(it may be in a captured graph, and giving it up costs a synchronisation, a free
and two allocations a call)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


def test_no_room_for_the_planes():
    import torch
    import paper_2305_01024_gb300 as ft
    n = 8192
    A, B = torch.rand(n, n, device="cuda") - 0.5, torch.rand(n, n, device="cuda") - 0.5
    C = torch.zeros(n, n, device="cuda")
    h = ft.Handle(0)
    # a workspace of 0.56 GB (A^T of 8192 x 16384), enough for the CUDA-core kernel
    # at 8192^3 (0.28 GB) but not for the planes and checksum segments (0.95 GB)
    wide = torch.rand(n, 2 * n, device="cuda")
    h.gemm(wide, torch.rand(2 * n, 256, device="cuda"), torch.zeros(n, 256, device="cuda"), level="thread")
    h.gemm(A[:1024, :1024], B[:1024, :1024], C[:1024, :1024], level="block")
    del wide
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    assert free > 2000 * MB
    filler = torch.empty(free - 200 * MB, dtype=torch.uint8, device="cuda")
    try:
        before = torch.cuda.mem_get_info()[0]
        for _ in range(2):
            rep = h.gemm(A, B, C, level="block")
            assert rep.detected == 0
            assert abs(torch.cuda.mem_get_info()[0] - before) < 64 * MB
        cores = C.cpu().numpy()
    finally:
        del filler
        torch.cuda.empty_cache()
    h.gemm(A, B, C, level="block")
    tensor = C.cpu().numpy()
    assert not np.array_equal(cores, tensor)  # the tensor cores once there is room
    ref = (A[:64].double() @ B.double()).cpu().numpy()
    bound = 2 * n * 2.0 ** -24 * (A[:64].double().abs() @ B.double().abs()).cpu().numpy()
    for got in (cores, tensor):
        assert np.all(np.abs(got[:64] - ref) <= bound)
    h.close()
