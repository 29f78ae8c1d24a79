"""fp64 units computed in 1, 4 or 8 pieces (the choice follows the unit count):
faults on every target in every piece, two faults in different pieces of a
unit, units partly outside the matrix.  Integers, against the oracle."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _key(r):
    g = r if isinstance(r, dict) else vars(r)
    return (g["tile_m"], g["tile_n"], g["kstep"], g["row"], g["col"], g["kind"])


# units of 128 x 128: 1 .. 19 (8 pieces), 72 (4), 152 (1)
@pytest.mark.parametrize("M,N,K", [(33, 20, 40), (128, 128, 64), (300, 260, 72), (1030, 1025, 24), (1024, 2432, 16)])
@pytest.mark.parametrize("cadence", [2, 0])
def test_dgemm_pieces(orc, M, N, K, cadence):
    import torch
    import paper_2305_01024_gb300 as ft
    A = synth.integers((M, K), 8600 + M, dtype=np.float64)
    B = synth.integers((K, N), 8700 + N, dtype=np.float64)
    tm, tn = (M - 1) // 128, (N - 1) // 128
    rl, cl = (M - 1) % 128, (N - 1) % 128  # last row / column of the last unit
    r0, c0 = (127 if M >= 128 else M - 1), (127 if N >= 128 else N - 1)
    faults = [(0, 0, 0, r0, 0, 64.0), (tm, tn, -1, rl, cl, -32.0), (0, 0, 1 if K < 24 else 2, min(40, r0), min(70, c0), 16.0, 1),
              (tm, 0, -1, 0, min(65, c0), 8.0, 2)]
    if K >= 40:  # two in one unit and period: uncorrectable
        faults += [(0, 0, 4, 0, 0, 64.0), (0, 0, 4, r0, c0, 128.0)]
    h = ft.Handle(0)
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    rep = h.dgemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, cadence=cadence, inject=faults)
    h.close()
    res = orc.gemm_ft(A, B, orc.dgemm_schedule(cadence=cadence or 10**6), faults=faults)
    assert np.array_equal(C.cpu().numpy(), res.C)
    assert [_key(r) for r in rep.records] == [_key(r) for r in res.records]
    for g, o in zip(rep.records, res.records):
        assert (g["delta"], g["residual_r"], g["residual_c"]) == (o.delta, o.residual_r, o.residual_c)


@pytest.mark.parametrize("M,N,K", [(17, 9, 24), (64, 64, 40), (150, 130, 48), (640, 1024, 16)])
def test_zgemm_pieces(orc, M, N, K):
    import torch
    import paper_2305_01024_gb300 as ft
    mk = lambda sh, s: synth.integers(sh, s, dtype=np.float64) + 1j * synth.integers(sh, s + 1, dtype=np.float64)
    A, B = mk((M, K), 8800 + M), mk((K, N), 8900 + N)
    tm, tn = (M - 1) // 64, (N - 1) // 64
    faults = [(0, 0, 0, min(33, M - 1), 0, 64.0, 0), (tm, tn, -1, (M - 1) % 64, (N - 1) % 64, 32.0, 4)]
    if tm or tn:
        faults += [(tm, 0, 1, 1, 2, 16.0, 1), (0, tn, 1, 2, 1, 16.0, 6)]
    h = ft.Handle(0)
    C = torch.zeros(M, N, dtype=torch.complex128, device="cuda")
    rep = h.zgemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, cadence=1, inject=faults)
    h.close()
    res = orc.zgemm_ft(A, B, tile=64, k_tb=8, cadence=1, faults=faults)
    assert np.array_equal(C.cpu().numpy(), res.C)
    assert [_key(r) for r in rep.records] == [_key(r) for r in res.records]
