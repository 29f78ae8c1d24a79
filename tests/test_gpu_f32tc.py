"""The tensor-core path of the fp32 GEMM (three exact bf16 planes per operand,
levels OFF, WARP and BLOCK) against the CPU oracle: shapes at the edges of its
tiles (256 x 256 and 256 x 128), chunks (32 of K) and checksum segments (256 of
K), every unit size, split-K, faults on every target, violations of the
single-event-upset model, and operands the planes cannot hold, which the
CUDA-core kernel computes.

Tolerances.  Integers: exact.  Floats: an fp32 result within the worst-case
bound 2*K*u*|A||B|, as for the CUDA-core kernel, and in the 2-norm within
u*sqrt(K/8) of the product: chunk results (32 of K) added with
round-to-nearest err by about 0.3*u*sqrt(K/32)/sqrt(2) of it, the truncated
accumulation inside a chunk by about 1u more.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
TUPLES = {
    "wide": (128, 128, 16, 64, 64, 16, 8),
    "wide32": (128, 128, 32, 64, 64, 16, 8),
    "huge": (128, 128, 8, 32, 64, 8, 8),
    "large": (64, 64, 8, 32, 64, 8, 8),
    "tall": (32, 128, 8, 16, 64, 4, 8),
    "medium": (32, 32, 8, 16, 32, 4, 4),
    "small": (16, 16, 16, 8, 16, 2, 2),
}
LEVELS = {"off": 0, "warp": 2, "block": 3}
FIELDS = ("m_tb", "n_tb", "k_tb", "m_w", "n_w", "m_t", "n_t")


@pytest.fixture(scope="module")
def ft():
    import torch
    import paper_2305_01024_gb300 as ft
    assert torch.cuda.is_available()
    ft.lib()
    return ft


def _sched(name, period=256, split_k=1):
    s = dict(zip(FIELDS, TUPLES[name]))
    return dict(s, cadence=period // s["k_tb"], split_k=split_k)


def _run(ft, A, B, Cin, alpha, beta, level, s, faults):
    import torch
    h = ft.Handle(0)
    h.set_schedule(s)
    C = torch.from_numpy(Cin.copy()).cuda()
    rep = h.gemm(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, alpha=alpha, beta=beta, level=level,
                 inject=faults)
    out = C.cpu().numpy().astype(np.float64)
    h.close()
    return out, rep


def _oracle(orc, A, B, Cin, alpha, beta, level, s, faults):
    return orc.gemm_ft(A, B, orc.Schedule(**{f: s[f] for f in FIELDS}, cadence=s["cadence"] or 10**6,  # 0: once per split
                                          split_k=s["split_k"],
                                          level=level, lam=32.0, u=U), faults=faults, alpha=alpha, beta=beta, Cin=Cin)


def _key(r):
    g = r if isinstance(r, dict) else vars(r)
    return (g["tile_m"], g["tile_n"], g["kstep"], g["row"], g["col"], g["kind"])


# (M, N, K): flop counts that take the tensor-core path, edges of 128 / 256
# rows and columns, of 32-element chunks (half chunks too) and 256-element
# segments and periods
SHAPES = [(640, 512, 352), (641, 385, 513), (255, 1153, 400), (129, 1000, 1041), (1027, 127, 777)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("name,level", [("wide32", "block"), ("wide", "warp"), ("huge", "block"), ("large", "block"),
                                        ("tall", "block"), ("tall", "warp"), ("medium", "block"), ("small", "block")])
def test_integers_and_faults_bit_exact(ft, orc, shape, name, level):
    M, N, K = shape
    s = _sched(name, period=128 if name == "wide32" else 256)
    lv = LEVELS[level]
    seed = 7000 + 13 * M + N
    A, B, Cin = synth.integers((M, K), seed), synth.integers((K, N), seed + 1), synth.integers((M, N), seed + 2)
    tm, tn, ks = -(-M // s["m_tb"]), -(-N // s["n_tb"]), -(-K // s["k_tb"])

    def at(i, j, k, r, c, delta, target=0):  # inside the (perhaps ragged) tile (i, j)
        return (i, j, k, min(r, M - i * s["m_tb"] - 1, s["m_tb"] - 1), min(c, N - j * s["n_tb"] - 1, s["n_tb"] - 1),
                delta, target)
    faults = [at(0, 0, 0, 0, 0, 512.0), at(tm - 1, tn - 1, -1, 128, 128, -256.0), at(tm // 2, 0, ks // 2, 9, 1, 128.0, 1),
              at(0, tn // 2, ks // 2, 1, 3, 64.0, 2), at(tm - 1, 0, ks - 2, 0, 128, 1024.0)]
    C, rep = _run(ft, A, B, Cin, -2.0, 3.0, lv, s, faults)
    ref = -2 * (A.astype(np.int64) @ B.astype(np.int64)) + 3 * Cin.astype(np.int64)
    res = _oracle(orc, A, B, Cin, -2.0, 3.0, lv, s, faults)
    assert np.array_equal(C, res.C)
    if res.uncorrectable == 0:  # no two of the faults in one unit and period
        assert np.array_equal(C, ref)
    assert [_key(r) for r in rep.records] == [_key(r) for r in res.records]
    for g, o in zip(rep.records, res.records):
        assert (g["delta"], g["residual_r"], g["residual_c"]) == (o.delta, o.residual_r, o.residual_c)
        assert g["tau"] == pytest.approx(o.tau, rel=1e-4, abs=1e-30)
    assert rep.corrected >= 1 and rep.detected == res.detected


@pytest.mark.parametrize("K,split,period", [(4096, 4, 256), (2049, 3, 256), (1024, 2, 0), (3000, 1, 0)])
def test_splits_and_periods_bit_exact(ft, orc, K, split, period):
    """Every split verifies its own partial; a period of 0 is one verification
    per split, over several checksum segments."""
    M, N = 520, 260
    s = _sched("wide32", period=period, split_k=split)
    A, B = synth.integers((M, K), 7100 + K), synth.integers((K, N), 7200 + K)
    faults = [(0, 0, 3, 1, 2, 512.0), (2, 2, -1, 43, 3, -512.0), (1, 1, K // 64, 100, 3, 256.0)]
    C, rep = _run(ft, A, B, np.zeros((M, N), np.float32), 1.0, 0.0, 3, s, faults)
    res = _oracle(orc, A, B, np.zeros((M, N), np.float32), 1.0, 0.0, 3, s, faults)
    assert np.array_equal(C, A.astype(np.int64) @ B.astype(np.int64))
    assert [_key(r) for r in rep.records] == [_key(r) for r in res.records]
    assert rep.corrected == 3


@pytest.mark.parametrize("shape", [(200, 130, 5000), (256, 256, 4099), (47, 300, 8192)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("name,level", [("wide32", "block"), ("wide", "warp"), ("large", "block"), ("tall", "block"),
                                        ("tall", "warp"), ("medium", "block"), ("medium", "warp"), ("small", "block"),
                                        ("wide", "off")])
def test_long_k_by_segments_bit_exact(ft, orc, shape, name, level):
    """Few tiles and a long K: the product by segments of K, then a scan that
    verifies period by period."""
    M, N, K = shape
    s, lv, seed = _sched(name), LEVELS[level], 7600 + M
    A, B, Cin = synth.integers((M, K), seed), synth.integers((K, N), seed + 1), synth.integers((M, N), seed + 2)
    tm, tn, ks = -(-M // s["m_tb"]), -(-N // s["n_tb"]), -(-K // s["k_tb"])
    faults = [(0, 0, 3, 5, 7, 512.0), (0, tn // 2, ks // 2, 2, 1, -256.0), (0, 0, ks // 3, 1, 2, 128.0, 1),
              (tm // 2, 0, ks - 1, 3, 4, 64.0, 2), (0, 0, ks // 2, 0, 0, 32.0), (0, 0, ks // 2, 9, 9, 64.0)]
    if level == "off":
        C, rep = _run(ft, A, B, Cin, -2.0, 3.0, lv, s, None)
        assert np.array_equal(C, -2 * (A.astype(np.int64) @ B.astype(np.int64)) + 3 * Cin.astype(np.int64))
        return
    C, rep = _run(ft, A, B, Cin, -2.0, 3.0, lv, s, faults)
    res = _oracle(orc, A, B, Cin, -2.0, 3.0, lv, s, faults)
    assert np.array_equal(C, res.C)
    assert [_key(r) for r in rep.records] == [_key(r) for r in res.records]
    for g, o in zip(rep.records, res.records):
        assert (g["delta"], g["residual_r"], g["residual_c"]) == (o.delta, o.residual_r, o.residual_c)
    assert rep.corrected >= 1 and rep.checksum_only >= 1


def test_two_faults_in_a_unit_stay_uncorrectable(ft, orc):
    M, N, K = 400, 700, 800
    s = _sched("wide")
    A, B = synth.integers((M, K), 7301), synth.integers((K, N), 7302)
    faults = [(1, 1, 1, 0, 0, 64.0), (1, 1, 2, 16, 32, 32.0)]
    C, rep = _run(ft, A, B, np.zeros((M, N), np.float32), 1.0, 0.0, 3, s, faults)
    res = _oracle(orc, A, B, np.zeros((M, N), np.float32), 1.0, 0.0, 3, s, faults)
    assert np.array_equal(C, res.C)
    assert [_key(r) for r in rep.records] == [_key(r) for r in res.records]
    assert rep.uncorrectable >= 1 and rep.corrected == 0


@pytest.mark.parametrize("level", ["off", "block"])
@pytest.mark.parametrize("kind", ["uniform", "positive"])
@pytest.mark.parametrize("shape", [(513, 1025, 1000), (600, 700, 6001)], ids=lambda s: "x".join(map(str, s)))
def test_floats_within_fp32_rounding(ft, shape, kind, level):
    M, N, K = shape
    A, B = synth.uniform((M, K), 7401), synth.uniform((K, N), 7402)
    if kind == "positive":
        A, B = np.abs(A), np.abs(B)
    C, rep = _run(ft, A, B, np.zeros((M, N), np.float32), 1.0, 0.0, LEVELS[level], _sched("wide32"), None)
    A, B = A.astype(np.float64), B.astype(np.float64)
    ref = A @ B
    assert np.all(np.abs(C - ref) <= 2 * K * U * (np.abs(A) @ np.abs(B)))
    assert np.linalg.norm(C - ref) <= U * np.sqrt(K / 8) * np.linalg.norm(ref)
    assert rep.detected == 0


@pytest.mark.parametrize("case", ["tiny", "huge", "one tiny", "inf", "nan"])
@pytest.mark.parametrize("aligned", [True, False])
def test_operands_outside_the_planes_take_the_cuda_cores(ft, case, aligned):
    """Magnitudes outside 2^-100 .. 2^60, infinities and NaN: what plain fp32
    arithmetic gives."""
    M, N, K = (640, 512, 512) if aligned else (641, 513, 515)
    A, B = synth.uniform((M, K), 7501), synth.uniform((K, N), 7502)
    if case == "tiny":
        A, B = A * np.float32(2.0 ** -110), B * np.float32(2.0 ** 20)
    elif case == "huge":
        A, B = A * np.float32(2.0 ** 90), B * np.float32(2.0 ** 10)
    elif case == "one tiny":
        A[3, 5] = 2.0 ** -120
    elif case == "inf":
        A[7, 9] = np.inf
    else:
        B[11, 200] = np.nan
    C, rep = _run(ft, A, B, np.zeros((M, N), np.float32), 1.0, 0.0, 0, _sched("wide32"), None)
    with np.errstate(invalid="ignore"):
        ref = A.astype(np.float64) @ B.astype(np.float64)
        bound = 2 * K * U * (np.abs(A.astype(np.float64)) @ np.abs(B.astype(np.float64)))
    fine = np.isfinite(ref)
    assert np.array_equal(np.isnan(ref), np.isnan(C))
    assert np.array_equal(C[~fine & ~np.isnan(ref)], ref[~fine & ~np.isnan(ref)])
    assert np.all(np.abs(C[fine] - ref[fine]) <= bound[fine])
    if case == "one tiny":  # (the fp32 norms of the others under- or overflow: no threshold to test against)
        C, rep = _run(ft, A, B, np.zeros((M, N), np.float32), 1.0, 0.0, 3, _sched("wide32"),
                      [(1, 2, 3, 4, 5, float(np.abs(ref).max() * 8))])
        assert rep.corrected == 1 and rep.detected == 1
        tau = rep.records[0]["tau"]
        assert np.all(np.abs(C - ref) <= bound + np.where(np.arange(M * N).reshape(M, N) == (128 + 4) * N + 256 + 5, tau, 0))
