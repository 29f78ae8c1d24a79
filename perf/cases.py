"""The calls this library is timed on: what its users have it do, through the
public Python binding, from the smallest call to the largest.

A case is a dict of plain values.  `kind` selects the entry point:

  sgemm   Handle.gemm on fp32 operands at any checksum level
  tc      Handle.gemm on bf16 operands (tensor cores), level tile or off
  fp8     Handle.quantize of one operand, then Handle.gemm on e4m3 codes
  group   Group.run over many bf16 GEMMs, then Handle.report_fetch
  fp64    Handle.dgemm / Handle.zgemm with block checksums

`prepare` makes what a program has in hand before the call (operands, output
buffer, handle, a group), `run` is one pass, `work` its least bytes and
flops, `exact` the same result in 64 bits by plain torch.
"""
import math
import random

import torch

import paper_2305_01024_gb300 as ft

# the 128 x 128 tile with k-steps of 32, verified every 256 of K: the schedule
# the benchmark fixes for its largest fp32 GEMM
K32 = dict(m_tb=128, n_tb=128, k_tb=32, m_w=64, n_w=64, m_t=16, n_t=8, cadence=8, split_k=1)
LEVEL = {"off": ft.FT_OFF, "thread": ft.FT_THREAD, "warp": ft.FT_WARP, "block": ft.FT_BLOCK, "tile": ft.FT_TILE}


def _sgemm(name, m, n, k, level="block", dist="uniform", beta=0.0, schedule="default", faults=0):
    return dict(name=name, kind="sgemm", m=m, n=n, k=k, level=level, dist=dist, beta=beta, schedule=schedule,
                faults=faults)


def _tc(name, m, n, k, level="tile"):
    return dict(name=name, kind="tc", m=m, n=n, k=k, level=level)


def listed():
    return [
        # one small protected GEMM, its report read at once: latency and launches
        _sgemm("sgemm_256_block", 256, 256, 256),
        # a ragged fp32 GEMM of middling size that is hit by one fault
        _sgemm("sgemm_777x1531x2049_block_fault", 777, 1531, 2049, dist="normal", faults=1),
        # a small output reduced over a very long K
        _sgemm("sgemm_256x256x65536_block", 256, 256, 65536, dist="normal"),
        # the finer checksum unit of Section 4.2.2
        _sgemm("sgemm_2048_warp", 2048, 2048, 2048, level="warp", beta=0.5),
        # the square sweep's middle, accumulating into C
        _sgemm("sgemm_4096_block", 4096, 4096, 4096, beta=0.5),
        # the headline: the square sweep's largest size on the benchmark's schedule
        _sgemm("sgemm_16384_block", 16384, 16384, 16384, beta=0.5, schedule="k32"),
        # a small bf16 GEMM with checksums through the MMA
        _tc("bf16_300x500x256_tile", 300, 500, 256),
        # an ordinary unprotected bf16 GEMM
        _tc("bf16_4096_off", 4096, 4096, 4096, level="off"),
        # a large protected bf16 GEMM
        _tc("bf16_8192_tile", 8192, 8192, 8192),
        # fp8 inference: fresh activations quantized, then multiplied by
        # weights that were quantized once
        dict(name="fp8_4096x4096x8192_tile", kind="fp8", m=4096, n=4096, k=8192),
        # many uneven bf16 GEMMs in one launch, 1% of the tiles hit by a fault
        dict(name="group_128_tile", kind="group", count=128, max_mn=4096, max_k=2048, level="tile", fault_pct=1),
        # double precision with block checksums
        dict(name="dgemm_2048_block", kind="fp64", m=2048, n=2048, k=2048, complex=False),
    ]


def _logint(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, int(v) // step * step)


def draw(rng):
    f = rng.randrange(10)
    if f == 0:
        m, n, k = (_logint(rng, 48, 640) for _ in range(3))
        c = _sgemm("", m, n, k, level=rng.choice(["block", "block", "off"]))
    elif f == 1:
        m, n, k = (_logint(rng, 640, 4096) for _ in range(3))
        c = _sgemm("", m, n, k, dist="normal", faults=1)
    elif f == 2:
        m, n = (_logint(rng, 64, 512) for _ in range(2))
        c = _sgemm("", m, n, _logint(rng, 8192, 65536), dist="normal")
    elif f == 3:
        m, n, k = (_logint(rng, 512, 4096) for _ in range(3))
        c = _sgemm("", m, n, k, level=rng.choice(["warp", "thread"]), beta=0.5)
    elif f == 4:
        m, n, k = (_logint(rng, 2048, 12288) for _ in range(3))
        c = _sgemm("", m, n, k, level=rng.choice(["block", "block", "off"]), beta=rng.choice([0.0, 0.5]),
                   dist=rng.choice(["uniform", "normal"]), schedule=rng.choice(["default", "k32"]))
    elif f == 5:
        c = _tc("", _logint(rng, 64, 1024), _logint(rng, 64, 1024), _logint(rng, 64, 1024, 8),
                rng.choice(["tile", "off"]))
    elif f == 6:
        c = _tc("", _logint(rng, 2048, 12288), _logint(rng, 2048, 12288), _logint(rng, 2048, 12288, 8),
                rng.choice(["tile", "off"]))
    elif f == 7:
        c = dict(kind="fp8", m=_logint(rng, 256, 8192), n=_logint(rng, 1024, 8192), k=_logint(rng, 1024, 8192, 16))
    elif f == 8:
        c = dict(kind="group", count=_logint(rng, 8, 160), max_mn=_logint(rng, 512, 4096, 16),
                 max_k=_logint(rng, 512, 2048, 16), level=rng.choice(["tile", "tile", "off"]), fault_pct=1)
    else:
        z = rng.random() < 0.4
        m, n, k = (_logint(rng, 128, 1536 if z else 3072) for _ in range(3))
        c = dict(kind="fp64", m=m, n=n, k=k, complex=z)
    c.pop("name", None)
    return c


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _matrix(g, shape, dist="normal", dtype=torch.float32):
    if dist == "normal":
        return torch.randn(shape, generator=g, device="cuda", dtype=dtype)
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype).mul_(2).sub_(1)


def _operands(case, seed):
    """The operands of a single GEMM, from the seed alone."""
    g = _gen(seed)
    m, n, k = case["m"], case["n"], case["k"]
    if case["kind"] == "sgemm":
        A, B = _matrix(g, (m, k), case["dist"]), _matrix(g, (k, n), case["dist"])
        return A, B, _matrix(g, (m, n), case["dist"]) if case["beta"] else None
    if case["kind"] == "tc":
        return _matrix(g, (m, k)).bfloat16(), _matrix(g, (k, n)).bfloat16(), None
    if case["kind"] == "fp8":
        return _matrix(g, (m, k)), _matrix(g, (k, n)), None
    dtype = torch.complex128 if case["complex"] else torch.float64
    return _matrix(g, (m, k), dtype=dtype), _matrix(g, (k, n), dtype=dtype), None


def _group_shapes(case):
    """Problem sizes as multiples of 16: a property of the case, not of the seed."""
    rng = random.Random(case["count"] * 7919 + case["max_mn"] * 31 + case["max_k"])
    return [(16 * rng.randint(4, case["max_mn"] // 16), 16 * rng.randint(4, case["max_mn"] // 16),
             16 * rng.randint(4, case["max_k"] // 16)) for _ in range(case["count"])]


def _group_operands(case, seed):
    g = _gen(seed)
    return [(_matrix(g, (m, k)).bfloat16(), _matrix(g, (k, n)).bfloat16()) for m, n, k in _group_shapes(case)]


def prepare(case, seed):
    kind = case["kind"]
    h = ft.Handle(0)
    if kind == "group":
        ops = _group_operands(case, seed)
        shapes = [(a.shape[0], b.shape[1]) for a, b in ops]
        flat = torch.zeros(sum(m * n for m, n in shapes), device="cuda")
        problems, at = [], 0
        for (a, b), (m, n) in zip(ops, shapes):
            problems.append((a, b, flat[at:at + m * n].view(m, n)))
            at += m * n
        level = LEVEL[case["level"]]
        group = ft.Group(h, problems, dtype=ft.BF16, level=level)
        if case["level"] == "tile" and case["fault_pct"]:
            rng = random.Random(seed)
            dm, dn = ft.tc_tile(ft.BF16, level)
            tm, tn = group.tiles()
            tiles = [(p, i, j) for p in range(len(ops)) for i in range(tm[p]) for j in range(tn[p])]
            faults = []
            for p, i, j in rng.sample(tiles, max(1, len(tiles) * case["fault_pct"] // 100)):
                m, n = shapes[p]
                r, c = rng.randrange(min(dm, m - i * dm)), rng.randrange(min(dn, n - j * dn))
                faults.append((p, i, j, -1, r, c, 64.0 * math.sqrt(ops[p][0].shape[1])))
            group.set_faults(faults)
        return dict(case=case, h=h, group=group, C=flat)
    A, B, C0 = _operands(case, seed)
    m, n, k = case["m"], case["n"], case["k"]
    st = dict(case=case, h=h, A=A, B=B, C0=C0)
    if kind == "fp64":
        st["C"] = torch.zeros((m, n), dtype=A.dtype, device="cuda")
        return st
    st["C"] = torch.zeros((m, n), device="cuda")
    if kind == "fp8":
        # the weights, quantized once
        st["B"], st["scale_b"] = h.quantize(B, ft.E4M3)
    if kind == "sgemm":
        if case["schedule"] == "k32":
            h.set_schedule(K32)
        st["inject"] = None
        if case["faults"]:
            # one corrupted accumulator at a fixed element, half way along K,
            # in the tiling the handle uses for this shape
            s = h.get_schedule(m, n, k, level=LEVEL[case["level"]])
            r, c = m // 3, n // 2
            st["inject"] = [(r // s.m_tb, c // s.n_tb, (k // 2) // s.k_tb, r % s.m_tb, c % s.n_tb,
                             64.0 * math.sqrt(k))]
    return st


def _result(C, rep):
    return dict(C=C, detected=rep.detected, corrected=rep.corrected, uncorrectable=rep.uncorrectable)


def run(st):
    case, h = st["case"], st["h"]
    kind = case["kind"]
    if kind == "group":
        st["group"].run()
        return _result(st["C"], h.report_fetch())
    A, B, C = st["A"], st["B"], st["C"]
    if kind == "sgemm":
        if case["beta"]:
            C.copy_(st["C0"])
        return _result(C, h.gemm(A, B, C, beta=case["beta"], level=LEVEL[case["level"]], inject=st["inject"]))
    if kind == "tc":
        return _result(C, h.gemm(A, B, C, level=LEVEL[case["level"]], dtype=ft.BF16))
    if kind == "fp8":
        codes, scale = h.quantize(A, ft.E4M3)
        h.set_fp8_scales(scale, st["scale_b"])
        out = _result(C, h.gemm(codes, B, C, level=ft.FT_TILE, dtype=ft.E4M3))
        out["codes"] = codes
        return out
    return _result(C, (h.zgemm if case["complex"] else h.dgemm)(A, B, C))


def work(case):
    if case["kind"] == "group":
        shapes = _group_shapes(case)
        return {"bytes": sum(2 * (m * k + k * n) + 4 * m * n for m, n, k in shapes),
                "flops": sum(2 * m * n * k for m, n, k in shapes)}
    m, n, k = case["m"], case["n"], case["k"]
    flops = 2 * m * n * k
    if case["kind"] == "sgemm":
        b = 4 * (m * k + k * n + m * n * (2 if case["beta"] else 1))
    elif case["kind"] == "tc":
        b = 2 * (m * k + k * n) + 4 * m * n
    elif case["kind"] == "fp8":
        b = 4 * m * k + m * k + k * n + 4 * m * n
    else:
        e = 16 if case["complex"] else 8
        b = e * (m * k + k * n + m * n)
        flops *= 4 if case["complex"] else 1
    return {"bytes": b, "flops": flops}


def _e4m3(x):
    """Per-tensor scale amax / 448 and round to nearest even, saturating."""
    scale = x.abs().max() / 448.0
    return (x / scale).clamp(-448.0, 448.0).to(torch.float8_e4m3fn).double(), scale.double()


def exact(case, seed):
    counts = dict(detected=None, corrected=None, uncorrectable=None)
    if case["kind"] == "group":
        return dict(C=torch.cat([(a.double() @ b.double()).reshape(-1) for a, b in _group_operands(case, seed)]), **counts)
    A, B, C0 = _operands(case, seed)
    if case["kind"] == "fp8":
        (qa, sa), (qb, sb) = _e4m3(A), _e4m3(B)
        return dict(C=(qa @ qb) * (sa * sb), codes=None, **counts)
    if case["kind"] == "fp64":
        return dict(C=A @ B, **counts)
    C = A.double() @ B.double()
    if C0 is not None:
        C += case["beta"] * C0.double()
    return dict(C=C, **counts)
