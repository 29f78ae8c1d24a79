"""Handles that come and go: each has its own report, though closed ones leave
their page-locked memory to the next.  More handles at once than are kept, closed
and opened in turn and from several threads, every one with its own faults."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_reports_stay_apart():
    import torch
    import paper_2305_01024_gb300 as ft
    n = 256
    A, B = torch.ones(n, n, device="cuda"), torch.ones(n, n, device="cuda")
    torch.cuda.synchronize()
    errors = []

    def use(h, C, tag):
        faults = [(t // 16, t % 16, 3, 1, 2, 1024.0 + tag) for t in range(tag % 5)]
        rep = h.gemm(A, B, C, level="block", inject=faults)
        if [r["delta"] for r in rep.records] != [1024.0 + tag] * (tag % 5) or rep.corrected != tag % 5:
            errors.append((tag, rep.records))
        codes, scale = h.quantize(A * (tag + 1), ft.E4M3)
        if abs(scale - (tag + 1) / 448.0) > 1e-6 * (tag + 1):
            errors.append((tag, scale))

    def run(base):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            C = torch.zeros(n, n, device="cuda")
            hs = [ft.Handle(0, stream=stream) for _ in range(8)]
            for rounds in range(3):
                for i, h in enumerate(hs):
                    use(h, C, base + 8 * rounds + i)
                for i in range(0, 8, 2):
                    hs[i].close()
                    hs[i] = ft.Handle(0, stream=stream)
            for h in hs:
                h.close()
    run(0)
    threads = [threading.Thread(target=run, args=(100 * t,)) for t in range(1, 5)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
