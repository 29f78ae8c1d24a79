"""How the fp32 tensor-core GEMM cuts K into checksum segments, on the host:
the kernel's own header, compiled by the C++ compiler.  Segments tile every
split, none is longer than asked for, none straddles the end of a verification
period, and all start on a chunk of 32."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2305_01024_gb300", "csrc")
SRC = """
#include "f32tc_seg.cuh"
extern "C" int layout(int span, int period, int most, int* per) {
  const ftg::F32TcSegs t = ftg::f32tc_segs(span, period, most);
  *per = t.per_period;
  return t.per_split;
}
extern "C" void segment(int span, int period, int most, int j, int here, int* out) {
  ftg::f32tc_segment(ftg::f32tc_segs(span, period, most), j, here, out, out + 1);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("seg")
    (d / "seg.cpp").write_text(SRC)
    so = str(d / "seg.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "seg.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("most", [256, 512, 4096])
@pytest.mark.parametrize("period", [32, 96, 128, 256, 384, 512, 1024, 3200, 3232, 8224, 10**6])
@pytest.mark.parametrize("span,last", [(16384, 16384), (16384, 100), (9340, 9340), (65536, 33000), (255, 255), (7, 7),
                                       (4096, 0)])
def test_segments_tile_the_periods(lib, span, last, period, most):
    per = ctypes.c_int()
    n = lib.layout(span, period, most, ctypes.byref(per))
    out = (ctypes.c_int * 2)()
    for here in (span, last):  # an ordinary split, the last one
        at = 0
        for j in range(n):
            lib.segment(span, period, most, j, here, out)
            first, length = out[0], out[1]
            if at == here:
                assert length == 0
                continue
            assert first == at and 0 < length <= most and first % 32 == 0
            assert first // period == (first + length - 1) // period
            assert (j // per.value == first // period) if period < span else per.value == n
            at += length
        assert at == here
