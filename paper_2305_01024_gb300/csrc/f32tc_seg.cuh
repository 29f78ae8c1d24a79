// f32tc_seg.cuh -- how the fp32 tensor-core GEMM cuts K into checksum segments
// (plain C++ as well, for tests on the host).
//
// A split of K is `span` elements and is verified every `period` of them (a
// multiple of 32, or the whole split).  Every period is cut on its own into
// segments of `seg` elements, its last one shorter where the period is no
// multiple of it, so that a period is always whole segments.
#pragma once

#ifdef __CUDACC__
#define F32TC_HD __host__ __device__ __forceinline__
#else
#define F32TC_HD inline
#endif

namespace ftg {

struct F32TcSegs {
  int period, seg;            // elements of K
  int per_period, per_split;  // segments
  int uneven;                 // a period's last segment is shorter than the others (and more periods follow)
};

// Segments of at most `most` elements (a multiple of 32).
F32TC_HD F32TcSegs f32tc_segs(int span, int period, int most) {
  F32TcSegs t;
  t.period = period < span ? period : span;
  t.seg = most < period ? most : period;
  t.per_period = (t.period + t.seg - 1) / t.seg;
  const int whole = span / t.period, rest = span - whole * t.period;
  t.per_split = whole * t.per_period + (rest + t.seg - 1) / t.seg;
  t.uneven = t.period < span && t.period % t.seg != 0;
  return t;
}

// Segment j of a split: its first element, counted from the split's, and its
// length; 0 where the split holds `here` elements only (the last one).
F32TC_HD void f32tc_segment(const F32TcSegs& t, int j, int here, int* first, int* len) {
  int at = j * t.seg, end = here;
  if (t.uneven) {  // (its division in every item took 1 % of 256 x 256 x 65536 in the thread that issues the MMAs)
    const int p = j / t.per_period, p0 = p * t.period;
    at = p0 + (j - p * t.per_period) * t.seg;
    end = here - p0 < t.period ? here : p0 + t.period;
  }
  const int left = end - at;
  *first = at;
  *len = left < 0 ? 0 : left < t.seg ? left : t.seg;
}

}  // namespace ftg
