// f32tc_scan.cu -- second half of the fp32 tensor-core GEMM when the product
// has few output tiles and a long K: f32tc_kernel has left the product of
// every checksum segment of K in memory (all segments in parallel), and these
// kernels add them up.  With checksums one CTA walks the segments of one
// verification unit, a warp holding a 32 x 32 (16 x 16, 16 x 32) piece of it in
// registers; at the end of each period it injects the scheduled faults
// (Section 5.3), verifies, locates and corrects (Section 4.2.1) exactly as the
// one-pass kernel does.
//
// Bound: the chain of one period (copy, sums, barriers, comparison: 0.7 us
// with one warp a unit); units run side by side, and units of one warp walk
// shares of their periods side by side (f32tc_scan_groups_kernel).  256 x 256 x
// 65536 with 16 x 16 units: 50 us after 128 us for the segments; one pass over K
// kept 2 of 76 CTA pairs busy for 1780 us.
#include "f32tc.cuh"

namespace ftg {

// N values summed over the lanes of bit `o`, each side keeping half of them.
template <int N>
__device__ __forceinline__ void scan_fold(float* v, int lane, int o) {
  const bool up = lane & o;
#pragma unroll
  for (int e = 0; e < N / 2; ++e) {
    const float lo = v[e], hi = v[N / 2 + e];
    v[e] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
  }
}

// Row and column sums of the piece a warp holds (the layout of the kernels
// below): rowp[UR], colp[CW].
template <int UR, int CW>
__device__ __forceinline__ void scan_sums(const float* acc, int lane, float* rowp, float* colp) {
  constexpr int EPT = UR * CW / 32;
  float t[EPT];
#pragma unroll
  for (int i = 0; i < EPT; ++i) t[i] = acc[i];
  // rows: over the CW lanes of a row
  if constexpr (EPT == 32) {
    scan_fold<32>(t, lane, 16);
    scan_fold<16>(t, lane, 8);
    scan_fold<8>(t, lane, 4);
    scan_fold<4>(t, lane, 2);
    scan_fold<2>(t, lane, 1);
    rowp[lane] = t[0];
  } else if constexpr (EPT == 16) {
    scan_fold<16>(t, lane, 16);
    scan_fold<8>(t, lane, 8);
    scan_fold<4>(t, lane, 4);
    scan_fold<2>(t, lane, 2);
    t[0] += __shfl_xor_sync(0xffffffffu, t[0], 1);
    if (!(lane & 1)) rowp[lane >> 1] = t[0];
  } else {
    static_assert(EPT == 8 && CW == 16, "pieces: 32 x 32, 16 x 32, 16 x 16");
    scan_fold<8>(t, lane, 8);
    scan_fold<4>(t, lane, 4);
    scan_fold<2>(t, lane, 2);
    t[0] += __shfl_xor_sync(0xffffffffu, t[0], 1);
    if (!(lane & 1)) rowp[lane / CW + 2 * ((lane & 15) >> 1)] = t[0];
  }
  // columns: this lane's rows (both half-warps' of a 16-wide piece)
#pragma unroll
  for (int i = 0; i < EPT; ++i) t[i] = acc[i];
#pragma unroll
  for (int st = EPT / 2; st > 0; st >>= 1)
#pragma unroll
    for (int i = 0; i < st; ++i) t[i] += t[i + st];
  if constexpr (CW == 16) t[0] += __shfl_xor_sync(0xffffffffu, t[0], 16);
  if (lane < CW) colp[lane] = t[0];
}

struct ScanShared {
  float rowp[4][128], colp[4][128];  // partial sums per warp column / row of the unit
  double sum64[256];
  unsigned long long bestr, bestc;
  double fix_delta;
  float fro[2];
  int nr, nc, fix_row, fix_col, reset;
  float reset_value;
  float c[256];
  uint8_t flag[256];
};

// UR x CW: the piece of the unit a warp holds.  The segments ahead travel
// through a ring of `depth` (a power of two) in shared memory, each thread
// copying and reading its own elements (256 x 256 x 65536: 182 us against 211
// with one segment ahead in registers).
// WARP: one warp of a larger block runs the unit (nthr = 32), else the block.
template <int UR, int CW, bool WARP>
__device__ void scan_unit(const F32TcParams& p, int depth, ScanShared& X, float* ring, int tid, int nthr) {
  constexpr int EPT = UR * CW / 32, STEP = 32 / CW;
  auto sync = [] {
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
  };
  const int lane = tid & 31, warp = tid >> 5;
  const int wcols = p.un / CW, wr = warp / wcols, wc = warp - wr * wcols;
  const int I = blockIdx.x / p.nw, J = blockIdx.x - I * p.nw;
  const int row0 = I * p.um, col0 = J * p.un, ne = p.um + p.un;
  const int rsub = lane / CW, lc = wc * CW + lane % CW;  // rows wr * UR + rsub + STEP i, column lc of the unit
  auto lrow = [&](int i) { return wr * UR + rsub + STEP * i; };
  const bool col_ok = col0 + lc < p.N;

  if (tid < 2) {  // Frobenius norms of the unit's rows and columns
    const float* sq = (tid ? p.sq16b : p.sq16a) + (tid ? col0 : row0) / 16;
    const int cnt = min((tid ? p.un : p.um) / 16, ((tid ? p.N - col0 : p.M - row0) + 15) / 16);
    float s = 0.f;
    for (int g = 0; g < cnt; ++g) s += sq[g];
    X.fro[tid] = sqrtf(s);
  }
  if (tid == 0) X.reset = -1;
  sync();
  // this thread's checksum entries: rows 0 .. um - 1, then columns
  const float* dsrc[2];
  long long dstride[2];
  float c[2], tn[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = tid + q * nthr;
    c[q] = tn[q] = 0.f;
    dsrc[q] = p.Dr;  // not read where the stride is 0
    dstride[q] = 0;
    if (e < p.um) {
      if (row0 + e < p.M) {
        dsrc[q] = p.Dr + (long long)J * p.ldr_d + row0 + e;
        dstride[q] = (long long)p.nw * p.ldr_d;
        tn[q] = __fmul_rn(__fmul_rn(p.lam_u, p.nA[row0 + e]), X.fro[1]);
      }
    } else if (e < ne && col0 + e - p.um < p.N) {
      dsrc[q] = p.Dc + (long long)I * p.ldc_d + col0 + e - p.um;
      dstride[q] = (long long)p.nv * p.ldc_d;
      tn[q] = __fmul_rn(__fmul_rn(p.lam_u, X.fro[0]), p.nB[col0 + e - p.um]);
    }
  }
  // scheduled faults of the schedule tile that holds this unit
  const int tile_m = row0 / p.m_tb, tile_n = col0 / p.n_tb, tile = tile_m * p.tiles_n_sched + tile_n;
  const int f0 = p.nfaults > 0 ? first_fault(p.faults, p.nfaults, tile) : 0;
  const bool has_fault = f0 < p.nfaults && p.faults[f0].tile == tile;

  float acc[EPT];
#pragma unroll
  for (int i = 0; i < EPT; ++i) acc[i] = 0.f;
  const float* src = p.P + (long long)row0 * p.ldp + col0 + lc;
  const int segs = p.sg.per_split;
  unsigned ok_rows = 0u;  // bit i: row lrow(i) of this lane's column is inside the matrix
#pragma unroll
  for (int i = 0; i < EPT; ++i) ok_rows |= (col_ok && row0 + lrow(i) < p.M ? 1u : 0u) << i;
  const float* next = src + (long long)lrow(0) * p.ldp;  // of the segment to fetch
  const long long row_step = (long long)STEP * p.ldp, seg_step = (long long)p.M * p.ldp;
  const uint32_t ring0 = (uint32_t)__cvta_generic_to_shared(ring + tid), line = 4u * nthr, slot = (EPT + 2) * line;
  int fetched = 0;
  // 4 bytes, or zeros where `in` is 0 (nothing is read then)
  auto copy = [](uint32_t dst, const float* from, int in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(from), "r"(in) : "memory");
  };
  auto fetch = [&]() {  // one copy group per segment, empty past the last
    if (fetched < segs) {
      uint32_t d = ring0 + (fetched & (depth - 1)) * slot;
      const float* from = next;
#pragma unroll
      for (int i = 0; i < EPT; ++i, d += line, from += row_step) {
        const int in = (ok_rows >> i & 1u) * 4;
        copy(d, in ? from : p.P, in);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q, d += line) copy(d, dsrc[q], dstride[q] ? 4 : 0);
      next += seg_step;
#pragma unroll
      for (int q = 0; q < 2; ++q) dsrc[q] += dstride[q];
    }
    ++fetched;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int g = 0; g < depth - 1; ++g) fetch();
  int left = p.sg.per_period;  // segments to the end of the period
  for (int seg = 0, period = 0; seg < segs; ++seg) {
    // segment `seg` has landed: all but the depth - 2 newest groups
    if (depth == 4) asm volatile("cp.async.wait_group 2;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    {
      const float* d = ring + (seg & (depth - 1)) * (EPT + 2) * nthr + tid;
#pragma unroll
      for (int i = 0; i < EPT; ++i) acc[i] += d[i * nthr];
#pragma unroll
      for (int q = 0; q < 2; ++q) c[q] += d[(EPT + q) * nthr];
    }
    fetch();  // into the slot read one segment ago
    if (--left > 0 && seg + 1 < segs) continue;
    left = p.sg.per_period;
    const int ks_first = period * p.cadence, ks = min((period + 1) * p.cadence, p.ksteps) - 1;
    ++period;
    if (has_fault) {
      for (int f = f0; f < p.nfaults && p.faults[f].tile == tile; ++f) {
        const Fault F = p.faults[f];
        const int fr = tile_m * p.m_tb + F.row - row0, fc = tile_n * p.n_tb + F.col - col0;
        if (F.kstep < ks_first || F.kstep > ks || fr < 0 || fr >= p.um || fc < 0 || fc >= p.un) continue;
        if (F.target == T_ACC) {
#pragma unroll
          for (int i = 0; i < EPT; ++i)
            if (lrow(i) == fr && lc == fc) acc[i] += F.delta;
        } else {
          const int e = F.target == T_ROWSUM ? fr : p.um + fc;
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if (e == tid + q * nthr) c[q] += F.delta;
        }
      }
    }
    // ----- verification -----
    scan_sums<UR, CW>(acc, lane, X.rowp[wc] + wr * UR, X.colp[wr] + wc * CW);
    sync();
    const float grow = __fmul_rn(p.mu_u, sqrtf((float)min((ks + 1) * p.k_tb, p.K)));
    unsigned flags = 0u;
    float tau[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + q * nthr;
      tau[q] = __fmaf_rn(grow, fabsf(c[q]), tn[q]);
      if (e >= ne) continue;
      float s = 0.f;
      if (e < p.um) for (int w = 0; w < wcols; ++w) s += X.rowp[w][e];
      else for (int w = 0; w < p.um / UR; ++w) s += X.colp[w][e - p.um];
      if (fabsf(s - c[q]) > kScreen * tau[q]) flags |= 1u << q;
    }
    bool any;
    if constexpr (WARP) any = __any_sync(0xffffffffu, flags != 0u);
    else any = __syncthreads_or(flags != 0u);
    if (!any) {
      if constexpr (WARP) __syncwarp();
      continue;
    }
    // ----- fp64 confirmation of the screened entries -----
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + q * nthr;
      if (e >= ne) continue;
      X.flag[e] = (flags >> q) & 1u;
      X.sum64[e] = 0.0;
      X.c[e] = c[q];
    }
    if (tid == 0) {
      X.nr = 0; X.nc = 0; X.bestr = 0ull; X.bestc = 0ull; X.fix_row = -1; X.reset = -1;
    }
    sync();
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      if (X.flag[lrow(i)]) atomicAdd(&X.sum64[lrow(i)], (double)acc[i]);
      if (X.flag[p.um + lc]) atomicAdd(&X.sum64[p.um + lc], (double)acc[i]);
    }
    sync();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + q * nthr;
      if (!((flags >> q) & 1u)) continue;
      const double d = X.sum64[e] - (double)c[q];
      if (!(fabs(d) > (double)tau[q])) continue;
      const float sc = flag_score((float)d, tau[q]);
      if (e < p.um) {
        atomicAdd(&X.nr, 1);
        atomicMax(&X.bestr, flag_key(sc, e));
      } else {
        atomicAdd(&X.nc, 1);
        atomicMax(&X.bestc, flag_key(sc, e - p.um));
      }
    }
    sync();
    if (tid == 0 && (X.nr | X.nc)) {
      const int nr = X.nr, nc = X.nc;
      const int ir = nr ? key_index(X.bestr) : -1, jc = nc ? key_index(X.bestc) : -1, ec = p.um + jc;
      const double dR = nr ? X.sum64[ir] - (double)X.c[ir] : 0.0, dC = nc ? X.sum64[ec] - (double)X.c[ec] : 0.0;
      const float tR = nr ? __fmaf_rn(grow, fabsf(X.c[ir]), __fmul_rn(__fmul_rn(p.lam_u, p.nA[row0 + ir]), X.fro[1])) : 0.f;
      const float tC = nc ? __fmaf_rn(grow, fabsf(X.c[ec]), __fmul_rn(__fmul_rn(p.lam_u, X.fro[0]), p.nB[col0 + jc])) : 0.f;
      ftgemm_fault_record rec;
      rec.tile_m = tile_m; rec.tile_n = tile_n; rec.kstep = ks;
      rec.problem = 0; rec.reserved = 0;
      rec.row = nr ? row0 + ir : -1;
      rec.col = nc ? col0 + jc : -1;
      rec.residual_r = dR; rec.residual_c = dC; rec.tau = (double)tR + (double)tC;
      rec.delta = 0.0;
      if (nr == 1 && nc == 1) {
        if (fabs(dR - dC) <= (double)tR + (double)tC) {
          rec.kind = K_CORRECTED; rec.delta = dR;
          X.fix_row = ir; X.fix_col = jc; X.fix_delta = dR;
        } else {
          rec.kind = K_UNCORRECTABLE;
        }
      } else if (nr == 1 && nc == 0) {
        rec.kind = K_CHECKSUM; rec.delta = -dR; X.reset = ir; X.reset_value = (float)X.sum64[ir];
      } else if (nr == 0 && nc == 1) {
        rec.kind = K_CHECKSUM; rec.delta = -dC; X.reset = ec; X.reset_value = (float)X.sum64[ec];
      } else {
        rec.kind = K_UNCORRECTABLE;
      }
      report_event(p.rep, p.recs, rec);
    }
    sync();
    // ----- correct the located element, or reset the checksum -----
#pragma unroll
    for (int i = 0; i < EPT; ++i)
      if (lrow(i) == X.fix_row && lc == X.fix_col) acc[i] = (float)((double)acc[i] - X.fix_delta);
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (tid + q * nthr == X.reset) c[q] = X.reset_value;
    sync();  // the shared state is reused
  }
  if (!col_ok) return;
  float* out = p.C + (long long)row0 * p.ldc + col0 + lc;
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    if (row0 + lrow(i) >= p.M) continue;
    float* d = out + (long long)lrow(i) * p.ldc;
    const float v = p.alpha * acc[i];
    *d = p.beta != 0.f ? fmaf(p.beta, *d, v) : v;
  }
}

template <int UR, int CW>
__global__ void __launch_bounds__(512) f32tc_scan_kernel(const __grid_constant__ F32TcParams p, int depth) {
  if (*p.bad == p.epoch) return;
  extern __shared__ float ring[];  // [depth][UR * CW / 32 + 2][threads]
  __shared__ ScanShared X;
  scan_unit<UR, CW, false>(p, depth, X, ring, threadIdx.x, blockDim.x);
}

// Units of one warp and many periods: a block per unit, SCAN_GROUPS warps with
// a share of the periods each.  A warp first adds up its segments, then starts
// from the sums of the shares before its own and walks its periods again,
// screening each as scan_unit does; the segments come from L2 the second time.
// Where a fault is scheduled, or anything was flagged (nothing has been written
// then), one warp runs the unit from the start, period by period.
// Bound: the chain of one period, SCAN_GROUPS of them side by side.  One warp a
// unit / this, us: 256 x 256 x 65536 with 16 x 16 units 182 / 50, with 32 x 32
// 306 / 92; 384 x 384 x 16384 (32 x 32) 82 / 30; at 16 periods 512 x 512 x 4096
// (16 x 16) 16 / 17, 640 x 384 x 4096 (32 x 32) 24 / 19.
constexpr int SCAN_GROUPS = 8;
template <int UR, int CW>
__global__ void __launch_bounds__(32 * SCAN_GROUPS) f32tc_scan_groups_kernel(const __grid_constant__ F32TcParams p, int depth) {
  if (*p.bad == p.epoch) return;
  constexpr int EPT = UR * CW / 32, STEP = 32 / CW, G = SCAN_GROUPS, NV = EPT + 2;
  extern __shared__ float ring[];  // [depth][NV][32]
  __shared__ ScanShared X;
  __shared__ float pre[G - 1][NV][32], rowp[G][UR], colp[G][CW];
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
  const int I = blockIdx.x / p.nw, J = blockIdx.x - I * p.nw, row0 = I * UR, col0 = J * CW;
  const int lc = lane % CW;
  auto lrow = [&](int i) { return lane / CW + STEP * i; };
  const bool col_ok = col0 + lc < p.N;
  if (tid < 2) {  // Frobenius norms of the unit's rows and columns
    const float* sq = (tid ? p.sq16b : p.sq16a) + (tid ? col0 : row0) / 16;
    const int cnt = min((tid ? CW : UR) / 16, ((tid ? p.N - col0 : p.M - row0) + 15) / 16);
    float s = 0.f;
    for (int i = 0; i < cnt; ++i) s += sq[i];
    X.fro[tid] = sqrtf(s);
  }
  __syncthreads();
  // this lane's checksum entries: rows 0 .. UR - 1, then columns
  const float* dsrc[2];
  long long dstride[2];
  float tn[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = lane + 32 * q;
    tn[q] = 0.f;
    dsrc[q] = nullptr;
    dstride[q] = 0;
    if (e < UR) {
      if (row0 + e < p.M) {
        dsrc[q] = p.Dr + (long long)J * p.ldr_d + row0 + e;
        dstride[q] = (long long)p.nw * p.ldr_d;
        tn[q] = __fmul_rn(__fmul_rn(p.lam_u, p.nA[row0 + e]), X.fro[1]);
      }
    } else if (e < UR + CW && col0 + e - UR < p.N) {
      dsrc[q] = p.Dc + (long long)I * p.ldc_d + col0 + e - UR;
      dstride[q] = (long long)p.nv * p.ldc_d;
      tn[q] = __fmul_rn(__fmul_rn(p.lam_u, X.fro[0]), p.nB[col0 + e - UR]);
    }
  }
  const int tile = row0 / p.m_tb * p.tiles_n_sched + col0 / p.n_tb;
  const int f0 = p.nfaults > 0 ? first_fault(p.faults, p.nfaults, tile) : 0;
  if (f0 < p.nfaults && p.faults[f0].tile == tile) {
    if (g == 0) scan_unit<UR, CW, true>(p, depth, X, ring, lane, 32);
    return;
  }
  bool redo = false;

  // this warp's periods and segments
  const int segs = p.sg.per_split, spp = p.sg.per_period;
  const int share = ((segs + spp - 1) / spp + G - 1) / G;
  const int s0 = min((long long)segs, (long long)g * share * spp), s1 = min((long long)segs, (long long)(g + 1) * share * spp);
  const float* src = p.P + (long long)row0 * p.ldp + col0 + lc;
  const long long seg_step = (long long)p.M * p.ldp;
  auto load = [&](int seg, float* v) {
#pragma unroll
    for (int i = 0; i < EPT; ++i)
      v[i] = col_ok && row0 + lrow(i) < p.M ? __ldg(src + seg * seg_step + lrow(i) * p.ldp) : 0.f;
#pragma unroll
    for (int q = 0; q < 2; ++q) v[EPT + q] = dsrc[q] ? __ldg(dsrc[q] + seg * dstride[q]) : 0.f;
  };
  float acc[NV], v[NV];  // the piece, then this lane's checksums
#pragma unroll
  for (int i = 0; i < NV; ++i) acc[i] = 0.f;
  if (g < G - 1) {
#pragma unroll 4
    for (int seg = s0; seg < s1; ++seg) {
      load(seg, v);
#pragma unroll
      for (int i = 0; i < NV; ++i) acc[i] += v[i];
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      pre[g][i][lane] = acc[i];
      acc[i] = 0.f;
    }
  }
  if (s0 < s1) load(s0, v);
  __syncthreads();
  for (int h = 0; h < g; ++h)
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] += pre[h][i][lane];
  for (int seg = s0, left = spp, period = g * share; seg < s1; ++seg) {
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] += v[i];
    if (seg + 1 < s1) load(seg + 1, v);
    if (--left > 0 && seg + 1 < segs) continue;
    left = spp;
    const int ks = min((period + 1) * p.cadence, p.ksteps) - 1;
    ++period;
    scan_sums<UR, CW>(acc, lane, rowp[g], colp[g]);
    __syncwarp();
    const float grow = __fmul_rn(p.mu_u, sqrtf((float)min((ks + 1) * p.k_tb, p.K)));
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = lane + 32 * q;
      if (e >= UR + CW) continue;
      const float c = acc[EPT + q], sum = e < UR ? rowp[g][e] : colp[g][e - UR];
      redo |= fabsf(sum - c) > kScreen * __fmaf_rn(grow, fabsf(c), tn[q]);
    }
    __syncwarp();
  }
  if (__syncthreads_or(redo)) {
    if (g == 0) scan_unit<UR, CW, true>(p, depth, X, ring, lane, 32);
    return;
  }
  if (s0 >= s1 || s1 < segs || !col_ok) return;  // the last share's warp holds the result
  float* out = p.C + (long long)row0 * p.ldc + col0 + lc;
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    if (row0 + lrow(i) >= p.M) continue;
    float* d = out + (long long)lrow(i) * p.ldc;
    const float o = p.alpha * acc[i];
    *d = p.beta != 0.f ? fmaf(p.beta, *d, o) : o;
  }
}

// Without checksums: C = alpha * (sum of the segments) + beta * C, after the
// scheduled faults (each on one accumulator).
__global__ void __launch_bounds__(256) f32tc_sum_kernel(const __grid_constant__ F32TcParams p) {
  if (*p.bad == p.epoch) return;
  const long long idx = (long long)blockIdx.x * 256 + threadIdx.x;
  if (idx >= (long long)p.M * p.N) return;
  const int r = (int)(idx / p.N), c = (int)(idx - (long long)r * p.N);
  const float* s = p.P + (long long)r * p.ldp + c;
  float v = 0.f;
#pragma unroll 8
  for (int g = 0; g < p.sg.per_split; ++g) v += __ldg(s + (long long)g * p.M * p.ldp);
  if (p.nfaults > 0) {
    const int tile = r / p.m_tb * p.tiles_n_sched + c / p.n_tb;
    for (int f = first_fault(p.faults, p.nfaults, tile); f < p.nfaults && p.faults[f].tile == tile; ++f)
      if (p.faults[f].row == r % p.m_tb && p.faults[f].col == c % p.n_tb) v += p.faults[f].delta;
  }
  float* d = p.C + (long long)r * p.ldc + c;
  const float o = p.alpha * v;
  *d = p.beta != 0.f ? fmaf(p.beta, *d, o) : o;
}

// Units a warp's pieces tile; others keep the one-pass kernel.
bool f32tc_scan_units(int um, int un) {
  return (um == 16 && un >= 16 && un <= 128) || (um >= 32 && un >= 32 && um <= 128 && un <= 128);
}

// Units of one warp, few enough that one warp each leaves the GPU idle, with
// enough periods for shares.  One warp a unit / shares, us: 512 x 512 x 8192 with
// 32 x 32 units 45 / 31, with 16 x 16 29 / 25; but 640 x 640 x 4096 (32 x 32) 26 /
// 36, 1024 x 512 x 4096 (16 x 16) 19 / 32, 1024 x 1024 x 8192 (32 x 32) 57 / 112.
bool f32tc_scan_groups(int M, int N, int um, int un, int periods) {
  return um <= 32 && un <= 32 && (long long)M * N <= 1 << 18 && periods >= 2 * SCAN_GROUPS;
}

cudaError_t launch_f32tc_scan(bool abft, const F32TcParams& p, int* launches, cudaStream_t st) {
  ++*launches;
  if (!abft) {
    f32tc_sum_kernel<<<(unsigned)(((long long)p.M * p.N + 255) / 256), 256, 0, st>>>(p);
    return cudaGetLastError();
  }
  if (!f32tc_scan_units(p.um, p.un)) return cudaErrorInvalidValue;
  const unsigned units = (unsigned)(p.nv * p.nw);
  const int ur = p.um < 32 ? p.um : 32, cw = p.un < 32 ? p.un : 32, threads = p.um / ur * (p.un / cw) * 32;
  const int depth = p.um * p.un <= 4096 ? 4 : 2;
  const size_t smem = sizeof(float) * depth * (ur * cw / 32 + 2) * threads;  // at most 139,264 bytes (128 x 128)
  auto go = [&](auto* k, int block) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // an ordinary launch: scheduled while the GEMM kernel drains, the small
    // blocks gather on the SMs that are free first (253 us against 182 for
    // 256 x 256 x 65536 with one warp a unit)
    k<<<units, block, smem, st>>>(p, depth);
    return cudaGetLastError();
  };
  if (f32tc_scan_groups(p.M, p.N, p.um, p.un, (p.sg.per_split + p.sg.per_period - 1) / p.sg.per_period)) {
    if (ur == 32) return go(f32tc_scan_groups_kernel<32, 32>, 32 * SCAN_GROUPS);
    if (cw == 32) return go(f32tc_scan_groups_kernel<16, 32>, 32 * SCAN_GROUPS);
    return go(f32tc_scan_groups_kernel<16, 16>, 32 * SCAN_GROUPS);
  }
  if (ur == 32) return go(f32tc_scan_kernel<32, 32>, threads);
  if (cw == 32) return go(f32tc_scan_kernel<16, 32>, threads);
  return go(f32tc_scan_kernel<16, 16>, threads);
}

}  // namespace ftg
