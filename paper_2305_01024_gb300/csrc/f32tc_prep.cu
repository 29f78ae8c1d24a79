// f32tc_prep.cu -- encode pass of the fp32 GEMM on the tensor cores: the
// three bf16 planes of A and B (f32tc.cuh), the checksum vectors e^T A per
// row unit and B e per column unit (Eq. 1-2) in fp32 and as planes, and the
// partials of the norms that scale the detection threshold.  Each operand is
// read once.
//
// The planes are written in the order the GEMM kernel reads them: every
// (128-row tile, 32-element chunk of K) of A, and every (64-column tile,
// chunk) of B, is one contiguous block holding its three planes as the
// swizzled shared-memory image the MMA descriptors name, so a TMA load moves
// whole 128-byte lines in sequence.  (Planes kept row-major, loaded as
// 64-byte rows of a 3-D box, held the kernel to 144 TFLOP/s at 8192^3: the
// loads, not the MMAs, set its pace.)
//
// Bound: HBM.  Per element 4 bytes are read and 6 written; a warp reads 8
// rows x 128 bytes of A (4 rows x 256 bytes of B) and writes 512 contiguous
// bytes per plane, four such cells in flight.
#include <cuda_bf16.h>

#include "f32tc.cuh"
#include "ptx.cuh"

namespace ftg {

// The largest and smallest magnitudes the split represents exactly (and whose
// sums cannot overflow): biased exponents 27 (2^-100) .. 186 (2^59); zero too.
__device__ __forceinline__ bool f32tc_outside(float x) {
  const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
  return u != 0u && u - (27u << 23) >= (160u << 23);
}

// Planes of two values, packed pairwise: x = p[0] + p[1] + p[2] exactly.
__device__ __forceinline__ void split2(float x0, float x1, uint32_t p[3]) {
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    p[s] = *reinterpret_cast<const uint32_t*>(&h);
    x0 -= __uint_as_float(p[s] << 16);
    x1 -= __uint_as_float(p[s] & 0xffff0000u);
  }
}

// Eight values as one 16-byte unit of each plane
__device__ __forceinline__ void store_planes8(uint16_t* dst, long long plane, const float* x) {
  uint32_t w[4][3];
#pragma unroll
  for (int i = 0; i < 4; ++i) split2(x[2 * i], x[2 * i + 1], w[i]);
#pragma unroll
  for (int s = 0; s < 3; ++s)
    *reinterpret_cast<uint4*>(dst + s * plane) = make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
}

// elements c .. c + 7 of a row (zero past `cols`)
__device__ __forceinline__ void load8(const float* row, int c, int cols, bool vec, float* x) {
  if (vec && c + 7 < cols) {
    const float4 u = __ldg(reinterpret_cast<const float4*>(row + c)), v = __ldg(reinterpret_cast<const float4*>(row + c) + 1);
    x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w;
    x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = c + e < cols ? __ldg(row + c + e) : 0.f;
  }
}

// Element offset of the 16-byte unit holding k .. k + 7 (k a multiple of 8)
// of row r, plane 0, in row-operand planes of nch chunks per 128-row tile.
__device__ __forceinline__ long long row_unit(int r, int k, int nch) {
  const int rl = r & 127, c = (k & 31) >> 3;
  return ((long long)(r >> 7) * nch + (k >> 5)) * (3 * F32TC_APLANE) + rl * 32 + ((c ^ ((rl >> 1) & 3)) << 3);
}

// One block: 128 rows x 128 elements of K of A (the first a_blocks blocks),
// or 128 columns x 128 elements of K of B; warp w takes chunk w % 4 and half
// w / 4 of the rows (columns).  With units (um > 0): V[u][k], the sum of the
// rows of unit u, W[u][k], the sum of the columns, both in fp32 and as row
// planes, and the squared-norm partials of every 128 elements of K.
__global__ void __launch_bounds__(256) f32tc_split_kernel(const float* __restrict__ A, long long lda,
                                                          const float* __restrict__ B, long long ldb,
                                                          const F32TcPrep e, int veca, int vecb, int a_blocks) {
  __shared__ __align__(16) float usum[8][128];  // unit sums per element of K (units of 128: two halves)
  __shared__ float sq4[4][128];                 // squared norms per chunk
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool side_a = (int)blockIdx.x < a_blocks;
  const int blk = side_a ? blockIdx.x : blockIdx.x - a_blocks;
  const int kgroups = (e.K + 127) / 128;
  const int kb = blk % kgroups, tile = blk / kgroups;
  const int ch = warp & 3, half = warp >> 2, chunk = kb * 4 + ch, nch = (e.K + 31) / 32;
  const int us = side_a ? e.um : e.un;
  bool out = false;
  if (chunk < nch) {
    if (side_a) {
      const int lr = lane >> 2, k = chunk * 32 + (lane & 3) * 8;
      float cs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int g4 = 0; g4 < 8; g4 += 4) {
        float x[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = tile * 128 + half * 64 + (g4 + i) * 8 + lr;
          load8(A + (long long)min(r, e.M - 1) * lda, k, r < e.M ? e.K : 0, veca, x[i]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int g = g4 + i, rl = half * 64 + g * 8 + lr;
          store_planes8(e.Ap + row_unit(tile * 128 + rl, k, nch), F32TC_APLANE, x[i]);
          float sq = 0.f;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            out |= f32tc_outside(x[i][j]);
            cs[j] += x[i][j];
            sq = fmaf(x[i][j], x[i][j], sq);
          }
          if (us) {
            sq += __shfl_xor_sync(0xffffffffu, sq, 1);
            sq += __shfl_xor_sync(0xffffffffu, sq, 2);
            if ((lane & 3) == 0) sq4[ch][rl] = sq;
            if (((g + 1) * 8) % min(us, 64) == 0) {  // a unit's rows (or this half of them) are complete
#pragma unroll
              for (int j = 0; j < 8; ++j) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) cs[j] += __shfl_xor_sync(0xffffffffu, cs[j], o);
              }
              if (lane < 4) {
                float* d = &usum[(half * 64 + g * 8) / min(us, 64)][ch * 32 + lane * 8];
                *reinterpret_cast<float4*>(d) = make_float4(cs[0], cs[1], cs[2], cs[3]);
                *reinterpret_cast<float4*>(d + 4) = make_float4(cs[4], cs[5], cs[6], cs[7]);
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) cs[j] = 0.f;
            }
          }
        }
      }
    } else {
      const int lk = lane >> 3, c = lane & 7, n = tile * 128 + half * 64 + c * 8;
      const long long base = ((long long)(tile * 2 + half) * nch + chunk) * (3 * F32TC_BPLANE);
      float sq[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int g4 = 0; g4 < 8; g4 += 4) {
        float x[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = chunk * 32 + (g4 + i) * 4 + lk;
          load8(B + (long long)min(k, e.K - 1) * ldb, n, k < e.K ? e.N : 0, vecb, x[i]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int kl = (g4 + i) * 4 + lk;
          store_planes8(e.Bp + base + kl * 64 + ((c ^ (kl & 7)) << 3), F32TC_BPLANE, x[i]);
          float s = 0.f;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            out |= f32tc_outside(x[i][j]);
            s += x[i][j];
            sq[j] = fmaf(x[i][j], x[i][j], sq[j]);
          }
          if (us) {
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            if (us > 16) s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (us > 32) s += __shfl_xor_sync(0xffffffffu, s, 4);
            const int u = min(us, 64);
            if ((c * 8) % u == 0) usum[(half * 64 + c * 8) / u][ch * 32 + kl] = s;
          }
        }
      }
      if (us) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          sq[j] += __shfl_xor_sync(0xffffffffu, sq[j], 8);
          sq[j] += __shfl_xor_sync(0xffffffffu, sq[j], 16);
          if (lane < 8) sq4[ch][half * 64 + c * 8 + j] = sq[j];
        }
      }
    }
  }
  if (__any_sync(0xffffffffu, out) && lane == 0) *e.bad = e.epoch;
  if (!us) return;
  __syncthreads();
  const int chunks = min(4, nch - kb * 4);
  if (threadIdx.x < 128) {
    const int line = tile * 128 + threadIdx.x, L = side_a ? e.M : e.N;
    float s = 0.f;
    for (int c = 0; c < chunks; ++c) s += sq4[c][threadIdx.x];
    if (line < L) (side_a ? e.pa : e.pb)[(long long)kb * L + line] = s;
  }
  // the units' sums, eight elements of K per thread
  const int nu = side_a ? e.nv : e.nw;
  float* S = side_a ? e.V : e.W;
  uint16_t* P = side_a ? e.Vp : e.Wp;
  const int t = threadIdx.x, u = t >> 4, k = kb * 128 + (t & 15) * 8, unit = tile * (128 / us) + u;
  if (u >= 128 / us || unit >= nu || k >= nch * 32) return;
  float s[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    s[j] = usum[u][(t & 15) * 8 + j];
    if (us == 128) s[j] += usum[1][(t & 15) * 8 + j];
  }
  if (k < e.K) {
    float4* d = reinterpret_cast<float4*>(S + (long long)unit * e.ldv + k);
    d[0] = make_float4(s[0], s[1], s[2], s[3]);
    d[1] = make_float4(s[4], s[5], s[6], s[7]);
  }
  store_planes8(P + row_unit(unit, k, nch), F32TC_APLANE, s);
}

__global__ void f32tc_clear_kernel(int* bad) { *bad = 0; }

// captured: the launches go into a graph.  Its replays all carry the epoch of
// the capture, so each clears the flag first: what one replay's operands held
// does not send the next one to the CUDA cores.
cudaError_t launch_f32tc_split(const float* A, long long lda, const float* B, long long ldb, const F32TcPrep& e,
                               bool captured, int* launches, cudaStream_t st) {
  const int veca = lda % 4 == 0 && ((uintptr_t)A & 15) == 0, vecb = ldb % 4 == 0 && ((uintptr_t)B & 15) == 0;
  const int kgroups = (e.K + 127) / 128;
  const long long ab = (long long)kgroups * ((e.M + 127) / 128), bb = (long long)kgroups * ((e.N + 127) / 128);
  if (ab + bb > 0x7fffffff) return cudaErrorInvalidValue;
  cudaError_t er = cudaSuccess;
  if (captured) {
    f32tc_clear_kernel<<<1, 1, 0, st>>>(e.bad);
    er = cudaGetLastError();
    if (er != cudaSuccess) return er;
    *launches += 1;
  }
  er = launch_pdl(f32tc_split_kernel, (unsigned)(ab + bb), 256, 0, st, A, lda, B, ldb, e, veca, vecb, (int)ab);
  *launches += 1;
  return er;
}

}  // namespace ftg
