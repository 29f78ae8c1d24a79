// f32tc.cuh -- fp32 GEMM with online ABFT on the tensor cores: types shared
// by its encode pass (f32tc_prep.cu), its kernel (f32tc_gemm.cu) and api.cu.
//
// An fp32 value x is the exact sum of three bf16 values,
//   x1 = bf16(x), x2 = bf16(x - x1), x3 = bf16(x - x1 - x2),
// as long as 2^-100 <= |x| < 2^60 or x = 0 (8 bits each; the remainders are
// exact in fp32).  A product a*b is then the sum of nine bf16 products, each
// exact in the fp32 tensor-core accumulation; the three smallest (a2 b3,
// a3 b2, a3 b3: together below 2^-25 |a b|) are left out, half an ulp of one
// fp32 product rounding.  The other six run as bf16 MMAs.
//
// The tensor-core accumulation truncates (a chunk's sum of one sign comes out
// 0.7 to 1 u too small, u = 2^-24), so it only ever runs over F32TC_KC elements
// of K, and a product of fewer stays on the CUDA cores.  Each chunk's products
// are summed in tensor memory in order of size, smallest first, and the chunk's
// result is added to an fp32 accumulator in registers with round-to-nearest.
// The registers are the accumulators the ABFT scheme protects: faults are added
// there, and every verification period the unit's row and column sums are formed
// from them.
#pragma once
#include "f32tc_seg.cuh"
#include "internal.cuh"

namespace ftg {

constexpr int F32TC_KC = 32;    // elements of K per pipeline stage and per tensor-core accumulation
constexpr int F32TC_BM = 128;   // rows of C per CTA (a CTA pair: 256)
constexpr int F32TC_SEG = 256;  // elements of K per checksum segment (f32tc_plan: or one period, if that is no multiple of it)

// Planes in memory: row operands (A, e^T A, (B e)^T) as blocks of 128 rows x
// 32 elements of K, three planes of 128 64-byte rows each, the 16-byte units
// of row r permuted by (r / 2) % 4 (the 64-byte swizzle); the column operand B
// as blocks of 32 elements of K x 64 columns, three planes of 32 128-byte rows,
// the units of row k permuted by k % 8 (the 128-byte swizzle).  Blocks run
// along K first.  Rows, columns and elements of K past the matrix are zero in
// A and B; rows past the last unit are undefined in the checksum planes (they
// only reach results that are not stored).
constexpr int F32TC_APLANE = 128 * F32TC_KC, F32TC_BPLANE = 64 * F32TC_KC;  // elements of a block's plane

struct F32TcParams {
  int M, N, K;
  int tiles_m2, tiles_n;       // CTA-pair tile rows (2 * F32TC_BM each), tile columns
  int group_m;                 // pair tile rows per raster group
  // MAIN: tiles of the launch; half_first > 0: tiles of 256 columns from that
  // one on, in halves of 128 (what the 256-column launch before it leaves over)
  int tiles, half_first;
  int nsplit, k_per_split;     // splits of K and their length in elements
  F32TcSegs sg;
  // verification units and the schedule's tiling (what records and faults refer to)
  int um, un;                  // unit rows / columns (powers of two, 16 .. 128)
  int nv, nw;                  // units along M and N
  int m_tb, n_tb, k_tb, tiles_n_sched, ks_per_split, cadence, ksteps;
  float* nA; float* nB;        // row norms of A, column norms of B
  float* sq16a; float* sq16b;  // sums of squares of every 16 rows of A / columns of B
  // what the SUMS launch forms them from: squared-norm partials
  // [ceil(K / 128)][M] and [ceil(K / 128)][N], or null (no checksums)
  const float* pa; const float* pb;
  float* Dc; float* Dr;        // checksum segments: [seg][nv][ldc_d] and [seg][nw][ldr_d]
  long long ldc_d, ldr_d;
  // the product itself by segments, [seg][M][ldp] (f32tc_scan.cu adds them
  // up; one split), or null: one pass over K per tile
  float* P; long long ldp;
  float lam_u, mu_u;
  float* C; long long ldc; int c_vec;
  float alpha, beta;
  float* partial;              // [split][M][N], or null
  const Fault* faults; int nfaults;
  DevReport* rep; ftgemm_fault_record* recs;
  // the encode pass sets *bad (the handle's own word) to `epoch`, the call's own
  // number, when an operand is outside the split's range: nothing to clear before
  // a call, except in a graph, whose replays share one number (launch_f32tc_split)
  const int* bad; int epoch;
};

// The encode pass: operand planes, and (um > 0) checksum vectors and squared-norm
// partials (the SUMS launch forms the norms from them).
struct F32TcPrep {
  int M, N, K;
  int um, un, nv, nw;
  uint16_t* Ap;                 // planes of A: [ceil(M / 128)][chunks][3][F32TC_APLANE]
  uint16_t* Bp;                 // planes of B: [2 * ceil(N / 128)][chunks][3][F32TC_BPLANE]
  float* V; float* W; long long ldv;  // e^T A [nv][ldv], B e [nw][ldv] (ldv a multiple of 8)
  uint16_t* Vp; uint16_t* Wp;   // their planes, as A's
  float* pa; float* pb;         // squared-norm partials [ceil(K / 128)][M], [ceil(K / 128)][N]
  float* nA; float* nB; float* sq16a; float* sq16b;
  int* bad; int epoch;
};

// 2-D maps over the planes as rows of 128 bytes, no swizzle (the planes are
// stored swizzled).
struct F32TcMaps {
  CUtensorMap A, V, W;  // row operands: box of one block (192 rows)
  CUtensorMap B;        // column operand: box of one block (96 rows)
  CUtensorMap An;       // A as the column operand: box of 64 rows of one plane (32 rows)
};

}  // namespace ftg
