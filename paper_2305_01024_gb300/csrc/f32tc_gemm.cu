// f32tc_gemm.cu -- fp32 GEMM with online block- and warp-level ABFT on the
// tensor cores (f32tc.cuh gives the arithmetic: three exact bf16 planes per
// operand, six bf16 MMAs per product, fp32 accumulation in registers).
//
// A 2-CTA cluster computes a 256 x BN tile of C with cta_group::2 MMAs, each
// CTA its own 128 rows, as the bf16 kernel does (tc_gemm.cu).  Warp 0 issues
// TMA loads (the three planes of an operand tile in one 3-D box), warp 1 of
// the even CTA the MMAs: per 32-element chunk of K the six plane products,
// smallest first, into one of the tensor-memory accumulators.  Eight (sixteen)
// epilogue warps read each finished chunk and add it to the accumulators they
// hold in registers (64 a thread: 4 rows x 16 columns), while the MMAs of the next
// chunks run.  At the end of a verification period they inject the scheduled faults
// (Section 5.3), form the unit's row and column sums, compare them with the
// checksums and locate and correct (Section 4.2.1), exactly as the CUDA-core
// kernel does on its fragments (simt_ftgemm.cuh).
//
// The checksums (Eq. 4) come from the same kernel (SUMS = true) run first on
// the encoded operands: (e^T A) B and A (B e), one result per segment of at
// most 256 of K (or a whole period, where that costs less: f32tc_plan), all in
// parallel; two warps of the main kernel add a period's segments to the running
// checksums ahead of its verification.  They cost the units' share of a tile
// (1/128 of the product each for 128 x 128 units)
// instead of an extra operand row in every MMA, so the verification unit
// stays the schedule's own tile.
#include <climits>
#include <cstddef>

#include "f32tc.cuh"
#include "ptx.cuh"

namespace ftg {

cudaError_t launch_f32tc_scan(bool abft, const F32TcParams& p, int* launches, cudaStream_t st);

// BN = 256: the large-problem tile, units of 64 rows and columns or more.
// BN = 128: finer waves for small problems, units from 16.  The issuing
// thread needs 64 cycles or more per MMA, which is what a 256 x 128 one runs
// for, and some 300 between chunks; a 256 x 256 one runs 128 and its queue
// covers the gap (8192^3 without checksums: 1080 cycles a chunk of 256 x 128,
// 1560 of 256 x 256, against 768 and 1536 of MMA time; 4.4 and 3.3 ms).
// What bounds it at BN = 256: the tensor cores without checksums (16384^3
// 28.7-30.6 ms, 295 TFLOP/s = 1770 of bf16 MMAs, the power cap); with block
// checksums the verification, which stops the MMAs once both accumulators are
// full (32-34 ms; the CUDA-core kernel 133.8).
template <int BN>
struct F32TcCfg {
  static constexpr int BM = F32TC_BM, KC = F32TC_KC;
  static constexpr int A_BYTES = 3 * BM * KC * 2;        // three planes, 64-byte rows
  static constexpr int B_BYTES = 3 * (BN / 2) * KC * 2;  // this CTA's half of the columns
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = 4;
  static constexpr int NBUF = 512 / BN;                  // tensor-memory accumulators
  // warps: TMA, MMA, two that keep the checksums (the SUMS launch: norms), then the epilogue's, EW / 4 per tensor-memory
  // lane quarter
  static constexpr int EW0 = 4, EW = BN == 256 ? 16 : 8, EPI_T = 32 * EW, THREADS = 32 * (EW0 + EW);
  static constexpr int CPT = BN / (EW / 4);              // columns per epilogue warp
  static constexpr int GC = BN == 256 ? 64 : 16;         // columns per row partial: the smallest unit
  static constexpr int GR = BN == 256 ? 32 : 16;         // rows per column partial
  static constexpr int MAXE = 128 * (BN / GC) + BN * (128 / GC);  // checksum entries with the smallest units
  static constexpr int MAXU = 128 / GC * (BN / GC);      // units per CTA tile
  static constexpr int MN_BOX = 64 * KC * 2;             // one plane's 64-column box
  // registers: 64 accumulators a thread and the rest of the epilogue need
  // more than an even split over 640 threads; the TMA / MMA group gives up
  // part of its share
  static constexpr bool SPLIT_REGS = BN == 256;
  static constexpr int REGS = 96, REGS_LOW = 64, REGS_EPI = 104;
  static_assert(4 * REGS_LOW + EW * REGS_EPI <= (4 + EW) * REGS, "register hand-over");
};

template <int BN>
struct F32TcTail {
  using Cfg = F32TcCfg<BN>;
  // verification: partial sums, and (while a flagged period is confirmed)
  // the fp64 sums and flags of its entries
  alignas(16) float colpart[128 / Cfg::GR][BN];  // column sums of GR rows
  float rowpart[BN / Cfg::GC][128];     // row sums of GC columns
  double sum64[Cfg::MAXE];
  uint8_t eflag[Cfg::MAXE];
  float c[Cfg::MAXE];                   // checksums at the end of the period: rows per column unit, then columns per row unit
  float tn[Cfg::MAXE];                  // norm term of each entry's threshold
  float sFA[128 / Cfg::GC], sFB[BN / Cfg::GC];
  uint64_t full[Cfg::STAGES], empty[Cfg::STAGES], acc_full[Cfg::NBUF], acc_empty[Cfg::NBUF];
  uint64_t chk_full, chk_empty;         // c (and tn) of a period ready, verified
  unsigned long long bestr[Cfg::MAXU], bestc[Cfg::MAXU];
  double fix_delta[Cfg::MAXU];
  int nr[Cfg::MAXU], nc[Cfg::MAXU], fix_row[Cfg::MAXU], fix_col[Cfg::MAXU];
  uint32_t tmem_base;
  int abort;
};

template <int BN>
constexpr size_t f32tc_smem() {
  static_assert(offsetof(F32TcTail<BN>, colpart) % 16 == 0 && offsetof(F32TcTail<BN>, sum64) % 8 == 0, "vector access");
  static_assert(1024 + F32TcCfg<BN>::STAGES * F32TcCfg<BN>::STAGE_BYTES + sizeof(F32TcTail<BN>) <= 227 * 1024,
                "shared memory of one CTA");
  return 1024 + (size_t)F32TcCfg<BN>::STAGES * F32TcCfg<BN>::STAGE_BYTES + sizeof(F32TcTail<BN>);
}

// Shared-memory descriptors: K-major tile of 64-byte rows, 64-byte swizzle
// (8-row groups 512 bytes apart); MN-major tile of 128-byte swizzled boxes of
// 64 columns x KC k-rows (8-row groups along K 1024 bytes apart, the next 64
// columns `group` bytes further).
__device__ __forceinline__ uint64_t desc_k_sw64(const void* p) {
  return (uint64_t)((smem_u32(p) & 0x3FFFFu) >> 4) | (uint64_t)1 << 16 | (uint64_t)(512 >> 4) << 32 |
         (uint64_t)1 << 46 | (uint64_t)4 << 61;
}
__device__ __forceinline__ uint64_t desc_mn_sw128(const void* p, uint32_t group) {
  return (uint64_t)((smem_u32(p) & 0x3FFFFu) >> 4) | (uint64_t)((group >> 4) & 0x3FFF) << 16 |
         (uint64_t)(1024 >> 4) << 32 | (uint64_t)1 << 46 | (uint64_t)2 << 61;
}

// 16 tensor-memory lanes x 32 columns in the 16x256b shape: registers 4j ..
// 4j + 3 hold (row t/4, columns 8j + 2(t%4), + 1) and (row t/4 + 8, the same
// columns) of lane t.
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Half of a reduce-scatter step: the N values of v, each summed with the
// partner's over lane bit `o`, the lanes with the bit set keeping the upper
// N / 2 of them (in v[0 .. N/2)).
template <int N>
__device__ __forceinline__ void fold(float* v, int lane, int o) {
  const bool up = lane & o;
#pragma unroll
  for (int e = 0; e < N / 2; ++e) {
    const float lo = v[e], hi = v[N / 2 + e];
    v[e] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
  }
}

// (d0, d1) += (a0, a1), packed
__device__ __forceinline__ void acc2(float& d0, float& d1, float a0, float a1) {
  asm("{\n.reg .b64 ra, rd;\n mov.b64 ra, {%2, %3};\n mov.b64 rd, {%0, %1};\n add.rn.f32x2 rd, rd, ra;\n"
      " mov.b64 {%0, %1}, rd;\n}"
      : "+f"(d0), "+f"(d1)
      : "f"(a0), "f"(a1));
}

// One unit of work of a CTA pair.  MAIN: a tile of C over one split of K.
// SUMS: a tile of a checksum product over one segment of K.
struct F32TcItem {
  int type;            // SUMS: 0 (e^T A) B, 1 (B e)^T A^T, 2 A B
  int row0, col0;      // of the pair's tile
  int z, seg;          // split (MAIN), segment (SUMS)
  int k0, klen;
};

// Tiles of one segment by type.
struct F32TcSums {
  int cols[3], n[3];
};
template <int BN>
__host__ __device__ __forceinline__ F32TcSums f32tc_sums(const F32TcParams& p) {
  F32TcSums t;
  t.cols[0] = t.cols[2] = (p.N + BN - 1) / BN;
  t.cols[1] = (p.M + BN - 1) / BN;
  t.n[0] = p.Dc ? (p.nv + 255) / 256 * t.cols[0] : 0;
  t.n[1] = p.Dc ? (p.nw + 255) / 256 * t.cols[1] : 0;
  t.n[2] = p.P ? p.tiles_m2 * t.cols[2] : 0;
  return t;
}

template <int BN, bool SUMS>
__device__ __forceinline__ int f32tc_items(const F32TcParams& p) {
  if constexpr (!SUMS) return p.tiles;
  const F32TcSums t = f32tc_sums<BN>(p);
  return p.nsplit * p.sg.per_split * (t.n[0] + t.n[1] + t.n[2]);
}

template <int BN, bool SUMS>
__device__ __forceinline__ F32TcItem f32tc_item(const F32TcParams& p, int id) {
  F32TcItem t;
  if constexpr (!SUMS) {
    const int tiles = p.tiles_m2 * p.tiles_n;
    int width = BN, half = 0;
    if (BN == 128 && p.half_first > 0) {
      width = 256;
      half = id % 2 * 128;
      id = p.half_first + id / 2;
    }
    t.z = id / tiles;
    id -= t.z * tiles;
    const int per_group = p.group_m * p.tiles_n, first = id / per_group * p.group_m;
    const int gsize = min(p.tiles_m2 - first, p.group_m), in = id % per_group;
    t.type = 0;
    t.seg = 0;
    t.row0 = (first + in % gsize) * 256;
    t.col0 = in / gsize * width + half;
    t.k0 = t.z * p.k_per_split;
    t.klen = min(p.k_per_split, p.K - t.k0);
  } else {
    const F32TcSums u = f32tc_sums<BN>(p);
    const int per = u.n[0] + u.n[1] + u.n[2];
    t.seg = id / per;
    int j = id - t.seg * per;
    t.type = j < u.n[0] ? 0 : j < u.n[0] + u.n[1] ? 1 : 2;
    if (t.type > 0) j -= u.n[0];
    if (t.type > 1) j -= u.n[1];
    const int cols = t.type == 1 ? u.cols[1] : u.cols[0];
    t.row0 = j / cols * 256;
    t.col0 = j % cols * BN;
    t.z = t.seg / p.sg.per_split;
    const int k0 = t.z * p.k_per_split;
    f32tc_segment(p.sg, t.seg - t.z * p.sg.per_split, min(p.k_per_split, p.K - k0), &t.k0, &t.klen);
    t.k0 += k0;
  }
  return t;
}

// Norms from the encode pass's squared partials, a line (row of A, column of B)
// per lane, and the sums of squares of each 16 lines; eight partial sums a line
// in a fixed order, so results repeat.  Two warps of every CTA of the SUMS launch,
// which have nothing else to do: a kernel of its own took 6-14 us of every call
// (256 .. 4096 rows) before the checksum products could start.
__device__ __forceinline__ void f32tc_norms(const F32TcParams& p, int w, int nw, int lane) {
  const int ga = (p.M + 31) / 32, gb = (p.N + 31) / 32, parts = (p.K + 127) / 128;
  for (int g = w; g < ga + gb; g += nw) {
    const bool side_a = g < ga;
    const int L = side_a ? p.M : p.N, line = (side_a ? g : g - ga) * 32 + lane;
    const float* part = (side_a ? p.pa : p.pb) + line;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (line < L) {
      for (int c = 0; c < parts; c += 8)
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c + u < parts) s[u] += part[(long long)(c + u) * L];
    }
    float t = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
    if (line < L) (side_a ? p.nA : p.nB)[line] = sqrtf(t);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (line < L && lane % 16 == 0) (side_a ? p.sq16a : p.sq16b)[line / 16] = t;
  }
}

template <int BN, bool ABFT, bool SUMS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(F32TcCfg<BN>::THREADS, 1)
    f32tc_kernel(const __grid_constant__ F32TcMaps maps, const __grid_constant__ F32TcParams p) {
  using Cfg = F32TcCfg<BN>;
  constexpr int S = Cfg::STAGES, NBUF = Cfg::NBUF, CPT = Cfg::CPT, KC = Cfg::KC, EPI_T = Cfg::EPI_T;
  pdl_wait();
  pdl_trigger();
  if (*p.bad == p.epoch) {  // an operand outside the split's range: the CUDA-core kernel runs instead
    if (SUMS && p.pa && threadIdx.x / 32 - 2 < 2u)  // (with the same norms)
      f32tc_norms(p, blockIdx.x * 2 + threadIdx.x / 32 - 2, gridDim.x * 2, threadIdx.x & 31);
    return;
  }
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = smem_raw + (-smem_u32(smem_raw) & 1023u);  // (shared address space kept)
  F32TcTail<BN>& T = *reinterpret_cast<F32TcTail<BN>*>(base + S * Cfg::STAGE_BYTES);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_ctarank();
  const bool leader = rank == 0;
  const int worker = blockIdx.x >> 1, workers = gridDim.x >> 1;
  const int items = f32tc_items<BN, SUMS>(p), nch = (p.K + KC - 1) / KC;
  auto sA = [&](int s) { return base + s * Cfg::STAGE_BYTES; };
  auto sB = [&](int s) { return base + s * Cfg::STAGE_BYTES + Cfg::A_BYTES; };

  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&T.full[s], 1);
      mbar_init(&T.empty[s], 1);
    }
    for (int a = 0; a < NBUF; ++a) {
      mbar_init(&T.acc_full[a], 1);
      mbar_init(&T.acc_empty[a], 2 * Cfg::EW);  // one arrival per epilogue warp of both CTAs
    }
    mbar_init(&T.chk_full, 2);
    mbar_init(&T.chk_empty, Cfg::EW);
    T.abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(&T.tmem_base, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the leader's barriers are initialised before the other CTA signals them
  tc_fence_after();
  const uint32_t tmem = T.tmem_base;

  if (warp < Cfg::EW0) {
    if constexpr (Cfg::SPLIT_REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Cfg::REGS_LOW));
  if (warp == 0 && lane == 0) {
    // ---- TMA producer: this CTA's 128 rows and its half of the columns ----
    uint32_t it = 0;
    bool dead = false;
    for (int id = worker; id < items && !dead; id += workers) {
      const F32TcItem x = f32tc_item<BN, SUMS>(p, id);
      const CUtensorMap* mA = !SUMS || x.type == 2 ? &maps.A : (x.type ? &maps.W : &maps.V);
      const bool kmajor_b = SUMS && x.type == 1;
      const int row = x.row0 + rank * 128, col = x.col0 + rank * (BN / 2);
      for (int k = 0; k < x.klen; k += KC, ++it) {
        const int s = it % S;
        if (it >= S && !mbar_wait(&T.empty[s], ((it / S) & 1u) ^ 1u)) {
          dead = true;
          break;
        }
        const uint32_t cbar = mapa_rank(&T.full[s], 0);
        if (leader) mbar_arrive_expect_tx(&T.full[s], 2 * Cfg::STAGE_BYTES);
        const int chunk = (x.k0 + k) / KC;
        tma_load_2d_pair(sA(s), mA, cbar, 0, (row / 128 * nch + chunk) * 192);
        if (kmajor_b) {
          // rows col .. col + BN/2 - 1 of A, plane by plane in 64-row pieces
#pragma unroll
          for (int pl = 0; pl < 3; ++pl)
#pragma unroll
            for (int g = 0; g < BN / 128; ++g)
              tma_load_2d_pair(sB(s) + (pl * (BN / 128) + g) * 4096, &maps.An, cbar, 0,
                               ((col + 64 * g) / 128 * nch + chunk) * 192 + pl * 64 + (col + 64 * g) % 128 / 2);
        } else {
#pragma unroll
          for (int g = 0; g < BN / 128; ++g)
            tma_load_2d_pair(sB(s) + g * 3 * Cfg::MN_BOX, &maps.B, cbar, 0, ((col / 64 + g) * nch + chunk) * 96);
        }
      }
    }
    if (dead) atomicExch(&T.abort, 1);
    // let the last loads land before the CTAs may exit (bounded)
    if (leader)
      for (uint32_t q = it > (uint32_t)S ? it - S : 0; q < it; ++q) mbar_wait(&T.full[q % S], (q / S) & 1u);
  } else if (SUMS && warp >= 2) {
    if (p.pa) f32tc_norms(p, blockIdx.x * 2 + warp - 2, gridDim.x * 2, lane);
  } else if (ABFT && warp >= 2) {
    // ---- the checksums of the epilogue's entries, a period ahead ------------
    // Their segments of the coming period are loaded while the current one
    // runs and added once it is verified; a tile's first period also forms the
    // thresholds' norm terms.  Done by the epilogue itself this kept the MMAs
    // waiting: the 256-column tiles of 8192^3 took 3.54 ms, now 3.35, those of
    // 4096^3's three full waves 430 us, now 407.  A tile's norms are loaded before
    // its turn too: 16384 x 16384 x 32, one period a tile, 550 us a call without
    // that, now 410.
    const int hq = (warp - 2) * 32 + lane;
    const int um_sh = 31 - __clz(p.um), un_sh = 31 - __clz(p.un);
    const int nRow = 128 * (BN >> un_sh), nE = nRow + BN * (128 >> um_sh);
    // entries a thread loads at a time (more would spill); one after the other
    // the 2048 entries of 16 x 16 units took far longer than their period (1300 x
    // 900 x 8192 584 us; now 315, still bound by these two warps)
    constexpr int AHEAD = BN == 128 ? 8 : 4;
    uint32_t checks = 0;
    bool dead = false;
    auto both = [] { asm volatile("bar.sync 2, 64;" ::: "memory"); };
    for (int id = worker; id < items; id += workers) {
      const F32TcItem x = f32tc_item<BN, SUMS>(p, id);
      const int row0 = x.row0 + rank * 128, col0 = x.col0;
      const int ks0 = x.z * p.ks_per_split, nks = min(p.ks_per_split, p.ksteps - ks0);
      // Frobenius norms of the units' rows and columns
      auto fro = [](const float* sq16, int first, int per, int count) {
        float v[8], s = 0.f;  // (loads first: per <= 8)
#pragma unroll
        for (int g = 0; g < 8; ++g) v[g] = g < per && first + g < count ? sq16[first + g] : 0.f;
#pragma unroll
        for (int g = 0; g < 8; ++g) s += v[g];
        return sqrtf(s);
      };
      both();  // the other warp is done with the tile before
      if (hq < 128 >> um_sh) T.sFA[hq] = fro(p.sq16a, row0 / 16 + hq * (p.um / 16), p.um / 16, (p.M + 15) / 16);
      if (hq < BN >> un_sh) T.sFB[hq] = fro(p.sq16b, col0 / 16 + hq * (p.un / 16), p.un / 16, (p.N + 15) / 16);
      both();
      for (int period = 0, done = 0; done < nks; ++period, done += p.cadence) {
        // segment g of this period at entry e: its address (null outside the
        // matrix) for g = 0 and the distance to the next
        const int s0 = x.z * p.sg.per_split + period * p.sg.per_period;
        const int J0 = col0 >> un_sh, I0 = row0 >> um_sh;
        const float* const dr = p.Dr + ((long long)s0 * p.nw + J0) * p.ldr_d + row0;
        const float* const dc = p.Dc + ((long long)s0 * p.nv + I0) * p.ldc_d + col0;
        auto seg_of = [&](int e, long long* stride) -> const float* {
          if (e < nRow) {
            const int J = e >> 7, r = e & 127;
            *stride = (long long)p.nw * p.ldr_d;
            return J0 + J < p.nw && row0 + r < p.M ? dr + J * p.ldr_d + r : nullptr;
          }
          const int I = (e - nRow) / BN, c = (e - nRow) % BN;
          *stride = (long long)p.nv * p.ldc_d;
          return I0 + I < p.nv && col0 + c < p.N ? dc + I * p.ldc_d + c : nullptr;
        };
        const int segs = min(p.sg.per_period, p.sg.per_split - period * p.sg.per_period);
        auto first = [&](int e) {
          long long stride;
          const float* src = e < nE ? seg_of(e, &stride) : nullptr;
          return src ? __ldg(src) : 0.f;
        };
        auto norm = [&](int e) {  // of the row or column of entry e
          const int gr = row0 + (e & 127), gc = col0 + (e - nRow) % BN;
          if (e < nRow) return gr < p.M ? p.nA[gr] : 0.f;
          return e < nE && gc < p.N ? p.nB[gc] : 0.f;
        };
        auto enter = [&](int e, float d, float nrm) {  // entry e, d its first segment
          float c = (period > 0 ? T.c[e] : 0.f) + d;
          if (segs > 1) {  // periods longer than a segment
            long long stride;
            const float* src = seg_of(e, &stride);
            for (int g = 1; src && g < segs; ++g) c += __ldg(src + g * stride);
          }
          T.c[e] = c;
          if (period == 0) {
            // lambda * u times the norms, rounded as ft_tau does
            T.tn[e] = e < nRow ? __fmul_rn(__fmul_rn(p.lam_u, nrm), T.sFB[e >> 7])
                               : __fmul_rn(__fmul_rn(p.lam_u, T.sFA[(e - nRow) / BN]), nrm);
          }
        };
#pragma unroll 1
        for (int e0 = hq; e0 < nE; e0 += 64 * AHEAD) {
          float d[AHEAD];
#pragma unroll
          for (int i = 0; i < AHEAD; ++i) d[i] = first(e0 + 64 * i);
          float nrm[AHEAD];
#pragma unroll
          for (int i = 0; i < AHEAD; ++i) nrm[i] = period == 0 ? norm(e0 + 64 * i) : 0.f;
          // (the loads of small units' further entries overlap the coming period)
          if (e0 == hq && checks > 0 && !dead && !mbar_wait(&T.chk_empty, (checks - 1) & 1u)) {
            dead = true;
            atomicExch(&T.abort, 1);
          }
#pragma unroll
          for (int i = 0; i < AHEAD; ++i)
            if (e0 + 64 * i < nE) enter(e0 + 64 * i, d[i], nrm[i]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&T.chk_full);
        ++checks;
      }
    }
  } else if (warp == 1 && lane == 0 && leader) {
    // ---- MMA issuer: per chunk the six plane products, smallest first ----
    constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((256u >> 4) << 24);
    uint32_t it = 0;
    bool dead = false;
    for (int id = worker; id < items && !dead; id += workers) {
      const F32TcItem x = f32tc_item<BN, SUMS>(p, id);
      const bool kmajor_b = SUMS && x.type == 1;
      const uint32_t id_t = kmajor_b ? idesc : idesc | (1u << 16);  // B MN-major
      for (int k = 0; k < x.klen; k += KC, ++it) {
        const int s = it % S, ab = it % NBUF;
        if ((it >= (uint32_t)NBUF && !mbar_wait(&T.acc_empty[ab], ((it / NBUF) & 1u) ^ 1u)) ||
            !mbar_wait(&T.full[s], (it / S) & 1u)) {
          dead = true;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(ab * BN);
        const uint64_t da = desc_k_sw64(sA(s));
        // planes of the operands, smallest product first; 16 elements of K at a time
        auto products = [&](uint64_t db, uint32_t pb, uint32_t kb, int nk16) {
          constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
          for (int q = 0; q < 6; ++q)
#pragma unroll
            for (int kk = 0; kk < KC / 16; ++kk)
              if (kk < nk16)
                tc_mma_f16_pair(d, da + (uint64_t)(PA[q] * (128 * KC * 2 >> 4) + kk * 2),
                                db + (uint64_t)(PB[q] * pb + kk * kb), id_t, (q | kk) != 0);
        };
        constexpr uint32_t PB_MN = Cfg::MN_BOX >> 4, PB_K = (BN / 2) * KC * 2 >> 4;
        if (!kmajor_b) {
          const uint64_t db = desc_mn_sw128(sB(s), 3 * Cfg::MN_BOX);
          if (x.klen - k > KC / 2) products(db, PB_MN, 16 * 128 >> 4, KC / 16);
          else products(db, PB_MN, 16 * 128 >> 4, 1);
        } else {
          const uint64_t db = desc_k_sw64(sB(s));
          if (x.klen - k > KC / 2) products(db, PB_K, 2, KC / 16);
          else products(db, PB_K, 2, 1);
        }
        tc_commit_pair(&T.empty[s], (uint16_t)3);
        tc_commit_pair(&T.acc_full[ab], (uint16_t)3);
      }
    }
    if (dead) atomicExch(&T.abort, 1);
    // let the last MMAs finish before tensor memory may be released (bounded)
    if (it > 0) mbar_wait(&T.acc_full[(it - 1) % NBUF], ((it - 1) / NBUF) & 1u);
    }
  } else {
    if constexpr (Cfg::SPLIT_REGS) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Cfg::REGS_EPI));
    // ---- epilogue: accumulate, verify, store -------------------------------
    // Thread layout of the accumulators (the 16x256b tensor-memory shape): rows
    // rbase + 8 i, columns cbase + 8 j + b.  Column sums then need 3 shuffle
    // levels instead of the 5 of one row per lane, and C is written straight
    // from registers in whole 32-byte sectors.
    constexpr int NJ = CPT / 8;
    const int lq = warp & 3, eh = (warp - Cfg::EW0) >> 2, q = (warp - Cfg::EW0) * 32 + lane;
    const int rbase = lq * 32 + (lane >> 2), cbase = eh * CPT + 2 * (lane & 3);
    uint32_t it = 0, checks = 0;
    bool dead = false;
    float acc[4][NJ][2];
    // Hand a chunk's accumulator back to the MMA thread (in the leader CTA).
    // Relaxed: the reads completed (wait::ld) and no store precedes, so the
    // arrival has nothing to publish.  With release at cluster scope, an
    // arrival cost each warp some 1700 cycles a chunk, twice the chunk's MMAs
    // of 256 x 128 (8192^3 without checksums: 7.0 ms against 4.9).
    auto acc_release = [&](int ab) {
      asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(mapa_rank(&T.acc_empty[ab], 0))
                   : "memory");
    };
    // the tile's rows < rows and columns < cols from the registers to memory
    auto store = [&](float* out, long long ld, int rows, int cols, float alpha, float beta, bool vec) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tr = rbase + 8 * i;
        if (tr >= rows) continue;
        float* line = out + (long long)tr * ld + cbase;
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          const int tc = cbase + 8 * j;
          float2 o = make_float2(alpha * acc[i][j][0], alpha * acc[i][j][1]);
          if (vec && tc + 1 < cols) {
            if (beta != 0.f) {
              const float2 ci = *reinterpret_cast<const float2*>(line + 8 * j);
              o = make_float2(fmaf(beta, ci.x, o.x), fmaf(beta, ci.y, o.y));
            }
            *reinterpret_cast<float2*>(line + 8 * j) = o;
          } else {
            if (tc < cols) line[8 * j] = beta != 0.f ? fmaf(beta, line[8 * j], o.x) : o.x;
            if (tc + 1 < cols) line[8 * j + 1] = beta != 0.f ? fmaf(beta, line[8 * j + 1], o.y) : o.y;
          }
        }
      }
    };

    for (int id = worker; id < items; id += workers) {
      const F32TcItem x = f32tc_item<BN, SUMS>(p, id);
      const int row0 = x.row0 + rank * 128, col0 = x.col0;
      // schedule k-steps of this split, and its verification periods
      const int ks0 = x.z * p.ks_per_split, ks1 = min(ks0 + p.ks_per_split, p.ksteps);
      const int um_sh = 31 - __clz(p.um), un_sh = 31 - __clz(p.un);
      const int nRow = ABFT ? 128 * (BN >> un_sh) : 0, nE = ABFT ? nRow + BN * (128 >> um_sh) : 0;
      // the k-step that ends the current period, and the elements of K up to it
      int period = 0, next_ks = INT_MAX, k_end = INT_MAX;
      bool has_fault = false;
      if constexpr (!SUMS) {
        next_ks = min(ks0 + (ABFT ? p.cadence : p.ks_per_split), ks1) - 1;
        k_end = min(x.klen, (next_ks + 1 - ks0) * p.k_tb);
        if (p.nfaults > 0) {
          // any scheduled fault in the schedule tiles this CTA tile covers?
          const int tm0 = row0 / p.m_tb, tn0 = col0 / p.n_tb;
          const int ntr = row0 < p.M ? (min(row0 + 128, p.M) - 1) / p.m_tb - tm0 + 1 : 0;
          const int ntc = (min(col0 + BN, p.N) - 1) / p.n_tb - tn0 + 1;
          bool mine = false;
          for (int t = lane; t < ntr * ntc; t += 32) {
            const int tile = (tm0 + t / ntc) * p.tiles_n_sched + tn0 + t % ntc;
            const int f = first_fault(p.faults, p.nfaults, tile);
            mine |= f < p.nfaults && p.faults[f].tile == tile;
          }
          has_fault = __any_sync(0xffffffffu, mine);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j][0] = acc[i][j][1] = 0.f;

      for (int k = 0; k < x.klen; k += KC, ++it) {
        const int ab = it % NBUF;
        const bool ok = !dead && mbar_wait(&T.acc_full[ab], (it / NBUF) & 1u);
        if (!ok && !dead) {
          dead = true;
          atomicExch(&T.abort, 1);
        }
        tc_fence_after();
        __syncwarp();
        if (ok) {
          const uint32_t tl = tmem + (uint32_t)(ab * BN + eh * CPT) + ((uint32_t)(lq * 32) << 16);
          // 32 columns of 16 rows are added while the next load is in flight
          constexpr int NL = CPT / 16;
          float v[2][16];
          auto load = [&](int l) { tmem_ld_16x256b_x4(tl + l / 2 * 32 + ((uint32_t)(l % 2 * 16) << 16), v[l & 1]); };
          load(0);
#pragma unroll
          for (int l = 0; l < NL; ++l) {
            tmem_wait_ld();
            if (l + 1 < NL) load(l + 1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              float(&lo)[2] = acc[2 * (l & 1)][4 * (l >> 1) + j];
              float(&hi)[2] = acc[2 * (l & 1) + 1][4 * (l >> 1) + j];
              acc2(lo[0], lo[1], v[l & 1][4 * j], v[l & 1][4 * j + 1]);
              acc2(hi[0], hi[1], v[l & 1][4 * j + 2], v[l & 1][4 * j + 3]);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) acc_release(ab);

        if constexpr (!SUMS) {
          if (k + KC < k_end) continue;
          const int ks = next_ks, ks_first = ks0 + period * (ABFT ? p.cadence : p.ks_per_split);
          if constexpr (ABFT) {  // the checksums through this period
            if (!dead && !mbar_wait(&T.chk_full, checks & 1u)) {
              dead = true;
              atomicExch(&T.abort, 1);
            }
            ++checks;
          }
          // ----- faults scheduled in this period (Section 5.3): additive
          // offsets on the accumulators or the running checksums -----
          if (has_fault) {
            const int tm0 = row0 / p.m_tb, tn0 = col0 / p.n_tb;
            const int tm1 = (min(row0 + 128, p.M) - 1) / p.m_tb, tn1 = (min(col0 + BN, p.N) - 1) / p.n_tb;
            for (int tm = tm0; tm <= tm1; ++tm)
              for (int tn = tn0; tn <= tn1; ++tn) {
                const int tile = tm * p.tiles_n_sched + tn;
                for (int f = first_fault(p.faults, p.nfaults, tile); f < p.nfaults && p.faults[f].tile == tile; ++f) {
                  const Fault F = p.faults[f];
                  if (F.kstep < ks_first || F.kstep > ks) continue;
                  const int fr = tm * p.m_tb + F.row - row0, fc = tn * p.n_tb + F.col - col0;
                  if (F.target == T_ACC) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                      for (int j = 0; j < NJ; ++j)
#pragma unroll
                        for (int b = 0; b < 2; ++b)
                          if (rbase + 8 * i == fr && cbase + 8 * j + b == fc) acc[i][j][b] += F.delta;
                  } else if constexpr (ABFT) {
                    const int e = F.target == T_ROWSUM ? fc / p.un * 128 + fr : nRow + fr / p.um * BN + fc;
                    if (e % EPI_T == q) T.c[e] += F.delta;  // the thread that keeps the entry
                  }
                }
              }
          }
          if constexpr (ABFT) {
            // ----- verification: partial sums of GC columns of each row and
            // of GR rows of each column -----
            constexpr int GC = Cfg::GC, GR = Cfg::GR;
            {
              // rows: this thread's columns of each group, then its quad's
              constexpr int NG = CPT / GC, JG = GC / 8;
              float t[NG * 4];
#pragma unroll
              for (int g = 0; g < NG; ++g)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  float s[JG][2];
#pragma unroll
                  for (int j = 0; j < JG; ++j) {
                    s[j][0] = acc[i][g * JG + j][0];
                    s[j][1] = acc[i][g * JG + j][1];
                  }
#pragma unroll
                  for (int st = JG / 2; st > 0; st >>= 1)
#pragma unroll
                    for (int j = 0; j < st; ++j) acc2(s[j][0], s[j][1], s[j + st][0], s[j + st][1]);
                  t[g * 4 + i] = s[0][0] + s[0][1];
                }
              fold<NG * 4>(t, lane, 2);
              fold<NG * 2>(t, lane, 1);
              const int v0 = (lane & 2 ? NG * 2 : 0) + (lane & 1 ? NG : 0);
#pragma unroll
              for (int e = 0; e < NG; ++e) T.rowpart[eh * NG + (v0 + e) / 4][rbase + 8 * ((v0 + e) % 4)] = t[e];
            }
            {
              // columns: this thread's rows of each group, then 8 lanes'
              constexpr int NG = 32 / GR, IG = 4 / NG, NV = NG * NJ * 2;
              static_assert(NV >= 16, "three folds leave pairs");
              float t[NV];
#pragma unroll
              for (int g = 0; g < NG; ++g)
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                  float(&d)[2] = *reinterpret_cast<float(*)[2]>(&t[(g * NJ + j) * 2]);
                  d[0] = acc[g * IG][j][0];
                  d[1] = acc[g * IG][j][1];
#pragma unroll
                  for (int i = 1; i < IG; ++i) acc2(d[0], d[1], acc[g * IG + i][j][0], acc[g * IG + i][j][1]);
                }
              fold<NV>(t, lane, 16);
              fold<NV / 2>(t, lane, 8);
              fold<NV / 4>(t, lane, 4);
              const int v0 = (lane & 16 ? NV / 2 : 0) + (lane & 8 ? NV / 4 : 0) + (lane & 4 ? NV / 8 : 0);
#pragma unroll
              for (int e = 0; e < NV / 8; e += 2) {
                const int g = (v0 + e) / (NJ * 2), j = (v0 + e) % (NJ * 2) / 2;
                *reinterpret_cast<float2*>(&T.colpart[lq * NG + g][cbase + 8 * j]) = make_float2(t[e], t[e + 1]);
              }
            }
            bar_red_or(1, EPI_T, 0);
            // growth term of the threshold after k elements of K in this split
            const float grow = __fmul_rn(p.mu_u, sqrtf((float)(min((ks + 1) * p.k_tb, p.K) - ks0 * p.k_tb)));
            // threshold of entry e with checksum c
            auto tau_of = [&](int e, float c) { return __fmaf_rn(grow, fabsf(c), T.tn[e]); };
            unsigned flags = 0u;
            const int row_per = p.un / GC, col_per = p.um / GR;
#pragma unroll 1
            for (int i = 0; i < Cfg::MAXE / EPI_T; ++i) {
              const int e = q + i * EPI_T;
              if (e >= nE) break;
              const float c = T.c[e];
              const bool is_row = e < nRow;
              const int sh = is_row ? 7 : BN == 256 ? 8 : 7;  // entries of a line of partial sums
              const int per = is_row ? row_per : col_per, at = is_row ? e : e - nRow;
              const float* src = (is_row ? &T.rowpart[0][0] : &T.colpart[0][0]) + ((at >> sh) * per << sh) + (at & ((1 << sh) - 1));
              float w[128 / (GC < GR ? GC : GR)], s = 0.f;
#pragma unroll
              for (int g = 0; g < 128 / (GC < GR ? GC : GR); ++g) w[g] = g < per ? src[g << sh] : 0.f;
#pragma unroll
              for (int g = 0; g < 128 / (GC < GR ? GC : GR); ++g) s += w[g];
              if (ok && fabsf(s - c) > kScreen * tau_of(e, c)) flags |= 1u << i;
            }
            if (bar_red_or(1, EPI_T, flags != 0u)) {
              // ----- fp64 confirmation of the screened entries -----
              const int units_n = BN / p.un, units = units_n * (128 / p.um);
              int i = 0;
              for (int e = q; e < nE; e += EPI_T, ++i) {
                T.eflag[e] = (flags >> i) & 1u;
                T.sum64[e] = 0.0;
              }
              if (q < units) {
                T.nr[q] = 0; T.nc[q] = 0; T.bestr[q] = 0ull; T.bestc[q] = 0ull; T.fix_row[q] = -1;
              }
              bar_red_or(1, EPI_T, 0);
              constexpr int RG = CPT / GC, CG = 32 / GR;  // entries of a row, of a column
              if constexpr (BN == 128) {
                // Which of the warp's entries are flagged first, then one at a
                // time in a loop: a branch around every entry's own code took
                // most of an event's time fetching code (777 x 1531 x 2049, the
                // kernel with one fault 72 us, now 68, without 58).  256-column
                // tiles have no registers for that.
                unsigned rm = 0u;
#pragma unroll
                for (int u = 0; u < 4 * RG; ++u)
                  rm |= (unsigned)T.eflag[((eh * CPT + GC * (u % RG)) >> un_sh) * 128 + rbase + 8 * (u / RG)] << u;
                for (unsigned m = __reduce_or_sync(0xffffffffu, rm); m; m &= m - 1u) {
                  const int u0 = __ffs(m) - 1;
                  double sum = 0.0;
#pragma unroll
                  for (int j = 0; j < GC / 4; ++j) {
                    float v = 0.f;
#pragma unroll
                    for (int u = 0; u < 4 * RG; ++u)
                      if (u == u0) v = acc[u / RG][u % RG * (GC / 8) + j / 2][j % 2];
                    sum += (double)v;
                  }
#pragma unroll
                  for (int o = 1; o < 4; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                  if ((rm >> u0 & 1u) && (lane & 3) == 0)
                    atomicAdd(&T.sum64[((eh * CPT + GC * (u0 % RG)) >> un_sh) * 128 + rbase + 8 * (u0 / RG)], sum);
                }
                unsigned cm = 0u;
#pragma unroll
                for (int u = 0; u < CG * NJ * 2; ++u)
                  cm |= (unsigned)T.eflag[nRow + ((lq * 32 + GR * (u / (NJ * 2))) >> um_sh) * BN + cbase + u % (NJ * 2) / 2 * 8 + u % 2] << u;
                for (unsigned m = __reduce_or_sync(0xffffffffu, cm); m; m &= m - 1u) {
                  const int u0 = __ffs(m) - 1;
                  double sum = 0.0;
#pragma unroll
                  for (int r = 0; r < GR / 8; ++r) {
                    float v = 0.f;
#pragma unroll
                    for (int u = 0; u < CG * NJ * 2; ++u)
                      if (u == u0) v = acc[u / (NJ * 2) * (GR / 8) + r][u % (NJ * 2) / 2][u % 2];
                    sum += (double)v;
                  }
#pragma unroll
                  for (int o = 4; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                  if ((cm >> u0 & 1u) && lane < 4)
                    atomicAdd(&T.sum64[nRow + ((lq * 32 + GR * (u0 / (NJ * 2))) >> um_sh) * BN + cbase + u0 % (NJ * 2) / 2 * 8 + u0 % 2], sum);
                }
              } else {
#pragma unroll
                for (int i2 = 0; i2 < 4; ++i2) {
                  const int r = rbase + 8 * i2;
#pragma unroll
                  for (int g = 0; g < CPT / GC; ++g) {
                    const int e = ((eh * CPT + GC * g) >> un_sh) * 128 + r;
                    if (T.eflag[e]) {
                      double s = 0.0;
#pragma unroll
                      for (int j = 0; j < GC / 8; ++j) s += (double)acc[i2][g * (GC / 8) + j][0] + (double)acc[i2][g * (GC / 8) + j][1];
                      atomicAdd(&T.sum64[e], s);
                    }
                  }
#pragma unroll
                  for (int j = 0; j < NJ; ++j)
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                      const int e = nRow + (r >> um_sh) * BN + cbase + 8 * j + b;
                      if (T.eflag[e]) atomicAdd(&T.sum64[e], (double)acc[i2][j][b]);
                    }
                }
              }
              bar_red_or(1, EPI_T, 0);
              i = 0;
              for (int e = q; e < nE; e += EPI_T, ++i) {
                if (!((flags >> i) & 1u)) continue;
                const float c = T.c[e], tau = tau_of(e, c);
                const double d = T.sum64[e] - (double)c;
                if (!(fabs(d) > (double)tau)) continue;
                const float sc = flag_score((float)d, tau);
                if (e < nRow) {
                  const int u = (e & 127) / p.um * units_n + (e >> 7);
                  atomicAdd(&T.nr[u], 1);
                  atomicMax(&T.bestr[u], flag_key(sc, e & 127));
                } else {
                  const int col = (e - nRow) % BN, u = (e - nRow) / BN * units_n + col / p.un;
                  atomicAdd(&T.nc[u], 1);
                  atomicMax(&T.bestc[u], flag_key(sc, col));
                }
              }
              bar_red_or(1, EPI_T, 0);
              if (q < units && (T.nr[q] | T.nc[q])) {
                const int nr = T.nr[q], nc = T.nc[q];
                const int ir = nr ? key_index(T.bestr[q]) : -1, jc = nc ? key_index(T.bestc[q]) : -1;
                const int er = nr ? q % units_n * 128 + ir : 0, ec = nc ? nRow + q / units_n * BN + jc : 0;
                const double dR = nr ? T.sum64[er] - (double)T.c[er] : 0.0, dC = nc ? T.sum64[ec] - (double)T.c[ec] : 0.0;
                const float tR = nr ? tau_of(er, T.c[er]) : 0.f, tC = nc ? tau_of(ec, T.c[ec]) : 0.f;
                ftgemm_fault_record rec;
                rec.tile_m = (row0 + q / units_n * p.um) / p.m_tb;
                rec.tile_n = (col0 + q % units_n * p.un) / p.n_tb;
                rec.kstep = ks;
                rec.problem = 0; rec.reserved = 0;
                rec.row = nr ? row0 + ir : -1;
                rec.col = nc ? col0 + jc : -1;
                rec.residual_r = dR; rec.residual_c = dC; rec.tau = (double)tR + (double)tC;
                rec.delta = 0.0;
                if (nr == 1 && nc == 1) {
                  if (fabs(dR - dC) <= (double)tR + (double)tC) {
                    rec.kind = K_CORRECTED; rec.delta = dR;
                    T.fix_row[q] = ir; T.fix_col[q] = jc; T.fix_delta[q] = dR;
                  } else {
                    rec.kind = K_UNCORRECTABLE;
                  }
                } else if (nr == 1 && nc == 0) {
                  rec.kind = K_CHECKSUM; rec.delta = -dR; T.c[er] = (float)T.sum64[er];
                } else if (nr == 0 && nc == 1) {
                  rec.kind = K_CHECKSUM; rec.delta = -dC; T.c[ec] = (float)T.sum64[ec];
                } else {
                  rec.kind = K_UNCORRECTABLE;
                }
                report_event(p.rep, p.recs, rec);
              }
              bar_red_or(1, EPI_T, 0);
              // ----- correct the located elements (Section 4.2.1) -----
#pragma unroll
              for (int i2 = 0; i2 < 4; ++i2)
#pragma unroll
                for (int g = 0; g < CPT / GC; ++g) {
                  const int r = rbase + 8 * i2, u = (r >> um_sh) * units_n + ((eh * CPT + GC * g) >> un_sh);
                  if (T.fix_row[u] == r) {
#pragma unroll
                    for (int j = g * (GC / 8); j < (g + 1) * (GC / 8); ++j)
#pragma unroll
                      for (int b = 0; b < 2; ++b)
                        if (T.fix_col[u] == cbase + 8 * j + b) acc[i2][j][b] = (float)((double)acc[i2][j][b] - T.fix_delta[u]);
                  }
                }
              bar_red_or(1, EPI_T, 0);  // the shared arrays are reused
            }
          }
          ++period;
          next_ks = min(next_ks + (ABFT ? p.cadence : p.ks_per_split), ks1 - 1);
          k_end = min(x.klen, (next_ks + 1 - ks0) * p.k_tb);
          if constexpr (ABFT) {
            __syncwarp();
            if (lane == 0) mbar_arrive(&T.chk_empty);
          }
        }
      }
      if (dead) continue;
      if constexpr (SUMS) {
        const int lines = x.type == 2 ? p.M : x.type ? p.nw : p.nv;
        const long long ld = x.type == 2 ? p.ldp : x.type ? p.ldr_d : p.ldc_d;
        float* out = (x.type == 2 ? p.P : x.type ? p.Dr : p.Dc) + ((long long)x.seg * lines + row0) * ld + col0;
        store(out, ld, lines - row0, (x.type == 1 ? p.M : p.N) - col0, 1.f, 0.f, true);
      } else if (p.partial) {
        store(p.partial + ((long long)x.z * p.M + row0) * p.N + col0, p.N, p.M - row0, p.N - col0, 1.f, 0.f,
              (p.N & 1) == 0);
      } else {
        store(p.C + (long long)row0 * p.ldc + col0, p.ldc, p.M - row0, p.N - col0, p.alpha, p.beta, p.c_vec);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && T.abort) atomicAdd(&p.rep->timeouts, 1);
  cluster_sync();  // both CTAs are done with each other's barriers and tensor memory
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}

template <int BN, bool ABFT, bool SUMS>
static cudaError_t f32tc_launch(const F32TcMaps& maps, const F32TcParams& p, int items, int sms, cudaStream_t st) {
  constexpr size_t smem = f32tc_smem<BN>();
  cudaError_t e = cudaFuncSetAttribute(f32tc_kernel<BN, ABFT, SUMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if constexpr (F32TcCfg<BN>::SPLIT_REGS) {
    // the hand-over draws on what the launch allocates
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, f32tc_kernel<BN, ABFT, SUMS>);
    if (e != cudaSuccess) return e;
    if (fa.numRegs != F32TcCfg<BN>::REGS) return cudaErrorInvalidConfiguration;
  }
  const int workers = items < sms / 2 ? items : sms / 2;
  return launch_pdl(f32tc_kernel<BN, ABFT, SUMS>, 2 * workers, F32TcCfg<BN>::THREADS, smem, st, maps, p);
}

// The product's tiles in one pass over K.
template <int BN>
static cudaError_t f32tc_product(bool abft, const F32TcMaps& maps, const F32TcParams& p, int sms, int* launches,
                                 cudaStream_t st) {
  ++*launches;
  return abft ? f32tc_launch<BN, true, false>(maps, p, p.tiles, sms, st)
              : f32tc_launch<BN, false, false>(maps, p, p.tiles, sms, st);
}

// The segments (checksums; the product too if it goes by segments), then the
// product in one pass or its scan.  bn: columns per tile; tail: tiles of 256
// columns left to a second launch.
template <int BN>
static cudaError_t f32tc_run_bn(bool abft, const F32TcMaps& maps, F32TcParams p, int tail, int sms, int* launches,
                                cudaStream_t st) {
  // the tile's shared arrays hold units of GC rows and columns or more
  if (abft && (p.um < F32TcCfg<BN>::GC || p.un < F32TcCfg<BN>::GC || p.um > 128 || p.un > 128)) return cudaErrorInvalidValue;
  if (abft || p.P) {
    const F32TcSums t = f32tc_sums<BN>(p);
    const long long items = ((long long)t.n[0] + t.n[1] + t.n[2]) * p.nsplit * p.sg.per_split;
    if (items > INT_MAX) return cudaErrorInvalidValue;
    cudaError_t e = f32tc_launch<BN, false, true>(maps, p, (int)items, sms, st);
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  if (p.P) return launch_f32tc_scan(abft, p, launches, st);
  const long long items = (long long)p.nsplit * p.tiles_m2 * p.tiles_n;
  if (items > INT_MAX || tail < 0 || tail >= items || (tail && BN != 256)) return cudaErrorInvalidValue;
  p.tiles = (int)items - tail;
  cudaError_t e = f32tc_product<BN>(abft, maps, p, sms, launches, st);
  if (e != cudaSuccess || !tail) return e;
  p.half_first = p.tiles;
  p.tiles = 2 * tail;
  return f32tc_product<128>(abft, maps, p, sms, launches, st);
}

cudaError_t launch_f32tc(int bn, int tail, bool abft, const F32TcMaps& maps, const F32TcParams& p, int sms,
                         int* launches, cudaStream_t st) {
  return bn == 256 ? f32tc_run_bn<256>(abft, maps, p, tail, sms, launches, st)
                   : f32tc_run_bn<128>(abft, maps, p, tail, sms, launches, st);
}

}  // namespace ftg
