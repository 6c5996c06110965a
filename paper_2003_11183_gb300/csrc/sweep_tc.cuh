// The integrand of a whole diagonal tile i in one kernel (Algorithm 6's per-tile step with eq. 2 over the
// tile): the tile's low-rank limit shifts, the sweep with its in-tile coupling, and the tile's projections
// for the later tiles, the products on the tensor cores.
//
// Four warps of a CTA own 128 samples, one per thread and per TMEM lane. The tile runs in sub-tiles of 64 variables. The
// sums that sub-tile q starts from are accumulated, by tcgen05 products issued by one thread, in 64 TMEM columns:
//     T[c][v] = sum_k U_i[q0 + v][k] W[k][c]           (the low-rank shifts: W the
//               rank-major projections of the earlier tiles, read MN-major; U
//               the tile's rows of the row factors; 16-bit operands, fp32 accumulation)
//             + sum_{u < q0} B_i[q0 + v][u] y_u[c]     (the coupling to the tile's
//               earlier sub-tiles: the CTA's own rows of the sample-major y, hi
//               and lo 16-bit parts, times the split copy of B_i, hi*hi + hi*lo +
//               lo*hi)
// for v < 64, the same sums as eq. 2 regrouped.  Each thread then runs the
// sub-tile's chain for its sample: 16 variables at a time, their sums over the
// sub-tile's earlier blocks accumulated together, then the block in order, each
// variable pushing its y into a shifting window of the block's later sums.  The
// products' sums come from the thread's TMEM lane (tcgen05.ld); the y of the
// sub-tile go to the same lane, into the columns whose sums have been read
// (tcgen05.st).  After each block its y are stored, sample-major 16-bit hi and
// lo, for the later products.  After the last sub-tile come the
// tile's projections W[k][c] = sum_v V_i[k][v] y_v[c], in steps of 64 ranks through
// the same columns, written as rows of W.  So neither the shifts nor the
// coupling go through global memory, the per-variable loads of B are
// shared-memory broadcasts, and the sample's log P is closed once per tile.
//
// Shared memory per CTA: stages of MMA operands (24 KB; float32 28), staged by TMA (128-byte swizzle where 64 deep, 64-byte
// where 32 deep), and what the sweep reads: a 96-byte record per
// variable (its window column of B, limits, reciprocal diagonal, lattice generator) and
// the six 16 x 16 blocks of the sub-tile's triangle that lie left of the windows.  Every wait is bounded; on expiry the
// CTA records an error code, skips the rest, waits (bounded) for its copies and products in flight, frees its
// TMEM and returns.
//
// What bounds it: the chain from a variable's sum to its y (about 110 instructions, most
// of them dependent) and, with six CTAs per SM, the issue slots; the arithmetic pipe
// (compares, selects, integer operations: half the rate of the FMA pipe) came first
// with 64 of 176 instructions a variable, so the step avoids them: see
// sov_step_f32_upper.  With that step, the constants' loads beside the products and the pairwise
// renormalisation and TMEM stores: n = 65,536, 20 x 5,000 samples, tiles of 512: 73.5 -> 60.4 ms a solve; n =
// 16,384, 10 x 1,000, tiles of 256: 10.0 -> 7.2 ms; two-sided limits (n = 3,900, 8 x 1,301): 4.43 -> 1.99 ms.  With one
// launch for all tiles (k_sweep_tc): 57.4, 6.77, 1.85; with the products beside the sweep (StcPlan) and the projections'
// row numbers read into shared memory together: 56.8, 5.94, 1.60.
#pragma once
#include "gemm.cuh"
#include "tcgen05.cuh"
#include "sweep.cuh"

namespace tlrmvn {

// Arithmetic of the products:
//   STC_BF16, STC_FP16  16-bit operands, the coupling's split into hi and lo parts (the BF16- and FP16-shift paths)
//   STC_FP32            every operand split into fp16 parts: the FP32 path's.  The tensor cores accumulate float32
//                       sums by truncation, which in one accumulator shifts a sum of 512 terms by about 1e-6 of
//                       itself, always towards zero (ten times the error of float32 FMAs).  So the factor's operands
//                       are scaled by powers of two into [-1, 1] (each row of U and of the tile's part left of the
//                       sub-tile, each row of V) and the projections to order 1, and hi parts are rounded to multiples
//                       of 2^-7 (the factor's) and 2^-11 (y, projections): the products hi*hi are multiples of 2^-18
//                       and their sums, below 64, exact; the other products (hi*lo, lo*hi, lo*lo), 2^-7 of those,
//                       have an accumulator of their own (128 TMEM columns).  The factor's operands have a third
//                       part, and hi*third is added there: their rounding to two parts, the same for all samples, was
//                       the largest error left, and the third part lets their grid be coarse.  With 2^-10 for
//                       both, sums were exact below 16 only, and rows of many equal entries pass that: the mean error of
//                       the samples' logs, as a share of them, 1.8e-7 at n = 512, b = -1, all entries 0.05 (now
//                       7e-9; float32 FMAs 4.5e-8), 1.8e-7 at n = 2,048, b = -3, positive random entries (6e-9; 5e-9).
//                       Errors of the samples' logs against 64 bits (rms; float32 FMAs in brackets): n = 2,000 points,
//                       tiles of 256, exponential kernel of range 0.1, b = -2: 9.8e-6 (1.5e-5), b = 1: 2.3e-6 (3.8e-6);
//                       range 0.5, b = 0: 5.9e-6 (6.2e-6); range 3, b = 0: 1.0e-5 (7.9e-6), b = 3: 1.3e-6 (2.4e-6).
//                       y is held to 23 bits, so sums that a few large y make up are less exact: all entries
//                       0.05, b = -5: 4.2e-5 of 327 (2.7e-5), b = -20: 1.8e-3 of 4,320 (4.6e-4).  Times against the float32 FMA products and sweeps: n = 16,384, 20
//                       x 5,000 samples: 55.0 -> 25.9 ms a solve; n = 4,096, nu = 7, 10 x 1,000: 4.41 -> 2.35 ms; 64
//                       batched problems, 10 x 2,000: 87.9 -> 18.8 ms.
enum StcMode { STC_BF16 = 0, STC_FP16 = 1, STC_FP32 = 2 };
constexpr int STC_SUB = 64;   // variables per sub-tile
constexpr int STC_NS = 128;   // samples per CTA (TMEM lanes)
constexpr int STC_KB = 32;    // K depth of a coupling k-block
// The largest y and projection that the operands hold (STC_FP32: with a margin for the grid of its leading parts).
__host__ __device__ constexpr float stc_range(int mode) {
  return mode == STC_FP32 ? 32768.0f : (mode == STC_FP16 ? 65504.0f : 3.38e38f);
}
using StcCfg = tc::Cfg<64, true, false, STC_KB, 1>;
using StcShiftCfg = tc::Cfg<64, false, true, 64, 1>;  // 16-bit shift k-block: W (MN-major) x U rows, 64 deep
using StcProjCfg = tc::Cfg<64, false, false, 64, 1>;  // 16-bit projection k-block: y rows x V rows, 64 deep
static_assert(StcProjCfg::SB == StcCfg::SB && StcShiftCfg::SB == StcCfg::SB, "they fill the same stage");

// The 16-bit operand type of the products: bf16 (BF16-shift path) or fp16
// (FP16-shift path), as raw 16-bit words.  pack rounds two floats to the type
// (round to nearest even) and returns them packed low word first, with their
// rounded values in ra, rb.
template <bool F16>
struct Op16;
template <>
struct Op16<false> {
  static __device__ __forceinline__ uint32_t pack(float a, float b, float& ra, float& rb) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    ra = __low2float(h);
    rb = __high2float(h);
    return ((uint32_t)__bfloat16_as_ushort(h.y) << 16) | __bfloat16_as_ushort(h.x);
  }
  static __device__ __forceinline__ unsigned short one(float a) { return __bfloat16_as_ushort(__float2bfloat16_rn(a)); }
};
template <>
struct Op16<true> {
  static __device__ __forceinline__ uint32_t pack(float a, float b, float& ra, float& rb) {
    const __half2 h = __floats2half2_rn(a, b);
    ra = __low2float(h);
    rb = __high2float(h);
    return ((uint32_t)__half_as_ushort(h.y) << 16) | __half_as_ushort(h.x);
  }
  static __device__ __forceinline__ unsigned short one(float a) { return __half_as_ushort(__float2half_rn(a)); }
};

// hi and lo fp16 parts of two floats for STC_FP32, packed low word first: hi a multiple of 2^-11 (of more above 1)
__device__ __forceinline__ void split_f32(float a, float b, uint32_t& hi, uint32_t& lo) {
  float ha, hb, la, lb;
  hi = Op16<true>::pack((a + 6144.0f) - 6144.0f, (b + 6144.0f) - 6144.0f, ha, hb);
  lo = Op16<true>::pack(a - ha, b - hb, la, lb);
}

// Per variable: [0, 16) the window column (for an even variable v B[v+2+k][v] at k < 14 and B[v+1][v] at 14,
// so that the pair update of the sweep reads aligned pairs; for an odd one B[v+1+k][v] at k < 15),
// then a, b, 1 / B_vv and (STC_FP32) the inverse of its row's scale, the lattice generator (8 bytes) and 8 spare bytes.
constexpr int STC_REC = 24;  // floats
// Entries after the lattice shifts' table: a sample's row is read up to three entries past a tile's last variable.
constexpr int STC_DPAD = 4;

// A diagonal tile: its first variable and size, its rank rows of W (first, count), its column ranks (first, count),
// and how many of its first ranks come from tiles before the one before it.
struct StcTile {
  int t0, mt, krow0, kr, kcol0, kc, kearly, pad;
};
// A tile for the sweeping warps.
struct SweepTcArgs {
  const float* rec;  // the factor's records at the tile's first variable (limits not filled in)
  const float* BT;   // transposed diagonal tile, BT[u * ldbt + v] = B[v][u]
  int64_t ldbt;
  int mt;            // variables in the tile
  const float* a;    // limits at the tile's first variable
  const float* b;
  int64_t ys_lo;     // offset of the lo parts in a sample's row of y
  int kr, kc;        // the tile's ranks (0: no low-rank shift), its column ranks (0: no projection)
  int64_t ldw;       // projections, rank-major: row vmap[r], ldw samples a row
  const int32_t* vmap;    // at the tile's first column rank
  const float* wscale;    // FP16 path: per column rank, the factor applied to a projection before it is
                          // stored (the inverse of the per-tile scales of U and V); null on the BF16 path
  float tscale;           // FP16 path: 1 / g, undoing the products' global scale g where the sweep reads them
  const float* rscale;    // STC_FP32: per variable of the tile, the inverse of its row's scale
  StcTile t;              // the tile (for the products)
  int wlo;                // STC_FP32: the lo parts' row offset in W
  int* err;               // [0] a bounded wait's code; [1] (STC_FP32, STC_FP16) a y or a projection beyond fp16's range

  // from the arguments as of tile 0, variable 0 and column rank 0 to those of tile i of at most m variables
  __device__ void at(const StcTile& tile, int i, int m) {
    t = tile;
    rec += (int64_t)i * m * STC_REC;
    BT += (int64_t)i * m * ldbt;
    mt = t.mt;
    a += t.t0;
    b += t.t0;
    kr = t.kr;
    kc = t.kc;
    vmap += t.kcol0;
    wscale += t.kcol0;
    rscale += (int64_t)i * m;
  }
};
constexpr int STC_ARGS = 256;  // shared memory of a tile's arguments
static_assert(sizeof(SweepTcArgs) <= STC_ARGS, "the arguments' place");
// The operands for the producing thread: tensor maps (32-deep boxes; 16-bit W, U and V, and mapYp, 64-deep), x offsets of the lo halves in the y and split-B maps,
// STC_FP32: of the lo parts in the W (rows), U and V maps (third parts: twice).
struct StcOps {
  const CUtensorMap *mapY, *mapYp, *mapB, *mapW, *mapU, *mapV;
  int alo, blo, wlo, ulo, vlo;
  int* err;
};

constexpr int STC_TRI = 6 * 256;  // floats: the 16 x 16 blocks (ub, vb), ub < vb, at vb (vb - 1) / 2 + ub
// A stage: [A hi][B hi][A lo][B lo] of a split k-block, 32 deep (STC_FP32: [B third] too), or [A][B] of a 16-bit shift
// or projection k-block, 64 deep.
__host__ __device__ constexpr uint32_t stc_stage_bytes(int mode) {
  return StcCfg::SB + (mode == STC_FP32 ? StcCfg::B_BYTES : 0);
}
// [NST stages][records][triangle blocks][barriers, TMEM slot, a tile][a tile's arguments] (the dynamic shared memory starts
// 1 KB-aligned: the kernels have no static shared memory, and the system's own part is 1 KB)
__host__ __device__ constexpr size_t sweep_tc_smem_bytes(int mode, int nst) {
  return (size_t)nst * stc_stage_bytes(mode) + (STC_SUB * STC_REC + STC_TRI) * sizeof(float) + 256 + STC_ARGS;
}
// TMEM columns of one accumulator (the sums, then the y, of a sub-tile; STC_FP32: and the second sums).
__host__ __device__ constexpr uint32_t stc_cols(int mode) { return mode == STC_FP32 ? 2 * STC_SUB : STC_SUB; }

// The producing thread's place: k-blocks gone through the stages, steps begun, steps whose first half and whole the
// sweeping warps are known to have done (overlapped), k-blocks of the coming step under way (otherwise).
struct StcRun {
  uint32_t count, step, half, whole;
  int pre;
};

// Shared-memory layout and per-CTA state of the whole-tile sweep (set up once per kernel).
struct StcCta {
  unsigned char* stage;
  float* rec;            // the sub-tile's records
  float* tri;            // its triangle blocks
  uint64_t* full;        // [NST] the stage's copies landed
  uint64_t* freeb;       // [NST] the products reading the stage are done
  uint64_t* acc;         // [2] the accumulator's products are done
  uint64_t* ready;       // [2] a step's first half, its whole is done (one arrival per sweeping warp)
  uint32_t tmem;         // first of the CTA's TMEM columns
  int* abort_flag;
  int* item;             // (persistent kernel) the work item
  SweepTcArgs* args;     // (k_sweep_tc) the tile's arguments
  StcTile* next;         // (k_sweep_tc) the coming tile
};

// Where the CTA's samples sit in the operand maps and the result buffers.
struct StcPlace {
  int wx;                // x coordinate of the CTA's first sample in the W map (samples are columns)
  int wy;                // row added to the tile's rank rows in the W map
  int yrow;              // row coordinate of the CTA's first sample in the y maps (samples are rows)
  unsigned short* ysrow; // the thread's row of sample-major y (hi; lo at + ys_lo)
  unsigned short* wcol;  // the thread's column of W (row k at wcol[k * ldw])
};

__device__ __forceinline__ void tmem_ld16(uint32_t (&r)[16], uint32_t addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
// Bounded wait: false when the limit expires (the error code set) or the CTA has given up.
__device__ __forceinline__ bool stc_wait(const StcCta& k, uint64_t* bar, uint32_t parity, int* err, int code) {
  for (uint32_t i = 0; i < tc::WAIT_LIMIT; i++) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    if ((i & 255) == 255 && *(volatile int*)k.abort_flag) return false;
  }
  atomicExch(err, code);
  return false;
}

// Who issues the products.  Overlapped (a launch of at most two CTAs an SM): a fifth warp's first thread, into two
// accumulators by turns, so that most of a step's products (a step: a sub-tile, or a projection pass) run while the
// step before is swept.  Otherwise thread 0 of the four sweeping warps, between the steps, one accumulator: with six CTAs
// an SM (float32: three) the others' sweeps fill that time.  A fifth warp's registers and a second accumulator
// leave four (two), and those are slower as soon as there are samples for more than two: n = 65,536, 20 x 5,000: 74 against
// 57 ms; two CTAs an SM, n = 8,192, 38,000 samples, tiles of 512: bf16 3.44 against 3.95 ms, float32 3.96
// against 4.86; one: n = 16,384, 10 x 1,000: 5.94 against 6.77; float32, n = 1,024: 0.55 against 0.61.
template <bool OV>
struct StcPlan;
template <>
struct StcPlan<true> {
  static constexpr int THREADS = 160, NBUF = 2;
};
template <>
struct StcPlan<false> {
  static constexpr int THREADS = 128, NBUF = 1;
};
__host__ __device__ constexpr int stc_stages(int mode, bool ov) {
  return mode == STC_FP32 ? (ov ? 3 : 2) : (ov ? 4 : 1);
}
// CTAs per SM: six (80 registers a thread), STC_FP32 three; overlapped two.
__host__ __device__ constexpr int stc_ctas(int mode, bool ov) { return ov ? 2 : (mode == STC_FP32 ? 3 : 6); }

// Step u of a tile: its k-blocks are nsh of ranks, then those of y.
template <int MODE>
struct StcStep {
  static constexpr bool SPLIT = MODE == STC_FP32;
  static constexpr int KS = SPLIT ? STC_KB : 64;  // depth of a shift or projection k-block
  int nsub, q0, r0, nsh, nk;
  bool proj;
  __device__ StcStep(const StcTile& t, int u) {
    nsub = (t.mt + STC_SUB - 1) / STC_SUB;
    proj = u >= nsub;
    q0 = u * STC_SUB;
    r0 = (u - nsub) * STC_SUB;
    nsh = proj ? 0 : (t.kr + KS - 1) / KS;
    nk = proj ? (t.mt + KS - 1) / KS : nsh + q0 / STC_KB;
  }
  // What k-block kb waits for, overlapped: nothing, the first half (32 variables) of the step before (1), all of it (2).
  __device__ int gate(const StcTile& t, int u, int kb) const {
    if (kb < nsh) return u == 0 && kb >= t.kearly / KS ? 2 : 0;
    const int j = kb - nsh;
    if (!proj) return j < nk - nsh - 2 ? 0 : (j == nk - nsh - 2 ? 1 : 2);
    if (u > nsub) return 0;
    if (!SPLIT) return j < nsub - 1 ? 0 : 2;
    return j < 2 * (nsub - 1) ? 0 : (j == 2 * (nsub - 1) ? 1 : 2);
  }
  // Starts the copies of k-block kb into stage st.
  __device__ void load(const StcOps& o, const StcTile& t, int row0, const StcCta& k, const StcPlace& pl, int kb,
                       uint32_t st) const {
    constexpr uint32_t A = StcCfg::A_BYTES, HALF = StcCfg::HALF, SB = stc_stage_bytes(MODE), B3 = 2 * HALF;
    unsigned char* s = k.stage + st * SB;
    uint64_t* bar = k.full + st;
    tc::mbar_expect_tx(bar, SB);
    if (kb < nsh) {  // two 64-sample MN-major boxes of W, a box of U rows
      const int y = pl.wy + t.krow0 + kb * KS;
      if constexpr (SPLIT) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
          tc::tma_load_2d(s + h * HALF, o.mapW, bar, pl.wx, y + h * o.wlo);
          tc::tma_load_2d(s + h * HALF + A / 2, o.mapW, bar, pl.wx + 64, y + h * o.wlo);
          tc::tma_load_2d(s + h * HALF + A, o.mapU, bar, kb * KS + h * o.ulo, row0 + q0);
        }
        tc::tma_load_2d(s + B3, o.mapU, bar, kb * KS + 2 * o.ulo, row0 + q0);
      } else {
        tc::tma_load_2d(s, o.mapW, bar, pl.wx, y);
        tc::tma_load_2d(s + StcShiftCfg::A_BYTES / 2, o.mapW, bar, pl.wx + 64, y);
        tc::tma_load_2d(s + StcShiftCfg::A_BYTES, o.mapU, bar, kb * KS, row0 + q0);
      }
    } else if (!SPLIT && proj) {
      tc::tma_load_2d(s, o.mapYp, bar, kb * KS, pl.yrow);
      tc::tma_load_2d(s + StcProjCfg::A_BYTES, o.mapV, bar, kb * KS, t.kcol0 + r0);
    } else {
      const int x = (kb - nsh) * STC_KB;
      const CUtensorMap* mb = proj ? o.mapV : o.mapB;
      const int lo = proj ? o.vlo : o.blo, y = proj ? t.kcol0 + r0 : row0 + q0;
      tc::tma_load_2d(s, o.mapY, bar, x, pl.yrow);
      tc::tma_load_2d(s + HALF, o.mapY, bar, o.alo + x, pl.yrow);
      tc::tma_load_2d(s + A, mb, bar, x, y);
      tc::tma_load_2d(s + HALF + A, mb, bar, lo + x, y);
      if constexpr (SPLIT) tc::tma_load_2d(s + B3, mb, bar, 2 * lo + x, y);
    }
  }
  // Issues its products into the accumulator at d (STC_FP32: all but hi x hi at d + 64).
  __device__ void mma(const StcCta& k, int kb, uint32_t st, uint32_t d) const {
    constexpr bool F16 = MODE != STC_BF16;
    constexpr uint32_t ID_K = F16 ? StcCfg::IDESC_F16 : StcCfg::IDESC;            // A K-major (y)
    constexpr uint32_t ID_M = F16 ? StcShiftCfg::IDESC_F16 : StcShiftCfg::IDESC;  // A MN-major (W)
    constexpr uint32_t A = StcCfg::A_BYTES, HALF = StcCfg::HALF;
    const uint32_t sa = tc::smem_u32(k.stage) + st * stc_stage_bytes(MODE);
    const bool sh = kb < nsh;
    if (!SPLIT && (sh || proj)) {
      // per 16-deep step MN-major W is two 1 KB K groups on (+128), K-major rows 32 bytes (+2)
      const uint64_t da = sh ? tc::sdesc_mn(sa, StcShiftCfg::A_BYTES / 2) : tc::sdesc<64>(sa);
      const uint64_t db = tc::sdesc<64>(sa + StcShiftCfg::A_BYTES), step = sh ? 128 : 2;
#pragma unroll
      for (int kk = 0; kk < 4; kk++)
        tc::mma_f16(d, da + step * (uint64_t)kk, db + (uint64_t)(2 * kk), sh ? ID_M : ID_K, (kb > 0 || kk > 0) ? 1u : 0u);
      return;
    }
    const uint64_t ah = SPLIT && sh ? tc::sdesc_mn(sa, A / 2) : tc::sdesc<STC_KB>(sa);
    const uint64_t al = SPLIT && sh ? tc::sdesc_mn(sa + HALF, A / 2) : tc::sdesc<STC_KB>(sa + HALF);
    const uint64_t bh = tc::sdesc<STC_KB>(sa + A), bl = tc::sdesc<STC_KB>(sa + HALF + A);
    const uint64_t step = SPLIT && sh ? 128 : 2;
    const uint32_t id = SPLIT && sh ? ID_M : ID_K, d2 = SPLIT ? d + STC_SUB : d;
#pragma unroll
    for (int kk = 0; kk < STC_KB / 16; kk++) {
      const uint64_t oa = step * (uint64_t)kk, ob = (uint64_t)(2 * kk);
      const uint32_t acc = (kb > 0 || kk > 0) ? 1u : 0u;
      tc::mma_f16(d, ah + oa, bh + ob, id, acc);
      tc::mma_f16(d2, ah + oa, bl + ob, id, SPLIT ? acc : 1u);
      tc::mma_f16(d2, al + oa, bh + ob, id, 1u);
      if constexpr (SPLIT) {
        tc::mma_f16(d2, al + oa, bl + ob, id, 1u);
        tc::mma_f16(d2, ah + oa, tc::sdesc<STC_KB>(sa + 2 * HALF) + ob, id, 1u);
      }
    }
  }
};

// The products of step u of a tile, by one thread: its k-blocks through a ring of NST stages, then the accumulator's
// barrier.  Overlapped, a step's accumulator is complete only after the step before it has been swept, but most of its
// k-blocks need nothing of that step: all but the last two of a sub-tile's coupling and of the first projection pass
// (the first of these waits for the step's first half), and all but the ranks of the tile before in a tile's first shift.
// Returns false (its copies and products in flight waited for, bounded) when a wait expired or the CTA gave up.
template <int MODE, int NST, bool OV>
__device__ __forceinline__ bool stc_products(const StcOps& o, const StcTile& t, int row0, const StcCta& k,
                                             const StcPlace& pl, int u, StcRun& r) {
  const StcStep<MODE> s(t, u);
  // the step before is swept: its first 32 variables, or all
  auto swept = [&](bool whole) -> bool {
    if (r.half < r.step) {
      if (!stc_wait(k, k.ready, (r.step - 1) & 1, o.err, 6)) return false;
      r.half = r.step;
    }
    if (whole && r.whole < r.step) {
      if (!stc_wait(k, k.ready + 1, (r.step - 1) & 1, o.err, 7)) return false;
      r.whole = r.step;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return true;
  };
  const uint32_t buf = OV ? r.step & 1 : 0;
  int issued = OV ? 0 : r.pre, kb = 0;
  bool ok = true;
  for (; kb < s.nk; kb++) {
    for (; issued < s.nk && issued < kb + NST; issued++) {
      if constexpr (OV) {
        const int g = s.gate(t, u, issued);
        if (g != 0 && (g == 1 ? r.half : r.whole) < r.step) {
          if (issued > kb) break;  // (first the products of what has been loaded)
          if (!swept(g == 2)) {
            ok = false;
            break;
          }
        }
      }
      const uint32_t i = r.count + (uint32_t)issued;
      if (i >= NST && !stc_wait(k, k.freeb + i % NST, (i / NST - 1) & 1, o.err, 9)) {
        ok = false;
        break;
      }
      s.load(o, t, row0, k, pl, issued, i % NST);
    }
    const uint32_t i = r.count + (uint32_t)kb;
    if (!ok || !stc_wait(k, k.full + i % NST, (i / NST) & 1, o.err, 8)) {
      ok = false;
      break;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    s.mma(k, kb, i % NST, k.tmem + buf * stc_cols(MODE));
    tc::mma_commit(k.freeb + i % NST);
  }
  if (OV && ok) ok = swept(true);
  if (!ok) {
    *(volatile int*)k.abort_flag = 1;
    for (int j = kb; j < issued; j++) {  // copies in flight
      const uint32_t i = r.count + (uint32_t)j;
      tc::mbar_wait(k.full + i % NST, (i / NST) & 1, o.err, 5);
    }
    if (r.count + (uint32_t)kb > 0) {  // products in flight (they complete in order)
      const uint32_t i = r.count + (uint32_t)kb - 1;
      tc::mbar_wait(k.freeb + i % NST, (i / NST) & 1, o.err, 5);
    }
    return false;
  }
  r.count += (uint32_t)s.nk;
  r.pre = 0;
  if (s.nk > 0) tc::mma_commit(k.acc + buf);
  else mbar_arrive(k.acc + buf);
  r.step++;
  return true;
}
// Not overlapped, after a step's products: the copies of the next sub-tile's first shift k-blocks, which land during
// the sweep (W and U are complete, all products have read their stages).
template <int MODE, int NST>
__device__ __forceinline__ void stc_prefetch(const StcOps& o, const StcTile& t, int row0, const StcCta& k,
                                             const StcPlace& pl, int u, StcRun& r) {
  const StcStep<MODE> s(t, u);
  if (s.proj) return;
  for (; r.pre < NST && r.pre < s.nsh; r.pre++) s.load(o, t, row0, k, pl, r.pre, (r.count + (uint32_t)r.pre) % NST);
}
// Overlapped: all products of a tile.
template <int MODE, int NST>
__device__ __forceinline__ bool stc_produce(const StcOps& o, const StcTile& t, int row0, const StcCta& k,
                                            const StcPlace& pl, StcRun& r) {
  const int steps = (t.mt + STC_SUB - 1) / STC_SUB + (t.kc + STC_SUB - 1) / STC_SUB;
  for (int u = 0; u < steps; u++)
    if (!stc_products<MODE, NST, true>(o, t, row0, k, pl, u, r)) return false;
  return true;
}

// A barrier of the sweeping warps; true (to all of them) when a wait before it failed.
template <bool OV>
__device__ __forceinline__ bool stc_bar(const StcCta& k, bool failed) {
  if constexpr (OV) {
    uint32_t any;
    __syncwarp();
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, 128, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(any)
        : "r"(failed ? 1u : 0u)
        : "memory");
    if (any) *(volatile int*)k.abort_flag = 1;
    return any != 0;
  } else {  // (thread 0 alone waits, and sets the flag)
    __syncthreads();
    return *(volatile int*)k.abort_flag != 0;
  }
}
// The arguments of tile i (of end, the largest of m variables) for the sweeping warps; base: those as of tile 0.  The
// tile after it is copied during the sweep.
template <bool OV>
__device__ __forceinline__ void stc_args(const StcCta& k, const SweepTcArgs& base, const StcTile* tiles, int i, int end,
                                         int m, bool first) {
  stc_bar<OV>(k, false);  // those of the tile before read by all
  if (threadIdx.x == 0) {
    SweepTcArgs p = base;
    p.at(first ? tiles[i] : *k.next, i, m);
    *k.args = p;
    if (i + 1 < end) {
      cp_async16(reinterpret_cast<float4*>(k.next), reinterpret_cast<const float*>(tiles + i + 1), 16);
      cp_async16(reinterpret_cast<float4*>(k.next) + 1, reinterpret_cast<const float*>(tiles + i + 1) + 4, 16);
      cp_async_commit();
    }
  }
  stc_bar<OV>(k, false);
}

// The warp's part of the step's first half (0) or whole (1) is done, its y or projections visible to copies, its TMEM
// accesses complete.
template <bool OV>
__device__ __forceinline__ void stc_done(const StcCta& k, int which) {
  asm volatile("fence.proxy.async;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if constexpr (OV) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(k.ready + which);
  }
}

// In FLAGS, for the batched kernel: its W goes from problem to problem, and one's padding rows, times zero, lie where
// another's projections were, so these have to stay finite (y is by itself: ndtri_tail_f32).  (The check costs a solve
// of n = 65,536 0.4 of 56.7 ms.)
constexpr int STC_GUARD = 4;

// One diagonal tile for the CTA's samples, by the sweeping warps: the float sweep of eq. 2 and the projections, of the
// products' sums.  step: steps so far.  o, run, row0: thread
// 0's, to issue the products when no other warp does.  act: the thread's
// sample exists (else it shadows one and writes nothing); Ds: its row of lattice shifts
// (read up to three entries past the tile); ks: its point
// index; rs: its MVT scale (1 for MVN).  The tile's log P is added to (prod, pe, lsum).
// Returns false (to all sweeping warps) when a bounded wait expired.
template <int FLAGS, int MODE, int NST, bool OV>
__device__ __forceinline__ bool stc_tile(const SweepTcArgs& p, const StcCta& k, const StcPlace& pl, uint32_t& step,
                                         const StcOps& o, StcRun& run, int row0, const bool act, const uint64_t* Ds, const uint32_t ks,
                                         const float rs,
                                         float& prod, float& lsum, int& pe) {
  constexpr bool PER = FLAGS & SWEEP_PERIODIZE, ONE = FLAGS & SWEEP_ONE_SIDED;
  constexpr bool F16 = MODE != STC_BF16, SPLIT = MODE == STC_FP32, GUARD = FLAGS & STC_GUARD;
  using Op = Op16<F16>;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int mt = p.mt;
  const uint32_t tmem = k.tmem + ((uint32_t)(32 * warp) << 16);  // this warp's 32 lanes
  for (int q0 = 0; q0 < mt; q0 += STC_SUB, step++) {
    const int mq = min(STC_SUB, mt - q0);
    const uint32_t buf = OV ? step & 1 : 0, tl = tmem + buf * stc_cols(MODE);
    stc_bar<OV>(k, false);  // every sweeping thread is past the previous sub-tile's reads of the records and its accumulator
    if (!OV && tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      stc_products<MODE, NST, OV>(o, p.t, row0, k, pl, q0 / STC_SUB, run);
    }
    if (OV || tid >= 32) {
      constexpr int T0 = OV ? 0 : 32;  // (the warp that issues the products is late)
      for (int t = tid - T0; t < mq * 6; t += STC_NS - T0) {
        const int v = t / 6, c = t - v * 6;
        const float* src = p.rec + (int64_t)(q0 + v) * STC_REC + 4 * c;
        if (c == 4)
          reinterpret_cast<float4*>(k.rec)[t] =
              make_float4(p.a[q0 + v], p.b[q0 + v], __ldg(src + 2), SPLIT ? __ldg(p.rscale + q0 + v) : 0.0f);
        else
          cp_async16(reinterpret_cast<float4*>(k.rec) + t, src, 16);
      }
      for (int t = tid - T0; t < STC_TRI / 4; t += STC_NS - T0) {
        const int blk = t >> 6, u = (t >> 2) & 15, c = t & 3;
        const int vb = blk < 1 ? 1 : (blk < 3 ? 2 : 3), ub = blk - vb * (vb - 1) / 2;
        if (16 * vb < mq)
          cp_async16(reinterpret_cast<float4*>(k.tri) + t,
                     p.BT + (int64_t)(q0 + 16 * ub + u) * p.ldbt + q0 + 16 * vb + 4 * c, 16);
      }
      cp_async_commit();
    }
    bool ok = true;  // (not overlapped, the others wait at the barrier: their polls would take the other CTAs' issue slots)
    if (OV || tid == 0) ok = stc_wait(k, k.acc + buf, (OV ? step >> 1 : step) & 1, p.err, 4);
    if (!OV && !ok) *(volatile int*)k.abort_flag = 1;
    if (!OV && tid == 0 && ok) stc_prefetch<MODE, NST>(o, p.t, row0, k, pl, q0 / STC_SUB + 1, run);
    cp_async_wait<0>();
    // records and triangle staged; shifts and coupling are in TMEM
    if (stc_bar<OV>(k, !ok)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    const uint64_t* Dp = Ds + p.t.t0 + q0;
    uint64_t d0 = Dp[0], d1 = Dp[1];  // the lattice shifts of a pair of variables, loaded one pair ahead
    for (int v0 = 0; v0 < mq; v0 += DIAG_VB) {
      const int nb = min(DIAG_VB, mq - v0);
      // acc[i] = sums of the block's variables 2i (x) and 2i + 1 (y), as pairs for the
      // paired float32 FMAs (each pair FMA rounds as two fmaf)
      float2 acc[DIAG_VB / 2];
      if (q0 > 0 || p.kr > 0) {
        uint32_t r[DIAG_VB];
        tmem_ld16(r, tl + (uint32_t)v0);
        if constexpr (SPLIT) {
          uint32_t l[DIAG_VB];
          tmem_ld16(l, tl + (uint32_t)(STC_SUB + v0));
          const float* sc = k.rec + v0 * STC_REC + 19;  // (rows past a ragged tile: stale, unused)
#pragma unroll
          for (int j = 0; j < DIAG_VB / 2; j++)
            acc[j] = make_float2(
                (__uint_as_float(r[2 * j]) + __uint_as_float(l[2 * j])) * sc[2 * j * STC_REC],
                (__uint_as_float(r[2 * j + 1]) + __uint_as_float(l[2 * j + 1])) * sc[(2 * j + 1) * STC_REC]);
        } else {
#pragma unroll
          for (int j = 0; j < DIAG_VB / 2; j++)
            acc[j] = F16 ? make_float2(__uint_as_float(r[2 * j]) * p.tscale, __uint_as_float(r[2 * j + 1]) * p.tscale)
                         : make_float2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
        }
      } else {
#pragma unroll
        for (int j = 0; j < DIAG_VB / 2; j++) acc[j] = make_float2(0.0f, 0.0f);
      }
      // sums over the sub-tile's earlier blocks for the block's 16 variables: y_u from this lane's TMEM columns
      const float* tri = k.tri + 256 * ((v0 >> 4) * ((v0 >> 4) - 1) / 2);
      for (int u0 = 0; u0 < v0; u0 += DIAG_VB, tri += 256) {
        uint32_t r[DIAG_VB];
        tmem_ld16(r, tl + (uint32_t)u0);
#pragma unroll
        for (int uu = 0; uu < DIAG_VB; uu++) {
          const float4* b4 = reinterpret_cast<const float4*>(tri + uu * DIAG_VB);
          const float4 q[4] = {b4[0], b4[1], b4[2], b4[3]};
          const float2 yy = make_float2(__uint_as_float(r[uu]), __uint_as_float(r[uu]));
#pragma unroll
          for (int h = 0; h < 4; h++) {
            acc[2 * h] = __ffma2_rn(make_float2(q[h].x, q[h].y), yy, acc[2 * h]);
            acc[2 * h + 1] = __ffma2_rn(make_float2(q[h].z, q[h].w), yy, acc[2 * h + 1]);
          }
        }
      }
      // one variable of eq. 2: sum = its sum over the earlier variables and the shifts, rp its record; returns its y
      // and multiplies its probability into the product (renormalised by the caller once a pair)
      auto step = [&](const float* rp, uint64_t dv, float sum) -> float {
        const float4 abi = *reinterpret_cast<const float4*>(rp + 16);
        const uint64_t qv = *reinterpret_cast<const uint64_t*>(rp + 20);
        const float bt = fmaf(abi.y, rs, -sum) * abi.z;
        float w, wc, f, y;
        lattice_wf((uint64_t)ks * qv + dv, PER ? 1 : 0, w, wc);
        if (ONE) {
          sov_step_f32_upper<F16 ? (int)stc_range(MODE) : 0>(bt, w, wc, f, lsum, y);
        } else {
          const float at = fmaf(abi.x, rs, -sum) * abi.z;
          sov_step_f32_prod<F16 ? (int)stc_range(MODE) : 0>(at, bt, w, wc, f, lsum, y);
        }
        prod *= f;
        return y;
      };
      // the block's variables in pairs (v even, v + 1): after y_v the pair's second sum
      // takes B[v+1][v] y_v and the window moves two places, the later sums taking
      // B[v+2+k][v] y_v; after y_{v+1} they take B[v+2+k][v+1] y_{v+1} (k < 14: the
      // rest of the block).  Each sum receives its terms in the order of the variables.
      const float* rp = k.rec + v0 * STC_REC;
#pragma unroll 1
      for (int j = 0; j < nb; j += 2, rp += 2 * STC_REC) {
        const uint64_t n0 = Dp[2], n1 = Dp[3];  // (at most three entries past the tile)
        Dp += 2;
        const float y0 = step(rp, d0, acc[0].x);
        float y1 = 0.0f;
        if (j + 1 < nb) {  // (uniform; false for a ragged tile's last variable only)
          float sum;
          {
            const float4* b4 = reinterpret_cast<const float4*>(rp);
            const float4 q[4] = {b4[0], b4[1], b4[2], b4[3]};
            sum = fmaf(q[3].z, y0, acc[0].y);
            const float2 yy = make_float2(y0, y0);
#pragma unroll
            for (int h = 0; h < 3; h++) {
              acc[2 * h] = __ffma2_rn(make_float2(q[h].x, q[h].y), yy, acc[2 * h + 1]);
              acc[2 * h + 1] = __ffma2_rn(make_float2(q[h].z, q[h].w), yy, acc[2 * h + 2]);
            }
            acc[6] = __ffma2_rn(make_float2(q[3].x, q[3].y), yy, acc[7]);
            acc[7] = make_float2(0.0f, 0.0f);
          }
          y1 = step(rp + STC_REC, d1, sum);
          {
            const float4* b4 = reinterpret_cast<const float4*>(rp + STC_REC);
            const float4 q[4] = {b4[0], b4[1], b4[2], b4[3]};
            const float2 yy = make_float2(y1, y1);
#pragma unroll
            for (int h = 0; h < 3; h++) {
              acc[2 * h] = __ffma2_rn(make_float2(q[h].x, q[h].y), yy, acc[2 * h]);
              acc[2 * h + 1] = __ffma2_rn(make_float2(q[h].z, q[h].w), yy, acc[2 * h + 1]);
            }
            acc[6] = __ffma2_rn(make_float2(q[3].x, q[3].y), yy, acc[6]);
          }
        }
        d0 = n0;
        d1 = n1;
        // prod in [1, 2) times two factors of at least 2.5e-19 each: a normal float
        const int pb = __float_as_int(prod);
        pe += (pb >> 23) - 127;
        prod = __int_as_float((pb & 0x007FFFFF) | 0x3F800000);
        __syncwarp();  // (the steps' rare branch)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(tl + (uint32_t)(v0 + j)),
                     "r"(__float_as_uint(y0)), "r"(__float_as_uint(y1))
                     : "memory");
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      // the block's y, sample-major 16-bit hi and lo (32 bytes each per sample), for
      // the later sub-tiles' products (read back by TMA: async proxy) and the projection
      {
        uint32_t r[DIAG_VB];
        tmem_ld16(r, tl + (uint32_t)v0);
        if (act) {
          unsigned short* row = pl.ysrow + q0 + v0;
          uint32_t hi2[DIAG_VB / 2], lo2[DIAG_VB / 2];
          float top = 0.0f;
#pragma unroll
          for (int j = 0; j < DIAG_VB; j += 2) {
            const float y0 = __uint_as_float(r[j]), y1 = __uint_as_float(r[j + 1]);
            if constexpr (SPLIT) {
              split_f32(y0, y1, hi2[j / 2], lo2[j / 2]);
            } else {
              float h0, h1, l0, l1;
              hi2[j / 2] = Op::pack(y0, y1, h0, h1);
              lo2[j / 2] = Op::pack(y0 - h0, y1 - h1, l0, l1);
            }
            if (F16) top = fmaxf(top, j < nb ? fmaxf(fabsf(y0), fabsf(y1)) : 0.0f);
          }
          if (F16 && top >= stc_range(MODE)) p.err[1] = 1;  // (the step cuts y to it: what follows stays finite)
          if (nb == DIAG_VB) {
            uint4* dh = reinterpret_cast<uint4*>(row);
            uint4* dlo = reinterpret_cast<uint4*>(row + p.ys_lo);
            dh[0] = make_uint4(hi2[0], hi2[1], hi2[2], hi2[3]);
            dh[1] = make_uint4(hi2[4], hi2[5], hi2[6], hi2[7]);
            dlo[0] = make_uint4(lo2[0], lo2[1], lo2[2], lo2[3]);
            dlo[1] = make_uint4(lo2[4], lo2[5], lo2[6], lo2[7]);
          } else {
            unsigned short* rh = row;
            unsigned short* rl = row + p.ys_lo;
#pragma unroll
            for (int j = 0; j < DIAG_VB; j++)
              if (j < nb) {
                rh[j] = (unsigned short)(hi2[j / 2] >> (16 * (j & 1)));
                rl[j] = (unsigned short)(lo2[j / 2] >> (16 * (j & 1)));
              }
          }
        }
      }
      if (OV && v0 == STC_KB - DIAG_VB && mq > STC_KB) stc_done<OV>(k, 0);
    }
    if (OV && mq <= STC_KB) stc_done<OV>(k, 0);
    stc_done<OV>(k, 1);
  }
  // the tile's projections for the later tiles, 64 ranks a step: W[vmap[r]][c] = sum_v V[kcol0 + r][v] y_v[c]; the
  // rows' places and scales are in the records' and the triangle's, up to RANKS at a time
  constexpr int RANKS = STC_SUB * STC_REC;
  static_assert(RANKS <= STC_TRI && RANKS % STC_SUB == 0, "room for the scales");
  int32_t* const vm = reinterpret_cast<int32_t*>(k.rec);
  float* const ws = k.tri;
#pragma unroll 1
  for (int r0 = 0, rb = 0; r0 < p.kc; r0 += STC_SUB, step++) {
    const uint32_t buf = OV ? step & 1 : 0, tl = tmem + buf * stc_cols(MODE);
    if (!OV || r0 % RANKS == 0) stc_bar<OV>(k, false);  // every sweeping thread is done with those, and the accumulator
    if (!OV && tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      stc_products<MODE, NST, OV>(o, p.t, row0, k, pl, (mt + STC_SUB - 1) / STC_SUB + r0 / STC_SUB, run);
    }
    if (r0 % RANKS == 0) {
      rb = r0;
      for (int t = tid; t < RANKS && r0 + t < p.kc; t += STC_NS) {
        vm[t] = __ldg(p.vmap + r0 + t);
        if (F16) ws[t] = __ldg(p.wscale + r0 + t);
      }
    }
    bool ok = true;
    if (OV || tid == 0) ok = stc_wait(k, k.acc + buf, (OV ? step >> 1 : step) & 1, p.err, 4);
    if (!OV && !ok) *(volatile int*)k.abort_flag = 1;
    if (stc_bar<OV>(k, !ok)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
    for (int h = 0; h < 64; h += 16) {
      uint32_t r[16];
      tmem_ld16(r, tl + (uint32_t)h);
      if constexpr (SPLIT) {
        uint32_t l[16];
        tmem_ld16(l, tl + (uint32_t)(STC_SUB + h));
        if (act) {
          float top = 0.0f;
#pragma unroll
          for (int j = 0; j < 16; j += 2)
            if (r0 + h + j < p.kc) {
              const bool two = r0 + h + j + 1 < p.kc;
              const int rr = r0 + h + j, r1 = two ? rr + 1 : rr;
              const float w0 = (__uint_as_float(r[j]) + __uint_as_float(l[j])) * ws[rr - rb];
              const float w1 = (__uint_as_float(r[j + 1]) + __uint_as_float(l[j + 1])) * ws[r1 - rb];
              uint32_t hi, lo;
              split_f32(w0, w1, hi, lo);
              top = max_nan(top, fabsf(w0), two ? fabsf(w1) : 0.0f);
              unsigned short* d0 = pl.wcol + (int64_t)vm[rr - rb] * p.ldw;
              d0[0] = (unsigned short)hi;
              d0[(int64_t)p.wlo * p.ldw] = (unsigned short)lo;
              if (two) {
                unsigned short* d1 = pl.wcol + (int64_t)vm[r1 - rb] * p.ldw;
                d1[0] = (unsigned short)(hi >> 16);
                d1[(int64_t)p.wlo * p.ldw] = (unsigned short)(lo >> 16);
              }
            }
          if (!(top <= stc_range(MODE))) p.err[1] = 1;
        }
      } else if (act) {
        float top = 0.0f;
#pragma unroll
        for (int j = 0; j < 16; j += 2)
          if (r0 + h + j < p.kc) {
            const int q = r0 - rb + h + j;
            const float w0 = F16 ? __uint_as_float(r[j]) * ws[q] : __uint_as_float(r[j]);
            pl.wcol[(int64_t)vm[q] * p.ldw] = Op::one(w0);
            float w1 = 0.0f;
            if (r0 + h + j + 1 < p.kc) {
              w1 = F16 ? __uint_as_float(r[j + 1]) * ws[q + 1] : __uint_as_float(r[j + 1]);
              pl.wcol[(int64_t)vm[q + 1] * p.ldw] = Op::one(w1);
            }
            if (F16 || GUARD) top = max_nan(top, fabsf(w0), fabsf(w1));
          }
        if (F16 && !(top <= stc_range(MODE))) p.err[1] = 1;
        if (!F16 && GUARD && !(top <= stc_range(MODE))) {
          // a NaN or an overflow makes the sample's log NaN, and W keeps finite values
          lsum = NAN;
#pragma unroll 1
          for (int j = 0; j < 16 && r0 + h + j < p.kc; j++) {
            unsigned short* const w = pl.wcol + (int64_t)vm[r0 - rb + h + j] * p.ldw;
            if ((*w & 0x7F80) == 0x7F80) *w = 0;
          }
        }
      }
    }
    if (OV) stc_done<OV>(k, 0);
    stc_done<OV>(k, 1);
  }
  return true;
}

// The CTA's stages, records, barriers and TMEM columns (dynamic shared memory of
// sweep_tc_smem_bytes(MODE, NST)); the barriers initialised and the columns allocated.
// Ends with every thread past the allocation.
template <int MODE, int NST, bool OV>
__device__ __forceinline__ StcCta stc_cta_setup(unsigned char* smem) {
  StcCta k;
  k.stage = smem;
  k.rec = reinterpret_cast<float*>(smem + NST * stc_stage_bytes(MODE));
  k.tri = k.rec + STC_SUB * STC_REC;
  k.full = reinterpret_cast<uint64_t*>(k.tri + STC_TRI);
  k.freeb = k.full + NST;
  k.acc = k.freeb + NST;
  k.ready = k.acc + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(k.ready + 2);
  static_assert((2 * NST + 4) * 8 + 12 <= 192, "the barriers' place");
  k.abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  k.item = k.abort_flag + 1;
  k.next = reinterpret_cast<StcTile*>(reinterpret_cast<unsigned char*>(k.full) + 192);
  k.args = reinterpret_cast<SweepTcArgs*>(reinterpret_cast<unsigned char*>(k.full) + 256);
  if (threadIdx.x == 0) {
    *k.abort_flag = 0;
#pragma unroll
    for (int s = 0; s < NST; s++) {
      tc::mbar_init(k.full + s, 1);
      tc::mbar_init(k.freeb + s, 1);
    }
#pragma unroll
    for (int s = 0; s < 2; s++) {
      tc::mbar_init(k.acc + s, 1);
      tc::mbar_init(k.ready + s, STC_NS / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tmem_slot)),
                 "r"(StcPlan<OV>::NBUF * stc_cols(MODE))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  k.tmem = *tmem_slot;
  return k;
}

// Frees the CTA's TMEM columns once every thread is done with them.
template <int MODE, bool OV>
__device__ __forceinline__ void stc_cta_release(const StcCta& k) {
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(k.tmem), "r"(StcPlan<OV>::NBUF * stc_cols(MODE))
                 : "memory");
}

struct SweepTcLaunch {
  SweepTcArgs base;      // the arguments as of tile 0 at variable, rank row and column rank 0
  const StcTile* tiles;
  int i0, i1;            // the launch's tiles
  int m;                 // largest tile
  int alo, blo, ulo, vlo;  // (StcOps)
  const uint64_t* D;
  int64_t ldD, sample0, N, C;
  const float* rs;
  unsigned short* Ys;
  int64_t ldys;
  unsigned short* W;
  double* logP;
};

// All tiles [i0, i1) of a chunk's samples in one launch; CTA x owns samples [128 x, 128 (x + 1)), whose tiles need
// nothing of the other CTAs.  (A launch for each tile has every tile end with its slowest CTA, and all CTAs
// allocate and load anew: n = 65,536, 20 x 5,000 samples, tiles of 512, bf16: 60.8 -> 57.4 ms a solve; n = 16,384,
// 10 x 1,000, tiles of 256: 7.22 -> 6.78; 20 requests of n = 512 to 4,096 on four streams: 11.0 -> 8.8.  A queue of (tile, block) items over fewer CTAs, the same number on each
// SM, was slower: 63 ms with four or five CTAs on each, for the CTAs then run out of step and their y out of L2.)
template <int FLAGS, int MODE, bool OV>
__global__ void __launch_bounds__(StcPlan<OV>::THREADS, stc_ctas(MODE, OV))
    k_sweep_tc(const __grid_constant__ CUtensorMap mapY, const __grid_constant__ CUtensorMap mapYp, const __grid_constant__ CUtensorMap mapB,
               const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapU,
               const __grid_constant__ CUtensorMap mapV, const __grid_constant__ SweepTcLaunch d) {
  extern __shared__ __align__(1024) unsigned char stc_smem[];
  constexpr int NST = stc_stages(MODE, OV);
  const StcCta k = stc_cta_setup<MODE, NST, OV>(stc_smem);
  const int tid = threadIdx.x;
  const int c0 = blockIdx.x * STC_NS;  // (a chunk holds fewer than 2^31 samples)
  StcPlace pl;
  pl.wx = c0;
  pl.wy = 0;
  pl.yrow = c0;
  const StcOps o{&mapY, &mapYp, &mapB, &mapW, &mapU, &mapV, d.alo, d.blo, d.base.wlo, d.ulo, d.vlo, d.base.err};
  StcRun run{0, 0, 0, 0, 0};
  if (OV && tid >= STC_NS) {
    if (tid == STC_NS) {
#pragma unroll 1
      for (int i = d.i0; i < d.i1; i++) {
        const StcTile t = d.tiles[i];
        if (!stc_produce<MODE, NST>(o, t, i * d.m, k, pl, run)) break;
      }
    }
  } else {
    const bool act = c0 + tid < d.C;
    const int cs = act ? c0 + tid : (int)d.C - 1;  // inactive lanes shadow a valid sample, write nothing
    const int64_t g = d.sample0 + cs;
    const int64_t sh = g / d.N;
    const uint64_t* Ds = d.D + sh * d.ldD;
    const uint32_t ks = (uint32_t)(g - sh * d.N) + 1u;  // lattice point index k = 1..N (N < 2^31)
    const float rs = d.rs ? d.rs[cs] : 1.0f;
    pl.ysrow = d.Ys + (int64_t)cs * d.ldys;
    pl.wcol = d.W + cs;
    uint32_t step = 0;
#pragma unroll 1
    for (int i = d.i0; i < d.i1; i++) {
      stc_args<OV>(k, d.base, d.tiles, i, d.i1, d.m, i == d.i0);
      // log P of the tile = log(prod) + pe log 2 + lsum, prod kept in [1, 2)
      float prod = 1.0f, lsum = 0.0f;
      int pe = 0;
      if (!stc_tile<FLAGS, MODE, NST, OV>(*k.args, k, pl, step, o, run, i * d.m, act, Ds, ks, rs, prod, lsum, pe))
        break;
      if (act) {
        const double lp = (double)(logf(prod) + lsum) + (double)pe * 0.69314718055994530942;
        if (i == 0) d.logP[g] = lp;
        else atomicAdd(d.logP + g, lp);  // (this thread's alone: an add that nothing waits for)
      }
    }
  }
  stc_cta_release<MODE, OV>(k);
}

}  // namespace tlrmvn
