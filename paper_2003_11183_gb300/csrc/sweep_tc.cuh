// The integrand of a whole diagonal tile i in one kernel (Algorithm 6's per-tile step with eq. 2 over the
// tile): the tile's low-rank limit shifts, the sweep with its in-tile coupling, and the tile's projections
// for the later tiles, the products on the tensor cores.
//
// One CTA of 128 threads owns 128 samples, one per thread and per TMEM lane, and
// 64 TMEM columns.  The tile runs in sub-tiles of 64 variables.  Before sub-tile
// q, one thread accumulates into the columns, by tcgen05 products,
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
// lo, for the later products.  After the last sub-tile the CTA computes the
// tile's projections W[k][c] = sum_v V_i[k][v] y_v[c] in passes of 64 ranks through
// the same columns and writes them as rows of W.  So neither the shifts nor the
// coupling go through global memory, the per-variable loads of B are
// shared-memory broadcasts, and the sample's log P is closed once per tile.
//
// Shared memory per CTA (36.1 KB, six CTAs per SM): one 24 KB stage of MMA operands,
// staged by TMA (shift and projection k-blocks 64 deep, 128-byte swizzle; coupling
// k-blocks 32 deep, 64-byte swizzle), and what the sweep reads: a 96-byte record per
// variable (its window column of B, limits, reciprocal diagonal, lattice generator) and
// the six 16 x 16 blocks of the sub-tile's triangle that lie left of the windows.
// These have a place of their own, so that the idle threads load them while one
// thread runs the products, and the first shift k-block of the next sub-tile is copied
// during the sweep.  Every wait is bounded; on expiry the CTA records an error code,
// skips the rest, waits (bounded) for its copies and products in flight, frees its
// TMEM and returns.
//
// What bounds it: the chain from a variable's sum to its y (about 110 instructions, most
// of them dependent) and, with five CTAs per SM, the issue slots; the arithmetic pipe
// (compares, selects, integer operations: half the rate of the FMA pipe) came first
// with 64 of 176 instructions a variable, so the step avoids them: see
// sov_step_f32_upper.  With that step, the constants' loads beside the products and the pairwise
// renormalisation and TMEM stores: n = 65,536, 20 x 5,000 samples, tiles of 512: 73.5 -> 60.4 ms a solve; n =
// 16,384, 10 x 1,000, tiles of 256: 10.0 -> 7.2 ms; two-sided limits (n = 3,900, 8 x 1,301): 4.43 -> 1.99 ms.
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
//                       of 2^-10: the products hi*hi are multiples of 2^-20 and their sums, below 16, exact; the
//                       other products (hi*lo, lo*hi, lo*lo), 2^-10 of those, have an accumulator of their own (128
//                       TMEM columns).  The factor's operands have a third part, and hi*third is added there: their
//                       rounding to two parts, the same for all samples, was the largest error left.  Errors of
//                       the samples' logs against 64 bits (rms; float32 FMAs before in brackets): n = 8,192, tiles
//                       of 256: 1.9e-5 (2.7e-5); n = 1,024, tiles of 128, nu = 7: 4.5e-6 (6.3e-6); n = 2,048, tiles
//                       of 512: 1.0e-5 (1.3e-5).  Times against the float32 FMA products and sweeps: n = 16,384, 20
//                       x 5,000 samples: 55.0 -> 25.9 ms a solve; n = 4,096, nu = 7, 10 x 1,000: 4.41 -> 2.35 ms; 64
//                       batched problems, 10 x 2,000: 87.9 -> 18.8 ms.
enum StcMode { STC_BF16 = 0, STC_FP16 = 1, STC_FP32 = 2 };
constexpr int STC_SUB = 64;   // variables per sub-tile
constexpr int STC_NS = 128;   // samples per CTA (TMEM lanes)
constexpr int STC_KB = 32;    // K depth of a coupling k-block
using StcCfg = tc::Cfg<64, true, false, STC_KB, 1>;

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

// hi and lo fp16 parts of two floats for STC_FP32, packed low word first: hi a multiple of 2^-10 (of more above 2)
__device__ __forceinline__ void split_f32(float a, float b, uint32_t& hi, uint32_t& lo) {
  float ha, hb, la, lb;
  hi = Op16<true>::pack((a + 12288.0f) - 12288.0f, (b + 12288.0f) - 12288.0f, ha, hb);
  lo = Op16<true>::pack(a - ha, b - hb, la, lb);
}

// Per variable: [0, 16) the window column (for an even variable v B[v+2+k][v] at k < 14 and B[v+1][v] at 14,
// so that the pair update of the sweep reads aligned pairs; for an odd one B[v+1+k][v] at k < 15),
// then a, b, 1 / B_vv and (STC_FP32) the inverse of its row's scale, the lattice generator (8 bytes) and 8 spare bytes.
constexpr int STC_REC = 24;  // floats
// Entries after the lattice shifts' table: a sample's row is read up to three entries past a tile's last variable.
constexpr int STC_DPAD = 4;

struct SweepTcArgs {
  const float* rec;  // the factor's records at the tile's first variable (limits not filled in)
  const float* BT;   // transposed diagonal tile, BT[u * ldbt + v] = B[v][u]
  int64_t ldbt;
  int mt;            // variables in the tile
  int t0;            // (k_sweep_tc) its first variable
  const float* a;    // limits at the tile's first variable
  const float* b;
  int64_t ys_lo;     // offset of the lo parts in a sample's row of y
  int brow0;     // row of the tile's first variable in the split-B map
  int alo, blo;  // x offsets of the lo halves in the y and split-B maps
  int urow0;     // row of the tile's first variable in the U map
  int krow0, kr; // the tile's rank rows in the W map (first, count; 0: no low-rank shift)
  int kcol0, kc; // the tile's column ranks: first row in the V map, count (0: no projection)
  int64_t ldw;   // projections, rank-major: row vmap[r], ldw samples a row
  const int32_t* vmap;    // at the tile's first column rank
  const float* wscale;    // FP16 path: per column rank, the factor applied to a projection before it is
                          // stored (the inverse of the per-tile scales of U and V); null on the BF16 path
  float tscale;           // FP16 path: 1 / g, undoing the products' global scale g where the sweep reads them
  const float* rscale;    // STC_FP32: per variable of the tile, the inverse of its row's scale
  int wlo, ulo, vlo;      // STC_FP32: the lo parts' row offset in W, x offsets in the U and V maps (third parts: twice)
  int* err;               // [0] a bounded wait's code; [1] (STC_FP32) a y or a projection beyond fp16's range
};
constexpr int STC_ARGS = 256;  // shared memory of a tile's arguments
static_assert(sizeof(SweepTcArgs) <= STC_ARGS, "the arguments' place");
using StcProjCfg = tc::Cfg<64, false, false, 64, 1>;  // projection k-block: y rows x V rows, 64 deep
static_assert(StcProjCfg::SB == StcCfg::SB, "a projection k-block fills the same stage");
using StcShiftCfg = tc::Cfg<64, false, true, 64, 1>;  // shift k-block: W (MN-major) x U rows, 64 deep
static_assert(StcShiftCfg::SB == StcCfg::SB, "a shift k-block fills the same stage");

constexpr int STC_TRI = 6 * 256;  // floats: the 16 x 16 blocks (ub, vb), ub < vb, at vb (vb - 1) / 2 + ub
// [NST stages][records][triangle blocks][barriers, TMEM slot][a tile's arguments] (the dynamic shared memory starts 1 KB-aligned: the
// kernels have no static shared memory, and the system's own part is 1 KB)
__host__ __device__ constexpr uint32_t stc_stage_bytes(int mode) {
  return StcCfg::SB + (mode == STC_FP32 ? StcCfg::B_BYTES : 0);  // (the third part of the factor's operand)
}
__host__ __device__ constexpr size_t sweep_tc_smem_bytes(int mode, int nst) {
  return (size_t)nst * stc_stage_bytes(mode) + (STC_SUB * STC_REC + STC_TRI) * sizeof(float) + 128 + STC_ARGS;
}
// TMEM columns of a CTA: the sums (and y) of a sub-tile, and STC_FP32's second accumulator
__host__ __device__ constexpr uint32_t stc_cols(int mode) { return mode == STC_FP32 ? 2 * STC_SUB : STC_SUB; }

// Shared-memory layout and per-CTA state of the whole-tile sweep (set up once per
// kernel: a persistent kernel runs many tiles through the same stage, barriers
// and TMEM columns).
struct StcCta {
  unsigned char* stage;
  float* rec;            // the sub-tile's records
  float* tri;            // its triangle blocks
  uint64_t* full;        // [NST] the stage's copies landed
  uint64_t* freeb;       // [NST] the products reading the stage are done
  uint32_t tmem;         // first of the CTA's TMEM columns
  uint32_t* count;       // k-blocks gone through the stages so far (block i uses stage i mod NST)
  int* abort_flag;
  int* item;             // the work item
  SweepTcArgs* args;     // (k_sweep_tc) the tile's arguments
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

// Thread 0's ring of NST stages.  load(i, st) starts the copies of k-block i into a stage, mma(i, st) issues its
// products.  Runs blocks [0, nk), of which the first `pre` were loaded before, and waits for all products; `count`
// numbers the blocks over the CTA's life.  Returns false (every copy and product in flight waited for, bounded) when
// a wait expired.
template <int NST, typename Load, typename Mma>
__device__ __forceinline__ bool stc_ring(const StcCta& k, uint32_t& count, int nk, int pre, int* err, Load load,
                                         Mma mma) {
  int issued = pre, kb = 0;
  bool ok = true;
  for (; kb < nk; kb++) {
    for (; issued < nk && issued < kb + NST; issued++) {
      const uint32_t i = count + (uint32_t)issued;
      if (i >= NST && !tc::mbar_wait(k.freeb + i % NST, (i / NST - 1) & 1, err, 9)) {
        ok = false;
        break;
      }
      load(issued, i % NST);
    }
    const uint32_t i = count + (uint32_t)kb;
    if (!ok || !tc::mbar_wait(k.full + i % NST, (i / NST) & 1, err, 8)) {
      ok = false;
      break;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    mma(kb, i % NST);
    tc::mma_commit(k.freeb + i % NST);
  }
  if (kb > 0) {  // (products complete in order)
    const uint32_t i = count + (uint32_t)kb - 1;
    if (!tc::mbar_wait(k.freeb + i % NST, (i / NST) & 1, err, 9)) ok = false;
  }
  if (!ok)
    for (; kb < issued; kb++) {
      const uint32_t i = count + (uint32_t)kb;
      tc::mbar_wait(k.full + i % NST, (i / NST) & 1, err, 5);
    }
  count += (uint32_t)nk;
  return ok;
}

// One diagonal tile for the CTA's samples: the low-rank shifts and in-tile
// coupling on tcgen05, the float sweep of eq. 2, the projections.  act: the thread's
// sample exists (else it shadows one and writes nothing); Ds: its row of lattice shifts
// at the tile's first variable (read up to three entries past the tile); ks: its point
// index; rs: its MVT scale (1 for MVN).  The tile's log P is added to (prod, pe, lsum).
// Returns false when a bounded wait expired.
template <int FLAGS, int MODE, int NST>
__device__ __forceinline__ bool stc_tile(const CUtensorMap* mapY, const CUtensorMap* mapB, const CUtensorMap* mapW,
                                         const CUtensorMap* mapU, const CUtensorMap* mapY64, const CUtensorMap* mapV,
                                         const SweepTcArgs& p, const StcCta& k, const StcPlace& pl, const bool act,
                                         const uint64_t* Ds, const uint32_t ks, const float rs, float& prod,
                                         float& lsum, int& pe) {
  constexpr bool PER = FLAGS & SWEEP_PERIODIZE, ONE = FLAGS & SWEEP_ONE_SIDED;
  constexpr bool F16 = MODE != STC_BF16, SPLIT = MODE == STC_FP32;
  using Op = Op16<F16>;
  constexpr uint32_t ID_C = F16 ? StcCfg::IDESC_F16 : StcCfg::IDESC;
  constexpr uint32_t ID_S = F16 ? StcShiftCfg::IDESC_F16 : StcShiftCfg::IDESC;
  constexpr uint32_t ID_P = F16 ? StcProjCfg::IDESC_F16 : StcProjCfg::IDESC;
  constexpr uint32_t CA = StcCfg::A_BYTES, CHALF = StcCfg::HALF, SA = StcShiftCfg::A_BYTES, PA = StcProjCfg::A_BYTES;
  constexpr uint32_t SB = stc_stage_bytes(MODE), CB3 = StcCfg::SB;  // (a stage; its third B part)
  constexpr int KS = SPLIT ? STC_KB : 64;  // depth of a shift or projection k-block
  unsigned char* stage = k.stage;
  volatile int* abort_flag = k.abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int mt = p.mt;
  const uint32_t tmem = k.tmem;
  const uint32_t tl = tmem + ((uint32_t)(32 * warp) << 16);  // this warp's 32 lanes
  const int nks = (p.kr + KS - 1) / KS;
  // the copies of shift k-block kb.  16-bit: two 64-sample MN-major boxes of W (64 ranks), one box of U rows.  Split:
  // [W hi: two 64-sample boxes of 32 ranks][U hi][W lo][U lo][U third]
  auto load_shift = [&](int kb, int q0, uint32_t st) {
    unsigned char* d = stage + st * SB;
    uint64_t* bar = k.full + st;
    tc::mbar_expect_tx(bar, SB);
    const int y = pl.wy + p.krow0 + kb * KS;
    if constexpr (SPLIT) {
#pragma unroll
      for (int h = 0; h < 2; h++) {
        tc::tma_load_2d(d + h * CHALF, mapW, bar, pl.wx, y + h * p.wlo);
        tc::tma_load_2d(d + h * CHALF + CA / 2, mapW, bar, pl.wx + 64, y + h * p.wlo);
        tc::tma_load_2d(d + h * CHALF + CA, mapU, bar, kb * KS + h * p.ulo, p.urow0 + q0);
      }
      tc::tma_load_2d(d + CB3, mapU, bar, kb * KS + 2 * p.ulo, p.urow0 + q0);
    } else {
      tc::tma_load_2d(d, mapW, bar, pl.wx, y);
      tc::tma_load_2d(d + SA / 2, mapW, bar, pl.wx + 64, y);
      tc::tma_load_2d(d + SA, mapU, bar, kb * 64, p.urow0 + q0);
    }
  };
  // the products of a split stage [A hi][B hi][A lo][B lo]([B third]), 32 deep: A's descriptors and their advance per 16-deep step
  auto mma_split = [&](uint64_t ah, uint64_t al, uint64_t astep, uint32_t sa, uint32_t idesc, bool first) {
    const uint64_t bh = tc::sdesc<STC_KB>(sa + CA), bl = tc::sdesc<STC_KB>(sa + CHALF + CA);
#pragma unroll
    for (int kk = 0; kk < STC_KB / 16; kk++) {
      const uint64_t oa = astep * (uint64_t)kk, ob = (uint64_t)(2 * kk);  // 32 bytes per 16-deep step of B
      const uint32_t acc = (!first || kk > 0) ? 1u : 0u;
      tc::mma_f16(tmem, ah + oa, bh + ob, idesc, acc);
      tc::mma_f16(SPLIT ? tmem + STC_SUB : tmem, ah + oa, bl + ob, idesc, SPLIT ? acc : 1u);
      tc::mma_f16(SPLIT ? tmem + STC_SUB : tmem, al + oa, bh + ob, idesc, 1u);
      if constexpr (SPLIT) {
        tc::mma_f16(tmem + STC_SUB, al + oa, bl + ob, idesc, 1u);
        tc::mma_f16(tmem + STC_SUB, ah + oa, tc::sdesc<STC_KB>(sa + CB3) + ob, idesc, 1u);
      }
    }
  };

  int pre = 0;  // (thread 0) shift k-blocks of the coming sub-tile already under way
  for (int q0 = 0; q0 < mt; q0 += STC_SUB) {
    const int mq = min(STC_SUB, mt - q0);
    // every thread is past the previous sub-tile's reads of the records and its TMEM accesses
    if (tid >= 32) {
      // the sub-tile's records, limits and triangle blocks, by the warps that do not run the products
      const int t0 = tid - 32;
      for (int t = t0; t < mq * 6; t += STC_NS - 32) {
        const int v = t / 6, c = t - v * 6;
        const float* src = p.rec + (int64_t)(q0 + v) * STC_REC + 4 * c;
        if (c == 4)
          reinterpret_cast<float4*>(k.rec)[t] =
              make_float4(p.a[q0 + v], p.b[q0 + v], __ldg(src + 2), SPLIT ? __ldg(p.rscale + q0 + v) : 0.0f);
        else
          cp_async16(reinterpret_cast<float4*>(k.rec) + t, src, 16);
      }
      for (int t = t0; t < STC_TRI / 4; t += STC_NS - 32) {
        const int blk = t >> 6, u = (t >> 2) & 15, c = t & 3;
        const int vb = blk < 1 ? 1 : (blk < 3 ? 2 : 3), ub = blk - vb * (vb - 1) / 2;
        if (16 * vb < mq)
          cp_async16(reinterpret_cast<float4*>(k.tri) + t,
                     p.BT + (int64_t)(q0 + 16 * ub + u) * p.ldbt + q0 + 16 * vb + 4 * c, 16);
      }
      cp_async_commit();
      cp_async_wait<0>();
    }
    if ((q0 > 0 || p.kr > 0) && tid == 0) {
      // T = W[ranks of row tile i, samples]^T U_i[q0 + v, ranks]^T     (the low-rank shifts)
      //   + y[:, <q0] B_i[q0 + v, <q0]^T                              (the coupling, 32-deep split stages)
      const uint32_t sa0 = tc::smem_u32(stage);
      uint32_t count = *k.count;
      const bool ok = stc_ring<NST>(
          k, count, nks + q0 / STC_KB, pre, p.err,
          [&](int kb, uint32_t st) {
            if (kb < nks) {
              load_shift(kb, q0, st);
              return;
            }
            unsigned char* d = stage + st * SB;
            uint64_t* bar = k.full + st;
            tc::mbar_expect_tx(bar, SB);
            const int x = (kb - nks) * STC_KB;
            tc::tma_load_2d(d, mapY, bar, x, pl.yrow);
            tc::tma_load_2d(d + CHALF, mapY, bar, p.alo + x, pl.yrow);
            tc::tma_load_2d(d + CA, mapB, bar, x, p.brow0 + q0);
            tc::tma_load_2d(d + CHALF + CA, mapB, bar, p.blo + x, p.brow0 + q0);
            if constexpr (SPLIT) tc::tma_load_2d(d + CB3, mapB, bar, 2 * p.blo + x, p.brow0 + q0);
          },
          [&](int kb, uint32_t st) {
            const uint32_t sa = sa0 + st * SB;
            if (kb >= nks) {
              mma_split(tc::sdesc<STC_KB>(sa), tc::sdesc<STC_KB>(sa + CHALF), 2, sa, ID_C, kb == 0);
            } else if constexpr (SPLIT) {
              // per 16-deep step MN-major W is two 1 KB K groups on (+128)
              mma_split(tc::sdesc_mn(sa, CA / 2), tc::sdesc_mn(sa + CHALF, CA / 2), 128, sa, ID_S, kb == 0);
            } else {
              const uint64_t dw = tc::sdesc_mn(sa, SA / 2), du = tc::sdesc<64>(sa + SA);
#pragma unroll
              for (int kk = 0; kk < 4; kk++)
                tc::mma_f16(tmem, dw + (uint64_t)(128 * kk), du + (uint64_t)(2 * kk), ID_S,
                            (kb > 0 || kk > 0) ? 1u : 0u);
            }
          });
      pre = 0;
      if (!ok) {
        *abort_flag = 1;
      } else if (q0 + STC_SUB < mt) {
        // these land during the sweep (W and U are complete; all products have read their stages)
        for (; pre < NST && pre < nks; pre++) load_shift(pre, q0 + STC_SUB, (count + (uint32_t)pre) % NST);
      }
      *k.count = count;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();  // records and triangle staged; shifts and coupling are in TMEM
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (*abort_flag) return false;

    const uint64_t* Dp = Ds + q0;
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
          sov_step_f32_upper(bt, w, wc, f, lsum, y);
        } else {
          const float at = fmaf(abi.x, rs, -sum) * abi.z;
          sov_step_f32_prod(at, bt, w, wc, f, lsum, y);
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
              top = fmaxf(top, j < nb ? fmaxf(fabsf(y0), fabsf(y1)) : 0.0f);
            } else {
              float h0, h1, l0, l1;
              hi2[j / 2] = Op::pack(y0, y1, h0, h1);
              lo2[j / 2] = Op::pack(y0 - h0, y1 - h1, l0, l1);
            }
          }
          if (SPLIT && top > 32768.0f) p.err[1] = 1;
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
    }
    // y stored and visible to the copies (global), the records free for the next sub-tile's (shared), the TMEM
    // columns free for the next products
    asm volatile("fence.proxy.async;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  }
  // the tile's projections for the later tiles, 64 ranks a pass through the same
  // TMEM columns: W[vmap[r]][c] = sum_v V[kcol0 + r][v] y_v[c] (y hi parts, 64-deep
  // stages of the CTA's y rows and of V rows)
  for (int r0 = 0; r0 < p.kc; r0 += 64) {
    if (tid == 0) {
      const uint32_t sa0 = tc::smem_u32(stage);
      uint32_t count = *k.count;
      const bool ok = stc_ring<NST>(
          k, count, (mt + KS - 1) / KS, 0, p.err,
          [&](int kb, uint32_t st) {
            unsigned char* d = stage + st * SB;
            uint64_t* bar = k.full + st;
            tc::mbar_expect_tx(bar, SB);
            if constexpr (SPLIT) {
              tc::tma_load_2d(d, mapY, bar, kb * KS, pl.yrow);
              tc::tma_load_2d(d + CHALF, mapY, bar, p.alo + kb * KS, pl.yrow);
              tc::tma_load_2d(d + CA, mapV, bar, kb * KS, p.kcol0 + r0);
              tc::tma_load_2d(d + CHALF + CA, mapV, bar, p.vlo + kb * KS, p.kcol0 + r0);
              tc::tma_load_2d(d + CB3, mapV, bar, 2 * p.vlo + kb * KS, p.kcol0 + r0);
            } else {
              tc::tma_load_2d(d, mapY64, bar, kb * 64, pl.yrow);
              tc::tma_load_2d(d + PA, mapV, bar, kb * 64, p.kcol0 + r0);
            }
          },
          [&](int kb, uint32_t st) {
            const uint32_t sa = sa0 + st * SB;
            if constexpr (SPLIT) {
              mma_split(tc::sdesc<STC_KB>(sa), tc::sdesc<STC_KB>(sa + CHALF), 2, sa, ID_C, kb == 0);
            } else {
              const uint64_t da = tc::sdesc<64>(sa), db = tc::sdesc<64>(sa + PA);
#pragma unroll
              for (int kk = 0; kk < 4; kk++)
                tc::mma_f16(tmem, da + (uint64_t)(2 * kk), db + (uint64_t)(2 * kk), ID_P, (kb > 0 || kk > 0) ? 1u : 0u);
            }
          });
      if (!ok) *abort_flag = 1;
      *k.count = count;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (*abort_flag) return false;
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
              const float w0 = (__uint_as_float(r[j]) + __uint_as_float(l[j])) * p.wscale[rr];
              const float w1 = (__uint_as_float(r[j + 1]) + __uint_as_float(l[j + 1])) * p.wscale[r1];
              uint32_t hi, lo;
              split_f32(w0, w1, hi, lo);
              top = fmaxf(top, fmaxf(fabsf(w0), two ? fabsf(w1) : 0.0f));
              unsigned short* d0 = pl.wcol + (int64_t)p.vmap[rr] * p.ldw;
              d0[0] = (unsigned short)hi;
              d0[(int64_t)p.wlo * p.ldw] = (unsigned short)lo;
              if (two) {
                unsigned short* d1 = pl.wcol + (int64_t)p.vmap[r1] * p.ldw;
                d1[0] = (unsigned short)(hi >> 16);
                d1[(int64_t)p.wlo * p.ldw] = (unsigned short)(lo >> 16);
              }
            }
          if (top > 32768.0f) p.err[1] = 1;
        }
      } else if (act) {
#pragma unroll
        for (int j = 0; j < 16; j++)
          if (r0 + h + j < p.kc)
            pl.wcol[(int64_t)p.vmap[r0 + h + j] * p.ldw] =
                Op::one(F16 ? __uint_as_float(r[j]) * p.wscale[r0 + h + j] : __uint_as_float(r[j]));
      }
    }
    // W visible to the copies of the next tile's shifts, when the same CTA runs it
    asm volatile("fence.proxy.async;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();  // the TMEM columns and the stage free for the next pass
  }
  return true;
}

// The CTA's stages, records, barriers and TMEM columns (dynamic shared memory of
// sweep_tc_smem_bytes(MODE, NST)); the barriers initialised and the columns allocated.
// Ends with every thread past the allocation.
template <int MODE, int NST>
__device__ __forceinline__ StcCta stc_cta_setup(unsigned char* smem) {
  StcCta k;
  k.stage = smem;
  k.rec = reinterpret_cast<float*>(smem + NST * stc_stage_bytes(MODE));
  k.tri = k.rec + STC_SUB * STC_REC;
  k.full = reinterpret_cast<uint64_t*>(k.tri + STC_TRI);
  k.freeb = k.full + NST;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(k.freeb + NST);
  k.count = tmem_slot + 1;
  k.abort_flag = reinterpret_cast<int*>(tmem_slot + 2);
  k.item = k.abort_flag + 1;
  k.args = reinterpret_cast<SweepTcArgs*>(reinterpret_cast<unsigned char*>(k.full) + 128);
  if (threadIdx.x == 0) {
    *k.abort_flag = 0;
    *k.count = 0;
#pragma unroll
    for (int s = 0; s < NST; s++) {
      tc::mbar_init(k.full + s, 1);
      tc::mbar_init(k.freeb + s, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tmem_slot)),
                 "r"(stc_cols(MODE))
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
template <int MODE>
__device__ __forceinline__ void stc_cta_release(const StcCta& k) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(k.tmem), "r"(stc_cols(MODE))
                 : "memory");
}

// CTAs per SM: six with one stage (80 registers each), three with two, two with three or four.
__host__ __device__ constexpr int stc_ctas(int nst) { return nst == 1 ? 6 : (nst == 2 ? 3 : 2); }

// A diagonal tile: its first variable and size, its rank rows of W (first, count), its column ranks (first, count).
struct StcTile {
  int t0, mt, krow0, kr, kcol0, kc, pad[2];
};
struct SweepTcLaunch {
  SweepTcArgs base;      // the arguments as of tile 0 at variable, rank row and column rank 0
  const StcTile* tiles;
  int i0, i1;            // the launch's tiles
  int m;                 // largest tile
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
template <int FLAGS, int MODE, int NST>
__global__ void __launch_bounds__(STC_NS, stc_ctas(NST))
    k_sweep_tc(const __grid_constant__ CUtensorMap mapY, const __grid_constant__ CUtensorMap mapB,
               const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapU,
               const __grid_constant__ CUtensorMap mapY64, const __grid_constant__ CUtensorMap mapV,
               const __grid_constant__ SweepTcLaunch d) {
  extern __shared__ __align__(1024) unsigned char stc_smem[];
  const StcCta k = stc_cta_setup<MODE, NST>(stc_smem);
  const int tid = threadIdx.x;
  const int c0 = blockIdx.x * STC_NS;  // (a chunk holds fewer than 2^31 samples)
  const bool act = c0 + tid < d.C;
  const int cs = act ? c0 + tid : (int)d.C - 1;  // inactive lanes shadow a valid sample, write nothing
  const int64_t g = d.sample0 + cs, sh = g / d.N;
  const uint32_t ks = (uint32_t)(g - sh * d.N) + 1u;  // lattice point index k = 1..N (N < 2^31)
  const float rs = d.rs ? d.rs[cs] : 1.0f;
  StcPlace pl;
  pl.wx = c0;
  pl.wy = 0;
  pl.yrow = c0;
  pl.ysrow = d.Ys + (int64_t)cs * d.ldys;
  pl.wcol = d.W + cs;
#pragma unroll 1
  for (int i = d.i0; i < d.i1; i++) {
    if (tid == 0) {
      const int4 t = __ldg(reinterpret_cast<const int4*>(d.tiles + i));
      const int2 c = __ldg(reinterpret_cast<const int2*>(d.tiles + i) + 2);
      SweepTcArgs& p = *k.args;
      p = d.base;
      p.rec += (int64_t)i * d.m * STC_REC;
      p.BT += (int64_t)i * d.m * p.ldbt;
      p.mt = t.y;
      p.t0 = t.x;
      p.a += t.x;
      p.b += t.x;
      p.brow0 = i * d.m;
      p.urow0 = i * d.m;
      p.krow0 = t.z;
      p.kr = t.w;
      p.kcol0 = c.x;
      p.kc = c.y;
      p.vmap += c.x;
      p.wscale += c.x;
      p.rscale += (int64_t)i * d.m;
    }
    __syncthreads();
    // log P of the tile = log(prod) + pe log 2 + lsum, prod kept in [1, 2)
    float prod = 1.0f, lsum = 0.0f;
    int pe = 0;
    if (!stc_tile<FLAGS, MODE, NST>(&mapY, &mapB, &mapW, &mapU, &mapY64, &mapV, *k.args, k, pl, act,
                                    d.D + sh * d.ldD + k.args->t0, ks, rs, prod, lsum, pe))
      break;
    if (act) {
      const double lp = (double)(logf(prod) + lsum) + (double)pe * 0.69314718055994530942;
      if (i == 0) d.logP[g] = lp;
      else atomicAdd(d.logP + g, lp);  // (this thread's alone: an add that nothing waits for)
    }
    __syncthreads();  // the arguments read by all
  }
  stc_cta_release<MODE>(k);
}

}  // namespace tlrmvn
