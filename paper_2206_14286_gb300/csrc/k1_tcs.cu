// k1_tcs.cu -- PartialReduce with bins j mod L (Alg. 1) fused with a tcgen05
// BF16 contraction, queries on the tensor-memory lanes and each bin's rows
// side by side in the accumulator.
//
// Row j = t*Lv + v lies in virtual bin v, Lv = fold * L (bins j mod Lv refine
// bins j mod L: virtual bin v merges into bin v mod L). The last, ragged grid
// row holds r = N mod Lv rows, so virtual bins below r have T + 1 rows and the
// others T = floor(N / Lv): the database is read as two [rows x bins] grids,
// A (bins 0..r-1, T + 1 rows) and B (bins r..Lv-1, T rows), with a tensor map
// each, and no row is left over. One pipeline step covers 16 virtual bins and
// 16 grid rows of one of the grids: 256 database rows, loaded per K block by
// ONE 3-D TMA box whose outer dimension is the bin, so accumulator column
// n = (b - b0)*16 + (t - t0)
// and every run of 16 consecutive columns holds 16 rows of ONE bin. The
// epilogue reduces such a run with a single tcgen05.ld.red.max (the load
// returns the 16 scores and their maximum) and compares the maximum once with
// the bin's best so far; only on a new best does it look for the column. That
// is about one compare per 16 scores instead of a compare (and a key pack)
// per score, which keeps the CUDA-core work well below the tensor-core time.
//
// One CTA (640 threads, one per SM) owns a contiguous run of steps and takes
// kq query tiles in turn over it, one segment each; kq > 1 only when the tiles
// do not spread evenly over the SMs (the host picks kq and the runs). A tile is
// NH query halves of up to 128 queries (MMA M = 128, A operand resident in
// shared memory unless the rows are too long), NH = 2 or 1; with one half the
// A operand holds only the queries there are (the MMA's other lanes read
// whatever follows and are ignored), which leaves the shared memory to the
// ring: calls of few queries are bound by the database read.
//   warp 0      : TMA producer (the query tile once per segment; per step and
//                 128-byte K block one 16 x 16-row box into a 32 KB stage of
//                 an S-stage ring).
//   warp 1      : TMEM allocation (512 columns: two 128 x 256 FP32
//                 accumulators) and tcgen05.mma issue. NH = 2: one accumulator
//                 per query half; half 0 of a step is computed and handed to
//                 its epilogue while half 1 is computed, so each half's drain
//                 overlaps the other's MMAs. NH = 1: the steps alternate
//                 between the accumulators.
//   warps 2, 3  : (L2 only) each step's half norms as an extra K = 16 block
//                 (-h split into three BF16 parts against a ones block of the
//                 queries), so the accumulator holds the relaxed score
//                 <q,x> - |x|^2/2 (App. A.2, Eq. 19).
//   warps 4..19 : epilogue, two warpgroups (column halves) per accumulator; a
//                 thread owns one query and 8 bins of the step; it keeps each
//                 bin's best score and grid row, and when the CTA moves to
//                 the next group of bins it merges them into G[query][bin] by
//                 64-bit atomicMax on the ordered key (score, ~row): ties
//                 keep the smaller row, and bins split between CTAs (or
//                 accumulators) merge exactly. Warps without a query only
//                 release the accumulators.
// Steps that reach past a grid's last row or bin take a column-by-column path
// with a validity test. All waits are bounded (see tc_ptx.cuh).
#include <algorithm>
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "dtypes.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace tpuknn {

namespace {

constexpr int kThreadsS = 640;   // 4 control warps + 4 epilogue warpgroups
constexpr int kQH = 128;         // queries per half: MMA M, TMEM lanes
constexpr int kRowsBin = 16;     // grid rows per bin per step
constexpr int kSpanS = 128;      // bytes of one 128-byte swizzle span (one K block)
constexpr int kExtAS = kQH * 32;             // ones block (K = 16 BF16)

// A step: 16 bins x 16 grid rows (or 256 consecutive rows): MMA N = 256, one
// K block of it 32 KB. (8-bin steps, N = 128 with two accumulators per query
// half, measured 0.320 against 0.195 ms on 1M x 128 rows, 1024 queries: their
// MMAs read 1.5x the shared-memory operand bytes per FLOP.)
constexpr int kStepBins = 16;
constexpr int kCols = kStepBins * kRowsBin;  // MMA N, accumulator columns
constexpr int kStage = kCols * kSpanS;       // one K block of a step
// Half-norm block of a step (K = 16, no swizzle): the 16-byte pieces of K
// index 0..7, eight columns after eight. The pieces of K index 8..15 are zero
// and one block of zeros serves every slot (the descriptor's leading offset
// leads to it). Four slots, two per half-norm warp: with two, a slot's values
// were written while the MMAs already waited for them.
constexpr int kExtB = kCols * 16;
constexpr int kXS = 4;
constexpr int kBPW = kStepBins / 2;          // bins per epilogue warpgroup
// Half norms on their way in (L2): a ring of kHS steps of 16 x 16 floats, one
// grid row (or, contiguous bins, one row of each run of 16) every kHP floats,
// loaded kHD steps ahead. At the HBM rate a step of 128-element rows takes 1.5
// us, about one load latency under load: one step ahead (in registers)
// stalled. The odd row length lets a warp write rows and read columns with at
// most two lanes on a bank.
constexpr int kHS = 8, kHD = 6, kHP = 17;
constexpr int kHStep = kRowsBin * kHP;
constexpr int kHRing = kHS * kHStep * 4;
// Register split (setmaxnreg): the control warpgroup gives up registers so
// the epilogue can keep four 16-column runs in flight. 128*64 + 512*104 =
// 61440 = 640*96, the registers the kernel is launched with (checked on the
// host before every launch).
constexpr int kCtrlRegsS = 64, kEpiRegsS = 104;

struct TcsArgs {
  int64_t N, M, L;
  int Lv, T, r;                    // virtual bins; full grid rows; rows of the ragged one
  int ntga, ntgb, nbga;            // 16-row groups of grids A and B, 16-bin groups of A
  uint32_t bq, br;                 // contiguous bins: q = N / L, r = N mod L
  int64_t steps_per_q, nqt;        // steps over the whole database; query tiles
  int64_t parts, steps_per_part;   // the database steps split into `parts` ranges
  int64_t kq, groups;              // query tiles one CTA takes in turn; tile groups
  int qrows;                       // query rows of a resident tile (multiple of 8)
  int nkb, nksteps, stages;
  uint32_t stage_bytes;            // one K block of a step (+ of the queries when streamed)
  uint32_t a_bytes;
  int ext;
  uint32_t idesc;
  const float* hnorm;
  const float* xscale;             // E4M3: the database-wide scale (xscale[0])
  unsigned long long* G;
};

// Where a step lies: bin group bg (A's groups first), 16-row group tg.
struct StepPos {
  int bg, tg;
};
__device__ __forceinline__ StepPos step_at(const TcsArgs& a, int64_t s) {
  const int64_t sa = (int64_t)a.nbga * a.ntga;
  if (s < sa) return StepPos{(int)(s / a.ntga), (int)(s % a.ntga)};
  return StepPos{a.nbga + (int)((s - sa) / a.ntgb), (int)((s - sa) % a.ntgb)};
}
// The next step; true when it starts another group of bins.
__device__ __forceinline__ bool step_next(const TcsArgs& a, StepPos& p) {
  if (++p.tg < (p.bg < a.nbga ? a.ntga : a.ntgb)) return false;
  p.tg = 0;
  ++p.bg;
  return true;
}
// The grid of bin group bg: its first local bin, rows, bins, and the virtual
// bin of its local bin 0.
struct StepGrid {
  int b0, rows, bins, base;
};
__device__ __forceinline__ StepGrid step_grid(const TcsArgs& a, int bg) {
  if (bg < a.nbga) return StepGrid{bg * kStepBins, a.T + 1, a.r, 0};
  return StepGrid{(bg - a.nbga) * kStepBins, a.T, a.Lv - a.r, a.r};
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool live) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src),
               "r"(live ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The smallest k with r[k] == m (one of them is). The equalities become 1.0 or
// 0.0 and add up powers of two, the largest for k = 0, so half of the work
// runs on the FMA pipe (16 compares and 16 selects all ran on the ALU, the
// pipe that bounds short bins: 2M x 96 E4M3 rows, L = 8192, 2000 queries, 1.085
// against 1.026 ms a search).
__device__ __forceinline__ int first_equal(const float (&r)[16], float m) {
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    float e;
    asm("set.eq.f32.f32 %0, %1, %2;" : "=f"(e) : "f"(r[k]), "f"(m));
    acc[k & 3] = fmaf(e, (float)(1 << (15 - k)), acc[k & 3]);
  }
  const float sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  return 15 + 127 - (int)(__float_as_uint(sum) >> 23);
}

// 64 columns of this thread's lane as four runs of 16 with their maxima, waited for.
__device__ __forceinline__ void tmem_ld4x16_max_s(uint32_t taddr, float (&r)[4][16], float (&m)[4]) {
  asm volatile(
      "tcgen05.ld.red.sync.aligned.32x32b.x16.max.f32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, %16, [%68];\n\t"
      "tcgen05.ld.red.sync.aligned.32x32b.x16.max.f32 {%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32}, %33, [%69];\n\t"
      "tcgen05.ld.red.sync.aligned.32x32b.x16.max.f32 {%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49}, %50, [%70];\n\t"
      "tcgen05.ld.red.sync.aligned.32x32b.x16.max.f32 {%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63,%64,%65,%66}, %67, [%71];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(r[0][0]), "=f"(r[0][1]), "=f"(r[0][2]), "=f"(r[0][3]), "=f"(r[0][4]), "=f"(r[0][5]), "=f"(r[0][6]), "=f"(r[0][7]), "=f"(r[0][8]), "=f"(r[0][9]), "=f"(r[0][10]), "=f"(r[0][11]), "=f"(r[0][12]), "=f"(r[0][13]), "=f"(r[0][14]), "=f"(r[0][15]), "=f"(m[0]),
        "=f"(r[1][0]), "=f"(r[1][1]), "=f"(r[1][2]), "=f"(r[1][3]), "=f"(r[1][4]), "=f"(r[1][5]), "=f"(r[1][6]), "=f"(r[1][7]), "=f"(r[1][8]), "=f"(r[1][9]), "=f"(r[1][10]), "=f"(r[1][11]), "=f"(r[1][12]), "=f"(r[1][13]), "=f"(r[1][14]), "=f"(r[1][15]), "=f"(m[1]),
        "=f"(r[2][0]), "=f"(r[2][1]), "=f"(r[2][2]), "=f"(r[2][3]), "=f"(r[2][4]), "=f"(r[2][5]), "=f"(r[2][6]), "=f"(r[2][7]), "=f"(r[2][8]), "=f"(r[2][9]), "=f"(r[2][10]), "=f"(r[2][11]), "=f"(r[2][12]), "=f"(r[2][13]), "=f"(r[2][14]), "=f"(r[2][15]), "=f"(m[2]),
        "=f"(r[3][0]), "=f"(r[3][1]), "=f"(r[3][2]), "=f"(r[3][3]), "=f"(r[3][4]), "=f"(r[3][5]), "=f"(r[3][6]), "=f"(r[3][7]), "=f"(r[3][8]), "=f"(r[3][9]), "=f"(r[3][10]), "=f"(r[3][11]), "=f"(r[3][12]), "=f"(r[3][13]), "=f"(r[3][14]), "=f"(r[3][15]), "=f"(m[3])
      : "r"(taddr), "r"(taddr + 16u), "r"(taddr + 32u), "r"(taddr + 48u)
      : "memory");
}

// 16 columns of this thread's lane, waited for.
__device__ __forceinline__ void tmem_ld16s(uint32_t taddr, float (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
      : "r"(taddr)
      : "memory");
}

// byte offset of (row r, 16-byte piece kc) in a K = 16 BF16 block without swizzle
__device__ __forceinline__ uint32_t ext_off_s(int r, int kc) {
  return (uint32_t)((r >> 3) * 256 + kc * 128 + (r & 7) * 16);
}

// Modes of the K loop:
//   kFused   : rows up to 128 elements. The whole step's K blocks are resident
//              together; each query half runs all its MMAs in one unrolled run
//              (NKS K-steps), so each half's drain overlaps the other's MMAs.
//   kKLoopA  : longer rows, query tile resident. The step walks its K blocks
//              one stage at a time, each stage feeding both halves; both
//              accumulators close at the end of the step (their drain is short
//              against a long step).
//   kKLoopQ  : rows too long for a resident query tile: a stage carries the K
//              block of the 256 queries too.
constexpr int kFused = 0, kKLoopA = 1, kKLoopQ = 2;

// Bin maps: kBinsMod (bin = j mod L, steps over the [T][L] grid view) and
// kBinsRun (Alg. 1's ShiftRight generalised to L balanced runs of consecutive
// rows; a step is 256 consecutive rows, and a thread follows one current bin).
constexpr int kBinsMod = 0, kBinsRun = 1;

// (row numbers and bin ends are below 2^31: 32-bit unsigned arithmetic)
__device__ __forceinline__ uint32_t run_bin_of(uint32_t p, uint32_t q, uint32_t r) {
  const uint64_t big = (uint64_t)r * (q + 1);
  return p < big ? p / (q + 1) : r + (uint32_t)(p - big) / q;
}
__device__ __forceinline__ uint32_t run_bin_end(uint32_t b, uint32_t q, uint32_t r) {
  return (b + 1) * q + min(b + 1, r);
}

template <int NKS, int MODE, int BM, int NH, int DT>
__global__ void __launch_bounds__(kThreadsS, 1)
k1_tcs_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmY,
              const __grid_constant__ CUtensorMap tmQ, const TcsArgs a) {
  // tmX: grid A (or the rows, contiguous bins), tmY: grid B.
  // queries of a tile; NB accumulators per query half
  constexpr int kQTile = NH * kQH;
  constexpr int NB = 2 / NH, XS = kXS, BPW = kBPW;
  // elements of one 128-byte K block (the x coordinate of a K block's box)
  constexpr int kElS = DT == KNN_E4M3 ? kSpanS : kSpanS / 2;
  // 128-byte K blocks per step
  const int NKB = MODE == kFused ? (NKS + 3) / 4 : a.nkb;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  const int S = a.stages;
  uint8_t* sA = smem;                                      // queries, SW128, [kb][qrows][128 B]
  uint8_t* sB = sA + a.a_bytes;                            // S stages of one K block
  uint8_t* sAext = sB + (size_t)S * a.stage_bytes;         // ones block (L2)
  uint8_t* sBext = sAext + (a.ext ? kExtAS : 0);           // XS half-norm blocks, zeros (L2)
  float* sH = reinterpret_cast<float*>(sBext + (a.ext ? (XS + 1) * kExtB : 0));  // half norms (L2)
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(sH) +
                                               (a.ext ? kHRing : 0));
  // accumulator (h, buf) of query half h: barriers b_accf / b_acce + 8 (h NB + buf),
  // TMEM columns (h NB + buf) kCols
  constexpr int NACC = 2;
  const uint32_t b_full = smem_u32(bars), b_empty = smem_u32(bars + S);
  const uint32_t b_accf = smem_u32(bars + 2 * S), b_acce = smem_u32(bars + 2 * S + NACC);
  const uint32_t b_xf = smem_u32(bars + 2 * S + 2 * NACC);
  const uint32_t b_xe = smem_u32(bars + 2 * S + 2 * NACC + XS);
  const uint32_t b_q = smem_u32(bars + 2 * S + 2 * NACC + 2 * XS);
  const uint32_t b_done = smem_u32(bars + 2 * S + 2 * NACC + 2 * XS + 1);
  const uint32_t b_qe = smem_u32(bars + 2 * S + 2 * NACC + 2 * XS + 2);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 2 * NACC + 2 * XS + 3);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // CTA = (part, group): the steps [s_begin, s_end) of the database for the
  // query tiles q0 .. q0 + nseg - 1, one after the other (a segment each).
  // The CTAs of one part walk the same rows at the same time, so the rows
  // they share meet in L2; their block indices are adjacent, which keeps
  // them on neighbouring SMs (the same die). Step i of the CTA is step
  // i mod ns of segment i / ns; barrier phases count i across segments.
  const int64_t part = blockIdx.x / a.groups;
  const int64_t q0 = (blockIdx.x % a.groups) * a.kq;
  const int nseg = (int)max((int64_t)0, min(a.kq, a.nqt - q0));
  const int64_t s_begin = part * a.steps_per_part;
  const int64_t s_end = min(a.steps_per_q, s_begin + a.steps_per_part);
  const int ns = (int)max((int64_t)0, s_end - s_begin);
  const int nt = nseg * ns;  // steps of this CTA

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(b_full + 8 * s, 1);
      mbar_init(b_empty + 8 * s, 1);
    }
    for (int c = 0; c < NACC; ++c) {
      mbar_init(b_accf + 8 * c, 1);
      mbar_init(b_acce + 8 * c, 8);  // the 8 warps of its two warpgroups
    }
    for (int e = 0; e < XS; ++e) {
      mbar_init(b_xf + 8 * e, 1);
      mbar_init(b_xe + 8 * e, 1);
    }
    mbar_init(b_q, 1);
    mbar_init(b_done, 1);
    mbar_init(b_qe, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (a.ext) {
    // the queries' ones block: K index 0..2 = 1, the rest 0; and the zeros
    // behind the half-norm blocks
    const __nv_bfloat16 one = __float2bfloat16_rn(1.0f), zero = __float2bfloat16_rn(0.0f);
    for (int r = threadIdx.x; r < kQH; r += kThreadsS) {
      __nv_bfloat16 v[8] = {one, one, one, zero, zero, zero, zero, zero};
      *reinterpret_cast<uint4*>(sAext + ext_off_s(r, 0)) = *reinterpret_cast<uint4*>(v);
      *reinterpret_cast<uint4*>(sAext + ext_off_s(r, 1)) = make_uint4(0, 0, 0, 0);
    }
    for (int t = threadIdx.x; t < kCols; t += kThreadsS)
      *reinterpret_cast<uint4*>(sBext + (size_t)XS * kExtB + t * 16) = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the prologue above touches no global memory; the queries and the zeroed
  // key array come from the preceding kernel
  pdl_wait();
  pdl_trigger();

  if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kCtrlRegsS));
  if (warp == 0) {
    // -------------------------------------------------------------- producer
    int s = 0, issued = 0, q_armed = 0;
    uint32_t ph = 0;
    bool prun = true;
    for (int sg = 0; sg < nseg && prun; ++sg) {
    const int64_t qtile = q0 + sg;
    // the segment's query tile (phase sg of b_q); from the second segment on
    // only after the MMAs of the previous one are done with the old tile
    if (MODE != kKLoopQ && sg > 0 &&
        !warp_all(mbar_wait_sleep(b_qe, (uint32_t)((sg - 1) & 1), abort_flag)))
      break;
    q_armed = sg + 1;
    if (lane == 0) {
      if (MODE == kKLoopQ) {
        mbar_arrive(b_q);  // the queries come with every stage
      } else {
        mbar_expect_tx(b_q, a.a_bytes);
        for (int kb = 0; kb < NKB; ++kb)
          tma_load_2d(smem_u32(sA + (size_t)kb * a.qrows * kSpanS), &tmQ, b_q, kb * kElS,
                      (int)(qtile * kQTile));
      }
    }
    __syncwarp();
    int kb = 0;
    StepPos sp = BM == kBinsMod ? step_at(a, s_begin) : StepPos{0, 0};
    const int total = ns * NKB;
    for (int g = 0; g < total; ++g) {
      if (issued >= S && !warp_all(mbar_wait_sleep(b_empty + 8 * s, ph ^ 1u, abort_flag))) {
        prun = false;
        break;
      }
      if (lane == 0) {
        mbar_expect_tx(b_full + 8 * s, a.stage_bytes);
        uint32_t dst = smem_u32(sB + (size_t)s * a.stage_bytes);
        if (MODE == kKLoopQ) {
          // the queries' K block first: [queries][128 B]
          tma_load_2d(dst, &tmQ, b_full + 8 * s, kb * kElS, (int)(qtile * kQTile));
          dst += a.qrows * kSpanS;
        }
        if constexpr (BM == kBinsRun) {
          // kCols consecutive rows; rows past N read the fill value (zero)
          tma_load_2d(dst, &tmX, b_full + 8 * s, kb * kElS,
                      (int)((s_begin + g / NKB) * kCols));
        } else {
          // one box: K block kb (128 bytes), 16 grid rows, 16 bins, landing as
          // [bin][grid row][128 B]; bins and rows past the grid's and
          // elements past the row read the fill value (zero)
          tma_load_3d(dst, sp.bg < a.nbga ? &tmX : &tmY, b_full + 8 * s, kb * kElS,
                      sp.tg * kRowsBin, step_grid(a, sp.bg).b0);
        }
      }
      __syncwarp();
      ++issued;
      if (++kb == NKB) {
        kb = 0;
        if (BM == kBinsMod) step_next(a, sp);
      }
      if (++s == S) {
        s = 0;
        ph ^= 1u;
      }
    }
    }
    // the copies still in flight land before the CTA can exit, also after a
    // give-up: the last min(issued, S) stages and the last query tile armed
    for (int k = 0; k < S && k < issued; ++k) {
      if (--s < 0) {
        s = S - 1;
        ph ^= 1u;
      }
      mbar_drain(b_full + 8 * s, ph);
    }
    if (MODE != kKLoopQ && q_armed > 0) mbar_drain(b_q, (uint32_t)((q_armed - 1) & 1));
    return;
  }
  if (warp == 1) {
    // -------------------------------------------------------------- MMA issuer
    // The whole warp runs the loop and the waits; one lane issues. The tensor
    // pipe holds few instructions, so nothing slow sits between the MMAs of a
    // half: every wait of a step (its stages, its L2 block, the accumulator
    // being free) comes before the unrolled run of MMAs it guards, and the
    // commits come after.
    // b_q phase sg: the query tile of segment sg has landed; a commit to b_qe
    // after a segment's last MMAs frees the tile for the next one
    if constexpr (MODE == kFused) {
    {
      const uint64_t a_desc = smem_desc_sw128(smem_u32(sA));
      const uint64_t b_desc = smem_desc_sw128(smem_u32(sB));
      const uint64_t ax_desc = smem_desc_noswz(smem_u32(sAext), 128, 256);
      // half-norm block of slot e
      auto bx_desc = [&](int e) {
        return smem_desc_noswz(smem_u32(sBext + e * kExtB), (XS - e) * kExtB, 128);
      };
      int s0 = 0;           // stage of K block 0 of the current step
      uint32_t ph0 = 0;
      bool run = true;
      for (int sg = 0; sg < nseg && run; ++sg) {
      if (!warp_all(mbar_wait(b_q, (uint32_t)(sg & 1), abort_flag))) break;
      for (int li = 0; li < ns && run; ++li) {
        const int i = sg * ns + li;
        const int e = i % XS;
        const int buf = i % NB;
        // the stages of this step (NKB consecutive ring slots)
        int sk[(NKS + 3) / 4];
        {
          int s = s0;
          uint32_t ph = ph0;
#pragma unroll
          for (int kb = 0; kb < NKB; ++kb) {
            sk[kb] = s;
            if (run && !warp_all(mbar_wait(b_full + 8 * s, ph, abort_flag))) run = false;
            if (++s == S) {
              s = 0;
              ph ^= 1u;
            }
          }
          s0 = s;
          ph0 = ph;
        }
        if (!run) break;
        if (a.ext && !warp_all(mbar_wait(b_xf + 8 * e, (uint32_t)((i / XS) & 1), abort_flag))) {
          run = false;
          break;
        }
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          // the accumulator's previous use (step i - NB) has been drained
          const int c = h * NB + buf;
          if (i >= NB &&
              !warp_all(mbar_wait(b_acce + 8 * c, (uint32_t)(((i / NB) & 1) ^ 1), abort_flag))) {
            run = false;
            break;
          }
          tc_fence_after();
          if (lane == 0) {
            const uint32_t d_tmem = tmem_base + (uint32_t)(c * kCols);
            const uint64_t ah = a_desc + (uint64_t)((h * kQH * kSpanS) >> 4);
#pragma unroll
            for (int ks = 0; ks < NKS; ++ks) {
              // descriptors advance by (bytes >> 4) in their address field
              const uint64_t ad = ah + (uint64_t)(((ks >> 2) * a.qrows * kSpanS + (ks & 3) * 32) >> 4);
              const uint64_t bd =
                  b_desc + (uint64_t)((sk[ks >> 2] * kStage + (ks & 3) * 32) >> 4);
              tc_mma<DT>(d_tmem, ad, bd, a.idesc, ks > 0 ? 1u : 0u);
              // the last half is a K block's last reader: its stage is free
              // once the MMAs so far complete (2-3% faster than freeing all
              // stages of the step after the half's last MMA)
              if (h == NH - 1 && ((ks & 3) == 3 || ks == NKS - 1))
                tc_commit(b_empty + 8 * sk[ks >> 2]);
            }
            if (a.ext)
              tc_mma<KNN_BF16>(d_tmem, ax_desc, bx_desc(e), a.idesc, 1u);
            tc_commit(b_accf + 8 * c);
            if (h == NH - 1 && a.ext) tc_commit(b_xe + 8 * e);
          }
          __syncwarp();
        }
      }
      if (!run) break;
      if (lane == 0) tc_commit(b_qe);
      __syncwarp();
      }
    }
    }
    if constexpr (MODE != kFused) {
    {
      const uint64_t a_desc = smem_desc_sw128(smem_u32(sA));
      const uint64_t ax_desc = smem_desc_noswz(smem_u32(sAext), 128, 256);
      // half-norm block of slot e
      auto bx_desc = [&](int e) {
        return smem_desc_noswz(smem_u32(sBext + e * kExtB), (XS - e) * kExtB, 128);
      };
      int s = 0;
      uint32_t ph = 0;
      bool run = true;
      for (int sg = 0; sg < nseg && run; ++sg) {
      if (!warp_all(mbar_wait(b_q, (uint32_t)(sg & 1), abort_flag))) break;
      for (int li = 0; li < ns && run; ++li) {
        const int i = sg * ns + li;
        const int e = i % XS;
        const int buf = i % NB;
        // the step's accumulators are written from its first K block on. (With
        // two halves, waiting for half 1 only before its own MMAs and closing
        // half 0 before half 1's last K block overlaps the drains with MMAs,
        // but the MMAs then take 203 cycles each instead of 139 and the step
        // is longer: 1.56 against 1.44 ms on 1M x 256 rows, 4096 queries.)
#pragma unroll
        for (int h = 0; h < NH; ++h)
          if (run && i >= NB &&
              !warp_all(mbar_wait(b_acce + 8 * (h * NB + buf), (uint32_t)(((i / NB) & 1) ^ 1),
                                  abort_flag)))
            run = false;
        if (!run) break;
        for (int kb = 0; kb < NKB; ++kb) {
          if (!warp_all(mbar_wait(b_full + 8 * s, ph, abort_flag))) {
            run = false;
            break;
          }
          tc_fence_after();
          if (lane == 0) {
            const uint32_t st = smem_u32(sB + (size_t)s * a.stage_bytes);
            const uint64_t bd = smem_desc_sw128(MODE == kKLoopQ ? st + a.qrows * kSpanS : st);
            const int steps = min(4, a.nksteps - kb * 4);
#pragma unroll
            for (int h = 0; h < NH; ++h) {
              const int c = h * NB + buf;
              const uint32_t d_tmem = tmem_base + (uint32_t)(c * kCols);
              const uint64_t ad =
                  MODE == kKLoopQ
                      ? smem_desc_sw128(st + (uint32_t)(h * kQH * kSpanS))
                      : a_desc + (uint64_t)((kb * a.qrows * kSpanS + h * kQH * kSpanS) >> 4);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                if (kk < steps)
                  tc_mma<DT>(d_tmem, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), a.idesc,
                             (kb | kk) ? 1u : 0u);
            }
            tc_commit(b_empty + 8 * s);
          }
          __syncwarp();
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (!run) break;
        if (a.ext) {
          if (!warp_all(mbar_wait(b_xf + 8 * e, (uint32_t)((i / XS) & 1), abort_flag))) {
            run = false;
            break;
          }
          tc_fence_after();
        }
        if (lane == 0) {
          if (a.ext) {
#pragma unroll
            for (int h = 0; h < NH; ++h)
              tc_mma<KNN_BF16>(tmem_base + (uint32_t)((h * NB + buf) * kCols), ax_desc,
                               bx_desc(e), a.idesc, 1u);
            tc_commit(b_xe + 8 * e);
          }
#pragma unroll
          for (int h = 0; h < NH; ++h) tc_commit(b_accf + 8 * (h * NB + buf));
        }
        __syncwarp();
      }
      if (!run) break;
      if (lane == 0) tc_commit(b_qe);
      __syncwarp();
      }
    }
    }
    // all MMAs have completed before tensor memory is released (also after a
    // give-up: the MMAs already issued still write their accumulators)
    if (lane == 0) tc_commit(b_done);
    __syncwarp();
    mbar_drain(b_done, 0);
    asm volatile("bar.sync 1, %0;" ::"n"(32 + 512) : "memory");
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
    return;
  }
  if (warp == 2 || warp == 3) {
    // ---------------------------------------------------------- L2 half norms
    if (!a.ext) return;
    // column n = j*16 + u of a step is bin b0 + j, grid row t0 + u. The values
    // come in by cp.async kHD steps ahead of the step being written, lane l of
    // copy k taking j = l % 16, u = l / 16 + 2 k, so that 16 lanes read 16
    // consecutive floats of one grid row. On the way out lane l writes columns
    // n = l + 32 k, whose 16-byte pieces are adjacent: written in the order
    // they come in, eight lanes meet in a bank, and a step's stores took 3,500
    // cycles of a shared memory that the MMAs' operands nearly fill. Warps 2 and 3 take the steps in turn, and a
    // block slot each: one warp for every step kept the MMAs waiting 6-8% of
    // the time (two query halves) to 25% (one).
    constexpr int HK = kCols / 32;
    StepPos sp = BM == kBinsMod ? step_at(a, s_begin) : StepPos{0, 0};
    int lsn = 0;  // step within the segment of the next load
    auto load = [&](int i) {
      const uint32_t dst = smem_u32(sH + (i % kHS) * kHStep);
      const bool own = (i & 1) == warp - 2;
      if (i < nt) {
        if (own) {
          if constexpr (BM == kBinsRun) {
            // column n is row step*256 + n
#pragma unroll
            for (int k = 0; k < HK; ++k) {
              const int n = lane + 32 * k;
              const int64_t p = (s_begin + lsn) * kCols + n;
              cp_async4(dst + 4 * ((n & 15) * kHP + (n >> 4)), a.hnorm + (p < a.N ? p : 0),
                        p < a.N);
            }
          } else {
            const StepGrid gr = step_grid(a, sp.bg);
            const int b = gr.b0 + (lane & 15), t = sp.tg * kRowsBin + (lane >> 4);
            const float* src = a.hnorm + ((int64_t)t * a.Lv + gr.base + b);
#pragma unroll
            for (int k = 0; k < HK; ++k) {
              const bool live = b < gr.bins && t + 2 * k < gr.rows;
              cp_async4(dst + 4 * (((lane >> 4) + 2 * k) * kHP + (lane & 15)),
                        live ? src + (int64_t)(2 * k) * a.Lv : a.hnorm, live);
            }
          }
        }
        if (BM == kBinsMod) step_next(a, sp);
        if (++lsn == ns) {  // the next segment repeats the steps
          lsn = 0;
          if (BM == kBinsMod) sp = step_at(a, s_begin);
        }
      }
      cp_async_commit();
    };
#pragma unroll 1
    for (int k = 0; k < kHD; ++k) load(k);
    {
      for (int i = 0; i < nt; ++i) {
        load(i + kHD);
        if ((i & 1) != warp - 2) continue;
        cp_async_wait<kHD>();
        __syncwarp();  // every lane's copies have landed
        const int e = i % XS;
        int ok = 1;
        if (lane == 0 && i >= XS)
          ok = mbar_wait_sleep(b_xe + 8 * e, (uint32_t)(((i / XS) & 1) ^ 1), abort_flag) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        uint8_t* ext = sBext + (size_t)e * kExtB;
        const float* hs = sH + (i % kHS) * kHStep;
        float hv[HK];
#pragma unroll
        for (int k = 0; k < HK; ++k) {
          const int n = lane + 32 * k;
          hv[k] = hs[(n & 15) * kHP + (n >> 4)];
        }
#pragma unroll
        for (int k = 0; k < HK; ++k) {
          const __nv_bfloat16 hi = __float2bfloat16_rn(hv[k]);
          const float rem1 = hv[k] - __bfloat162float(hi);
          const __nv_bfloat16 mid = __float2bfloat16_rn(rem1);
          const __nv_bfloat16 lo = __float2bfloat16_rn(rem1 - __bfloat162float(mid));
          const __nv_bfloat16 z = __float2bfloat16_rn(0.0f);
          __nv_bfloat16 v[8] = {__hneg(hi), __hneg(mid), __hneg(lo), z, z, z, z, z};
          *reinterpret_cast<uint4*>(ext + (lane + 32 * k) * 16) = *reinterpret_cast<uint4*>(v);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(b_xf + 8 * e);
      }
    }
    cp_async_wait<0>();
    return;
  }
  if (warp < 4) return;

  // ---------------------------------------------------------------- epilogue
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegsS));
  const int quad = warp & 3;
  const int egrp = (warp - 4) >> 2;  // 0..3
  const int acc = egrp >> 1;         // accumulator: query half (NH = 2) or step parity
  const int h = NH == 2 ? acc : 0;   // query half
  const int cq = egrp & 1;           // bins cq*BPW .. cq*BPW+BPW-1 of each step
  constexpr int NLD = BPW / 4;       // 64-column loads per step and thread
  // this thread's query in the current segment
  bool q_ok = false, w_ok = false;  // this thread's query exists; any of the warp's
  unsigned long long* gq = a.G;
  // E4M3: keys hold the raw dot of the codes times the database scale (the
  // per-query scale is left out: it does not change the order in a query)
  const float xs0 = DT == KNN_E4M3 ? a.xscale[0] : 1.0f;
  auto scaled = [&](float v) { return DT == KNN_E4M3 ? __fmul_rn(v, xs0) : v; };
  auto set_query = [&](int sg) {
    const int64_t qi = (q0 + sg) * kQTile + h * kQH + quad * 32 + lane;
    q_ok = qi < a.M;
    w_ok = __ballot_sync(0xffffffffu, q_ok) != 0u;
    gq = a.G + (q_ok ? qi : 0) * a.L;
  };
  // TMEM lanes of this warp and this warpgroup's columns of an accumulator
  const uint32_t tlane = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(cq * BPW * 16);
  const uint32_t tb = tlane + (uint32_t)(acc * kCols);
  const uint32_t bf = b_accf + 8 * acc, be = b_acce + 8 * acc;
  // whether step i is this warpgroup's, and the phase of its accumulator
  auto mine = [&](int i) { return NB == 1 || (i & 1) == acc; };
  auto phase = [&](int i) { return (uint32_t)((i / NB) & 1); };
  if constexpr (BM == kBinsRun) {
    // Contiguous bins: this warpgroup sees rows s*kCols + cq*kCols/2 .. + kCols/2 - 1
    // of every step s, in increasing order. A thread follows the current bin
    // (the same for every lane: bins depend on rows only) with its best score
    // and row, and merges it into G when the rows leave the bin.
    const uint32_t nrows = (uint32_t)a.N;
    const uint32_t first = (uint32_t)min((s_begin * kCols + cq * (kCols / 2)), a.N - 1);
    uint32_t cur = 0, seg_end = 0;
    int32_t brow = -1;
    float bv = __uint_as_float(kNegInfBits);
    auto flush_run = [&]() {
      if (q_ok && brow >= 0)
        atomicMax(&gq[cur], (unsigned long long)make_key(scaled(bv), brow));
    };
    bool erun = true;
    for (int sg = 0; sg < nseg && erun; ++sg) {
    if (sg > 0) flush_run();
    set_query(sg);
    cur = run_bin_of(first, a.bq, a.br);
    seg_end = run_bin_end(cur, a.bq, a.br);
    bv = __uint_as_float(kNegInfBits);
    brow = -1;
    for (int li = 0; li < ns; ++li) {
      const int i = sg * ns + li;
      if (!mine(i)) continue;
      if (!warp_all(mbar_wait_sleep(bf, phase(i), abort_flag))) {
        erun = false;
        break;
      }
      tc_fence_after();
      if (!w_ok) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(be);
        continue;
      }
      const uint32_t p0 = (uint32_t)((s_begin + li) * kCols + cq * (kCols / 2));
#pragma unroll
      for (int half64 = 0; half64 < NLD; ++half64) {
        float r[4][16], m[4];
        __syncwarp();
        tmem_ld4x16_max_s(tb + (uint32_t)(half64 * 64), r, m);
        if (half64 == NLD - 1) {
          // everything of this accumulator is in registers: release it
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(be);
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const uint32_t pg = p0 + half64 * 64 + g * 16;
          if (pg + 16 <= seg_end) {  // (the last bin ends at N)
            // the 16 rows lie inside the current bin: one compare
            if (m[g] > bv) {
              bv = m[g];
              brow = (int32_t)pg + first_equal(r[g], m[g]);
            }
          } else {
            // a bin boundary or the end of the rows falls in this run
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const uint32_t p = pg + k;
              if (p < nrows) {
                while (p >= seg_end) {
                  flush_run();
                  ++cur;
                  seg_end = run_bin_end(cur, a.bq, a.br);
                  bv = __uint_as_float(kNegInfBits);
                  brow = -1;
                }
                if (r[g][k] > bv) {
                  bv = r[g][k];
                  brow = (int32_t)p;
                }
              }
            }
          }
        }
      }
    }
    }
    tc_fence_before();
    asm volatile("bar.arrive 1, %0;" ::"n"(32 + 512) : "memory");
    flush_run();
    return;
  }
  StepPos sp{0, 0};
  float best[BPW];
  int32_t bt[BPW];
#pragma unroll
  for (int g = 0; g < BPW; ++g) {
    best[g] = __uint_as_float(kNegInfBits);
    bt[g] = -1;
  }
  auto flush = [&](int bg) {
    const StepGrid gr = step_grid(a, bg);
#pragma unroll
    for (int g = 0; g < BPW; ++g) {
      const int b = gr.b0 + cq * BPW + g;
      if (q_ok && bt[g] >= 0 && b < gr.bins) {
        const int vb = gr.base + b;  // virtual bin; bin vb mod L
        atomicMax(&gq[a.Lv == a.L ? vb : vb % (int)a.L],
                  (unsigned long long)make_key(scaled(best[g]), bt[g] * a.Lv + vb));
      }
      best[g] = __uint_as_float(kNegInfBits);
      bt[g] = -1;
    }
  };
  auto record = [&](float (&r)[4][16], float (&m)[4], int g0, int32_t t0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int g = g0 + q;
      if (m[q] > best[g]) {
        best[g] = m[q];
        bt[g] = t0 + first_equal(r[q], m[q]);
      }
    }
  };
  bool erun = true;
  for (int sg = 0; sg < nseg && erun; ++sg) {
  if (sg > 0) flush(sp.bg);  // the previous segment's last group of bins
  set_query(sg);
  sp = step_at(a, s_begin);
  StepGrid gr = step_grid(a, sp.bg);
  for (int li = 0; li < ns; ++li) {
    const int i = sg * ns + li;
    if (mine(i)) {
      if (!warp_all(mbar_wait_sleep(bf, phase(i), abort_flag))) {
        erun = false;
        break;
      }
      tc_fence_after();
      const int32_t t0 = sp.tg * kRowsBin;
      const int bw = gr.b0 + cq * BPW;  // first bin of this warpgroup
      if (!w_ok) {
        // no query in this warp
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(be);
      } else if (t0 + kRowsBin <= gr.rows && bw + BPW <= gr.bins) {
        // every column valid (warp-uniform): one compare per 16 scores. The
        // accumulator is released as soon as the last run is in registers.
        float r[4][16], m[4];
#pragma unroll
        for (int ld = 0; ld < NLD; ++ld) {
          __syncwarp();
          tmem_ld4x16_max_s(tb + (uint32_t)(ld * 64), r, m);
          if (ld == NLD - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(be);
          }
          record(r, m, 4 * ld, t0);
        }
      } else {
        // past the grid's last row or bin: column by column
#pragma unroll
        for (int g = 0; g < BPW; ++g) {
          float r[16];
          __syncwarp();
          tmem_ld16s(tb + (uint32_t)(g * 16), r);
          if (bw + g < gr.bins) {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              if (t0 + k < gr.rows && r[k] > best[g]) {
                best[g] = r[k];
                bt[g] = t0 + k;
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(be);
      }
    }
    const int bg = sp.bg;
    if (step_next(a, sp)) {
      flush(bg);
      if (li + 1 < ns) gr = step_grid(a, sp.bg);
    }
  }
  }
  tc_fence_before();
  asm volatile("bar.arrive 1, %0;" ::"n"(32 + 512) : "memory");
  flush(sp.bg);
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode_s() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

CUtensorMapDataType map_type(int esz) {
  return esz == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
}

// 2-D map of BF16 (esz 2) or E4M3 codes (esz 1): inner extent `inner`
// elements, `rows` rows `stride_el` elements apart, box of 128 bytes x
// box_rows, 128-byte swizzle.
bool make_map_s(CUtensorMap* m, const void* base, int64_t inner, int64_t rows, int64_t stride_el,
                int box_rows, int esz) {
  auto enc = get_encode_s();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)stride_el * esz};
  cuuint32_t box[2] = {(cuuint32_t)(kSpanS / esz), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(m, map_type(esz), 2, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3-D view of one grid of the database for the step boxes: element d of grid
// row t, bin b is row t*Lv + b from `base`. Dimensions (d, t, b) with the bin
// outermost, so a box of (128 bytes, 16, 16) lands as [bin][grid row][128 B]:
// each bin's 16 rows are consecutive accumulator columns.
bool make_map_grid(CUtensorMap* m, const void* base, int64_t pitch, int64_t Lv, int64_t rows,
                   int64_t bins, int esz) {
  auto enc = get_encode_s();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)pitch, (cuuint64_t)rows, (cuuint64_t)bins};
  cuuint64_t strides[2] = {(cuuint64_t)(Lv * pitch * esz), (cuuint64_t)(pitch * esz)};
  cuuint32_t box[3] = {(cuuint32_t)(kSpanS / esz), (cuuint32_t)kRowsBin, (cuuint32_t)kStepBins};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(m, map_type(esz), 3, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Steps over the two grids of an N-row database with Lv virtual bins.
int64_t grid_steps(int64_t N, int64_t Lv, TcsArgs* a) {
  const int64_t T = N / Lv, r = N % Lv;
  a->Lv = (int)Lv;
  a->T = (int)T;
  a->r = (int)r;
  a->ntga = (int)cdiv(T + 1, kRowsBin);
  a->ntgb = (int)cdiv(T, kRowsBin);
  a->nbga = (int)cdiv(r, kStepBins);
  return (int64_t)a->nbga * a->ntga + cdiv(Lv - r, kStepBins) * a->ntgb;
}

// How many virtual bins per bin: the grids are padded to groups of 16 bins, so
// few bins waste MMAs (L = 20: two groups of 16, 1.6x the steps). The fold with
// the least time, in microseconds:
//   - the steps of a CTA, 0.45 per K block and query half, each further fold
//     counted as one per cent for its position searches;
//   - the merges into fewer than 16 bins, which all CTAs make at once: with L = 3
//     the 304 (CTA, accumulator) pairs of up to 128 queries add 5 ns for each
//     virtual bin (60,000 x 64 rows, 64 queries: fold 1, 3, 5 took 22, 24, 45 us, and
//     300,000 rows 45, 40, 56; 256 queries 24, 23, 30), more bins spread them over
//     more lines (L = 5, 7, 10: 40, 30, 24 us at 16 virtual bins). Few queries have
//     few merges (1 query: 19-20 us whatever the fold).
int64_t pick_fold(int64_t N, int64_t L, int64_t row_bytes, int64_t M, int64_t sms) {
  int64_t best = 1;
  double cost = 0.0;
  const double halves = (double)cdiv(M, kQH);
  const double step = 0.45 * (double)cdiv(row_bytes, kSpanS) * halves / (double)sms;
  const double merge = 0.005 * 2.0 * (double)sms / halves * std::min(1.0, 3.0 / (double)L) *
                       std::min(1.0, (double)M / 64.0);
  for (int64_t f = 1; f <= 16; ++f) {
    if (f > 1 && (f * L * kRowsBin > N || f * L * row_bytes >= ((int64_t)1 << 40))) break;
    TcsArgs a{};
    const double c = (double)grid_steps(N, f * L, &a) * step * (1.0 + 0.01 * (double)(f - 1)) +
                     merge * (double)std::min<int64_t>(f * L, kStepBins);
    if (f == 1 || c < cost) {
      best = f;
      cost = c;
    }
  }
  return best;
}

// One CTA per SM at most: the database steps split into `parts` ranges and
// the query tiles into groups of kq; CTA (group, part) runs the tiles of its
// group one after the other over its range. Picks the kq (and the parts it
// allows) with the least work per CTA, counting a query-tile reload as one
// step; ties go to the smaller kq (fewer reloads, fewer database passes).
void tcs_schedule(int64_t nqt, int64_t steps, int64_t sms, int64_t* kq_out, int64_t* parts_out,
                  int64_t* spp_out, int64_t* groups_out) {
  if (sms < 1) sms = 1;
  const int64_t kq_min = cdiv(nqt, sms);
  int64_t best = -1;
  for (int64_t kq = kq_min; kq <= min(nqt, kq_min + 16); ++kq) {
    const int64_t groups = cdiv(nqt, kq);
    if (groups > sms) continue;
    int64_t parts = min(sms / groups, steps);
    const int64_t spp = cdiv(steps, parts);
    parts = cdiv(steps, spp);
    const int64_t work = kq * (spp + 1);
    if (best < 0 || work < best) {
      best = work;
      *kq_out = kq;
      *parts_out = parts;
      *spp_out = spp;
      *groups_out = groups;
    }
  }
}

struct TcsShape {
  int mode, nkb, nksteps, stages, qrows;
  uint32_t a_bytes, stage_bytes;
  size_t smem;
};

// The first mode whose shared memory fits: kFused (resident query tile, the
// whole step's K blocks plus one of look-ahead), kKLoopA (resident query
// tile, at least 2 stages of one K block; 4 with one query half, whose calls
// live on bytes in flight), kKLoopQ (query K block streamed in every stage).
// nh query halves per tile; a single half holds only the M queries there are.
bool tcs_shape(int D, int metric, int esz, int nh, int64_t M, TcsShape* sh) {
  const int pitch = (int)round_up(D, 16);
  const size_t budget = 227 * 1024;
  const int ext = metric == KNN_L2;
  sh->qrows = nh == 2 ? 2 * kQH : (int)std::min<int64_t>(kQH, round_up(M < 1 ? 1 : M, 8));
  // 128-byte K blocks and 32-byte MMA K-steps (16 BF16 or 32 E4M3 elements)
  sh->nkb = (int)cdiv((int64_t)pitch * esz, kSpanS);
  const int nks = (int)cdiv((int64_t)pitch * esz, 32);
  const uint32_t a_res = (uint32_t)(sh->nkb * sh->qrows * kSpanS);
  const size_t fixed = 1024 + (ext ? kExtAS + (kXS + 1) * kExtB + kHRing : 0) + 512;
  // kFused: K-steps rounded up to an even count (the extra step multiplies
  // zero query columns: the query box reads zeros past the row)
  const int nks_even = (int)round_up(nks, 2);
  if (nks_even <= 8) {
    const int need = sh->nkb + 1 > 3 ? sh->nkb + 1 : 3;
    if (fixed + a_res + (size_t)need * kStage <= budget) {
      sh->mode = kFused;
      sh->nksteps = nks_even;
      sh->a_bytes = a_res;
      sh->stage_bytes = (uint32_t)kStage;
      sh->stages = (int)std::min<size_t>(16, (budget - fixed - a_res) / kStage);
      sh->smem = fixed + a_res + (size_t)sh->stages * kStage;
      return true;
    }
  }
  sh->nksteps = nks;
  if (fixed + a_res + (nh == 2 ? 2 : 4) * (size_t)kStage <= budget) {
    sh->mode = kKLoopA;
    sh->a_bytes = a_res;
    sh->stage_bytes = (uint32_t)kStage;
    sh->stages = (int)std::min<size_t>(8, (budget - fixed - a_res) / kStage);
  } else {
    sh->mode = kKLoopQ;
    sh->a_bytes = 0;
    sh->stage_bytes = (uint32_t)(sh->qrows * kSpanS + kStage);
    sh->stages = (int)std::min<size_t>(6, (budget - fixed) / sh->stage_bytes);
    if (sh->stages < 2) return false;
  }
  sh->smem = fixed + sh->a_bytes + (size_t)sh->stages * sh->stage_bytes;
  return true;
}

template <int NKS, int MODE, int BM, int NH, int DT>
cudaError_t launch_tcs(const CUtensorMap (&mx)[2], const CUtensorMap& mq, const TcsArgs& a,
                       size_t smem, int64_t blocks, cudaStream_t st) {
  auto kern = k1_tcs_kernel<NKS, MODE, BM, NH, DT>;
  // setmaxnreg.inc waits until the registers it asks for are free: refuse to
  // launch unless the launch-time allocation covers the split.
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kern);
  if (e != cudaSuccess) return e;
  if ((int64_t)round_up(fa.numRegs, 8) * kThreadsS < 128 * kCtrlRegsS + 512 * kEpiRegsS)
    return cudaErrorNotSupported;
  e = allow_dynamic_smem(kern);
  if (e != cudaSuccess) return e;
  if constexpr (BM == kBinsRun) {
    // Contiguous bins: a plain launch. Started early behind the query prep,
    // the CTAs land on SMs in the order those free up, and the sharers of a
    // part end up far apart (measured: 0.244 -> 0.284 ms per search).
    kern<<<(unsigned)blocks, kThreadsS, smem, st>>>(mx[0], mx[1], mq, a);
    return cudaGetLastError();
  } else {
    return launch_pdl(kern, dim3((unsigned)blocks), dim3(kThreadsS), smem, st, mx[0], mx[1], mq, a);
  }
}

}  // namespace

// KNN_BF16 with any metric; KNN_E4M3_T (one database-wide scale) with IP
// and COS (the L2 half norm enters the BF16 contraction as an extra K block,
// which the E4M3 MMAs do not take).
bool k1_tcs_supported(int dtype, int D, int metric, int64_t N, int64_t L) {
  TcsShape sh;
  if (metric < KNN_IP || metric > KNN_COS) return false;
  if (dtype != KNN_BF16 && !(dtype == KNN_E4M3_T && metric != KNN_L2)) return false;
  const int esz = dtype == KNN_BF16 ? 2 : 1;
  if (!tcs_shape(D, metric, esz, 2, 0, &sh)) return false;
  if (L < 1 || L > N || N >= ((int64_t)1 << 31)) return false;
  // the grid view's row stride (L rows) must stay below 2^40 bytes
  return L * round_up(D, 16) * esz < ((int64_t)1 << 40);
}

template <int BM, int NH, int DT>
cudaError_t launch_tcs_mode(const TcsShape& sh, const CUtensorMap (&mx)[2], const CUtensorMap& mq,
                            const TcsArgs& a, int64_t blocks, cudaStream_t st) {
  if (sh.mode == kKLoopA) return launch_tcs<4, kKLoopA, BM, NH, DT>(mx, mq, a, sh.smem, blocks, st);
  if (sh.mode == kKLoopQ) return launch_tcs<4, kKLoopQ, BM, NH, DT>(mx, mq, a, sh.smem, blocks, st);
  switch (sh.nksteps) {
    case 2: return launch_tcs<2, kFused, BM, NH, DT>(mx, mq, a, sh.smem, blocks, st);
    case 4: return launch_tcs<4, kFused, BM, NH, DT>(mx, mq, a, sh.smem, blocks, st);
    case 6: return launch_tcs<6, kFused, BM, NH, DT>(mx, mq, a, sh.smem, blocks, st);
    case 8: return launch_tcs<8, kFused, BM, NH, DT>(mx, mq, a, sh.smem, blocks, st);
    default: return cudaErrorNotSupported;
  }
}
template <int NH, int DT>
cudaError_t launch_tcs_bins(bool runs, const TcsShape& sh, const CUtensorMap (&mx)[2],
                            const CUtensorMap& mq, const TcsArgs& a, int64_t blocks,
                            cudaStream_t st) {
  return runs ? launch_tcs_mode<kBinsRun, NH, DT>(sh, mx, mq, a, blocks, st)
              : launch_tcs_mode<kBinsMod, NH, DT>(sh, mx, mq, a, blocks, st);
}

cudaError_t launch_k1_tcs(int64_t N, int64_t M, int64_t L, int D, int metric, int dtype,
                          int bin_map, const void* X, const float* xscale, const float* hnorm,
                          const void* Qp, unsigned long long* G, cudaStream_t st) {
  const bool e4 = dtype == KNN_E4M3_T;
  const int esz = e4 ? 1 : 2;
  if (!k1_tcs_supported(dtype, D, metric, N, L)) return cudaErrorNotSupported;
  if (metric == KNN_L2 && !hnorm) return cudaErrorInvalidValue;
  if (e4 && !xscale) return cudaErrorInvalidValue;
  if ((reinterpret_cast<uintptr_t>(X) & 15) || (reinterpret_cast<uintptr_t>(Qp) & 15))
    return cudaErrorInvalidValue;
  if (M <= 0) return cudaSuccess;
  const bool runs = bin_map == KNN_BINS_CONTIGUOUS;
  const int pitch = (int)round_up(D, 16);
  TcsArgs a{};
  a.N = N;
  a.M = M;
  a.L = L;
  a.bq = (uint32_t)(N / L);
  a.br = (uint32_t)(N % L);
  // a step: 16 bins x 16 grid rows (j mod L), or 256 consecutive rows
  const int64_t sms = std::max(1, device_sm_count());
  const int64_t grid =
      grid_steps(N, runs ? L : L * pick_fold(N, L, (int64_t)pitch * esz, M, sms), &a);
  a.steps_per_q = runs ? cdiv(N, kCols) : grid;
  // One or two query halves per tile: a step costs its halves' MMAs, so one
  // half is taken where the halves do not pair up (M <= 128, or 333 queries: 3
  // halves instead of 2 x 2). With one half every step is read from L2 for 128
  // queries instead of 256, counted as a tenth of its time; with contiguous
  // bins the epilogue also meets every bin in four warpgroups, which counts as
  // half of it (333 queries on 700,001 x 100 rows, L2: 118 us with one half, 106
  // with two; bins mod L: 90 and 110). On 1M x 128 rows (L2) a search of 1, 128
  // and 333 queries took 61, 74 and 113 us with two halves and takes 51, 55 and
  // 101 us; 64 queries on 4M x 768 rows 2.0 ms and 0.95 ms (6.5 TB/s).
  int64_t kq1 = 1, parts1 = 1, spp1 = 1, groups1 = 1;
  tcs_schedule(cdiv(M, 2 * kQH), a.steps_per_q, sms, &a.kq, &a.parts, &a.steps_per_part, &a.groups);
  tcs_schedule(cdiv(M, kQH), a.steps_per_q, sms, &kq1, &parts1, &spp1, &groups1);
  int nh = 2;
  if ((runs ? 1.5 : 1.1) * (double)kq1 * (double)(spp1 + 1) <
      2.0 * (double)a.kq * (double)(a.steps_per_part + 1)) {
    nh = 1;
    a.kq = kq1;
    a.parts = parts1;
    a.steps_per_part = spp1;
    a.groups = groups1;
  }
  a.nqt = cdiv(M, nh * kQH);
  TcsShape sh;
  if (!tcs_shape(D, metric, esz, nh, M, &sh)) return cudaErrorNotSupported;
  // step counters of a CTA are 32-bit
  if (a.kq * a.steps_per_part * sh.nkb >= ((int64_t)1 << 31)) return cudaErrorNotSupported;
  a.qrows = sh.qrows;
  a.nkb = sh.nkb;
  a.nksteps = sh.nksteps;
  a.stages = sh.stages;
  a.a_bytes = sh.a_bytes;
  a.stage_bytes = sh.stage_bytes;
  a.ext = metric == KNN_L2 ? 1 : 0;
  // D = F32, A = B = BF16 (kind::f16) or E4M3 (kind::f8f6f4, format 0), both
  // K-major, N = 256, M = 128
  a.idesc = (1u << 4) | (e4 ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)(kCols >> 3) << 17) |
            ((uint32_t)(kQH >> 4) << 24);
  a.hnorm = hnorm;
  a.xscale = xscale;
  a.G = G;
  CUtensorMap mx[2], mq;
  bool mapped;
  if (runs) {
    mapped = make_map_s(&mx[0], X, pitch, N, pitch, kCols, esz);
    mx[1] = mx[0];
  } else {
    const char* xb = static_cast<const char*>(X) + (int64_t)a.r * pitch * esz;
    mapped = make_map_grid(&mx[1], xb, pitch, a.Lv, a.T, a.Lv - a.r, esz);
    if (a.r > 0)
      mapped = mapped && make_map_grid(&mx[0], X, pitch, a.Lv, a.T + 1, a.r, esz);
    else
      mx[0] = mx[1];
  }
  if (!mapped) return cudaErrorInvalidValue;
  if (!make_map_s(&mq, Qp, pitch, M, pitch, sh.qrows, esz)) return cudaErrorInvalidValue;
  const int64_t blocks = a.groups * a.parts;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (e4)
    return nh == 2 ? launch_tcs_bins<2, KNN_E4M3>(runs, sh, mx, mq, a, blocks, st)
                   : launch_tcs_bins<1, KNN_E4M3>(runs, sh, mx, mq, a, blocks, st);
  return nh == 2 ? launch_tcs_bins<2, KNN_BF16>(runs, sh, mx, mq, a, blocks, st)
                 : launch_tcs_bins<1, KNN_BF16>(runs, sh, mx, mq, a, blocks, st);
}

bool k1_tcs_take_timeout() { return tc_take_timeout_local(); }
bool k1_tcs_set_wait_limit(unsigned long long ns) { return tc_set_wait_limit_local(ns); }

}  // namespace tpuknn
