// k1_simt.cu -- PartialReduce (Alg. 1) fused with an FP32 SIMT contraction.
//
// The plain FP32 path: no tensor cores, exact FP32 scores and exact indices.
// Tiling follows Alg. 2 (App. A.3): a block of BQ queries stays fixed
// while the CTA walks tiles of BW database rows; the D loop runs in
// chunks of BD = 16 through double-buffered shared memory (the next chunk's
// global loads are in registers while the current chunk is multiplied), with
// a TQ x TB register tile per thread (TQ = 8: 128 queries; TQ = 4: 64, for calls
// of at most 64; TB = 4: 64 rows); after each tile the compare/select of Alg. 1 (strict '>'
// while the row index grows, so ties keep the smaller index) updates the
// running best of each (query, bin) the thread owns. The bins never change
// across tiles (tile t covers rows t*Lk + strip*64 + [0, 64)); the running
// (value, row) state of the CTA's BQ x 64 pairs lives in shared memory (one
// 16-byte load and at most two 16-byte stores per query row and tile), which
// leaves the registers to the accumulators and the operand prefetch. At the
// end the pairs merge into the [M][L] array of ordered 64-bit (score, ~row)
// keys by atomicMax, across the splits of the rows and the folds of the bins:
// the rescoring then reads L keys per query, not L pairs per split.
//
// The products are two to an instruction (fma.rn.f32x2: each half an FP32 fused
// multiply-add, so every score is the same chain as with scalar ones):
// bound by the FFMA rate and, with scalar ones, by instruction issue. 64 queries
// on 16,384 x 128 rows (L = 1024) 19.5 -> 13.4 us with 64-query tiles; an exact
// search's scores, 100 queries on 1M x 128 rows, 1.09 -> 0.65 ms (50 TFLOP/s of
// the 78 that FFMA reaches, counting the tile's 28 idle query rows).
//
// kScores: an exact search's chunk, one bin per row: the scores themselves are
// written (4 bytes each), no state and no merge; 128 rows per tile (TB = 8, with
// 128 queries and tiles for half of the SMs or more), which halves the
// shared-memory operand reads per product.
#include "common.cuh"
#include "kernels.h"

namespace tpuknn {

namespace {
constexpr int BD = 16;
constexpr int kSimtThreads = 256;  // (BQ / TQ) x (BW / TB) threads

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

template <int METRIC, int TQ, int TB, bool kScores>
__global__ void __launch_bounds__(kSimtThreads, 2)
k1_simt_kernel(const float* __restrict__ X, const float* __restrict__ hnorm,
               const float* __restrict__ Qp, K1Plan p, float* __restrict__ scores,
               unsigned long long* __restrict__ G) {
  constexpr int BQ = 16 * TQ, BW = 16 * TB, NQ4 = BQ / 64, NW4 = BW / 64;
  constexpr int PADQ = BQ + 4, PADW = BW + 4;  // row padding of the transposed tiles
  static_assert(kScores || TB == 4, "the running state is laid out for 4 bins per thread");
  __shared__ __align__(16) float Qs[2][BD][PADQ];
  __shared__ __align__(16) float Xs[2][BD][PADW];
  // running best (value, row) of each (query, bin) of the CTA: [BQ][BW]
  extern __shared__ __align__(16) float simt_state[];
  float* sv = simt_state;
  int32_t* sa = reinterpret_cast<int32_t*>(simt_state + BQ * BW);
  const int tid = threadIdx.x, tq = tid >> 4, tb = tid & 15;
  int64_t cta = blockIdx.x;
  const int64_t qtile = cta % p.nqtiles;
  cta /= p.nqtiles;
  const int64_t strip = cta % p.nstrips;
  const int64_t split = cta / p.nstrips;
  const int64_t i0 = qtile * BQ, b0 = strip * BW;
  const int64_t t_begin = split * p.tiles_per_split;
  const int64_t t_end = min(p.ntiles, t_begin + p.tiles_per_split);

  if (!kScores) {
    // this thread's entries: rows tq*TQ + r, columns tb*TB .. tb*TB + 3
#pragma unroll
    for (int r = 0; r < TQ; ++r) {
      const int o = (tq * TQ + r) * BW + tb * TB;
      *reinterpret_cast<float4*>(sv + o) = make_float4(neg_inf(), neg_inf(), neg_inf(), neg_inf());
      *reinterpret_cast<int4*>(sa + o) = make_int4(-1, -1, -1, -1);
    }
  }
  // the queries and the zeroed keys come from the preceding kernel
  pdl_wait();
  pdl_trigger();

  // loader mapping: a chunk is BQ query rows and BW database rows of BD
  // floats; thread tid loads the float4 at column lcol of rows lrow (and
  // lrow + 64 for 128 queries)
  const int lrow = tid >> 2, lcol = (tid & 3) * 4;
  const float* qp[NQ4];
  bool qv[NQ4];
#pragma unroll
  for (int u = 0; u < NQ4; ++u) {
    qv[u] = i0 + lrow + 64 * u < p.M;
    qp[u] = Qp + (qv[u] ? (i0 + lrow + 64 * u) * p.pitch + lcol : 0);
  }
  const int nchunks = p.pitch / BD;

  for (int64_t t = t_begin; t < t_end; ++t) {
    const int64_t row0 = t * p.Lk + b0;
    const float* xp[NW4];
    bool xv[NW4];
#pragma unroll
    for (int u = 0; u < NW4; ++u) {
      const int64_t xrow = row0 + lrow + 64 * u;
      xv[u] = (b0 + lrow + 64 * u < p.Lk) && (xrow < p.N);
      xp[u] = X + (xv[u] ? xrow * p.pitch + lcol : 0);
    }
    uint64_t acc[TQ / 2][TB];  // queries 2r, 2r + 1 of bin c
#pragma unroll
    for (int r = 0; r < TQ / 2; ++r)
#pragma unroll
      for (int c = 0; c < TB; ++c) acc[r][c] = 0;

    float4 nq[NQ4], nx[NW4];
    auto fetch = [&](int d0) {
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < NQ4; ++u)
        nq[u] = qv[u] ? __ldg(reinterpret_cast<const float4*>(qp[u] + d0)) : z;
#pragma unroll
      for (int u = 0; u < NW4; ++u)
        nx[u] = xv[u] ? __ldg(reinterpret_cast<const float4*>(xp[u] + d0)) : z;
    };
    auto stash = [&](int buf) {
#pragma unroll
      for (int u = 0; u < NQ4; ++u) {
        Qs[buf][lcol + 0][lrow + 64 * u] = nq[u].x;
        Qs[buf][lcol + 1][lrow + 64 * u] = nq[u].y;
        Qs[buf][lcol + 2][lrow + 64 * u] = nq[u].z;
        Qs[buf][lcol + 3][lrow + 64 * u] = nq[u].w;
      }
#pragma unroll
      for (int u = 0; u < NW4; ++u) {
        Xs[buf][lcol + 0][lrow + 64 * u] = nx[u].x;
        Xs[buf][lcol + 1][lrow + 64 * u] = nx[u].y;
        Xs[buf][lcol + 2][lrow + 64 * u] = nx[u].z;
        Xs[buf][lcol + 3][lrow + 64 * u] = nx[u].w;
      }
    };
    fetch(0);
    // the previous tile's last chunk may still be read from buffer 0 or 1:
    // every thread has passed its compare/select before buffers are refilled
    __syncthreads();
    stash(0);
    __syncthreads();
    for (int ch = 0; ch < nchunks; ++ch) {
      const int buf = ch & 1;
      if (ch + 1 < nchunks) fetch((ch + 1) * BD);
#pragma unroll
      for (int dd = 0; dd < BD; ++dd) {
        uint64_t q2[TQ / 2];
#pragma unroll
        for (int r = 0; r < TQ / 4; ++r) {
          const ulonglong2 v =
              *reinterpret_cast<const ulonglong2*>(&Qs[buf][dd][tq * TQ + 4 * r]);
          q2[2 * r] = v.x;
          q2[2 * r + 1] = v.y;
        }
#pragma unroll
        for (int w = 0; w < TB / 4; ++w) {
          const float4 x4 = *reinterpret_cast<const float4*>(&Xs[buf][dd][64 * w + tb * 4]);
          const uint64_t x2[4] = {pack2(x4.x, x4.x), pack2(x4.y, x4.y), pack2(x4.z, x4.z),
                                  pack2(x4.w, x4.w)};
#pragma unroll
          for (int r = 0; r < TQ / 2; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) fma2(acc[r][4 * w + c], q2[r], x2[c]);
        }
      }
      if (ch + 1 < nchunks) {
        // the other buffer was last read in chunk ch - 1, before the barrier
        // that ended it
        stash(buf ^ 1);
        __syncthreads();
      }
    }
    // tile column of this thread's c-th bin
    auto col = [&](int c) { return 64 * (c >> 2) + tb * 4 + (c & 3); };
    float hb[TB];
    bool valid[TB];
#pragma unroll
    for (int c = 0; c < TB; ++c) {
      const int64_t b = b0 + col(c);
      const int64_t j = row0 + col(c);
      valid[c] = (b < p.Lk) && (j < p.N);
      hb[c] = (METRIC == KNN_L2 && valid[c]) ? hnorm[j] : 0.0f;
    }
#pragma unroll
    for (int r2 = 0; r2 < TQ / 2; ++r2) {
      float sc[2][TB];
#pragma unroll
      for (int c = 0; c < TB; ++c) unpack2(acc[r2][c], sc[0][c], sc[1][c]);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int r = 2 * r2 + u;
#pragma unroll
        for (int c = 0; c < TB; ++c) sc[u][c] -= hb[c];
        if (kScores) {
          const int64_t i = i0 + tq * TQ + r;
          if (i < p.M) {
#pragma unroll
            for (int w = 0; w < TB; w += 4) {
              float* o = scores + i * ((p.Lk + 3) & ~(int64_t)3) + b0 + col(w);
              if (valid[w + 3]) {
                *reinterpret_cast<float4*>(o) =
                    make_float4(sc[u][w], sc[u][w + 1], sc[u][w + 2], sc[u][w + 3]);
              } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                  if (valid[w + c]) o[c] = sc[u][w + c];
              }
            }
          }
        } else {
          // Alg. 1 compare/select per (query, bin), against the state in shared memory
          const int o = (tq * TQ + r) * BW + tb * TB;
          float4 bv = *reinterpret_cast<const float4*>(sv + o);
          int4 ba = *reinterpret_cast<const int4*>(sa + o);
          float* bvp = reinterpret_cast<float*>(&bv);
          int* bap = reinterpret_cast<int*>(&ba);
          bool upd = false;
#pragma unroll
          for (int c = 0; c < TB; ++c) {
            if (valid[c] && sc[u][c] > bvp[c]) {
              bvp[c] = sc[u][c];
              bap[c] = (int32_t)(row0 + tb * TB + c);
              upd = true;
            }
          }
          if (upd) {
            *reinterpret_cast<float4*>(sv + o) = bv;
            *reinterpret_cast<int4*>(sa + o) = ba;
          }
        }
      }
    }
  }
  if (kScores) return;
  // merge: neighbouring threads, neighbouring keys
  __syncthreads();
  for (int e = tid; e < BQ * BW; e += kSimtThreads) {
    const int64_t i = i0 + e / BW, b = b0 + e % BW;
    if (i < p.M && b < p.Lk && sa[e] >= 0)
      atomicMax(&G[i * p.L + (p.g == 1 ? b : b % p.L)], (unsigned long long)make_key(sv[e], sa[e]));
  }
}

template <int METRIC, int TQ, int TB, bool kScores>
cudaError_t launch_simt(const K1Plan& p, const float* X, const float* hnorm, const float* Qp,
                        float* v, int64_t blocks, cudaStream_t st) {
  auto kern = k1_simt_kernel<METRIC, TQ, TB, kScores>;
  size_t smem = kScores ? 0 : (size_t)(16 * TQ) * (16 * TB) * 8;
  // Launched early, behind the query prep, CTAs go two to an SM where the first
  // SMs are free, and others stay empty. No more CTAs than SMs: each asks for
  // enough shared memory to have an SM to itself (333 queries on 3000 x 768 rows,
  // L2, 144 CTAs: 93 us a call without, 65 launched in order, 61 so; 4096 elements
  // 468, 293 and 290).
  const int64_t sms = device_sm_count();
  constexpr int kOwnSm = 96 * 1024;
  if (blocks <= sms) smem = kOwnSm;
  // Up to two to an SM, with many of them short (the last of few splits) or all of
  // them long: launched in order the short ones share SMs with the others (1000
  // queries on 3000 x 768 rows, L = 1024, 3 tiles in splits of 2 and 1: 178 and 139
  // us), and those alone on an SM are worth more than the early start (256 queries on
  // 9000 x 2000 rows, L = 2000: 479 and 380). Short even ones gain from the early
  // start (65 queries on 16,384 x 128 rows: 24 and 27 us).
  const bool in_order =
      blocks > sms && blocks < 2 * sms &&
      (4 * (p.nsplits * p.tiles_per_split - p.ntiles) >= p.ntiles ||
       p.tiles_per_split * p.pitch >= 1536);
  if (smem > 0) {
    cudaError_t e = allow_dynamic_smem(kern, kOwnSm);
    if (e != cudaSuccess) return e;
  }
  unsigned long long* G = reinterpret_cast<unsigned long long*>(v);
  if (in_order) {
    kern<<<(unsigned)blocks, kSimtThreads, smem, st>>>(X, hnorm, Qp, p, v, G);
    return cudaGetLastError();
  }
  return launch_pdl(kern, dim3((unsigned)blocks), dim3(kSimtThreads), smem, st, X, hnorm, Qp, p, v,
                    G);
}
template <int METRIC>
cudaError_t launch_simt_tile(const K1Plan& p, const float* X, const float* hnorm, const float* Qp,
                             Partials out, int64_t blocks, cudaStream_t st) {
  if (out.keys64)
    return p.BQ == 64 ? launch_simt<METRIC, 4, 4, false>(p, X, hnorm, Qp, out.v, blocks, st)
                      : launch_simt<METRIC, 8, 4, false>(p, X, hnorm, Qp, out.v, blocks, st);
  return p.BQ == 64   ? launch_simt<METRIC, 4, 4, true>(p, X, hnorm, Qp, out.v, blocks, st)
         : p.BW == 64 ? launch_simt<METRIC, 8, 4, true>(p, X, hnorm, Qp, out.v, blocks, st)
                      : launch_simt<METRIC, 8, 8, true>(p, X, hnorm, Qp, out.v, blocks, st);
}
}  // namespace

cudaError_t launch_k1_simt(const K1Plan& p, const float* X, const float* hnorm, const float* Qp,
                           Partials out, cudaStream_t st) {
  if ((p.BW != 64 && (p.BW != 128 || out.keys64 || p.BQ != 128)) ||
      (p.BQ != 64 && p.BQ != 128) || (p.pitch % BD) != 0)
    return cudaErrorInvalidValue;
  if (!out.keys64 && p.ntiles != 1) return cudaErrorInvalidValue;
  int64_t blocks = p.nsplits * p.nstrips * p.nqtiles;
  if (blocks <= 0) return cudaSuccess;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  return p.metric == KNN_L2 ? launch_simt_tile<KNN_L2>(p, X, hnorm, Qp, out, blocks, st)
                            : launch_simt_tile<KNN_IP>(p, X, hnorm, Qp, out, blocks, st);
}

}  // namespace tpuknn
