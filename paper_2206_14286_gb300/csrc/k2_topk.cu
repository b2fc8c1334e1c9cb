// k2_topk.cu -- ExactRescoring (Sec. 5): per query, merge the partial bin
// winners of every split (and fold) and select the best Kp (score, index)
// keys; fused with the FP32 re-rank for searches (rescore_kernel, k23_kernel).
//
// One CTA per query holds its L <= 8192 keys in registers. Up to Kp = 128 the
// Kp-th largest of the 256 threads' maxima bounds the selection from below:
// few keys beyond Kp reach it, and those are gathered and sorted. Larger Kp: a
// radix select. What is left streams through shared memory against the running
// Kp-th best key: more candidates (L > 8192), or a sorted selection of Kp > 1024.
#include <algorithm>

#include "common.cuh"
#include "dtypes.cuh"
#include "kernels.h"

namespace tpuknn {

namespace {

// Packed partials: a float whose low `bits` bits hold (2^bits - 1 - t_local),
// t_local the tile ordinal inside the split; the bin's row is then
// j = (s * tiles_per_split + t_local) * Lk + bin.
struct PackedSource {
  const uint32_t* p;
  int64_t M, Lk, L, nsplits, tiles_per_split, index_offset;
  int g, bits;
  __device__ __forceinline__ uint64_t key(int64_t i, int64_t b) const {
    const uint32_t mask = bits ? ((1u << bits) - 1u) : 0u;
    uint64_t best = 0;
#pragma unroll 4
    for (int64_t s = 0; s < nsplits; ++s) {
      const int64_t base = (s * M + i) * Lk + b;
      for (int f = 0; f < g; ++f) {
        const uint32_t w = p[base + (int64_t)f * L];
        if (w == kNegInfBits) continue;  // no row reached this (split, bin)
        const int64_t tl = (int64_t)(mask - (w & mask));
        const int64_t bin = b + (int64_t)f * L;
        const int64_t j = (s * tiles_per_split + tl) * Lk + bin + index_offset;
        const uint64_t k = make_key(__uint_as_float(w & ~mask), (int32_t)j);
        best = k > best ? k : best;
      }
    }
    return best;
  }
};

// Merged partials: G[i][bin] = order-mapped packed key (0 = empty) whose
// low `bits` bits hold (2^bits - 1 - t), t the global tile ordinal; the row is
// j = t * Lk + bin.
struct MergedSource {
  const uint32_t* G;
  int64_t M, Lk, L, index_offset;
  int g, bits;
  __device__ __forceinline__ uint64_t key(int64_t i, int64_t b) const {
    const uint32_t mask = bits ? ((1u << bits) - 1u) : 0u;
    uint64_t best = 0;
    for (int f = 0; f < g; ++f) {
      const int64_t bin = b + (int64_t)f * L;
      const uint32_t u = G[i * Lk + bin];
      if (u == 0u) continue;
      const uint32_t w = __float_as_uint(ordered_to_float(u));
      const int64_t t = (int64_t)(mask - (w & mask));
      const int64_t j = t * Lk + bin + index_offset;
      const uint64_t k = make_key(__uint_as_float(w & ~mask), (int32_t)j);
      best = k > best ? k : best;
    }
    return best;
  }
};

// 64-bit keys already merged per (query, bin).
struct KeySource {
  const uint64_t* G;
  int64_t L;
  __device__ __forceinline__ uint64_t key(int64_t i, int64_t b) const { return G[i * L + b]; }
};

// Descending sort of KPL keys held in registers (bitonic network).
template <int KPL>
__device__ __forceinline__ void reg_sort_desc(uint64_t (&k)[KPL]) {
#pragma unroll
  for (int size = 2; size <= KPL; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll
      for (int t = 0; t < KPL / 2; ++t) {
        const int lo = 2 * t - (t & (stride - 1));
        const int hi = lo + stride;
        const bool desc = (lo & size) == 0;
        const uint64_t x = k[lo], y = k[hi];
        const bool sw = desc ? (x < y) : (x > y);
        k[lo] = sw ? y : x;
        k[hi] = sw ? x : y;
      }
    }
  }
}

__device__ __forceinline__ uint64_t shfl_xor_u64(uint64_t v, int o) {
  const uint32_t lo = __shfl_xor_sync(0xffffffffu, (uint32_t)v, o);
  const uint32_t hi = __shfl_xor_sync(0xffffffffu, (uint32_t)(v >> 32), o);
  return ((uint64_t)hi << 32) | lo;
}

template <class Src>
__global__ void __launch_bounds__(256)
k2_topk_kernel(Src src, int64_t nelem, int Kp, int CH, int CAP, const uint64_t* __restrict__ run_in,
               uint64_t* __restrict__ out_keys) {
  extern __shared__ uint64_t sk[];
  __shared__ int cnt;
  __shared__ uint64_t thr;
  const int64_t i = blockIdx.x;
  for (int t = threadIdx.x; t < Kp; t += blockDim.x) sk[t] = run_in ? run_in[i * Kp + t] : 0;
  if (threadIdx.x == 0) {
    cnt = 0;
    thr = run_in ? run_in[i * Kp + Kp - 1] : 0;
  }
  __syncthreads();
  auto flush = [&]() {
    const int used = Kp + cnt;
    for (int t = used + threadIdx.x; t < CAP; t += blockDim.x) sk[t] = 0;
    bitonic_sort_desc(sk, CAP);
    if (threadIdx.x == 0) {
      thr = sk[Kp - 1];
      cnt = 0;
    }
    __syncthreads();
  };
  for (int64_t base = 0; base < nelem; base += blockDim.x) {
    // every thread reads the count before any thread appends again, so the
    // flush decision (which contains barriers) is the same in every thread
    const int c = cnt;
    __syncthreads();
    if (c + (int)blockDim.x > CH) flush();
    const int64_t e = base + threadIdx.x;
    if (e < nelem) {
      const uint64_t k = src.key(i, e);
      if (k > thr) {
        const int pos = atomicAdd(&cnt, 1);
        sk[Kp + pos] = k;
      }
    }
    __syncthreads();
  }
  if (cnt > 0 || run_in == nullptr) flush();
  for (int t = threadIdx.x; t < Kp; t += blockDim.x) out_keys[i * Kp + t] = sk[t];
}

template <class Src>
__global__ void merge_bins_kernel(Src src, int64_t M, int64_t L, float* __restrict__ out_v,
                                  int32_t* __restrict__ out_a) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= M * L) return;
  const uint64_t k = src.key(t / L, t % L);
  out_v[t] = k ? key_score(k) : neg_inf();
  out_a[t] = k ? key_index(k) : -1;
}

template <class Src>
cudaError_t run_k2(const Src& src, int64_t M, int64_t nelem, int Kp, const uint64_t* run_in,
                   uint64_t* out, cudaStream_t st) {
  const int threads = 256;
  const int64_t ch64 = round_up(nelem, threads);
  int CH = (int)(ch64 < 4 * threads ? ch64 : 4 * threads);
  if (CH < threads) CH = threads;
  const int CAP = next_pow2(Kp + CH);
  const size_t smem = (size_t)CAP * sizeof(uint64_t);
  constexpr int kLargest = 200 * 1024;
  if (smem > kLargest) return cudaErrorInvalidValue;
  auto kern = k2_topk_kernel<Src>;
  if (smem > 48 * 1024) {
    cudaError_t e = allow_dynamic_smem(kern, kLargest);
    if (e != cudaSuccess) return e;
  }
  if (M <= 0) return cudaSuccess;
  kern<<<(unsigned)M, threads, smem, st>>>(src, nelem, Kp, CH, CAP, run_in, out);
  return cudaGetLastError();
}

// ExactRescoring and the FP32 re-rank in one CTA of 4 warps per query, for
// the merged 64-bit keys of K1 (L <= 256, Kp <= 32, K <= 32, 16-byte
// aligned FP32 rows with D % 4 == 0). Warp 0 takes the best Kp of the L keys:
// each lane sorts its KPL keys, then every round the warp's maximum key
// comes from two 32-bit max-reductions (high word, then the low word among
// the lanes that hold the high maximum) and the lane that holds it shifts
// its list. The 4 warps then score the Kp candidates against the FP32 rows
// (a lane reads 4 consecutive elements; a warp has up to 8 rows in flight),
// and warp 0 sorts the Kp exact keys across its lanes and writes the best K.
// Same results as the two-kernel path: the candidates are the Kp largest
// keys, and the re-rank scores and orders them the same way.
template <int METRIC, int KPL>
__global__ void __launch_bounds__(128)
k23_kernel(const uint64_t* __restrict__ G, int64_t L, int Kp, int K, int D,
           const float* __restrict__ qf32, int64_t q_stride, const float* __restrict__ xf32,
           int64_t N, float* __restrict__ out_val, int32_t* __restrict__ out_idx) {
  constexpr int kWarps = 4, kPerWarp = 8;  // 4 x 8 = 32 candidates at most
  __shared__ uint64_t s_cand[32];
  __shared__ uint64_t s_key[32];
  const int64_t i = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();  // the keys come from the contraction
  pdl_trigger();  // the next call's query prep may launch (it waits for this kernel)
  if (warp == 0) {
    uint64_t k[KPL];
#pragma unroll
    for (int r = 0; r < KPL; ++r) {
      const int64_t b = lane + 32 * r;
      k[r] = b < L ? G[i * L + b] : 0;
    }
    reg_sort_desc<KPL>(k);
    uint64_t mine = 0;
    for (int r = 0; r < Kp; ++r) {
      const uint32_t hi = (uint32_t)(k[0] >> 32);
      const uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
      const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? (uint32_t)k[0] : 0u);
      const uint64_t m = ((uint64_t)mh << 32) | ml;
      if (lane == r) mine = m;
      // keys are unique (distinct rows), so one lane pops
      if (m != 0 && k[0] == m) {
#pragma unroll
        for (int t = 0; t + 1 < KPL; ++t) k[t] = k[t + 1];
        k[KPL - 1] = 0;
      }
    }
    s_cand[lane] = mine;
  }
  __syncthreads();
  const float* q = qf32 + i * q_stride;
  {
    int32_t js[kPerWarp];
    float acc[kPerWarp];
#pragma unroll
    for (int u = 0; u < kPerWarp; ++u) {
      const int c = warp + kWarps * u;
      const uint64_t key = c < Kp ? s_cand[c] : 0;
      const int32_t j = key ? key_index(key) : -1;
      js[u] = (j >= 0 && j < N) ? j : -1;
      acc[u] = 0.0f;
    }
    for (int d0 = 0; d0 < D; d0 += 128) {
      const int d = d0 + lane * 4;
      const bool in = d < D;
      const float4 qv = in ? *reinterpret_cast<const float4*>(q + d) : make_float4(0, 0, 0, 0);
      float4 xv[kPerWarp];
#pragma unroll
      for (int u = 0; u < kPerWarp; ++u)
        xv[u] = (in && js[u] >= 0)
                    ? __ldg(reinterpret_cast<const float4*>(xf32 + (int64_t)js[u] * D + d))
                    : make_float4(0, 0, 0, 0);
#pragma unroll
      for (int u = 0; u < kPerWarp; ++u) {
        if (METRIC == KNN_L2) {
          // elements past D contribute 0: both sides are zero there
          const float t0 = qv.x - xv[u].x, t1 = qv.y - xv[u].y, t2 = qv.z - xv[u].z,
                      t3 = qv.w - xv[u].w;
          acc[u] = fmaf(t0, t0, acc[u]);
          acc[u] = fmaf(t1, t1, acc[u]);
          acc[u] = fmaf(t2, t2, acc[u]);
          acc[u] = fmaf(t3, t3, acc[u]);
        } else {
          acc[u] = fmaf(qv.x, xv[u].x, acc[u]);
          acc[u] = fmaf(qv.y, xv[u].y, acc[u]);
          acc[u] = fmaf(qv.z, xv[u].z, acc[u]);
          acc[u] = fmaf(qv.w, xv[u].w, acc[u]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kPerWarp; ++u) {
      float v = acc[u];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const int c = warp + kWarps * u;
      if (lane == 0 && c < 32)
        s_key[c] = js[u] >= 0 ? make_key(METRIC == KNN_L2 ? -v : v, js[u]) : 0;
    }
  }
  __syncthreads();
  if (warp != 0) return;
  uint64_t mine = s_key[lane];
#pragma unroll
  for (int k2 = 2; k2 <= 32; k2 <<= 1) {
#pragma unroll
    for (int jj = k2 >> 1; jj > 0; jj >>= 1) {
      const uint64_t other = shfl_xor_u64(mine, jj);
      const bool up = (lane & k2) == 0, lower = (lane & jj) == 0;
      const bool keep_max = (up == lower);
      mine = keep_max ? (other > mine ? other : mine) : (other < mine ? other : mine);
    }
  }
  if (lane < K) {
    const float sc = key_score(mine);
    out_idx[i * K + lane] = mine ? key_index(mine) : -1;
    out_val[i * K + lane] = mine ? (METRIC == KNN_L2 ? -sc : sc) : __int_as_float(0x7fc00000);
  }
}

template <int METRIC>
cudaError_t run_k23(const uint64_t* G, int64_t M, int64_t L, int Kp, int K, int D,
                    const float* qf32, int64_t q_stride, const float* xf32, int64_t N,
                    float* out_val, int32_t* out_idx, cudaStream_t st) {
  const int kpl = next_pow2((int)cdiv(L, 32));
  const unsigned blocks = (unsigned)M;
#define K23_CASE(P)                                                                          \
  case P:                                                                                    \
    return launch_pdl(k23_kernel<METRIC, P>, dim3(blocks), dim3(128), 0, st, G, L, Kp, K, D, \
                      qf32, q_stride, xf32, N, out_val, out_idx);
  switch (kpl) {
    K23_CASE(1)
    K23_CASE(2)
    K23_CASE(4)
    K23_CASE(8)
    default: return cudaErrorNotSupported;
  }
#undef K23_CASE
}


// Warp 0 of a radix-select pass: the digit where the count of the histogram's
// bins from the top reaches `need`, the keys in the bins above it, and
// whether every key in it is needed.
__device__ __forceinline__ void pick_digit(const uint32_t* hist, int need, int lane, int& s_digit,
                                           int& s_above, int& s_stop) {
  // lane l sums bins 255-8l .. 248-8l; counts from the top by a warp scan
  uint32_t c[8], sum = 0;
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    c[t] = hist[255 - 8 * lane - t];
    sum += c[t];
  }
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const uint32_t excl = incl - sum;  // keys matching the prefix in higher bins
  const bool mine = excl < (uint32_t)need && (uint32_t)need <= incl;
  const unsigned who = __ballot_sync(0xffffffffu, mine);
  if (who == 0) {
    // fewer matching keys than needed cannot happen for need <= L
    if (lane == 0) {
      s_digit = 0;
      s_above = 0;
      s_stop = 1;
    }
  } else if (mine) {
    uint32_t above = excl, ct = 0;
    int tf = 7;
    bool found = false;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (!found) {
        if (above + c[t] >= (uint32_t)need) {
          tf = t;
          ct = c[t];
          found = true;
        } else {
          above += c[t];
        }
      }
    }
    s_digit = 255 - 8 * lane - tf;
    s_above = (int)above;
    s_stop = (above + ct == (uint32_t)need) ? 1 : 0;
  }
}

constexpr int kTopkElems = 8192, kTopkCap = 1024, kThrMaxK = 128;

// The selection of one CTA of 256 threads.
struct SelectSmem {
  uint64_t buf[kTopkCap];
  uint32_t w[256];  // maxima, or a histogram
  int cnt, digit, above, stop;
};

// The K-th largest of the 256 threads' x (K <= 256): a bitonic sort, one value
// per thread.
__device__ __forceinline__ uint32_t kth_of_threads(uint32_t x, int K, uint32_t* w) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int size = 2; size <= 256; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      uint32_t y;
      if (stride >= 32) {
        __syncthreads();
        w[tid] = x;
        __syncthreads();
        y = w[tid ^ stride];
      } else {
        y = __shfl_xor_sync(0xffffffffu, x, stride);
      }
      const bool keep_max = ((tid & stride) == 0) == ((tid & size) == 0);
      x = keep_max ? max(x, y) : min(x, y);
    }
  }
  __syncthreads();
  w[tid] = x;
  __syncthreads();
  return w[K - 1];
}

// The keys of buf[0..c), c <= kTopkCap, sorted best first; buf is zero from c
// to `fill` afterwards. All 256 threads; ends with a barrier.
__device__ __forceinline__ void sort_buf(uint64_t* buf, int c, int fill) {
  const int tid = threadIdx.x, lane = tid & 31;
  if (c <= 32) {
    if (tid < 32) {
      uint64_t x = lane < c ? buf[lane] : 0;
#pragma unroll
      for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
          const uint64_t y = shfl_xor_u64(x, stride);
          const bool keep_max = ((lane & stride) == 0) == ((lane & size) == 0);
          x = keep_max ? (y > x ? y : x) : (y < x ? y : x);
        }
      }
      buf[lane] = x;
    }
    for (int t = 32 + tid; t < fill; t += 256) buf[t] = 0;
    __syncthreads();
    return;
  }
  const int P2 = next_pow2(c);
  for (int t = c + tid; t < max(P2, fill); t += 256) buf[t] = 0;
  bitonic_sort_desc(buf, P2);
}

// The best Kp of the CTA's L keys (thread t holds keys t + 256 u) into
// dst[0..Kp): sorted best first if `sorted`, else as a set. dst is sm.buf for
// Kp <= kTopkCap; more keys, as a set only, go to global memory.
//
// Up to kThrMaxK: the Kp-th largest of the threads' maxima (high words) is a
// lower bound of the Kp-th largest key; the keys that reach it are gathered.
// Beyond, or if more reach it than the buffer holds (ties): a radix select,
// 8 bits per pass from the top, a 256-bin histogram of the keys that match
// the digits chosen so far, stopping once every matching key is needed. Keys
// are distinct but for empty ones (0), so the set is that of a sort.
template <int KPT>
__device__ __forceinline__ void select_topk(const uint64_t (&k)[KPT], int L, int Kp, bool sorted,
                                            SelectSmem& sm, uint64_t* dst) {
  const int tid = threadIdx.x, lane = tid & 31;
  bool radix = Kp > kThrMaxK;
  if (tid == 0) sm.cnt = 0;
  if (!radix) {
    uint32_t mx = 0;
#pragma unroll
    for (int u = 0; u < KPT; ++u) mx = max(mx, (uint32_t)(k[u] >> 32));
    const uint32_t thr = max(kth_of_threads(mx, Kp, sm.w), 1u);
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      if ((uint32_t)(k[u] >> 32) >= thr) {
        const int p = atomicAdd(&sm.cnt, 1);
        if (p < kTopkCap) sm.buf[p] = k[u];
      }
    }
    __syncthreads();
    const int c = sm.cnt;
    radix = c > kTopkCap;
    if (!radix) {
      if (sorted || c > Kp) {
        sort_buf(sm.buf, c, Kp);
      } else {
        for (int t = c + tid; t < Kp; t += 256) sm.buf[t] = 0;
        __syncthreads();
      }
      return;
    }
  }
  uint64_t prefix = 0, mask = 0;
  int need = min(Kp, L);  // keys still to take among those matching the prefix
  for (int shift = 56; shift >= 0; shift -= 8) {
    __syncthreads();
    sm.w[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < KPT; ++u)
      if (u * 256 + tid < L && (k[u] & mask) == prefix)
        atomicAdd(&sm.w[(uint32_t)(k[u] >> shift) & 255u], 1u);
    __syncthreads();
    if (tid < 32) pick_digit(sm.w, need, lane, sm.digit, sm.above, sm.stop);
    __syncthreads();
    prefix |= (uint64_t)sm.digit << shift;
    mask |= (uint64_t)0xFF << shift;
    need -= sm.above;
    if (sm.stop) break;
  }
  // the keys above the prefix (masked), then `need` of those matching it
  const int n_hi = min(Kp, L) - need;
  __syncthreads();
  if (tid == 0) {
    sm.cnt = 0;
    sm.above = 0;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < KPT; ++u) {
    if (u * 256 + tid >= L) continue;
    const uint64_t m = k[u] & mask;
    if (m > prefix) {
      dst[atomicAdd(&sm.cnt, 1)] = k[u];
    } else if (m == prefix) {
      const int p = atomicAdd(&sm.above, 1);
      if (p < need) dst[n_hi + p] = k[u];
    }
  }
  for (int t = L + tid; t < Kp; t += 256) dst[t] = 0;  // Kp > L: empty
  __syncthreads();
  if (sorted) sort_buf(sm.buf, Kp, Kp);
}

template <class Src, int KPT>
__device__ __forceinline__ void load_keys(const Src& src, int64_t i, int L, uint64_t (&k)[KPT]) {
#pragma unroll
  for (int u = 0; u < KPT; ++u) {
    const int b = u * 256 + threadIdx.x;
    k[u] = b < L ? src.key(i, b) : 0;
  }
}

// ExactRescoring alone: the best Kp keys of each query, as keys or (out_val
// given) as values, negated when `neg`, and indices. kDirect: more than kTopkCap
// keys (a set for a re-rank) are written as they are gathered: 1000 queries, L =
// 8192, 1600 candidates of 64 elements 375 us a search; the streaming kernel
// below, whose sorted buffer holds them all, 1513.
// (three CTAs per SM with up to 8192 keys: 10,000 queries 1.18 -> 0.91 ms)
template <class Src, int KPT, bool kDirect>
__global__ void __launch_bounds__(256, KPT == 32 ? 3 : 4)
k2_select_kernel(Src src, int L, int Kp, bool sorted, uint64_t* __restrict__ out_keys, int neg,
                 float* __restrict__ out_val, int32_t* __restrict__ out_idx) {
  __shared__ SelectSmem sm;
  const int64_t i = blockIdx.x;
  pdl_wait();
  uint64_t k[KPT];
  load_keys(src, i, L, k);
  if constexpr (kDirect) {
    select_topk(k, L, Kp, false, sm, out_keys + i * Kp);
    return;
  }
  select_topk(k, L, Kp, sorted, sm, sm.buf);
  for (int t = threadIdx.x; t < Kp; t += 256) {
    const uint64_t key = sm.buf[t];
    if (out_val) {
      out_val[i * Kp + t] =
          key ? (neg ? -key_score(key) : key_score(key)) : __int_as_float(0x7fc00000);
      out_idx[i * Kp + t] = key ? key_index(key) : -1;
    } else {
      out_keys[i * Kp + t] = key;
    }
  }
}

// ExactRescoring and the FP32 re-rank of its Kp candidates in one launch: the
// candidates stay in shared memory, the 8 warps score four of them at a time
// (eight in the re-rank alone; their row loads in flight together), and the
// best K of the exact keys are sorted and written: 4096 queries, L = 605, 64
// candidates of 256 elements 160 -> 75 us, against one warp per query for the
// selection and a second launch. The re-rank alone of 2000 x 800 rows of 96:
// 224 -> 180 us (3.4 TB/s of gathered rows). The scores are those of the separate re-rank, sum by
// sum: VEC4 (Kp <= 32, 16-byte aligned FP32 rows) a lane owns 4 adjacent
// elements of each 128, else every 32nd element. KPT = 0: the re-rank alone, of
// Kp <= 1024 candidates that src holds.
struct RescoreArgs {
  int L, Kp, K, D, metric, dtype, pitch;
  const float* qf32;
  int64_t q_stride;
  const float* xf32;
  const void* xlp;
  const float* xscale;
  int64_t N;
  float* out_val;
  int32_t* out_idx;
};

template <class Src, int KPT, bool VEC4>
__global__ void __launch_bounds__(256) rescore_kernel(Src src, RescoreArgs a) {
  __shared__ SelectSmem sm;
  const int64_t i = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_wait();     // the keys come from the contraction
  pdl_trigger();  // the next call's query prep may launch (it waits for this kernel)
  if constexpr (KPT == 0) {
    for (int t = tid; t < a.Kp; t += 256) sm.buf[t] = src.key(i, t);
    __syncthreads();
  } else {
    uint64_t k[KPT];
    load_keys(src, i, a.L, k);
    select_topk(k, a.L, a.Kp, false, sm, sm.buf);
  }
  const float* q = a.qf32 + i * a.q_stride;
  constexpr int kCand = KPT == 0 ? 8 : 4;
  for (int c0 = warp * kCand; c0 < a.Kp; c0 += 8 * kCand) {
    int32_t jj[kCand];
    float acc[kCand];
#pragma unroll
    for (int u = 0; u < kCand; ++u) {
      const uint64_t key = c0 + u < a.Kp ? sm.buf[c0 + u] : 0;
      const int32_t j = key ? key_index(key) : -1;
      jj[u] = (j >= 0 && j < a.N) ? j : -1;
      acc[u] = 0.0f;
    }
    if constexpr (VEC4) {
      for (int d0 = 0; d0 < a.D; d0 += 128) {
        const int d = d0 + lane * 4;
        const bool in = d < a.D;
        const float4 qv = in ? *reinterpret_cast<const float4*>(q + d) : make_float4(0, 0, 0, 0);
        float4 xv[kCand];
#pragma unroll
        for (int u = 0; u < kCand; ++u)
          xv[u] = (in && jj[u] >= 0)
                      ? __ldg(reinterpret_cast<const float4*>(a.xf32 + (int64_t)jj[u] * a.D + d))
                      : make_float4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < kCand; ++u) {
          if (a.metric == KNN_L2) {
            // elements past D contribute 0: both sides are zero there
            const float t0 = qv.x - xv[u].x, t1 = qv.y - xv[u].y, t2 = qv.z - xv[u].z,
                        t3 = qv.w - xv[u].w;
            acc[u] = fmaf(t0, t0, acc[u]);
            acc[u] = fmaf(t1, t1, acc[u]);
            acc[u] = fmaf(t2, t2, acc[u]);
            acc[u] = fmaf(t3, t3, acc[u]);
          } else {
            acc[u] = fmaf(qv.x, xv[u].x, acc[u]);
            acc[u] = fmaf(qv.y, xv[u].y, acc[u]);
            acc[u] = fmaf(qv.z, xv[u].z, acc[u]);
            acc[u] = fmaf(qv.w, xv[u].w, acc[u]);
          }
        }
      }
    } else {
      for (int d = lane; d < a.D; d += 32) {
        const float qq = q[d];
        float xv[kCand];
#pragma unroll
        for (int u = 0; u < kCand; ++u)
          xv[u] = jj[u] < 0 ? 0.0f
                            : (a.xf32 ? a.xf32[(int64_t)jj[u] * a.D + d]
                                      : load_stored(a.xlp, a.dtype, jj[u], a.pitch, d, a.xscale));
#pragma unroll
        for (int u = 0; u < kCand; ++u) {
          if (a.metric == KNN_L2) {
            const float t = qq - xv[u];
            acc[u] = fmaf(t, t, acc[u]);
          } else {
            acc[u] = fmaf(qq, xv[u], acc[u]);
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kCand; ++u) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
    }
    __syncwarp();  // every lane has read these candidates
    if (lane == 0) {
#pragma unroll
      for (int u = 0; u < kCand; ++u)
        if (c0 + u < a.Kp)
          sm.buf[c0 + u] =
              jj[u] < 0 ? 0 : make_key(a.metric == KNN_L2 ? -acc[u] : acc[u], jj[u]);
    }
  }
  __syncthreads();
  if (a.Kp <= 256 || a.K > kThrMaxK) {
    sort_buf(sm.buf, a.Kp, a.Kp);
  } else {
    // many candidates, few wanted: select again, from registers
    uint64_t k[kTopkCap / 256];
#pragma unroll
    for (int u = 0; u < kTopkCap / 256; ++u) {
      const int c = u * 256 + tid;
      k[u] = c < a.Kp ? sm.buf[c] : 0;
    }
    __syncthreads();
    select_topk(k, a.Kp, a.K, true, sm, sm.buf);
  }
  for (int t = tid; t < a.K; t += 256) {
    const uint64_t key = sm.buf[t];
    const float sc = key_score(key);
    a.out_idx[i * a.K + t] = key ? key_index(key) : -1;
    a.out_val[i * a.K + t] =
        key ? (a.metric == KNN_L2 ? -sc : sc) : __int_as_float(0x7fc00000);
  }
}

// ExactRescoring of few bins, as values and indices, by one warp per query: each
// lane sorts its KPL keys, then K rounds take the warp's maximum key (see
// k23_kernel). For many queries: a CTA of 256 threads for each leaves most of
// them without a key. 10,000 queries, K = 10, L = 16, 128, 256, 512: 50, 50, 58, 71 us
// a call by CTAs, 23, 25, 35, 55 by warps (K = 64: 75 and 60 at L = 128, 109 and 126
// at 512); up to 3000 queries both take the same.
template <int KPL>
__global__ void __launch_bounds__(256)
k2_warp_kernel(const uint64_t* __restrict__ G, int64_t M, int L, int K, int neg,
               float* __restrict__ out_val, int32_t* __restrict__ out_idx) {
  const int lane = threadIdx.x & 31;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= M) return;
  uint64_t k[KPL];
#pragma unroll
  for (int r = 0; r < KPL; ++r) {
    const int b = lane + 32 * r;
    k[r] = b < L ? G[i * L + b] : 0;
  }
  reg_sort_desc<KPL>(k);
  for (int r = 0; r < K; ++r) {
    const uint32_t hi = (uint32_t)(k[0] >> 32);
    const uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? (uint32_t)k[0] : 0u);
    const uint64_t m = ((uint64_t)mh << 32) | ml;
    if (lane == (r & 31)) {
      out_val[i * K + r] = m ? (neg ? -key_score(m) : key_score(m)) : __int_as_float(0x7fc00000);
      out_idx[i * K + r] = m ? key_index(m) : -1;
    }
    if (m != 0 && k[0] == m) {
#pragma unroll
      for (int t = 0; t + 1 < KPL; ++t) k[t] = k[t + 1];
      k[KPL - 1] = 0;
    }
  }
}
bool k2_warp_better(int64_t M, int64_t L, int K) {
  return M >= 16 * device_sm_count() && (L <= 256 ? K <= 64 : L <= 512 && K <= 16);
}
cudaError_t run_k2_warp(const uint64_t* G, int64_t M, int64_t L, int K, int neg, float* out_val,
                        int32_t* out_idx, cudaStream_t st) {
  const int64_t blocks = cdiv(M, 8);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto kern = L <= 32    ? k2_warp_kernel<1>
              : L <= 64  ? k2_warp_kernel<2>
              : L <= 128 ? k2_warp_kernel<4>
              : L <= 256 ? k2_warp_kernel<8>
                         : k2_warp_kernel<16>;
  kern<<<(unsigned)blocks, 256, 0, st>>>(G, M, (int)L, K, neg, out_val, out_idx);
  return cudaGetLastError();
}

// Launches a kernel of one CTA per query that selects (and re-ranks) Kp keys.
// Launched early behind a contraction it saves about 2 us, but its CTAs then go
// where the first SMs fall free, four to eight to an SM while others idle: with
// 100 queries, L = 1024 and 1024 candidates of 64 elements 90 us a search,
// launched in order 49. It is launched early where the CTAs are short (Kp <= 32:
// in order the same or up to 9% longer, M = 1 to 800), few (16 queries, Kp = 256:
// 0-12% longer; 1024 candidates of 16 queries on 200,000 rows 31% less), or so many
// that they fill the chip either way (800 queries 0-8% longer; 450 queries, Kp = 40,
// 128, 512: 0-3, 4-15, 4-23% less).
template <typename... KArgs, typename... Args>
cudaError_t launch_per_query(void (*kernel)(KArgs...), int64_t M, bool early, cudaStream_t st,
                             Args... args) {
  if (early) return launch_pdl(kernel, dim3((unsigned)M), dim3(256), 0, st, args...);
  kernel<<<(unsigned)M, 256, 0, st>>>(args...);
  return cudaGetLastError();
}
bool early_better(int64_t M, int Kp) {
  return Kp <= 32 || M <= 8 || (M <= 32 && Kp <= 256) || M >= 4 * device_sm_count();
}

template <class Src>
cudaError_t run_k2_select(const Src& src, int64_t M, int64_t L, int Kp, bool sorted, uint64_t* out,
                          int neg, float* out_val, int32_t* out_idx, cudaStream_t st) {
  auto kern = L <= 1024   ? k2_select_kernel<Src, 4, false>
              : L <= 2048 ? k2_select_kernel<Src, 8, false>
              : L <= 4096 ? k2_select_kernel<Src, 16, false>
                          : k2_select_kernel<Src, 32, false>;
  if (Kp > kTopkCap)
    kern = L <= 2048   ? k2_select_kernel<Src, 8, true>
           : L <= 4096 ? k2_select_kernel<Src, 16, true>
                       : k2_select_kernel<Src, 32, true>;
  // (values and indices follow kernels that let nothing start early: no crowding)
  return launch_per_query(kern, M, out_val || early_better(M, Kp), st, src, (int)L, Kp, sorted,
                          out, neg, out_val, out_idx);
}
template <class Src, bool VEC4>
cudaError_t run_rescore(const Src& src, int64_t M, const RescoreArgs& a, cudaStream_t st) {
  auto kern = a.L <= 1024 ? rescore_kernel<Src, 4, VEC4> : rescore_kernel<Src, 8, VEC4>;
  return launch_per_query(kern, M, early_better(M, a.Kp), st, src, a);
}

// ---------------------------------------------------------------------------
// Top-K of an exact search: a CTA takes the best K of up to 8192 elements of
// one query, so that many CTAs share a query's scores (one CTA per query
// streaming all of them left 100 queries on 100 SMs: 3.4 ms for 1M rows), and
// a second launch takes the best K of the CTAs' and the earlier chunks' keys.
//
// Up to K = kThrMaxK: each of 256 threads holds 32 elements; the K-th largest
// of the 256 threads' maxima is a lower bound of the K-th largest element, and
// few elements beyond K reach it (about 126 for K = 100 of 8192), so those are
// gathered and sorted, and no element is looked at more than twice: 0.18 ms
// for 100 queries of 1M scores, K = 10, with the merge. Larger K,
// or more elements at the bound than the buffer holds (ties): a radix select
// over the keys, read again in every pass.
// ---------------------------------------------------------------------------
// Scores of a chunk: element e of query i as an ordered 64-bit key (0: no
// candidate, which -inf and NaN are not). raw() is what a thread loads, with
// no condition around it, so that its loads are all in flight together.
struct ScoreSource {
  const float* v;
  int64_t ld, row0;
  typedef float Raw;
  __device__ __forceinline__ float raw(int64_t i, int64_t e) const { return v[i * ld + e]; }
  static __device__ __forceinline__ uint32_t high(float s) {
    return s > neg_inf() ? float_to_ordered(s) : 0u;
  }
  __device__ __forceinline__ uint64_t key(int64_t i, int64_t e) const {
    const uint32_t h = high(raw(i, e));
    return h ? ((uint64_t)h << 32) | (uint32_t)~(uint32_t)(row0 + e) : 0;
  }
};
// The K keys of the running set (if any), then the CTAs' keys.
struct MergeSource {
  const uint64_t* run;
  const uint64_t* cand;
  int64_t nrun, ncand;  // per query
  typedef uint32_t Raw;
  __device__ __forceinline__ const uint64_t* at(int64_t i, int64_t e) const {
    return e < nrun ? run + (i * nrun + e) : cand + (i * ncand + e - nrun);
  }
  __device__ __forceinline__ uint32_t raw(int64_t i, int64_t e) const {
    return reinterpret_cast<const uint32_t*>(at(i, e))[1];
  }
  static __device__ __forceinline__ uint32_t high(uint32_t h) { return h; }
  __device__ __forceinline__ uint64_t key(int64_t i, int64_t e) const { return *at(i, e); }
};

template <class Src>
__global__ void __launch_bounds__(256)
block_topk_kernel(Src src, int64_t n, int64_t nblk, int K, uint64_t* __restrict__ out) {
  constexpr int KPT = kTopkElems / 256;
  __shared__ SelectSmem sm;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t i = blockIdx.x / nblk, blk = blockIdx.x % nblk;
  const int64_t e0 = blk * kTopkElems;
  const int m = (int)min((int64_t)kTopkElems, n - e0);  // elements of this CTA
  uint64_t* o = out + (i * nblk + blk) * K;
  if (tid == 0) sm.cnt = 0;
  bool overflow = K > kThrMaxK;
  if (!overflow) {
    typename Src::Raw raw[KPT];
#pragma unroll
    for (int u = 0; u < KPT; ++u) raw[u] = src.raw(i, e0 + min(u * 256 + tid, m - 1));
    uint32_t h[KPT], mx = 0;
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      h[u] = u * 256 + tid < m ? Src::high(raw[u]) : 0u;
      mx = max(mx, h[u]);
    }
    const uint32_t thr = max(kth_of_threads(mx, K, sm.w), 1u);
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      if (h[u] >= thr) {
        const int p = atomicAdd(&sm.cnt, 1);
        if (p < kTopkCap) sm.buf[p] = src.key(i, e0 + u * 256 + tid);
      }
    }
    __syncthreads();
    overflow = sm.cnt > kTopkCap;
  }
  if (!overflow) {
    sort_buf(sm.buf, sm.cnt, K);
    for (int t = tid; t < K; t += 256) o[t] = sm.buf[t];
    return;
  }
  // radix select, 8 bits per pass from the top, over the keys in memory
  uint64_t prefix = 0, mask = 0;
  int need = min(K, m);
  for (int shift = 56; shift >= 0; shift -= 8) {
    __syncthreads();
    sm.w[tid] = 0;
    __syncthreads();
    for (int e = tid; e < m; e += 256) {
      const uint64_t k = src.key(i, e0 + e);
      if ((k & mask) == prefix) atomicAdd(&sm.w[(uint32_t)(k >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (tid < 32) pick_digit(sm.w, need, lane, sm.digit, sm.above, sm.stop);
    __syncthreads();
    prefix |= (uint64_t)sm.digit << shift;
    mask |= (uint64_t)0xFF << shift;
    need -= sm.above;
    if (sm.stop) break;
  }
  // the keys above the prefix, then `need` of those matching it (all of them,
  // but for repeated empty keys)
  const int total = min(K, m), n_hi = total - need;
  __syncthreads();
  if (tid == 0) {
    sm.cnt = 0;
    sm.above = 0;
  }
  __syncthreads();
  for (int e = tid; e < m; e += 256) {
    const uint64_t k = src.key(i, e0 + e);
    if ((k & mask) > prefix) {
      o[atomicAdd(&sm.cnt, 1)] = k;
    } else if ((k & mask) == prefix) {
      const int p = atomicAdd(&sm.above, 1);
      if (p < need) o[n_hi + p] = k;
    }
  }
  for (int t = total + tid; t < K; t += 256) o[t] = 0;
}

}  // namespace

// Per query: one CTA with the candidates in registers up to 8192 of them, and
// 1024 selected if they are to be sorted; the streaming CTA kernel everything else.
template <class Src>
cudaError_t dispatch_k2(const Src& s, const K1Plan& p, int Kp, uint64_t* out_keys, bool sorted,
                        cudaStream_t st) {
  if (p.L <= kTopkElems && (Kp <= kTopkCap || !sorted) && p.M <= 0x7fffffffLL)
    return run_k2_select(s, p.M, p.L, Kp, sorted, out_keys, 0, nullptr, nullptr, st);
  return run_k2(s, p.M, p.L, Kp, nullptr, out_keys, st);
}

// f(source) for the form the partials have.
template <class F>
cudaError_t with_source(const K1Plan& p, const Partials& parts, F f) {
  if (parts.keys64) return f(KeySource{reinterpret_cast<const uint64_t*>(parts.v), p.L});
  if (parts.merged)
    return f(MergedSource{reinterpret_cast<const uint32_t*>(parts.v), p.M, p.Lk, p.L,
                          parts.index_offset, p.g, p.code_bits});
  return f(PackedSource{reinterpret_cast<const uint32_t*>(parts.v), p.M, p.Lk, p.L, p.nsplits,
                        p.tiles_per_split, parts.index_offset, p.g, p.code_bits});
}

cudaError_t launch_merge_bins(const K1Plan& p, Partials parts, float* out_v, int32_t* out_a,
                              cudaStream_t st) {
  const int64_t n = p.M * p.L;
  if (n <= 0) return cudaSuccess;
  return with_source(p, parts, [&](auto s) {
    merge_bins_kernel<<<(unsigned)cdiv(n, 256), 256, 0, st>>>(s, p.M, p.L, out_v, out_a);
    return cudaGetLastError();
  });
}

cudaError_t launch_k2(const K1Plan& p, Partials parts, int Kp, uint64_t* out_keys, cudaStream_t st,
                      bool sorted) {
  if (p.M <= 0) return cudaSuccess;
  return with_source(
      p, parts, [&](auto s) { return dispatch_k2(s, p, Kp, out_keys, sorted, st); });
}

cudaError_t launch_k2_pairs(const uint64_t* keys, int64_t M, int64_t L, int K, int neg,
                            uint64_t* scratch, float* out_val, int32_t* out_idx,
                            cudaStream_t st) {
  if (M <= 0) return cudaSuccess;
  if (k2_warp_better(M, L, K)) return run_k2_warp(keys, M, L, K, neg, out_val, out_idx, st);
  const KeySource s{keys, L};
  if (L <= kTopkElems && K <= kTopkCap && M <= 0x7fffffffLL)
    return run_k2_select(s, M, L, K, true, nullptr, neg, out_val, out_idx, st);
  cudaError_t e = run_k2(s, M, L, K, nullptr, scratch, st);
  return e == cudaSuccess ? launch_keys_to_pairs(scratch, M * K, neg, out_val, out_idx, st) : e;
}

// (With up to 8192 keys the selection holds 64 registers of them a thread and
// two CTAs fit an SM, too few for the re-rank's row loads: 2M x 96 E4M3 rows, L
// = 8192, 800 candidates, 2000 queries, 1.107 ms a search against 1.011 with
// two launches. At the line, 60,000 x 64 BF16 rows: 6000 queries and 132 candidates
// 305 us fused with L = 2048, 341 by two launches with 2049; 1000 and 800, 110 and 120.)
bool rescore_supported(const K1Plan& p, int Kp) {
  return p.L <= 2048 && Kp <= kTopkCap && p.M <= 0x7fffffffLL;
}

cudaError_t launch_rescore(const K1Plan& p, Partials parts, int Kp, int K, const float* qf32,
                           int64_t q_stride, const float* xf32, const void* xlp, int dtype,
                           const float* xscale, int64_t N, float* out_val, int32_t* out_idx,
                           cudaStream_t st) {
  if (p.M <= 0) return cudaSuccess;
  if (!rescore_supported(p, Kp)) return cudaErrorNotSupported;
  const RescoreArgs a{(int)p.L, Kp,   K,   p.D,    p.metric, dtype,   p.pitch, qf32,
                      q_stride, xf32, xlp, xscale, N,        out_val, out_idx};
  // the sums of the separate re-rank's vector kernel, where that would run
  const bool vec4 = Kp <= 32 && K <= 32 && xf32 && p.D % 4 == 0 && q_stride % 4 == 0 &&
                    (reinterpret_cast<uintptr_t>(xf32) & 15) == 0 &&
                    (reinterpret_cast<uintptr_t>(qf32) & 15) == 0;
  return with_source(p, parts, [&](auto s) {
    return vec4 ? run_rescore<decltype(s), true>(s, p.M, a, st)
                : run_rescore<decltype(s), false>(s, p.M, a, st);
  });
}

cudaError_t launch_rerank(int64_t M, int D, int metric, const uint64_t* cand, int Kp, int K,
                          const float* qf32, int64_t q_stride, const float* xf32, const void* xlp,
                          int dtype, int pitch, const float* xscale, int64_t N, float* out_val,
                          int32_t* out_idx, cudaStream_t st) {
  if (M <= 0) return cudaSuccess;
  if (Kp > kTopkCap || M > 0x7fffffffLL) return cudaErrorNotSupported;
  const RescoreArgs a{Kp,       Kp,   K,   D,      metric, dtype,   pitch, qf32,
                      q_stride, xf32, xlp, xscale, N,      out_val, out_idx};
  return launch_pdl(rescore_kernel<KeySource, 0, false>, dim3((unsigned)M), dim3(256), 0, st,
                    KeySource{cand, Kp}, a);
}

int64_t exact_chunk_rows(int K) {
  // the second launch merges the running K keys and every CTA's in one CTA
  return std::max<int64_t>(1, kTopkElems / K - 1) * kTopkElems;
}

size_t exact_cand_bytes(int64_t M, int64_t n, int K) {
  return (size_t)(M * cdiv(n, kTopkElems) * K) * 8;
}

cudaError_t launch_exact_topk(const float* scores, int64_t ld, int64_t M, int64_t n, int64_t row0,
                              int K, const uint64_t* run_in, uint64_t* run_out, uint64_t* cand,
                              cudaStream_t st) {
  if (M <= 0 || n <= 0) return cudaSuccess;
  const int64_t nblk = cdiv(n, kTopkElems);
  const int64_t nmerge = (run_in ? K : 0) + nblk * K;
  if (K < 1 || K > kExactMaxK || nmerge > kTopkElems || M * nblk > 0x7fffffffLL)
    return cudaErrorInvalidValue;
  const ScoreSource s{scores, ld, row0};
  if (nblk == 1 && !run_in) {
    block_topk_kernel<<<(unsigned)M, 256, 0, st>>>(s, n, (int64_t)1, K, run_out);
    return cudaGetLastError();
  }
  block_topk_kernel<<<(unsigned)(M * nblk), 256, 0, st>>>(s, n, nblk, K, cand);
  const MergeSource ms{run_in, cand, run_in ? K : 0, nblk * K};
  block_topk_kernel<<<(unsigned)M, 256, 0, st>>>(ms, nmerge, (int64_t)1, K, run_out);
  return cudaGetLastError();
}

cudaError_t launch_k2_scores(const float* scores, int64_t ld, int64_t M, int64_t n, int64_t row0,
                             int K, const uint64_t* run_in, uint64_t* run_out, cudaStream_t st) {
  return run_k2(ScoreSource{scores, ld, row0}, M, n, K, run_in, run_out, st);
}

bool k23_supported(int64_t M, int64_t L, int Kp, int K, int D, const float* qf32,
                   int64_t q_stride, const float* xf32) {
  return M > 0 && M <= 0x7fffffffLL && L >= 1 && L <= 256 && Kp >= 1 && Kp <= 32 &&
         K >= 1 && K <= 32 && xf32 && D % 4 == 0 && q_stride % 4 == 0 &&
         (reinterpret_cast<uintptr_t>(xf32) & 15) == 0 &&
         (reinterpret_cast<uintptr_t>(qf32) & 15) == 0;
}

cudaError_t launch_k23(const uint64_t* G, int64_t M, int64_t L, int Kp, int K, int D, int metric,
                       const float* qf32, int64_t q_stride, const float* xf32, int64_t N,
                       float* out_val, int32_t* out_idx, cudaStream_t st) {
  if (M <= 0) return cudaSuccess;
  if (!k23_supported(M, L, Kp, K, D, qf32, q_stride, xf32)) return cudaErrorNotSupported;
  return metric == KNN_L2 ? run_k23<KNN_L2>(G, M, L, Kp, K, D, qf32, q_stride, xf32, N, out_val,
                                            out_idx, st)
                          : run_k23<KNN_IP>(G, M, L, Kp, K, D, qf32, q_stride, xf32, N, out_val,
                                            out_idx, st);
}

}  // namespace tpuknn
