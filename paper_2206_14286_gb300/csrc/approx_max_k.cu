// approx_max_k.cu -- the approx_max_k / approx_min_k operator on a score
// matrix the caller already holds (App. A.1: the operator behind Alg. 1,
// without the fused contraction). For every row i of S (M x N, FP32 or BF16,
// row-major) and bin l it keeps the best score and its column, bins j mod L
// or L balanced runs of consecutive columns; optionally ExactRescoring then
// keeps the best K of the L winners (aggregate_to_topk).
//
// The operator reads every score once and is HBM-bound. Bin winners merge in
// an M x L array of ordered 64-bit keys (score, ~column) by atomicMax, so ties
// keep the smaller column whatever the order of the CTAs; approx_min_k
// negates the scores on the way in and the values on the way out.
#include <algorithm>
#include <cmath>
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"

namespace tpuknn {

namespace {

// The score, negated for approx_min_k; adding +0 turns -0 into +0, so that
// the two zeros make equal keys and tie to the smaller column.
template <int DT>
__device__ __forceinline__ float load_score(const void* S, int64_t t, float sg) {
  const float v = DT == KNN_BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(S)[t])
                                 : reinterpret_cast<const float*>(S)[t];
  return sg * v + 0.0f;
}

// The larger of two scores of load_score's form, a NaN above every other, and
// whether it is not `a` (by its bits: a score of that form has one NaN, the
// arithmetic's canonical positive one, and one zero).
__device__ __forceinline__ float max_nan(float a, float b, bool& changed) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  changed = __float_as_uint(m) != __float_as_uint(a);
  return m;
}
// make_key of a score, a NaN's too. (On the bits of a float the compiler turns
// make_key's "| 0x80000000" into a negation, which loses a NaN's bits: a NaN
// came out as -0. The empty asm makes them an integer's.)
__device__ __forceinline__ uint64_t score_key(float v, int32_t j) {
  uint32_t u = __float_as_uint(v);
  asm("" : "+r"(u));
  return ((uint64_t)((u & 0x80000000u) ? ~u : (u | 0x80000000u)) << 32) | (uint32_t)~j;
}

// Bins j mod L: a thread owns V bins b0 .. b0 + V - 1 of a row and walks their
// columns, every bdy-th grid row of the CTA's chunk of grid rows, keeping each
// bin's best value and grid row in registers (a later column leads only by a
// larger score, which keeps the smaller column on ties). V = 8 BF16 or 4 FP32
// columns of one 16-byte load (L and N multiples of V, S 16-byte aligned), else
// V = 1.
//
// Bound by HBM. threadIdx.x runs over the vectors of a grid row, however many
// there are (tpr of them, up to 256), and threadIdx.y over grid rows, so the
// CTA's threads read bdy whole grid rows, which are adjacent in memory, and no
// lane idles for padding: rounded up to warps, 22 vectors of L = 176 left 10 of
// 32 lanes without work (1024 x 1M BF16: 510 us). The bdy rows' bests merge in
// shared memory before one atomicMax per bin. kRows: threadIdx.z runs over rows
// of S, where a row's columns are too few for more threads (an instance of its
// own: with the row a thread's, not a CTA's, 250 x 100,003 FP32 was 3% slower).
// CTAs to an SM (by registers; with four of V = 8, 1024 x 1M BF16 took 374 us,
// with five 316).
constexpr int mod_ctas(int V) { return V == 8 ? 5 : V == 4 ? 6 : 8; }
template <int DT, int V, bool kRows>
__global__ void __launch_bounds__(256, mod_ctas(V))
bin_max_mod_kernel(const void* __restrict__ S, int M, int64_t N, int L, int kchunk, int neg,
                   unsigned long long* __restrict__ G) {
  constexpr int kEsz = DT == KNN_BF16 ? 2 : 4, U = V == 1 ? 8 : 4;
  __shared__ uint64_t part[V == 1 ? 1 : V][256];
  const int bdy = blockDim.y;
  const int zt = kRows ? threadIdx.z * bdy * blockDim.x : 0;  // first thread of this row
  const int64_t i = kRows ? (int64_t)blockIdx.y * blockDim.z + threadIdx.z : blockIdx.y;
  const int b0 = ((int)blockIdx.x * blockDim.x + threadIdx.x) * V;
  const bool live = b0 < L && (!kRows || i < M);
  const uint32_t T = (uint32_t)((N + L - 1) / L);  // grid rows, the last one maybe ragged
  const uint32_t k0 = blockIdx.z * (uint32_t)kchunk, k1 = min(T, k0 + kchunk);
  const float sg = neg ? -1.0f : 1.0f;
  // every grid row but the last is whole
  const uint32_t kfull = live && (int64_t)(k1 - 1) * L + b0 + V <= N ? k1 : k1 - 1;
  // the first column leads with -inf until a score is larger
  const bool any = live && k0 + threadIdx.y < kfull;
  float bv[V];
  uint32_t bk[V];
#pragma unroll
  for (int c = 0; c < V; ++c) {
    bv[c] = neg_inf();
    bk[c] = k0 + threadIdx.y;
  }
  if (any) {
    const char* row = static_cast<const char*>(S) + (i * N + b0) * kEsz;
    auto take = [&](const uint4& raw, float one, uint32_t k) {
      float x[V];
      if constexpr (V == 1) {
        x[0] = one;
      } else if constexpr (DT == KNN_BF16) {
        const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&raw);
#pragma unroll
        for (int c = 0; c < V; ++c) x[c] = __bfloat162float(h[c]);
      } else {
        const float* f = reinterpret_cast<const float*>(&raw);
#pragma unroll
        for (int c = 0; c < V; ++c) x[c] = f[c];
      }
#pragma unroll
      for (int c = 0; c < V; ++c) {
        // adding +0 turns -0 into +0: the two zeros tie
        const float v = sg * x[c] + 0.0f;
        bool lead;
        bv[c] = max_nan(bv[c], v, lead);
        if (lead) bk[c] = k;
      }
    };
    auto load = [&](uint32_t k, uint4& raw, float& one) {
      const char* p = row + (int64_t)k * L * kEsz;
      if constexpr (V == 1)
        one = load_score<DT>(p, 0, 1.0f);
      else
        raw = __ldg(reinterpret_cast<const uint4*>(p));
    };
    uint32_t k = k0 + threadIdx.y;
    for (; k + (U - 1) * bdy < kfull; k += U * bdy) {
      uint4 raw[U];
      float one[U];
#pragma unroll
      for (int u = 0; u < U; ++u) load(k + u * bdy, raw[u], one[u]);
#pragma unroll
      for (int u = 0; u < U; ++u) take(raw[u], one[u], k + u * bdy);
    }
    for (; k < kfull; k += bdy) {
      uint4 raw;
      float one;
      load(k, raw, one);
      take(raw, one, k);
    }
  }
  auto key = [&](int c) -> uint64_t {
    return any ? score_key(bv[c], (int32_t)(bk[c] * (uint32_t)L + b0 + c)) : (uint64_t)0;
  };
  if (bdy == 1) {
#pragma unroll
    for (int c = 0; c < V; ++c) {
      const uint64_t best = key(c);
      if (best) atomicMax(&G[i * L + b0 + c], (unsigned long long)best);
    }
    return;
  }
  const int t0 = threadIdx.y * blockDim.x + threadIdx.x;
#pragma unroll
  for (int c = 0; c < V; ++c) part[V == 1 ? 0 : c][zt + t0] = key(c);
  __syncthreads();
  for (int t = t0; t < (int)blockDim.x * V; t += blockDim.x * bdy) {
    const int c = t / blockDim.x, x = t % blockDim.x;
    const int b = ((int)blockIdx.x * blockDim.x + x) * V + c;
    uint64_t best = 0;
    for (int y = 0; y < bdy; ++y) {
      const uint64_t o = part[c][zt + y * blockDim.x + x];
      best = o > best ? o : best;
    }
    if (best && b < L) atomicMax(&G[i * L + b], (unsigned long long)best);
  }
}

__device__ __forceinline__ int64_t runs_bin_of(int64_t j, int64_t q, int64_t r) {
  const int64_t big = r * (q + 1);
  return j < big ? j / (q + 1) : r + (j - big) / q;
}

// Contiguous bins: a CTA sweeps `chunk` consecutive columns of one row; a
// thread keeps the best of its current bin and merges it when its columns
// (blockDim apart) move to another bin.
template <int DT>
__global__ void __launch_bounds__(256)
bin_max_runs_kernel(const void* __restrict__ S, int64_t N, int64_t L, int64_t chunk, int neg,
                    unsigned long long* __restrict__ G) {
  const int64_t i = blockIdx.y;
  const int64_t j0 = (int64_t)blockIdx.x * chunk;
  const int64_t j1 = min(N, j0 + chunk);
  const int64_t q = N / L, r = N % L;
  const float sg = neg ? -1.0f : 1.0f;
  int64_t cur = -1, end = 0;
  uint64_t best = 0;
  const int64_t step = blockDim.x;
  for (int64_t j8 = j0 + threadIdx.x; j8 < j1; j8 += 8 * step) {
    // eight independent loads in flight per thread
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t j = j8 + u * step;
      v[u] = j < j1 ? load_score<DT>(S, i * N + j, sg) : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t j = j8 + u * step;
      if (j < j1) {
        if (j >= end) {
          if (best) atomicMax(&G[i * L + cur], (unsigned long long)best);
          cur = runs_bin_of(j, q, r);
          end = (cur + 1) * q + min(cur + 1, r);
          best = 0;
        }
        const uint64_t key = score_key(v[u], (int32_t)j);
        best = key > best ? key : best;
      }
    }
  }
  if (best) atomicMax(&G[i * L + cur], (unsigned long long)best);
}

// The same with 16-byte loads (N a multiple of the V columns a load holds, S
// 16-byte aligned): a thread reads V consecutive columns at a time, blockDim
// * V columns apart, and keeps the best value and column of its current bin.
template <int DT>
__global__ void __launch_bounds__(256)
bin_max_runs_vec_kernel(const void* __restrict__ S, int64_t N, int64_t L, int64_t chunk, int neg,
                        unsigned long long* __restrict__ G) {
  constexpr int V = DT == KNN_BF16 ? 8 : 4;
  constexpr int kEsz = DT == KNN_BF16 ? 2 : 4;
  const int64_t i = blockIdx.y;
  const int64_t j0 = (int64_t)blockIdx.x * chunk;
  const int64_t j1 = min(N, j0 + chunk);
  const int64_t q = N / L, r = N % L;
  const float sg = neg ? -1.0f : 1.0f;
  const char* row = static_cast<const char*>(S) + i * N * kEsz;
  int64_t cur = -1, end = 0;
  float bv = neg_inf();
  int32_t bj = -1;
  auto flush = [&]() {
    if (bj >= 0) atomicMax(&G[i * L + cur], (unsigned long long)score_key(bv, bj));
  };
  const int64_t step = (int64_t)blockDim.x * V;
  for (int64_t jv = j0 + (int64_t)threadIdx.x * V; jv < j1; jv += 4 * step) {
    uint4 raw[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t j = jv + u * step;
      raw[u] = j < j1 ? __ldg(reinterpret_cast<const uint4*>(row + j * kEsz))
                      : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t j = jv + u * step;
      if (j < j1) {
        float x[V];
        if constexpr (DT == KNN_BF16) {
          const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&raw[u]);
#pragma unroll
          for (int c = 0; c < V; ++c) x[c] = __bfloat162float(h[c]);
        } else {
          const float* f = reinterpret_cast<const float*>(&raw[u]);
#pragma unroll
          for (int c = 0; c < V; ++c) x[c] = f[c];
        }
#pragma unroll
        for (int c = 0; c < V; ++c) {
          const int64_t jj = j + c;
          if (jj >= end) {
            flush();
            cur = runs_bin_of(jj, q, r);
            end = (cur + 1) * q + min(cur + 1, r);
            bv = neg_inf();
            bj = (int32_t)jj;
          }
          const float v = sg * x[c] + 0.0f;
          bool lead;
          bv = max_nan(bv, v, lead);
          if (lead) bj = (int32_t)jj;
        }
      }
    }
  }
  flush();
}

// How the columns of j mod L bins are shared out: a CTA takes the bdx vectors of
// bdy grid rows at a time of bdz rows of S, kchunk grid rows of them, kz chunks
// to a row.
struct ModShape {
  int bdx, bdy, bdz;
  int64_t kz, kchunk;
};
// A thread has 32 loads or more before its CTA's bests merge, so few grid rows
// are shared by few threads, and the CTA's other threads take other rows of S
// (5000 x 4096 FP32, L = 128, 32 grid rows: 42 us a call with 8 threads over them,
// 28 with 1; 20,000 x 1024, L = 8, 128 grid rows: 29.4 us with 8, 28.4 with 4).
// The chunks: the time is the waves of CTAs times a chunk's loads per thread plus
// about eight loads' time for its start and its merge. (With at least 32 loads
// a chunk and up to 48 CTAs per SM, waves were left part empty: 3 x 20M FP32, L =
// 8, 61 us with 610 chunks a row, 47 with 304; 500 x 65,536, L = 128: 44 and 34; and
// one row of 1M BF16, L = 2064, had 30 CTAs.) More than 304 chunks queue for their
// bins' keys: one row of 1M FP32, L = 128, 41 us with 869, 20 with 300 or fewer.
ModShape mod_shape(int64_t M, int64_t grid_rows, int64_t tpr, int V) {
  constexpr int64_t kLoads = 32, kEdge = 8, kMaxChunks = 304;
  ModShape s;
  s.bdx = (int)std::min<int64_t>(256, tpr);
  const int64_t room = 256 / s.bdx;
  s.bdy = (int)std::min(room, std::max<int64_t>(1, grid_rows / kLoads));
  s.bdz = (int)std::min(std::min(room / s.bdy, M), (int64_t)64);
  const int64_t warps = cdiv((int64_t)s.bdx * s.bdy * s.bdz, 32);
  const int64_t slots = device_sm_count() * std::min<int64_t>(32, mod_ctas(V) * 8 / warps);
  const int64_t ctas = cdiv(tpr, s.bdx) * cdiv(M, s.bdz);  // of one chunk
  // chunk counts that end a wave; beyond two waves the CTAs no longer run in step,
  // and about half a chunk is left over at the end (1024 x 1M BF16: 337 us with 2
  // chunks a row, in 2.7 waves, 316 with 8, in 10.8)
  double best = -1.0;
  s.kz = 1;
  s.kchunk = grid_rows;
  const int64_t w0 = std::max<int64_t>(1, cdiv(ctas, slots));
  for (int64_t w = w0; w < w0 + 12; ++w) {
    const int64_t kz = std::min(std::min(w * slots / ctas, grid_rows), kMaxChunks);
    const int64_t kchunk = cdiv(grid_rows, kz), n = cdiv(grid_rows, kchunk);
    const double waves = (double)(ctas * n) / (double)slots;
    const double cost = (waves <= 2.0 ? std::ceil(waves) : waves + 0.5) *
                        (double)(cdiv(kchunk, s.bdy) + kEdge);
    if (best < 0.0 || cost < best) {
      best = cost;
      s.kz = n;
      s.kchunk = kchunk;
    }
    if (kz == grid_rows || kz == kMaxChunks) break;
  }
  return s;
}

template <bool kRows>
auto mod_kernel(int dtype, bool vec) {
  return dtype == KNN_BF16 ? (vec ? bin_max_mod_kernel<KNN_BF16, 8, kRows>
                                  : bin_max_mod_kernel<KNN_BF16, 1, kRows>)
                           : (vec ? bin_max_mod_kernel<KNN_F32, 4, kRows>
                                  : bin_max_mod_kernel<KNN_F32, 1, kRows>);
}

// Keys to (value, index) pairs, values back in the caller's orientation.
__global__ void keys_to_pairs_kernel(const uint64_t* __restrict__ keys, int64_t n, int neg,
                                     float* __restrict__ out_v, int32_t* __restrict__ out_a) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const uint64_t k = keys[t];
  out_v[t] = k ? (neg ? -key_score(k) : key_score(k)) : __int_as_float(0x7fc00000);
  out_a[t] = k ? key_index(k) : -1;
}

}  // namespace

cudaError_t launch_bin_max(const void* S, int dtype, int64_t M, int64_t N, int64_t L, int bin_map,
                           int neg, unsigned long long* G, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (M > 65535) {
    // grid y holds at most 65535 rows: split the rows
    const int esz = dtype == KNN_BF16 ? 2 : 4;
    for (int64_t m0 = 0; m0 < M; m0 += 65535) {
      const int64_t mc = min((int64_t)65535, M - m0);
      cudaError_t e = launch_bin_max(static_cast<const char*>(S) + m0 * N * esz, dtype, mc, N, L,
                                     bin_map, neg, G + m0 * L, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  const int sms = device_sm_count();
  const int vcols = dtype == KNN_BF16 ? 8 : 4;
  if (bin_map == KNN_BINS_MOD) {
    const bool vec = L % vcols == 0 && N % vcols == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0;
    const int64_t tpr = vec ? L / vcols : L;  // threads that cover a grid row
    const int64_t grid_rows = cdiv(N, L);
    if (cdiv(tpr, 256) > 0x7fffffffLL) return cudaErrorInvalidValue;
    const ModShape c = mod_shape(M, grid_rows, tpr, vec ? vcols : 1);
    dim3 grid((unsigned)cdiv(tpr, c.bdx), (unsigned)cdiv(M, c.bdz), (unsigned)c.kz),
        block((unsigned)c.bdx, (unsigned)c.bdy, (unsigned)c.bdz);
    auto kern = c.bdz > 1 ? mod_kernel<true>(dtype, vec) : mod_kernel<false>(dtype, vec);
    kern<<<grid, block, 0, st>>>(S, (int)M, N, (int)L, (int)c.kchunk, neg, G);
  } else {
    const bool vec = N % vcols == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0;
    // columns per CTA: 32 vectors per thread, or 32 columns per thread
    const int64_t chunk = 256 * 32 * (vec ? vcols : 1);
    const int64_t bx = cdiv(N, chunk);
    if (bx > 0x7fffffffLL) return cudaErrorInvalidValue;
    dim3 grid((unsigned)bx, (unsigned)M);
    if (vec) {
      if (dtype == KNN_BF16)
        bin_max_runs_vec_kernel<KNN_BF16><<<grid, 256, 0, st>>>(S, N, L, chunk, neg, G);
      else
        bin_max_runs_vec_kernel<KNN_F32><<<grid, 256, 0, st>>>(S, N, L, chunk, neg, G);
    } else if (dtype == KNN_BF16) {
      bin_max_runs_kernel<KNN_BF16><<<grid, 256, 0, st>>>(S, N, L, chunk, neg, G);
    } else {
      bin_max_runs_kernel<KNN_F32><<<grid, 256, 0, st>>>(S, N, L, chunk, neg, G);
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_keys_to_pairs(const uint64_t* keys, int64_t n, int neg, float* out_v,
                                 int32_t* out_a, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  keys_to_pairs_kernel<<<(unsigned)cdiv(n, 256), 256, 0, st>>>(keys, n, neg, out_v, out_a);
  return cudaGetLastError();
}

}  // namespace tpuknn
