// prep.cu -- row preparation for the contraction (database once, queries per
// call): optional cosine normalisation (Sec. 2), conversion to the stored
// element type (FP32 / BF16 / E4M3 with a per-row scale or with one scale for
// the whole database), half squared norms
// for L2 (App. A.2, Eq. 19), zero padding of each row to the row pitch.
//
// What defines the result is FP64 arithmetic: for COS the squared norm summed
// in index order, inv = 1 / sqrt, y = round32(x * inv); for L2 half the FP64
// sum of the stored values' squares, rounded to FP32. GB300's FP64 pipe takes
// about 26 cycles per warp instruction and SM, so that arithmetic bounded the
// kernel (38.6 ms for 2M x 96 cosine rows, against 0.26 ms of HBM traffic).
// The kernel therefore computes in pairs of FP32 numbers (error-free sums and
// products, Dekker / Knuth / Ogita-Rump-Oishi), whose error bound is known,
// and takes the FP64 result only for a row where that bound leaves the
// rounding of some element undecided (about one row in 1,000 at 96 elements):
// the bytes are the same as those of FP64 throughout. The kernel is then bound
// by HBM and instruction issue: 0.37 ms for those rows, 4.7 TB/s of its 1.74 GB
// (0.52 ms with every element scaled twice and divided by the E4M3 scale).
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "dtypes.cuh"
#include "kernels.h"

namespace tpuknn {

namespace {

// ---------------------------------------------------------------------------
// Pairs of FP32 numbers: value = h + l. Every operation is written with the
// _rn intrinsics, which the compiler does not contract.
// ---------------------------------------------------------------------------
struct Pair {
  float h, l;
};

// s + p = t + e exactly (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float s, float p, float& e) {
  const float t = __fadd_rn(s, p);
  const float z = __fsub_rn(t, s);
  e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
  return t;
}
// acc += v * v: the product and the sum are error-free, their two error terms
// go into the low part by plain adds. After n terms the low part's terms are
// at most (n + 1) 2^-24 of the sum and its 2n adds round by 2^-24 of that:
// |error| <= 2 n (n + 1) 2^-48 of the sum, 2^-36.9 for n = 32 (a lane's
// elements; the cross-lane sums below add 5 more terms of the same size).
__device__ __forceinline__ void add_square(Pair& a, float v) {
  const float p = __fmul_rn(v, v);
  const float e = __fmaf_rn(v, v, -p);
  float q;
  a.h = two_sum(a.h, p, q);
  a.l = __fadd_rn(a.l, __fadd_rn(q, e));
}
// The same with the low part's own rounding errors kept (a third component):
// what is left is the rounding of the two error terms' sum, 2^-47 of the
// running sum a term, 2 n 2^-48 in all: 2^-42 for n = 32.
struct Triple {
  float h, l, m;
};
__device__ __forceinline__ void add_square(Triple& a, float v) {
  const float p = __fmul_rn(v, v);
  const float e = __fmaf_rn(v, v, -p);
  float q, r;
  a.h = two_sum(a.h, p, q);
  a.l = two_sum(a.l, __fadd_rn(q, e), r);
  a.m = __fadd_rn(a.m, r);
}

// Magnitudes for which the pairs behave (anything else, zero rows too, takes
// the FP64 way). square_range, for the half norm: squares and their error terms
// neither overflow nor lose bits that matter against the sum of the row's
// squares: an element's square and its error term lose up to 2^-149, 2^-137 for
// the longest row, 2^-37 of the largest element's square. unit_range, for the
// inverse norm: its square, at least 2^(-2 kUnitHi) / kMaxD, is also
// held exactly as two FP32 numbers: its last bit, 2^-48 of it, is no smaller
// than FP32's smallest number, 2^-149. (With elements up to 2^50 that bit was
// lost, and 1 / |x| was off by up to 2^-41 at D = 1024.)
constexpr int kUnitHi = 40;
static_assert(2 * kUnitHi + 48 <= 149 - 12 && kMaxD <= 1 << 12, "1 / |x|^2 loses bits");
__device__ __forceinline__ bool square_range(float mx) { return mx >= 0x1p-50f && mx <= 0x1p50f; }
__device__ __forceinline__ bool unit_range(float mx) {
  return mx >= 0x1p-40f && mx <= (float)(1ll << kUnitHi);
}

// Sum over the G lanes of a row's group (G a power of two, groups aligned).
template <int G>
__device__ __forceinline__ Pair group_sum(Pair a) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, a.h, o);
    const float ol = __shfl_xor_sync(0xffffffffu, a.l, o);
    float q;
    a.h = two_sum(a.h, oh, q);
    a.l = __fadd_rn(__fadd_rn(a.l, ol), q);
  }
  return a;
}
template <int G>
__device__ __forceinline__ Triple group_sum(Triple a) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, a.h, o);
    const float ol = __shfl_xor_sync(0xffffffffu, a.l, o);
    const float om = __shfl_xor_sync(0xffffffffu, a.m, o);
    float q, r, u;
    a.h = two_sum(a.h, oh, q);
    a.l = two_sum(a.l, ol, u);
    a.l = two_sum(a.l, q, r);
    a.m = __fadd_rn(__fadd_rn(a.m, om), __fadd_rn(r, u));
  }
  return a;
}
template <int G>
__device__ __forceinline__ float group_max(float m) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  return m;
}
template <int G>
__device__ __forceinline__ double group_sum(double a) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}
// Whether any lane of this lane's group says so.
template <int G>
__device__ __forceinline__ bool group_any(bool p) {
  const unsigned m = __ballot_sync(0xffffffffu, p);
  const int lane = threadIdx.x & 31;
  const unsigned own = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (lane & ~(G - 1));
  return (m & own) != 0u;
}

// 1 / sqrt(n.h + n.l) as a pair: one Newton step from the hardware's
// reciprocal square root y (relative error below 2^-22), the residual
// 1 - n y^2 evaluated with error-free products (unit_range keeps y^2's two
// parts out of the subnormals). Terms of the residual are below 2^-21 and
// round by 2^-24 of that; the cubic term left out is below 2^-66: relative
// error below 2^-43.
__device__ __forceinline__ Pair inv_sqrt(float nh, float nl) {
  const float y = rsqrtf(nh);
  const float a = __fmul_rn(y, y), b = __fmaf_rn(y, y, -a);  // y^2 = a + b
  const float p = __fmul_rn(nh, a), e = __fmaf_rn(nh, a, -p);
  // 1 - p is exact (p within 2^-20 of 1)
  const float h = __fsub_rn(__fsub_rn(1.0f, p), __fmaf_rn(nh, b, __fmaf_rn(nl, a, e)));
  return Pair{y, __fmul_rn(y, __fmul_rn(h, __fmaf_rn(0.375f, h, 0.5f)))};
}

// round32(v * (inv.h + inv.l)) and whether it is decided. With at most 32
// elements per lane the product p + r is within 2^-41.5 of v / |x| (half the
// squared norm's error: 2^-43 from its terms, 2^-43.7 from its rounding to a
// pair; 2^-43 from the inverse root, 2^-46 from r) and the FP64 product within
// (D + 1) 2^-54, 2^-44 at D = 1024: where p + r and 2^-41 |p| to either side
// of it round to one number, both round to it. Longer rows (up to 128
// elements per lane, D = 4096: 2^-39.9 and 2^-42) take 2^-39. Products so
// small that r loses bits are left undecided.
template <int VPL>
__device__ __forceinline__ float scaled(float v, Pair inv, bool& undecided) {
  const float p = __fmul_rn(v, inv.h);
  const float r = __fmaf_rn(v, inv.l, __fmaf_rn(v, inv.h, -p));
  const float m = __fmul_rn(fabsf(p), VPL > 0 ? 0x1p-41f : 0x1p-39f);
  const float up = __fadd_rn(p, __fadd_rn(r, m)), dn = __fadd_rn(p, __fsub_rn(r, m));
  // (written so that a NaN is undecided)
  undecided = undecided || !(up == dn) || (v != 0.0f && !(fabsf(p) >= 0x1p-70f));
  return copysignf(up, v);  // -0 stays -0
}

// The defining arithmetic: FP64 squared norm in index order, summed by one
// lane; -1 marks a zero row (all its elements become 0).
__device__ __forceinline__ double inv_norm64(const float* xr, int D) {
  double n2 = 0.0;
  for (int d = 0; d < D; ++d) {
    const double t = (double)xr[d];
    n2 = __dadd_rn(n2, __dmul_rn(t, t));
  }
  return n2 == 0.0 ? -1.0 : __ddiv_rn(1.0, __dsqrt_rn(n2));
}
__device__ __forceinline__ float scaled64(float v, double inv) {
  return inv < 0.0 ? 0.0f : __double2float_rn(__dmul_rn((double)v, inv));
}

__device__ __forceinline__ float e4m3_scale_of(float mx) {
  return mx > 0.0f ? __fdiv_rn(mx, 448.0f) : 1.0f;
}

// E4M3 codes of y[0..3] / s, the quotient rounded to FP32 first. The code is
// decided without the division where y times 1/s, raised and lowered by 2^-21
// (8 units against the 4 that the reciprocal, its factor, the product and the
// quotient's own rounding can move it), converts to the same code: all but
// one element in 2^16.
struct E4m3Scale {
  float s, up, dn;
  bool usable;
};
__device__ __forceinline__ E4m3Scale e4m3_scale(float s) {
  const float r = __frcp_rn(s);
  return E4m3Scale{s, __fmul_rn(r, 1.0f + 0x1p-21f), __fmul_rn(r, 1.0f - 0x1p-21f),
                   s >= 0x1p-100f && s <= 0x1p100f};
}
__device__ __forceinline__ uint32_t e4m3x4(float a, float b, float c, float d) {
  const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3);
  const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(c, d), __NV_SATFINITE, __NV_E4M3);
  return lo | (hi << 16);
}
__device__ __forceinline__ uint32_t e4m3_codes(const float (&y)[4], const E4m3Scale& k) {
  const uint32_t u = e4m3x4(__fmul_rn(y[0], k.up), __fmul_rn(y[1], k.up), __fmul_rn(y[2], k.up),
                            __fmul_rn(y[3], k.up));
  const uint32_t l = e4m3x4(__fmul_rn(y[0], k.dn), __fmul_rn(y[1], k.dn), __fmul_rn(y[2], k.dn),
                            __fmul_rn(y[3], k.dn));
  if (u == l && k.usable) return u;
  return e4m3x4(__fdiv_rn(y[0], k.s), __fdiv_rn(y[1], k.s), __fdiv_rn(y[2], k.s),
                __fdiv_rn(y[3], k.s));
}

// A row's elements as a group of G lanes holds them: lane l of the group owns
// elements 4 (l + G t) .. + 3, t < VPL. VPL = 0: rows too long for
// registers; the elements are read again in every pass (t < nv).
template <int G, int VPL>
struct RowRegs {
  float v[VPL > 0 ? VPL : 1][4];
};

__device__ __forceinline__ void load4(const float* xr, int d, int D, bool vec, float (&o)[4]) {
  if (vec) {  // D a multiple of 4, rows 16-byte aligned
    const float4 f = d < D ? __ldg(reinterpret_cast<const float4*>(xr + d))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    o[0] = f.x;
    o[1] = f.y;
    o[2] = f.z;
    o[3] = f.w;
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) o[u] = d + u < D ? __ldg(xr + d + u) : 0.0f;
  }
}

// The rows' y (the row itself, or for COS the row scaled to unit length) is
// what f(d, y) sees: four consecutive elements from d at a time. For COS the
// row must be decided by `norm_of` first.
struct RowNorm {
  Pair inv;      // FP32 pair (fast way)
  double inv64;  // FP64 (exact way)
  bool fast;
};

// Finds the norm of a row held in x (VPL > 0) and turns x into the unit row;
// VPL = 0: only the norm, and the caller scales what it reads again.
template <int G, int VPL>
__device__ __forceinline__ RowNorm norm_of(const float* xr, int D, bool vec, RowRegs<G, VPL>& x,
                                           bool live) {
  const int lane = threadIdx.x & 31, gl = lane & (G - 1);
  const int nv = VPL > 0 ? VPL : (D + 4 * G - 1) / (4 * G);
  RowNorm n;
  Triple s{0.f, 0.f, 0.f};
  float mx = 0.0f;
  auto elements = [&](int t, float (&v)[4]) {
    if constexpr (VPL > 0) {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = x.v[t][u];
    } else {
      load4(xr, 4 * (gl + G * t), live ? D : 0, vec, v);
    }
  };
#pragma unroll
  for (int t = 0; t < nv; ++t) {
    float v[4];
    elements(t, v);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      add_square(s, v[u]);
      mx = fmaxf(mx, fabsf(v[u]));
    }
  }
  s = group_sum<G>(s);
  mx = group_max<G>(mx);
  // renormalise to a pair: |l| within 2^-24 of h
  float e;
  const float h = two_sum(s.h, __fadd_rn(s.l, s.m), e);
  n.inv = inv_sqrt(h, e);
  n.inv64 = 0.0;
  bool undecided = !unit_range(mx) || !(h <= 3.0e38f);
#pragma unroll
  for (int t = 0; t < nv; ++t) {
    float v[4];
    elements(t, v);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float y = scaled<VPL>(v[u], n.inv, undecided);
      if constexpr (VPL > 0) x.v[t][u] = y;
    }
  }
  n.fast = !group_any<G>(undecided && live);
  if (!n.fast && live) {
    double inv = 0.0;
    if (gl == 0) inv = inv_norm64(xr, D);
    const unsigned own = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (lane & ~(G - 1));
    n.inv64 = __shfl_sync(own, inv, lane & ~(G - 1));
    if constexpr (VPL > 0) {
#pragma unroll 1
      for (int t = 0; t < VPL; ++t) {
        float v[4];
        load4(xr, 4 * (gl + G * t), D, vec, v);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          v[u] = 4 * (gl + G * t) + u < D ? scaled64(v[u], n.inv64) : 0.0f;
#pragma unroll
        for (int k = 0; k < VPL; ++k)  // x.v[t] without a dynamic register index
          if (k == t) {
#pragma unroll
            for (int u = 0; u < 4; ++u) x.v[k][u] = v[u];
          }
      }
    }
  }
  return n;
}

// Element d of a long row's unit row (0 past the row's end, whatever the norm).
__device__ __forceinline__ float unit_value(float v, int d, int D, const RowNorm& n) {
  bool dummy = false;
  const float y = n.fast ? scaled<0>(v, n.inv, dummy) : scaled64(v, n.inv64);
  return d < D ? y : 0.0f;
}

// The largest |y| over all rows, merged into *mx_bits as the bits of a
// non-negative float (their integer order is the float order).
template <int G, int VPL>
__global__ void __launch_bounds__(256)
rows_absmax_kernel(const float* __restrict__ x, int64_t rows, int D, int metric, int vec,
                   unsigned* __restrict__ mx_bits) {
  pdl_wait();
  const int gl = threadIdx.x & (G - 1);
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const bool live = r < rows;
  const float* xr = x + (live ? r : 0) * (int64_t)D;
  const int nv = VPL > 0 ? VPL : (D + 4 * G - 1) / (4 * G);
  RowRegs<G, VPL> xs;
  if constexpr (VPL > 0) {
#pragma unroll
    for (int t = 0; t < VPL; ++t) load4(xr, 4 * (gl + G * t), live ? D : 0, vec != 0, xs.v[t]);
  }
  RowNorm n{};
  if (metric == KNN_COS) n = norm_of<G, VPL>(xr, D, vec != 0, xs, live);
  float mx = 0.0f;
#pragma unroll
  for (int t = 0; t < nv; ++t) {
    float v[4];
    if constexpr (VPL > 0) {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = xs.v[t][u];
    } else {
      load4(xr, 4 * (gl + G * t), live ? D : 0, vec != 0, v);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      mx = fmaxf(mx, fabsf(VPL == 0 && metric == KNN_COS
                               ? unit_value(v[u], 4 * (gl + G * t) + u, D, n)
                               : v[u]));
  }
  mx = group_max<32>(mx);
  __shared__ float s_mx[8];
  if ((threadIdx.x & 31) == 0) s_mx[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) mx = fmaxf(mx, s_mx[w]);
    if (mx > 0.0f) atomicMax(mx_bits, __float_as_uint(mx));
  }
}

__global__ void set_word_kernel(unsigned* p, unsigned v) { *p = v; }
// the database-wide scale into the first row's slot, from the maximum held there
__global__ void tensor_scale_kernel(float* scale) {
  scale[0] = e4m3_scale_of(__uint_as_float(*reinterpret_cast<const unsigned*>(scale)));
}

// A group of G lanes per row, its elements in registers. The E4M3 scale uses
// a maximum (order-free): the row's own (KNN_E4M3) or, when gmax_bits is
// given, the database-wide one (KNN_E4M3_T; then row 0's scale slot holds
// that maximum during this kernel and is written afterwards). If zero_buf is
// given, the CTAs also clear zero_n 32-bit words of it.
//
// Eight lanes per row up to 256 elements: a warp has four rows in flight with
// VPL 16-byte loads per lane each (a warp per row left 384 bytes per warp in
// flight at 96 elements), and a row's 8 x 16-byte pieces fill whole sectors.
template <int DT, bool COS, int G, int VPL>
__global__ void __launch_bounds__(256)
prep_rows_kernel(const float* __restrict__ x, int64_t rows, int D, int pitch, int vec,
                 void* __restrict__ out_lp, float* __restrict__ out_scale,
                 float* __restrict__ out_hnorm, float* __restrict__ out_f32,
                 uint32_t* __restrict__ zero_buf, int64_t zero_n,
                 const unsigned* __restrict__ gmax_bits) {
  // Launched behind whatever the stream ran before: wait for it (its output
  // may be these rows, or it may still read the buffers written here), then
  // let the contraction launch and run its prologue.
  pdl_wait();
  pdl_trigger();
  if (zero_buf) {
    // 16-byte stores where the buffer allows, then the odd words
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t done = 0;
    if ((reinterpret_cast<uintptr_t>(zero_buf) & 15) == 0) {
      const int64_t n4 = zero_n / 4;
      for (int64_t t = t0; t < n4; t += stride)
        reinterpret_cast<uint4*>(zero_buf)[t] = make_uint4(0u, 0u, 0u, 0u);
      done = n4 * 4;
    }
    for (int64_t t = done + t0; t < zero_n; t += stride) zero_buf[t] = 0u;
  }
  const int gl = threadIdx.x & (G - 1);
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const bool live = r < rows;  // the same in every lane of a group
  if (__ballot_sync(0xffffffffu, live) == 0u) return;
  const float* xr = x + (live ? r : 0) * (int64_t)D;
  const int nv = VPL > 0 ? VPL : (pitch + 4 * G - 1) / (4 * G);
  RowRegs<G, VPL> xs;
  if constexpr (VPL > 0) {
#pragma unroll
    for (int t = 0; t < VPL; ++t) load4(xr, 4 * (gl + G * t), live ? D : 0, vec & 1, xs.v[t]);
  }
  RowNorm n{};
  if constexpr (COS) n = norm_of<G, VPL>(xr, D, vec & 1, xs, live);
  // four values y of this lane from d = 4 (gl + G t)
  auto yvals = [&](int t, float (&y)[4]) {
    if constexpr (VPL > 0) {
#pragma unroll
      for (int u = 0; u < 4; ++u) y[u] = xs.v[t][u];
    } else {
      load4(xr, 4 * (gl + G * t), live ? D : 0, vec & 1, y);
      if (COS) {
#pragma unroll
        for (int u = 0; u < 4; ++u) y[u] = unit_value(y[u], 4 * (gl + G * t) + u, D, n);
      }
    }
  };
  float s = 1.0f;
  if (DT == KNN_E4M3) {
    if (gmax_bits) {
      s = e4m3_scale_of(__uint_as_float(*gmax_bits));
      if (out_scale && gl == 0 && r > 0 && live) out_scale[r] = s;
    } else {
      float mx = 0.0f;
#pragma unroll
      for (int t = 0; t < nv; ++t) {
        float y[4];
        yvals(t, y);
#pragma unroll
        for (int u = 0; u < 4; ++u) mx = fmaxf(mx, fabsf(y[u]));
      }
      mx = group_max<G>(mx);
      s = e4m3_scale_of(mx);
      if (out_scale && gl == 0 && live) out_scale[r] = s;
    }
  }
  Pair h2{0.0f, 0.0f};
  float smx = 0.0f;
  const E4m3Scale es = e4m3_scale(s);
  // the four stored values of y (what the contraction sees), and the bytes
  auto stored4 = [&](const float (&y)[4], float (&st)[4], uint32_t& code) {
    code = DT == KNN_E4M3 ? e4m3_codes(y, es) : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (DT == KNN_F32)
        st[u] = y[u];
      else if (DT == KNN_BF16)
        st[u] = __bfloat162float(__float2bfloat16_rn(y[u]));
      else
        st[u] = e4m3_code_to_float((uint8_t)(code >> (8 * u))) * s;
    }
  };
  if (live) {
#pragma unroll
    for (int t = 0; t < nv; ++t) {
      const int d = 4 * (gl + G * t);
      if (d >= pitch) break;
      float y[4], st[4];
      uint32_t code;
      yvals(t, y);
      stored4(y, st, code);
      if (DT == KNN_F32) {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(out_lp) + r * pitch + d) =
            make_float4(y[0], y[1], y[2], y[3]);
      } else if (DT == KNN_BF16) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(y[0], y[1]),
                             hi = __floats2bfloat162_rn(y[2], y[3]);
        uint2 w;
        w.x = *reinterpret_cast<const uint32_t*>(&lo);
        w.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(out_lp) + r * pitch + d) = w;
      } else {
        *reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(out_lp) + r * pitch + d) = code;
      }
      if (!COS && out_hnorm) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          add_square(h2, st[u]);
          smx = fmaxf(smx, fabsf(st[u]));
        }
      }
      if (COS && out_f32) {
        float* o = out_f32 + r * (int64_t)D + d;
        if (vec & 2) {
          if (d < D) *reinterpret_cast<float4*>(o) = make_float4(y[0], y[1], y[2], y[3]);
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (d + u < D) o[u] = y[u];
        }
      }
    }
  }
  if (!COS && out_hnorm) {
    // half the sum, rounded once; the FP64 sum where the pair's error bound
    // (2^-36 of the sum with 32 elements per lane, 2^-32 with 128) leaves the
    // rounding open. A row of zeros is 0 (50,000 x 257 rows of zeros or of
    // elements at 2^-45 took 122 us in both, 79 in FP64 alone)
    h2 = group_sum<G>(h2);
    smx = group_max<G>(smx);
    const float m = __fmul_rn(h2.h, VPL > 0 ? 0x1p-35f : 0x1p-31f);
    const float up = __fadd_rn(h2.h, __fadd_rn(h2.l, m)), dn = __fadd_rn(h2.h, __fsub_rn(h2.l, m));
    const bool zero = smx == 0.0f && h2.h == 0.0f;  // (a NaN is in h2.h only)
    const bool open = !zero && !(up == dn && square_range(smx));
    float hn = zero ? 0.0f : 0.5f * up;
    if (group_any<32>(open && live)) {
      double a = 0.0;
      if (live) {
#pragma unroll
        for (int t = 0; t < nv; ++t) {
          const int d = 4 * (gl + G * t);
          if (d >= pitch) break;
          float y[4], st[4];
          uint32_t code;
          yvals(t, y);
          stored4(y, st, code);
#pragma unroll
          for (int u = 0; u < 4; ++u) a += (double)st[u] * (double)st[u];
        }
      }
      a = group_sum<G>(a);
      if (open) hn = (float)(0.5 * a);
    }
    if (gl == 0 && live) out_hnorm[r] = hn;
  }
}

// Lanes per row and 16-byte pieces per lane for a row pitch.
template <class F>
cudaError_t by_length(int pitch, F f) {
  if (pitch <= 64) return f(std::integral_constant<int, 8>(), std::integral_constant<int, 2>());
  if (pitch <= 96) return f(std::integral_constant<int, 8>(), std::integral_constant<int, 3>());
  if (pitch <= 128) return f(std::integral_constant<int, 8>(), std::integral_constant<int, 4>());
  if (pitch <= 256) return f(std::integral_constant<int, 8>(), std::integral_constant<int, 8>());
  if (pitch <= 512) return f(std::integral_constant<int, 32>(), std::integral_constant<int, 4>());
  if (pitch <= 1024) return f(std::integral_constant<int, 32>(), std::integral_constant<int, 8>());
  return f(std::integral_constant<int, 32>(), std::integral_constant<int, 0>());
}

template <int DT>
cudaError_t launch_rows(const float* x, int64_t rows, int D, int pitch, int metric, void* out_lp,
                        float* out_scale, float* h, float* f, cudaStream_t st, uint32_t* zero_buf,
                        int64_t zero_n, const unsigned* gmax_bits) {
  const int threads = 256;
  // bit 0: 16-byte loads of x; bit 1: 16-byte stores of the unit rows
  const int vec = (D % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0 ? 1 : 0) |
                  (D % 4 == 0 && (reinterpret_cast<uintptr_t>(f) & 15) == 0 ? 2 : 0);
  return by_length(pitch, [&](auto g, auto v) {
    int64_t blocks = cdiv(rows * decltype(g)::value, threads);
    // a block clears 16 KB or more, up to four blocks per SM (131 MB of keys
    // by 64 blocks: 46 us)
    if (zero_buf)
      blocks = std::max(blocks, std::max<int64_t>(64, std::min<int64_t>(4 * device_sm_count(),
                                                                      cdiv(zero_n, 4096))));
    if (blocks < 1) blocks = 1;
    auto kern = metric == KNN_COS
                    ? prep_rows_kernel<DT, true, decltype(g)::value, decltype(v)::value>
                    : prep_rows_kernel<DT, false, decltype(g)::value, decltype(v)::value>;
    return launch_pdl(kern, dim3((unsigned)blocks), dim3(threads), 0, st, x, rows, D, pitch, vec,
                      out_lp, out_scale, h, f, zero_buf, zero_n, gmax_bits);
  });
}

}  // namespace

cudaError_t launch_prep(const float* x, int64_t rows, int D, int pitch, int metric, int dtype,
                        void* out_lp, float* out_scale, float* out_hnorm, float* out_f32,
                        cudaStream_t st, uint32_t* zero_buf, int64_t zero_n) {
  if (rows <= 0 && zero_n <= 0) return cudaSuccess;
  float* h = metric == KNN_L2 ? out_hnorm : nullptr;
  float* f = metric == KNN_COS ? out_f32 : nullptr;
  switch (dtype) {
    case KNN_F32:
      return launch_rows<KNN_F32>(x, rows, D, pitch, metric, out_lp, nullptr, h, f, st, zero_buf,
                                  zero_n, nullptr);
    case KNN_BF16:
      return launch_rows<KNN_BF16>(x, rows, D, pitch, metric, out_lp, nullptr, h, f, st, zero_buf,
                                   zero_n, nullptr);
    case KNN_E4M3_T: {
      // the database-wide maximum, accumulated in row 0's scale slot
      if (rows <= 0 || !out_scale) return cudaErrorInvalidValue;
      unsigned* mx = reinterpret_cast<unsigned*>(out_scale);
      set_word_kernel<<<1, 1, 0, st>>>(mx, 0u);
      const int vec = D % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0 ? 1 : 0;
      cudaError_t e = by_length(pitch, [&](auto g, auto v) {
        return launch_pdl(rows_absmax_kernel<decltype(g)::value, decltype(v)::value>,
                          dim3((unsigned)cdiv(rows * decltype(g)::value, 256)), dim3(256), 0, st, x,
                          rows, D, metric, vec, mx);
      });
      if (e != cudaSuccess) return e;
      e = launch_rows<KNN_E4M3>(x, rows, D, pitch, metric, out_lp, out_scale, h, f, st, zero_buf,
                                zero_n, mx);
      if (e != cudaSuccess) return e;
      tensor_scale_kernel<<<1, 1, 0, st>>>(out_scale);
      return cudaGetLastError();
    }
    default:
      return launch_rows<KNN_E4M3>(x, rows, D, pitch, metric, out_lp, out_scale, h, f, st,
                                   zero_buf, zero_n, nullptr);
  }
}

}  // namespace tpuknn
