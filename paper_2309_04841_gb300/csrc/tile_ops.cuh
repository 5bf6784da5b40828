// tile_ops.cuh -- what the on-chip and the small-tile kernels share: arithmetic per
// precision, costs and phases, and slots of tile offsets in shared memory that are
// linear over XOR and free of bank conflicts in every round of a tile.
#pragma once

#include "qaoa_common.cuh"

namespace qaoa {
namespace tile {

__device__ __forceinline__ double ld_cost(const void *cost, int kind, uint32_t x) {
  if (kind == kCostI32) return (double)reinterpret_cast<const int *>(cost)[x];
  if (kind == kCostU16) return (double)reinterpret_cast<const unsigned short *>(cost)[x];
  if (kind == kCostF32) return (double)reinterpret_cast<const float *>(cost)[x];
  return reinterpret_cast<const double *>(cost)[x];
}

// ---- per precision: vector arithmetic, costs, phases, sums
template <typename Real> struct Ops;

template <> struct Ops<float> {
  using C2 = float2;
  using F = float2;  // a cost value as float pair hi + lo
  __device__ static __forceinline__ F integer(int f) {
    const float h = (float)f;
    return make_float2(h, (float)((long long)f - (long long)h));
  }
  __device__ static __forceinline__ C2 mk(float x, float y) { return make_float2(x, y); }
  __device__ static __forceinline__ C2 axpy(float t, C2 a, C2 b) { return __ffma2_rn(make_float2(t, t), a, b); }
  // exact for int32 and float32 costs, about 2^-48 relative for float64 ones
  __device__ static __forceinline__ F cost(const void *c, int kind, uint32_t x) {
    if (kind == kCostI32) return integer(reinterpret_cast<const int *>(c)[x]);
    if (kind == kCostU16) return make_float2((float)reinterpret_cast<const unsigned short *>(c)[x], 0.f);
    if (kind == kCostF32) return make_float2(reinterpret_cast<const float *>(c)[x], 0.f);
    const double f = reinterpret_cast<const double *>(c)[x];
    const float h = (float)f;
    return make_float2(h, (float)(f - (double)h));
  }
  __device__ static __forceinline__ float value(F f) { return f.x; }
  // scl exp(-i g f) with g / 2pi = g_hi + g_lo: Dekker's two-product by fma,
  // only the fraction reaches sincospi
  template <class L>
  __device__ static __forceinline__ C2 phase(const L &l, F f, float scl) {
    const float p = l.g_hi * f.x;
    const float e = fmaf(l.g_hi, f.x, -p);
    const float r = (p - rintf(p)) + (e + fmaf(l.g_hi, f.y, l.g_lo * f.x));
    float sn, cs;
    sincospif(2.0f * r, &sn, &cs);
    return make_float2(cs * scl, -sn * scl);
  }
  // The same for a table, (scl + scl_lo) exp(-i g f) rounded about once: every amplitude of
  // a digit shares an entry's error, so it is formed in float pairs -- the angle in
  // quarter turns + [-pi/4, pi/4], its sine and cosine by their Taylor polynomials -- which
  // is about as exact as entries from float64 (3e7 angles: within 0.55 ulp of scl) at the
  // price of sincospif.  (In float64 the entries of n = 14 took 27 us of a 110 us gradient.)
  template <class L>
  __host__ __device__ static __forceinline__ C2 entry(const L &l, F f, float scl, float scl_lo) {
    const float p = l.g_hi * f.x;
    const float e0 = fmaf(l.g_hi, f.x, -p) + fmaf(l.g_hi, f.y, l.g_lo * f.x), e = e0 - rintf(e0);
    const float r = p - rintf(p), k = rintf(4.f * (r + e)), a = fmaf(k, -0.25f, r);
    const float t = a + e, bb = t - a, tl = (a - (t - bb)) + (e - bb);  // a + e = t + tl turns
    const float h = 6.28318548f * t, hl = fmaf(6.28318548f, t, -h) + fmaf(-1.74845553e-7f, t, 6.28318548f * tl);
    const float q = h * h;
    const float sp = fmaf(q, fmaf(q, fmaf(q, 1.f / 362880.f, -1.f / 5040.f), 1.f / 120.f), -1.f / 6.f);
    const float cp = fmaf(q, fmaf(q, fmaf(q, -1.f / 3628800.f, 1.f / 40320.f), -1.f / 720.f), 1.f / 24.f);
    const float sl = fmaf(h * q, sp, fmaf(-0.5f * q, hl, hl));  // sine: h + sl
    const float w = fmaf(-0.5f, q, 1.f), wl = fmaf(-0.5f, q, 1.f - w);
    const float cl = wl + fmaf(q * q, cp, fmaf(-0.5f, fmaf(h, h, -q), -h * hl));  // cosine: w + cl
    const int n = (int)k & 3;  // quarter turns
    float ch = (n & 1) ? h : w, cx = (n & 1) ? sl : cl, sh = (n & 1) ? w : h, sx = (n & 1) ? cl : sl;
    const float cs = n == 1 || n == 2 ? -1.f : 1.f, ss = n >= 2 ? 1.f : -1.f;  // signs of cos and of -sin
    auto scaled = [&](float hi, float lo, float sign) {
      const float y = hi * scl, yl = fmaf(hi, scl, -y) + fmaf(lo, scl, hi * scl_lo);
      return sign * (y + yl);
    };
    return make_float2(scaled(ch, cx, cs), scaled(sh, sx, ss));
  }
  // a float32 or float64 cost
  __device__ static __forceinline__ F real(const void *c, int kind, uint64_t x) {
    if (kind == kCostF32) return make_float2(__ldg(reinterpret_cast<const float *>(c) + x), 0.f);
    const double f = __ldg(reinterpret_cast<const double *>(c) + x);
    const float h = (float)f;
    return make_float2(h, (float)(f - (double)h));
  }
  // Slot of tile offset i with EB register bits (rounds over consecutive bits):
  // 16 lanes of a half-warp hit 16 bank pairs in the layouts of EB 2 and 3 (and
  // all but a two-way conflict for EB 1).
  template <int EB>
  __host__ __device__ static constexpr uint32_t slot(uint32_t i) {
    return EB == 3 ? i ^ ((i >> 4) & 7u) ^ ((i >> 3) & 8u) : i ^ ((i >> 4) & 3u) ^ ((i >> 2) & 12u);
  }
  // running sum as a float pair (Knuth's TwoSum)
  struct Sum {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float x) {
      const float s = hi + x, bb = s - hi;
      lo += (hi - (s - bb)) + (x - bb);
      hi = s;
    }
    __device__ __forceinline__ void warp() {  // lane 0 gets the warp's sum
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float h = __shfl_down_sync(0xffffffffu, hi, o), l = __shfl_down_sync(0xffffffffu, lo, o);
        add(h);
        lo += l;
      }
    }
    __device__ __forceinline__ float get() const { return hi + lo; }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
  };
};

template <> struct Ops<double> {
  using C2 = double2;
  using F = double;
  __device__ static __forceinline__ F integer(int f) { return (double)f; }
  __device__ static __forceinline__ C2 mk(double x, double y) { return make_double2(x, y); }
  __device__ static __forceinline__ C2 axpy(double t, C2 a, C2 b) {
    return make_double2(fma(t, a.x, b.x), fma(t, a.y, b.y));
  }
  __device__ static __forceinline__ F cost(const void *c, int kind, uint32_t x) { return ld_cost(c, kind, x); }
  __device__ static __forceinline__ double value(F f) { return f; }
  template <class L>
  __device__ static __forceinline__ C2 phase(const L &l, F f, double scl) {
    const double t = l.g_hi * f;
    double sn, cs;
    sincospi(2.0 * (t - rint(t)), &sn, &cs);
    return make_double2(cs * scl, -sn * scl);
  }
  // for a table: from both parts of g / 2pi (a phase per amplitude takes the first alone, as it
  // always did: the two FMAs more are 3% of a complex128 pass)
  template <class L>
  __device__ static __forceinline__ C2 entry(const L &l, F f, double scl, double) {
    const double p = l.g_hi * f;
    double sn, cs;
    sincospi(2.0 * ((p - rint(p)) + fma(l.g_lo, f, fma(l.g_hi, f, -p))), &sn, &cs);
    return make_double2(cs * scl, -sn * scl);
  }
  __device__ static __forceinline__ F real(const void *c, int kind, uint64_t x) {
    return kind == kCostF32 ? (double)__ldg(reinterpret_cast<const float *>(c) + x)
                            : __ldg(reinterpret_cast<const double *>(c) + x);
  }
  // 8 lanes of a quarter-warp hit 8 slots of 16 bytes
  template <int EB>
  __host__ __device__ static constexpr uint32_t slot(uint32_t i) {
    return EB == 3 ? i ^ ((i >> 3) & 7u) : i ^ ((i >> 3) & 3u) ^ ((i >> 2) & 4u);
  }
  struct Sum {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void warp() {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    __device__ __forceinline__ double get() const { return s; }
    __device__ __forceinline__ double value() const { return s; }
  };
};

template <typename C2>
__device__ __forceinline__ C2 cm(C2 a, C2 b) {
  C2 r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}

// z * i^k
template <typename C2>
__device__ __forceinline__ C2 ipow(C2 z, int k) {
  C2 r = z;
  if (k & 1) {
    r.x = -z.y;
    r.y = z.x;
  }
  if (k & 2) {
    r.x = -r.x;
    r.y = -r.y;
  }
  return r;
}

template <typename C2>
__device__ __forceinline__ C2 neg(C2 a) {
  a.x = -a.x;
  a.y = -a.y;
  return a;
}

template <int I> struct Int { static constexpr int value = I; };

// f(Int<0>()), ..., f(Int<N - 1>())
template <int N, int I = 0, class F>
__device__ __forceinline__ void unroll(F f) {
  if constexpr (I < N) {
    f(Int<I>());
    unroll<N, I + 1>(f);
  }
}

}  // namespace tile
}  // namespace qaoa
