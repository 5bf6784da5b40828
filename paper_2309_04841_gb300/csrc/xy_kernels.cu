// xy_kernels.cu -- the Hamming-weight-preserving XY mixers (Sec. 3.2: the
// SU(4) extension of Algorithms 1-2) and the Dicke initial state.
//
// One XY gate exp(-i b (X_i X_j + Y_i Y_j) / 2) leaves the basis states whose
// bits i, j are 00 or 11 alone and rotates each pair (bits 10, bits 01) by
// [[cos b, -i sin b], [-i sin b, cos b]] (as three shears, see xy_pair).  A
// layer's mixer is the ordered product of its edge gates, so consecutive
// gates share qubits and must run in order.  k_xy_tile stages a tile of 2^tb amplitudes in shared memory
// (2^c contiguous "passenger" qubits 0..c-1 times rows of two windows of qubits)
// and applies a run of gates whose qubits all lie in the tile, with the layer's
// phase fused into the load of its first pass.  The gates run in rounds of up to six
// on four register bits, 16 amplitudes a thread, one sweep over shared memory and
// one barrier a round instead of one a gate (complete graph n = 19, 28 gates a pass
// on average: 20.9 -> 17.6 us a pass).
#include "qaoa_common.cuh"
#include "kernels.h"

namespace qaoa {

namespace {

template <typename C2> struct XyR;
template <> struct XyR<float2> { using R = float; };
template <> struct XyR<double2> { using R = double; };

template <typename C2>
__device__ __forceinline__ C2 xmk(typename XyR<C2>::R x, typename XyR<C2>::R y) {
  C2 r;
  r.x = x;
  r.y = y;
  return r;
}

template <typename C2>
__device__ __forceinline__ C2 xmul(C2 a, C2 b) {
  return xmk<C2>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// (u, w) <- (cos b u - i sin b w, -i sin b u + cos b w).  With v = i w this is
// the real rotation (u, v) <- (c u - s v, s u + c v), applied as Paeth's three
// shears (t = tan(b/2), s = sin b; b reduced to |b| <= pi/2, the rest an
// exact sign `neg`): every shear has determinant 1, so the rounding of t and
// s adds no systematic growth or decay of the norm over many gates, as a
// rounded (cos, sin) pair would.
template <typename C2, typename R>
__device__ __forceinline__ void xy_pair(C2 &u, C2 &w, R t, R s, bool neg) {
  const C2 v = xmk<C2>(-w.y, w.x);  // i w
  const C2 x1 = xmk<C2>(u.x - t * v.x, u.y - t * v.y);
  C2 y1 = xmk<C2>(v.x + s * x1.x, v.y + s * x1.y);
  C2 x2 = xmk<C2>(x1.x - t * y1.x, x1.y - t * y1.y);
  if (neg) {
    x2 = xmk<C2>(-x2.x, -x2.y);
    y1 = xmk<C2>(-y1.x, -y1.y);
  }
  u = x2;
  w = xmk<C2>(y1.y, -y1.x);  // -i v
}

// Two neighbouring amplitudes (p 16-byte aligned): one 16-byte access for
// complex64.
__device__ __forceinline__ void ld2(const float2 *p, float2 &a, float2 &b) {
  const float4 q = *reinterpret_cast<const float4 *>(p);
  a = make_float2(q.x, q.y);
  b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void ld2(const double2 *p, double2 &a, double2 &b) {
  a = p[0];
  b = p[1];
}
__device__ __forceinline__ void st2(float2 *p, float2 a, float2 b) {
  *reinterpret_cast<float4 *>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st2(double2 *p, double2 a, double2 b) {
  p[0] = a;
  p[1] = b;
}

// k with zero bits inserted at positions lo < hi (32-bit: tile offsets).
__device__ __forceinline__ uint32_t insert2_32(uint32_t k, int lo, int hi) {
  k = ((k >> lo) << (lo + 1)) | (k & ((1u << lo) - 1u));
  return ((k >> hi) << (hi + 1)) | (k & ((1u << hi) - 1u));
}

// Slot of tile offset i.  The low four offset bits pick the bank pair; read as two
// numbers of GF(4), offset bits 4-5 are added to both (the point (1, 1) of the
// projective line) and bits 6-7 as (1, w), beside (1, 0) and (0, 1) of bits 0-1 and
// 2-3: any two of these four bit pairs are independent, so whatever two pairs a
// round holds in registers, the 16 lanes of a half-warp hit 16 bank pairs.
__host__ __device__ constexpr uint32_t xy_slot(uint32_t i) {
  const uint32_t a = (i >> 4) & 3u, b = (i >> 6) & 3u;
  const uint32_t wb = ((b & 1u) << 1) ^ ((b >> 1) * 3u);  // w b
  return i ^ a ^ (a << 2) ^ b ^ (wb << 2);
}

__device__ __forceinline__ double xy_cost(const void *cost, int kind, uint64_t x) {
  if (kind == kCostI32) return (double)__ldg(reinterpret_cast<const int *>(cost) + x);
  if (kind == kCostU16) return (double)__ldg(reinterpret_cast<const unsigned short *>(cost) + x);
  if (kind == kCostF32) return (double)__ldg(reinterpret_cast<const float *>(cost) + x);
  return __ldg(reinterpret_cast<const double *>(cost) + x);
}

// exp(-i g f_x): complex64 reduces g f / 2pi as a float-float (Dekker's
// two-product by fma) and takes sincospif of the fraction; complex128 reduces
// in float64.
__device__ __forceinline__ float2 xy_phase(const XyPass &P, float2, uint64_t x) {
  const double fd = xy_cost(P.cost, P.cost_kind, x);
  const float fh = (float)fd, fl = (float)(fd - (double)fh);
  const float p = P.g_hi * fh;
  const float e = fmaf(P.g_hi, fh, -p);
  const float r = (p - rintf(p)) + (e + fmaf(P.g_hi, fl, P.g_lo * fh));
  float sn, cs;
  sincospif(2.0f * r, &sn, &cs);
  return make_float2(cs, -sn);
}

__device__ __forceinline__ double2 xy_phase(const XyPass &P, double2, uint64_t x) {
  const double t = P.g2pi * xy_cost(P.cost, P.cost_kind, x);
  const double r = t - rint(t);
  double sn, cs;
  sincospi(2.0 * r, &sn, &cs);
  return make_double2(cs, -sn);
}

// exp(-i g f_x) from the digit tables (copy q of entry e at e * 16 + q; see
// PhaseDigits), integer costs only.
__device__ __forceinline__ float2 xy_phase_tab(const XyPass &P, const float2 *tab, float2, uint64_t x) {
  const int f = P.cost_kind == kCostU16 ? (int)__ldg(reinterpret_cast<const unsigned short *>(P.cost) + x)
                                        : __ldg(reinterpret_cast<const int *>(P.cost) + x);
  const uint32_t d = (uint32_t)(f - P.ph.fmin) >> P.ph.shift;
  const uint32_t q = threadIdx.x & (kPhaseCopies - 1);
  if (P.ph.nd == 2) {
    const float2 a = tab[((d & 63u) << 4) | q];
    const float2 b = tab[((64u + min(d >> 6, (uint32_t)P.ph.last)) << 4) | q];
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
  }
  const float2 a = tab[((d & 31u) << 4) | q];
  const float2 b = tab[((32u + ((d >> 5) & 31u)) << 4) | q];
  const float2 c = tab[((64u + min(d >> 10, (uint32_t)P.ph.last)) << 4) | q];
  const float2 ab = make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
  return make_float2(ab.x * c.x - ab.y * c.y, ab.x * c.y + ab.y * c.x);
}

__device__ __forceinline__ double2 xy_phase_tab(const XyPass &P, const float2 *, double2, uint64_t x) {
  return xy_phase(P, double2(), x);  // complex128 always computes
}

// Global index of tile offset t in tile T: t's bits are qubits 0..c-1, h1.. and
// h2.., T fills the gaps between and above them in order.
__device__ __forceinline__ uint64_t xy_index(const XyPass &P, uint64_t T, uint32_t t) {
  const int g1 = P.h1 - P.c, top1 = P.h1 + P.w1, g2 = P.h2 - top1;
  const uint64_t lo = T & ((1ull << g1) - 1ull), mid = (T >> g1) & ((1ull << g2) - 1ull), top = T >> (g1 + g2);
  const uint32_t r1 = (t >> P.c) & ((1u << P.w1) - 1u), r2 = t >> (P.c + P.w1);
  return (uint64_t)(t & ((1u << P.c) - 1u)) | (lo << P.c) | ((uint64_t)r1 << P.h1) | (mid << top1) |
         ((uint64_t)r2 << P.h2) | (top << (P.h2 + P.w2));
}

// Registers per thread for the next tile's amplitudes (complex64; tiles of
// up to 2^12 amplitudes over 256 threads, two neighbours per load).
constexpr int kXyPrefetchPairs = (1 << kXyMaxTb) / 512;

template <typename C2>
__device__ __forceinline__ C2 xy_phased(const XyPass &P, const float2 *tab, bool table, C2 v, uint64_t x) {
  return table ? xmul(v, xy_phase_tab(P, tab, v, x)) : xmul(v, xy_phase(P, v, x));
}

// PF (complex64): the next tile's amplitudes are loaded into registers while
// the gates run on the current one in shared memory; otherwise the tile is
// loaded just before its gates.
// SINGLE: no rounds, a gate at a time, a pair a thread (xy_single in api.cu).
template <typename C2, bool PF, bool SINGLE>
__global__ void __launch_bounds__(256, PF ? 2 : 1) k_xy_tile(const __grid_constant__ XyPass P) {
  using R = typename XyR<C2>::R;
  extern __shared__ __align__(16) unsigned char xy_smem[];
  C2 *s = reinterpret_cast<C2 *>(xy_smem);
  C2 *psi = reinterpret_cast<C2 *>(P.psi);
  const uint32_t TE = 1u << P.tb;
  float2 *tab = reinterpret_cast<float2 *>(xy_smem + (size_t)TE * sizeof(C2));
  const R th = (R)P.tb2, sn = (R)P.sb;
  const bool neg = P.neg != 0;
  const bool table = P.has_phase && P.ph.mode == 0;
  if (table) {
    for (int i = threadIdx.x; i < P.ph.nent * kPhaseCopies; i += blockDim.x) tab[i] = P.ph.d[i >> 4];
    __syncthreads();
  }
  // pairs of neighbouring amplitudes (tile bit 0 is qubit 0, c >= 1): one
  // 16-byte load per complex64 pair; thread tid holds offsets 2 (tid + 256 i)
  C2 r[PF ? 2 * kXyPrefetchPairs : 1];
  auto load_regs = [&](uint64_t T) {
    if constexpr (PF) {
#pragma unroll
      for (int i = 0; i < kXyPrefetchPairs; ++i) {
        const uint32_t t = 2 * (threadIdx.x + 256u * i);
        if (t < TE) ld2(psi + xy_index(P, T, t), r[2 * i], r[2 * i + 1]);
      }
    }
  };
  if (blockIdx.x < P.ntiles) load_regs(blockIdx.x);
  for (uint64_t T = blockIdx.x; T < P.ntiles; T += gridDim.x) {
    if constexpr (PF) {
#pragma unroll
      for (int i = 0; i < kXyPrefetchPairs; ++i) {
        const uint32_t t = 2 * (threadIdx.x + 256u * i);
        if (t < TE) {
          C2 v0 = r[2 * i], v1 = r[2 * i + 1];
          if (P.has_phase) {
            const uint64_t x = xy_index(P, T, t);
            v0 = xy_phased(P, tab, table, v0, x);
            v1 = xy_phased(P, tab, table, v1, x + 1);
          }
          s[xy_slot(t)] = v0;
          s[xy_slot(t + 1)] = v1;
        }
      }
      __syncthreads();
      if (T + gridDim.x < P.ntiles) load_regs(T + gridDim.x);
    } else {
      for (uint32_t t = 2 * threadIdx.x; t < TE; t += 2 * blockDim.x) {
        const uint64_t x = xy_index(P, T, t);  // even
        C2 v0, v1;
        ld2(psi + x, v0, v1);
        if (P.has_phase) {
          v0 = xy_phased(P, tab, table, v0, x);
          v1 = xy_phased(P, tab, table, v1, x + 1);
        }
        s[xy_slot(t)] = v0;
        s[xy_slot(t + 1)] = v1;
      }
      __syncthreads();
    }
    for (int k = 0; k < P.nrounds; ++k) {
      const XyRound rd = P.rounds[k];
      if constexpr (!SINGLE) {
        uint32_t e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) e[j] = xy_slot(1u << rd.bit[j]);
        for (uint32_t i = threadIdx.x; i < (TE >> 4); i += blockDim.x) {
          uint32_t o = i;
#pragma unroll
          for (int j = 0; j < 4; ++j) o = ((o >> rd.bit[j]) << (rd.bit[j] + 1)) | (o & ((1u << rd.bit[j]) - 1u));
          C2 v[16];
          o = xy_slot(o);  // (linear over XOR)
          auto at = [&](int q) -> C2 & {
            return s[o ^ ((q & 1) ? e[0] : 0u) ^ ((q & 2) ? e[1] : 0u) ^ ((q & 4) ? e[2] : 0u) ^ ((q & 8) ? e[3] : 0u)];
          };
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = at(q);
#pragma unroll
          for (int g = 0; g < 6; ++g)
            if ((rd.mask >> g) & 1) {
              const int a = xy_gate_a(g), b = xy_gate_b(g);
#pragma unroll
              for (int q = 0; q < 16; ++q)
                if (((q >> a) & 1) && !((q >> b) & 1))
                  xy_pair<C2, R>(v[q], v[q ^ (1 << a) ^ (1 << b)], th, sn, neg);
            }
#pragma unroll
          for (int q = 0; q < 16; ++q) at(q) = v[q];
        }
        __syncthreads();
      } else {
        const uint32_t bits = rd.bit[0] | rd.bit[1] << 8 | rd.bit[2] << 16 | (uint32_t)rd.bit[3] << 24;
#pragma unroll 1
        for (int g = 0; g < 6; ++g)
          if ((rd.mask >> g) & 1) {
            const int a = (bits >> (8 * xy_gate_a(g))) & 255u, b = (bits >> (8 * xy_gate_b(g))) & 255u;
            for (uint32_t i = threadIdx.x; i < (TE >> 2); i += blockDim.x) {
              const uint32_t t0 = insert2_32(i, a, b);
              xy_pair<C2, R>(s[xy_slot(t0 | (1u << a))], s[xy_slot(t0 | (1u << b))], th, sn, neg);
            }
            __syncthreads();
          }
      }
    }
    for (uint32_t t = 2 * threadIdx.x; t < TE; t += 2 * blockDim.x) {
      st2(psi + xy_index(P, T, t), s[xy_slot(t)], s[xy_slot(t + 1)]);
    }
    __syncthreads();
  }
}

// |D^n_k>: amplitude C(n, k)^{-1/2} on every x of Hamming weight k, else 0.
template <typename C2>
__global__ void __launch_bounds__(256) k_dicke(C2 *psi, int n, int k, double amp) {
  using R = typename XyR<C2>::R;
  const uint64_t N = 1ull << n;
  for (uint64_t x = blockIdx.x * 256ull + threadIdx.x; x < N; x += (uint64_t)gridDim.x * 256ull)
    psi[x] = xmk<C2>(__popcll(x) == k ? (R)amp : (R)0, (R)0);
}

unsigned grid_n(uint64_t work, int nsm) {
  const uint64_t b = (work + 255) / 256, cap = (uint64_t)nsm * 8;
  return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

template <typename C2, bool PF, bool SINGLE>
static cudaError_t launch_xy_tile_t(const XyPass &P, cudaStream_t s, int nsm) {
  const size_t tabb = (size_t)kPhaseTabEntries * sizeof(float2);
  const size_t smem = sizeof(C2) << P.tb, most = (sizeof(C2) << kXyMaxTb) + (sizeof(C2) == 8 ? tabb : 0);
  auto kern = k_xy_tile<C2, PF, SINGLE>;
  static int per_sm = 0;  // resident CTAs per SM (registers, shared memory)
  if (!per_sm) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e != cudaSuccess) return e;
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, 256, most) != cudaSuccess || b < 1) b = 1;
    per_sm = b;
  }
  const uint64_t cap = (uint64_t)nsm * per_sm;
  const unsigned grid = (unsigned)(P.ntiles < cap ? P.ntiles : cap);
  kern<<<grid, 256, smem + (P.has_phase && P.ph.mode == 0 ? tabb : 0), s>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_xy_tile(const XyPass &P, bool c128, cudaStream_t s, int nsm) {
  if (!P.single && P.tb < 4) return cudaErrorInvalidValue;  // a round holds four tile bits
  if (c128)
    return P.single ? launch_xy_tile_t<double2, false, true>(P, s, nsm) : launch_xy_tile_t<double2, false, false>(P, s, nsm);
  // prefetching the next tile into registers pays on tiles that fill the CTA; the smallest ones
  // are bound by fetching that code (ring n = 6 p = 6 33 -> 28 us of device time without)
  if (P.single) return launch_xy_tile_t<float2, false, true>(P, s, nsm);
  return P.tb > 9 ? launch_xy_tile_t<float2, true, false>(P, s, nsm) : launch_xy_tile_t<float2, false, false>(P, s, nsm);
}

cudaError_t launch_dicke(void *psi, bool c128, int n, int k, double amp, cudaStream_t s, int nsm) {
  const unsigned grid = grid_n(1ull << n, nsm);
  if (c128)
    k_dicke<double2><<<grid, 256, 0, s>>>(reinterpret_cast<double2 *>(psi), n, k, amp);
  else
    k_dicke<float2><<<grid, 256, 0, s>>>(reinterpret_cast<float2 *>(psi), n, k, amp);
  return cudaGetLastError();
}

}  // namespace qaoa
