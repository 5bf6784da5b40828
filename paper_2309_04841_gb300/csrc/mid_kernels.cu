// mid_kernels.cu -- passes over n <= 20 vectors, both precisions: small tiles.
//
// A pass there is bound by the latency of one tile, not by bandwidth (the vectors
// stay in L2): 2^13-amplitude tiles left n = 18 with 32 CTAs of 8 warps, 12 to 20 us
// a pass.  Here a tile has 2^8 to 2^11 amplitudes, 4 a thread (two index bits), so
// that n = 18 spreads over 128 CTAs and every scheduler has two warps to switch
// between; HIGH tiles have 4-amplitude segments (one 32-byte sector, one thread's
// registers), so two groups of TB and TB - 2 qubits cover n.  Rounds of two bits
// with one exchange buffer pair each way, everything a template constant
// (tile_ops.cuh).  What the next pass can do before the previous one has ended --
// phase tables, costs, indexes -- it does: passes are launched with programmatic
// stream serialisation and wait (griddepcontrol.wait) before they touch the
// vectors.  The adjoint's partial sums are added by an extra CTA of the next pass,
// off the critical path.  Rotations are the reduced ones of pass_kernels.cu, in the
// standard basis.  Measured (objective and gradient, a library call): complex64
// p = 12 LABS n = 14 391 -> 111 us, n = 18 393 -> 187 us, without symmetry n = 18
// 394 -> 231 us; complex128 p = 2 n = 14 253 -> 77 us, p = 4 n = 18 655 -> 386 us.
#include "kernels.h"
#include "overlap.cuh"
#include "tile_ops.cuh"

namespace qaoa {

namespace {

using namespace tile;

#ifdef QAOA_MID_F64
using Real = double;
#else
using Real = float;
#endif
using O = Ops<Real>;
using C2 = O::C2;
using F = O::F;

constexpr int kH1 = 1, kPH = 2, kH2 = 4, kRED = 8, kINIT = 8;
constexpr int EB = 2, REGS = 4;

// exp(-i b X) in reduced form (pass_kernels.cu) on the register bits in mask.
__device__ __forceinline__ void rot_std(C2 (&v)[REGS], uint32_t mask, Real t, int form) {
#pragma unroll
  for (int j = 0; j < EB; ++j)
    if ((mask >> j) & 1u) {
#pragma unroll
      for (int r = 0; r < REGS; ++r)
        if (!((r >> j) & 1)) {
          C2 &x = v[r], &y = v[r | (1 << j)];
          const C2 a = x, b = y;
          if (form == 0) {
            x = O::mk(fma(t, b.y, a.x), fma(-t, b.x, a.y));
            y = O::mk(fma(t, a.y, b.x), fma(-t, a.x, b.y));
          } else {
            x = O::mk(fma(t, a.x, b.y), fma(t, a.y, -b.x));
            y = O::mk(fma(t, b.x, a.y), fma(t, b.y, -a.x));
          }
        }
    }
}

// Im <lambda| X |psi> over the pairs of the register bits in mask.
__device__ __forceinline__ Real inner_std(const C2 (&v)[REGS], const C2 (&w)[REGS], uint32_t mask) {
  Real g[2] = {0, 0};
#pragma unroll
  for (int j = 0; j < EB; ++j)
    if ((mask >> j) & 1u) {
#pragma unroll
      for (int r = 0; r < REGS; ++r)
        if (!((r >> j) & 1)) {
          const C2 pa = v[r], pb = v[r | (1 << j)], la = w[r], lb = w[r | (1 << j)];
          g[0] = fma(la.x, pb.y, g[0]);
          g[1] = fma(-la.y, pb.x, g[1]);
          g[0] = fma(lb.x, pa.y, g[0]);
          g[1] = fma(-lb.y, pa.x, g[1]);
        }
    }
  return g[0] + g[1];
}

// A tile of TB bits.  Round k holds bits 2k, 2k+1 in registers (the last round
// bits TB-2, TB-1), the others in the thread number, in order.  HIGH: bits 0, 1 are
// the segment and not rotated.  CP: tile bit TB-1 selects the box of a complement
// pair (qaoa_common.cuh).
template <int TB_, bool HIGH_, bool CP_>
struct Tile {
  static constexpr int TB = TB_, R = mid_rounds(TB), NT = 1 << (TB - EB);
  static constexpr bool HIGH = HIGH_, CP = CP_;
  __host__ __device__ static constexpr int shift(int k) { return mid_shift(TB, k); }
};

template <class TL>
struct Ctx {
  uint32_t t;          // thread of the tile
  uint32_t sb[TL::R];  // slot of its offset base in each round
  uint64_t base;       // index of tile offset 0
  __device__ __forceinline__ static uint32_t off_base(uint32_t t, int k) {
    const int s = TL::shift(k);
    return (t & ((1u << s) - 1u)) | ((t >> s) << (s + EB));
  }
  __device__ __forceinline__ uint32_t slot(int k, int r) const {
    return sb[k] ^ O::slot<EB>((uint32_t)r << TL::shift(k));
  }
  // index of the amplitude in register r of round k
  __device__ __forceinline__ uint64_t index(const Geom &g, int k, int r) const {
    uint32_t o = off_base(t, k) | ((uint32_t)r << TL::shift(k));
    const bool box1 = TL::CP && (o >> (TL::TB - 1)) != 0u;
    if (TL::CP) o &= (1u << (TL::TB - 1)) - 1u;
    const uint64_t x = base + (TL::HIGH ? (uint64_t)(o & 3u) + ((uint64_t)(o >> 2) << g.h) : (uint64_t)o);
    return box1 ? g.comp - x : x;
  }
};

template <class TL>
__device__ __forceinline__ Ctx<TL> make_ctx(const Geom &g, uint64_t T) {
  Ctx<TL> c;
  c.t = threadIdx.x;
#pragma unroll
  for (int k = 0; k < TL::R; ++k) c.sb[k] = O::slot<EB>(Ctx<TL>::off_base(c.t, k));
  c.base = TL::HIGH ? tile_base(g, T) : T << TL::TB;
  return c;
}

// Cost values of a round's registers; raw integers for the phase tables.
struct Costs {
  F f[REGS];
  int q[REGS];
};
template <class TL>
__device__ __forceinline__ void load_costs(Costs &c, const Ctx<TL> &x, const Geom &g, int k, const void *cost,
                                           int kind) {
#pragma unroll
  for (int r = 0; r < REGS; ++r) {
    const uint64_t i = x.index(g, k, r);
    c.q[r] = 0;
    if (kind == kCostI32 || kind == kCostU16) {
      c.q[r] = kind == kCostI32 ? __ldg(reinterpret_cast<const int *>(cost) + i)
                                : (int)__ldg(reinterpret_cast<const unsigned short *>(cost) + i);
      c.f[r] = O::integer(c.q[r]);
    } else {
      c.f[r] = O::real(cost, kind, i);
    }
  }
}

template <int NT>
__device__ __forceinline__ void fill_tables(C2 *tab, const PhaseData<Real> &ph) {
  for (int i = threadIdx.x; i < ph.entries; i += NT) {
    const int digit = min(i >> 6, ph.nd - 1), j = (i - 64 * digit) << (6 * digit + ph.shift);
    const bool last = i >= 64 * (ph.nd - 1);
    tab[i] = O::entry(ph, O::integer(last ? ph.fmin + j : j), last ? ph.scl : (Real)1, last ? ph.scl_lo : (Real)0);
  }
}

__device__ __forceinline__ C2 phase_of(const PhaseData<Real> &ph, const C2 *tab, F f, int q) {
  if (ph.mode == 0) {
    const uint32_t d = (uint32_t)(q - ph.fmin) >> ph.shift;
    if (ph.nd == 2) return cm(tab[d & 63u], tab[64u + min(d >> 6, (uint32_t)ph.last)]);
    return cm(cm(tab[d & 63u], tab[64u + ((d >> 6) & 63u)]), tab[128u + min(d >> 12, (uint32_t)ph.last)]);
  }
  return O::phase(ph, f, ph.scl);
}

template <int NT>
__device__ __forceinline__ void sync() {
  if constexpr (NT == 32)
    __syncwarp();
  else
    __syncthreads();
}

// Registers of round K1 -> K2 (v, and w where two), through buffer `b` of two.
template <class TL, int K1, int K2, bool TWO>
__device__ __forceinline__ void exchange(C2 (&v)[REGS], C2 (&w)[REGS], const Ctx<TL> &c, C2 *buf) {
#pragma unroll
  for (int r = 0; r < REGS; ++r) {
    buf[c.slot(K1, r)] = v[r];
    if (TWO) buf[c.slot(K1, r) + (1u << TL::TB)] = w[r];
  }
  sync<TL::NT>();
#pragma unroll
  for (int r = 0; r < REGS; ++r) {
    v[r] = buf[c.slot(K2, r)];
    if (TWO) w[r] = buf[c.slot(K2, r) + (1u << TL::TB)];
  }
}

template <class TL>
__device__ __forceinline__ void load_vec(C2 (&v)[REGS], const C2 *p, const Ctx<TL> &c, const Geom &g) {
  // round 0: four consecutive amplitudes, in descending order in box 1
  const bool down = TL::CP && (c.t >> (TL::TB - EB - 1)) != 0u;
  const uint64_t x = c.index(g, 0, down ? REGS - 1 : 0);
  const float4 *q = reinterpret_cast<const float4 *>(p + x);
  C2 t[REGS];
#pragma unroll
  for (int i = 0; i < (int)(REGS * sizeof(C2) / 16); ++i) reinterpret_cast<float4 *>(t)[i] = q[i];
#pragma unroll
  for (int r = 0; r < REGS; ++r) v[r] = down ? t[REGS - 1 - r] : t[r];
}

template <class TL>
__device__ __forceinline__ void store_vec(const C2 (&v)[REGS], C2 *p, const Ctx<TL> &c, const Geom &g, int k,
                                          uint64_t mirror) {
#pragma unroll
  for (int r = 0; r < REGS; ++r) {
    const uint64_t x = c.index(g, k, r);
    p[x] = v[r];
    if (mirror) p[mirror - x] = v[r];
  }
}

// Sum of K values over the CTA, thread 0 gets it: float pairs (complex64) within
// the warp, float64 across warps.
template <int K, int NT>
__device__ __forceinline__ void cta_sum(O::Sum (&a)[K], double (&out)[K], double *red) {
  constexpr int W = NT < 32 ? 1 : NT / 32;
#pragma unroll
  for (int k = 0; k < K; ++k) a[k].warp();
  sync<NT>();
  if ((threadIdx.x & 31u) == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[(threadIdx.x >> 5) * K + k] = a[k].value();
  sync<NT>();
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double s = 0.0;
      for (int i = 0; i < W; ++i) s += red[i * K + k];
      out[k] = s;
    }
}

// Sums of all tiles' partials [ntiles][K], by one CTA in a fixed order.
template <int K, int NT, class Fin>
__device__ __forceinline__ void sum_partials(const double *partials, uint64_t ntiles, double *red, Fin fin) {
  constexpr int W = NT < 32 ? 1 : NT / 32;
  double a[K];
#pragma unroll
  for (int k = 0; k < K; ++k) a[k] = 0.0;
  for (uint64_t i = threadIdx.x; i < ntiles; i += NT)
#pragma unroll
    for (int k = 0; k < K; ++k) a[k] += __ldcg(partials + i * K + k);
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_down_sync(0xffffffffu, a[k], o);
  sync<NT>();
  if ((threadIdx.x & 31u) == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[(threadIdx.x >> 5) * K + k] = a[k];
  sync<NT>();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      for (int i = 1; i < W; ++i) a[k] += red[i * K + k];
    fin(a);
  }
}

template <class TL, int K>
__global__ void __launch_bounds__(TL::NT) k_mid_fwd(const __grid_constant__ MidParams<Real> P) {
  constexpr bool H1 = (K & kH1) != 0, PH = (K & kPH) != 0, H2 = (K & kH2) != 0, RED = (K & kRED) != 0;
  constexpr int R = TL::R, RS = H1 && H2 ? 0 : R - 1, KP = H1 ? R - 1 : 0;  // rounds of the store and of the phase
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2 *buf = reinterpret_cast<C2 *>(smem_raw), *tab = buf + (2u << TL::TB);
  double *red = reinterpret_cast<double *>(tab + kTileTable);
  const Geom g = P.g;
  if (PH && P.ph.mode == 0) fill_tables<TL::NT>(tab, P.ph);
  const Ctx<TL> c = make_ctx<TL>(g, blockIdx.x);
  Costs cost;
  if (!P.overlap) pdl_wait();
  if (PH) load_costs(cost, c, g, KP, P.cost, P.cost_kind);
  if (P.overlap) pdl_wait();
  pdl_launch();
  C2 v[REGS], w[REGS];
  if (P.init_plus) {
#pragma unroll
    for (int r = 0; r < REGS; ++r) v[r] = O::mk(P.amp, 0);
  } else {
    load_vec(v, P.psi, c, g);
  }
  sync<TL::NT>();  // the tables
  auto phase = [&]() {
#pragma unroll
    for (int r = 0; r < REGS; ++r) v[r] = cm(v[r], phase_of(P.ph, tab, cost.f[r], cost.q[r]));
  };
  int cur = 0;
  auto next = [&]() { return buf + ((uint32_t)(cur ^= 1) << TL::TB); };
  auto sweep_up = [&](Real t, int form) {
    unroll<R>([&](auto I) {
      constexpr int k = I.value;
      if constexpr (k > 0) exchange<TL, (k > 0 ? k - 1 : 0), k, false>(v, w, c, next());
      rot_std(v, mid_mask(TL::TB, P.rot, k), t, form);
    });
  };
  if constexpr (PH && !H1) phase();
  if constexpr (H1) {
    sweep_up(P.t1, P.form1);
    if constexpr (PH) phase();
    if constexpr (H2)
      unroll<R>([&](auto I) {
        constexpr int k = R - 1 - I.value;
        if constexpr (I.value > 0) exchange<TL, (I.value > 0 ? k + 1 : 0), k, false>(v, w, c, next());
        rot_std(v, mid_mask(TL::TB, P.rot, k), P.t2, P.form2);
      });
  } else {
    sweep_up(P.t2, P.form2);
  }
  if (P.post_scale != (Real)1) {
#pragma unroll
    for (int r = 0; r < REGS; ++r) v[r] = O::mk(v[r].x * P.post_scale, v[r].y * P.post_scale);
  }
  store_vec(v, P.psi, c, g, RS, P.mirror);
  if constexpr (RED) {
    load_costs(cost, c, g, RS, P.cost, P.cost_kind);
    O::Sum a[2];
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      const Real pr = v[r].x * v[r].x + v[r].y * v[r].y;
      bool at_min = cost.q[r] == (int)P.fmin_d;  // in the cost's own type
      if (P.cost_kind == kCostF32) at_min = O::value(cost.f[r]) == (Real)P.fmin_d;
      if (P.cost_kind == kCostF64)
        at_min = __ldg(reinterpret_cast<const double *>(P.cost) + c.index(g, RS, r)) == P.fmin_d;
      a[0].add(pr * O::value(cost.f[r]));
      a[1].add(at_min ? pr : (Real)0);
    }
    double s[2];
    cta_sum<2, TL::NT>(a, s, red);
    __shared__ int last;
    if (threadIdx.x == 0) {
      P.partials[blockIdx.x * 2] = s[0];
      P.partials[blockIdx.x * 2 + 1] = s[1];
      __threadfence();
      last = atomicAdd(P.counter, 1u) == gridDim.x - 1u;
    }
    sync<TL::NT>();
    if (!last) return;
    __threadfence();
    sum_partials<2, TL::NT>(P.partials, gridDim.x, red, [&](double(&e)[2]) {
      P.out[0] = P.out_scale * e[0];
      P.out[1] = P.out_scale * e[1];
      *P.counter = 0u;
    });
  }
}

// Adds the partial sums of one adjoint pass to its gradient slots.
template <int NT>
__device__ __forceinline__ void add_gradients(const MidSums &S, double *red) {
  sum_partials<3, NT>(S.partials, S.ntiles, red, [&](double(&a)[3]) {
    if (S.out_b1) *S.out_b1 += S.scale * a[0];
    if (S.out_g) *S.out_g += S.scale * a[1];
    if (S.out_b2) *S.out_b2 += S.scale * a[2];
  });
}

__global__ void __launch_bounds__(256) k_mid_sum(const __grid_constant__ MidSums S) {
  __shared__ double red[8 * 3];
  pdl_wait();
  pdl_launch();
  add_gradients<256>(S, red);
}

template <class TL, int K>
__global__ void __launch_bounds__(TL::NT) k_mid_bwd(const __grid_constant__ MidParams<Real> P) {
  constexpr bool PH = (K & kPH) != 0, H2 = (K & kH2) != 0, INIT = (K & kINIT) != 0;
  constexpr int R = TL::R, RS = H2 ? 0 : R - 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2 *buf = reinterpret_cast<C2 *>(smem_raw), *tab = buf + (4u << TL::TB);
  double *red = reinterpret_cast<double *>(tab + kTileTable);
  const Geom g = P.g;
  if (blockIdx.x == g.ntiles) {  // the extra CTA: the previous pass's sums
    pdl_wait();
    pdl_launch();
    add_gradients<TL::NT>(P.prev, red);
    return;
  }
  if (PH && P.ph.mode == 0) fill_tables<TL::NT>(tab, P.ph);
  const Ctx<TL> c = make_ctx<TL>(g, blockIdx.x);
  Costs cost;
  if (!P.overlap) pdl_wait();
  if (INIT) load_costs(cost, c, g, 0, P.cost, P.cost_kind);
  if (PH) load_costs(cost, c, g, R - 1, P.cost, P.cost_kind);
  if (P.overlap) pdl_wait();
  pdl_launch();
  C2 v[REGS], w[REGS];
  load_vec(v, P.psi, c, g);
  const Real fc = INIT || PH ? (Real)cost_shift(P.energy) : (Real)0;
  if constexpr (INIT) {
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      const Real f = O::value(cost.f[r]) - fc;
      w[r] = O::mk(f * v[r].x, f * v[r].y);
    }
  } else {
    load_vec(w, P.lam, c, g);
  }
  sync<TL::NT>();
  int cur = 0;
  auto next = [&]() { return buf + ((uint32_t)(cur ^= 1) << (TL::TB + 1)); };
  O::Sum a[3];
  unroll<R>([&](auto I) {
    constexpr int k = I.value;
    if constexpr (k > 0) exchange<TL, (k > 0 ? k - 1 : 0), k, true>(v, w, c, next());
    const uint32_t m = mid_mask(TL::TB, P.rot, k);
    if (m != 0u) {
      a[0].add(inner_std(v, w, m) * P.w1[k]);
      rot_std(v, m, P.t1, P.form1);
      rot_std(w, m, P.t1, P.form1);
    }
  });
  if constexpr (PH) {
    Real raw = 0;
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      raw += (O::value(cost.f[r]) - fc) * (w[r].x * v[r].y - w[r].y * v[r].x);
      const C2 ph = phase_of(P.ph, tab, cost.f[r], cost.q[r]);
      v[r] = cm(v[r], ph);
      w[r] = cm(w[r], ph);
    }
    a[1].add(raw * P.wg);
  }
  if constexpr (H2)
    unroll<R>([&](auto I) {
      constexpr int k = R - 1 - I.value;
      if constexpr (I.value > 0) exchange<TL, (I.value > 0 ? k + 1 : 0), k, true>(v, w, c, next());
      const uint32_t m = mid_mask(TL::TB, P.rot, k);
      if (m != 0u) {
        a[2].add(inner_std(v, w, m) * P.w2[k]);
        rot_std(v, m, P.t2, P.form2);
        rot_std(w, m, P.t2, P.form2);
      }
    });
  if (P.post_scale != (Real)1) {
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      v[r] = O::mk(v[r].x * P.post_scale, v[r].y * P.post_scale);
      w[r] = O::mk(w[r].x * P.post_scale, w[r].y * P.post_scale);
    }
  }
  store_vec(v, P.psi, c, g, RS, P.mirror);
  store_vec(w, P.lam, c, g, RS, 0);
  double s[3];
  cta_sum<3, TL::NT>(a, s, red);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < 3; ++k) P.partials[blockIdx.x * 3 + k] = s[k];
  }
}

// ---------------------------------------------------------------- launchers

template <class TL, int K>
cudaError_t launch_fwd_k(const MidParams<Real> &P, cudaStream_t s) {
  constexpr size_t smem = (((size_t)2 << TL::TB) + kTileTable) * sizeof(C2) + 16 * 3 * 8;
  static const cudaError_t init =
      cudaFuncSetAttribute(k_mid_fwd<TL, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (init != cudaSuccess) return init;
  return launch_pdl(k_mid_fwd<TL, K>, (unsigned)P.g.ntiles, TL::NT, smem, P, P.overlap, s);
}

template <class TL, int K>
cudaError_t launch_bwd_k(const MidParams<Real> &P, cudaStream_t s) {
  constexpr size_t smem = (((size_t)4 << TL::TB) + kTileTable) * sizeof(C2) + 16 * 3 * 8;
  static const cudaError_t init =
      cudaFuncSetAttribute(k_mid_bwd<TL, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (init != cudaSuccess) return init;
  return launch_pdl(k_mid_bwd<TL, K>, (unsigned)P.g.ntiles + (P.prev.ntiles ? 1u : 0u), TL::NT, smem, P, P.overlap, s);
}

// The kinds that schedules of two groups produce: LOW starts, either ends.
template <class TL>
cudaError_t fwd_kind(const MidParams<Real> &P, int k, cudaStream_t s) {
  switch (k) {
    case kH1 | kPH | kH2: return launch_fwd_k<TL, kH1 | kPH | kH2>(P, s);
    case kH1: return launch_fwd_k<TL, kH1>(P, s);
    case kH1 | kRED: return launch_fwd_k<TL, kH1 | kRED>(P, s);
    case kPH | kH2:
      if constexpr (!TL::HIGH) return launch_fwd_k<TL, kPH | kH2>(P, s);
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
}
template <class TL>
cudaError_t bwd_kind(const MidParams<Real> &P, int k, cudaStream_t s) {
  switch (k) {
    case kPH | kH2: return launch_bwd_k<TL, kPH | kH2>(P, s);
    case kPH: return launch_bwd_k<TL, kPH>(P, s);
    case kINIT:
      if constexpr (!TL::HIGH) return launch_bwd_k<TL, kINIT>(P, s);
      return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
  }
}

template <int TB>
cudaError_t fwd_tb(const MidParams<Real> &P, bool high, int k, cudaStream_t s) {
  if (!high) return P.g.comp ? cudaErrorInvalidValue : fwd_kind<Tile<TB, false, false>>(P, k, s);
  return P.g.comp ? fwd_kind<Tile<TB, true, true>>(P, k, s) : fwd_kind<Tile<TB, true, false>>(P, k, s);
}
template <int TB>
cudaError_t bwd_tb(const MidParams<Real> &P, bool high, int k, cudaStream_t s) {
  if (!high) return P.g.comp ? cudaErrorInvalidValue : bwd_kind<Tile<TB, false, false>>(P, k, s);
  return P.g.comp ? bwd_kind<Tile<TB, true, true>>(P, k, s) : bwd_kind<Tile<TB, true, false>>(P, k, s);
}

}  // namespace

cudaError_t launch_mid_fwd(const MidParams<Real> &P, bool high, int tb, cudaStream_t s) {
  if (high && P.g.c != kMidC) return cudaErrorInvalidValue;
  switch (tb) {
    case 8: return fwd_tb<8>(P, high, P.kind, s);
    case 9: return fwd_tb<9>(P, high, P.kind, s);
    case 10: return fwd_tb<10>(P, high, P.kind, s);
    case 11: return fwd_tb<11>(P, high, P.kind, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_mid_bwd(const MidParams<Real> &P, bool high, int tb, cudaStream_t s) {
  if (high && P.g.c != kMidC) return cudaErrorInvalidValue;
  switch (tb) {
    case 8: return bwd_tb<8>(P, high, P.kind, s);
    case 9: return bwd_tb<9>(P, high, P.kind, s);
    case 10: return bwd_tb<10>(P, high, P.kind, s);
    case 11: return bwd_tb<11>(P, high, P.kind, s);
    default: return cudaErrorInvalidValue;
  }
}

#ifndef QAOA_MID_F64
cudaError_t launch_mid_sum(const MidSums &S, bool overlap, cudaStream_t s) {
  return launch_pdl(k_mid_sum, 1, 256, 0, S, overlap, s);
}
#endif

}  // namespace qaoa
