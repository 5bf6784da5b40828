// small_kernels.cu -- n <= 12: one CTA holds the whole state (and lambda) on
// chip and runs many layers of Algorithm 3 (and their adjoint) in a single
// launch.
//
// Bound by latency: one CTA, a few warps, a chain of layers.  The state sits in
// registers, up to 8 amplitudes a thread (3 index bits), so a layer of d index
// bits takes ceil(d / 3) rounds of up to three rotations with no data movement and
// one shared-memory exchange (one barrier) between rounds, instead of a barrier
// and a sweep over shared memory per qubit; consecutive layers walk the rounds
// in opposite directions, so no exchange is spent on returning.  Costs with the
// complement symmetry are run on the d = n - 1 index bits of half the state; the
// top qubit's rotation then reads each amplitude's complement at the first
// exchange.  Rotations are the reduced real ones of the twisted basis
// (kernels.h), 2 packed FMAs a pair; a thread's gradient terms of a layer go to
// shared memory and are summed for several layers at once.  Compiled once per
// precision.  LABS n = 10 p = 12 objective and gradient: 222 -> 37 us
// a call, n = 12 586 -> 66 us; complex128 877 -> 254 and 3577 -> 953 us.
#include <cstring>

#include "kernels.h"
#include "tile_ops.cuh"

namespace qaoa {

namespace {

using namespace tile;

// Deterministic block sum (fixed tree); thread 0 gets the result.
template <int K>
__device__ __forceinline__ void bsum(double (&a)[K], double *red) {
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_down_sync(0xffffffffu, a[k], o);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[w * K + k] = a[k];
  __syncthreads();
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double s = 0.0;
      for (int i = 0; i < nw; ++i) s += red[i * K + k];
      a[k] = s;
    }
  __syncthreads();
}

// Rotations of the register bits in MASK (bit j: register bit j), in reduced form.
template <typename Real, int EB, uint32_t MASK>
__device__ __forceinline__ void rot(typename Ops<Real>::C2 (&v)[1 << EB], Real t, int form) {
  using O = Ops<Real>;
  auto pairs = [&](auto upd) {
#pragma unroll
    for (int j = 0; j < EB; ++j)
      if ((MASK >> j) & 1u) {
#pragma unroll
        for (int r = 0; r < (1 << EB); ++r)
          if (!((r >> j) & 1)) upd(v[r], v[r | (1 << j)]);
      }
  };
  if (form == 0)
    pairs([&](typename O::C2 &x, typename O::C2 &y) {
      const typename O::C2 a = x, b = y;
      x = O::axpy(t, b, a);
      y = O::axpy(-t, a, b);
    });
  else
    pairs([&](typename O::C2 &x, typename O::C2 &y) {
      const typename O::C2 a = x, b = y;
      x = O::axpy(t, a, b);
      y = O::axpy(t, b, neg(a));
    });
}

// Sum over the masked bits' pairs of Im <lambda| X |psi> (twisted basis).
template <typename Real, int EB, uint32_t MASK>
__device__ __forceinline__ Real inner(const typename Ops<Real>::C2 (&v)[1 << EB],
                                      const typename Ops<Real>::C2 (&w)[1 << EB]) {
  using O = Ops<Real>;
  typename O::C2 p[2] = {O::mk(0, 0), O::mk(0, 0)}, q[2] = {O::mk(0, 0), O::mk(0, 0)};
#pragma unroll
  for (int j = 0; j < EB; ++j)
    if ((MASK >> j) & 1u) {
#pragma unroll
      for (int r = 0; r < (1 << EB); ++r)
        if (!((r >> j) & 1)) {
          const int k = (r >> (j == 0 ? 1 : 0)) & 1, h = r | (1 << j);
          if constexpr (sizeof(Real) == 4) {
            p[k] = __ffma2_rn(w[r], v[h], p[k]);
            q[k] = __ffma2_rn(w[h], v[r], q[k]);
          } else {
            p[k] = O::mk(fma(w[r].x, v[h].x, p[k].x), fma(w[r].y, v[h].y, p[k].y));
            q[k] = O::mk(fma(w[h].x, v[r].x, q[k].x), fma(w[h].y, v[r].y, q[k].y));
          }
        }
    }
  return ((p[0].x + p[1].x) + (p[0].y + p[1].y)) - ((q[0].x + q[1].x) + (q[0].y + q[1].y));
}

}  // namespace

// mode 0: forward layers [0, nl) (+ optional E/O reduction)
// mode 1: forward all layers, E/O, then the whole adjoint sweep (grad)
// mode 2: adjoint sweep over layers [0, nl) in reverse, continuing from the
//         psi / lambda stored by a previous launch (or lambda = (f - E) psi)
//
// Thread t < 2^(D-EB) holds, in the layout of round k, the 2^EB amplitudes whose
// index bits s .. s+EB-1 (s = SmallTile::shift(D, k)) are the register number and the
// others are t.  D is a template argument: rounds, masks and register slots are
// constants (with D at run time a layer took 2.5 us at any size, most of it
// integer instructions).  Slots of indices are linear over XOR.  Two exchange
// buffers take one barrier an exchange: a buffer is written again only after the
// barrier of the exchange between; the largest complex128 tiles have room for one
// and take two.
template <typename Real, int D>
__device__ __forceinline__ void small_run(const SmallJob<Real> &P) {
  using O = Ops<Real>;
  using C2 = typename O::C2;
  using F = typename O::F;
  using T = SmallTile<Real>;
  constexpr bool DBL = T::buffers(D) == 2;
  constexpr int EB = T::eb(D), REGS = 1 << EB, R = T::rounds(D);
  constexpr uint32_t N = 1u << D, NT = 1u << (D - EB), all = N - 1u;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const bool grad = P.mode != 0, half = P.half != 0;
  C2 *buf = reinterpret_cast<C2 *>(smem_raw);  // psi, lambda, then the second pair
  F *fs = reinterpret_cast<F *>(buf + N * (uint32_t)((DBL ? 2 : 1) * (grad ? 2 : 1)));
  C2 *tab = reinterpret_cast<C2 *>(fs + N);  // phase tables of some layers
  C2 *terms = tab + kSmallTableBytes / sizeof(C2);  // [small_term_layers][NT + 1] of (d/d beta, d/d gamma)
  double *red = reinterpret_cast<double *>(terms + (grad ? SmallTile<Real>::kTermLayers * (int)(NT + 1u) : 0));
  SmallLayer<Real> *Ls = reinterpret_cast<SmallLayer<Real> *>(red + 64);
  auto sync = [] {
    if constexpr (T::threads(D) == 32)
      __syncwarp();
    else
      __syncthreads();
  };
  const uint32_t tid = threadIdx.x, t = tid & (NT - 1u);  // threads beyond the tile shadow others
  const bool act = tid < NT;

  // this thread's index base and its slot in the layout of each round
  auto base_of = [&](auto K) {
    constexpr int s = T::shift(D, K.value);
    return (t & ((1u << s) - 1u)) | ((t >> s) << (s + EB));
  };
  auto index = [&](auto K, int r) { return base_of(K) | ((uint32_t)r << T::shift(D, K.value)); };
  uint32_t sb[R];
  unroll<R>([&](auto K) { sb[K.value] = O::template slot<EB>(base_of(K)); });
  auto slot = [&](auto K, int r) { return sb[K.value] ^ O::template slot<EB>((uint32_t)r << T::shift(D, K.value)); };

  for (uint32_t x = tid; x < N; x += blockDim.x) fs[O::template slot<EB>(x)] = O::cost(P.cost, P.cost_kind, x);
  {  // a copy of the layers: every layer starts with them, and from shared memory they take one latency
    static_assert(sizeof(SmallLayer<Real>) % 8 == 0, "copied in 8-byte words");
    const uint64_t *src = reinterpret_cast<const uint64_t *>(P.L);
    uint64_t *dst = reinterpret_cast<uint64_t *>(Ls);
    for (uint32_t i = tid; i < (uint32_t)P.nl * (sizeof(SmallLayer<Real>) / 8); i += blockDim.x) dst[i] = src[i];
  }
  // table digits (f - fmin) >> shift of this thread's amplitudes in the layouts
  // of the first and the last round, where the phases are applied (a cost
  // outside its statistics' range stays inside the table)
  uint16_t dg[2][REGS];
  if (P.entries) {
    const uint32_t top = P.ndig ? 64u * (uint32_t)P.ndig - 1u : (uint32_t)P.entries - 1u;
    auto digit = [&](uint32_t x) {
      if (P.by_x) return (uint16_t)x;
      const int f = P.cost_kind == kCostI32 ? reinterpret_cast<const int *>(P.cost)[x]
                                            : (int)reinterpret_cast<const unsigned short *>(P.cost)[x];
      return (uint16_t)min((uint32_t)(f - P.fmin) >> P.shift, top);
    };
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      dg[0][r] = digit(index(Int<0>(), r));
      dg[1][r] = digit(index(Int<R - 1>(), r));
    }
  }
  C2 v[REGS], w[REGS];
#pragma unroll
  for (int r = 0; r < REGS; ++r) {
    const uint32_t x = index(Int<0>(), r);
    v[r] = ipow(P.init_plus ? O::mk(P.amp, 0) : P.psi[x], -__popc(x));
  }
  bool up = true;  // the registers are in the layout of round 0 (else R - 1)
  sync();

  // complement rotation (half): kappa = i^(D-1) (-1)^popc(x), see kernels.h; a at
  // x, b at ~x, ep the sign of kappa
  constexpr bool odd = (D & 1) != 0;
  auto rot_u = [&](C2 a, C2 b, Real ep, Real tau, int form) {
    const C2 kb = odd ? O::mk(ep * b.x, ep * b.y) : O::mk(-ep * b.y, ep * b.x);
    return form == 0 ? O::axpy(tau, kb, a) : O::axpy(tau, a, kb);
  };
  int cur = 0;
  // registers in the layout of round K1 -> K2; with the complement rotation (cu),
  // whose Im <lambda| X |psi> is summed over both members of each pair
  auto exchange = [&](auto K1, auto K2, auto two, bool cu, Real tau, int form, Real &uterm) {
    C2 *bv = buf + (cur ? N * (grad ? 2u : 1u) : 0u), *bw = bv + N;
    if (act) {
#pragma unroll
      for (int r = 0; r < REGS; ++r) {
        const uint32_t i = slot(K1, r);
        bv[i] = v[r];
        if (two.value) bw[i] = w[r];
      }
    }
    sync();
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      v[r] = bv[slot(K2, r)];
      if (two.value) w[r] = bw[slot(K2, r)];
    }
    if (cu) {
      const Real eb = (((D - 1) >> 1) + __popc(base_of(K2))) & 1 ? (Real)-1 : (Real)1;
#pragma unroll
      for (int r = 0; r < REGS; ++r) {
        const uint32_t j = slot(K2, r) ^ O::template slot<EB>(all);
        const Real ep = (popc_c(r) & 1) ? -eb : eb;
        const C2 b = bv[j];
        if (two.value) {
          const C2 q = w[r];
          uterm += ep * (odd ? q.x * b.x + q.y * b.y : q.y * b.x - q.x * b.y);
          w[r] = rot_u(q, bw[j], ep, tau, form);
        }
        v[r] = rot_u(v[r], b, ep, tau, form);
      }
    }
    if (DBL)
      cur ^= 1;
    else
      sync();
  };

  // Phase tables of the layers from l0 on (as many as fit): exp(-i g f), times
  // the scale pending there, or for the adjoint the inverse phases and scales.
  // An entry costs about one sincospi, an amplitude then its lookups.
  const int TE = P.entries, LB = TE ? small_table_layers<Real>(TE) : 1;
  auto tables = [&](int l0, bool adj) {
    const int cnt = min(LB, P.nl - l0) * TE;
    sync();
    for (int i = (int)tid; i < cnt; i += (int)blockDim.x) {
      const int li = l0 + i / TE, e = i % TE;
      const SmallLayer<Real> &L = Ls[li];
      const bool low = P.ndig && e < 64;  // the low digit of two
      const Real scl = low ? (Real)1 : adj ? L.sig_adj : li == 0 ? (Real)1 : Ls[li - 1].sig;
      const int j = low ? e << P.shift : P.fmin + ((P.ndig ? (e - 64) * 64 : e) << P.shift);
      const F f = P.by_x ? fs[O::template slot<EB>((uint32_t)e)] : O::integer(j);
      // (complex64 n = 13: entries as exact as that size's always were, 102.8 -> 104.5 us; below,
      // as exact as a phase per amplitude was)
      C2 z = sizeof(Real) == 8 || (D == kSmallMaxN && half) ? O::entry(L, f, scl, (Real)0) : O::phase(L, f, scl);
      if (adj) z.y = -z.y;
      tab[i] = z;
    }
    sync();
  };
  auto table_phase = [&](int tl, uint32_t q) {
    const C2 *z = tab + tl * TE;
    return P.ndig ? cm(z[q & 63u], z[64u + (q >> 6)]) : z[q];
  };

  Real pend = 1;  // psi (and lambda) are stored divided by this
  int tl = 0;     // the layer's place in the tables
  auto forward_layer = [&](auto UP, const SmallLayer<Real> &L) {
    constexpr int E = UP.value ? 0 : 1;  // the layout the layer starts in
    Real none = 0;
    if (P.entries) {
#pragma unroll
      for (int r = 0; r < REGS; ++r) v[r] = cm(v[r], table_phase(tl, dg[E][r]));
    } else {
#pragma unroll
      for (int r = 0; r < REGS; ++r) v[r] = cm(v[r], O::phase(L, fs[slot(Int<(E ? R - 1 : 0)>(), r)], pend));
    }
    unroll<R>([&](auto I) {
      constexpr int K = UP.value ? I.value : R - 1 - I.value, K0 = UP.value ? K - 1 : K + 1;
      if constexpr (I.value > 0)
        exchange(Int<K0>(), Int<K>(), Int<0>(), I.value == 1 && half, L.tau, L.form, none);
      rot<Real, EB, T::mask(D, K)>(v, L.tau, L.form);
    });
    if (R == 1 && half) exchange(Int<0>(), Int<0>(), Int<0>(), true, L.tau, L.form, none);
    pend = L.sig;
  };
  // one adjoint layer: un-rotate (tan / cot of -beta), d/d beta and d/d gamma, un-phase
  Real fc = 0;  // costs are taken from E (cost_shift)
  auto adjoint_layer = [&](auto UP, const SmallLayer<Real> &L, int row) {
    constexpr int E = UP.value && R > 1 ? 1 : 0;  // the layout the layer ends in
    constexpr int KE = E ? R - 1 : 0;
    typename O::Sum gb;
    const Real tau = -L.tau;
    unroll<R>([&](auto I) {
      constexpr int K = UP.value ? I.value : R - 1 - I.value, K0 = UP.value ? K - 1 : K + 1;
      if constexpr (I.value > 0) {
        Real u = 0;
        exchange(Int<K0>(), Int<K>(), Int<1>(), I.value == 1 && half, tau, L.form, u);
        if (I.value == 1 && half) gb.add(u * L.w_comp[UP.value]);
      }
      gb.add(inner<Real, EB, T::mask(D, K)>(v, w) * L.w[UP.value][I.value]);
      rot<Real, EB, T::mask(D, K)>(v, tau, L.form);
      rot<Real, EB, T::mask(D, K)>(w, tau, L.form);
    });
    if (R == 1 && half) {
      Real u = 0;
      exchange(Int<0>(), Int<0>(), Int<1>(), true, tau, L.form, u);
      gb.add(u * L.w_comp[UP.value]);
    }
    Real raw = 0;
#pragma unroll
    for (int r = 0; r < REGS; ++r)
      raw += (O::value(fs[slot(Int<KE>(), r)]) - fc) * (w[r].x * v[r].y - w[r].y * v[r].x);
    if (P.entries) {
#pragma unroll
      for (int r = 0; r < REGS; ++r) {
        const C2 ph = table_phase(tl, dg[E][r]);
        v[r] = cm(v[r], ph);
        w[r] = cm(w[r], ph);
      }
    } else {
#pragma unroll
      for (int r = 0; r < REGS; ++r) {
        C2 ph = O::phase(L, fs[slot(Int<KE>(), r)], L.sig_adj);
        ph.y = -ph.y;  // exp(+i g f): the inverse phase
        v[r] = cm(v[r], ph);
        w[r] = cm(w[r], ph);
      }
    }
    if (act) terms[row * (NT + 1u) + t] = O::mk(gb.get(), raw * L.wg);
  };
  // Sums of the last `rows` layers' terms (layers l0 ..): 2 rows sums over NT
  // threads' terms, as 16-term pieces in parallel, then the pieces in order.
  auto sum_terms = [&](int l0, int rows) {
    constexpr int PIECES = NT >= 16 ? (int)(NT / 16) : 1, PER = (int)NT / PIECES;
    // (between layers the exchange buffers are free)
    double *part = 2 * SmallTile<Real>::kTermLayers * PIECES <= 64 ? red : reinterpret_cast<double *>(buf);
    sync();
    for (int i = (int)tid; i < 2 * rows * PIECES; i += (int)blockDim.x) {
      const int row = (i >> 1) % rows, piece = (i >> 1) / rows;
      typename O::Sum a;
      for (int j = 0; j < PER; ++j) {
        const C2 z = terms[row * (int)(NT + 1u) + piece * PER + j];
        a.add((i & 1) ? z.y : z.x);
      }
      part[i] = a.value();
    }
    sync();
    const double sc = half ? 4.0 : 2.0;
    for (int i = (int)tid; i < 2 * rows; i += (int)blockDim.x) {
      double a = 0.0;
      for (int piece = 0; piece < PIECES; ++piece) a += part[2 * rows * piece + i];
      ((i & 1) ? P.out_dg : P.out_db)[l0 + (i >> 1)] = sc * a;
    }
    sync();
  };

  double energy = 0.0;
  if (P.mode == 0 || P.mode == 1) {
    for (int li = 0; li < P.nl; ++li) {
      if (P.entries && li % LB == 0) tables(li, false);
      tl = li % LB;
      if (up || R == 1)
        forward_layer(Int<1>(), Ls[li]);
      else
        forward_layer(Int<0>(), Ls[li]);
      up = R == 1 || !up;
    }
#pragma unroll
    for (int r = 0; r < REGS; ++r) v[r] = O::mk(v[r].x * pend, v[r].y * pend);
    if (P.reduce) {
      double a[2] = {0.0, 0.0};
      if (act) {
#pragma unroll
        for (int r = 0; r < REGS; ++r) {
          const double f = ld_cost(P.cost, P.cost_kind, up ? index(Int<0>(), r) : index(Int<R - 1>(), r));
          const double pr = (double)v[r].x * v[r].x + (double)v[r].y * v[r].y;
          a[0] += pr * f;
          a[1] += (f == P.fmin_d) ? pr : 0.0;
        }
      }
      bsum<2>(a, red);
      if (tid == 0) {
        P.out[0] = red[0] = half ? 2.0 * a[0] : a[0];
        P.out[1] = half ? 2.0 * a[1] : a[1];
      }
      sync();
      energy = red[0];
      sync();
    }
  }

  auto at = [&](int r) { return up ? index(Int<0>(), r) : index(Int<R - 1>(), r); };
  if (grad) {
    if (P.mode == 2) energy = P.out[0];
    fc = (Real)(isfinite(energy) ? energy : 0.0);
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      if (P.mode == 1 || P.init_lambda) {
        const Real f = O::value(fs[O::template slot<EB>(at(r))]) - fc;
        w[r] = O::mk(f * v[r].x, f * v[r].y);
      } else {
        w[r] = ipow(P.lam[at(r)], -__popc(at(r)));
      }
    }
    constexpr int RB = SmallTile<Real>::kTermLayers;
    for (int li = P.nl - 1; li >= 0; --li) {
      if (P.entries && (li == P.nl - 1 || li % LB == LB - 1)) tables(li - li % LB, true);
      tl = li % LB;
      if (up || R == 1)
        adjoint_layer(Int<1>(), Ls[li], li % RB);
      else
        adjoint_layer(Int<0>(), Ls[li], li % RB);
      up = R == 1 || !up;
      if (li % RB == 0) sum_terms(li, min(RB, P.nl - li));
    }
    if (act) {
#pragma unroll
      for (int r = 0; r < REGS; ++r) P.lam[at(r)] = ipow(w[r], __popc(at(r)));
    }
  }
  if (act) {
#pragma unroll
    for (int r = 0; r < REGS; ++r) {
      const uint32_t x = at(r);
      const C2 z = ipow(v[r], __popc(x));
      P.psi[x] = z;
      if (half) P.psi[2u * N - 1u - x] = z;
    }
  }
}

template <typename Real, int D, int CAP>
__global__ void __launch_bounds__(SmallTile<Real>::threads(D)) k_small(const __grid_constant__ SmallParams<Real, CAP> P) {
  SmallJob<Real> J = P.job;
  J.L = P.L;
  small_run<Real, D>(J);
}

// Many independent requests on D index bits in one launch: CTA b runs jobs[b] (serving).
template <typename Real, int D>
__global__ void __launch_bounds__(SmallTile<Real>::threads(D)) k_small_batch(const SmallJob<Real> *jobs) {
  const SmallJob<Real> J = jobs[blockIdx.x];
  small_run<Real, D>(J);
}

// Shared memory of a job: exchange buffers, costs, phase tables, nl layers,
// block sums and per-thread gradient terms.
template <typename Real, int D>
static constexpr size_t small_smem(int nl, bool grad) {
  const size_t e = (size_t)1 << D, nt = (size_t)1 << (D - SmallTile<Real>::eb(D));
  const size_t bufs = SmallTile<Real>::buffers(D) * (grad ? 2 : 1);
  return e * (2 * sizeof(Real) * bufs + 8) + kSmallTableBytes + (size_t)nl * sizeof(SmallLayer<Real>) + 64 * 8 +
         (grad ? (nt + 1) * SmallTile<Real>::kTermLayers * 2 * sizeof(Real) : 0);
}

template <typename Real, int D, class Kernel>
static cudaError_t small_attr(Kernel kern) {
  constexpr size_t most = small_smem<Real, D>(SmallTile<Real>::kMaxLayers, true);
  static_assert(most <= 227 * 1024, "shared memory of one SM");
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

template <typename Real, int D, int CAP>
static cudaError_t launch_small_t(const SmallJob<Real> &J, const SmallLayer<Real> *layers, cudaStream_t st) {
  static const cudaError_t init = small_attr<Real, D>(k_small<Real, D, CAP>);
  if (init != cudaSuccess) return init;
  SmallParams<Real, CAP> P;
  memset(&P, 0, sizeof(P));
  P.job = J;
  for (int i = 0; i < J.nl; ++i) P.L[i] = layers[i];
  k_small<Real, D, CAP><<<1, SmallTile<Real>::threads(D), small_smem<Real, D>(J.nl, J.mode != 0), st>>>(P);
  return cudaGetLastError();
}

#ifdef QAOA_SMALL_F64
using SmallReal = double;
#else
using SmallReal = float;
#endif

// f.template operator()<D>() for the run-time d in 1 .. kSmallMaxN
template <int D = 1, class F>
static cudaError_t small_dispatch(int d, F f) {
  if (d == D) return f(Int<D>());
  if constexpr (D < kSmallMaxN) return small_dispatch<D + 1>(d, f);
  return cudaErrorInvalidValue;
}

cudaError_t launch_small(const SmallJob<SmallReal> &J, const SmallLayer<SmallReal> *layers, cudaStream_t s) {
  constexpr int ML = SmallTile<SmallReal>::kMaxLayers;
  if (J.nl < 1 || J.nl > ML) return cudaErrorInvalidValue;
  return small_dispatch(small_dims(J.n, J.half), [&](auto D) {
    return J.nl <= 16 ? launch_small_t<SmallReal, D.value, 16>(J, layers, s)
                      : launch_small_t<SmallReal, D.value, ML>(J, layers, s);
  });
}

#ifndef QAOA_SMALL_F64
cudaError_t launch_small_batch(const SmallJob<float> *d_jobs, int count, int d, int max_nl, cudaStream_t st) {
  return small_dispatch(d, [&](auto D) {
    static const cudaError_t init = small_attr<float, D.value>(k_small_batch<float, D.value>);
    if (init != cudaSuccess) return init;
    k_small_batch<float, D.value>
        <<<count, SmallTile<float>::threads(D.value), small_smem<float, D.value>(max_nl, true), st>>>(d_jobs);
    return cudaGetLastError();
  });
}
#endif

}  // namespace qaoa
