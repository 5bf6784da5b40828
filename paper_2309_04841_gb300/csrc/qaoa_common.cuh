// qaoa_common.cuh -- device helpers, tile plans and kernel parameter blocks
// shared by the kernels and the host planner of the sm_103a QAOA library.
//
// A "pass" streams the whole state vector through the SMs once.  The state
// is cut into tiles of 2^TB amplitudes; tile bit j maps to basis-index bit
//   j            for j <  c   (low segment: contiguous, gives coalescing)
//   h + (j - c)  for j >= c   (high segment: any run of qubits)
// so a pass can rotate any TB-qubit window (Algorithm 1 on each of them)
// while every global access still moves whole 2^c-amplitude segments.
// Inside a tile each thread holds 2^EB amplitudes in registers; a "round"
// assigns EB tile bits to registers, 5 to lanes and the rest to warps, and
// smem transposes move between rounds.  Rotations of register bits need no
// data movement at all.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace qaoa {

template <typename R> struct C2T;
template <> struct C2T<float> { using type = float2; };
template <> struct C2T<double> { using type = double2; };

// Scatter the low bits of v into the set bits of mask (parallel bit deposit).
__host__ __device__ constexpr uint32_t pdep(uint32_t v, uint32_t mask) {
  uint32_t out = 0;
  int k = 0;
  for (int b = 0; b < 32; ++b) {
    if ((mask >> b) & 1u) {
      if ((v >> k) & 1u) out |= 1u << b;
      ++k;
    }
  }
  return out;
}

__host__ __device__ constexpr int popc_c(uint32_t m) {
  int c = 0;
  for (int b = 0; b < 32; ++b) c += (m >> b) & 1u;
  return c;
}

__host__ __device__ constexpr int log2_c(int v) { return v <= 1 ? 0 : 1 + log2_c(v >> 1); }

// Tile plan: TB tile bits, 2^EB registers per thread, NT threads, NR rounds
// given as (register, lane, warp) masks over tile bits; smem slot swizzle
// s = t ^ ((t >> SWS) & m) with m = 15 for 8-byte and 7 for 16-byte
// amplitudes, chosen so every round's smem access pattern is bank-conflict
// free (each half-warp / quarter-warp hits distinct 128-byte bank rows).
template <int TB_, int EB_, int NT_, int SWS_, int NR_, uint32_t R0, uint32_t L0,
          uint32_t W0, uint32_t R1, uint32_t L1, uint32_t W1, uint32_t R2 = 0,
          uint32_t L2 = 0, uint32_t W2 = 0>
struct Plan {
  static constexpr int TB = TB_, EB = EB_, NT = NT_, SWS = SWS_, NR = NR_;
  static constexpr int NREG = 1 << EB_;
  __host__ __device__ static constexpr uint32_t reg(int r) { return r == 0 ? R0 : r == 1 ? R1 : R2; }
  __host__ __device__ static constexpr uint32_t lane(int r) { return r == 0 ? L0 : r == 1 ? L1 : L2; }
  __host__ __device__ static constexpr uint32_t warp(int r) { return r == 0 ? W0 : r == 1 ? W1 : W2; }
  __host__ __device__ static constexpr bool valid_round(int r) {
    return popc_c(reg(r)) == EB && popc_c(lane(r)) == 5 &&
           popc_c(warp(r)) == log2_c(NT / 32) && (reg(r) & lane(r)) == 0 &&
           (reg(r) & warp(r)) == 0 && (lane(r) & warp(r)) == 0 &&
           (reg(r) | lane(r) | warp(r)) == ((1u << TB) - 1u);
  }
  __host__ __device__ static constexpr bool valid() {
    return (1 << TB) == NT * NREG && valid_round(0) && valid_round(1) &&
           (NR < 3 || valid_round(2)) && (lane(0) & 0x1Fu) == 0x1Fu;
  }
};

// complex64 forward: 8192-amplitude tiles (64 KB), 32 amplitudes/thread.
using PlanF13Low = Plan<13, 5, 256, 5, 3, 0x1F00, 0x001F, 0x00E0,
                        0x001F, 0x03E0, 0x1C00, 0x03E0, 0x001F, 0x1C00>;
using PlanF13High = Plan<13, 5, 256, 5, 2, 0x1F00, 0x001F, 0x00E0,
                         0x01F0, 0x020F, 0x1C00>;
// 4096-amplitude tiles, 16 amplitudes/thread: complex64 adjoint (two
// vectors, 64 KB) and complex128 forward (64 KB).
using PlanT12Low = Plan<12, 4, 256, 4, 3, 0x0F00, 0x001F, 0x00E0,
                        0x000F, 0x01F0, 0x0E00, 0x00F0, 0x010F, 0x0E00>;
using PlanT12High = Plan<12, 4, 256, 4, 2, 0x0F00, 0x001F, 0x00E0,
                         0x00F0, 0x010F, 0x0E00>;
// 2048-amplitude tiles, 16 amplitudes/thread: complex128 adjoint.
using PlanT11Low = Plan<11, 4, 128, 4, 3, 0x0780, 0x001F, 0x0060,
                        0x000F, 0x01F0, 0x0600, 0x00F0, 0x010F, 0x0600>;
using PlanT11High = Plan<11, 4, 128, 4, 2, 0x0780, 0x001F, 0x0060,
                         0x00F0, 0x010F, 0x0600>;

static_assert(PlanF13Low::valid() && PlanF13High::valid(), "bad F13 plan");
static_assert(PlanT12Low::valid() && PlanT12High::valid(), "bad T12 plan");
static_assert(PlanT11Low::valid() && PlanT11High::valid(), "bad T11 plan");

// Passenger (low-segment) bits of a HIGH pass: 2^4 contiguous amplitudes
// (128 B for complex64, 256 B for complex128) per global segment.
constexpr int kHighC = 4;
constexpr int kMidC = 2;  // of the small tiles (mid_kernels.cu)

// The gradient is the same for f and f - c, any c: d/d beta and d/d gamma are
// commutators' expectations.  With c = E the vector lambda = (f - c) psi is as
// short as it can be, and Im <lambda|(f - c)|psi> sums terms of the size of the
// costs' spread instead of their mean, so the roundings that both carry weigh
// less.  NULL: c = 0 (streamed complex64 passes over integer costs; api.cu says why).
__device__ __forceinline__ double cost_shift(const double *energy) {
  if (!energy) return 0.0;
  const double e = __ldcg(energy);
  return isfinite(e) ? e : 0.0;
}

enum CostKind : int { kCostI32 = 0, kCostF32 = 1, kCostF64 = 2, kCostU16 = 3 };

// Tile geometry of one pass (see file comment).  A complement pair (comp != 0,
// the all-ones mask of the vector's index): tile bit tb - 1 is no index bit but
// selects one of two boxes of 2^(tb-1) amplitudes, tile offset t with that bit
// set being the amplitude whose index is the complement of the one at t without
// it, so the rotation that pairs x with ~x acts on that tile bit.
struct Geom {
  int n, c, h, tb;
  uint64_t ntiles;
  uint64_t comp;
};

__device__ __forceinline__ uint64_t tile_base(const Geom &g, uint64_t T) {
  const int mid = g.h - g.c;  // outer bits between the two segments
  const uint64_t lo = T & ((1ull << mid) - 1ull);
  const uint64_t hi = T >> mid;
  return (lo << g.c) | (hi << (g.h + g.tb - g.c - (g.comp ? 1 : 0)));
}

__device__ __forceinline__ uint64_t tile_off(const Geom &g, uint32_t t) {
  return (uint64_t)(t & ((1u << g.c) - 1u)) + ((uint64_t)(t >> g.c) << g.h);
}

// Rotation schedule of one sweep: for round r, bit i of m[r] says "rotate
// register bit i in this round" and bit i of lm[r] "rotate the tile bit held
// by lane-index bit i, with a warp shuffle" (TMA kernels only).
struct Sweep {
  uint8_t m[4];
  uint8_t lm[4];
};

// ------------------------------------------------------------ parameters
// Per-layer phase data.  Mode 0, integer costs of a small range, with
// d = (f - fmin) >> shift: exp(-i g f) = T0[d & 63] T1[d >> 6] (nd 2), or three
// digits, T0[d & 63] T1[(d >> 6) & 63] T2[d >> 12]; each CTA builds the `entries`
// of its tables (fill_phase).  Mode 1: computed per amplitude.  Both reduce
// g f / 2 pi from g / 2 pi as a pair of Reals: rounded to one it would be off by a
// relative error that all amplitudes share.
constexpr int kTileTable = 192;  // most entries
template <typename Real>
struct PhaseData {
  using C2 = typename C2T<Real>::type;
  int mode;
  int fmin, shift;
  int nd, last, entries;  // digits; entries of the last table - 1; of all
  Real g_hi, g_lo;   // g / 2pi = g_hi + g_lo
  Real scl, scl_lo;  // factor applied with the phase (the last table carries it), as a pair
};

template <typename Real>
struct FwdParams {
  using C2 = typename C2T<Real>::type;
  C2 *psi;
  const void *cost;
  int cost_kind;
  Geom g;
  Sweep s1, s2;         // s1 before the phase, s2 after
  // the sweeps' rotations in reduced form (rot_tan): multiplier and form;
  // the state is stored divided by the product of the dropped factors, which
  // the host folds into the next phase or into post_scale
  Real t1, t2;
  int form1, form2;
  Real post_scale;      // the pass's result times this before the reduction and the store
  int has_phase;
  int init_plus;        // ignore psi, start from |+>
  Real amp;             // 2^{-n/2}
  int reduce;           // fused energy/overlap in the final layout
  double fmin_d;        // ground-state value for the overlap
  double *partials;     // [ntiles][2]
  unsigned *counter;
  double *out;          // [2]: E, O
  double out_scale;     // E and O times this (2 where half of the amplitudes are held)
  uint64_t mirror;      // nonzero (2^n - 1): amplitude x is also stored at its complement
  PhaseData<Real> ph;
};

template <typename Real>
struct BwdParams {
  using C2 = typename C2T<Real>::type;
  C2 *psi, *lam;
  const void *cost;
  int cost_kind;
  Geom g;
  Sweep s1, s2;
  Real t1, t2;            // un-rotations in reduced form (rot_tan of -beta)
  int form1, form2;
  // psi and lambda are stored divided by a common real factor sigma; a raw
  // inner product is the true one divided by sigma^2, so each round's sum is
  // weighted by that round's sigma^2 (w1 / w2 per round, wg for the phase)
  Real w1[3], w2[3], wg;
  Real post_scale;        // psi and lambda times this before the store
  int has_phase;          // g_gamma accumulation + un-phase between sweeps
  int init_lambda;        // lambda <- (f - E) psi at load
  const double *energy;   // E of the forward sweep or NULL (cost_shift)
  double *partials;       // [ntiles][3]
  unsigned *counter;
  double *out_b1, *out_g, *out_b2;  // gradient slots (accumulated: +=)
  double out_scale;       // inner products times this before they are added
  uint64_t mirror;        // nonzero (2^n - 1): psi[x] is also stored at its complement
  PhaseData<Real> ph;     // un-phase data (exp(+i g f))
};

// ---- small-tile passes, n <= 20 (mid_kernels.cu)
constexpr int kMidMaxN = 20, kMidMaxRounds = 6;

// Partial sums [ntiles][3] of an adjoint pass and the slots that scale times
// their sums are added to; ntiles 0: none.
struct MidSums {
  const double *partials;
  uint64_t ntiles;
  double *out_b1, *out_g, *out_b2;
  double scale;
};

// The register bits that round k of a tile of TB bits rotates: round k holds bits
// 2k, 2k+1 (the last one TB-2, TB-1) and leaves what an earlier round has rotated.
__host__ __device__ constexpr int mid_rounds(int TB) { return (TB + 1) / 2; }
__host__ __device__ constexpr int mid_shift(int TB, int k) { return 2 * k < TB - 2 ? 2 * k : TB - 2; }
__host__ __device__ constexpr uint32_t mid_mask(int TB, uint32_t rot, int k) {
  const uint32_t fresh = mid_shift(TB, k) < 2 * k ? 2u : 3u;
  return (rot >> mid_shift(TB, k)) & fresh;
}

template <typename Real>
struct MidParams {
  using C2 = typename C2T<Real>::type;
  C2 *psi, *lam;
  const void *cost;
  int cost_kind;
  Geom g;
  int kind;             // as the TMA passes': kernels.h
  uint32_t rot;         // tile bits rotated by each sweep
  Real t1, t2;          // sweeps before and after the phase, reduced (FwdParams, BwdParams)
  int form1, form2;
  Real w1[kMidMaxRounds], w2[kMidMaxRounds], wg;
  Real post_scale;
  int init_plus;
  int overlap;          // launched to overlap the pass before it, whose own costs were complete
  Real amp;
  double fmin_d;
  const double *energy;
  double *partials;
  unsigned *counter;
  double *out;
  double out_scale;
  uint64_t mirror;
  MidSums prev;         // summed by an extra CTA
  PhaseData<Real> ph;
};

// ---- single-CTA kernels (small_kernels.cu)
constexpr int kSmallMaxN = 12;  // most index bits one CTA holds
constexpr int kSmallMaxLayers = 128;  // most layers of a request that the server batches

// A register tile of d index bits holds 2^eb amplitudes a thread: few where that
// fills more of a warp, or more warps.  complex128 takes fewer than complex64:
// its phases are long dependent chains, which only other warps overlap (d = 8, costs
// without tables, n = 8 p = 6 gradient: 146 us with 4 amplitudes a thread, 116 with 2).  Its
// rounds, the lowest register bit of round k, and (bit j: register bit j) the
// index bits that round k rotates: eb k .. eb (k + 1) - 1.
__host__ __device__ constexpr int small_dims(int n, int half) { return n - half; }
template <typename Real>
struct SmallTile {
  static constexpr bool F64 = sizeof(Real) == 8;
  static constexpr int kMaxRounds = F64 ? 8 : 6;
  static constexpr int kMaxLayers = F64 ? 96 : 128;  // layers a launch
  // exchange buffers: two save a barrier, where they fit
  __host__ __device__ static constexpr int buffers(int d) { return F64 && d > 10 ? 1 : 2; }
  static constexpr int kTermLayers = F64 ? 4 : 8;    // adjoint layers whose gradient terms are summed at once
  __host__ __device__ static constexpr int eb(int d) {
    return F64 ? (d <= 8 ? 1 : d <= 11 ? 2 : 3) : (d <= 6 ? 1 : d <= 9 ? 2 : 3);
  }
  __host__ __device__ static constexpr int threads(int d) { return d - eb(d) < 5 ? 32 : 1 << (d - eb(d)); }
  __host__ __device__ static constexpr int rounds(int d) { return (d + eb(d) - 1) / eb(d); }
  __host__ __device__ static constexpr int shift(int d, int k) {
    return eb(d) * k < d - eb(d) ? eb(d) * k : d - eb(d);
  }
  // index bits that round k rotates: the bits of mask(d, k)
  __host__ __device__ static constexpr int rotated(int d, int k) { return eb(d) * (k + 1) <= d ? eb(d) : d - eb(d) * k; }
  __host__ __device__ static constexpr uint32_t mask(int d, int k) {
    uint32_t m = 0;
    for (int j = 0; j < eb(d); ++j)
      if (shift(d, k) + j >= eb(d) * k) m |= 1u << j;
    return m;
  }
};

// Phase tables: bytes, and layers whose tables are built at once.
constexpr int kSmallTableBytes = 8192;
template <typename Real>
__host__ __device__ constexpr int small_table_layers(int entries) {
  return kSmallTableBytes / (entries * 2 * (int)sizeof(Real));
}

// One layer.  Rotations are reduced (kernels.h): multiplier tau of form `form`,
// sig / sig_adj the product of the dropped factors over the layer's rotations,
// forward and adjoint.  An inner product taken part-way through an adjoint layer
// is weighted by the square of the factors dropped so far in that layer: before
// step i of the rounds upward / downward, w_comp at the complement rotation, wg
// after the last rotation.
template <typename Real>
struct SmallLayer {
  Real tau, sig, sig_adj, wg;
  Real w[2][SmallTile<Real>::kMaxRounds], w_comp[2];  // [1] upward, [0] downward
  Real g_hi, g_lo;  // g / 2pi = g_hi + g_lo
  int form;
  int pad;  // to 8-byte words (copied as such)
};

// One request for the on-chip kernels (a launch of k_small runs one, a launch
// of k_small_batch runs one per CTA from a device array of these).
template <typename Real>
struct SmallJob {
  using C2 = typename C2T<Real>::type;
  C2 *psi, *lam;
  const void *cost;
  int cost_kind;
  int n, nl;        // qubits; layers in this launch
  int mode;         // 0 forward, 1 forward + adjoint, 2 adjoint only
  // integer costs of a small range, d = (f - fmin) >> shift: phases from a table
  // by d (ndig 0), or from two, of 64 entries by its low digit and of ndig by the
  // rest; entries of both.  by_x: a table by the amplitude, any costs.  entries 0:
  // phases computed
  int entries, ndig, shift, fmin, by_x;
  int half;         // complement symmetry: n - 1 index bits are held
  int init_plus, init_lambda, reduce;
  Real amp;
  double fmin_d;
  double *out;              // [E, O] (mode 2 with init_lambda reads E)
  double *out_dg, *out_db;  // per-layer gradient outputs
  const SmallLayer<Real> *L;
};

// Launch parameters with room for CAP layers (a launch copies all of it, so
// short circuits take a small block).
template <typename Real, int CAP>
struct SmallParams {
  SmallJob<Real> job;  // job.L unused
  SmallLayer<Real> L[CAP];
};

}  // namespace qaoa
