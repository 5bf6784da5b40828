// kernels.h -- launcher declarations between the host planner (api.cu) and
// the kernel translation units.  Internal to the library.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

#include "qaoa_common.cuh"

namespace qaoa {


enum TermMode : int { kTermI32 = 0, kTermFixed = 1, kTermF64 = 2 };

constexpr int kTermChunk = 1024;  // terms per launch (parameter block)
constexpr int kEdgeMax = 1536;    // edges per MaxCut launch (parameter block)

struct TermChunk {
  int n, nterms, mode, out_kind, accumulate;
  double scale, inv_scale;  // fixed mode: weights are wl * inv_scale
  void *out;
  uint64_t mask[kTermChunk];
  int64_t wl[kTermChunk];
  double wd[kTermChunk];
};

// Terms of exactly added weights for k_walsh: value(x) = (acc(x) >> shift), or
// acc(x) * inv_scale for float outputs, acc the sum of +-w.
struct WalshTerms {
  int n, nterms, out_kind, accumulate, shift;
  double scale, inv_scale;
  void *out;
  uint32_t mask[kTermChunk];
  int64_t w[kTermChunk];
};
constexpr int kWalshBits = 13;  // index bits of a tile: the smallest n

struct EdgeChunk {
  int n, m, mode, out_kind;
  double inv_scale;
  void *out;
  uint8_t ei[kEdgeMax], ej[kEdgeMax];
  int64_t wl[kEdgeMax];
  double wd[kEdgeMax];
};

cudaError_t launch_terms(const TermChunk &P, cudaStream_t s, int nsm);
cudaError_t launch_walsh(const WalshTerms &P, bool wide, cudaStream_t s, int nsm);
cudaError_t launch_labs(int n, int32_t *out, cudaStream_t s, int nsm);
cudaError_t launch_labs_u16(int n, uint16_t *out, cudaStream_t s, int nsm);
cudaError_t launch_probs(int n, void *psi, bool c128, void *out, cudaStream_t s, int nsm);
cudaError_t launch_convert(int n, const void *src, int src_kind, void *dst, int dst_kind,
                           cudaStream_t s, int nsm);
cudaError_t launch_maxcut(const EdgeChunk &P, cudaStream_t s, int nsm);
unsigned reduce_grid(int n, int nsm);
cudaError_t launch_cost_stats(int n, const void *cost, int kind, double *partials,
                              unsigned *counter, double *out, cudaStream_t s, int nsm);
cudaError_t launch_expect(int n, const void *psi, bool c128, const void *cost, int kind,
                          double fmin, double *partials, unsigned *counter, double *out, int which,
                          cudaStream_t s, int nsm);

// Small-tile passes (n <= 20), tb = 8 .. 11, one CTA a tile; k_mid_sum adds the
// last adjoint pass's sums.
cudaError_t launch_mid_fwd(const MidParams<float> &P, bool high, int tb, cudaStream_t s);
cudaError_t launch_mid_fwd(const MidParams<double> &P, bool high, int tb, cudaStream_t s);
cudaError_t launch_mid_bwd(const MidParams<float> &P, bool high, int tb, cudaStream_t s);
cudaError_t launch_mid_bwd(const MidParams<double> &P, bool high, int tb, cudaStream_t s);
cudaError_t launch_mid_sum(const MidSums &S, bool overlap, cudaStream_t s);

// tb: log2 of the tile (float: 13 forward, 12 adjoint; double: 12 forward, 11
// adjoint); other values fail with cudaErrorInvalidValue.
cudaError_t launch_fwd(const FwdParams<float> &P, bool high, int tb, cudaStream_t s, int nsm);
cudaError_t launch_fwd(const FwdParams<double> &P, bool high, int tb, cudaStream_t s, int nsm);
cudaError_t launch_bwd(const BwdParams<float> &P, bool high, int tb, cudaStream_t s, int nsm);
cudaError_t launch_bwd(const BwdParams<double> &P, bool high, int tb, cudaStream_t s, int nsm);

// Launch profiling (profile.cu): returns a record id, or -1 when disabled.
int prof_begin(cudaStream_t s);
void prof_end(int id, cudaStream_t s, const char *kind, double bytes);

// ---- complex64 passes streamed by TMA (tma_kernels.cu)
// Round plans for the TMA 128-byte swizzle (conflict-free at 8 and 16 bytes).
using PlanTmaF13Low = Plan<13, 5, 256, 0, 3, 0x1F00, 0x001F, 0x00E0,
                           0x020F, 0x01F0, 0x1C00, 0x01F0, 0x020F, 0x1C00>;
using PlanTmaF13High = Plan<13, 5, 256, 0, 2, 0x1F00, 0x001F, 0x00E0,
                            0x01F0, 0x020F, 0x1C00>;
using PlanTmaB12Low = Plan<12, 4, 256, 0, 3, 0x0F00, 0x001F, 0x00E0,
                           0x000F, 0x01F0, 0x0E00, 0x00F0, 0x010F, 0x0E00>;
using PlanTmaB12High = Plan<12, 4, 256, 0, 2, 0x0F00, 0x001F, 0x00E0,
                            0x00F0, 0x010F, 0x0E00>;
static_assert(PlanTmaF13Low::valid() && PlanTmaF13High::valid(), "bad TMA F13 plan");
static_assert(PlanTmaB12Low::valid() && PlanTmaB12High::valid(), "bad TMA B12 plan");
// Adjoint HIGH groups of 9 qubits on one 512-thread CTA per SM ("wide"): the
// 2^13-amplitude tile of psi and lambda (16 contiguous amplitudes x rows
// h..h+8, 128 KB) in one CTA; round 0 holds tile bits 8-11 in registers,
// round 1 tile bits 4-7 and tile bit 12 as lane bit 4 (a shuffle rotation).
using PlanTmaB13High = Plan<13, 4, 512, 0, 2, 0x0F00, 0x001F, 0x10E0, 0x00F0, 0x100F, 0x0F00>;
static_assert(PlanTmaB13High::valid(), "bad TMA B13 plan");
// Complement pairs: on a cost vector with f(x) = f(~x) the state keeps
// psi(x) = psi(~x), so the passes hold the 2^(n-1) amplitudes with the top
// qubit 0 (m = n - 1 index bits).  The rotation of the top qubit pairs x with
// its m-bit complement.  The one group that carries it has tiles of two boxes,
// T and ~T, of 2^(TB-1) amplitudes: tile bit TB - 1 selects the box, and tile
// offset t of box 1 is the amplitude ~x of the x at offset t of box 0.  The
// shared-memory slot of (box 1, t) is the bitwise complement of t, a constant
// XOR, so the loads stay two plain boxes.  Tile bit TB - 1 must be the last
// register bit of round 0 and a warp bit of round 1, or a warp bit of round 0 and
// the last lane bit of round 1 (the 512-thread plan: the pair's rotation is then the
// shuffle that the full vector's top qubit takes in the same place, so that both
// round every amplitude alike).
template <class PL>
constexpr bool comp_plan() {
  const int b = PL::TB - 1;
  return PL::NR == 2 && (((PL::reg(0) >> b) == 1u && (PL::warp(1) >> b) == 1u) ||
                         ((PL::warp(0) >> b) == 1u && (PL::lane(1) >> b) == 1u));
}
static_assert(comp_plan<PlanTmaF13High>() && comp_plan<PlanTmaB12High>() && comp_plan<PlanTmaB13High>(),
              "complement tile bit");

// The TMA passes hold vectors in the twisted basis s(x) = (-i)^popc(x) psi(x),
// where exp(-i b X_q) acts on a pair as the real rotation
// [[cos b, sin b], [-sin b, cos b]].  Rotations run in reduced ("tan") form,
// exp(-i b X) = sigma * G with
//   form 0: sigma = cos b,  G(a, b) = (a + t b, b - t a),  t = tan b
//   form 1: sigma = sin b,  G(a, b) = (u a + b, u b - a),  u = cot b
// (the adjoint uses -b), |t|, |u| <= 1; the host tracks the product of the
// sigmas and folds it into the next phase's tables or applies it at the end of the
// pass (scl_end).

// Phase factors of the TMA passes.  Mode 0 (integer costs): with
// d = (f - fmin) >> shift (every f - fmin a multiple of 2^shift),
//   nd = 2:  exp(-i g f) = D0[d & 63] * D1[d >> 6],
//   nd = 3:  exp(-i g f) = D0[d & 31] * D1[(d >> 5) & 31] * D2[d >> 10],
// the last table also carrying exp(-i g fmin) and the pending scale; the
// tables lie back to back in d[] (nent entries).  Shared memory holds each
// entry as 16 interleaved copies, so the 16 lanes of a half-warp read 16
// different bank pairs whatever their costs.  Mode 1: computed from
// g / 2pi = g_hi + g_lo (float-float): the fraction r of g f / 2pi splits into
// k / 64, looked up in d[] = scale * exp(-2 pi i k / 64), and a rest of at most
// 1 / 128, whose sine and cosine are their Taylor polynomials (to the third and
// fourth power; the next terms are 2e-9).  64 r has to be a small number for that: its
// integer part must fit the mantissa beside the rounding constant.  The low part of
// g f / 2pi, up to 2^-25 of it, is part of r, so from |g f / 2pi| = 2^36 on (penalties of
// 1e12, say) nd = 0 takes the form that reduces r once more; nd = 1 (float32 costs below)
// does without, 0.8% of a weighted MaxCut n = 28 gradient.  It is the pivots' arithmetic that costs
// there: weighted MaxCut n = 28 pivots 658 -> 559 us forward and 1339 -> 1161 us
// adjoint against sincospi and a scale multiply per amplitude; the phase's error is
// smaller (32 equal layers, beta = 0: 1.7e-6 -> 1.2e-6 rms).
constexpr int kPhaseCopies = 16;
constexpr int kPhaseMaxEntries = 112;
constexpr int kPhaseTabEntries = kPhaseMaxEntries * kPhaseCopies;

struct PhaseDigits {
  int mode;
  int fmin;
  int shift;
  int nd;     // 2 or 3 digits; mode 1: float32 costs of ordinary size (1) or any (0)
  int real;   // mode 1: float32 costs
  int last;   // entries of the last table - 1 (its index is clamped to this)
  int nent;   // entries in use
  float g_hi, g_lo;
  float2 d[kPhaseMaxEntries];
};

struct alignas(64) TmaFwdParams {
  CUtensorMap map_psi;   // state, 8-byte elements, 128-byte swizzle (loads)
  CUtensorMap map_cost;  // cost vector, 4-byte elements
  float2 *psi;           // the state (finished tiles are stored from registers)
  uint64_t ntiles;
  int h, c, cost_kind;  // tile = 2^c contiguous amplitudes x rows at qubits h..
  int mid2;             // the outer bits c..h-1 are view dimension 2 (else 1), see make_tile_map
  int comp;             // complement pair: the index bits m of the half vector, else 0
  Sweep s1, s2;
  float tau1, tau2;
  int form1, form2;
  float2 scl_end;
  int end_scale;
  int has_phase, init_plus, reduce;
  int twist_in;  // first pass on a caller's state: into the twisted basis
  int untwist;   // last pass (with end_scale): back to the standard basis
  uint64_t mirror;   // with untwist, nonzero (2^n - 1): amplitude x is also stored at its complement
  double out_scale;  // E and O times this (2 where half of the amplitudes are held)
  float amp;
  uint32_t fmin_word;  // f_min as the cost vector stores it (int32 or float32 bits)
  double *partials;
  unsigned *counter;
  double *out;
  unsigned *err;
  PhaseDigits ph;
};

struct alignas(64) TmaBwdParams {
  CUtensorMap map_psi, map_lam, map_cost;  // loads
  float2 *psi, *lam;                       // stores, from registers
  uint64_t ntiles;
  int h, c, cost_kind;
  int mid2, comp;     // as in TmaFwdParams
  Sweep s1, s2;
  float tau1, tau2;
  int form1, form2;
  float w1[4], w2[4]; // |scale|^2 weights of the inner products taken in each round
  float wg;           // |scale|^2 weight of the d/d gamma inner product
  int has_phase, init_lambda;
  const double *energy;  // E of the forward sweep or NULL (cost_shift)
  int untwist;  // last pass: psi back to the standard basis, lambda not stored
  uint64_t mirror;   // with untwist, nonzero (2^n - 1): psi[x] is also stored at its complement
  double out_scale;  // inner products times this before they are added
  // HIGH group of 9 new qubits (c = 4) on a 2^13-amplitude tile: 1 = cluster
  // pair, two CTAs holding its two halves (k_bwd_pair; map_cost is then the
  // pair cost map of the phase layout for passes with a phase); 2 = one
  // 512-thread CTA (k_bwd_tma with PlanTmaB13High); 0 = neither
  int cluster;
  double *partials;
  unsigned *counter;
  double *out_b1, *out_g, *out_b2;
  unsigned *err;
  PhaseDigits ph;
};

// The tile view whose outer bits c..h-1 are dimension 2 (else dimension 1): segments
// of 32 amplitudes and more, and tiles of fewer than 256 rows.
constexpr bool tile_map_mid2(int tb, int c) { return c >= 5 || tb - c < 8; }
cudaError_t make_tile_map(CUtensorMap *map, void *base, int n, int tb, int h, int c, int esz,
                          int swizzle_bytes);
// Cost tile of one CTA of a pair in the phase layout: 16 contiguous elements
// x qubits h..h+3 and h+5..h+8, qubit h+4 fixed by the box coordinate.
cudaError_t make_pair_cost_map(CUtensorMap *map, void *base, int n, int h, int esz);
// TMA passes over 4-byte (int32 / float32) and 2-byte (uint16) cost vectors.
cudaError_t launch_fwd_tma(const TmaFwdParams &P, bool high, cudaStream_t s, int nsm);
// one bounded device-side wait that nothing completes (sets *err after ~1 s)
cudaError_t launch_wait_selftest(unsigned *err, cudaStream_t s);
cudaError_t launch_bwd_tma(const TmaBwdParams &P, bool high, cudaStream_t s, int nsm);
cudaError_t launch_fwd_tma_u16(const TmaFwdParams &P, bool high, cudaStream_t s, int nsm);
cudaError_t launch_bwd_tma_u16(const TmaBwdParams &P, bool high, cudaStream_t s, int nsm);

// ---- XY ring mixer passes streamed by TMA (complex64).  A ring layer is the
// ordered chain of gates (q, q + 1), then (n - 1, 0).  Tiles of 2^13
// amplitudes; a round holds 5 consecutive tile bits in registers and applies
// the chain's gates among them in order, consecutive rounds sharing one bit:
//   LOW pass (qubits 0..12):  rounds over tile bits 0-4, 4-8, 8-12;
//   HIGH pass (16 contiguous amplitudes x rows h..h+8 at tile bits 4..12):
//                             rounds over tile bits 4-8, 8-12.
// em[r] bit i: apply the gate on the round's register bits (i, i + 1).  wrap:
// after the last round, the gate (tile bit 12, tile bit 0) = (n - 1, 0), tile
// bit 0 being lane bit 0 there (a shuffle).
using PlanXyLow = Plan<13, 5, 256, 0, 3, 0x001F, 0x03E0, 0x1C00, 0x01F0, 0x020F, 0x1C00,
                       0x1F00, 0x001F, 0x00E0>;
using PlanXyHigh = Plan<13, 5, 256, 0, 2, 0x01F0, 0x020F, 0x1C00, 0x1F00, 0x001F, 0x00E0>;
static_assert(PlanXyLow::valid_round(0) && PlanXyLow::valid_round(1) && PlanXyLow::valid_round(2) &&
                  PlanXyHigh::valid_round(0) && PlanXyHigh::valid_round(1),
              "bad XY plans");

struct alignas(64) XyTmaParams {
  CUtensorMap map_psi, map_cost;
  float2 *psi;
  uint64_t ntiles;
  int h, c, cost_kind;
  int has_phase;       // the layer's phase before the gates (LOW pass)
  uint32_t em[3];      // gate masks per round
  int wrap;            // the gate (n - 1, 0) after the last round
  float t, s;          // tan(b/2), sin(b) of the layer's beta reduced to |b| <= pi/2
  int neg;             // the reduction took out a factor -1
  unsigned *err;
  PhaseDigits ph;
};
cudaError_t launch_xy_tma(const XyTmaParams &P, bool low, cudaStream_t s, int nsm);
cudaError_t launch_xy_tma_u16(const XyTmaParams &P, bool low, cudaStream_t s, int nsm);

// One XY-mixer pass over tiles of 2^tb amplitudes: qubits 0..c-1 (contiguous),
// h1..h1+w1-1 and h2..h2+w2-1, in rounds: round k holds the four tile bits of
// rounds[k].bit (ascending) in registers and applies, for each set bit of its mask,
// the gate on register bits xy_gate_a, xy_gate_b, in that (lexicographic) order.
constexpr int kXyMaxTb = 12;
constexpr int kXyMaxRounds = 32;
// register bits of gate g: (0,1) (0,2) (0,3) (1,2) (1,3) (2,3)
__host__ __device__ constexpr int xy_gate_a(int g) { return g < 3 ? 0 : g < 5 ? 1 : 2; }
__host__ __device__ constexpr int xy_gate_b(int g) { return g < 3 ? g + 1 : g < 5 ? g - 1 : 3; }
struct XyRound {
  uint8_t bit[4];
  uint8_t mask;
};
struct XyPass {
  void *psi;
  const void *cost;
  uint64_t ntiles;
  int tb, c, h1, w1, h2, w2;
  int cost_kind, has_phase;  // phase exp(-i g f) applied while loading
  float g_hi, g_lo;          // complex64: g / 2pi = g_hi + g_lo
  double g2pi;               // complex128: g / 2pi
  double tb2, sb;            // tan(b/2), sin(b) of the layer's beta reduced to |b| <= pi/2
  int neg;                   // the reduction took out a factor -1
  int nrounds;
  int single;  // a gate at a time in shared memory (xy_single)
  XyRound rounds[kXyMaxRounds];
  PhaseDigits ph;  // complex64 integer costs: digit tables (mode 0), else computed
};

cudaError_t launch_xy_tile(const XyPass &P, bool c128, cudaStream_t s, int nsm);
cudaError_t launch_dicke(void *psi, bool c128, int n, int k, double amp, cudaStream_t s, int nsm);

// The phase tables of a job (entries, ndig, shift, fmin) from its cost type and
// statistics.  Computing a phase takes about as long as 10 of the products that
// two tables add per amplitude: the cheapest of computing all N, one table and two.
template <typename Real>
void small_digits(SmallJob<Real> &J, double f_min, double f_max, unsigned step_log2) {
  J.entries = J.ndig = 0;
  const int d = small_dims(J.n, J.half);
  // one warp with fewer threads at work than it has lanes: they compute the phases for each other
  J.by_x = 1 << (d - SmallTile<Real>::eb(d)) < 32;
  if (J.by_x) {
    J.entries = 1 << d;
    return;
  }
  if (J.cost_kind != kCostI32 && J.cost_kind != kCostU16) return;
  const int shift = step_log2 < 31u ? (int)step_log2 : 0;
  const double top = std::floor((f_max - f_min) / std::ldexp(1.0, shift));  // the largest d
  if (!(top >= 0.0 && top < 8192.0 && f_min >= -2147483648.0 && f_max <= 2147483647.0)) return;
  const int N = 1 << d, one = (int)top + 1, hi = (int)top / 64 + 1;
  const int t1 = 10 * one, t2 = 10 * (64 + hi) + N, most = kSmallTableBytes / (2 * (int)sizeof(Real));
  if (t1 <= t2 && t1 < 10 * N && one <= most) {
    J.entries = one;
  } else if (t2 < 10 * N && 64 + hi <= most) {
    J.entries = 64 + hi;
    J.ndig = hi;
  }
  J.shift = shift;
  J.fmin = (int)f_min;
}
// count jobs on d index bits (small_dims) each, of max_nl layers at most
cudaError_t launch_small_batch(const SmallJob<float> *d_jobs, int count, int d, int max_nl, cudaStream_t s);
cudaError_t launch_small(const SmallJob<float> &J, const SmallLayer<float> *layers, cudaStream_t s);
cudaError_t launch_small(const SmallJob<double> &J, const SmallLayer<double> *layers, cudaStream_t s);

// The factor sigma = 1 / sqrt(1 + t^2) of a rotation by tan t, |t| <= 1, and its powers
// as pairs of doubles.  A layer applies sigma once per qubit: in single doubles its
// three roundings, all of one sign over the layer, cost complex128 states twice the norm
// error of sigma = cos(beta) (n = 23, p = 4: 5.5e-15 against 2.6e-15); as pairs a power
// is rounded once.
struct SigmaPair {
  double hi, lo;
};
inline SigmaPair sigma_pair(double t, double sign) {
  const double s = 1.0 / std::sqrt(1.0 + t * t);
  const double u = s * s, ue = std::fma(s, s, -u), v = t * t, ve = std::fma(t, t, -v);
  // r = 1 - s^2 (1 + t^2); 1 - u is exact (u in [1/2, 1])
  const double r = std::fma(-u, v, 1.0 - u) - (ue + ue * v + u * ve);
  return SigmaPair{std::copysign(s, sign), std::copysign(s, sign) * (0.5 * r)};
}
inline SigmaPair sigma_mul(SigmaPair a, SigmaPair b) {
  const double p = a.hi * b.hi;
  const double e = std::fma(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi);
  const double h = p + e;
  return SigmaPair{h, e - (h - p)};
}
inline double sigma_pow(SigmaPair s, int k) {
  SigmaPair r{1.0, 0.0};
  for (; k > 0; k >>= 1, s = sigma_mul(s, s))
    if (k & 1) r = sigma_mul(r, s);
  return r.hi + r.lo;
}

// gamma / 2 pi as a pair of Reals.  Rounded to one double it was most of the error of a
// shallow complex128 circuit: gradients against long double, geometric means over ten
// angle sets, weighted MaxCut n = 14 p = 2 1.1e-15 -> 7.9e-16 of the norm, LABS n = 12
// p = 4 3.0e-15 -> 7.5e-16 (cosines of the unreduced product and the cosine as a rotation's
// factor: 2.1e-15 and 4.0e-15).
template <typename Real>
void turns_pair(double gamma, Real &hi, Real &lo) {
  const double inv_hi = 0x1.45f306dc9c883p-3, inv_lo = -0x1.6b01ec5417056p-57;  // 1 / (2 pi)
  const double h = gamma * inv_hi, l = std::fma(gamma, inv_hi, -h) + gamma * inv_lo;
  hi = (Real)h;
  lo = sizeof(Real) == 8 ? (Real)l : (Real)((h - (double)hi) + l);
}

// The layer data of angles (gamma, beta) for n qubits.  A server batch of long requests is
// bound by this (512 requests of n = 8 p = 100: 24 ms, with 27 powers of sigma and loops
// over mask bits, 17.4 ms now).
template <typename Real>
SmallLayer<Real> small_layer(double gamma, double beta, int n, int half) {
  SmallLayer<Real> L = {};
  const double c = std::cos(beta), s = std::sin(beta);
  L.form = std::fabs(c) >= std::fabs(s) ? 0 : 1;
  L.tau = (Real)(L.form ? c / s : s / c);
  // the factor of one rotation by the rounded tau (unitary); the adjoint's is its negative in form 1
  const double t = (double)L.tau;
  double pw[kSmallMaxN + 2];  // sigma^(2 i); pairs where the results are doubles
  if constexpr (sizeof(Real) == 8) {
    const SigmaPair sigma = sigma_pair(t, L.form ? s : c), sq = sigma_mul(sigma, sigma);
    SigmaPair run{1.0, 0.0};
    for (int i = 0; i <= n; ++i, run = sigma_mul(run, sq)) pw[i] = run.hi + run.lo;
    L.sig = (Real)sigma_pow(sigma, n);
  } else {
    const double sigma = std::copysign(1.0 / std::sqrt(1.0 + t * t), L.form ? s : c), sq = sigma * sigma;
    pw[0] = 1.0;
    for (int i = 1; i <= n; ++i) pw[i] = pw[i - 1] * sq;
    L.sig = (Real)(pw[n / 2] * ((n & 1) ? sigma : 1.0));
  }
  L.sig_adj = L.form && (n & 1) ? -L.sig : L.sig;
  L.wg = (Real)pw[n];
  using T = SmallTile<Real>;
  const int d = small_dims(n, half), R = T::rounds(d);
  for (int up = 0; up < 2; ++up) {
    int done = 0;
    for (int i = 0; i < T::kMaxRounds; ++i) {
      L.w[up][i] = (Real)pw[done];
      if (i < R) done += T::rotated(d, up ? i : R - 1 - i);
      if (i == 0) {
        L.w_comp[up] = (Real)pw[done];
        done += half;
      }
    }
  }
  turns_pair(gamma, L.g_hi, L.g_lo);
  return L;
}

}  // namespace qaoa
