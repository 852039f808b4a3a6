// kc_pair.cuh -- the mixed path's evaluation of two observations at a time
// in packed single precision (fma / add / mul .f32x2).
//
// What bounds the mixed kernels is FP32 issue and the register file's read
// ports.  On a GB300 a packed instruction takes the FMA pipe as long as two
// scalar ones but one issue slot (measured, clocks per warp and SM
// sub-partition: FFMA 1.04, FFMA2 2.06; with three different registers, or
// pairs, as operands 1.51 and 3.11), so a packed body leaves slots to the
// MUFU, integer and shared-memory work: the same body ran the 2^20-system
// sweep in 2067 us packed and 2221 scalar.  The body itself is cut to about
// 45 FMA-pipe operations, 40 clocks of MUFU and one shared-memory gather per
// planet-observation evaluation (before: 68 operations, 44 clocks): 68
// clocks per warp and sub-partition in steady state, 104 before.
//
//  - mean anomaly, 8 operations instead of 13: the observation times and
//    1/P are split at fixed binary places (2^-6 d and 2^-17 cycles/d), so
//    that their product is a multiple of 2^-23 cycles and its difference
//    from the nearest integer of the phase is exact in one FMA;
//  - Mikkola's cubic start with its quintic correction replaced by a
//    degree-four fit (below): within 8e-4 rad of the root (1.37e-3 just past
//    pi) instead of 3.6e-3, which lets one Newton step (4 operations) stand
//    for Halley's (9);
//  - sin/cos of the start from a table at multiples of 2^-8 rad in shared
//    memory and a rotation by the remainder (8 operations instead of 15);
//  - the velocity as (A cos E - B sin E)/(1 - e cos E) with its last product
//    inside the first operation of the compensated planet sum.
// The whole solve runs on |M| (E is odd in M), with M's sign put back on
// sin E.
//
// Accuracy, a float emulation of both forms over 2^20 draws each (P in 1 ..
// 4000 d, 4000 d of observations; errors of M in rad, of v in units of K,
// rms): M 6.9e-8 (scalar form 9.8e-8), v 7.9e-8 for e < 0.3 (9.1e-8),
// 6.6e-8 for e in 0.3 .. 0.8 (8.2e-8), 5.9e-8 for 0.8 .. 0.95 (8.6e-8),
// 7.3e-8 for 0.95 .. 0.99 (1.0e-7), 1.3e-7 for 0.99 .. 0.999 (1.4e-7).
#pragma once

#include "kc_device.cuh"

namespace kc {

// ------------------------------------------------ packed arithmetic

typedef unsigned long long f32x2;      // two floats, the first in the low half

__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f32x2 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ float lo2(f32x2 a) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
  return x;
}
__device__ __forceinline__ float hi2(f32x2 a) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
  return y;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return pack2(-lo2(a), -hi2(a)); }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return add2(a, neg2(b)); }
__device__ __forceinline__ f32x2 rcp2(f32x2 a) {
  return pack2(rcp_fast(lo2(a)), rcp_fast(hi2(a)));
}

// Two compensated sums side by side (Kahan, as in kc_device.cuh).
struct Kahan2 {
  f32x2 big, small;
};

// k += x where y = x - k.small is already formed (its subtraction can ride
// in the FMA that produces x).
__device__ __forceinline__ void kahan_add_y(Kahan2 &k, f32x2 y) {
  const f32x2 t = add2(k.big, y);
  k.small = sub2(sub2(t, k.big), y);
  k.big = t;
}
__device__ __forceinline__ void kahan_add(Kahan2 &k, f32x2 x) { kahan_add_y(k, sub2(x, k.small)); }

// The two sums of a pair as one.
__device__ __forceinline__ Kahan kahan_join(const Kahan2 &k) {
  Kahan a = {lo2(k.big), lo2(k.small)};
  const Kahan b = {hi2(k.big), hi2(k.small)};
  kahan_merge(a, b);
  return a;
}

// ------------------------------------------------ sin/cos table

// sin and cos at k 2^-8 rad, k = 0 .. 1023, rounded to float: 8 KB.  The start
// of the solve lies in [0, 1.04 pi], below 3.3.  A power of two of entries,
// so that the index of any start (NaN included, for an invalid planet) is
// masked into the table.  Two arrays, not (sin, cos) words: two 4-byte
// gathers land in the halves of the packed registers, where one 8-byte
// gather per observation needed moves (1995 us against 2067 on the sweep).
constexpr int kAngTabN = 1024;
constexpr float kAngRound = 49152.0f;              // 1.5 * 2^15: rounds to 2^-8

struct AngTab {
  float s[kAngTabN], c[kAngTabN];
};

// Taylor series about 0 in double: below 2e-15 absolute for x < 4.
constexpr double ang_series(double x, bool cosine) {
  double term = cosine ? 1.0 : x, sum = 0.0;
  for (int n = cosine ? 0 : 1; n < 50; n += 2) {
    sum += term;
    term *= -x * x / ((n + 1.0) * (n + 2.0));
  }
  return sum;
}
// vers: 1 - cos in place of cos (= 2 sin^2 of half the angle).
constexpr AngTab make_ang_tab(bool vers) {
  AngTab t{};
  for (int k = 0; k < kAngTabN; ++k) {
    const double h = ang_series(k / 512.0, false);
    t.s[k] = (float)ang_series(k / 256.0, false);
    t.c[k] = vers ? (float)(2.0 * h * h) : (float)ang_series(k / 256.0, true);
  }
  return t;
}
static __device__ const __align__(16) AngTab kAngTab = make_ang_tab(false);
static __device__ const __align__(16) AngTab kAngTabV = make_ang_tab(true);

// The CTA's copy in shared memory (16-byte copies; a barrier must follow).
// VERS: the form kepler_pair<true> takes.
template <bool VERS>
__device__ __forceinline__ void ang_tab_load(float *tab, int tid, int nthreads) {
  const float4 *src = reinterpret_cast<const float4 *>(VERS ? &kAngTabV : &kAngTab);
  for (int i = tid; i < kAngTabN / 2; i += nthreads) reinterpret_cast<float4 *>(tab)[i] = src[i];
}

// ------------------------------------------------ observation times

// tau = th + tl with th a multiple of 2^-6 d (or tau_hi itself from 2^17 d
// on, whose last place is no finer) and |tl| <= 2^-7 d, rounded to 2^-32 d and
// finer (err: what it lost).
constexpr float kTauPlace = 64.0f;
__device__ __forceinline__ void tau_place(float &hi, float &lo, float &err) {
  const float th = fabsf(hi) < 131072.0f ? rintf(hi * kTauPlace) * (1.0f / kTauPlace) : hi;
  two_sum(__fsub_rn(hi, th), lo, lo, err);
  hi = th;
}
__device__ __forceinline__ void tau_place(float &hi, float &lo) {
  const float th = fabsf(hi) < 131072.0f ? rintf(hi * kTauPlace) * (1.0f / kTauPlace) : hi;
  lo = __fadd_rn(__fsub_rn(hi, th), lo);
  hi = th;
}

// Limits of the short form of the mean anomaly (mean_anomaly_pair): 1/P up
// to 2 cycles/d, |tau| below 2^14 d (45 years).  Beyond them the wide form
// runs, and what the binary places would lose is kept:
//  - a time beyond the limit: every time stays the plain pair (tau_hi, tau_lo),
//    and every 1/P (n_hi, n_lo) (planet_plain).  Placed, 1/P is known to 2^-42
//    cycles/d: 4.5e-7 rad (rms) in M at P = 3000 d and 1e6 d, 2e-4 where times
//    and periods are given in seconds;
//  - 1/P above the limit: that planet keeps the plain pair;
//  - 1/P above kPairExactFreq: the system's times are read as plain pairs.
//    Placed, they are known to 2^-33 d: 6.5e-7 rad at P = 1e-3 d (6e-9 at the
//    limit).
// So M is within 2.1e-7 rad (4e-8 to 8e-8 rms) wherever |tau/P| < 2^22.
constexpr float kPairMaxFreq = 2.0f;
constexpr float kPairExactFreq = 16.0f;
constexpr float kPairMaxTau = 16384.0f;

__device__ __forceinline__ bool far_time(float th) { return !(fabsf(th) < kPairMaxTau); }

// Whether one of the thread's times from the first-th on is a far one (out of line:
// few batches have more than one tile).
static __device__ __noinline__ bool far_later(const double *t, int first, int n_obs) {
  const double t_ref = t[0];
  bool far = false;
#pragma unroll 4
  for (int k = first + threadIdx.x; k < n_obs; k += blockDim.x)
    far |= !(fabs(t[k] - t_ref) < (double)kPairMaxTau);
  return far;
}

// Observations k and k + 1 of t (n of them; the padding has tau = 0) as plain
// pairs, for the rare systems of the last case: one FP64 subtraction each, on a pipe
// that is idle otherwise (65536 x 4 x 256 with P in 0.001 .. 0.01 d: 188 us; the
// float expansions of the staging, 100 instructions, took 239).
__device__ __forceinline__ void plain_times(const double *t, int k, int n, f32x2 &th,
                                            f32x2 &tl) {
  const double t_ref = t[0];
  float ah, al, bh, bl;
  split_d(k < n ? t[k] - t_ref : 0.0, ah, al);
  split_d(k + 1 < n ? t[k + 1] - t_ref : 0.0, bh, bl);
  th = pack2(ah, bh);
  tl = pack2(al, bl);
}

// ------------------------------------------------ per-planet constants

// The start.  With a = (1 - e)/(4 e + 1/2), the real root of Mikkola's
// cubic s^3 + 3 a s = M/(4 e + 1/2) is s = sqrt(a) (z - 1/z), z = (b +
// sqrt(b^2 + 1))^(1/3), b = M bs, bs = 1/((8 e + 1) a^(3/2)); s is close to
// sin(E/3), and sin E = 3 s - 4 s^3 there.  Instead of correcting s (his
// -0.078 s^5/(1 + e)), sin E is taken as s (3 + c1 x + c2 x^2 + c3 x^3 +
// c4 x^4), x = s^2, with c1 .. c4 cubics in e fitted to keep the error of
// ONE NEWTON STEP small (weighted least squares with the weights iterated
// towards the largest error, kepler_start_fit.py, which fits up to |M| = 1.02 pi
// and checks beyond).  For every 0 <= e < 1, in exact arithmetic: for |M| <= pi
// the start is within 8e-4 rad and the step within 5.1e-9 rad of the root (as
// Halley's step from the quintic correction), up to 1.02 pi within 1.06e-3 and
// 5.1e-9, up to 1.038 pi, where the short mean anomaly ends, within 1.37e-3 and
// 1.7e-8.  Scaled to s' = z - 1/z: E0 = M + s' (q0 + q1 x' + .. + q4 x'^4), q_i = e c_i
// a^(i + 1/2).
__device__ __forceinline__ float start_fit(float e, float k0, float k1, float k2, float k3) {
  return __fmaf_rn(e, __fmaf_rn(e, __fmaf_rn(e, k3, k2), k1), k0);
}

struct StartP {
  float bs, q[5];
};

// a = (1 - e)/(4 e + 1/2), sa = sqrt(a) and bs are given.
__device__ __forceinline__ StartP start_from(float e, float a, float sa, float bs) {
  StartP p;
  p.bs = bs;
  float f = e * sa;
  p.q[0] = 3.0f * f;
  f *= a;
  p.q[1] = f * start_fit(e, -3.9074f, -0.4550f, 0.5740f, -0.2644f);
  f *= a;
  p.q[2] = f * start_fit(e, -0.8507f, 3.2176f, -3.9800f, 1.8248f);
  f *= a;
  p.q[3] = f * start_fit(e, 2.1773f, -6.5683f, 8.0450f, -3.7069f);
  f *= a;
  p.q[4] = f * start_fit(e, -0.8390f, 3.4927f, -4.6815f, 2.2459f);
  return p;
}

__device__ __forceinline__ StartP start_constants(float e) {
  const float r = 1.0f / __fmaf_rn(4.0f, e, 0.5f);
  const float a = fmaxf((1.0f - e) * r, 1e-8f);      // e rounded up to 1: finite
  const float sa = sqrtf(a);
  return start_from(e, a, sa, 0.5f * r / (a * sa));
}

// The same for one evaluation (every (M, e) of the Kepler-only solver has its
// own e): approximate reciprocals; e up to kEccFast.
__device__ __forceinline__ StartP start_constants_fast(float e) {
  const float r = rcp_fast(__fmaf_rn(4.0f, e, 0.5f)), a = (1.0f - e) * r, is = rsqrt_fast(a);
  return start_from(e, a, a * is, 0.5f * r * (is * is * is));
}

// Phase: n = 1/P rounded; nq its multiple of 2^-17 (n itself in a plain pair),
// nlo the rest; c a multiple of 2^-23, clo the rest, both low parts and n2pi
// times 2 pi.  Start: st, above.
// Velocity: v = (A cos E - B sin E)/(1 - e cos E), A = K cos w (1 - e^2),
// B = K sqrt(1 - e^2) sin w.
struct __align__(16) PlanetP {
  float n, nq, c, nlo2pi;
  float clo2pi, n2pi, e;
  StartP st;
  float A, B, ome;           // ome = 1 - e (gradient only)
};

// What planet_setup_pair derives besides the phase and the start: sin and cos
// of w, b2 = 1 - e^2 (one rounding) and b = sqrt(b2).
struct OrbitF {
  float sw, cw, b2, b;
};

// x y z with the product x y's remainder and x's low part carried (x, y, z
// rounded once each, the result once more).
__device__ __forceinline__ float product3(float x_hi, float x_lo, float y, float z) {
  float u, ue;
  two_prod(x_hi, y, u, ue);
  return __fmaf_rn(u, z, __fmaf_rn(x_lo, y, ue) * z);
}

// Whether a planet's period is too short for the short form.
__device__ __forceinline__ bool short_period(const PlanetP &q) { return !(q.n <= kPairMaxFreq); }

// Phase, start and orbit constants of one planet; the caller sets A and B.
// An invalid planet gets e = NaN, which makes its velocities NaN.  plain: 1/P
// as a plain pair whatever its size.
__device__ __forceinline__ PlanetP planet_setup_orbit(const double *p, double t_ref, double t0,
                                                      bool plain, OrbitF &o) {
  PlanetP q;
  float n_hi, n_lo, c_hi, c_lo;
  phase_setup_ds(p[0], p[4], t_ref, t0, n_hi, n_lo, c_hi, c_lo);
  constexpr float kPlaceN = 131072.0f, kPlaceC = 8388608.0f;          // 2^17, 2^23
  q.n = n_hi;
  q.nq = n_hi <= kPairMaxFreq && !plain ? rintf(n_hi * kPlaceN) * (1.0f / kPlaceN) : n_hi;
  q.nlo2pi = __fadd_rn(__fsub_rn(n_hi, q.nq), n_lo) * kTwoPiF;
  q.c = rintf(c_hi * kPlaceC) * (1.0f / kPlaceC);
  q.clo2pi = __fadd_rn(__fsub_rn(c_hi, q.c), c_lo) * kTwoPiF;
  q.n2pi = n_hi * kTwoPiF;
  const float ef = d2f(p[2]);
  q.e = planet_valid(p[0], p[1], p[2], p[3], p[4]) ? ef : __int_as_float(0x7fc00000);
  q.st = start_constants(q.e);
  float w_hi, w_lo;
  split_d(p[3], w_hi, w_lo);
  float sw, cw;
  sincosf(w_hi, &sw, &cw);
  o.sw = __fmaf_rn(w_lo, cw, sw);
  o.cw = __fmaf_rn(-w_lo, sw, cw);
  o.b2 = __fmaf_rn(-ef, ef, 1.0f);
  o.b = sqrtf(o.b2);
  q.ome = 0.0f;
  return q;
}

__device__ __forceinline__ PlanetP planet_setup_pair(const double *p, double t_ref, double t0,
                                                     bool plain) {
  OrbitF o;
  PlanetP q = planet_setup_orbit(p, t_ref, t0, plain, o);
  float K_hi, K_lo;
  split_d(p[1], K_hi, K_lo);
  q.A = product3(K_hi, K_lo, o.cw, o.b2);
  q.B = product3(K_hi, K_lo, o.sw, o.b);
  return q;
}

// 1/P of a planet that is set up, made a plain pair (a far time is known only
// after the setup).
__device__ __forceinline__ void planet_plain(PlanetP &q, double P) {
  float n_lo;
  frequency_ds(P, q.nq, n_lo);
  q.nlo2pi = n_lo * kTwoPiF;
}

// The gradient's planet: A and B of the solve without K, and the constants
// of the partials (grad_terms).
struct __align__(16) GradPlanetP {
  PlanetP p;
  float K, C, sw, esw, cw, beta, ibeta, swo;     // C = beta cos w, esw = e sin w, swo = (1 - e) sin w
};

__device__ __forceinline__ GradPlanetP grad_setup_pair(const double *p, double t_ref, double t0,
                                                       bool plain) {
  GradPlanetP g;
  OrbitF o;
  g.p = planet_setup_orbit(p, t_ref, t0, plain, o);
  float e_hi, e_lo;
  split_d(p[2], e_hi, e_lo);
  g.p.ome = __fsub_rn(__fsub_rn(1.0f, e_hi), e_lo);
  o.b2 = g.p.ome * (1.0f + g.p.e);
  o.b = sqrtf(o.b2);
  g.p.A = o.cw * o.b2;
  g.p.B = o.sw * o.b;
  g.K = d2f(p[1]);
  g.C = o.cw * o.b;
  g.sw = o.sw;
  g.cw = o.cw;
  g.esw = g.p.e * o.sw;
  g.swo = o.sw * g.p.ome;
  g.beta = o.b;
  g.ibeta = 1.0f / o.b;
  return g;
}

// ------------------------------------------------ mean anomaly

// M of two observations, |M| < 1.038 pi.  k is the integer nearest to the phase
// without tl n, up to 2^-6 cycles (1/P = 2, |tl| = 2^-7 d), without 1/P's low part,
// up to 2^-10, and rounded to float, up to 2^-9 (both at |tau/P| = 2^15): |phase -
// k| < 0.519 cycles; th nq is a multiple of 2^-23 and its distance from k below
// 2, so the FMA is exact, and so is the sum with c.  The low parts (below 0.1
// cycles) add three roundings near 2^-26 rad and the final FMA one: 2.1e-7 rad
// at worst, 6.9e-8 rms.
__device__ __forceinline__ f32x2 mean_anomaly_pair(f32x2 th, f32x2 tl, const PlanetP &q) {
  const f32x2 magic = dup2(kRoundMagic);
  const f32x2 y = fma2(th, dup2(q.n), dup2(q.c));
  const f32x2 k = sub2(add2(y, magic), magic);
  const f32x2 u = add2(fma2(th, dup2(q.nq), neg2(k)), dup2(q.c));
  const f32x2 lo = fma2(tl, dup2(q.n2pi), fma2(th, dup2(q.nlo2pi), dup2(q.clo2pi)));
  return fma2(u, dup2(kTwoPiF), lo);
}

__device__ __forceinline__ f32x2 round2(f32x2 x) {
  return sub2(add2(x, dup2(kRoundMagic)), dup2(kRoundMagic));
}

// M at any period and time the double-single phase covers (|tau/P| < 2^22): tau
// as the float pair of its leading 48 bits, the product's FMA remainder and the
// sum's TwoSum remainder kept, every part wrapped before the last sum, 2 pi with
// its own low part.  |M| <= 1.0001 pi.
__device__ __forceinline__ f32x2 mean_anomaly_wide(f32x2 th, f32x2 tl, const PlanetP &q) {
  const f32x2 hi = add2(th, tl), lo = sub2(tl, sub2(hi, th));
  const f32x2 n = dup2(q.nq), p = mul2(hi, n), pe = fma2(hi, n, neg2(p));
  f32x2 lc = fma2(lo, dup2(q.n), pe);
  lc = fma2(fma2(hi, dup2(q.nlo2pi), dup2(q.clo2pi)), dup2((float)kInvTwoPi), lc);
  lc = sub2(lc, round2(lc));
  const f32x2 f = sub2(p, round2(p)), c = dup2(q.c);
  f32x2 u = add2(f, c);
  const f32x2 v = sub2(u, f);
  lc = add2(lc, add2(sub2(f, sub2(u, v)), sub2(c, v)));
  u = sub2(u, round2(u));
  u = sub2(u, round2(add2(u, lc)));
  constexpr float kTwoPiLo = (float)(kTwoPi - (double)kTwoPiF);
  return fma2(u, dup2(kTwoPiF), fma2(u, dup2(kTwoPiLo), mul2(lc, dup2(kTwoPiF))));
}

// The form of a wide body's lane: `brief` if its system takes the short form all
// the same, `some` and `all` (for the warp) if any lane's or every lane's does.  So
// a system's bits do not hang on the others of its warp, which run the rest of the
// solve together.
struct MeanForm {
  bool some = false, all = false, brief = false;
};

template <bool WIDE>
__device__ __forceinline__ f32x2 mean_anomaly2(f32x2 th, f32x2 tl, const PlanetP &q,
                                               MeanForm form = {}) {
  if (!WIDE) return mean_anomaly_pair(th, tl, q);
  f32x2 M = mean_anomaly_wide(th, tl, q);
  if (form.some) {
    const f32x2 m = mean_anomaly_pair(th, tl, q);
    M = form.brief ? m : M;
  }
  return M;
}

// ------------------------------------------------ Kepler's equation

// s' = z - 1/z of the start for one |M|.  1/z is the exponential of the
// negated logarithm: ex2 runs at twice the rate of rcp (4 clocks per warp
// against 8).
__device__ __forceinline__ float start_root(float b, float w) {
  const float l = lg2_fast(b + sqrt_fast(w)) * (1.0f / 3.0f);
  return ex2_fast(l) - ex2_fast(-l);
}

// Table index of the angle behind k = angle + kAngRound.
__device__ __forceinline__ unsigned ang_index(float k) {
  return __float_as_uint(k) & (kAngTabN - 1);
}

// Solves E - e sin E = |M| for two mean anomalies: sin E >= 0-signed as for
// |M| (s, without M's sign), cos E (c) and, for a residual, E.
// The table's angle a = E0 rounded to 2^-8 is exact in float, and so is b =
// E0 - a, |b| <= 2^-9: sin b = b and cos b = 1 - b^2/2 to 1.3e-9.
// VERS: from the table of 1 - cos, c is 1 - cos E and D = (1 - e) + e (1 - cos
// E), to full relative precision where e is high and E small: the partials take
// 1/D squared, and cos E rounded near 1 cost them up to 4e-6 there (ragged batches
// whose gradient norm one such system dominates: 1.6e-6 off, now 5.7e-7; the
// scalar form 4.6e-7; the geometric mean over 90 batches 0.81 of the scalar
// form's error).  Two packed additions more: 65536 x 3 x 512 260 us both, 20000 x
// 6 x 256 90 -> 94.
template <bool VERS>
__device__ __forceinline__ void kepler_pair(f32x2 m, const PlanetP &q, const float *tab, f32x2 &s,
                                            f32x2 &c, f32x2 &E) {
  const f32x2 b = mul2(m, dup2(q.st.bs));
  const f32x2 w = fma2(b, b, dup2(1.0f));
  const f32x2 r = pack2(start_root(lo2(b), lo2(w)), start_root(hi2(b), hi2(w)));
  const f32x2 x = mul2(r, r);
  f32x2 p = fma2(x, dup2(q.st.q[4]), dup2(q.st.q[3]));
  p = fma2(x, p, dup2(q.st.q[2]));
  p = fma2(x, p, dup2(q.st.q[1]));
  p = fma2(x, p, dup2(q.st.q[0]));
  const f32x2 E0 = fma2(r, p, m);
  // sin, cos of E0
  const f32x2 k = add2(E0, dup2(kAngRound));
  const f32x2 d0 = sub2(E0, sub2(k, dup2(kAngRound)));
  const unsigned i0 = ang_index(lo2(k)), i1 = ang_index(hi2(k));
  const f32x2 S = pack2(tab[i0], tab[i1]), T = pack2(tab[kAngTabN + i0], tab[kAngTabN + i1]);
  const f32x2 C = VERS ? sub2(dup2(1.0f), T) : T;
  const f32x2 h0 = mul2(d0, dup2(-0.5f));
  const f32x2 s0 = fma2(d0, fma2(h0, S, C), S);
  // Newton: d = (E0 - e sin E0 - m)/(1 - e cos E0), E = E0 - d
  const f32x2 ne = dup2(-q.e);
  const f32x2 f = fma2(ne, s0, sub2(E0, m));
  if constexpr (VERS) {
    const f32x2 v0 = fma2(d0, fma2(neg2(h0), C, S), T), c0 = sub2(dup2(1.0f), v0);
    const f32x2 d = mul2(f, rcp2(fma2(dup2(q.e), v0, dup2(q.ome))));
    const f32x2 h = mul2(d, dup2(-0.5f));
    s = fma2(d, neg2(fma2(neg2(h), s0, c0)), s0);
    c = fma2(d, neg2(fma2(h, c0, s0)), v0);
    E = sub2(E0, d);
  } else {
    const f32x2 c0 = fma2(d0, fma2(h0, C, neg2(S)), C);
    const f32x2 d = mul2(f, rcp2(fma2(ne, c0, dup2(1.0f))));
    const f32x2 h = mul2(d, dup2(-0.5f));
    s = fma2(d, neg2(fma2(neg2(h), s0, c0)), s0);
    c = fma2(d, fma2(h, c0, s0), c0);
    E = sub2(E0, d);
  }
}

// x with M's sign (x's own kept: an exclusive or).
__device__ __forceinline__ f32x2 signed_as(f32x2 x, f32x2 M) {
  const unsigned a = __float_as_uint(lo2(x)) ^ (__float_as_uint(lo2(M)) & 0x80000000u);
  const unsigned b = __float_as_uint(hi2(x)) ^ (__float_as_uint(hi2(M)) & 0x80000000u);
  return pack2(__uint_as_float(a), __uint_as_float(b));
}

__device__ __forceinline__ f32x2 abs2(f32x2 x) { return pack2(fabsf(lo2(x)), fabsf(hi2(x))); }

// V += v with sin E already signed.
__device__ __forceinline__ void velocity_sum(Kahan2 &V, const PlanetP &q, f32x2 s, f32x2 c) {
  const f32x2 D = fma2(dup2(-q.e), c, dup2(1.0f));
  const f32x2 num = fma2(dup2(q.A), c, neg2(mul2(dup2(q.B), s)));
  kahan_add_y(V, fma2(num, rcp2(D), neg2(V.small)));
}

// ------------------------------------------------ partials

// One planet of a pair of observations, for the gradient: with y = 1/D,
//   dK = v/K = (A cos E - B sin E) y,
//   Q  = sin(w + f) = (sin w cos E + C sin E - e sin w) y;
// the other partials follow (GradSums).  V takes K dK.
struct GradTerms {
  f32x2 s, dK, Q, y;
};

__device__ __forceinline__ GradTerms grad_terms_at(f32x2 M, const GradPlanetP &g,
                                                   const float *tab, Kahan2 &V) {
  GradTerms o;
  f32x2 s, c, E;
  kepler_pair<true>(abs2(M), g.p, tab, s, c, E);      // c = 1 - cos E
  o.s = signed_as(s, M);
  o.y = rcp2(fma2(dup2(g.p.e), c, dup2(g.p.ome)));
  o.dK = mul2(fma2(dup2(-g.p.A), c, fma2(dup2(-g.p.B), o.s, dup2(g.p.A))), o.y);
  o.Q = mul2(fma2(dup2(g.C), o.s, fma2(dup2(-g.sw), c, dup2(g.swo))), o.y);
  kahan_add_y(V, fma2(dup2(g.K), o.dK, neg2(V.small)));
  return o;
}

template <bool WIDE>
__device__ __forceinline__ GradTerms grad_terms(f32x2 th, f32x2 tl, const GradPlanetP &g,
                                                const float *tab, Kahan2 &V,
                                                MeanForm form = {}) {
  return grad_terms_at(mean_anomaly2<WIDE>(th, tl, g.p, form), g, tab, V);
}

// Sums over the observations, a = 2 w r: of a dt Q y^2 (compensated: the
// period's terms cancel heavily), a dK, a Q y sin E (1/beta + beta y), a Q, a
// Q y^2.  The partials by (P, K, e, w, M0) are
//   2 pi n^2 K beta dt Q y^2,  dK,  K cos w - K Q y sin E (1/beta + beta y),
//   -K (Q + e sin w),  -K beta Q y^2,
// so their factors, and the parts a alone multiplies, are applied once per
// system (grad_finish): 17 packed operations per pair and planet for all five
// where the partials formed one by one took about 40 scalar ones each.
struct GradSums {
  Kahan2 P;
  f32x2 K, e, w, M;
};

__device__ __forceinline__ void grad_add(GradSums &G, const GradTerms &o, const GradPlanetP &g,
                                         f32x2 a, f32x2 adt) {
  const f32x2 Qy = mul2(o.Q, o.y), Qyy = mul2(Qy, o.y);
  const f32x2 h = fma2(dup2(g.beta), o.y, dup2(g.ibeta));
  kahan_add_y(G.P, fma2(adt, Qyy, neg2(G.P.small)));
  G.K = fma2(a, o.dK, G.K);
  G.e = fma2(mul2(a, Qy), mul2(o.s, h), G.e);
  G.w = fma2(a, o.Q, G.w);
  G.M = fma2(a, Qyy, G.M);
}

// The same sums with the pair's two halves added one after the other: six
// registers a planet instead of twelve.  A packed multiply-add of three
// register pairs reads as many registers as two scalar ones, so it is no
// faster; from four planets on (where twelve registers a planet spill) the
// kernels sum this way.
struct GradSumsS {
  Kahan P;
  float K, e, w, M;
};

__device__ __forceinline__ void add_halves(float &sum, f32x2 a, f32x2 b) {
  sum = __fmaf_rn(hi2(a), hi2(b), __fmaf_rn(lo2(a), lo2(b), sum));
}

__device__ __forceinline__ void grad_add(GradSumsS &G, const GradTerms &o, const GradPlanetP &g,
                                         f32x2 a, f32x2 adt) {
  const f32x2 Qy = mul2(o.Q, o.y), Qyy = mul2(Qy, o.y);
  const f32x2 h = fma2(dup2(g.beta), o.y, dup2(g.ibeta));
  const f32x2 P = mul2(adt, Qyy);
  kahan_add(G.P, lo2(P));
  kahan_add(G.P, hi2(P));
  add_halves(G.K, a, o.dK);
  add_halves(G.e, mul2(a, Qy), mul2(o.s, h));
  add_halves(G.w, a, o.Q);
  add_halves(G.M, a, Qyy);
}

template <int J>
struct GradSumsFor {
  typedef GradSums type;
};
#define KC_SCALAR_SUMS(J)   \
  template <>               \
  struct GradSumsFor<J> {   \
    typedef GradSumsS type; \
  }
KC_SCALAR_SUMS(4);
KC_SCALAR_SUMS(5);
KC_SCALAR_SUMS(6);
KC_SCALAR_SUMS(7);
KC_SCALAR_SUMS(8);
#undef KC_SCALAR_SUMS

// The same planet's row of sqrt(w) J for the Gauss-Newton matrix, each column
// over its per-planet factor (gn_scale), and its gradient sums from the row
// with a = 2 sqrt(w) r; swdt = sqrt(w) (t - t0).
__device__ __forceinline__ void gn_add(GradSums &G, const GradTerms &o, const GradPlanetP &g,
                                       f32x2 sw, f32x2 swdt, f32x2 a, f32x2 *u) {
  const f32x2 Qy = mul2(o.Q, o.y), Qyy = mul2(Qy, o.y);
  const f32x2 h = fma2(dup2(g.beta), o.y, dup2(g.ibeta));
  u[0] = mul2(swdt, Qyy);
  u[1] = mul2(sw, o.dK);
  u[2] = mul2(sw, sub2(dup2(g.cw), mul2(Qy, mul2(o.s, h))));
  u[3] = mul2(sw, add2(o.Q, dup2(g.esw)));
  u[4] = mul2(sw, Qyy);
  kahan_add_y(G.P, fma2(a, u[0], neg2(G.P.small)));
  G.K = fma2(a, u[1], G.K);
  G.e = fma2(a, u[2], G.e);
  G.w = fma2(a, u[3], G.w);
  G.M = fma2(a, u[4], G.M);
}

// Factor of parameter p (0 .. 5 n_pl) of a system's rows: the columns are (dt
// Q y^2, dK, cos w - .., Q + e sin w, Q y^2) per planet, then 1.
__device__ __forceinline__ float gn_scale(const GradPlanetP *q, int J, int p) {
  const int j = p / 5, i = p - 5 * j;
  if (j >= J) return 1.0f;
  const GradPlanetP &g = q[j];
  const float Kb = g.K * g.beta;
  switch (i) {
    case 0: return Kb * (kTwoPiF * (g.p.n * g.p.n));
    case 1: return 1.0f;
    case 2: return g.K;
    case 3: return -g.K;
    default: return -Kb;
  }
}

__device__ __forceinline__ float join2(f32x2 x) { return lo2(x) + hi2(x); }

// A planet's five sums of one lane (the pair joined).
struct GradLane {
  Kahan P;
  float K, e, w, M;
};
__device__ __forceinline__ GradLane grad_join(const GradSums &G) {
  return GradLane{kahan_join(G.P), join2(G.K), join2(G.e), join2(G.w), join2(G.M)};
}
__device__ __forceinline__ GradLane grad_join(const GradSumsS &G) {
  return GradLane{G.P, G.K, G.e, G.w, G.M};
}
__device__ __forceinline__ void grad_combine(GradLane &g, int m) {
  const Kahan o = {shfl_xor(g.P.big, m), shfl_xor(g.P.small, m)};
  kahan_merge(g.P, o);
  g.K += shfl_xor(g.K, m);
  g.e += shfl_xor(g.e, m);
  g.w += shfl_xor(g.w, m);
  g.M += shfl_xor(g.M, m);
}
// The planet's gradient from the system's sums; sum_a = sum of a.
__device__ __forceinline__ void grad_finish(const GradLane &s, const GradPlanetP &g, float sum_a,
                                            float poison, float *out) {
  const float Kb = g.K * g.beta;
  out[0] = __fmaf_rn(Kb * (kTwoPiF * (g.p.n * g.p.n)), kahan_value(s.P), poison);
  out[1] = s.K + poison;
  out[2] = __fmaf_rn(g.K, __fmaf_rn(g.cw, sum_a, -s.e), poison);
  out[3] = __fmaf_rn(-g.K, __fmaf_rn(g.esw, sum_a, s.w), poison);
  out[4] = __fmaf_rn(-Kb, s.M, poison);
}

}  // namespace kc
