// kc_f64.cuh -- one planet-observation evaluation of the FP64 path, with the
// double-precision work that single-precision expansions can carry taken off
// the FP64 pipe.
//
// What bounds the FP64 kernels is that pipe: one FP64 instruction of a warp
// takes 64 clocks of a GB300 sub-partition (measured), an FP32 or integer
// instruction one to three.  The evaluation needs 53 bits in few places: the
// phase, f(E) = E - e sin E - M near its root, and the leading part of the
// velocity.  Everything else is a small correction to a tabulated value:
//
//  - the single-precision solve (kc_pair.cuh's start, one Newton step) gives
//    Ef within about 4e-7 of the root (|M| < 1.04 pi, solve_x); a, the multiple
//    of 2^-9 rad nearest to its start, has sin a and cos a in a table as doubles
//    and as float pairs;
//  - sin and cos of a + b (b = Ef - a exact in float, |b| < 1.8e-3 for |M| <= pi,
//    2.4e-3 just beyond) and of the corrected E differ from them by less than
//    3e-3, so a float pair (48 bits) holds the difference to 1e-17: rotation,
//    Newton's correction and the update run in float expansions (products with
//    their FMA remainders, sums by TwoSum);
//  - f(Ef) takes two FP64 FMAs, (Ef - 2 pi u) - e sin a, minus e times the
//    float-pair difference;
//  - v = N/D with N = A cos E - B sin E: N at the table's angle by two FP64
//    operations, times 1/D (a float pair assembled into a double on the
//    integer pipe) onto the planet sum, and the difference of N in float
//    pairs, summed compensated and added to V once per observation.
//
// FP64 instructions per evaluation: 7 (11 where 1/D is corrected, velocity_x),
// and 4 per observation (before: 33 and 3).  Error of v without that
// correction, in units of K, against 64-bit mantissas in an emulation (rms over
// 2.6e5 draws; P in 1 .. 4000 d, 4000 d of observations), with the form of one
// FP64 Halley step and one FP64 Newton step for 1/D in brackets: e < 0.3 1.5e-15
// (5.4e-15), 0.3 .. 0.8 1.8e-15 (4.4e-15), 0.8 .. 0.95 2.9e-15 (2.6e-15: hence the
// correction).  Valid for e <= kEccFast and amplitudes a float pair holds
// (amplitude_fits); a planet outside takes two FP64 quartic steps and an FP64
// velocity (PlanetX::high, eval_high), beside the others of its system.
#pragma once

#include "kc_device.cuh"
#include "kc_pair.cuh"

namespace kc {

// ------------------------------------------------ table

// sin and cos at k 2^-9 rad up to 1.057 pi, correctly rounded: the
// angle-addition recurrence in double-double from the Taylor series at 2^-9,
// evaluated by the compiler.
constexpr int kF64TabN = 1700;
constexpr float kF64Round = 24576.0f;              // 1.5 * 2^14: rounds to 2^-9

struct __align__(16) F64Tab {
  double sc[kF64TabN][2];       // sin, cos
  float f[kF64TabN][4];         // sin hi, lo, cos hi, lo
};

struct DD {
  double h, l;
};
constexpr DD dd_sum(double a, double b) {
  const double s = a + b, bv = s - a;
  return DD{s, (a - (s - bv)) + (b - bv)};
}
constexpr DD dd_prod(double a, double b) {          // Dekker's exact product
  const double p = a * b, t = 134217729.0 * a, ah = t - (t - a), al = a - ah;
  const double u = 134217729.0 * b, bh = u - (u - b), bl = b - bh;
  return DD{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD dd_mul(DD a, DD b) {
  const DD p = dd_prod(a.h, b.h);
  return dd_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD dd_add(DD a, DD b) {
  const DD s = dd_sum(a.h, b.h);
  return dd_sum(s.h, s.l + (a.l + b.l));
}
constexpr DD dd_inv(double a) {
  const double r = 1.0 / a;
  const DD e = dd_prod(a, r);
  return DD{r, ((1.0 - e.h) - e.l) / a};
}
constexpr F64Tab make_f64_tab() {
  F64Tab t{};
  const DD x{1.0 / 512.0, 0.0}, x2 = dd_mul(x, x), nx2{-x2.h, -x2.l};
  DD s = x, c{1.0, 0.0}, ps = x, pc{1.0, 0.0};
  for (int n = 1; n < 8; ++n) {
    ps = dd_mul(dd_mul(ps, nx2), dd_inv((2.0 * n) * (2.0 * n + 1.0)));
    pc = dd_mul(dd_mul(pc, nx2), dd_inv((2.0 * n - 1.0) * (2.0 * n)));
    s = dd_add(s, ps);
    c = dd_add(c, pc);
  }
  DD S{0.0, 0.0}, C{1.0, 0.0};
  for (int k = 0; k < kF64TabN; ++k) {
    const double sd = S.h + S.l, cd = C.h + C.l;
    t.sc[k][0] = sd;
    t.sc[k][1] = cd;
    t.f[k][0] = (float)sd;
    t.f[k][1] = (float)(sd - (double)(float)sd);
    t.f[k][2] = (float)cd;
    t.f[k][3] = (float)(cd - (double)(float)cd);
    const DD S1 = dd_add(dd_mul(S, c), dd_mul(C, s)), m = dd_mul(S, s);
    C = dd_add(dd_mul(C, c), DD{-m.h, -m.l});
    S = S1;
  }
  return t;
}
static __device__ const F64Tab kF64Tab = make_f64_tab();

// ------------------------------------------------ conversions

// As d2f / f2d / split_d of kc_device.cuh for values known to be far from
// overflow, in half the instructions: truncation instead of rounding, zero
// below 2^-74 (d2f_cut, split_cut); a zero float becomes 2^-127 (f2d_cut).
__device__ __forceinline__ float d2f_cut(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned m = (__funnelshift_l(l, h, 3) - (896u << 23)) & 0x7fffffffu;
  return __uint_as_float((h & 0x7fffffffu) < 0x3b500000u ? 0u : (m | (h & 0x80000000u)));
}
__device__ __forceinline__ double f2d_cut(float f) {
  const int b = __float_as_int(f);
  return __hiloint2double(((b >> 3) & 0x8fffffff) + 0x38000000, b << 29);
}
// x = hi + lo, hi the leading 24 bits of x, |lo| < ulp(hi) with 24 bits.
__device__ __forceinline__ void split_cut(double x, float &hi, float &lo) {
  hi = d2f_cut(x);
  const unsigned rest = (unsigned)__double2loint(x) & 0x1fffffffu;
  const unsigned sc = (__float_as_uint(hi) & 0xff800000u) - (52u << 23);   // +-2^(ex - 1075)
  lo = hi != 0.0f ? (float)(int)rest * __uint_as_float(sc) : 0.0f;
}
// h + l in double, |l| <= ulp(h), h zero or normal: the sum of the two
// significands on the integer pipe (about 16 instructions, where an FP64
// addition costs 64 clocks).  A negative l is taken from the float below |h|,
// so that the significand never borrows across a binade.  Below 2^-60 only h
// is kept.
__device__ __forceinline__ double pair_d(float h, float l) {
  const unsigned sign = __float_as_uint(h) & 0x80000000u;
  l = __uint_as_float(__float_as_uint(l) ^ sign);
  unsigned b = __float_as_uint(h) & 0x7fffffffu;
  const bool tiny = b < 0x21800000u, down = l < 0.0f;
  b -= down ? 1u : 0u;
  const float scale = __uint_as_float((306u << 23) - (b & 0x7f800000u));   // 2^52 / 2^E
  int r = __float2int_rn(l * scale) + (down ? 1 << 29 : 0);
  r = tiny ? 0 : r;
  const unsigned lo = b << 29, sum = lo + (unsigned)r;
  const unsigned hi = (b >> 3) + 0x38000000u + (sum < lo ? 1u : 0u);
  return __hiloint2double((int)(hi | sign), (int)sum);
}
// pair_d for a pair that may be no number: NaN where h is infinite or NaN.
__device__ __forceinline__ double pair_or_nan(float h, float l) {
  const double d = pair_d(h, l);
  const bool none = (__float_as_uint(h) & 0x7f800000u) == 0x7f800000u;
  return __hiloint2double(none ? 0x7ff80000 : __double2hiint(d), __double2loint(d));
}
__device__ __forceinline__ double xor_sign(double x, unsigned sign) {
  return __hiloint2double(__double2hiint(x) ^ (int)sign, __double2loint(x));
}
__device__ __forceinline__ float xor_sign(float x, unsigned sign) {
  return __uint_as_float(__float_as_uint(x) ^ sign);
}

// ------------------------------------------------ per-planet constants

// inv_P, c0, e, A, B as in PlanetD (A and B the velocity constants of the
// E-form); their float pairs, 1/P and 2 pi times its low part in single
// precision, and the start's constants (start_constants).  high: the velocity
// takes the form without float expansions (eval_high).
struct __align__(8) PlanetX {
  double inv_P, c0, e, A, B;
  float inv_P_f, inv_P_lo2pi, c0f;
  StartP st;
  float eh, el, Ah, Al, Bh, Bl;
  int high;
};

// Whether the velocity's differences, of 1e-3 K and less, fit the float pairs:
// |K| in [2^-30, 2^100) or zero (leading words compared).  Below it pair_d drops
// bits (2^-84 absolute), above it the pairs overflow.
__device__ __forceinline__ bool amplitude_fits(double K) {
  const unsigned h = (unsigned)__double2hiint(K) & 0x7fffffffu;
  return h - 0x3e100000u < 0x46300000u - 0x3e100000u || K == 0.0;
}

// sin and cos of any finite w from the table: w - 2 pi k in three FP64
// FMAs (2 pi as two doubles; k below 2^30, else the library's sincos), then
// the table's angle and the series of the remainder (|b| <= 2^-10: b^7/5040
// below 2e-25).
__device__ __forceinline__ void sincos_w(double w, double &s, double &c) {
  if (!(fabs(w) < 1e9)) {
    sincos(w, &s, &c);
    return;
  }
  const double k = rint(w * kInvTwoPi);
  double r = fma(-k, kTwoPi, w);
  r = fma(-k, 2.4492935982947064e-16, r);               // 2 pi - kTwoPi
  const unsigned sign = (unsigned)__double2hiint(r) & 0x80000000u;
  r = fabs(r);
  const float kf = __fadd_rn(d2f_cut(r), kF64Round);
  const int i = min((int)(__float_as_uint(kf) - __float_as_uint(kF64Round)), kF64TabN - 1);
  const double b = r - f2d(__fsub_rn(kf, kF64Round));
  const double b2 = b * b;
  const double sb = fma(b * b2, fma(b2, 1.0 / 120.0, -1.0 / 6.0), b);
  const double cb = fma(b2, fma(b2, fma(b2, -1.0 / 720.0, 1.0 / 24.0), -0.5), 1.0);
  const double S = kF64Tab.sc[i][0], C = kF64Tab.sc[i][1];
  s = xor_sign(fma(S, cb, C * sb), sign);
  c = fma(C, cb, -(S * sb));
}

// sqrt of x in [0, 1]: the single-precision root and two Newton steps whose
// corrections are formed in single precision (relative errors 6e-8, 4e-15,
// then below the last rounding).
__device__ __forceinline__ double sqrt_unit(double x) {
  const float s = sqrtf(d2f(x));
  if (s == 0.0f) return sqrt(x);
  const float h = 0.5f / s;
  double r = f2d(s);
  r += f2d(d2f(fma(-r, r, x)) * h);
  return r + f2d(d2f(fma(-r, r, x)) * h);
}

// Constants of one planet; dref = t_ref - t0.  sw, cw, beta: sin w, cos w and
// sqrt(1 - e^2), for the gradient.
__device__ __forceinline__ PlanetX planet_setup_x(const double *p, double dref, double &sw,
                                                  double &cw, double &beta) {
  const double P = p[0], K = p[1], e = p[2], w = p[3], M0 = p[4];
  PlanetX q;
  double n, nl;
  recip_checked(P, n, nl);
  q.inv_P = n;
  q.inv_P_f = d2f(n);
  q.inv_P_lo2pi = d2f(nl) * kTwoPiF;
  q.c0 = phase_cycles(dref, n, nl, M0 * kInvTwoPi);
  q.c0f = d2f(q.c0);
  q.e = e;
  sincos_w(w, sw, cw);
  const double b2 = (1.0 - e) * (1.0 + e);
  beta = sqrt_unit(b2);
  q.A = K * cw * b2;
  q.B = K * beta * sw;
  split_d(e, q.eh, q.el);
  split_d(q.A, q.Ah, q.Al);
  split_d(q.B, q.Bh, q.Bl);
  q.high = e > (double)kEccFast || !amplitude_fits(K);
  q.st = start_constants(q.eh);
  return q;
}

// ------------------------------------------------ one evaluation

// A float pair.
struct FF {
  float h, l;
};

// 1 - e (c + x) as a float pair from pairs e, c and x (x the small one):
// absolute error about 2^-49.  Also c + x.
__device__ __forceinline__ FF one_minus_e(float eh, float el, FF c, FF x, FF &cx) {
  float err;
  two_sum(c.h, x.h, cx.h, err);
  cx.l = (err + c.l) + x.l;
  float z, ze;
  two_prod(eh, cx.h, z, ze);
  FF D;
  D.h = __fsub_rn(1.0f, z);
  const float er = __fsub_rn(__fsub_rn(1.0f, D.h), z);
  D.l = __fmaf_rn(-el, cx.h, __fmaf_rn(-eh, cx.l, er - ze));
  return D;
}

// x + p y + q for the pair x with q small: the update of a difference.
__device__ __forceinline__ FF pair_step(FF x, float p, float p_lo, FF y, float q) {
  float m, me, err;
  FF r;
  two_prod(p, y.h, m, me);
  two_sum(x.h, m, r.h, err);
  float t = __fmaf_rn(p_lo, y.h, me);
  t = __fmaf_rn(p, y.l, t) + q;
  r.l = x.l + (t + err);
  return r;
}

// The solved Kepler's equation of one (planet, observation): |E|'s sine and
// cosine as the table's S, C plus the pairs ds, dc, 1/D = y (D = 1 - e cos
// E), and the sign of M (and so of sin E) as a sign bit.
struct EvalX {
  double S, C;
  FF ds, dc, y;
  unsigned sign;
  double u;          // |M| / 2 pi without the low part lo2pi, for the residual
  float lo2pi, Ef, d0, d1;
};

__device__ __forceinline__ EvalX solve_x(double tau, float tf, const PlanetX &p) {
  EvalX o;
  // phase: n is the integer nearest to it in single precision (three roundings),
  // so u = tau/P - n + c0 lies within 0.5 + 1.5 2^-23 |tau/P| of 0: 0.518 without
  // the wrap below (the table covers 0.528)
  const float n = rintf(__fmaf_rn(tf, p.inv_P_f, p.c0f));
  double u = fma(tau, p.inv_P, -f2d(n)) + p.c0;
  // (a vote, so that the usual case skips the FP64 work instead of predicating
  // it; the value is each lane's own, so that no lane's bits hang on the others)
  const bool wrap = fabsf(n) > 1e5f;
  if (__any_sync(__activemask(), wrap)) {
    const double w = u - f2d(rintf(d2f(u)));
    u = wrap ? w : u;
  }
  o.sign = (unsigned)__double2hiint(u) & 0x80000000u;
  u = xor_sign(u, o.sign);
  o.u = u;
  // n 0: NaN for a time or phase that is none (or beyond float's range).  The
  // conversions below turn it into some number; from here it reaches every float
  // pair of the solution, and pair_or_nan hands it on.
  o.lo2pi = xor_sign(__fmaf_rn(n, 0.0f, __fmul_rn(tf, p.inv_P_lo2pi)), o.sign);
  // single-precision solve
  const float m = d2f_cut(u) * kTwoPiF;
  const float sb = m * p.st.bs;
  const float r = start_root(sb, __fmaf_rn(sb, sb, 1.0f)), x = r * r;
  float pq = __fmaf_rn(x, p.st.q[4], p.st.q[3]);
  pq = __fmaf_rn(x, pq, p.st.q[2]);
  pq = __fmaf_rn(x, pq, p.st.q[1]);
  pq = __fmaf_rn(x, pq, p.st.q[0]);
  const float E0 = __fmaf_rn(r, pq, m);
  const float kf = __fadd_rn(E0, kF64Round), a = __fsub_rn(kf, kF64Round);
  const unsigned i = min(__float_as_uint(kf) - __float_as_uint(kF64Round), (unsigned)(kF64TabN - 1));
  const float4 tf4 = *reinterpret_cast<const float4 *>(kF64Tab.f[i]);
  const double2 td = *reinterpret_cast<const double2 *>(kF64Tab.sc[i]);
  const FF S = {tf4.x, tf4.y}, C = {tf4.z, tf4.w};
  o.S = td.x;
  o.C = td.y;
  float b = __fsub_rn(E0, a);
  {
    const float h = -0.5f * b;
    const float s0 = __fmaf_rn(b, __fmaf_rn(h, S.h, C.h), S.h);
    const float c0 = __fmaf_rn(b, __fmaf_rn(h, C.h, -S.h), C.h);
    const float f = __fmaf_rn(-p.eh, s0, __fsub_rn(E0, m));
    o.Ef = __fsub_rn(E0, f * rcp_fast(__fmaf_rn(-p.eh, c0, 1.0f)));
  }
  b = __fsub_rn(o.Ef, a);
  // sin, cos of Ef minus S, C: sin b = b + t3, cos b - 1 = m2h + m2l
  float b2, b2e;
  two_prod(b, b, b2, b2e);
  const float m2h = -0.5f * b2, m2l = __fmaf_rn(b2e, -0.5f, b2 * b2 * (1.0f / 24.0f));
  const float t3 = b * b2 * __fmaf_rn(b2, 1.0f / 120.0f, -1.0f / 6.0f);
  FF ds, dc;
  {
    float q, qe, w, we, err;
    two_prod(C.h, b, q, qe);
    two_prod(S.h, m2h, w, we);
    two_sum(q, w, ds.h, err);
    float t = __fmaf_rn(C.l, b, qe);
    t = __fmaf_rn(C.h, t3, t);
    t = __fmaf_rn(S.l, m2h, t);
    t = __fmaf_rn(S.h, m2l, t);
    ds.l = (t + we) + err;
    two_prod(S.h, -b, q, qe);
    two_prod(C.h, m2h, w, we);
    two_sum(q, w, dc.h, err);
    t = __fmaf_rn(-S.l, b, qe);
    t = __fmaf_rn(-S.h, t3, t);
    t = __fmaf_rn(C.l, m2h, t);
    t = __fmaf_rn(C.h, m2l, t);
    dc.l = (t + we) + err;
  }
  // f(Ef) = (Ef - M) - e S - e ds, as a pair
  float fh, fl;
  {
    const double g = fma(u, -kTwoPi, f2d_cut(o.Ef));
    float gh, gl, z, ze, err;
    split_cut(fma(-p.e, o.S, g), gh, gl);
    two_prod(p.eh, ds.h, z, ze);
    two_sum(gh, -z, fh, err);
    fl = __fmaf_rn(-p.eh, ds.l, err - ze);
    fl = __fmaf_rn(-p.el, ds.h, fl);
    fl = (fl + gl) - o.lo2pi;
    const float F = fh + fl;
    fl = fl - __fsub_rn(F, fh);
    fh = F;
  }
  // E = Ef - d, d = f/f' + (f''/2f') d^2
  FF c1, s1;
  const FF D1 = one_minus_e(p.eh, p.el, C, dc, c1);
  {
    float err;
    two_sum(S.h, ds.h, s1.h, err);
    s1.l = (err + S.l) + ds.l;
  }
  const float ri = rcp_fast(D1.h);
  const float d0 = fh * ri, hd2 = 0.5f * d0 * d0;
  float rem = __fmaf_rn(-d0, D1.h, fh);
  rem = __fmaf_rn(-d0, D1.l, rem + fl);
  rem = __fmaf_rn(p.eh * s1.h, hd2, rem);
  const float d1 = rem * ri;
  o.d0 = d0;
  o.d1 = d1;
  o.ds = pair_step(ds, -d0, -d1, c1, -hd2 * s1.h);
  o.dc = pair_step(dc, d0, d1, s1, -hd2 * c1.h);
  // 1/D as a pair: the reciprocal refined once in float, then its remainder
  FF cE;
  const FF D = one_minus_e(p.eh, p.el, C, o.dc, cE);
  float y = rcp_fast(D.h);
  y = __fmaf_rn(y, __fmaf_rn(-D.h, y, 1.0f), y);
  const float ep = __fmaf_rn(-D.l, y, __fmaf_rn(-D.h, y, 1.0f));
  fast_two_sum(y, y * __fmaf_rn(ep, ep, ep), o.y.h, o.y.l);
  return o;
}

// E of one (M, e) in double, for |M| in [2^-30, 1.02 pi] and 0 <= e <=
// kEccFast: solve_x's way with M itself and e of every evaluation, and with
// small E to full relative precision: of sin Ef = S + C b + q, b = Ef - a, the
// table's doubles take the first two terms, only q (below 2.1e-6 S and 7e-7 C b)
// is a float pair.  Five FP64 instructions, where an FP64 Halley step from
// the single-precision solution took some 16.
__device__ __forceinline__ double kepler_x(double M, double e) {
  const unsigned sign = (unsigned)__double2hiint(M) & 0x80000000u;
  M = xor_sign(M, sign);
  float eh, el;
  split_d(e, eh, el);
  const StartP st = start_constants_fast(eh);
  const float m = d2f_cut(M), sb = m * st.bs;
  const float r = start_root(sb, __fmaf_rn(sb, sb, 1.0f)), x = r * r;
  float pq = __fmaf_rn(x, st.q[4], st.q[3]);
  pq = __fmaf_rn(x, pq, st.q[2]);
  pq = __fmaf_rn(x, pq, st.q[1]);
  pq = __fmaf_rn(x, pq, st.q[0]);
  const float E0 = __fmaf_rn(r, pq, m);
  const float kf = __fadd_rn(E0, kF64Round), a = __fsub_rn(kf, kF64Round);
  const unsigned i = min(__float_as_uint(kf) - __float_as_uint(kF64Round), (unsigned)(kF64TabN - 1));
  const float4 tf = *reinterpret_cast<const float4 *>(kF64Tab.f[i]);
  const double2 td = *reinterpret_cast<const double2 *>(kF64Tab.sc[i]);
  const FF S = {tf.x, tf.y}, C = {tf.z, tf.w};
  float b = __fsub_rn(E0, a);
  float Ef;
  {
    const float h = -0.5f * b;
    const float s0 = __fmaf_rn(b, __fmaf_rn(h, S.h, C.h), S.h);
    const float c0 = __fmaf_rn(b, __fmaf_rn(h, C.h, -S.h), C.h);
    const float f = __fmaf_rn(-eh, s0, __fsub_rn(E0, m));
    Ef = __fsub_rn(E0, f * rcp_fast(__fmaf_rn(-eh, c0, 1.0f)));
  }
  b = __fsub_rn(Ef, a);
  // cos b - 1 = m2 and sin b - b = t3 as pairs
  float b2, b2e, b3, b3e;
  two_prod(b, b, b2, b2e);
  FF m2, t3, q;
  m2.h = -0.5f * b2;
  m2.l = __fmaf_rn(b2e, -0.5f, b2 * b2 * (1.0f / 24.0f));
  two_prod(b, b2, b3, b3e);
  constexpr float kSixth = -1.0f / 6.0f, kSixthLo = (float)(-1.0 / 6.0 - (double)kSixth);
  two_prod(b3, kSixth, t3.h, t3.l);
  t3.l = __fmaf_rn(b3, kSixthLo, t3.l);
  t3.l = __fmaf_rn(__fmaf_rn(b, b2e, b3e), kSixth, t3.l);
  t3.l = __fmaf_rn(b3 * b2, 1.0f / 120.0f, t3.l);
  {
    float w, we, y, ye, err;
    two_prod(S.h, m2.h, w, we);
    two_prod(C.h, t3.h, y, ye);
    two_sum(w, y, q.h, err);
    float t = __fmaf_rn(S.h, m2.l, we) + ye;
    t = __fmaf_rn(S.l, m2.h, t);
    t = __fmaf_rn(C.h, t3.l, t);
    t = __fmaf_rn(C.l, t3.h, t);
    fast_two_sum(q.h, t + err, q.h, q.l);
  }
  // f(Ef) = (Ef - M) - e S - e (C b + q), as a pair
  const double R = fma(td.y, f2d_cut(b), pair_d(q.h, q.l));
  float fh, fl;
  split_cut(fma(-e, R, fma(-e, td.x, f2d_cut(Ef) - M)), fh, fl);
  // E = Ef - d, d = f/f' + (f''/2f') d^2
  float dc, dce, z, ze, err;
  two_prod(S.h, -b, z, ze);
  two_sum(z, __fmaf_rn(C.h, m2.h, -S.h * t3.h), dc, dce);
  FF c1;
  const FF D = one_minus_e(eh, el, C, FF{dc, dce + ze}, c1);
  const float ri = rcp_fast(D.h), d0 = fh * ri;
  float rem = __fmaf_rn(-d0, D.h, fh);
  rem = __fmaf_rn(-d0, D.l, rem + fl);
  rem = __fmaf_rn(eh * __fmaf_rn(C.h, b, S.h), 0.5f * d0 * d0, rem);
  float h, l;
  two_sum(-d0, -(rem * ri), h, l);
  return xor_sign(f2d_cut(Ef) + pair_d(h, l), sign);
}

// V + (vh, vl) += v, v = (A cos E - B sin E)/D: the part at the table's angle
// on the FP64 pipe, the difference in float pairs.
// fine: 1/D corrected once in FP64 (four instructions more), for planets above
// kEccFine and for model velocities.  The pair's 48 bits of D, relative to D = 1
// - e cos E, are what limits v: the error of model velocities was 2.2e-15 of
// their rms with the pair (2.1e-15 to 2.5e-15 in the form before it) and is
// 3e-16 to 7e-16 so; that of chi2 with all e in 0.85 .. 0.95 was 2.5e-15 (1.35e-15
// before it) and is 6.6e-16.  At lower e it averages out in chi2 (e in 0.1 .. 0.4:
// 3.6e-16, 1.9e-15 before).  The vote makes it a branch (a
// predicated FP64 instruction takes the pipe's time all the same).
constexpr float kEccFine = 0.6f;
__device__ __forceinline__ void velocity_x(const EvalX &o, const PlanetX &p, bool fine, double &V,
                                           float &vh, float &vl) {
  const double N = fma(xor_sign(p.B, o.sign ^ 0x80000000u), o.S, p.A * o.C);
  double y = pair_d(o.y.h, o.y.l);
  if (__any_sync(__activemask(), fine)) {
    float h, l;
    two_sum(o.dc.h, o.dc.l, h, l);
    const double yf = fma(y, fma(-fma(-p.e, o.C + pair_d(h, l), 1.0), y, 1.0), y);
    y = fine ? yf : y;
  }
  V = fma(N, y, V);
  const float Bh = xor_sign(p.Bh, o.sign), Bl = xor_sign(p.Bl, o.sign);
  float x1, e1, x2, e2, nh, nl, err;
  two_prod(p.Ah, o.dc.h, x1, e1);
  two_prod(Bh, o.ds.h, x2, e2);
  two_sum(x1, -x2, nh, err);
  nl = (err + e1) - e2;
  nl = __fmaf_rn(p.Ah, o.dc.l, nl);
  nl = __fmaf_rn(p.Al, o.dc.h, nl);
  nl = __fmaf_rn(-Bh, o.ds.l, nl);
  nl = __fmaf_rn(-Bl, o.ds.h, nl);
  float w, we;
  two_prod(nh, o.y.h, w, we);
  we = __fmaf_rn(nl, o.y.h, __fmaf_rn(nh, o.y.l, we));
  two_sum(vh, w, vh, err);
  vl += err + we;
}

// V + (vh, vl) for a compensated pair (NaN where a time was; a zero pair, whose
// pair_d is 2^-127, adds nothing).
__device__ __forceinline__ double add_pair(double V, float vh, float vl) {
  float h, l;
  two_sum(vh, vl, h, l);
  const double d = pair_or_nan(h, l);
  return V + __hiloint2double(h == 0.0f ? 0 : __double2hiint(d), __double2loint(d));
}

// sin E (with M's sign), cos E and 1/D in double, the reciprocal's pair (48
// bits) corrected once in FP64: the partials take its square, and their
// largest terms stand where D is small.
__device__ __forceinline__ void solved_d(const EvalX &o, double e, double &sE, double &cE,
                                         double &y) {
  float h, l;
  two_sum(o.ds.h, o.ds.l, h, l);
  sE = xor_sign(o.S + pair_d(h, l), o.sign);
  two_sum(o.dc.h, o.dc.l, h, l);
  cE = o.C + pair_d(h, l);
  y = pair_or_nan(o.y.h, o.y.l);
  y = fma(y, fma(-fma(-e, cE, 1.0), y, 1.0), y);
}

// sin and cos of |x| <= 1.05 pi from the table, 11 FP64 instructions where the
// polynomials of sincos_f64 take 24: the series of the remainder end below 3e-25
// (sin) and 2e-21 (cos).
__device__ __forceinline__ void sincos_angle(double x, double &s, double &c) {
  const unsigned sign = (unsigned)__double2hiint(x) & 0x80000000u;
  x = xor_sign(x, sign);
  const float kf = __fadd_rn(d2f_cut(x), kF64Round);
  const unsigned i =
      min(__float_as_uint(kf) - __float_as_uint(kF64Round), (unsigned)(kF64TabN - 1));
  const double b = x - f2d_cut(__fsub_rn(kf, kF64Round)), b2 = b * b;
  const double2 t = *reinterpret_cast<const double2 *>(kF64Tab.sc[i]);
  const double sb = fma(b * b2, fma(b2, 1.0 / 120.0, -1.0 / 6.0), b);
  const double cb = fma(b2, fma(b2, 1.0 / 24.0, -0.5), 1.0);
  s = xor_sign(fma(t.x, cb, t.y * sb), sign);
  c = fma(t.y, cb, -(t.x * sb));
}

// kepler_f64<true>'s two quartic steps with that sine and cosine.  FP64 chi2 of
// 4096 x 4 x 256 with every e in 0.951 .. 0.99: 658 us, 805 with the
// polynomials (680 in the form before the float expansions, whose table lay in
// shared memory).
__device__ __forceinline__ double kepler_high(double M, double e, double &sE, double &cE) {
  float sf, cf;
  double E = f2d(kepler_f32(d2f(M), d2f(e), sf, cf)), s, c;
  sincos_angle(E, s, c);
  E += danby_delta_f64(E, M, e, s, c);
  sincos_angle(E, s, c);
  const double d = danby_delta_f64(E, M, e, s, c);
  const float df = d2f(d);
  const double hd2 = f2d(0.5f * df * df);
  sE = fma(d, c, fma(-hd2, s, s));
  cE = fma(-d, s, fma(-hd2, c, c));
  return E + d;
}

// The same V += v for a `high` planet.  Also sin E, cos E and |E - M - e sin E|.
__device__ __forceinline__ double eval_high(double tau, float tf, const PlanetX &p, double V,
                                            double &sE, double &cE, double &resid) {
  const double n = f2d(rintf(tf * p.inv_P_f));
  double u = fma(tau, p.inv_P, -n) + p.c0;
  u -= f2d(rintf(d2f(u)));
  const double M = fma(u, kTwoPi, f2d(tf * p.inv_P_lo2pi));
  const double E = kepler_high(M, p.e, sE, cE);
  resid = fabs((E - M) - p.e * sE);
  return fma(fma(p.A, cE, -(p.B * sE)), rcp_f64(fma(-p.e, cE, 1.0)), V);
}

// The model velocity gamma + sum_j v_j at tau.  HI: a planet of the system (or
// of the warp) is a `high` one; each planet takes its own form.
template <bool HI>
__device__ __forceinline__ double model_velocity(double tau, const PlanetX *q, int J, double gam) {
  const float tf = d2f(tau);
  double V = gam;
  float vh = 0.0f, vl = 0.0f;
#pragma unroll 1
  for (int j = 0; j < J; ++j) {
    if (HI && q[j].high) {
      double sE, cE, res;
      V = eval_high(tau, tf, q[j], V, sE, cE, res);
    } else {
      velocity_x(solve_x(tau, tf, q[j]), q[j], true, V, vh, vl);
    }
  }
  return add_pair(V, vh, vl);
}

// |E - M - e sin E| of the solution, in double.
__device__ __forceinline__ double resid_x(const EvalX &o, const PlanetX &p) {
  const double E = (f2d(o.Ef) - f2d(o.d0)) - f2d(o.d1);
  const double s = (o.S + f2d(o.ds.h)) + f2d(o.ds.l);
  return fabs((fma(o.u, -kTwoPi, E) - f2d(o.lo2pi)) - p.e * s);
}

}  // namespace kc
