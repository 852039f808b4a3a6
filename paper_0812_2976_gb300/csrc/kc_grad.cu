// kc_grad.cu -- adjoint of the fused chi-square: d chi2 / d(P, K, e, w, M0)
// for every planet and d chi2 / d gamma, for every system.
//
// Sec. 6 of the paper proposes evaluating partial derivatives of the
// goodness-of-fit statistic in parallel for derivative-based searches.  This
// kernel does it in the same pass as chi2, without storing anything per
// observation: per (observation, planet) it solves Kepler's equation (the
// same fixed-count solver as the forward kernel), keeps sin E and cos E
// in registers until the residual r_k of the observation is known, then adds
// 2 w_k r_k dv/dtheta to per-thread accumulators.  The derivatives follow
// from implicit differentiation of Kepler's equation,
//   dE = (dM + sin E de)/D,  D = 1 - e cos E,
// and of the true anomaly, df/dE = beta/D, df/de|E = sin E/(beta D) with
// beta = sqrt(1 - e^2):
//   dv/dK  = cos(w+f) + e cos w
//   dv/dw  = -K [sin(w+f) + e sin w]
//   dv/dM0 = -K sin(w+f) beta / D^2
//   dv/de  = K cos w - K sin(w+f) (sin E / D) (1/beta + beta/D)
//   dv/dP  = dv/dM0 * (-2 pi (t - t0) / P^2)     (frac() jumps ignored)
//   dV/dgamma = 1.
// Each system is handled by G <= 32 consecutive threads (one warp segment),
// combined by shuffles.
#include <algorithm>
#include <cmath>

#include "kc_device.cuh"
#include "kc_f64.cuh"
#include "kc_internal.h"
#include "kc_pair.cuh"
#include "kc_tcgen05.cuh"

namespace kc {

namespace {

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Planet constants for the gradient, single precision.
// ibeta = 1/beta, once per planet: the partials need it per observation.
struct GradPlanetF {
  PlanetF base;    // phase and velocity constants of the forward path
  float K, cw, sw, beta, n2, ibeta;   // n2 = (1/P)^2
  StartF m;        // the e-only constants of Mikkola's start
};

struct GradPlanetD {
  PlanetD base;
  double K, cw, sw, n2, ibeta;
};

__device__ inline GradPlanetF grad_setup_mixed(const double *p, double t_ref, double t0) {
  GradPlanetF g;
  g.base = planet_setup_mixed(p, t_ref, t0);
  float w_hi, w_lo;
  split_d(p[3], w_hi, w_lo);
  float sw, cw;
  sincosf(w_hi, &sw, &cw);
  g.sw = __fmaf_rn(w_lo, cw, sw);
  g.cw = __fmaf_rn(-w_lo, sw, cw);
  g.K = d2f(p[1]);
  const float e = g.base.e;
  g.beta = sqrtf((1.0f - e) * (1.0f + e));
  g.ibeta = 1.0f / g.beta;
  const float n = g.base.n_hi;
  g.n2 = n * n;
  g.m = kepler_start_setup(e);
  return g;
}

__device__ inline GradPlanetD grad_setup_f64(const double *p, double dref) {
  GradPlanetD g;
  g.base = planet_setup_f64(p, dref);
  sincos(p[3], &g.sw, &g.cw);
  g.K = p[1];
  g.n2 = g.base.inv_P * g.base.inv_P;
  g.ibeta = 1.0 / g.base.beta;
  return g;
}

__device__ inline double nan_d() { return __longlong_as_double(0x7ff8000000000000ll); }

__device__ inline double system_gamma_g(const double *p, int J) {
  bool ok = finite_bits(p[5 * J]);
  for (int j = 0; j < J; ++j)
    ok = ok && planet_valid(p[5 * j], p[5 * j + 1], p[5 * j + 2], p[5 * j + 3], p[5 * j + 4]);
  return ok ? p[5 * J] : nan_d();
}

// Free jitter of a system whose parameters end with (gamma, sigma_j).
__device__ inline double system_jitter_g(const double *p, int J) {
  const double sj = p[5 * J + 1];
  return finite_bits(sj) ? sj : nan_d();
}

constexpr double kLn2PiG = 1.8378770664093454836;      // ln(2 pi)

__device__ inline double inv_variance_g(double sigma, double jitter2) {
  const double var = fma(sigma, sigma, jitter2);
  return (var > 0.0) ? recip_d(var) : nan_d();
}

template <typename T>
struct Partials {
  T dP, dK, de, dw, dM;
};

// Partials of one planet's velocity from sin E, cos E and 1/D,
// D = 1 - e cos E (shared by both precisions).
template <typename T>
__device__ __forceinline__ void velocity_partials(T e, T K, T cw, T sw, T beta, T ibeta, T sE, T cE,
                                                  T invD, Partials<T> &d) {
  const T cf = (cE - e) * invD;           // cos f
  const T sf = beta * sE * invD;          // sin f
  const T c_wf = cw * cf - sw * sf;       // cos(w + f)
  const T s_wf = sw * cf + cw * sf;       // sin(w + f)
  d.dK = c_wf + e * cw;
  d.dw = -K * (s_wf + e * sw);
  const T ks = K * s_wf * invD;
  d.dM = -ks * beta * invD;
  d.de = K * cw - ks * sE * (ibeta + beta * invD);
}

// Shared memory of the packed gradient: the sin/cos table, the planets, the
// systems' gamma, six arrays of staged observations.
struct MixedGradLayout {
  size_t tab, pl, gam, obs, total;
  __host__ __device__ MixedGradLayout(int ST, int J, int tile) {
    tab = 0;
    pl = tab + sizeof(AngTab);
    gam = pl + sizeof(GradPlanetP) * ST * J;
    obs = align_up(gam + sizeof(float) * ST, 16);
    total = obs + sizeof(float) * 6 * tile;
  }
};
// obs_tile rounded up to whole pairs of every lane of a system.
__host__ __device__ inline int grad_tile(int obs_tile, int G) {
  return (obs_tile + 2 * G - 1) / (2 * G) * (2 * G);
}

struct ScalarGradLayout {
  size_t pl, gam, sj, obs, w, total;
  __host__ __device__ ScalarGradLayout(int ST, int J, int obs_tile) {
    pl = 0;
    gam = pl + sizeof(GradPlanetF) * ST * J;
    sj = gam + sizeof(float) * ST;
    obs = align_up(sj + sizeof(float) * ST, 16);
    w = obs + sizeof(float4) * obs_tile;
    total = align_up(w + sizeof(float2) * obs_tile, 16);
  }
};

struct ObsGD {
  double tau, v, w, dt;    // dt = t - t0
};

// Staged observation of the FP64 gradient (tf = tau in single precision).
struct __align__(16) ObsXD {
  double tau, v, w, dt;    // dt = t - t0
  float tf, pad;
  double pad2;
};

// Planet constants of the FP64 gradient: the solve's, and those of the
// partials in the form below.
struct __align__(8) GradPlanetX {
  PlanetX base;
  double K, sw, cw, A1, B1, C1, esw, beta, ibeta, n2;
};

struct F64GradLayout {
  size_t pl, gam, sj, obs, total;
  __host__ __device__ F64GradLayout(int ST, int J, int obs_tile) {
    pl = 0;
    gam = pl + sizeof(GradPlanetX) * ST * J;
    sj = gam + sizeof(double) * ST;
    obs = align_up(sj + sizeof(double) * ST, 16);
    total = align_up(obs + sizeof(ObsXD) * obs_tile, 16);
  }
};

// ------------------------------------------------------------ mixed

// Two observations per lane at a time, packed (kc_pair.cuh).  Bound by FP32
// issue and register ports like the forward kernel: 103 clocks per warp,
// planet and observation and sub-partition (68 of them the forward part);
// 128 registers hold the packed sums of up to three planets.  65536 x 3 x
// 512, us: 375 with the scalar kernel, 277 at its launch shape, 260 at the
// shape of kc_api.cu's model.
template <int J>
__global__ void __launch_bounds__(256, 2)
grad_mixed_kernel(UniformArgs a, int G, int obs_tile, float *__restrict__ chi2_out,
                  float *__restrict__ grad_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NP = 5 * J + 1;
  const int block = blockDim.x;
  const int ST = block / G;
  const int tile = grad_tile(obs_tile, G);
  const MixedGradLayout L(ST, J, tile);
  float *tab_s = reinterpret_cast<float *>(smem + L.tab);
  GradPlanetP *pl_s = reinterpret_cast<GradPlanetP *>(smem + L.pl);
  float *gam_s = reinterpret_cast<float *>(smem + L.gam);
  float *obs_s = reinterpret_cast<float *>(smem + L.obs);   // th, tl, v hi, v lo, w, t - t0

  const int tid = threadIdx.x;
  const int64_t sys0 = (int64_t)blockIdx.x * ST;
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  const Split3 tr3 = split3(t_ref), te3 = split3(a.t0);
  const float dref_f = (tr3.x0 - te3.x0) + (tr3.x1 - te3.x1);     // t_ref - t0, float
  const float jit2 = d2f(a.jitter2);
  ang_tab_load<true>(tab_s, tid, block);

  bool wide = false, plain = false;
  for (int i = tid; i < ST * J; i += block) {
    const int sl = i / J, j = i - sl * J;
    const int64_t s = sys0 + sl;
    GradPlanetP q = {};
    if (s < a.n_sys && dbg_ok(a.invalid, s * NP + 5 * j + 4 < a.n_sys * NP, kDbgParam, s * NP)) {
      q = grad_setup_pair(a.params + s * NP + 5 * j, t_ref, a.t0, false);
      wide |= short_period(q.p);
    }
    pl_s[i] = q;
  }
  for (int i = block - 1 - tid; i < ST; i += block) {
    const int64_t s = sys0 + i;
    gam_s[i] = s < a.n_sys ? d2f(system_gamma_g(a.params + s * NP, J)) : 0.0f;
  }

  // the tile that starts at k0; the padding has zero weight; plain: the times
  // stay as they are.  Returns whether one is a far one.
  auto stage = [&](int k0) {
    const int nk = min(obs_tile, a.n_obs - k0), npad = grad_tile(nk, G);
    bool far = false;
    for (int k = block - 1 - tid; k < npad; k += block) {
      float th = 0.0f, tl = 0.0f, vh = 0.0f, vl = 0.0f, wk = 0.0f, dt = 0.0f;
      if (k < nk && dbg_ok(a.invalid, k0 + k < a.n_obs, kDbgObs, k0 + k)) {
        sub_ds(split3(a.t[k0 + k]), tr3, th, tl);
        dt = th + dref_f;
        if (!plain) tau_place(th, tl);
        far |= far_time(th);
        split_d(a.v[k0 + k], vh, vl);
        const float sg = d2f(a.sigma[k0 + k]);
        const float var = __fmaf_rn(sg, sg, jit2);
        wk = var > 0.0f ? 1.0f / var : __int_as_float(0x7fc00000);
      }
      obs_s[k] = th;
      obs_s[tile + k] = tl;
      obs_s[2 * tile + k] = vh;
      obs_s[3 * tile + k] = vl;
      obs_s[4 * tile + k] = wk;
      obs_s[5 * tile + k] = dt;
    }
    return far;
  };
  bool far = stage(0);
  if (a.n_obs > obs_tile) far |= far_later(a.t, obs_tile, a.n_obs);
  wide = __syncthreads_or(wide || far);

  const int sl = tid / G, c = tid - sl * G;
  const int64_t s = sys0 + sl;
  const GradPlanetP *q = pl_s + sl * J;

  // all tiles' sums, their combination, the results (compiled twice from here on,
  // so that the short form keeps its registers)
  with_high_e(wide, [&](auto tag) {
    constexpr bool WIDE = decltype(tag)::value;
    MeanForm form;
    bool exact = false;
    if (WIDE) {
      plain = __syncthreads_or(far);
      if (plain) {
        // the planets and the first tile's times as plain pairs
        for (int i = tid; i < ST * J; i += block) {
          const int64_t at = (sys0 + i / J) * NP + 5 * (i % J);
          if (sys0 + i / J < a.n_sys && dbg_ok(a.invalid, at < a.n_sys * NP, kDbgParam, at))
            planet_plain(pl_s[i].p, a.params[at]);
        }
        for (int k = tid; k < min(obs_tile, a.n_obs); k += block)
          sub_ds(split3(a.t[k]), tr3, obs_s[k], obs_s[tile + k]);
        __syncthreads();
      }
      float n_max = 0.0f;                        // the system's shortest period
#pragma unroll
      for (int j = 0; j < J; ++j) n_max = fmaxf(n_max, q[j].p.n);
      form.brief = !plain && n_max <= kPairMaxFreq;
      form.some = __any_sync(0xffffffffu, form.brief);
      form.all = __all_sync(0xffffffffu, form.brief);
      exact = n_max > kPairExactFreq;
    }
    const float gam = gam_s[sl];
    Kahan2 acc = {0, 0};
    f32x2 sum_a = 0;
    typename GradSumsFor<J>::type g[J];
#pragma unroll
    for (int j = 0; j < J; ++j) g[j] = {{0, 0}, 0, 0, 0, 0};

    for (int k0 = 0; k0 < a.n_obs; k0 += obs_tile) {
      if (k0 > 0) {
        __syncthreads();
        stage(k0);
        __syncthreads();
      }
      const int npad = grad_tile(min(obs_tile, a.n_obs - k0), G);
      // (a warp of short-form systems alone in a wide CTA takes the short body)
      with_high_e(WIDE && !form.all, [&](auto body) {
        constexpr bool W = decltype(body)::value;
        for (int k = 2 * c; k < npad; k += 2 * G) {
          // the planets' constants are read again in every iteration: hoisted
          // for all J planets they would not fit the registers
          asm volatile("" ::: "memory");
          auto at = [&](int array) {
            return *reinterpret_cast<const f32x2 *>(obs_s + array * tile + k);
          };
          f32x2 th = at(0), tl = at(1);
          if (W && exact) plain_times(a.t, k0 + k, a.n_obs, th, tl);
          GradTerms o[J];
          Kahan2 V = {dup2(gam), 0};
#pragma unroll
          for (int j = 0; j < J; ++j) o[j] = grad_terms<W>(th, tl, q[j], tab_s, V, form);
          const f32x2 r = sub2(sub2(V.big, at(2)), add2(V.small, at(3)));
          const f32x2 wr = mul2(at(4), r), a2 = add2(wr, wr);
          kahan_add(acc, mul2(wr, r));
          sum_a = add2(sum_a, a2);
          const f32x2 adt = mul2(a2, at(5));
#pragma unroll
          for (int j = 0; j < J; ++j) grad_add(g[j], o[j], q[j], a2, adt);
        }
      });
    }

    Kahan chi = kahan_join(acc);
    float sa = join2(sum_a);
    GradLane gl[J];
#pragma unroll
    for (int j = 0; j < J; ++j) gl[j] = grad_join(g[j]);
    for (int m = G >> 1; m >= 1; m >>= 1) {
      const Kahan o = {shfl_xor(chi.big, m), shfl_xor(chi.small, m)};
      kahan_merge(chi, o);
      sa += shfl_xor(sa, m);
#pragma unroll
      for (int j = 0; j < J; ++j) grad_combine(gl[j], m);
    }
    if (c == 0 && s < a.n_sys) {
      // NaN for an invalid system
      const float poison = 0.0f * gam_s[sl];
      const float value = kahan_value(chi) + poison;
      if (chi2_out) chi2_out[s] = value;
      note_invalid(a.invalid, value);
      float *out = grad_out + s * NP;
#pragma unroll
      for (int j = 0; j < J; ++j) grad_finish(gl[j], q[j], sa, poison, out + 5 * j);
      out[5 * J] = sa + poison;
    }
  });
}

// One observation per lane at a time, in scalar single precision: the
// gradient behind autograd (which widens it to double, so that it carries single
// precision all the same) and of the free-jitter likelihood, whose per-system
// variance grad_mixed_kernel above has no form for.  65536 x 3 x 512: 375 us,
// the packed kernel 260.
// NLL = true: the free-jitter negative log-likelihood (see kc_fwd.cu) and
// its gradient, including d nll / d sigma_j = sigma_j sum_k w_k (1 - w_k r_k^2)
// (the planet and gamma terms carry w_k r_k instead of 2 w_k r_k).
template <int J, bool NLL = false>
__global__ void __launch_bounds__(256, 2)
grad_scalar_kernel(UniformArgs a, int G, int obs_tile, float *__restrict__ chi2_out,
                  float *__restrict__ grad_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NP = 5 * J + 1 + (NLL ? 1 : 0);
  const int block = blockDim.x;
  const int ST = block / G;
  const ScalarGradLayout L(ST, J, obs_tile);
  GradPlanetF *pl_s = reinterpret_cast<GradPlanetF *>(smem + L.pl);
  float *gam_s = reinterpret_cast<float *>(smem + L.gam);
  float *sj_s = reinterpret_cast<float *>(smem + L.sj);
  float4 *obs_s = reinterpret_cast<float4 *>(smem + L.obs);
  float2 *wt_s = reinterpret_cast<float2 *>(smem + L.w);   // (w_k, t_k - t0)

  const int tid = threadIdx.x;
  const int64_t sys0 = (int64_t)blockIdx.x * ST;
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  const Split3 tr3 = split3(t_ref), te3 = split3(a.t0);
  const float dref_f = (tr3.x0 - te3.x0) + (tr3.x1 - te3.x1);     // t_ref - t0, float
  const float jit2 = d2f(a.jitter2);

  for (int i = tid; i < ST * J; i += block) {
    const int sl = i / J, j = i - sl * J;
    const int64_t s = sys0 + sl;
    GradPlanetF q = {};
    if (s < a.n_sys && dbg_ok(a.invalid, s * NP + 5 * j + 4 < a.n_sys * NP, kDbgParam, s * NP))
      q = grad_setup_mixed(a.params + s * NP + 5 * j, t_ref, a.t0);
    pl_s[i] = q;
  }
  for (int i = tid; i < ST; i += block) {
    const int64_t s = sys0 + i;
    gam_s[i] = s < a.n_sys ? d2f(system_gamma_g(a.params + s * NP, J)) : 0.0f;
    if (NLL) sj_s[i] = s < a.n_sys ? d2f(system_jitter_g(a.params + s * NP, J)) : 0.0f;
  }

  const int sl = tid / G, c = tid - sl * G;
  const int64_t s = sys0 + sl;
  Kahan acc = {0.0f, 0.0f};
  // d/dP terms carry (t - t0)/P^2 and cancel heavily across observations, so
  // they are summed with compensation (plain FP32 sums lost up to ~3e-3)
  Kahan gP[J];
  float g[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) g[i] = 0.0f;
#pragma unroll
  for (int j = 0; j < J; ++j) gP[j] = Kahan{0.0f, 0.0f};

  for (int k0 = 0; k0 < a.n_obs; k0 += obs_tile) {
    const int nk = min(obs_tile, a.n_obs - k0);
    __syncthreads();
    for (int k = tid; k < nk; k += block) {
      if (!dbg_ok(a.invalid, k0 + k < a.n_obs, kDbgObs, k0 + k)) continue;
      float th, tl, vh, vl;
      sub_ds(split3(a.t[k0 + k]), tr3, th, tl);
      split_d(a.v[k0 + k], vh, vl);
      obs_s[k] = make_float4(th, tl, vh, vl);
      const float sg = d2f(a.sigma[k0 + k]);
      const float var = __fmaf_rn(sg, sg, jit2);
      wt_s[k] = make_float2(NLL ? sg * sg : (var > 0.0f ? 1.0f / var : __int_as_float(0x7fc00000)),
                            th + dref_f);
    }
    __syncthreads();
    const float gam = gam_s[sl];
    const float sj = NLL ? sj_s[sl] : 0.0f;
    const GradPlanetF *q = pl_s + sl * J;
    for (int k = c; k < nk; k += G) {
      const float4 o = obs_s[k];
      const float2 wt = wt_s[k];
      float sEj[J], cEj[J];
      Kahan V = {0.0f, 0.0f};
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const PlanetF p = q[j].base;
        const float M = mean_anomaly_mixed(o.x, o.y, p);
        kepler_f32_h(M, p.e, q[j].m, sEj[j], cEj[j]);
        kahan_add(V, velocity_mixed(p, sEj[j], cEj[j]));
      }
      const float r = __fadd_rn(__fsub_rn(V.big, o.z), __fsub_rn(gam, __fadd_rn(V.small, o.w)));
      float wk = wt.x, a2;
      if (NLL) {
        const float var = __fmaf_rn(sj, sj, wt.x);           // sigma_k^2 + sigma_j^2
        wk = var > 0.0f ? rcp_fast(var) : __int_as_float(0x7fc00000);
        const float wr = wk * r;
        kahan_add(acc, __fmaf_rn(wr, r, lg2_fast(var) * 0.693147180559945309f));
        a2 = wr;
        g[NP - 1] = __fmaf_rn(sj * wk, __fmaf_rn(-wr, r, 1.0f), g[NP - 1]);
      } else {
        const float wr = wk * r;
        kahan_add(acc, wr * r);
        a2 = 2.0f * wr;
      }
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const GradPlanetF qj = q[j];
        Partials<float> d;
        const float invD = rcp_fast(__fmaf_rn(-qj.base.e, cEj[j], 1.0f));
        velocity_partials(qj.base.e, qj.K, qj.cw, qj.sw, qj.beta, qj.ibeta, sEj[j], cEj[j], invD,
                            d);
        d.dP = d.dM * (-kTwoPiF * wt.y * qj.n2);
        kahan_add(gP[j], a2 * d.dP);
        g[5 * j + 1] = fmaf(a2, d.dK, g[5 * j + 1]);
        g[5 * j + 2] = fmaf(a2, d.de, g[5 * j + 2]);
        g[5 * j + 3] = fmaf(a2, d.dw, g[5 * j + 3]);
        g[5 * j + 4] = fmaf(a2, d.dM, g[5 * j + 4]);
      }
      g[5 * J] += a2;
    }
  }

  for (int m = G >> 1; m >= 1; m >>= 1) {
    Kahan o = {shfl_xor(acc.big, m), shfl_xor(acc.small, m)};
    kahan_merge(acc, o);
#pragma unroll
    for (int j = 0; j < J; ++j) {
      Kahan op = {shfl_xor(gP[j].big, m), shfl_xor(gP[j].small, m)};
      kahan_merge(gP[j], op);
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) g[i] += shfl_xor(g[i], m);
  }
#pragma unroll
  for (int j = 0; j < J; ++j) g[5 * j] = kahan_value(gP[j]);
  if (c == 0 && s < a.n_sys) {
    // NaN for an invalid system
    const float poison = 0.0f * gam_s[sl] + (NLL ? 0.0f * sj_s[sl] : 0.0f);
    const float value = NLL ? 0.5f * (kahan_value(acc) + (float)a.n_obs * (float)kLn2PiG) + poison
                            : kahan_value(acc) + poison;
    if (chi2_out) chi2_out[s] = value;
    note_invalid(a.invalid, value);
#pragma unroll
    for (int i = 0; i < NP; ++i) grad_out[s * NP + i] = g[i] + poison;
  }
}

// ------------------------------------------------------------ FP64

// Bound by the FP64 pipe: 27 FP64 instructions per evaluation (kc_f64.cuh's
// solve 4, sin E, cos E and 1/D 5, the velocity and Q 7, the partials and
// their sums 11), 105 before.  With
// y = 1/D, A1 = cos w (1 - e^2), B1 = beta sin w, C1 = beta cos w,
//   dv/dK  = (A1 cos E - B1 sin E) y = v/K,
//   Q      = sin(w + f) = (sin w cos E + C1 sin E - e sin w) y,
//   dv/dw  = -K (Q + e sin w),   dv/dM0 = -K beta Q y^2,
//   dv/de  = K cos w - K Q y sin E (1/beta + beta y),
// so the sums over the observations need only those of a v/K, a Q, a Q y^2,
// a dt Q y^2 and a Q y sin E (1/beta + beta y), a = 2 w r: the per-planet
// factors, and the parts a alone multiplies (its sum is gamma's gradient),
// are applied once per system.
__device__ inline GradPlanetX grad_setup_x(const double *p, double dref) {
  GradPlanetX g;
  double sw, cw, beta;
  g.base = planet_setup_x(p, dref, sw, cw, beta);
  const double e = p[2];
  g.K = p[1];
  g.sw = sw;
  g.cw = cw;
  g.A1 = cw * ((1.0 - e) * (1.0 + e));
  g.B1 = beta * sw;
  g.C1 = beta * cw;
  g.esw = e * sw;
  g.beta = beta;
  g.ibeta = 1.0 / beta;
  g.n2 = g.base.inv_P * g.base.inv_P;
  return g;
}

template <int J, bool NLL = false>
__global__ void __launch_bounds__(256, 2)
grad_f64_kernel(UniformArgs a, int G, int obs_tile, double *__restrict__ chi2_out,
                double *__restrict__ grad_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NP = 5 * J + 1 + (NLL ? 1 : 0);
  const int block = blockDim.x;
  const int ST = block / G;
  const F64GradLayout L(ST, J, obs_tile);
  GradPlanetX *pl_s = reinterpret_cast<GradPlanetX *>(smem + L.pl);
  double *gam_s = reinterpret_cast<double *>(smem + L.gam);
  double *sj_s = reinterpret_cast<double *>(smem + L.sj);
  ObsXD *obs_s = reinterpret_cast<ObsXD *>(smem + L.obs);

  const int tid = threadIdx.x;
  const int64_t sys0 = (int64_t)blockIdx.x * ST;
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  const double dref = t_ref - a.t0;

  for (int i = block - 1 - tid; i < ST; i += block) {
    const int64_t s = sys0 + i;
    gam_s[i] = s < a.n_sys ? system_gamma_g(a.params + s * NP, J) : 0.0;
    if (NLL) sj_s[i] = s < a.n_sys ? system_jitter_g(a.params + s * NP, J) : 0.0;
  }
  // the planets' setup dealt densely to one warp, another in each CTA
  int first = tid - 32 * (int)(blockIdx.x % (unsigned)(block >> 5));
  if (first < 0) first += block;
  for (int i = first; i < ST * J; i += block) {
    const int sl = i / J, j = i - sl * J;
    const int64_t s = sys0 + sl;
    GradPlanetX q = {};
    if (s < a.n_sys && dbg_ok(a.invalid, s * NP + 5 * j + 4 < a.n_sys * NP, kDbgParam, s * NP))
      q = grad_setup_x(a.params + s * NP + 5 * j, dref);
    pl_s[i] = q;
  }

  const int sl = tid / G, c = tid - sl * G;
  const int64_t s = sys0 + sl;
  double acc = 0.0, sum_a = 0.0, sum_j = 0.0;
  double g[5 * J];
#pragma unroll
  for (int i = 0; i < 5 * J; ++i) g[i] = 0.0;

  for (int k0 = 0; k0 < a.n_obs; k0 += obs_tile) {
    const int nk = min(obs_tile, a.n_obs - k0);
    if (k0 > 0) __syncthreads();
    for (int k = tid; k < nk; k += block) {
      if (!dbg_ok(a.invalid, k0 + k < a.n_obs, kDbgObs, k0 + k)) continue;
      ObsXD o;
      const double tk = a.t[k0 + k];
      o.tau = tk - t_ref;
      o.v = a.v[k0 + k];
      o.w = NLL ? a.sigma[k0 + k] * a.sigma[k0 + k] : inv_variance_g(a.sigma[k0 + k], a.jitter2);
      o.dt = tk - a.t0;
      o.tf = d2f(o.tau);
      o.pad = 0.0f;
      o.pad2 = 0.0;
      obs_s[k] = o;
    }
    __syncthreads();
    const double gam = gam_s[sl];
    const GradPlanetX *q = pl_s + sl * J;
    bool hi = false;
#pragma unroll
    for (int j = 0; j < J; ++j) hi = hi || q[j].base.e > (double)kEccFast;
    with_high_e(any_high_e(hi), [&](auto tag) {
      constexpr bool HI = decltype(tag)::value;
      for (int k = c; k < nk; k += G) {
        const ObsXD o = obs_s[k];
        double sE[J], dK[J], Q[J], y[J];
        double r = gam - o.v;
#pragma unroll (J <= 3 ? J : 1)
        for (int j = 0; j < J; ++j) {
          const GradPlanetX &p = q[j];
          double cE;
          if (HI && p.base.e > (double)kEccFast) {
            double res;
            eval_high(o.tau, o.tf, p.base, 0.0, sE[j], cE, res);
            y[j] = 1.0 / fma(-p.base.e, cE, 1.0);
          } else {
            solved_d(solve_x(o.tau, o.tf, p.base), p.base.e, sE[j], cE, y[j]);
          }
          dK[j] = fma(p.A1, cE, -(p.B1 * sE[j])) * y[j];
          Q[j] = fma(p.C1, sE[j], fma(p.sw, cE, -p.esw)) * y[j];
          r = fma(p.K, dK[j], r);
        }
        double a2;
        if (NLL) {
          const double sj = sj_s[sl];
          const double var = fma(sj, sj, o.w);
          const double wk = var > 0.0 ? recip_d(var) : nan_d();
          const double wr = wk * r;
          acc += fma(wr, r, log(var));
          a2 = wr;
          sum_j = fma(wk, fma(-wr, r, 1.0), sum_j);
        } else {
          const double wr = o.w * r;
          acc = fma(wr, r, acc);
          a2 = 2.0 * wr;
        }
        sum_a += a2;
        const double adt = a2 * o.dt;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const GradPlanetX &p = q[j];
          const double Qy = Q[j] * y[j], Qyy = Qy * y[j];
          const double h = fma(p.beta, y[j], p.ibeta);
          g[5 * j + 0] = fma(adt, Qyy, g[5 * j + 0]);
          g[5 * j + 1] = fma(a2, dK[j], g[5 * j + 1]);
          g[5 * j + 2] = fma(a2 * Qy, sE[j] * h, g[5 * j + 2]);
          g[5 * j + 3] = fma(a2, Q[j], g[5 * j + 3]);
          g[5 * j + 4] = fma(a2, Qyy, g[5 * j + 4]);
        }
      }
    });
  }
  if (a.n_obs == 0) __syncthreads();            // gam_s, sj_s written by other threads

  for (int m = G >> 1; m >= 1; m >>= 1) {
    acc += shfl_xor(acc, m);
    sum_a += shfl_xor(sum_a, m);
    if (NLL) sum_j += shfl_xor(sum_j, m);
#pragma unroll
    for (int i = 0; i < 5 * J; ++i) g[i] += shfl_xor(g[i], m);
  }
  if (c == 0 && s < a.n_sys) {
    const double poison = 0.0 * gam_s[sl] + (NLL ? 0.0 * sj_s[sl] : 0.0);
    const double value = NLL ? 0.5 * (acc + a.n_obs * kLn2PiG) + poison : acc + poison;
    if (chi2_out) chi2_out[s] = value;
    note_invalid(a.invalid, value);
    double *out = grad_out + s * NP;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const GradPlanetX &p = pl_s[sl * J + j];
      const double Kb = p.K * p.beta;
      out[5 * j + 0] = fma(Kb * (kTwoPi * p.n2), g[5 * j + 0], poison);
      out[5 * j + 1] = g[5 * j + 1] + poison;
      out[5 * j + 2] = fma(p.K, fma(p.cw, sum_a, -g[5 * j + 2]), poison);
      out[5 * j + 3] = fma(-p.K, fma(p.esw, sum_a, g[5 * j + 3]), poison);
      out[5 * j + 4] = fma(-Kb, g[5 * j + 4], poison);
    }
    out[5 * J] = sum_a + poison;
    if (NLL) out[5 * J + 1] = fma(sj_s[sl], sum_j, poison);
  }
}

// ------------------------------------------------------------ Gauss-Newton
//
// H = sum_k w_k J_k J_k^T per system (J_k = dV_k/dtheta), with chi2 and its
// gradient from the same pass: the matrix and the right-hand side of a
// Levenberg-Marquardt step (Sec. 6 lists derivatives for least-squares
// refinement as future work).  One warp per system; each lane evaluates one
// observation of a batch of 32 and writes u_k = sqrt(w_k) J_k as a row of a
// 32 x n matrix U in shared memory; the warp then adds U^T U to its
// accumulators.  Mixed path: that update is a rank-32 dense contraction per
// batch on the tensor cores (mma.sync m16n8k8 here; the tcgen05 form
// follows), TF32 inputs in the three-
// product split hi*hi + hi*lo + lo*hi, FP32 accumulation), only the tiles
// on or above the diagonal.  Each element of U is split into its (hi, lo)
// pair once, when its row is written; since B = U and A = U^T cover the
// same elements, the B fragments are halves of the A fragments.  FP64 path:
// FMAs on the FP64 pipe, the packed upper-triangle entries spread over the
// lanes.

constexpr int kGnWarps = 4;      // mixed: systems (warps) per CTA
constexpr int kGnWarpsD = 2;     // FP64
constexpr int kGnObsTile = 256;
constexpr int kGnAhead = 4;      // systems a warp of a pair kernel sets up together
constexpr int kTcObsTile = 512;  // observations the pair kernels stage at a time
constexpr int kGnRows = 64;      // observations per batch of the pair kernels: two per lane

__host__ __device__ constexpr int gn_np(int J) { return 5 * J + 1; }
__host__ __device__ constexpr int gn_mt(int J) { return (gn_np(J) + 15) / 16; }
__host__ __device__ constexpr int gn_nt(int J) { return (gn_np(J) + 7) / 8; }
// Row stride of U in (hi, lo) pairs: the tiled width 16 MT (>= 8 NT) plus 4,
// which is 4 mod 16 pairs, so that with the column swizzle below the 64-bit
// row writes and fragment loads of each half-warp hit 32 different banks.
__host__ __device__ constexpr int gn_row2(int J) { return gn_mt(J) * 16 + 4; }


struct GnMixedLayout {
  size_t pl, gam, obs, w, u, total;
  __host__ __device__ GnMixedLayout(int J, int obs_tile) {
    pl = 0;
    gam = pl + sizeof(GradPlanetF) * kGnWarps * J;
    obs = align_up(gam + sizeof(float) * kGnWarps, 16);
    w = obs + sizeof(float4) * obs_tile;
    u = align_up(w + sizeof(float4) * obs_tile, 16);
    total = align_up(u + sizeof(float2) * kGnWarps * 32 * gn_row2(J), 16);
  }
};

struct GnPairLayout {
  size_t tab, pl, obs, u, total;
  __host__ __device__ GnPairLayout(int J, int obs_tile) {
    tab = 0;
    pl = tab + sizeof(AngTab);
    obs = align_up(pl + sizeof(GradPlanetP) * kGnWarps * kGnAhead * J, 16);
    u = align_up(obs + sizeof(float) * 5 * obs_tile, 16);
    total = align_up(u + sizeof(float2) * kGnWarps * kGnRows * gn_row2(J), 16);
  }
};

struct GnF64Layout {
  size_t pl, gam, obs, pq, u, total;
  __host__ __device__ GnF64Layout(int J, int obs_tile) {
    const int np = gn_np(J), ntri = np * (np + 1) / 2;
    pl = 0;
    gam = pl + sizeof(GradPlanetD) * kGnWarpsD * J;
    obs = align_up(gam + sizeof(double) * kGnWarpsD, 16);
    pq = obs + sizeof(ObsGD) * obs_tile;
    u = align_up(pq + sizeof(short2) * ntri, 16);
    total = align_up(u + sizeof(double) * kGnWarpsD * 32 * (np | 1), 16);
  }
};

// Index of H[p][q], q >= p, in the packed upper triangle (row by row).
__device__ __forceinline__ int tri_index(int np, int p, int q) {
  return p * np - (p * (p - 1)) / 2 + (q - p);
}

// x = hi + lo + err with hi, lo TF32 numbers (FP32 with the 13 low
// significand bits zero): hi keeps the leading 11 significant bits of x, so
// |x - hi| < 2^-10 |x| and x - hi is exact in FP32; lo keeps the leading 11
// bits of x - hi, so |err| < 2^-20 |x|.  A product from the three terms
// hi*hi + hi*lo + lo*hi is then within about 3 * 2^-20 of the FP32 one.
__device__ __forceinline__ float2 tf32_pair(float x) {
  constexpr unsigned kTf32Mask = 0xffffe000u;
  const float hi = __uint_as_float(__float_as_uint(x) & kTf32Mask);
  const float lo = __uint_as_float(__float_as_uint(__fsub_rn(x, hi)) & kTf32Mask);
  return make_float2(hi, lo);
}

// D = A B + D for one 16 x 8 tile, A 16 x 8 (row), B 8 x 8 (col), TF32.
__device__ __forceinline__ void mma_tf32(float (&d)[4], const unsigned (&a)[4],
                                         const unsigned (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, "
      "{%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// The observations of one tile staged for the Gauss-Newton kernels: five
// arrays of STRIDE floats (th, tl, v hi, v lo, sqrt w), padded with zero weight
// to whole batches.  plain: the times stay as they are.  Returns whether one is
// a far one.
template <int STRIDE>
__device__ __forceinline__ bool gn_stage(const UniformArgs &a, int k0, int nk, int npad, int tid,
                                         int nthreads, const Split3 &tr3, float jit2, bool plain,
                                         float *obs) {
  bool far = false;
  // four observations' loads in flight: a tile is staged again for every four
  // systems where the observations exceed it
  for (int k4 = tid; k4 < npad; k4 += 4 * nthreads) {
    double t[4], v[4], sigma[4];
    bool real[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k4 + i * nthreads;
      real[i] = k < nk && dbg_ok(a.invalid, k0 + k < a.n_obs, kDbgObs, k0 + k);
      t[i] = real[i] ? a.t[k0 + k] : 0.0;
      v[i] = real[i] ? a.v[k0 + k] : 0.0;
      sigma[i] = real[i] ? a.sigma[k0 + k] : 1.0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k4 + i * nthreads;
      if (k >= npad) break;
      float th = 0.0f, tl = 0.0f, vh = 0.0f, vl = 0.0f, wk = 0.0f;
      if (real[i]) {
        sub_ds(split3(t[i]), tr3, th, tl);
        if (!plain) tau_place(th, tl);
        far |= far_time(th);
        split_d(v[i], vh, vl);
        const float sg = d2f(sigma[i]);
        const float var = __fmaf_rn(sg, sg, jit2);
        wk = var > 0.0f ? 1.0f / var : __int_as_float(0x7fc00000);
      }
      const float o[5] = {th, tl, vh, vl, sqrtf(wk)};
#pragma unroll
      for (int j = 0; j < 5; ++j) obs[j * STRIDE + k] = o[j];
    }
  }
  return far;
}

// The observations staged where they fit one tile, before the first system: as
// plain pairs if any time is a far one, which it returns.  Contains barriers.
template <int TILE, int ROWS>
__device__ __forceinline__ bool gn_prepare(const UniformArgs &a, bool staged_once, int tid,
                                           int nthreads, const Split3 &tr3, float jit2,
                                           float *obs) {
  const int npad = (a.n_obs + ROWS - 1) / ROWS * ROWS;
  bool far = false;
  if (staged_once)
    far = gn_stage<TILE>(a, 0, a.n_obs, npad, tid, nthreads, tr3, jit2, false, obs);
  far = __syncthreads_or(far);
  if (far) {
    for (int k = tid; k < a.n_obs; k += nthreads)
      sub_ds(split3(a.t[k]), tr3, obs[k], obs[TILE + k]);
    __syncthreads();
  }
  return far;
}

// One pair of observations of a lane (columns k, k + 1 of the staged tile):
// chi2 and gradient sums, and the rows of sqrt(w) J over their factors.
// dref = t_ref - t0; k0: the tile's first observation.
template <int J, int STRIDE, bool WIDE>
__device__ __forceinline__ void gn_pair(const UniformArgs &a, const float *obs, int k0, int k,
                                        float dref, const GradPlanetP *q,
                                        const float *tab, float gam, Kahan2 &acc, f32x2 &sum_a,
                                        GradSums (&g)[J], f32x2 (&u)[5 * J + 1]) {
  auto at = [&](int array) { return *reinterpret_cast<const f32x2 *>(obs + array * STRIDE + k); };
  f32x2 th = at(0), tl = at(1);
  if (WIDE) {
    float n_max = 0.0f;
#pragma unroll
    for (int j = 0; j < J; ++j) n_max = fmaxf(n_max, q[j].p.n);
    if (n_max > kPairExactFreq) plain_times(a.t, k0 + k, a.n_obs, th, tl);
  }
  GradTerms o[J];
  Kahan2 V = {dup2(gam), 0};
#pragma unroll
  for (int j = 0; j < J; ++j) o[j] = grad_terms<WIDE>(th, tl, q[j], tab, V);
  const f32x2 r = sub2(sub2(V.big, at(2)), add2(V.small, at(3)));
  const f32x2 sw = at(4), sr = mul2(sw, r), a2 = add2(sr, sr);
  kahan_add(acc, mul2(sr, sr));
  sum_a = fma2(a2, sw, sum_a);
  const f32x2 swdt = mul2(sw, add2(add2(th, tl), dup2(dref)));
#pragma unroll
  for (int j = 0; j < J; ++j) gn_add(g[j], o[j], q[j], sw, swdt, a2, u + 5 * j);
  u[5 * J] = sw;
}

// A warp's next kGnAhead systems, s0 + i stride, set up together: planet j of
// system i by lane i J + j into q[i J + j], gamma of system i by lane 16 + i (the
// lane's return value).  One system's setup is a chain of some 500
// instructions in J lanes; alone it took a tenth of the time of a system of
// 3 planets and 512 observations, and half of one of 1 and 256.  wide: bit l
// set if lane l's planet asks for the wide mean anomaly.
template <int J>
__device__ __forceinline__ float gn_setup_ahead(const UniformArgs &a, int64_t s0, int64_t stride,
                                                int lane, double t_ref, bool plain,
                                                GradPlanetP *q, unsigned &wide) {
  static_assert(kGnAhead * J <= 16, "planets in lanes 0 .. 15, gamma from lane 16");
  constexpr int NP = 5 * J + 1;
  bool brief = false;
  float gam = 0.0f;
  __syncwarp();                                        // the last systems' use of q
  if (lane < kGnAhead * J) {
    const int i = lane / J, j = lane - i * J;
    const int64_t s = s0 + i * stride;
    GradPlanetP p = {};
    if (s < a.n_sys && dbg_ok(a.invalid, s * NP + 5 * j + 4 < a.n_sys * NP, kDbgParam, s * NP)) {
      p = grad_setup_pair(a.params + s * NP + 5 * j, t_ref, a.t0, plain);
      brief = short_period(p.p);
    }
    q[lane] = p;
  } else if (lane >= 16 && lane < 16 + kGnAhead) {
    const int64_t s = s0 + (lane - 16) * stride;
    if (s < a.n_sys) gam = d2f(system_gamma_g(a.params + s * NP, J));
  }
  wide = __ballot_sync(0xffffffffu, brief);
  return gam;
}

// The planets of the warp's kGnAhead systems made plain pairs: the first far time
// of a series longer than a tile is met with the planets set up.
template <int J>
__device__ __forceinline__ void gn_ahead_plain(const UniformArgs &a, int64_t s0, int64_t stride,
                                               int lane, GradPlanetP *q) {
  constexpr int NP = 5 * J + 1;
  __syncwarp();
  if (lane < kGnAhead * J) {
    const int i = lane / J, j = lane - i * J;
    const int64_t s = s0 + i * stride;
    if (s < a.n_sys && dbg_ok(a.invalid, s * NP + 5 * j < a.n_sys * NP, kDbgParam, s * NP))
      planet_plain(q[lane].p, a.params[s * NP + 5 * j]);
  }
  __syncwarp();
}

// chi2 and gradient of a warp's system: the lanes' sums combined and written.
// scale: the factors of the rows' columns (gn_scale).
template <int J>
__device__ __forceinline__ void gn_write_grad(const UniformArgs &a, int64_t s, int lane,
                                              float poison, const Kahan2 &acc2, f32x2 sum_a,
                                              const GradSums (&g)[J], const float *scale,
                                              float *chi2_out, float *grad_out) {
  constexpr int NP = 5 * J + 1;
  Kahan acc = kahan_join(acc2);
  float sa = join2(sum_a);
  GradLane gl[J];
#pragma unroll
  for (int j = 0; j < J; ++j) gl[j] = grad_join(g[j]);
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    const Kahan o = {shfl_xor(acc.big, m), shfl_xor(acc.small, m)};
    kahan_merge(acc, o);
    sa += shfl_xor(sa, m);
#pragma unroll
    for (int j = 0; j < J; ++j) grad_combine(gl[j], m);
  }
  if (s >= a.n_sys) return;
  if (lane == 0) {
    const float value = kahan_value(acc) + poison;
    if (chi2_out) chi2_out[s] = value;
    note_invalid(a.invalid, value);
  }
  if (grad_out) {
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const float v[5] = {kahan_value(gl[j].P), gl[j].K, gl[j].e, gl[j].w, gl[j].M};
#pragma unroll
      for (int i = 0; i < 5; ++i)
        if (lane == ((5 * j + i) & 31))
          grad_out[s * NP + 5 * j + i] = __fmaf_rn(scale[5 * j + i], v[i], poison);
    }
    if (lane == ((5 * J) & 31)) grad_out[s * NP + 5 * J] = sa + poison;
  }
}

template <int J>
__global__ void __launch_bounds__(kGnWarps * 32)
gn_mixed_kernel(UniformArgs a, float *__restrict__ chi2_out, float *__restrict__ grad_out,
                float *__restrict__ jtj_out) {
  constexpr int NP = gn_np(J), MT = gn_mt(J), NT = gn_nt(J), ROW2 = gn_row2(J);
  constexpr int NTRI = NP * (NP + 1) / 2;
  extern __shared__ __align__(16) unsigned char smem[];
  const GnMixedLayout L(J, kGnObsTile);
  GradPlanetF *pl_s = reinterpret_cast<GradPlanetF *>(smem + L.pl);
  float *gam_s = reinterpret_cast<float *>(smem + L.gam);
  float4 *obs_s = reinterpret_cast<float4 *>(smem + L.obs);
  float4 *wt_s = reinterpret_cast<float4 *>(smem + L.w);
  float2 *u_all = reinterpret_cast<float2 *>(smem + L.u);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int block = kGnWarps * 32;
  const int64_t sys0 = (int64_t)blockIdx.x * kGnWarps;
  const int64_t s = sys0 + warp;
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  const Split3 tr3 = split3(t_ref), te3 = split3(a.t0);
  const float dref_f = (tr3.x0 - te3.x0) + (tr3.x1 - te3.x1);     // t_ref - t0
  const float jit2 = d2f(a.jitter2);

  for (int i = tid; i < kGnWarps * J; i += block) {
    const int64_t si = sys0 + i / J;
    GradPlanetF q = {};
    if (si < a.n_sys &&
        dbg_ok(a.invalid, si * NP + 5 * (i % J) + 4 < a.n_sys * NP, kDbgParam, si * NP))
      q = grad_setup_mixed(a.params + si * NP + 5 * (i % J), t_ref, a.t0);
    pl_s[i] = q;
  }
  for (int i = tid; i < kGnWarps; i += block)
    gam_s[i] = sys0 + i < a.n_sys ? d2f(system_gamma_g(a.params + (sys0 + i) * NP, J)) : 0.0f;
  for (int i = tid; i < kGnWarps * 32 * ROW2; i += block)
    u_all[i] = make_float2(0.0f, 0.0f);                           // incl. padding

  // The (hi, lo) pair of element (row r, column c) of U sits at
  // r * ROW2 + (c ^ ((r >> 2) & 3)): with ROW2 = 4 mod 16 both the row writes
  // (one row per lane) and the fragment loads touch 32 different banks in
  // each half-warp.
  float2 *u = u_all + warp * 32 * ROW2;
  const int gid = lane >> 2, tig = lane & 3;
  const int sw_row = (lane >> 2) & 3;
  Kahan acc = {0.0f, 0.0f};
  Kahan gP[J];
  float g[NP];
  float C[MT][NT][4];
#pragma unroll
  for (int i = 0; i < NP; ++i) g[i] = 0.0f;
#pragma unroll
  for (int j = 0; j < J; ++j) gP[j] = Kahan{0.0f, 0.0f};
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) C[mt][nt][i] = 0.0f;

  for (int k0 = 0; k0 < a.n_obs; k0 += kGnObsTile) {
    const int nk = min(kGnObsTile, a.n_obs - k0);
    __syncthreads();
    for (int k = tid; k < nk; k += block) {
      if (!dbg_ok(a.invalid, k0 + k < a.n_obs, kDbgObs, k0 + k)) continue;
      float th, tl, vh, vl;
      sub_ds(split3(a.t[k0 + k]), tr3, th, tl);
      split_d(a.v[k0 + k], vh, vl);
      obs_s[k] = make_float4(th, tl, vh, vl);
      const float sg = d2f(a.sigma[k0 + k]);
      const float var = __fmaf_rn(sg, sg, jit2);
      const float wk = var > 0.0f ? 1.0f / var : __int_as_float(0x7fc00000);
      wt_s[k] = make_float4(wk, th + dref_f, sqrtf(wk), 0.0f);
    }
    __syncthreads();
    const float gam = gam_s[warp];
    const GradPlanetF *q = pl_s + warp * J;
    for (int kb = 0; kb < nk; kb += 32) {
      const int k = kb + lane;
      float urow[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) urow[i] = 0.0f;
      if (k < nk) {
        const float4 o = obs_s[k];
        const float4 wt = wt_s[k];
        float sEj[J], cEj[J];
        Kahan V = {0.0f, 0.0f};
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const PlanetF p = q[j].base;
          const float M = mean_anomaly_mixed(o.x, o.y, p);
          kepler_f32_h(M, p.e, q[j].m, sEj[j], cEj[j]);
          kahan_add(V, velocity_mixed(p, sEj[j], cEj[j]));
        }
        const float r = __fadd_rn(__fsub_rn(V.big, o.z), __fsub_rn(gam, __fadd_rn(V.small, o.w)));
        const float wk = wt.x, wr = wk * r, a2 = 2.0f * wr;
        kahan_add(acc, wr * r);
        const float sw = wt.z;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const GradPlanetF qj = q[j];
          Partials<float> d;
          const float invD = rcp_fast(__fmaf_rn(-qj.base.e, cEj[j], 1.0f));
          velocity_partials(qj.base.e, qj.K, qj.cw, qj.sw, qj.beta, qj.ibeta, sEj[j], cEj[j], invD,
                            d);
          d.dP = d.dM * (-kTwoPiF * wt.y * qj.n2);
          kahan_add(gP[j], a2 * d.dP);
          g[5 * j + 1] = fmaf(a2, d.dK, g[5 * j + 1]);
          g[5 * j + 2] = fmaf(a2, d.de, g[5 * j + 2]);
          g[5 * j + 3] = fmaf(a2, d.dw, g[5 * j + 3]);
          g[5 * j + 4] = fmaf(a2, d.dM, g[5 * j + 4]);
          urow[5 * j + 0] = sw * d.dP;
          urow[5 * j + 1] = sw * d.dK;
          urow[5 * j + 2] = sw * d.de;
          urow[5 * j + 3] = sw * d.dw;
          urow[5 * j + 4] = sw * d.dM;
        }
        g[5 * J] += a2;
        urow[5 * J] = sw;
      }
#pragma unroll
      for (int i = 0; i < NP; ++i) u[lane * ROW2 + (i ^ sw_row)] = tf32_pair(urow[i]);
      __syncwarp();
      // H += U^T U: k-steps of 8 rows; A = U^T (16 x 8 per m-tile), B = U (8 x 8 per n-tile)
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        const float2 *r0 = u + (ks * 8 + tig) * ROW2;
        const float2 *r1 = r0 + 4 * ROW2;
        const int g0 = gid ^ ((2 * ks) & 3), g1 = gid ^ ((2 * ks + 1) & 3);   // row swizzles
        unsigned ah[MT][4], al[MT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
          const float2 x[4] = {r0[16 * mt + g0], r0[16 * mt + g0 + 8], r1[16 * mt + g1],
                               r1[16 * mt + g1 + 8]};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            ah[mt][i] = __float_as_uint(x[i].x);
            al[mt][i] = __float_as_uint(x[i].y);
          }
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          // columns 8 nt .. 8 nt + 7 of U: half h of m-tile nt / 2
          const int m = nt >> 1, h = nt & 1;
          const unsigned bh[2] = {ah[m][h], ah[m][2 + h]}, bl[2] = {al[m][h], al[m][2 + h]};
#pragma unroll
          for (int mt = 0; mt < MT; ++mt) {
            if (8 * nt + 7 >= 16 * mt) {        // a tile on or above the diagonal
              mma_tf32(C[mt][nt], al[mt], bh);
              mma_tf32(C[mt][nt], ah[mt], bl);
              mma_tf32(C[mt][nt], ah[mt], bh);
            }
          }
        }
      }
      __syncwarp();
    }
  }

  for (int m = 16; m >= 1; m >>= 1) {
    Kahan o = {shfl_xor(acc.big, m), shfl_xor(acc.small, m)};
    kahan_merge(acc, o);
#pragma unroll
    for (int j = 0; j < J; ++j) {
      Kahan op = {shfl_xor(gP[j].big, m), shfl_xor(gP[j].small, m)};
      kahan_merge(gP[j], op);
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) g[i] += shfl_xor(g[i], m);
  }
#pragma unroll
  for (int j = 0; j < J; ++j) g[5 * j] = kahan_value(gP[j]);
  if (s >= a.n_sys) return;
  const float poison = 0.0f * gam_s[warp];             // NaN for an invalid system
  if (lane == 0) {
    const float value = kahan_value(acc) + poison;
    if (chi2_out) chi2_out[s] = value;
    note_invalid(a.invalid, value);
  }
  if (grad_out) {
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (lane == (i & 31)) grad_out[s * NP + i] = g[i] + poison;
  }
  float *H = jtj_out + s * NTRI;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (8 * nt + 7 < 16 * mt) continue;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = 16 * mt + gid + (i >= 2 ? 8 : 0);
        const int col = 8 * nt + 2 * tig + (i & 1);
        if (row < NP && col < NP && col >= row) H[tri_index(NP, row, col)] = C[mt][nt][i] + poison;
      }
    }
}

// The pair form (kc_pair.cuh) with mma.sync, n_pl <= 3: the same chi2, bit for
// bit, as the tcgen05 kernel.  From four planets on its registers (192 to 255)
// leave too few warps: 20000 x 4 x 256 ran 267 us against 217 for the kernel
// above, 10000 x 8 x 256 476 against 296.
template <int J>
__global__ void __launch_bounds__(kGnWarps * 32)
gn_pair_kernel(UniformArgs a, float *__restrict__ chi2_out, float *__restrict__ grad_out,
               float *__restrict__ jtj_out) {
  constexpr int NP = gn_np(J), MT = gn_mt(J), NT = gn_nt(J), ROW2 = gn_row2(J);
  constexpr int NTRI = NP * (NP + 1) / 2, kTile = kTcObsTile;
  extern __shared__ __align__(16) unsigned char smem[];
  const GnPairLayout L(J, kTile);
  float *tab_s = reinterpret_cast<float *>(smem + L.tab);
  float *obs_s = reinterpret_cast<float *>(smem + L.obs);
  float2 *u_all = reinterpret_cast<float2 *>(smem + L.u);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int block = kGnWarps * 32;
  GradPlanetP *ahead = reinterpret_cast<GradPlanetP *>(smem + L.pl) + warp * kGnAhead * J;
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  const Split3 tr3 = split3(t_ref), te3 = split3(a.t0);
  const float dref_f = (tr3.x0 - te3.x0) + (tr3.x1 - te3.x1);     // t_ref - t0
  const float jit2 = d2f(a.jitter2);

  ang_tab_load<true>(tab_s, tid, block);
  for (int i = tid; i < kGnWarps * kGnRows * ROW2; i += block)
    u_all[i] = make_float2(0.0f, 0.0f);                           // incl. padding
  // observations that fit one tile are staged once for all of the CTA's systems
  const bool staged_once = a.n_obs <= kTile;
  bool plain = gn_prepare<kTile, kGnRows>(a, staged_once, tid, block, tr3, jit2, obs_s);

  // The (hi, lo) pair of element (row r, column c) of U sits at
  // r * ROW2 + (c ^ ((r >> 2) & 3)): with ROW2 = 4 mod 16 both the row writes
  // (rows l and 32 + l for lane l) and the fragment loads touch 32 different
  // banks in each half-warp.
  float2 *u = u_all + warp * kGnRows * ROW2;
  const int gid = lane >> 2, tig = lane & 3;
  const int sw_row = (lane >> 2) & 3;

  // a system per warp; the CTA's warps step together (they share the tile)
  const int64_t stride = (int64_t)gridDim.x * kGnWarps;
  int ahead_i = kGnAhead;                              // systems used of those set up
  unsigned wide_ahead = 0;
  float gam_ahead = 0.0f;
  for (int64_t s = (int64_t)blockIdx.x * kGnWarps + warp; s - warp < a.n_sys; s += stride) {
    if (ahead_i == kGnAhead) {
      ahead_i = 0;
      gam_ahead = gn_setup_ahead<J>(a, s, stride, lane, t_ref, plain, ahead, wide_ahead);
    }
    const GradPlanetP *q = ahead + ahead_i * J;
    const float gam = __shfl_sync(0xffffffffu, gam_ahead, 16 + ahead_i);
    bool wide = plain || ((wide_ahead >> (ahead_i * J)) & ((1u << J) - 1u)) != 0u;
    ++ahead_i;
    __syncwarp();
    Kahan2 acc = {0, 0};
    f32x2 sum_a = 0;
    GradSums g[J];
    float C[MT][NT][4];
#pragma unroll
    for (int j = 0; j < J; ++j) g[j] = GradSums{{0, 0}, 0, 0, 0, 0};
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) C[mt][nt][i] = 0.0f;

    for (int k0 = 0; k0 < a.n_obs; k0 += kTile) {
      const int nk = min(kTile, a.n_obs - k0);
      const int npad = (nk + kGnRows - 1) / kGnRows * kGnRows;
      if (!staged_once) {
        __syncthreads();
        const bool far = gn_stage<kTile>(a, k0, nk, npad, tid, block, tr3, jit2, plain, obs_s);
        if (__syncthreads_or(far) && !plain) {
          // the first far time: these systems again from the first tile
          plain = wide = true;
          gn_ahead_plain<J>(a, s - (ahead_i - 1) * stride, stride, lane, ahead);
          acc = Kahan2{0, 0};
          sum_a = 0;
#pragma unroll
          for (int j = 0; j < J; ++j) g[j] = GradSums{{0, 0}, 0, 0, 0, 0};
#pragma unroll
          for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
              for (int i = 0; i < 4; ++i) C[mt][nt][i] = 0.0f;
          k0 = -kTile;
          continue;
        }
      }
      for (int kb = 0; kb < npad; kb += kGnRows) {
        {
          f32x2 urow[NP];
          if (wide)
            gn_pair<J, kTile, true>(a, obs_s, k0, kb + 2 * lane, dref_f, q, tab_s, gam, acc,
                                    sum_a, g, urow);
          else
            gn_pair<J, kTile, false>(a, obs_s, k0, kb + 2 * lane, dref_f, q, tab_s, gam, acc,
                                     sum_a, g, urow);
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            u[lane * ROW2 + (i ^ sw_row)] = tf32_pair(lo2(urow[i]));
            u[(32 + lane) * ROW2 + (i ^ sw_row)] = tf32_pair(hi2(urow[i]));
          }
        }
        __syncwarp();
        // H += U^T U: k-steps of 8 rows, as in gn_mixed_kernel
#pragma unroll
        for (int ks = 0; ks < kGnRows / 8; ++ks) {
          const float2 *r0 = u + (ks * 8 + tig) * ROW2;
          const float2 *r1 = r0 + 4 * ROW2;
          const int g0 = gid ^ ((2 * ks) & 3), g1 = gid ^ ((2 * ks + 1) & 3);   // row swizzles
          const float2 x[4] = {r0[g0], r0[g0 + 8], r1[g1], r1[g1 + 8]};
          static_assert(MT == 1, "n_pl <= 3");
          unsigned ah[4], al[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            ah[i] = __float_as_uint(x[i].x);
            al[i] = __float_as_uint(x[i].y);
          }
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const unsigned bh[2] = {ah[nt], ah[2 + nt]}, bl[2] = {al[nt], al[2 + nt]};
            mma_tf32(C[0][nt], al, bh);
            mma_tf32(C[0][nt], ah, bl);
            mma_tf32(C[0][nt], ah, bh);
          }
        }
        __syncwarp();
      }
    }

    float scale[NP];                       // the rows' columns over their factors
#pragma unroll
    for (int p = 0; p < NP; ++p) scale[p] = gn_scale(q, J, p);
    const float poison = 0.0f * gam;                   // NaN for an invalid system
    gn_write_grad<J>(a, s, lane, poison, acc, sum_a, g, scale, chi2_out, grad_out);
    if (s < a.n_sys) {
      float *H = jtj_out + s * NTRI;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = gid + (i >= 2 ? 8 : 0);
          const int col = 8 * nt + 2 * tig + (i & 1);
          if (row < NP && col < NP && col >= row)
            H[tri_index(NP, row, col)] =
                __fmaf_rn(gn_scale(q, J, row) * gn_scale(q, J, col), C[0][nt][i], poison);
        }
    }
  }
}

// ---------------------------------------------- Gauss-Newton on tcgen05
//
// The same pass with the U^T U update on the fifth-generation tensor cores:
// the operands come from shared memory through matrix descriptors, the
// accumulator stays in tensor memory (TMEM) for the whole launch, and one
// thread issues each batch's MMAs, so the warps evaluating observations
// spend no issue slots or shared-memory loads on the contraction.  The
// smallest tcgen05 tile is M = 64 rows, four times one system's 16 (n_pl
// <= 3: 5 n_pl + 1 <= 16 parameters; rows beyond them never reach a kept
// entry), so the CTA's four warps write their systems' U^T rows into one
// 64-row tile (rows 16 w .. 16 w + 15 for warp w; TF32 (hi, lo) pairs as in
// gn_mixed_kernel, in two tiles, K-major, 128-byte swizzle), and thread 0
// issues the batch's MMAs (M = 64, N = 64, K = 8 per step).  H = U^T U is
// symmetric, so of the three products of the split, hi hi^T + lo hi^T +
// hi lo^T, the last is the transpose of the second: two accumulators in
// TMEM, D1 += hi hi^T and D2 += lo hi^T (two MMAs per K step, not three),
// give H = D1 + D2 + D2^T in the epilogue.  The four diagonal 16 x 16
// blocks are kept; 3/4 of the products are cross-system terms that are
// thrown away.  A batch is 64 observations, two per lane in packed form
// (kc_pair.cuh); its tile is two 64 x 32 halves.  The columns go in over their
// per-planet factors (gn_add), which the epilogue applies to H.  The order of the observations along K is free (the
// sum runs over all of them), so lane l puts its pair at K = 2l and 2l + 1
// and writes both words of an element with one 8-byte store.
// One tile suffices: a warp rewrites it only after evaluating the next 64
// observations, by which time the MMAs that read it have long completed
// (its lane 0 still waits on the mbarrier their commit arrives on).  A CTA
// barrier per batch hands the written tile to the issuing thread (an earlier
// version ran 822 us on 65536 x 3 x 512 this way against 891 us with a "full"
// mbarrier that let the other warps run a batch ahead of warp 0).  The CTAs
// are persistent: the table and the observations are staged once, and a warp
// sets four of its systems up at a time.  On 65536 x 3 x 512: 732 us with the
// scalar evaluation, 685 packed, 640 persistent, 619 with the setups
// together.  Bound by latency: 16 warps per SM (registers, TMEM and shared
// memory all end there), issue slots 44 % busy.  With
// M = 64 the accumulator's row r sits in TMEM lane 32 (r / 16) + r % 16, so
// warp w reads its system's blocks from its own lanes 32 w .. 32 w + 15,
// columns 16 w .. 16 w + 15 (D1) and 64 + 16 w .. 64 + 16 w + 15 (D2), and
// transposes D2's block through shared memory.  Every wait is bounded; a
// wait that gives up makes the CTA's results NaN (counted by the
// invalid-system counter) and the TMEM is still freed.

constexpr int kTcHalfBytes = 64 * 32 * 4;       // 64 rows x 32 observations, TF32
constexpr int kTcBatch = 64;                    // observations per batch
constexpr int kTcCols = 128;                    // TMEM columns per CTA: D1, D2
constexpr uint64_t kTcWaitLimit = 20000000;     // ns an mbarrier wait may take (20 ms)

struct GnTcLayout {
  size_t u, tab, pl, obs, bar, slot, total;
  __host__ __device__ GnTcLayout(int J) {
    u = 0;                                       // hi halves, then lo halves: 1024-aligned
    tab = u + 4 * kTcHalfBytes;
    pl = tab + sizeof(AngTab);
    obs = align_up(pl + sizeof(GradPlanetP) * kGnWarps * kGnAhead * J, 16);
    bar = align_up(obs + sizeof(float) * 5 * kTcObsTile, 8);
    slot = bar + sizeof(uint64_t);
    total = align_up(slot + 16, 16) + 1024;     // 1024 bytes to align the base
  }
};

// Lane 0 waits; the warp learns the outcome (and is ordered after it).
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, uint64_t limit, int lane) {
  bool ok = true;
  if (lane == 0) ok = tc::mbar_wait(bar, parity, limit);
  return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

// Writes the lane's two observations, columns 2 l and 2 l + 1 of U^T for
// lane l, into the tile: element (row 16 warp + p, column c) of a half
// (columns 0-31 and 32-63 of the batch) sits in 8-row group 2 warp + p / 8
// (1024 bytes each), row p % 8 (128 bytes), 16-byte chunk (c / 4) ^ (p % 8),
// word c % 4, so the pair is one aligned 8-byte word.  `rows` points at the
// lane's half, 8-row group and word; `lane_q` is its chunk before the
// swizzle.  The hi parts are TF32 (low 13 bits cleared), so that hi + lo is
// exact; the lo parts are stored whole: the tensor core takes their upper
// 19 bits, as clearing the rest here would (were it to round them instead,
// an element would move by less than 2^-20 of itself).
template <int NP>
__device__ __forceinline__ void gn_tc_store(unsigned char *rows, uint32_t lane_q,
                                            const f32x2 (&u)[NP]) {
  constexpr unsigned kTf32Mask = 0xffffe000u;
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const f32x2 h = pack2(__uint_as_float(__float_as_uint(lo2(u[p])) & kTf32Mask),
                          __uint_as_float(__float_as_uint(hi2(u[p])) & kTf32Mask));
    const uint32_t off = (p >> 3) * 1024 + (p & 7) * 128 + ((lane_q ^ (p & 7)) << 4);
    *reinterpret_cast<f32x2 *>(rows + off) = h;
    *reinterpret_cast<f32x2 *>(rows + 2 * kTcHalfBytes + off) = sub2(u[p], h);
  }
}

template <int J>
__global__ void __launch_bounds__(kGnWarps * 32, 4)
gn_mixed_tc_kernel(UniformArgs a, float *__restrict__ chi2_out, float *__restrict__ grad_out,
                   float *__restrict__ jtj_out) {
  constexpr int NP = gn_np(J);
  constexpr int NTRI = NP * (NP + 1) / 2;
  static_assert(NP <= 16, "one system's U^T fits 16 rows of the M = 64 tile");
  static_assert(kGnWarps == 4, "four systems per M = 64 tile");
  constexpr uint32_t IDESC = tc::idesc_tf32(64, 64);
  constexpr int kThreads = kGnWarps * 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char *smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
  const GnTcLayout L(J);
  float *tab_s = reinterpret_cast<float *>(smem + L.tab);
  float *obs_s = reinterpret_cast<float *>(smem + L.obs);       // th, tl, v hi, v lo, sqrt w
  uint64_t *bar = reinterpret_cast<uint64_t *>(smem + L.bar);   // commits of the MMAs
  uint32_t *slot = reinterpret_cast<uint32_t *>(smem + L.slot);
  unsigned char *tiles = smem + L.u;
  const uint32_t tiles_a = tc::smem_u32(tiles), bar_a = tc::smem_u32(bar);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  GradPlanetP *ahead = reinterpret_cast<GradPlanetP *>(smem + L.pl) + warp * kGnAhead * J;

  if (warp == 0) tc::tmem_alloc(tc::smem_u32(slot), kTcCols);
  if (tid == 0) {
    tc::mbar_init(bar_a, 1);                   // one commit per batch
    tc::mbar_init_fence();
  }
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  const Split3 tr3 = split3(t_ref), te3 = split3(a.t0);
  const float dref_f = (tr3.x0 - te3.x0) + (tr3.x1 - te3.x1);     // t_ref - t0
  const float jit2 = d2f(a.jitter2);
  ang_tab_load<true>(tab_s, tid, kThreads);
  // observations that fit one tile are staged once for all of the CTA's systems
  const bool staged_once = a.n_obs <= kTcObsTile;
  tc::fence_before_sync();
  bool plain =
      gn_prepare<kTcObsTile, kTcBatch>(a, staged_once, tid, kThreads, tr3, jit2, obs_s);
  tc::fence_after_sync();
  const uint32_t taddr = *slot;

  // lane l: columns 2 l, 2 l + 1 of the batch, in half l / 16
  const uint32_t lane_q = (uint32_t)(lane & 15) >> 1;
  unsigned char *my_rows = tiles + (lane >> 4) * kTcHalfBytes + 2048 * warp + 8 * (lane & 1);
  // The descriptors of the batch's K steps differ from the tile's in the
  // start address alone (bits 0-13: the address / 16; the tiles end below
  // 2^18 bytes, so an offset adds without a carry out of the field).
  const uint64_t dtile = tc::desc_kmajor_sw128(tiles_a);
  uint32_t nb = 0;                                   // batches (commits) so far
  bool ok = true;

  // Four systems at a time, one per warp.  A warp sets its own system up; the
  // barrier of a batch is the only one the systems share, and the first one
  // of a group also orders the group's first MMA (which overwrites the
  // accumulators) after every warp's read of the group before.
  const int64_t stride = (int64_t)gridDim.x * kGnWarps;
  int ahead_i = kGnAhead;                            // systems used of those set up
  unsigned wide_ahead = 0;
  float gam_ahead = 0.0f;
  for (int64_t s = (int64_t)blockIdx.x * kGnWarps + warp; s - warp < a.n_sys; s += stride) {
    if (ahead_i == kGnAhead) {
      ahead_i = 0;
      gam_ahead = gn_setup_ahead<J>(a, s, stride, lane, t_ref, plain, ahead, wide_ahead);
    }
    const GradPlanetP *q = ahead + ahead_i * J;
    const float gam = __shfl_sync(0xffffffffu, gam_ahead, 16 + ahead_i);
    bool wide = plain || ((wide_ahead >> (ahead_i * J)) & ((1u << J) - 1u)) != 0u;
    ++ahead_i;
    __syncwarp();
    Kahan2 acc2 = {0, 0};
    f32x2 sum_a = 0;
    GradSums g[J];
#pragma unroll
    for (int j = 0; j < J; ++j) g[j] = GradSums{{0, 0}, 0, 0, 0, 0};
    uint32_t nb0 = nb;

    for (int k0 = 0; k0 < a.n_obs; k0 += kTcObsTile) {
      const int nk = min(kTcObsTile, a.n_obs - k0);
      const int npad = (nk + kTcBatch - 1) / kTcBatch * kTcBatch;
      if (!staged_once) {
        __syncthreads();
        const bool far =
            gn_stage<kTcObsTile>(a, k0, nk, npad, tid, kThreads, tr3, jit2, plain, obs_s);
        if (__syncthreads_or(far) && !plain) {
          // the first far time: these systems again from the first tile (whose
          // first MMA overwrites the accumulators)
          plain = wide = true;
          gn_ahead_plain<J>(a, s - (ahead_i - 1) * stride, stride, lane, ahead);
          acc2 = Kahan2{0, 0};
          sum_a = 0;
#pragma unroll
          for (int j = 0; j < J; ++j) g[j] = GradSums{{0, 0}, 0, 0, 0, 0};
          nb0 = nb;
          k0 = -kTcObsTile;
          continue;
        }
      }
      for (int kb = 0; kb < npad; kb += kTcBatch) {
        f32x2 u[NP];
        if (wide)
          gn_pair<J, kTcObsTile, true>(a, obs_s, k0, kb + 2 * lane, dref_f, q, tab_s, gam, acc2,
                                       sum_a, g, u);
        else
          gn_pair<J, kTcObsTile, false>(a, obs_s, k0, kb + 2 * lane, dref_f, q, tab_s, gam, acc2,
                                        sum_a, g, u);
        if (nb > 0 && ok)                  // the MMAs that read the tile before
          ok = warp_wait(bar_a, (nb - 1) & 1u, kTcWaitLimit, lane);
        gn_tc_store<NP>(my_rows, lane_q, u);
        tc::fence_proxy_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        if (tid == 0) {
          tc::fence_after_sync();
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {
            // K step ks: columns 8 ks .. 8 ks + 7 of the batch, in half ks / 4
            const uint32_t off = ((ks >> 2) * kTcHalfBytes + 32 * (ks & 3)) >> 4;
            const uint64_t hi = dtile + off, lo = dtile + off + (2 * kTcHalfBytes >> 4);
            const uint32_t accumulate = ((nb - nb0) | ks) != 0;
            tc::mma_tf32(taddr, hi, hi, IDESC, accumulate);                 // D1 += hi hi^T
            tc::mma_tf32(taddr + kTcCols / 2, lo, hi, IDESC, accumulate);   // D2 += lo hi^T
          }
          tc::commit(bar_a);
        }
        ++nb;
      }
    }

    // Every MMA is complete once the last commit's phase is; a longer wait if
    // a wait gave up before.
    float h[16];
    if (nb > nb0) {
      const bool last_ok = warp_wait(bar_a, (nb - 1) & 1u, ok ? kTcWaitLimit : 4 * kTcWaitLimit,
                                     lane);
      ok = ok && last_ok;
      tc::fence_after_sync();
      const uint32_t blk = taddr + ((uint32_t)(32 * warp) << 16) + 16u * warp;
      float h2[16];
      tc::tmem_ld16(blk, h);
      tc::tmem_ld16(blk + kTcCols / 2, h2);
      // H = D1 + D2 + D2^T: lane r < 16 holds row r of both blocks; D2's is
      // transposed through 16 x 17 floats of the warp's own 2 KB of the
      // operand tile (no MMA reads the tile any more, and only this warp
      // writes there).
      float *tr = reinterpret_cast<float *>(tiles + 2048 * warp);
      __syncwarp();
      if (lane < 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) tr[lane * 17 + i] = h2[i];
      }
      __syncwarp();
      if (lane < 16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) h[i] += h2[i] + tr[i * 17 + lane];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i) h[i] = 0.0f;
    }

    // NaN for an invalid system, or where a wait on the tensor cores gave up
    const float poison = ok ? 0.0f * gam : __int_as_float(0x7fc00000);
    float scale[NP];                       // the rows' columns over their factors
#pragma unroll
    for (int p = 0; p < NP; ++p) scale[p] = gn_scale(q, J, p);
    gn_write_grad<J>(a, s, lane, poison, acc2, sum_a, g, scale, chi2_out, grad_out);
    if (s < a.n_sys && lane < NP) {
      float *H = jtj_out + s * NTRI;
      const float mine = gn_scale(q, J, lane);
#pragma unroll
      for (int c = 0; c < NP; ++c)
        if (c >= lane) H[tri_index(NP, lane, c)] = __fmaf_rn(mine * scale[c], h[c], poison);
    }
  }

  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_free(taddr, kTcCols);
  }
}

template <int J>
__global__ void __launch_bounds__(kGnWarpsD * 32)
gn_f64_kernel(UniformArgs a, double *__restrict__ chi2_out, double *__restrict__ grad_out,
              double *__restrict__ jtj_out) {
  constexpr int NP = gn_np(J), ROWD = NP | 1;
  constexpr int NTRI = NP * (NP + 1) / 2, E = (NTRI + 31) / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const GnF64Layout L(J, kGnObsTile);
  GradPlanetD *pl_s = reinterpret_cast<GradPlanetD *>(smem + L.pl);
  double *gam_s = reinterpret_cast<double *>(smem + L.gam);
  ObsGD *obs_s = reinterpret_cast<ObsGD *>(smem + L.obs);
  short2 *pq_s = reinterpret_cast<short2 *>(smem + L.pq);
  double *u_all = reinterpret_cast<double *>(smem + L.u);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int block = kGnWarpsD * 32;
  const int64_t sys0 = (int64_t)blockIdx.x * kGnWarpsD;
  const int64_t s = sys0 + warp;
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  const double dref = t_ref - a.t0;

  for (int i = tid; i < kGnWarpsD * J; i += block) {
    const int64_t si = sys0 + i / J;
    GradPlanetD q = {};
    if (si < a.n_sys &&
        dbg_ok(a.invalid, si * NP + 5 * (i % J) + 4 < a.n_sys * NP, kDbgParam, si * NP))
      q = grad_setup_f64(a.params + si * NP + 5 * (i % J), dref);
    pl_s[i] = q;
  }
  for (int i = tid; i < kGnWarpsD; i += block)
    gam_s[i] = sys0 + i < a.n_sys ? system_gamma_g(a.params + (sys0 + i) * NP, J) : 0.0;
  for (int p = tid; p < NP; p += block) {               // packed (p, q) table
    const int base = p * NP - (p * (p - 1)) / 2;
    for (int q = p; q < NP; ++q) pq_s[base + q - p] = make_short2((short)p, (short)q);
  }

  double *u = u_all + warp * 32 * ROWD;
  double acc = 0.0, g[NP], h[E];
#pragma unroll
  for (int i = 0; i < NP; ++i) g[i] = 0.0;
#pragma unroll
  for (int i = 0; i < E; ++i) h[i] = 0.0;

  for (int k0 = 0; k0 < a.n_obs; k0 += kGnObsTile) {
    const int nk = min(kGnObsTile, a.n_obs - k0);
    __syncthreads();
    for (int k = tid; k < nk; k += block) {
      if (!dbg_ok(a.invalid, k0 + k < a.n_obs, kDbgObs, k0 + k)) continue;
      ObsGD o;
      const double tk = a.t[k0 + k];
      o.tau = tk - t_ref;
      o.v = a.v[k0 + k];
      o.w = inv_variance_g(a.sigma[k0 + k], a.jitter2);
      o.dt = tk - a.t0;
      obs_s[k] = o;
    }
    __syncthreads();
    const double gam = gam_s[warp];
    const GradPlanetD *q = pl_s + warp * J;
    bool hi = false;                        // uniform: the warp holds one system
#pragma unroll
    for (int j = 0; j < J; ++j) hi = hi || q[j].base.e > (double)kEccFast;
    for (int kb = 0; kb < nk; kb += 32) {
      const int k = kb + lane;
      double urow[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) urow[i] = 0.0;
      if (k < nk) {
        const ObsGD o = obs_s[k];
        double sEj[J], cEj[J];
        double V = gam;
        with_high_e(hi, [&](auto tag) {
          constexpr bool HI = decltype(tag)::value;
#pragma unroll
          for (int j = 0; j < J; ++j) {
            const PlanetD p = q[j].base;
            const double M = mean_anomaly_f64(o.tau, p);
            kepler_f64<HI>(M, p.e, sEj[j], cEj[j]);
            V = velocity_add_f64(p, sEj[j], cEj[j], V);
          }
        });
        const double r = V - o.v;
        const double a2 = 2.0 * o.w * r;
        acc = fma(o.w * r, r, acc);
        const double sw = sqrt(o.w);
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const GradPlanetD qj = q[j];
          Partials<double> d;
          const double invD = 1.0 / fma(-qj.base.e, cEj[j], 1.0);
          velocity_partials(qj.base.e, qj.K, qj.cw, qj.sw, qj.base.beta, qj.ibeta, sEj[j], cEj[j],
                            invD, d);
          d.dP = d.dM * (-kTwoPi * o.dt * qj.n2);
          g[5 * j + 0] = fma(a2, d.dP, g[5 * j + 0]);
          g[5 * j + 1] = fma(a2, d.dK, g[5 * j + 1]);
          g[5 * j + 2] = fma(a2, d.de, g[5 * j + 2]);
          g[5 * j + 3] = fma(a2, d.dw, g[5 * j + 3]);
          g[5 * j + 4] = fma(a2, d.dM, g[5 * j + 4]);
          urow[5 * j + 0] = sw * d.dP;
          urow[5 * j + 1] = sw * d.dK;
          urow[5 * j + 2] = sw * d.de;
          urow[5 * j + 3] = sw * d.dw;
          urow[5 * j + 4] = sw * d.dM;
        }
        g[5 * J] += a2;
        urow[5 * J] = sw;
      }
#pragma unroll
      for (int i = 0; i < NP; ++i) u[lane * ROWD + i] = urow[i];
      __syncwarp();
      const int rows = min(32, nk - kb);
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int e = lane + 32 * i;
        if (e < NTRI) {
          const short2 pq = pq_s[e];
          double sum = 0.0;
          for (int rr = 0; rr < rows; ++rr) sum = fma(u[rr * ROWD + pq.x], u[rr * ROWD + pq.y], sum);
          h[i] += sum;
        }
      }
      __syncwarp();
    }
  }

  for (int m = 16; m >= 1; m >>= 1) {
    acc += shfl_xor(acc, m);
#pragma unroll
    for (int i = 0; i < NP; ++i) g[i] += shfl_xor(g[i], m);
  }
  if (s >= a.n_sys) return;
  const double poison = 0.0 * gam_s[warp];
  if (lane == 0) {
    const double value = acc + poison;
    if (chi2_out) chi2_out[s] = value;
    note_invalid(a.invalid, value);
  }
  if (grad_out) {
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (lane == (i & 31)) grad_out[s * NP + i] = g[i] + poison;
  }
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int e = lane + 32 * i;
    if (e < NTRI) jtj_out[s * NTRI + e] = h[i] + poison;
  }
}

template <typename Kern>
cudaError_t set_smem(Kern k, size_t bytes) {
  return raise_smem_limit(reinterpret_cast<const void *>(k), bytes);
}

}  // namespace

// Launch shape of a gradient tile: as many observations at a time as fit
// beside the planets of the CTA's systems, and a smaller CTA where the planets
// alone do not fit (tiles of few threads per system).
struct GradShape {
  int block, obs_tile;
  size_t smem;
};
enum class GradKernel { F64, Packed, Scalar };
static GradShape grad_shape(int n_pl, const Tile &t, GradKernel kernel) {
  GradShape f{t.block, t.obs_tile, 0};
  auto bytes = [&] {
    const int ST = f.block / t.G;
    if (kernel == GradKernel::F64) return F64GradLayout(ST, n_pl, f.obs_tile).total;
    if (kernel == GradKernel::Scalar) return ScalarGradLayout(ST, n_pl, f.obs_tile).total;
    return MixedGradLayout(ST, n_pl, grad_tile(f.obs_tile, t.G)).total;
  };
  constexpr size_t kMax = 227 * 1024;
  while (bytes() > kMax) {
    if (f.obs_tile > 32)
      f.obs_tile = (f.obs_tile + 1) / 2;
    else if (f.block > 32)
      f.block = (f.block / 2 + 31) / 32 * 32;
    else
      break;
  }
  f.smem = bytes();
  return f;
}

#define KC_DISPATCH_J(J, MACRO) \
  switch (J) {                  \
    case 1: MACRO(1); break;    \
    case 2: MACRO(2); break;    \
    case 3: MACRO(3); break;    \
    case 4: MACRO(4); break;    \
    case 5: MACRO(5); break;    \
    case 6: MACRO(6); break;    \
    case 7: MACRO(7); break;    \
    case 8: MACRO(8); break;    \
    default: return cudaErrorInvalidValue; \
  }

cudaError_t launch_grad_mixed(const UniformArgs &a, const Tile &tile, float *chi2, float *grad,
                              cudaStream_t st) {
  if (tile.G > 32) return cudaErrorInvalidValue;
  const GradShape f = grad_shape(a.n_pl, tile, GradKernel::Packed);
  const int ST = f.block / tile.G;
  const int grid = (int)((a.n_sys + ST - 1) / ST);
  cudaError_t err = cudaSuccess;
#define KC_LAUNCH(JJ)                                                                    \
  err = set_smem(grad_mixed_kernel<JJ>, f.smem);                                         \
  if (err == cudaSuccess)                                                                \
    grad_mixed_kernel<JJ><<<grid, f.block, f.smem, st>>>(a, tile.G, f.obs_tile, chi2, grad);
  KC_DISPATCH_J(a.n_pl, KC_LAUNCH)
#undef KC_LAUNCH
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

cudaError_t launch_grad_scalar(const UniformArgs &a, const Tile &tile, float *chi2, float *grad,
                               cudaStream_t st, bool nll) {
  if (tile.G > 32) return cudaErrorInvalidValue;
  const GradShape f = grad_shape(a.n_pl, tile, GradKernel::Scalar);
  const int ST = f.block / tile.G;
  const int grid = (int)((a.n_sys + ST - 1) / ST);
  cudaError_t err = cudaSuccess;
#define KC_LAUNCH_NLL(JJ, NN)                                                                   \
  err = set_smem(grad_scalar_kernel<JJ, NN>, f.smem);                                           \
  if (err == cudaSuccess)                                                                       \
    grad_scalar_kernel<JJ, NN><<<grid, f.block, f.smem, st>>>(a, tile.G, f.obs_tile, chi2, grad);
#define KC_LAUNCH(JJ)                      \
  if (nll) {                               \
    KC_LAUNCH_NLL(JJ, true)                \
  } else {                                 \
    KC_LAUNCH_NLL(JJ, false)               \
  }
  KC_DISPATCH_J(a.n_pl, KC_LAUNCH)
#undef KC_LAUNCH
#undef KC_LAUNCH_NLL
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

cudaError_t launch_grad_f64(const UniformArgs &a, const Tile &tile, double *chi2, double *grad,
                            cudaStream_t st, bool nll) {
  if (tile.G > 32) return cudaErrorInvalidValue;
  const GradShape f = grad_shape(a.n_pl, tile, GradKernel::F64);
  const size_t smem = f.smem;
  const int ST = f.block / tile.G;
  const int grid = (int)((a.n_sys + ST - 1) / ST);
  cudaError_t err = cudaSuccess;
#define KC_LAUNCH_NLL(JJ, NN)                                                                 \
  err = set_smem(grad_f64_kernel<JJ, NN>, smem);                                              \
  if (err == cudaSuccess)                                                                     \
    grad_f64_kernel<JJ, NN><<<grid, f.block, smem, st>>>(a, tile.G, f.obs_tile, chi2,           \
                                                            grad);
#define KC_LAUNCH(JJ)                      \
  if (nll) {                               \
    KC_LAUNCH_NLL(JJ, true)                \
  } else {                                 \
    KC_LAUNCH_NLL(JJ, false)               \
  }
  KC_DISPATCH_J(a.n_pl, KC_LAUNCH)
#undef KC_LAUNCH
#undef KC_LAUNCH_NLL
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

// The pair form with mma.sync (split 0, n_pl <= 3): persistent, as many CTAs
// as are resident at once.
template <int J>
cudaError_t launch_gn_pair(const UniformArgs &a, void *chi2, void *grad, void *jtj,
                           cudaStream_t st) {
  const size_t smem = GnPairLayout(J, kTcObsTile).total;
  cudaError_t err = set_smem(gn_pair_kernel<J>, smem);
  if (err != cudaSuccess) return err;
  int per_sm = 0;
  err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gn_pair_kernel<J>, kGnWarps * 32,
                                                      smem);
  if (err != cudaSuccess) return err;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int64_t groups = (a.n_sys + kGnWarps - 1) / kGnWarps;
  const int grid = (int)std::min<int64_t>(groups, (int64_t)sm_count() * per_sm);
  gn_pair_kernel<J><<<grid, kGnWarps * 32, smem, st>>>(a, (float *)chi2, (float *)grad,
                                                       (float *)jtj);
  return cudaGetLastError();
}

// The tcgen05 variant (split 4): n_pl <= 3.  Every resident CTA holds
// kTcCols TMEM columns, so the launch is refused unless the SM's 512
// columns cover all CTAs that can be resident at once (an allocation would
// otherwise wait for another CTA to finish).
template <int J>
cudaError_t launch_gn_tc(const UniformArgs &a, void *chi2, void *grad, void *jtj,
                         cudaStream_t st) {
  const size_t smem = GnTcLayout(J).total;
  cudaError_t err = set_smem(gn_mixed_tc_kernel<J>, smem);
  if (err != cudaSuccess) return err;
  int per_sm = 0;
  err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gn_mixed_tc_kernel<J>,
                                                      kGnWarps * 32, smem);
  if (err != cudaSuccess) return err;
  if (per_sm < 1 || per_sm * kTcCols > 512) return cudaErrorInvalidConfiguration;
  // persistent: the resident CTAs take the groups of four systems in turn.
  // As many as the SM's TMEM, shared memory and registers hold (the occupancy
  // query counts one for a kernel that allocates TMEM).
  const int64_t groups = (a.n_sys + kGnWarps - 1) / kGnWarps;
  const int fit = std::min(512 / kTcCols, (int)(228 * 1024 / (smem + 1024)));
  const int grid = (int)std::min<int64_t>(groups, (int64_t)sm_count() * std::max(fit, 1));
  gn_mixed_tc_kernel<J><<<grid, kGnWarps * 32, smem, st>>>(a, (float *)chi2, (float *)grad,
                                                           (float *)jtj);
  return cudaGetLastError();
}

// Without a tuned entry the mixed Gauss-Newton kernel updates U^T U on
// tcgen05 where it can (n_pl <= 3): 65536 systems x 3 planets x 512 observations
// take 617 us against 713 with mma.sync, 20000 x 2 x 400 147 against 164.  One
// planet's evaluation is too short to hide the hand-off to the tensor core, and
// from some 128 observations on mma.sync is the faster there (65536 x 1 x 512 367
// against 412 us, 20000 x 1 x 256 74 against 78); but its H is three times as far
// off (2.9e-6 against 9.4e-7 of sqrt(H_pp H_qq) at 300 observations, rms, 8.9e-6
// against 2.8e-6 at 900), so it is taken only where it is asked for.
int gn_default_variant(int n_pl) { return n_pl <= 3 ? 4 : 0; }

bool gn_variant_ok(int variant, int n_pl) {
  return variant == 0 || (variant == 4 && n_pl >= 1 && n_pl <= 3);
}

cudaError_t launch_gauss_newton(const UniformArgs &a, bool f64, void *chi2, void *grad,
                                void *jtj, cudaStream_t st, int variant) {
  cudaError_t err = cudaSuccess;
  if (!f64 && variant != 0) {
    if (!gn_variant_ok(variant, a.n_pl)) return cudaErrorInvalidValue;
    switch (a.n_pl) {
      case 1: return launch_gn_tc<1>(a, chi2, grad, jtj, st);
      case 2: return launch_gn_tc<2>(a, chi2, grad, jtj, st);
      default: return launch_gn_tc<3>(a, chi2, grad, jtj, st);
    }
  }
  if (f64) {
    const int grid = (int)((a.n_sys + kGnWarpsD - 1) / kGnWarpsD);
#define KC_LAUNCH(JJ)                                                                        \
  {                                                                                          \
    const size_t smem = GnF64Layout(JJ, kGnObsTile).total;                                   \
    err = set_smem(gn_f64_kernel<JJ>, smem);                                                 \
    if (err == cudaSuccess)                                                                  \
      gn_f64_kernel<JJ><<<grid, kGnWarpsD * 32, smem, st>>>(a, (double *)chi2, (double *)grad, \
                                                            (double *)jtj);                  \
  }
    KC_DISPATCH_J(a.n_pl, KC_LAUNCH)
#undef KC_LAUNCH
  } else {
    const int grid = (int)((a.n_sys + kGnWarps - 1) / kGnWarps);
#define KC_LAUNCH(JJ)                                                                     \
  {                                                                                       \
    const size_t smem = GnMixedLayout(JJ, kGnObsTile).total;                              \
    err = set_smem(gn_mixed_kernel<JJ>, smem);                                            \
    if (err == cudaSuccess)                                                               \
      gn_mixed_kernel<JJ><<<grid, kGnWarps * 32, smem, st>>>(a, (float *)chi2, (float *)grad, \
                                                             (float *)jtj);               \
  }
    switch (a.n_pl) {
      case 1: return launch_gn_pair<1>(a, chi2, grad, jtj, st);
      case 2: return launch_gn_pair<2>(a, chi2, grad, jtj, st);
      case 3: return launch_gn_pair<3>(a, chi2, grad, jtj, st);
      case 4: KC_LAUNCH(4) break;
      case 5: KC_LAUNCH(5) break;
      case 6: KC_LAUNCH(6) break;
      case 7: KC_LAUNCH(7) break;
      case 8: KC_LAUNCH(8) break;
      default: return cudaErrorInvalidValue;
    }
#undef KC_LAUNCH
  }
  if (err != cudaSuccess) return err;
  return cudaGetLastError();
}

}  // namespace kc
