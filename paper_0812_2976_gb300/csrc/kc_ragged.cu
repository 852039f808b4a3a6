// kc_ragged.cu -- ragged batches: systems with their own planet count and
// their own observations, evaluated by one persistent kernel that takes
// whole systems from a device work queue, replayed as a CUDA graph.
//
// The paper evaluates uniform batches (every model of one star shares the
// observations, Sec. 4.1).  A ragged batch (n_obs 16..1024, n_pl 1..6 per
// system) varies the work per system by ~400x, so a static split of
// systems over threads leaves most SMs idle at the end.  Here:
//  - a plan orders the systems by planet count, then by decreasing work
//    (n_pl * n_obs), and keeps that order on the device: big systems start
//    first, the smallest fill the tail, and warps running together mostly
//    share one unrolled body;
//  - each warp of a persistent grid takes the next system from an atomic
//    counter and evaluates it with its 32 lanes over the observations, the
//    planet count being warp-uniform so the planet loop is fully unrolled
//    for that count;
//  - the observations, fixed for the plan (Sec. 4.1 treats them as
//    constants for every model), are converted once per plan to the form the
//    kernel reads (packed pairs for the mixed path).
// The per-planet arithmetic is that of the uniform kernels (kc_device.cuh).
#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

#include "kc_device.cuh"
#include "kc_f64.cuh"
#include "kc_internal.h"
#include "kc_pair.cuh"
#include "kc_ragged.h"

namespace kc {

namespace {

__device__ inline double nan_r() { return __longlong_as_double(0x7ff8000000000000ll); }

// KC_DEBUG checks of a ragged system's descriptors (always true in a normal
// build): its observation range inside the plan's observations, its planet
// count, its parameter range inside the packed parameters.
__device__ __forceinline__ bool ragged_obs_ok(const RaggedDev &d, int64_t s, int64_t o0,
                                              int64_t o1) {
  return dbg_ok(d.invalid, 0 <= o0 && o0 <= o1 && o1 <= d.n_obs_total, kDbgObsOff, s);
}

__device__ __forceinline__ bool ragged_system_ok(const RaggedDev &d, int64_t s, int J,
                                                 int64_t o0, int64_t o1) {
  if (!dbg_ok(d.invalid, J >= 1 && J <= KC_MAX_PLANETS, kDbgPlanets, s)) return false;
  if (!ragged_obs_ok(d, s, o0, o1)) return false;
  const int64_t p0 = d.par_off[s];
  return dbg_ok(d.invalid, 0 <= p0 && p0 + 5 * J + 1 <= d.n_par_total, kDbgParOff, s);
}

__device__ inline double system_gamma_r(const double *p, int J) {
  bool ok = finite_bits(p[5 * J]);
  for (int j = 0; j < J; ++j)
    ok = ok && planet_valid(p[5 * j], p[5 * j + 1], p[5 * j + 2], p[5 * j + 3], p[5 * j + 4]);
  return ok ? p[5 * J] : nan_r();
}

// ------------------------------------------------------------ observation prep

// One warp per system, a lane per pair of observations: tau = t - t_ref (t_ref
// = the system's first observation) at fixed binary places and v as float
// pairs, w = 1/(sigma^2 + jitter^2), t - t0.
__global__ void prep_obs_mixed(RaggedDev d, const double *__restrict__ t,
                               const double *__restrict__ v, const double *__restrict__ sigma,
                               double jitter2, float4 *__restrict__ oa, float4 *__restrict__ ob,
                               double *__restrict__ t_ref) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = warp; s < d.n_sys; s += nwarp) {
    const int64_t o0 = d.obs_off[s], o1 = d.obs_off[s + 1];
    if (!ragged_obs_ok(d, s, o0, o1)) continue;
    const double tr = o1 > o0 ? t[o0] : d.t0;
    if (lane == 0) t_ref[s] = tr;
    // no FP64 instruction: differences from exact three-float splits
    const Split3 tr3 = split3(tr), te3 = split3(d.t0);
    const float jit2 = d2f(jitter2);
    const int64_t pair0 = ragged_pair(o0, s);
    // a far time leaves all of the system's as plain pairs
    bool seen = false;
    for (int64_t k = o0 + lane; k < o1; k += 32) {
      float th, tl;
      sub_ds(split3(t[k]), tr3, th, tl);
      tau_place(th, tl);
      seen |= far_time(th);
    }
    const bool far = __any_sync(0xffffffffu, seen);
    for (int64_t k = o0 + 2 * lane; k < o1; k += 64) {
      float th[2], tl[2], vh[2], vl[2], w[2], dt[2], err[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        th[i] = tl[i] = vh[i] = vl[i] = w[i] = dt[i] = err[i] = 0.0f;
        if (k + i < o1) {
          const Split3 tk = split3(t[k + i]);
          sub_ds(tk, tr3, th[i], tl[i]);
          if (!far) tau_place(th[i], tl[i], err[i]);
          split_d(v[k + i], vh[i], vl[i]);
          const float sg = d2f(sigma[k + i]);
          const float var = __fmaf_rn(sg, sg, jit2);
          w[i] = var > 0.0f ? 1.0f / var : __int_as_float(0x7fc00000);
          dt[i] = (tk.x0 - te3.x0) + (tk.x1 - te3.x1);
        }
      }
      const int64_t p = pair0 + ((k - o0) >> 1);
      oa[2 * p] = make_float4(th[0], th[1], tl[0], tl[1]);
      oa[2 * p + 1] = make_float4(vh[0], vh[1], vl[0], vl[1]);
      ob[p] = make_float4(w[0], w[1], dt[0], dt[1]);
      d.tau_err[p] = make_float2(err[0], err[1]);
    }
    if (lane == 0) d.far[s] = far ? 1 : 0;
  }
}

__global__ void prep_obs_f64(RaggedDev d, const double *__restrict__ t,
                             const double *__restrict__ v, const double *__restrict__ sigma,
                             double jitter2, ObsR64 *__restrict__ od,
                             double *__restrict__ t_ref) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = warp; s < d.n_sys; s += nwarp) {
    const int64_t o0 = d.obs_off[s], o1 = d.obs_off[s + 1];
    if (!ragged_obs_ok(d, s, o0, o1)) continue;
    const double tr = o1 > o0 ? t[o0] : d.t0;
    if (lane == 0) t_ref[s] = tr;
    for (int64_t k = o0 + lane; k < o1; k += 32) {
      const double var = fma(sigma[k], sigma[k], jitter2);
      od[k] = ObsR64{t[k] - tr, v[k], var > 0.0 ? 1.0 / var : nan_r(), t[k] - d.t0};
    }
  }
}

// FP64 model velocities of a ragged batch, one warp per system, its planets
// set up once by the first lanes, KC_MAX_PLANETS of them at a time: the counts
// are device data that no host check sees, and nothing else here limits them.
__global__ void __launch_bounds__(256)
predict_ragged_kernel(const double *__restrict__ params,
                                      const int64_t *__restrict__ par_off,
                                      const int32_t *__restrict__ n_pl,
                                      const double *__restrict__ t,
                                      const int64_t *__restrict__ obs_off, int64_t n_sys,
                                      double t0, double *__restrict__ v_out,
                                      unsigned long long *words) {
  __shared__ PlanetX pl_s[8][KC_MAX_PLANETS];
  const int lane = threadIdx.x & 31;
  PlanetX *pl = pl_s[threadIdx.x >> 5];
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarp = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = warp; s < n_sys; s += nwarp) {
    const int64_t o0 = obs_off[s], o1 = obs_off[s + 1];
    if (o1 <= o0) continue;
    const int J = n_pl[s];
    // the caller's arrays (no totals known here): ordered offsets, a planet
    if (!dbg_ok(words, o0 >= 0 && par_off[s] >= 0, kDbgObsOff, s) ||
        !dbg_ok(words, J >= 1, kDbgPlanets, s))
      continue;
    const double *p = params + par_off[s];
    const double tr = t[o0];
    const double gam = system_gamma_r(p, J);
    for (int j0 = 0; j0 == 0 || j0 < J; j0 += KC_MAX_PLANETS) {
      const int n = min(J - j0, KC_MAX_PLANETS);
      __syncwarp();
      if (lane < n) {
        double sw, cw, beta;
        pl[lane] = planet_setup_x(p + 5 * (j0 + lane), tr - t0, sw, cw, beta);
      }
      __syncwarp();
      const bool hi = any_high_e(lane < n && pl[lane].high);
      for (int64_t k = o0 + lane; k < o1; k += 32) {
        const double V = j0 == 0 ? gam : v_out[k];       // the lane's own sum so far
        v_out[k] = hi ? model_velocity<true>(t[k] - tr, pl, n, V)
                      : model_velocity<false>(t[k] - tr, pl, n, V);
      }
    }
  }
}

// ------------------------------------------------------------ per-system bodies

struct RPlanetD {
  PlanetD base;
  double K, cw, sw, n2, ibeta;
};

__device__ inline RPlanetD rsetup_f64(const double *p, double dref, bool grad) {
  RPlanetD g;
  g.base = planet_setup_f64(p, dref);
  g.K = g.cw = g.sw = g.n2 = g.ibeta = 0.0;
  if (grad) {
    sincos(p[3], &g.sw, &g.cw);
    g.K = p[1];
    g.n2 = g.base.inv_P * g.base.inv_P;
    g.ibeta = 1.0 / g.base.beta;
  }
  return g;
}

template <typename T>
__device__ __forceinline__ void partials_r(T e, T K, T cw, T sw, T beta, T ibeta, T sE, T cE,
                                           T invD,
                                           T &dK, T &dw, T &dM, T &de) {
  const T cf = (cE - e) * invD;
  const T sf = beta * sE * invD;
  const T c_wf = cw * cf - sw * sf;
  const T s_wf = sw * cf + cw * sf;
  dK = c_wf + e * cw;
  dw = -K * (s_wf + e * sw);
  const T ks = K * s_wf * invD;
  dM = -ks * beta * invD;
  de = K * cw - ks * sE * (ibeta + beta * invD);
}

// The planet constants of a mixed plan: with or without the partials'.
template <bool GRAD>
struct RaggedPlanet;
template <>
struct RaggedPlanet<true> {
  typedef GradPlanetP type;
};
template <>
struct RaggedPlanet<false> {
  typedef PlanetP type;
};

// One system of J planets and n observations by a warp, a pair of
// observations per lane at a time (kc_pair.cuh), the next pair loaded while
// this one is evaluated.  wide: the wide mean anomaly; with err != NULL the times
// completed to plain pairs by the plan's tau_err.
// The gradient has one body for both forms, a branch for the warp in front of the
// mean anomalies of three planets at a time: with a body of each, warps of both
// forms on an SM waited for instructions.  us with two bodies, with one, all periods
// above half a day and half of the systems with a shorter one: 50000 systems of 16
// to 1024 observations 336, 337 and 720, 391; 6000 of 16 to 512 38.1, 40.9 and 87,
// 44; 5000 of 100 to 1000 58, 58 and 138, 67; 20000 of 4 to 20 43.1, 39.5 and 53,
// 42.  (Half of the planets at a time, with the times completed outside the branch,
// it ran 47 us at 6000 and 69 at 5000; both bodies kept, with the one for both
// forms taken by all systems once one asks for it, 358 and 461 at 50000.)  The
// forward bodies are short enough for two (50000 of 16 to 1024: 220 us, 227 with
// one; the mixture 63 and 47).
template <int J, bool GRAD, bool WIDE>
__device__ __forceinline__ void body_mixed(const typename RaggedPlanet<GRAD>::type *pl, float gam,
                                           const float *tab, const float4 *oa, const float4 *ob,
                                           const float2 *err, bool wide, int64_t pair0, int n,
                                           int lane, float *chi2_out, float *grad_out) {
  constexpr int JG = GRAD ? J : 1;
  Kahan2 acc = {0, 0};
  f32x2 sum_a = 0;
  typename GradSumsFor<JG>::type g[JG];
#pragma unroll
  for (int j = 0; j < JG; ++j) g[j] = {{0, 0}, 0, 0, 0, 0};
  const int pairs = (n + 1) >> 1;
  oa += 2 * pair0;
  ob += pair0;
  float4 t_next = make_float4(0.f, 0.f, 0.f, 0.f), v_next = t_next, w_next = t_next;
  if (lane < pairs) {
    t_next = oa[2 * lane];
    v_next = oa[2 * lane + 1];
    w_next = ob[lane];
  }
  for (int p = lane; p < pairs; p += 32) {
    // the planets' constants are read from shared memory again in every
    // iteration instead of being hoisted into registers for all J planets (the
    // forward kernel spilled 3 KB so: 50000 systems of 16 to 1024 observations
    // in 287 us against 222)
    asm volatile("" ::: "memory");
    const float4 tt = t_next, vv = v_next, ww = w_next;
    if (p + 32 < pairs) {
      t_next = oa[2 * (p + 32)];
      v_next = oa[2 * (p + 32) + 1];
      w_next = ob[p + 32];
    }
    f32x2 th = pack2(tt.x, tt.y), tl = pack2(tt.z, tt.w);
    auto complete = [&]() {
      const float2 e = err[pair0 + p];
      float h0, l0, h1, l1;
      two_sum(tt.x, tt.z, h0, l0);
      two_sum(tt.y, tt.w, h1, l1);
      th = pack2(h0, h1);
      tl = pack2(l0 + e.x, l1 + e.y);
    };
    if (!GRAD && WIDE && err != nullptr) complete();
    Kahan2 V = {dup2(gam), 0};
    GradTerms o[JG];
    if constexpr (GRAD) {
      constexpr int H = J > 3 ? 3 : J;
#pragma unroll
      for (int j0 = 0; j0 < J; j0 += H) {
        f32x2 M[H];
        if (wide) {
          if (j0 == 0 && err != nullptr) complete();
#pragma unroll
          for (int j = 0; j < H && j0 + j < J; ++j) M[j] = mean_anomaly_wide(th, tl, pl[j0 + j].p);
        } else {
#pragma unroll
          for (int j = 0; j < H && j0 + j < J; ++j) M[j] = mean_anomaly_pair(th, tl, pl[j0 + j].p);
        }
#pragma unroll
        for (int j = 0; j < H && j0 + j < J; ++j)
          o[j0 + j] = grad_terms_at(M[j], pl[j0 + j], tab, V);
      }
    } else {
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const f32x2 M = mean_anomaly2<WIDE>(th, tl, pl[j]);
        f32x2 s, c, E;
        kepler_pair<false>(abs2(M), pl[j], tab, s, c, E);
        velocity_sum(V, pl[j], signed_as(s, M), c);
      }
    }
    const f32x2 r = sub2(sub2(V.big, pack2(vv.x, vv.y)), add2(V.small, pack2(vv.z, vv.w)));
    const f32x2 wr = mul2(pack2(ww.x, ww.y), r);
    kahan_add(acc, mul2(wr, r));
    if constexpr (GRAD) {
      const f32x2 a2 = add2(wr, wr), adt = mul2(a2, pack2(ww.z, ww.w));
      sum_a = add2(sum_a, a2);
#pragma unroll
      for (int j = 0; j < J; ++j) grad_add(g[j], o[j], pl[j], a2, adt);
    }
  }
  Kahan chi = kahan_join(acc);
  float sa = join2(sum_a);
  GradLane gl[JG];
#pragma unroll
  for (int j = 0; j < JG; ++j) gl[j] = grad_join(g[j]);
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    const Kahan o = {shfl_xor(chi.big, m), shfl_xor(chi.small, m)};
    kahan_merge(chi, o);
    if constexpr (GRAD) {
      sa += shfl_xor(sa, m);
#pragma unroll
      for (int j = 0; j < JG; ++j) grad_combine(gl[j], m);
    }
  }
  if (lane == 0) {
    float poison = 0.0f * gam;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      if constexpr (GRAD)
        poison += 0.0f * pl[j].p.e;
      else
        poison += 0.0f * pl[j].e;
    }
    *chi2_out = kahan_value(chi) + poison;
    if constexpr (GRAD) {
#pragma unroll
      for (int j = 0; j < JG; ++j) grad_finish(gl[j], pl[j], sa, poison, grad_out + 5 * j);
      grad_out[5 * J] = sa + poison;
    }
  }
}

template <int J, bool GRAD, bool HI>
__device__ __forceinline__ void body_f64(const RPlanetD *pl, double gam, const ObsR64 *od,
                                         int64_t o0, int n, int lane, double *chi2_out,
                                         double *grad_out) {
  constexpr int NP = 5 * J + 1;
  double acc = 0.0;
  double g[GRAD ? NP : 1];
#pragma unroll
  for (int i = 0; i < (GRAD ? NP : 1); ++i) g[i] = 0.0;
  ObsR64 o_next = {0.0, 0.0, 0.0, 0.0};
  if (lane < n) o_next = od[o0 + lane];
  for (int k = lane; k < n; k += 32) {
    const ObsR64 o = o_next;
    if (k + 32 < n) o_next = od[o0 + k + 32];
    double sEj[J], cEj[J];
    double V = gam;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const PlanetD q = pl[j].base;
      const double M = mean_anomaly_f64(o.tau, q);
      kepler_f64<HI>(M, q.e, sEj[j], cEj[j]);
      V = velocity_add_f64(q, sEj[j], cEj[j], V);
    }
    const double r = V - o.v;
    acc = fma(o.w * r, r, acc);
    if (GRAD) {
      const double a2 = 2.0 * o.w * r;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const RPlanetD q = pl[j];
        double dK, dw, dM, de;
        const double invD = 1.0 / fma(-q.base.e, cEj[j], 1.0);
        partials_r(q.base.e, q.K, q.cw, q.sw, q.base.beta, q.ibeta, sEj[j], cEj[j], invD, dK,
                   dw, dM, de);
        const double dP = dM * (-kTwoPi * o.dt * q.n2);
        g[5 * j + 0] = fma(a2, dP, g[5 * j + 0]);
        g[5 * j + 1] = fma(a2, dK, g[5 * j + 1]);
        g[5 * j + 2] = fma(a2, de, g[5 * j + 2]);
        g[5 * j + 3] = fma(a2, dw, g[5 * j + 3]);
        g[5 * j + 4] = fma(a2, dM, g[5 * j + 4]);
      }
      g[GRAD ? 5 * J : 0] += a2;
    }
  }
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    acc += shfl_xor(acc, m);
    if (GRAD) {
#pragma unroll
      for (int i = 0; i < (GRAD ? NP : 1); ++i) g[i] += shfl_xor(g[i], m);
    }
  }
  if (lane == 0) {
    const double poison = 0.0 * gam;
    *chi2_out = acc + poison;
    if (GRAD) {
#pragma unroll
      for (int i = 0; i < (GRAD ? NP : 1); ++i) grad_out[i] = g[i] + poison;
    }
  }
}

// ------------------------------------------------------------ persistent kernels

constexpr int kMaxWarps = 8;   // block <= 256

#define KC_RAGGED_SWITCH(BODY)                      \
  switch (J) {                                      \
    case 1: BODY(1); break;                         \
    case 2: BODY(2); break;                         \
    case 3: BODY(3); break;                         \
    case 4: BODY(4); break;                         \
    case 5: BODY(5); break;                         \
    case 6: BODY(6); break;                         \
    case 7: BODY(7); break;                         \
    default: BODY(8); break;                        \
  }

// Each warp: take the next kAhead systems from the queue (systems in
// decreasing order of work), set all their planets up at once (lane 8 i + j
// the planet j of the i-th), evaluate them one after the other with 32 lanes
// over the observations, reduce, write; until the queue is empty.  The queue
// counter must be zero at launch.  Taken one at a time, each system would wait
// for the counter, its descriptors, its parameters and a setup chain of some
// 500 instructions in J lanes.
// At most 128 registers, two CTAs of 256 threads per SM.  For the forward
// kernel three or four (80 or 64 registers) gain up to 6 % on large batches
// and lose on small ones, where each CTA's table load and the queue count:
// 50000 systems of 16 to 1024 observations 224 us (two), 222 (three), 210
// (four); 3000 of them 30, 36, 36; 20000 of 4 to 20 observations 29, 35, 33.
// Bound by the FP32 pipe's instructions (packed ones take two issue slots) at
// large sizes.  Measured before, one observation per instruction and a system
// at a time: forward 50000 systems 310 us, 3000 51, 20000 tiny 31; gradient
// 50000 systems 440 us (now 337), 200000 1734 (now 1186).
constexpr int kAhead = 4;
static_assert(kAhead * KC_MAX_PLANETS == 32, "a lane per planet of the systems taken");

template <bool GRAD>
__global__ void __launch_bounds__(256, 2)
ragged_mixed_kernel(RaggedDev d, const float4 *__restrict__ oa, const float4 *__restrict__ ob,
                    const double *__restrict__ params, float *__restrict__ chi2,
                    float *__restrict__ grad, unsigned long long *__restrict__ queue) {
  typedef typename RaggedPlanet<GRAD>::type Planet;
  __shared__ AngTab tab_s;
  __shared__ Planet pl_s[kMaxWarps][kAhead * KC_MAX_PLANETS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ang_tab_load<GRAD>(tab_s.s, threadIdx.x, blockDim.x);
  __syncthreads();
  const int mine = lane / KC_MAX_PLANETS, mine_j = lane % KC_MAX_PLANETS;
  // fewer at a time where the queue holds few per warp (300 systems taken four
  // at a time ran 40 us against 17); systems of one round of the lanes' pairs are
  // about alike, and half as many rounds balance them (14192 systems of 2 to 17
  // observations, one and two at a time: gradient 39.0, 32.8 us, forward 28.8, 22.5)
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int rounds = d.n_obs_total > 64 * d.n_sys ? 4 : 2;
  const int take = (int)max((int64_t)1, min((int64_t)kAhead, d.n_sys / (rounds * warps)));
  for (;;) {
    unsigned long long idx = 0;
    if (lane == 0) idx = atomicAdd(queue, (unsigned long long)take);
    idx = __shfl_sync(0xffffffffu, idx, 0);
    if (idx >= (unsigned long long)d.n_sys) break;
    // this lane's system of the ones taken (J = 0: none), and its planet
    int64_t s = -1, o0 = 0, p0 = 0;
    int J = 0, n = 0;
    float gam = 0.0f;
    bool wide_me = false, exact_me = false;
    if (mine < take && idx + mine < (unsigned long long)d.n_sys) {
      s = d.order[idx + mine];
      if (dbg_ok(d.invalid, 0 <= s && s < d.n_sys, kDbgOrder, (int64_t)(idx + mine))) {
        J = d.n_pl[s];
        o0 = d.obs_off[s];
        const int64_t o1 = d.obs_off[s + 1];
        p0 = d.par_off[s];
        n = (int)(o1 - o0);
        if (!ragged_system_ok(d, s, J, o0, o1)) J = 0;
      }
    }
    __syncwarp();                                // the last systems' use of the planets
    if (mine_j < J) {
      const double *p = params + p0 + 5 * mine_j;
      const bool far = d.far[s] != 0;
      const PlanetP *mine_p;
      if constexpr (GRAD) {
        pl_s[warp][lane] = grad_setup_pair(p, d.t_ref[s], d.t0, far);
        mine_p = &pl_s[warp][lane].p;
      } else {
        pl_s[warp][lane] = planet_setup_pair(p, d.t_ref[s], d.t0, far);
        mine_p = &pl_s[warp][lane];
      }
      wide_me = far || short_period(*mine_p);
      exact_me = !far && !(mine_p->n <= kPairExactFreq);
      if (mine_j == 0) {
        const double gd = params[p0 + 5 * J];
        gam = finite_bits(gd) ? d2f(gd) : __int_as_float(0x7fc00000);
      }
    }
    const unsigned wide = __ballot_sync(0xffffffffu, wide_me);
    const unsigned exact = __ballot_sync(0xffffffffu, exact_me);
    __syncwarp();
    for (int i = 0; i < take; ++i) {
      const int from = i * KC_MAX_PLANETS;
      const int Ji = __shfl_sync(0xffffffffu, J, from);
      if (Ji == 0) continue;
      const int64_t si = __shfl_sync(0xffffffffu, s, from);
      const int64_t oi = __shfl_sync(0xffffffffu, o0, from);
      const int64_t pi = __shfl_sync(0xffffffffu, p0, from);
      const int ni = __shfl_sync(0xffffffffu, n, from);
      const float gi = __shfl_sync(0xffffffffu, gam, from);
      const Planet *pl = pl_s[warp] + from;
      const bool wi = ((wide >> from) & 0xffu) != 0u;
      const float2 *err = ((exact >> from) & 0xffu) != 0u ? d.tau_err : nullptr;
      float *gout = GRAD ? grad + pi : nullptr;
      const int64_t pair0 = ragged_pair(oi, si);
      const int J = Ji;
#define KC_BODY(JJ)                                                                        \
  if (wi && !GRAD)                                                                         \
    body_mixed<JJ, GRAD, true>(pl, gi, tab_s.s, oa, ob, err, wi, pair0, ni, lane,          \
                               chi2 + si, gout);                                           \
  else                                                                                     \
    body_mixed<JJ, GRAD, false>(pl, gi, tab_s.s, oa, ob, err, wi, pair0, ni, lane,         \
                                chi2 + si, gout)
      KC_RAGGED_SWITCH(KC_BODY)
#undef KC_BODY
      if (lane == 0) note_invalid(d.invalid, chi2[si]);      // lane 0 wrote it
    }
  }
}

template <bool GRAD>
__global__ void __launch_bounds__(256)
ragged_f64_kernel(RaggedDev d, const ObsR64 *__restrict__ od, const double *__restrict__ params,
                  double *__restrict__ chi2, double *__restrict__ grad,
                  unsigned long long *__restrict__ queue) {
  __shared__ RPlanetD pl_s[kMaxWarps][KC_MAX_PLANETS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  RPlanetD *pl = pl_s[warp];
  for (;;) {
    unsigned long long idx = 0;
    if (lane == 0) idx = atomicAdd(queue, 1ull);
    idx = __shfl_sync(0xffffffffu, idx, 0);
    if (idx >= (unsigned long long)d.n_sys) break;
    const int64_t s = d.order[idx];
    if (!dbg_ok(d.invalid, 0 <= s && s < d.n_sys, kDbgOrder, (int64_t)idx)) continue;
    const int J = d.n_pl[s];
    const int64_t o0 = d.obs_off[s];
    if (!ragged_system_ok(d, s, J, o0, d.obs_off[s + 1])) continue;
    const int n = (int)(d.obs_off[s + 1] - o0);
    const double *p = params + d.par_off[s];
    const double dref = d.t_ref[s] - d.t0;
    if (lane < J) pl[lane] = rsetup_f64(p + 5 * lane, dref, GRAD);
    const double gam = system_gamma_r(p, J);
    __syncwarp();
    const bool hi = any_high_e(lane < J && pl[lane].base.e > (double)kEccFast);
    double *gout = GRAD ? grad + d.par_off[s] : nullptr;
#define KC_BODY(JJ)                                                                  \
  if (hi)                                                                            \
    body_f64<JJ, GRAD, true>(pl, gam, od, o0, n, lane, chi2 + s, gout);              \
  else                                                                               \
    body_f64<JJ, GRAD, false>(pl, gam, od, o0, n, lane, chi2 + s, gout)
    KC_RAGGED_SWITCH(KC_BODY)
#undef KC_BODY
    if (lane == 0) note_invalid(d.invalid, chi2[s]);      // lane 0 wrote it
    __syncwarp();
  }
}

}  // namespace

// ------------------------------------------------------------ launchers

cudaError_t ragged_prep(const RaggedDev &d, int mode, const double *t, const double *v,
                        const double *sigma, double jitter2, void *obs_a, void *obs_b,
                        double *t_ref, cudaStream_t st) {
  const int64_t warps = d.n_sys;
  int64_t blocks = (warps * 32 + 255) / 256;
  if (blocks > (int64_t)sm_count() * 64) blocks = (int64_t)sm_count() * 64;
  if (blocks < 1) blocks = 1;
  if (mode == KC_MIXED)
    prep_obs_mixed<<<(int)blocks, 256, 0, st>>>(d, t, v, sigma, jitter2, (float4 *)obs_a,
                                                (float4 *)obs_b, t_ref);
  else
    prep_obs_f64<<<(int)blocks, 256, 0, st>>>(d, t, v, sigma, jitter2, (ObsR64 *)obs_a, t_ref);
  return cudaGetLastError();
}

cudaError_t launch_predict_ragged(const double *params, const int64_t *par_off,
                                  const int32_t *n_pl, const double *t, const int64_t *obs_off,
                                  int64_t n_sys, double t0, double *v_out, cudaStream_t st) {
  int64_t blocks = (n_sys * 32 + 255) / 256;
  if (blocks > (int64_t)sm_count() * 64) blocks = (int64_t)sm_count() * 64;
  predict_ragged_kernel<<<(int)(blocks > 0 ? blocks : 1), 256, 0, st>>>(
      params, par_off, n_pl, t, obs_off, n_sys, t0, v_out, invalid_counter());
  return cudaGetLastError();
}

const void *ragged_kernel_fn(int mode, bool grad) {
  if (mode == KC_MIXED)
    return grad ? (const void *)ragged_mixed_kernel<true> : (const void *)ragged_mixed_kernel<false>;
  return grad ? (const void *)ragged_f64_kernel<true> : (const void *)ragged_f64_kernel<false>;
}

int ragged_max_blocks_per_sm(int mode, bool grad, int block) {
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, ragged_kernel_fn(mode, grad), block, 0);
  return n;
}

cudaError_t ragged_launch(const RaggedDev &d, int mode, bool grad, const void *obs_a,
                          const void *obs_b, const double *params, void *chi2, void *gradp,
                          unsigned long long *queue, int grid, int block, cudaStream_t st) {
  if (mode == KC_MIXED) {
    if (grad)
      ragged_mixed_kernel<true><<<grid, block, 0, st>>>(d, (const float4 *)obs_a,
                                                        (const float4 *)obs_b, params,
                                                        (float *)chi2, (float *)gradp, queue);
    else
      ragged_mixed_kernel<false><<<grid, block, 0, st>>>(d, (const float4 *)obs_a,
                                                         (const float4 *)obs_b, params,
                                                         (float *)chi2, (float *)gradp, queue);
  } else {
    if (grad)
      ragged_f64_kernel<true><<<grid, block, 0, st>>>(d, (const ObsR64 *)obs_a, params,
                                                      (double *)chi2, (double *)gradp, queue);
    else
      ragged_f64_kernel<false><<<grid, block, 0, st>>>(d, (const ObsR64 *)obs_a, params,
                                                       (double *)chi2, (double *)gradp, queue);
  }
  return cudaGetLastError();
}

}  // namespace kc
