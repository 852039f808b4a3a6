// kc_chi2_warp.cu -- the mixed-precision chi-square of a uniform batch with
// G = 8, 16, 32, 64 or 128 lanes per system (one warp per system at G = 32,
// two or four at 64 and 128), sized by the host so that the CTAs spread
// evenly over the SMs.
//
// The mixed path of the fused kernel of kc_fwd.cu (double-single phase,
// Sec. 5; Kepler's equation in single precision, Sec. 4.3; Eq. 3 velocity;
// Kahan sums of the planet velocities and of chi2, Sec. 4.4) in the packed
// two-observation form of kc_pair.cuh, laid out for the SMs rather than for
// a tile.  Bound by FP32 issue and register ports (68 clocks per warp,
// planet and observation and sub-partition in steady state).  Measured, us
// per launch, before (scalar form) and now: 2^20 x 4 x 256 3224 -> 1977, 4096
// x 4 x 256 back to back 14.3 -> 11.2, 300 x 3 x 101 5.9 -> 4.3; 65536 x 4 x 256
// with ordinary periods 191 -> 127, with 1, 10 and 100 % of the planets below half
// a day 142, 163 and 166, with a time beyond 2^14 d 169, with periods of 0.001 ..
// 0.01 d 188.
//
//  - A CTA of W warps evaluates W * 32 / G systems (one round).  The host
//    picks G and W by a cost model (pick_warp_tile) so that the CTAs land
//    evenly on the SMs and share their staging (for 4096 systems, 27 warps per
//    CTA: one CTA and 27 systems on every SM, where tiles of 16 systems leave
//    some SMs with 32 and others with 16).  Larger batches run many waves; the
//    hardware then overlaps one CTA's prologue with the work of the others on
//    its SM.
//  - Prologue: every global load (the reference time, this thread's
//    observation and its planet's parameters) is issued before any of them
//    is used, so the CTA waits for memory once.
//  - The observations (shared by every system, Sec. 4.1) are converted to
//    float pairs and staged in shared memory, padded with zero-weight
//    entries to whole chunks, so the inner loops have no tail; the last
//    threads of the CTA stage while the first set the planets up.
//  - Each lane holds a chunk of kChunk observations (two packed pairs: their
//    phases and their compensated velocity sums) in registers and streams
//    the planets over it: a planet's constants (PlanetP, computed once per
//    (system, planet)) are read from shared memory once per chunk, and the
//    chunk's Kepler solves are independent chains for the scheduler.
//  - A CTA with a period or a time outside the short mean anomaly's range runs
//    the wide body (kc_pair.cuh), in which a system without either still takes
//    the short form (a warp of such systems the short body); the first far time
//    has the planets and the staged times made plain pairs.  So a system's bits
//    hang on its own planets, the observations and the launch shape alone.
//  - The lanes of a system combine their compensated sums with TwoSum
//    shuffles, and the warps of a system (G > 32) through a few words of
//    shared memory; no atomics, no scratch memory.  Splitting a system over
//    several warps keeps the SMs' warp slots filled when the batch is small
//    (2048 systems: 28 warps per SM instead of 14).
//  - Programmatic dependent launch: the kernel waits for the grids before
//    it in the stream to complete (griddepcontrol.wait, ahead of its first
//    global access) and at once lets the next launch on the stream begin
//    (griddepcontrol.launch_dependents), so that a following batch's CTAs
//    are placed on the SMs as this grid's CTAs exit instead of after the
//    whole grid has completed (back-to-back 4096 x 4 x 256 batches: 14.0 us
//    each instead of 16.4 us, with the scalar body).  The launch asks for it
//    only outside stream capture: as programmatic edges in the DE-MC driver's
//    graph (4096 chains, halves of 2048) it cost a quarter of the generations
//    per second (2.36e4 against 3.12e4), where back-to-back launches of 1024 to
//    4096 systems gained 2.7-2.9 us each.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "kc_demc.cuh"
#include "kc_device.cuh"
#include "kc_internal.h"
#include "kc_pair.cuh"

namespace kc {

namespace {

constexpr int kChunk = 4;           // observations per lane in registers
constexpr int kObsTileMax = 1024;   // observations staged per CTA at a time

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) / 16 * 16; }
__host__ __device__ inline int round_up(int x, int m) { return (x + m - 1) / m * m; }
// x rounded up to a multiple of the power of two m (no division)
__device__ __forceinline__ int round_up_pow2(int x, int m) { return (x + m - 1) & -m; }

// Shared memory: the sin/cos table, the planets' constants, the systems'
// gamma, the staged observations (one float array per quantity, so that a
// lane reads the pair of observations it packs as one 8-byte word), and the
// words that combine a system's warps.
struct WarpLayout {
  size_t tab, pl, gam, obs, red, total;
  __host__ __device__ WarpLayout(int spr, int J, int tile, int nwarps) {
    tab = 0;
    pl = tab + sizeof(AngTab);
    gam = pl + sizeof(PlanetP) * spr * J;
    obs = align16(gam + sizeof(float) * spr);
    red = obs + sizeof(float) * 5 * tile;         // G > 32: 3 words per warp
    total = align16(red + sizeof(float) * 3 * nwarps);
  }
};

// Observations held per CTA: all of them (padded to whole chunks of every
// lane of a system) when they fit, else tiles of kObsTileMax.
__host__ __device__ inline int warp_obs_tile(int n_obs, int G) {
  return n_obs <= kObsTileMax ? round_up(n_obs > 0 ? n_obs : 1, G * kChunk) : kObsTileMax;
}

// Setup of one item of the CTA's round: items 0 .. spr*J - 1 are the
// (system, planet) constants, items spr*J .. spr*(J+1) - 1 the systems'
// gamma.  p holds the item's parameters (five, or gamma in p[0]); an
// invalid planet carries e = NaN, which poisons its system.
// Returns whether the planet's period asks for the wide mean anomaly.
template <int J>
__device__ __forceinline__ bool setup_item(int i, int spr, int64_t sys0, int64_t n_sys,
                                           const double (&p)[5], double t_ref, double t0,
                                           PlanetP *pl_s, float *gam_s, unsigned long long *dbg) {
  if (!dbg_ok(dbg, i < spr * (J + 1), kDbgSmem, i)) return false;
  bool brief = false;
  if (i < spr * J) {
    const int64_t s = sys0 + i / J;
    PlanetP q = {};
    if (s < n_sys) {
      q = planet_setup_pair(p, t_ref, t0, false);
      brief = short_period(q);
    }
    pl_s[i] = q;
  } else {
    const int sl = i - spr * J;
    float g = 0.0f;
    if (sys0 + sl < n_sys) g = finite_bits(p[0]) ? d2f(p[0]) : __int_as_float(0x7fc00000);
    gam_s[sl] = g;
  }
  return brief;
}

// The item's parameters.  DEMC: the launch evaluates DE-MC proposals; with
// a.demc.z set they are formed here from the chains' states and the draws
// (and stored to the proposals, which a.params points at).
template <int J, bool DEMC>
__device__ __forceinline__ void load_item(int i, int spr, int64_t sys0, const UniformArgs &a,
                                          double (&p)[5]) {
  const int npar = 5 * J + 1;
  if (i < spr * J) {
    const int sl = i / J, j = i - sl * J;
    const int64_t s = sys0 + sl;
    const int64_t at = s * npar + 5 * j;
    if (s < a.n_sys && dbg_ok(a.invalid, at + 4 < a.n_sys * npar, kDbgParam, at)) {
      if (DEMC && a.demc.z) {
        demc_form(a, s, 5 * j, npar, p);
      } else {
#pragma unroll
        for (int k = 0; k < 5; ++k) p[k] = a.params[at + k];
      }
    }
  } else {
    const int64_t s = sys0 + (i - spr * J);
    if (s < a.n_sys && dbg_ok(a.invalid, s * npar + 5 * J < a.n_sys * npar, kDbgParam,
                              s * npar + 5 * J)) {
      if (DEMC && a.demc.z) {
        double g[1];
        demc_form(a, s, 5 * J, npar, g);
        p[0] = g[0];
      } else {
        p[0] = a.params[s * npar + 5 * J];
      }
    }
  }
}

// The thread's observations of one staged tile: npad (whole chunks), nk of
// them real.  The thread takes kChunk observations at a time as kChunk / 2
// packed pairs.  WIDE: form as in kc_pair.cuh; with t != NULL the times as plain
// pairs, from t (n_obs of them, the tile's first one at k0).
template <int J, bool RESID, bool WIDE>
__device__ __forceinline__ void warp_tile_sum(const float *th_s, int tile, const PlanetP *q,
                                              const float *tab, float gam, int c, int lg,
                                              int npad, int nk, Kahan2 &acc, float &rmax,
                                              unsigned long long *dbg, MeanForm form = {},
                                              const double *t = nullptr, int k0 = 0,
                                              int n_obs = 0) {
  constexpr int kPairs = kChunk / 2;
  const int step = kChunk << lg;
  for (int base = 2 * c; base < npad; base += step) {
    if (!dbg_ok(dbg, base + ((kPairs - 1) << (lg + 1)) + 1 < tile, kDbgSmem, base)) break;
    f32x2 th[kPairs], tl[kPairs];
    Kahan2 V[kPairs];
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
      const float *o = th_s + base + (i << (lg + 1));
      th[i] = *reinterpret_cast<const f32x2 *>(o);
      tl[i] = *reinterpret_cast<const f32x2 *>(o + tile);
      if (WIDE && t != nullptr)
        plain_times(t, k0 + base + (i << (lg + 1)), n_obs, th[i], tl[i]);
      V[i].big = dup2(gam);
      V[i].small = 0;
    }
    // two planets per iteration: the second one's constants load while the
    // first one's chains run (2074 us against 2195 for one at a time on the
    // 2^20-system sweep; all four at once spill: 2171)
#pragma unroll 2
    for (int j = 0; j < J; ++j) {
      const PlanetP &qj = q[j];
#pragma unroll
      for (int i = 0; i < kPairs; ++i) {
        const f32x2 M = mean_anomaly2<WIDE>(th[i], tl[i], qj, form);
        const f32x2 m = abs2(M);
        f32x2 s, cE, E;
        kepler_pair<false>(m, qj, tab, s, cE, E);
        if (RESID) {
          const f32x2 r = fma2(dup2(-qj.e), s, sub2(E, m));
          const int k = base + (i << (lg + 1));
          rmax = fmaxf(rmax, k < nk ? fabsf(lo2(r)) : 0.0f);
          rmax = fmaxf(rmax, k + 1 < nk ? fabsf(hi2(r)) : 0.0f);
        }
        velocity_sum(V[i], qj, signed_as(s, M), cE);
      }
    }
#pragma unroll
    for (int i = 0; i < kPairs; ++i) {
      const float *o = th_s + 2 * tile + base + (i << (lg + 1));
      const f32x2 vh = *reinterpret_cast<const f32x2 *>(o);
      const f32x2 vl = *reinterpret_cast<const f32x2 *>(o + tile);
      const f32x2 w = *reinterpret_cast<const f32x2 *>(o + 2 * tile);
      // residual V - v_obs with the model and the observation as float pairs
      const f32x2 r = sub2(sub2(V[i].big, vh), add2(V[i].small, vl));
      kahan_add(acc, mul2(mul2(w, r), r));
    }
  }
}

// Observation k of a staged tile: tau = t - t_ref as (th, tl) and v as float
// pairs, w = 1/(sigma^2 + jitter^2); the padding up to whole chunks has zero
// weight (and tau = v = 0).  plain: tau stays as it is (kc_pair.cuh).  Returns
// whether the time is a far one.
__device__ __forceinline__ bool stage_obs(float *obs_s, int tile, int k, bool real, double t,
                                          double v, double sigma, const Split3 &tr3, float jit2,
                                          bool plain, unsigned long long *dbg) {
  if (!dbg_ok(dbg, k < tile, kDbgSmem, k)) return false;
  float th = 0.0f, tl = 0.0f, vh = 0.0f, vl = 0.0f, wk = 0.0f;
  if (real) {
    sub_ds(split3(t), tr3, th, tl);
    if (!plain) tau_place(th, tl);
    split_d(v, vh, vl);
    const float sg = d2f(sigma);
    const float var = __fmaf_rn(sg, sg, jit2);
    wk = var > 0.0f ? 1.0f / var : __int_as_float(0x7fc00000);
  }
  obs_s[k] = th;
  obs_s[tile + k] = tl;
  obs_s[2 * tile + k] = vh;
  obs_s[3 * tile + k] = vl;
  obs_s[4 * tile + k] = wk;
  return far_time(th);
}

// The CTA's shared memory.
template <int J>
struct WarpSmem {
  float *tab, *gam, *obs, *red;
  PlanetP *pl;
  __device__ __forceinline__ WarpSmem(unsigned char *smem, int spr, int tile, int nwarps) {
    const WarpLayout L(spr, J, tile, nwarps);
    tab = reinterpret_cast<float *>(smem + L.tab);
    pl = reinterpret_cast<PlanetP *>(smem + L.pl);
    gam = reinterpret_cast<float *>(smem + L.gam);
    obs = reinterpret_cast<float *>(smem + L.obs);
    red = reinterpret_cast<float *>(smem + L.red);
  }
};

// The CTA's systems, one per G lanes, once the first tile is staged: all tiles'
// sums, their combination, the results.  poison: NaN for an invalid system.  WIDE:
// plain, form and te as in wide_systems.  The short and the wide form part before
// it and do not meet again: joined after each tile, the wide body's registers cost
// the short one's 1 to 4 %.
template <int J, bool RESID, bool DEMC, bool WIDE>
__device__ __forceinline__ void systems(const UniformArgs &a, unsigned char *smem, int lg, int tile,
                                        int ntiles, float *out, float *resid_out, bool plain,
                                        MeanForm form, const double *te, float gam,
                                        float poison) {
  const int block = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = 1 << lg, spr = block >> lg, step = G * kChunk;
  const WarpSmem<J> m(smem, spr, tile, block >> 5);
  int slot = tid >> lg;
  if (!dbg_ok(a.invalid, slot < spr, kDbgSmem, slot)) slot = 0;
  const int c = tid & (G - 1);                   // the thread's place in its system
  const int64_t s = (int64_t)blockIdx.x * spr + slot;
  const PlanetP *q = m.pl + slot * J;
  Kahan2 acc2 = {0, 0};
  float rmax = 0.0f;

  for (int t = 0; t < ntiles; ++t) {
    const int k0 = t * tile;
    const int nk = min(tile, a.n_obs - k0);
    const int npad = round_up_pow2(nk, step);
    if (t > 0) {
      __syncthreads();
      const Split3 tr3 = split3(a.t[0]);
      const float jit2 = d2f(a.jitter2);
      for (int k = tid; k < npad; k += block) {
        const bool real = k < nk && dbg_ok(a.invalid, k0 + k < a.n_obs, kDbgObs, k0 + k);
        stage_obs(m.obs, tile, k, real, real ? a.t[k0 + k] : 0.0, real ? a.v[k0 + k] : 0.0,
                  real ? a.sigma[k0 + k] : 1.0, tr3, jit2, plain, a.invalid);
      }
      __syncthreads();
    }
    // (a warp of short-form systems alone in a wide CTA)
    if (WIDE && !form.all)
      warp_tile_sum<J, RESID, true>(m.obs, tile, q, m.tab, gam, c, lg, npad, nk, acc2, rmax,
                                    a.invalid, form, te, k0, a.n_obs);
    else
      warp_tile_sum<J, RESID, false>(m.obs, tile, q, m.tab, gam, c, lg, npad, nk, acc2, rmax,
                                     a.invalid);
  }
  Kahan acc = kahan_join(acc2);

  // combine the system's lanes within each of its warps (G a power of two)
  for (int d = (G < 32 ? G : 32) >> 1; d >= 1; d >>= 1) {
    Kahan o = {shfl_xor(acc.big, d), shfl_xor(acc.small, d)};
    kahan_merge(acc, o);
    if (RESID) rmax = fmaxf(rmax, shfl_xor(rmax, d));
  }
  if (G > 32) {
    // then its G / 32 warps, in warp order, through shared memory (lg is
    // the same for the whole CTA, so every thread reaches the barrier)
    float *red_s = m.red;
    if (lane == 0) {
      red_s[3 * warp] = acc.big;
      red_s[3 * warp + 1] = acc.small;
      red_s[3 * warp + 2] = rmax;
    }
    __syncthreads();
    if (c == 0) {
      for (int w = warp + 1; w < warp + (G >> 5); ++w) {
        if (!dbg_ok(a.invalid, w < (block >> 5), kDbgSmem, w)) break;
        const Kahan o = {red_s[3 * w], red_s[3 * w + 1]};
        kahan_merge(acc, o);
        rmax = fmaxf(rmax, red_s[3 * w + 2]);
      }
    }
  }
  if (c == 0 && s < a.n_sys) {
    const float value = kahan_value(acc) + poison;   // NaN survives n_obs == 0
    out[s] = value;
    note_invalid(a.invalid, value);
    if (RESID) resid_out[s] = rmax;
    // the proposals this CTA formed are visible here after the barrier
    if (DEMC) demc_accept<5 * J + 1>(a, s, value);
  }
}

// The systems of a CTA with a period or a time outside the short mean anomaly's
// range; far: one of the thread's times is.  All threads of the CTA call it.
template <int J, bool RESID, bool DEMC>
__device__ __forceinline__ void wide_systems(const UniformArgs &a, unsigned char *smem, int lg,
                                             int tile, int ntiles, float *out, float *resid_out,
                                             bool far, float gam, float poison) {
  const int block = blockDim.x, tid = threadIdx.x, spr = block >> lg;
  const int64_t sys0 = (int64_t)blockIdx.x * spr;
  const WarpSmem<J> m(smem, spr, tile, block >> 5);
  const bool plain = __syncthreads_or(far);
  if (plain) {
    // the planets and the first tile's times as plain pairs
    for (int i = tid; i < spr * J; i += block) {
      const int64_t at = (sys0 + i / J) * (5 * J + 1) + 5 * (i % J);
      if (sys0 + i / J < a.n_sys && dbg_ok(a.invalid, at < a.n_sys * (5 * J + 1), kDbgParam, at))
        planet_plain(m.pl[i], a.params[at]);
    }
    const Split3 tr3 = split3(a.t[0]);
    for (int k = tid; k < min(tile, a.n_obs); k += block)
      sub_ds(split3(a.t[k]), tr3, m.obs[k], m.obs[tile + k]);
    __syncthreads();
  }
  int slot = tid >> lg;
  if (!dbg_ok(a.invalid, slot < spr, kDbgSmem, slot)) slot = 0;
  float n_max = 0.0f;                            // the system's shortest period
#pragma unroll
  for (int j = 0; j < J; ++j) n_max = fmaxf(n_max, m.pl[slot * J + j].n);
  MeanForm form;
  form.brief = !plain && n_max <= kPairMaxFreq;
  form.some = __any_sync(0xffffffffu, form.brief);
  form.all = __all_sync(0xffffffffu, form.brief);
  systems<J, RESID, DEMC, true>(a, smem, lg, tile, ntiles, out, resid_out, plain, form,
                                n_max > kPairExactFreq ? a.t : nullptr, gam, poison);
}

// RESID: also the per-system max Kepler residual.  DEMC: the batch is a
// DE-MC step's proposals (a.demc): formed in the prologue, Metropolis
// decision in the epilogue; plain evaluations contain neither.
template <int J, bool RESID, bool DEMC>
__global__ void __maxnreg__(64)
chi2_mixed_warp_kernel(UniformArgs a, int lg, int tile, int ntiles, float *__restrict__ out,
                       float *__restrict__ resid_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  // everything written by earlier grids in the stream is visible after the
  // wait; the next grid may then start placing its CTAs (it waits likewise)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int block = blockDim.x;
  const int tid = threadIdx.x;
  const int G = 1 << lg;
  const int spr = block >> lg;                   // systems of this CTA
  const WarpSmem<J> m(smem, spr, tile, block >> 5);
  float *tab_s = m.tab, *gam_s = m.gam, *obs_s = m.obs;
  PlanetP *pl_s = m.pl;

  const int64_t sys0 = (int64_t)blockIdx.x * spr;
  const int nitems = spr * (J + 1);
  const int step = G * kChunk;                   // a power of two
  const int nk0 = min(tile, a.n_obs);
  const int npad0 = round_up_pow2(nk0, step);

  // ---- prologue: every global load first ----
  const double t_ref = a.n_obs > 0 ? a.t[0] : a.t0;
  double p[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (tid < nitems) load_item<J, DEMC>(tid, spr, sys0, a, p);
  // the observations are staged from the last thread down, so that in a
  // large CTA other warps convert them than set the planets up
  const int ob = block - 1 - tid;
  const bool has0 = ob < nk0 && dbg_ok(a.invalid, ob < a.n_obs, kDbgObs, ob);
  const bool has1 = ob + block < nk0 && dbg_ok(a.invalid, ob + block < a.n_obs, kDbgObs,
                                               ob + block);
  double t0v = 0.0, v0v = 0.0, s0v = 1.0, t1v = 0.0, v1v = 0.0, s1v = 1.0;
  if (has0) { t0v = a.t[ob]; v0v = a.v[ob]; s0v = a.sigma[ob]; }
  if (has1) { t1v = a.t[ob + block]; v1v = a.v[ob + block]; s1v = a.sigma[ob + block]; }
  ang_tab_load<false>(tab_s, tid, block);

  // the reference time's split, needed by the threads that stage
  Split3 tr3 = {0.0f, 0.0f, 0.0f};
  if (ob < npad0) tr3 = split3(t_ref);
  const float jit2 = d2f(a.jitter2);
  bool far = false, wide = false;
  if (tid < nitems)
    wide = setup_item<J>(tid, spr, sys0, a.n_sys, p, t_ref, a.t0, pl_s, gam_s, a.invalid);
  for (int i = tid + block; i < nitems; i += block) {       // more items than threads
    double q[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    load_item<J, DEMC>(i, spr, sys0, a, q);
    wide |= setup_item<J>(i, spr, sys0, a.n_sys, q, t_ref, a.t0, pl_s, gam_s, a.invalid);
  }
  if (ob < npad0)
    far |= stage_obs(obs_s, tile, ob, has0, t0v, v0v, s0v, tr3, jit2, false, a.invalid);
  if (ob + block < npad0)
    far |= stage_obs(obs_s, tile, ob + block, has1, t1v, v1v, s1v, tr3, jit2, false, a.invalid);
  for (int k = ob + 2 * block; k < npad0; k += block) {
    const bool real = k < nk0 && dbg_ok(a.invalid, k < a.n_obs, kDbgObs, k);
    far |= stage_obs(obs_s, tile, k, real, real ? a.t[k] : 0.0, real ? a.v[k] : 0.0,
                     real ? a.sigma[k] : 1.0, tr3, jit2, false, a.invalid);
  }
  if (ntiles > 1) far |= far_later(a.t, tile, a.n_obs);
  wide = __syncthreads_or(wide || far);

  int slot = tid >> lg;
  if (!dbg_ok(a.invalid, slot < spr, kDbgSmem, slot)) slot = 0;
  const float gam = gam_s[slot];
  float poison = 0.0f * gam;                     // NaN for an invalid system
#pragma unroll
  for (int j = 0; j < J; ++j) poison += 0.0f * pl_s[slot * J + j].e;
  if (wide)
    wide_systems<J, RESID, DEMC>(a, smem, lg, tile, ntiles, out, resid_out, far, gam, poison);
  else
    systems<J, RESID, DEMC, false>(a, smem, lg, tile, ntiles, out, resid_out, false, {}, nullptr,
                                   gam, poison);
}

// Variants: 0 plain, 1 with the Kepler residual, 2 DE-MC step.
template <int J>
const void *warp_kernel_fn(int variant) {
  switch (variant) {
    case 0: return reinterpret_cast<const void *>(chi2_mixed_warp_kernel<J, false, false>);
    case 1: return reinterpret_cast<const void *>(chi2_mixed_warp_kernel<J, true, false>);
    case 2: return reinterpret_cast<const void *>(chi2_mixed_warp_kernel<J, false, true>);
  }
  return nullptr;
}

const void *warp_kernel_for(int J, int variant) {
  switch (J) {
    case 1: return warp_kernel_fn<1>(variant);
    case 2: return warp_kernel_fn<2>(variant);
    case 3: return warp_kernel_fn<3>(variant);
    case 4: return warp_kernel_fn<4>(variant);
    case 5: return warp_kernel_fn<5>(variant);
    case 6: return warp_kernel_fn<6>(variant);
    case 7: return warp_kernel_fn<7>(variant);
    case 8: return warp_kernel_fn<8>(variant);
  }
  return nullptr;
}

// CTAs of the kernel resident per SM (occupancy API), remembered per device,
// planet count, block and shared-memory size; 0 when the shape does not fit.
// The shared-memory limit is not remembered here: it belongs to the kernel, not
// to a size.
std::mutex g_occ_mu;
std::map<std::tuple<int, int, int, size_t>, int> g_occ;

int blocks_per_sm(int J, int variant, int block, size_t smem) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 1;                                    // no device: shapes stay valid
  }
  const void *fn = warp_kernel_for(J, variant);
  if (!fn) return 0;
  if (raise_smem_limit(fn, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const auto key = std::make_tuple(dev * 16 + J, block, variant, smem);
  {
    std::lock_guard<std::mutex> lk(g_occ_mu);
    auto it = g_occ.find(key);
    if (it != g_occ.end()) return it->second;
  }
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, block, smem) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  std::lock_guard<std::mutex> lk(g_occ_mu);
  g_occ[key] = n;
  return n;
}

size_t warp_smem(int J, int G, int block, int n_obs) {
  return WarpLayout(block / G, J, warp_obs_tile(n_obs, G), block / 32).total;
}

int log2_lanes(int G) {
  int lg = 3;
  while ((8 << (lg - 3)) < G) ++lg;
  return lg;
}

}  // namespace

bool warp_tile_ok(int G, int block) {
  const bool lanes = G == 8 || G == 16 || G == 32 || G == 64 || G == 128;
  return lanes && block >= 32 && block <= 1024 && !(block & 31) && block % G == 0;
}

bool warp_lanes_fit(int G, int n_obs) { return G == 8 || n_obs >= G * kChunk; }

// Resident CTAs per SM of `block` threads at the kernel's 64 registers and
// `smem` bytes: the occupancy API's answer by arithmetic (the choice below
// asks for 145 shapes).
static int warp_occupancy(int block, size_t smem, int smem_sm) {
  const int by_regs = 65536 / (64 * block);
  const int by_smem = (int)((size_t)smem_sm / (smem + 1024));      // 1 KB reserved per CTA
  return std::min(std::min(by_regs, 2048 / block), std::min(by_smem, 32));
}

static Tile pick_warp_tile(int64_t n_sys, int n_pl, int n_obs, bool multi_warp) {
  // Predicted clocks of one SM for every shape of G lanes per system and W
  // warps per CTA, the smallest wins.  An SM runs ceil(CTAs / n_sm) CTAs,
  // each costing its four sub-partitions
  //  - kEval clocks per warp and planet for every observation of a lane (the
  //    measured steady state of the packed body), or the body's latency
  //    shared by the resident warps where they are too few to cover it
  //    (kChain clocks per chunk of kChunk observations);
  //  - the prologue's instructions: kSetup clocks per warp of (system,
  //    planet) items, kStage per warp of staged observations.
  // Few lanes per system share the staged observations and the planets'
  // setup among many systems (2^20 x 4 x 256: 1963 us at G = 8 against 2539
  // at G = 32), many lanes spread a small batch over the SMs (300 x 3 x 101:
  // 4.3 us at G = 32, 5.1 at 16; 256 x 4 x 256: G = 64); a CTA count just
  // above a multiple of the SM count leaves most of them idle at the end
  // (4096 x 4 x 256: 11.3 us in 152 CTAs of 27 warps, 13.2 in 256 of 16).
  // W counts half as rounded up to whole warps per sub-partition (9-warp
  // CTAs measured between the two).
  constexpr double kEval = 68.0, kChain = 560.0, kSetup = 600.0, kStage = 180.0;
  const int64_t n_sm = sm_count() > 1 ? sm_count() : 152;     // no device: a GB300's shapes
  int dev = 0, smem_sm = 228 * 1024;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
          cudaSuccess) {
    cudaGetLastError();
    smem_sm = 228 * 1024;                        // no device: shapes stay valid
  }
  Tile best{8, 128, 0, 3};
  double best_cost = 1e300;
  for (int G : {8, 16, 32, 64, 128}) {
    if (G > 32 && (!multi_warp || !warp_lanes_fit(G, n_obs))) continue;
    const int npad = round_up(n_obs > 0 ? n_obs : 1, G * kChunk);
    const double chunks = (double)npad / (G * kChunk);
    for (int W = 4; W <= 32; ++W) {
      const int block = 32 * W;
      if (block % G) continue;
      const int occ = warp_occupancy(block, warp_smem(n_pl, G, block, n_obs), smem_sm);
      if (occ < 1) continue;
      const int64_t spc = block / G;                 // systems per CTA
      const int64_t per_sm = ((n_sys + spc - 1) / spc + n_sm - 1) / n_sm;
      const int resident = (int)std::min<int64_t>(per_sm, occ);
      const int quads = (W + 3) / 4;                 // warps of the fullest sub-partition
      const double load = resident == 1 ? quads : 0.5 * (0.25 * W + quads);
      const double chunk = std::max(kEval * kChunk, kChain / (0.25 * W * resident));
      const double items = (double)((spc * n_pl + 31) / 32), stage = (double)((npad + 31) / 32);
      const double cost = (double)per_sm * (load * n_pl * chunks * chunk +
                                            0.25 * (items * kSetup + stage * kStage));
      if (cost < best_cost * (1.0 - 1e-9)) {
        best_cost = cost;
        best = Tile{G, block, 0, 3};
      }
    }
  }
  best.obs_tile = warp_obs_tile(n_obs, best.G);
  return best;
}

// The choice is the same for every call of a size: remembered, up to a
// bounded number of sizes.
Tile warp_tile(int64_t n_sys, int n_pl, int n_obs, bool multi_warp) {
  typedef std::tuple<int64_t, int, int, int, int> Key;
  static std::mutex mu;
  static std::map<Key, Tile> known;
  const Key key(n_sys, n_pl, n_obs, multi_warp, sm_count());
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = known.find(key);
    if (it != known.end()) return it->second;
  }
  const Tile t = pick_warp_tile(n_sys, n_pl, n_obs, multi_warp);
  std::lock_guard<std::mutex> lk(mu);
  if (known.size() >= 256) known.clear();
  known[key] = t;
  return t;
}

cudaError_t launch_chi2_mixed_warp(const UniformArgs &a, const Tile &tile, float *out,
                                   float *resid, cudaStream_t st) {
  const int G = tile.G, block = tile.block;
  if (!warp_tile_ok(G, block)) return cudaErrorInvalidValue;
  // a DE-MC step reports no residual (the DE-MC entry point has none)
  const int variant = a.demc.states ? 2 : (resid != nullptr ? 1 : 0);
  if (variant == 2) resid = nullptr;
  const void *fn = warp_kernel_for(a.n_pl, variant);
  if (!fn) return cudaErrorInvalidValue;
  const int spr = block / G;
  const int obs_tile = warp_obs_tile(a.n_obs, G);
  const size_t smem = WarpLayout(spr, a.n_pl, obs_tile, block / 32).total;
  if (blocks_per_sm(a.n_pl, variant, block, smem) < 1) return cudaErrorInvalidConfiguration;
  const int64_t ctas = (a.n_sys + spr - 1) / spr;
  if (ctas > 0x7fffffff) return cudaErrorInvalidConfiguration;
  UniformArgs args = a;
  int lg = log2_lanes(G), tl = obs_tile, nt = (a.n_obs + obs_tile - 1) / obs_tile;
  void *params[] = {&args, &lg, &tl, &nt, &out, &resid};
  // programmatic stream serialisation (the kernel's griddepcontrol.wait
  // keeps it ordered after the grids before it), not under stream capture
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return cudaGetLastError();
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace kc
