// GRPO step signals (Phase 2), JAGG aggregation (Phase 3) and gradient reductions.
//
// Both backbone families of Eq. logprob have a transition mean that is affine in the model
// output y_j (the velocity v_j or the noise prediction eps_j): mu_j = a_j z_j + c_j y_j, with
//   rectified flow       a_j = 1,                        c_j = t_{j+1} - t_j;
//   epsilon prediction   a_j = alpha_{j+1} / alpha_j,    c_j = -alpha_{j+1} (sigma_j / alpha_j
//                                                               - sigma_{j+1} / alpha_{j+1})
// ((alpha, sigma) the diffusion schedule at the window's times).  So r_ij = z_{j+1} - mu_j and
// d logp / d y_ij = r_ij c_j / sigma_j^2 for both, and one set of kernels serves both.
//
// grpo_step_signals runs in three launches:
//   1. ||r_ij||^2, one CTA per (i, j, chunk of D), partial sums in f64 written to the
//      workspace (fixed order: deterministic); the first CTA of a sample also forms its
//      advantage A_i (Eq. advantage) from the group's rewards;
//   2. a warp per (i, j): log-prob (Eq. logprob), ratio, clip decision (Eq. grpo_loss), the
//      coefficient k_ij = scale (-A_i) rho_ij c_j / sigma_j^2 (0 when clipped);
//   3. one elementwise pass writes s_ij = k_ij r_ij and/or the aggregated cotangents
//      sum_j (1 - alpha_j) s_ij and sum_j alpha_j s_ij (Eq. alpha, Eq. s_base_corr).
// The v-hat / z tiles of a window are read twice; at the paper's shapes they fit in L2.
// f64 runs at a small fraction of the f32 rate here, so each f64 value is formed once (the
// coefficients by one thread per CTA, a chunk's sum by four warps): a window of 4 x 4 steps
// of 262144 bf16 elements took 80 us with an f64 coefficient set and butterfly in every thread
// and five launches, 67 us with the log-prob part repeated by every CTA of the elementwise
// pass (two launches), and takes 28 to 32 us like this (reading and writing its 38 MB once is
// 5.6 us; the kernels alone take 11.8, 6.2 and 7.7); 8 x 4 steps of 16384 elements 37 -> 25 to 27 us.
#include <mutex>

#include "common.cuh"

namespace jagg {

int unit_status_signals(unsigned* v, int clear) { return read_unit_status(v, clear); }

namespace {

constexpr int SIG_THREADS = 1024;
constexpr int SIG_PER_THREAD = 8;  // consecutive elements: two 16-byte loads of each f32 row
constexpr int SIG_CHUNK = SIG_THREADS * SIG_PER_THREAD;  // elements of D per CTA of the residual sums
constexpr int APPLY_THREADS = 256;

// An f64 mean coefficient as an unevaluated sum of two floats (hi + lo).  Rounding a_j or c_j
// to one float shifts r_ij by the same relative amount at every element, an error that does
// not average out over D and reaches the log-prob as ~1e-7 * sqrt(D) |z| |r| / sigma^2.
struct Coef2 {
  float hi, lo;
};
__device__ __forceinline__ Coef2 split_coef(double x) {
  const float hi = (float)x;
  return Coef2{hi, (float)(x - (double)hi)};
}
// r = z1 - a z0 - c y: the hi products cancel most of z1 exactly inside the first two fmas; the
// lo terms are small corrections.
__device__ __forceinline__ float resid(float z1, float z0, float y, Coef2 a, Coef2 c) {
  float r = fmaf(-a.hi, z0, z1);
  r = fmaf(-c.hi, y, r);
  r = fmaf(-a.lo, z0, r);
  return fmaf(-c.lo, y, r);
}

// The mean coefficients (a_j, c_j) of one step: the flow Euler step, or (eps) the DDIM step
// of the schedule values a0 = alpha_j, a1 = alpha_{j+1}, s0 = sigma_j, s1 = sigma_{j+1}.
// False (and a = c = 0) when an alpha is not positive.  The step signals and the rollout
// sampler both take their coefficients from here, so both see the same f64 values.
__device__ __forceinline__ bool mean_coef(double t0, double t1, bool eps, double a0, double a1, double s0, double s1,
                                          double* a, double* c) {
  if (!eps) {
    *a = 1.0;
    *c = t1 - t0;
    return true;
  }
  if (a0 > 0.0 && a1 > 0.0) {
    *a = a1 / a0;
    *c = -a1 * (s0 / a0 - s1 / a1);
    return true;
  }
  *a = 0.0;
  *c = 0.0;
  return false;
}

// Elements k .. k + 7 of a row (zeros past D).  `vec`: the row is 16-byte aligned.
__device__ __forceinline__ void load8(const float* p, int64_t k, int64_t D, bool vec, float (&x)[8]) {
  if (vec && k + 8 <= D) {
    const float4 a = *reinterpret_cast<const float4*>(p + k), b = *reinterpret_cast<const float4*>(p + k + 4);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
    x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = k + e < D ? p[k + e] : 0.f;
  }
}
__device__ __forceinline__ void load8_any(const void* p, int64_t base, int is_f32, int64_t k, int64_t D, bool vec,
                                          float (&x)[8]) {
  if (is_f32) {
    load8(static_cast<const float*>(p) + base, k, D, vec, x);
  } else if (vec && k + 8 <= D) {
    const uint4 raw = *reinterpret_cast<const uint4*>(static_cast<const bf16*>(p) + base + k);
    const bf16* h = reinterpret_cast<const bf16*>(&raw);
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = __bfloat162float(h[e]);
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e)
      x[e] = k + e < D ? __bfloat162float(static_cast<const bf16*>(p)[base + k + e]) : 0.f;
  }
}

// sum over the CTA's chunk of D of one f32 value per thread (the sum of r^2 over the thread's
// 8 consecutive elements, blockIdx.x * SIG_CHUNK + 8 threadIdx.x + ...) in f64, in a fixed
// order; valid in thread 0.  The f32 values meet in shared memory and 128 threads fold 8
// each, so f64 adds run on full warps.  The rollout sampler and the step signals share it
// and the element-to-thread map, so equal residuals give equal log-probs.
__device__ __forceinline__ double chunk_sum(float part) {
  __shared__ float vals[SIG_THREADS];
  __shared__ double red[4];
  vals[threadIdx.x] = part;
  __syncthreads();
  if (threadIdx.x < 128) {
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < SIG_THREADS / 128; ++q) s += (double)vals[q * 128 + threadIdx.x];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x / 32] = s;
  }
  __syncthreads();
  return threadIdx.x == 0 ? (red[0] + red[1]) + (red[2] + red[3]) : 0.0;
}
// sum of a row's chunk partials by one warp, in a fixed order (every lane gets it).
__device__ __forceinline__ double sum_partials(const double* partial, int chunks) {
  double s = 0.0;
  for (int c = threadIdx.x & 31; c < chunks; c += 32) s += partial[c];
  return warp_sum(s);
}

// Eq. logprob from the squared residual norm.  Written with explicitly rounded operations so
// that no call site contracts it into a different fused multiply-add: the rollout sampler
// and the step signals must agree to the last bit.
__device__ __forceinline__ double gauss_logp(double rr, double sg, int64_t D) {
  const double quad = __ddiv_rn(rr, __dmul_rn(2.0, __dmul_rn(sg, sg)));
  const double norm = __dmul_rn((double)D, log(__dmul_rn(sqrt(2.0 * 3.14159265358979323846), sg)));
  return __dsub_rn(-quad, norm);
}

// The inputs of one window's step signals; sched_alpha == nullptr selects the rectified-flow
// step.  vec: every row of v and z starts on a 16-byte boundary.
struct Window {
  const void* v;
  int v_f32, vec;
  const float* z;
  const double* t;
  const double* sched_alpha;
  const double* sched_sigma;
  int G, W;
  int64_t D;
};

// The mean coefficients of step j of the window (false: a bad schedule).
__device__ __forceinline__ bool window_coef(const Window& w, int j, double* a, double* c) {
  const bool eps = w.sched_alpha != nullptr;
  return mean_coef(w.t[j], w.t[j + 1], eps, eps ? w.sched_alpha[j] : 0.0, eps ? w.sched_alpha[j + 1] : 0.0,
                   eps ? w.sched_sigma[j] : 0.0, eps ? w.sched_sigma[j + 1] : 0.0, a, c);
}

// Advantage of sample i by one warp: A_i = clamp((r_i - mean) / (std + eps), +-clip).
__device__ __forceinline__ void advantage(const float* rewards, int G, int i, double adv_eps, double adv_clip,
                                          double* adv) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int g = lane; g < G; g += 32) s += (double)rewards[g];
  const double mu = warp_sum(s) / G;
  s = 0.0;
  for (int g = lane; g < G; g += 32) {
    const double d = (double)rewards[g] - mu;
    s += d * d;
  }
  s = warp_sum(s);
  if (lane != 0) return;
  const double sd = G > 1 ? sqrt(s / (G - 1)) : 0.0;
  const double a = ((double)rewards[i] - mu) / (sd + adv_eps);
  adv[i] = a > adv_clip ? adv_clip : (a < -adv_clip ? -adv_clip : a);
}

// grid: (chunks, G*W).  Bound by reading v and z once from DRAM; every load of a thread is
// issued before the first use.
__global__ void __launch_bounds__(SIG_THREADS) resid_norm_kernel(Window w, const float* rewards, double adv_eps,
                                                                 double adv_clip, double* adv, double* partial) {
  pdl_wait();
  const int ij = blockIdx.y;
  const int i = ij / w.W, j = ij % w.W;
  const float* z0 = w.z + ((int64_t)i * (w.W + 1) + j) * w.D;
  const int64_t vb = ((int64_t)i * w.W + j) * w.D;
  const int64_t k = (int64_t)blockIdx.x * SIG_CHUNK + (int64_t)threadIdx.x * SIG_PER_THREAD;
  float x0[8], x1[8], y[8];
  load8(z0, k, w.D, w.vec, x0);
  load8(z0 + w.D, k, w.D, w.vec, x1);
  load8_any(w.v, vb, w.v_f32, k, w.D, w.vec, y);
  __shared__ Coef2 coef[2];
  if (threadIdx.x == 0) {
    double ad, cd;
    if (!window_coef(w, j, &ad, &cd) && blockIdx.x == 0) set_device_status(JAGG_DEV_BADARG);
    coef[0] = split_coef(ad);
    coef[1] = split_coef(cd);
  }
  __syncthreads();
  const Coef2 a = coef[0], c = coef[1];
  float part = 0.f;
#pragma unroll
  for (int e = 0; e < 8; ++e) {  // elements past D loaded as zeros: r = 0
    const float r = resid(x1[e], x0[e], y[e], a, c);
    part = fmaf(r, r, part);
  }
  const double s = chunk_sum(part);
  if (threadIdx.x == 0) partial[(int64_t)ij * gridDim.x + blockIdx.x] = s;
  if (blockIdx.x == 0 && j == 0 && threadIdx.x < 32) advantage(rewards, w.G, i, adv_eps, adv_clip, adv);
}

// One warp per (i, j).  What the elementwise pass needs of a step goes back into the workspace:
// mc[j] = the mean coefficients (a.hi, a.lo, c.hi, c.lo), and the signal's coefficient and
// the aggregation weight (k, alpha) over the first of the step's own partial sums.
__global__ void __launch_bounds__(32) logprob_kernel(Window w, double* partial, int chunks, const double* sigma,
                                                     const double* logp_old, const double* adv, double clip_eps,
                                                     double scale, int aggregate, double* logp_new, double* ratio,
                                                     uint8_t* clipped, float4* mc) {
  pdl_wait();
  const int ij = blockIdx.x;
  const int i = ij / w.W, j = ij % w.W;
  const double rr = sum_partials(partial + (int64_t)ij * chunks, chunks);
  if (threadIdx.x != 0) return;
  double am, c;
  window_coef(w, j, &am, &c);
  const double sg = sigma[j];
  const double lp = gauss_logp(rr, sg, w.D);
  const double rho = exp(lp - logp_old[ij]);
  const double a = adv[i];
  const bool clip = (a > 0.0 && rho > 1.0 + clip_eps) || (a < 0.0 && rho < 1.0 - clip_eps);
  logp_new[ij] = lp;
  ratio[ij] = rho;
  clipped[ij] = clip ? 1 : 0;
  float2 q = make_float2(clip ? 0.f : (float)(scale * (-a) * rho * c / (sg * sg)), 0.f);
  if (aggregate) {
    const double den = w.t[0] - w.t[w.W - 1];
    if (den != 0.0)
      q.y = (float)((w.t[0] - w.t[j]) / den);
    else
      set_device_status(JAGG_DEV_BADARG);
  }
  *reinterpret_cast<float2*>(partial + (int64_t)ij * chunks) = q;
  if (i == 0) {
    const Coef2 ca = split_coef(am), cc = split_coef(c);
    mc[j] = make_float4(ca.hi, ca.lo, cc.hi, cc.lo);
  }
}

// grid: (ceil(D / 4 / APPLY_THREADS), G).  Each thread: 4 consecutive elements of D over every
// step.
__global__ void __launch_bounds__(APPLY_THREADS) apply_kernel(Window w, const double* partial, int chunks,
                                                              const float4* mc, float* s_out, float* cot_out,
                                                              int vec_out) {
  pdl_wait();
  const int i = blockIdx.y;
  const int64_t D = w.D;
  const int64_t kbase = ((int64_t)blockIdx.x * APPLY_THREADS + threadIdx.x) * 4;
  if (kbase >= D) return;
  const bool full = kbase + 4 <= D;
  auto load4 = [&](const float* p, bool vec, float (&x)[4]) {
    if (vec && full) {
      const float4 f = *reinterpret_cast<const float4*>(p + kbase);
      x[0] = f.x; x[1] = f.y; x[2] = f.z; x[3] = f.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = kbase + e < D ? p[kbase + e] : 0.f;
    }
  };
  auto store4 = [&](float* p, const float (&x)[4]) {
    if (vec_out && full) {
      *reinterpret_cast<float4*>(p + kbase) = make_float4(x[0], x[1], x[2], x[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (kbase + e < D) p[kbase + e] = x[e];
    }
  };
  float base[4] = {0.f, 0.f, 0.f, 0.f}, corr[4] = {0.f, 0.f, 0.f, 0.f};
  float x0[4];
  load4(w.z + (int64_t)i * (w.W + 1) * D, w.vec, x0);
#pragma unroll 4
  for (int j = 0; j < w.W; ++j) {
    const int64_t vb = ((int64_t)i * w.W + j) * D;
    float x1[4], y[4], s[4];
    load4(w.z + ((int64_t)i * (w.W + 1) + j + 1) * D, w.vec, x1);
    if (w.v_f32) {
      load4(static_cast<const float*>(w.v) + vb, w.vec, y);
    } else if (w.vec && full) {
      const uint2 raw = *reinterpret_cast<const uint2*>(static_cast<const bf16*>(w.v) + vb + kbase);
      const bf16* h = reinterpret_cast<const bf16*>(&raw);
#pragma unroll
      for (int e = 0; e < 4; ++e) y[e] = __bfloat162float(h[e]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        y[e] = kbase + e < D ? __bfloat162float(static_cast<const bf16*>(w.v)[vb + kbase + e]) : 0.f;
    }
    const float2 q = *reinterpret_cast<const float2*>(partial + ((int64_t)i * w.W + j) * chunks);
    const float4 m = mc[j];
    const Coef2 a{m.x, m.y}, c{m.z, m.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      s[e] = q.x * resid(x1[e], x0[e], y[e], a, c);
      base[e] += (1.f - q.y) * s[e];
      corr[e] += q.y * s[e];
      x0[e] = x1[e];
    }
    if (s_out) store4(s_out + vb, s);
  }
  if (cot_out) {
    store4(cot_out + (int64_t)i * D, base);
    store4(cot_out + ((int64_t)w.G + i) * D, corr);
  }
}

// Rollout sampler step.  grid: (chunks, G).  z_{j+1} = a z_j + c y + sigma xi, rounded to f32
// and stored, then its residual against the mean enters the same chunk sums as the signals.
struct RolloutStep {
  const void* y;
  int y_f32, vec;  // vec: every row of y, z, xi and z_model starts on a 16-byte boundary
  const float* z_cur;
  const float* xi;
  float* z_next;
  void* z_model;  // optional dense [G, D] copy of z_next in the model's dtype (next forward's input)
  int zm_f32;
  int64_t D, z_ld, y_ld, xi_ld;
  double t0, t1, sigma, a0, a1, s0, s1;
  int eps;
  double* partial;
};

__global__ void __launch_bounds__(SIG_THREADS) rollout_step_kernel(RolloutStep p) {
  pdl_wait();
  const int i = blockIdx.y;
  const int64_t D = p.D;
  const int64_t k = (int64_t)blockIdx.x * SIG_CHUNK + (int64_t)threadIdx.x * SIG_PER_THREAD;
  float zc[8], y[8], xi[8];
  load8(p.z_cur + (int64_t)i * p.z_ld, k, D, p.vec, zc);
  load8_any(p.y, (int64_t)i * p.y_ld, p.y_f32, k, D, p.vec, y);
  load8(p.xi + (int64_t)i * p.xi_ld, k, D, p.vec, xi);
  __shared__ Coef2 coef[2];
  if (threadIdx.x == 0) {
    double ad, cd;
    if (!mean_coef(p.t0, p.t1, p.eps != 0, p.a0, p.a1, p.s0, p.s1, &ad, &cd) && blockIdx.x == 0 && i == 0)
      set_device_status(JAGG_DEV_BADARG);
    coef[0] = split_coef(ad);
    coef[1] = split_coef(cd);
  }
  __syncthreads();
  const Coef2 a = coef[0], c = coef[1];
  const float sg = (float)p.sigma;
  float zn[8];
  float part = 0.f;
#pragma unroll
  for (int e = 0; e < 8; ++e) {  // elements past D loaded as zeros: z_next = r = 0 there
    float m = fmaf(a.lo, zc[e], c.lo * y[e]);
    m = fmaf(c.hi, y[e], m);
    m = fmaf(a.hi, zc[e], m);
    zn[e] = fmaf(sg, xi[e], m);
    const float r = resid(zn[e], zc[e], y[e], a, c);
    part = fmaf(r, r, part);
  }
  float* z1 = p.z_next + (int64_t)i * p.z_ld;
  float* zmf = p.zm_f32 ? static_cast<float*>(p.z_model) : nullptr;
  bf16* zmb = p.zm_f32 ? nullptr : static_cast<bf16*>(p.z_model);
  if (p.vec && k + 8 <= D) {
    const float4 lo = make_float4(zn[0], zn[1], zn[2], zn[3]), hi = make_float4(zn[4], zn[5], zn[6], zn[7]);
    *reinterpret_cast<float4*>(z1 + k) = lo;
    *reinterpret_cast<float4*>(z1 + k + 4) = hi;
    if (zmf) {
      *reinterpret_cast<float4*>(zmf + (int64_t)i * D + k) = lo;
      *reinterpret_cast<float4*>(zmf + (int64_t)i * D + k + 4) = hi;
    } else if (zmb) {
      uint4 raw;
      __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&raw);
#pragma unroll
      for (int e = 0; e < 4; ++e) h[e] = __floats2bfloat162_rn(zn[2 * e], zn[2 * e + 1]);
      *reinterpret_cast<uint4*>(zmb + (int64_t)i * D + k) = raw;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (k + e >= D) break;
      z1[k + e] = zn[e];
      if (zmf) zmf[(int64_t)i * D + k + e] = zn[e];
      if (zmb) zmb[(int64_t)i * D + k + e] = __float2bfloat16_rn(zn[e]);
    }
  }
  const double s = chunk_sum(part);
  if (threadIdx.x == 0) p.partial[(int64_t)i * gridDim.x + blockIdx.x] = s;
}

// One warp per sample.
__global__ void __launch_bounds__(32) rollout_logp_kernel(const double* partial, int chunks, double sigma, int64_t D,
                                                          double* logp, int64_t logp_ld) {
  pdl_wait();
  const int i = blockIdx.x;
  const double rr = sum_partials(partial + (int64_t)i * chunks, chunks);
  if (threadIdx.x == 0) logp[(int64_t)i * logp_ld] = gauss_logp(rr, sigma, D);
}

__global__ void check_alpha_kernel(const double* t, int W) {
  pdl_wait();
  if (threadIdx.x == 0 && blockIdx.x == 0 && !(t[0] - t[W - 1] != 0.0)) set_device_status(JAGG_DEV_BADARG);
}

__global__ void aggregate_kernel(const float* s, const double* t, int G, int W, int64_t D, float* cot) {
  pdl_wait();
  const int i = blockIdx.y;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= D) return;
  const double den = t[0] - t[W - 1];
  float base = 0.f, corr = 0.f;
  if (den != 0.0) {
    for (int j = 0; j < W; ++j) {
      const float al = (float)((t[0] - t[j]) / den);
      const float v = s[((int64_t)i * W + j) * D + k];
      base += (1.f - al) * v;
      corr += al * v;
    }
  }
  cot[(int64_t)i * D + k] = base;
  cot[((int64_t)G + i) * D + k] = corr;
}

__global__ void aggregate_span_kernel(const float* s, int64_t ld, const double* t, double t_first, double t_last, int G,
                                      int n, int64_t D, float* cot, int accumulate) {
  pdl_wait();
  const int i = blockIdx.y;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= D) return;
  const double den = t_first - t_last;
  float base = 0.f, corr = 0.f;
  for (int j = 0; j < n; ++j) {
    const float al = (float)((t_first - t[j]) / den);
    const float v = s[(int64_t)i * ld + (int64_t)j * D + k];
    base += (1.f - al) * v;
    corr += al * v;
  }
  float* b = cot + (int64_t)i * D + k;
  float* c = cot + ((int64_t)G + i) * D + k;
  if (accumulate) {
    *b += base;
    *c += corr;
  } else {
    *b = base;
    *c = corr;
  }
}

// ------------------------------------------------------------------ grad_reduce
constexpr int GR_BLOCKS = 1024;  // the most CTAs (rows of partial sums in the workspace)
constexpr int GR_THREADS = 256;
constexpr int GR_UNROLL = 4;
constexpr int GR_RUN = GR_THREADS * GR_UNROLL;  // float4 of a vector per CTA and iteration

// HAS_B: a second vector b (else <a, b> = |b|^2 = |a|^2 and b is not read); HAS_ACC: the
// update acc += alpha a.  A CTA walks runs of GR_RUN consecutive float4 of each vector; each
// thread issues its GR_UNROLL loads of every input before using any; f32 sums over 16 terms fold
// into f64.  Bound by DRAM.  CTAs per SM and cache policy by form, each at its best of 2 to 5 CTAs with streaming
// and with plain accesses (130 M elements; us with the sums' second launch where there are sums):
//   acc, a, b   4, plain      304   (streaming 315; 3 CTAs 309)
//   acc, a      4, plain      232   (streaming, 3 CTAs: 248)
//   a, b        5, streaming  175   (3 CTAs 220; plain 185)
//   a           3, streaming   91   (plain 107)
// 435, 236, 265 and 166 when a thread's eight loads were a grid apart, 1024 CTAs ran in more than one
// wave and one thread per sum added the partials.
constexpr int gr_ctas_per_sm(bool has_b, bool has_acc) { return has_acc ? 4 : has_b ? 5 : 3; }
template <bool PLAIN>
__device__ __forceinline__ float4 gr_load(const float4* p) { return PLAIN ? *p : __ldcs(p); }

template <bool HAS_B, bool HAS_ACC>
__global__ void __launch_bounds__(GR_THREADS) grad_reduce_kernel(const float* a, const float* b, int64_t P,
                                                                 float alpha, float* acc, double* partial) {
  pdl_wait();
  double sab = 0.0, saa = 0.0, sbb = 0.0;
  const int64_t nvec = P / 4;
  const float4* a4 = reinterpret_cast<const float4*>(a);
  const float4* b4 = reinterpret_cast<const float4*>(b);
  float4* c4 = reinterpret_cast<float4*>(acc);
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int64_t i0 = (int64_t)blockIdx.x * GR_RUN + threadIdx.x; i0 < nvec; i0 += (int64_t)gridDim.x * GR_RUN) {
    float4 x[GR_UNROLL], y[GR_UNROLL], c[GR_UNROLL];
#pragma unroll
    for (int r = 0; r < GR_UNROLL; ++r) {
      const int64_t q = i0 + r * GR_THREADS;
      const bool in = q < nvec;
      x[r] = in ? gr_load<HAS_ACC>(a4 + q) : zero;
      if constexpr (HAS_B) y[r] = in ? gr_load<HAS_ACC>(b4 + q) : zero;
      if constexpr (HAS_ACC) c[r] = in ? c4[q] : zero;
    }
    float fab = 0.f, faa = 0.f, fbb = 0.f;
#pragma unroll
    for (int r = 0; r < GR_UNROLL; ++r) {
      faa += x[r].x * x[r].x + x[r].y * x[r].y + x[r].z * x[r].z + x[r].w * x[r].w;
      if constexpr (HAS_B) {
        fab += x[r].x * y[r].x + x[r].y * y[r].y + x[r].z * y[r].z + x[r].w * y[r].w;
        fbb += y[r].x * y[r].x + y[r].y * y[r].y + y[r].z * y[r].z + y[r].w * y[r].w;
      }
      if constexpr (HAS_ACC) {
        const int64_t q = i0 + r * GR_THREADS;
        c[r].x += alpha * x[r].x; c[r].y += alpha * x[r].y; c[r].z += alpha * x[r].z; c[r].w += alpha * x[r].w;
        if (q < nvec) c4[q] = c[r];
      }
    }
    if constexpr (!HAS_B) fab = fbb = faa;
    sab += fab;
    saa += faa;
    sbb += fbb;
  }
  // scalar tail (P % 4), handled by block 0
  if (blockIdx.x == 0) {
    for (int64_t k = nvec * 4 + threadIdx.x; k < P; k += GR_THREADS) {
      const float x = a[k], y = b ? b[k] : a[k];
      sab += (double)x * y;
      saa += (double)x * x;
      sbb += (double)y * y;
      if (acc) acc[k] += alpha * x;
    }
  }
  if (!partial) return;
  sab = warp_sum(sab);
  saa = warp_sum(saa);
  sbb = warp_sum(sbb);
  __shared__ double red[3][GR_THREADS / 32];
  const int w = threadIdx.x / 32;
  if ((threadIdx.x & 31) == 0) {
    red[0][w] = sab;
    red[1][w] = saa;
    red[2][w] = sbb;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
    for (int i = 0; i < GR_THREADS / 32; ++i) s += red[threadIdx.x][i];
    partial[(int64_t)blockIdx.x * 3 + threadIdx.x] = s;
  }
}

// Three warps: the sums over the CTAs' partials of <a, b>, |a|^2, |b|^2.
__global__ void __launch_bounds__(96) grad_reduce_final(const double* partial, int blocks, double* out3) {
  pdl_wait();
  const int w = threadIdx.x / 32;
  double s = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x & 31; i < blocks; i += 32) s += partial[(int64_t)i * 3 + w];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) out3[w] = s;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// The mean coefficients (a_j, c_j as hi, lo floats) at the head of the signals workspace.
int64_t mean_coef_bytes(int W) { return ((int64_t)2 * W * 8 + 15) / 16 * 16; }

}  // namespace

}  // namespace jagg

using namespace jagg;

// ------------------------------------------------------------------ C ABI
extern "C" int64_t jagg_signals_workspace_bytes(int G, int W, int64_t D) {
  if (G <= 0 || W <= 0 || D <= 0) return 0;
  const int64_t chunks = (D + SIG_CHUNK - 1) / SIG_CHUNK;
  // the mean coefficients, the partial sums, and G W floats that no kernel uses any more: the
  // size stays what callers, and the bound of the static variant, have been given
  return mean_coef_bytes(W) + (int64_t)G * W * chunks * 8 + (int64_t)G * W * 4 + 64;
}

namespace jagg {
namespace {
int step_signals(const char* name, const void* v_hat, int v_dtype, const float* z, const double* t,
                 const double* sched_alpha, const double* sched_sigma, const double* sigma, const double* logp_old,
                 const float* rewards, int G, int W, int64_t D, double clip_eps, double adv_clip, double adv_eps,
                 double scale, float* s_out, float* cot_out, double* logp_new, double* ratio, uint8_t* clipped,
                 double* adv_out, void* ws, size_t ws_bytes, cudaStream_t stream) {
  JAGG_CHECK_ARG(G > 0 && W > 0 && D > 0, "%s: G=%d W=%d D=%lld must be positive", name, G, W, (long long)D);
  JAGG_CHECK_ARG(G <= 65535 && (int64_t)G * W <= 65535, "%s: G*W too large", name);
  JAGG_CHECK_ARG(v_dtype == JAGG_DTYPE_F32 || v_dtype == JAGG_DTYPE_BF16, "%s: bad v_dtype", name);
  JAGG_CHECK_ARG(v_hat && z && t && sigma && logp_old && rewards && logp_new && ratio && clipped && adv_out && ws,
                 "%s: null pointer", name);
  JAGG_CHECK_ARG(!cot_out || W >= 2, "%s: aggregation needs W >= 2", name);
  JAGG_CHECK_ARG(clip_eps >= 0.0 && adv_clip >= 0.0 && adv_eps >= 0.0, "%s: negative constant", name);
  const int64_t need = jagg_signals_workspace_bytes(G, W, D);
  if ((int64_t)ws_bytes < need) {
    set_last_error("%s: workspace %zu < %lld bytes", name, ws_bytes, (long long)need);
    return JAGG_ERR_WORKSPACE;
  }
  JAGG_CHECK_ARG(aligned16(ws), "%s: workspace not 16-byte aligned", name);
  const int chunks = (int)((D + SIG_CHUNK - 1) / SIG_CHUNK);
  float4* mc = static_cast<float4*>(ws);
  double* partial = reinterpret_cast<double*>(static_cast<char*>(ws) + mean_coef_bytes(W));
  const int vf32 = v_dtype == JAGG_DTYPE_F32;
  // 16-byte rows: z rows of D floats and v rows of D elements from aligned bases
  const bool vec = D % 8 == 0 && aligned16(v_hat) && aligned16(z);
  const bool vec_out = D % 4 == 0 && (!s_out || aligned16(s_out)) && (!cot_out || aligned16(cot_out));
  const Window win{v_hat, vf32, vec ? 1 : 0, z, t, sched_alpha, sched_sigma, G, W, D};
  const int tok = prof_start(stream);
  JAGG_CUDA_TRY(launch(resid_norm_kernel, dim3(chunks, G * W), SIG_THREADS, 0, stream, win, rewards, adv_eps,
                       adv_clip, adv_out, partial));
  JAGG_LAUNCHED();
  JAGG_CUDA_TRY(launch(logprob_kernel, G * W, 32, 0, stream, win, partial, chunks, sigma, logp_old, adv_out,
                       clip_eps, scale,
                                           cot_out ? 1 : 0, logp_new, ratio, clipped, mc));
  JAGG_LAUNCHED();
  if (s_out || cot_out) {
    const int gx = ceil_div(D, (int64_t)APPLY_THREADS * 4);
    JAGG_CUDA_TRY(launch(apply_kernel, dim3(gx, G), APPLY_THREADS, 0, stream, win, partial, chunks, mc, s_out,
                         cot_out, vec_out ? 1 : 0));
    JAGG_LAUNCHED();
  }
  // algorithmic bytes: v-hat and the W + 1 latents of every sample read once, the signals
  // (G W rows) or the cotangents (2G rows) written in f32
  const double out_rows = s_out ? (double)G * W : (cot_out ? 2.0 * G : 0.0);
  prof_stop(tok, stream, PROF_SIGNALS, 0.0,
            (double)D * ((double)G * W * (vf32 ? 4.0 : 2.0) + (double)G * (W + 1) * 4.0 + out_rows * 4.0));
  return JAGG_OK;
}
}  // namespace
}  // namespace jagg

extern "C" int grpo_step_signals(const void* v_hat, int v_dtype, const float* z, const double* t, const double* sigma,
                                 const double* logp_old, const float* rewards, int G, int W, int64_t D,
                                 double clip_eps, double adv_clip, double adv_eps, double scale, float* s_out,
                                 float* cot_out, double* logp_new, double* ratio, uint8_t* clipped, double* adv_out,
                                 void* ws, size_t ws_bytes, cudaStream_t stream) {
  return step_signals("grpo_step_signals", v_hat, v_dtype, z, t, nullptr, nullptr, sigma, logp_old, rewards, G, W, D,
                      clip_eps, adv_clip, adv_eps, scale, s_out, cot_out, logp_new, ratio, clipped, adv_out, ws,
                      ws_bytes, stream);
}

extern "C" int grpo_step_signals_eps(const void* eps_hat, int eps_dtype, const float* z, const double* t,
                                     const double* sched_alpha, const double* sched_sigma, const double* sigma,
                                     const double* logp_old, const float* rewards, int G, int W, int64_t D,
                                     double clip_eps, double adv_clip, double adv_eps, double scale, float* s_out,
                                     float* cot_out, double* logp_new, double* ratio, uint8_t* clipped,
                                     double* adv_out, void* ws, size_t ws_bytes, cudaStream_t stream) {
  JAGG_CHECK_ARG(sched_alpha && sched_sigma, "grpo_step_signals_eps: null schedule");
  return step_signals("grpo_step_signals_eps", eps_hat, eps_dtype, z, t, sched_alpha, sched_sigma, sigma, logp_old,
                      rewards, G, W, D, clip_eps, adv_clip, adv_eps, scale, s_out, cot_out, logp_new, ratio, clipped,
                      adv_out, ws, ws_bytes, stream);
}

extern "C" int64_t jagg_rollout_workspace_bytes(int G, int64_t D) {
  if (G <= 0 || D <= 0) return 0;
  return (int64_t)G * ((D + SIG_CHUNK - 1) / SIG_CHUNK) * 8 + 64;
}

extern "C" int jagg_rollout_step(const void* y_hat, int y_dtype, int64_t y_sample_stride, const float* z_cur,
                                 float* z_next, int64_t z_sample_stride, const float* xi, int64_t xi_sample_stride,
                                 int G, int64_t D, double t_cur, double t_next, double sigma, const double* sched,
                                 double* logp, int64_t logp_stride, void* z_model, int z_model_dtype, void* ws,
                                 size_t ws_bytes, cudaStream_t stream) {
  JAGG_CHECK_ARG(y_hat && z_cur && z_next && xi && logp && ws, "jagg_rollout_step: null pointer");
  JAGG_CHECK_ARG(G > 0 && G <= 65535 && D > 0, "jagg_rollout_step: bad G=%d or D=%lld", G, (long long)D);
  JAGG_CHECK_ARG(y_dtype == JAGG_DTYPE_F32 || y_dtype == JAGG_DTYPE_BF16, "jagg_rollout_step: bad y_dtype");
  JAGG_CHECK_ARG(sigma > 0.0, "jagg_rollout_step: sigma %g must be positive", sigma);
  const int64_t zl = z_sample_stride ? z_sample_stride : D, yl = y_sample_stride ? y_sample_stride : D,
                xl = xi_sample_stride ? xi_sample_stride : D;
  JAGG_CHECK_ARG(zl >= D && yl >= D && xl >= D, "jagg_rollout_step: a sample stride is below D");
  JAGG_CHECK_ARG(logp_stride >= 1, "jagg_rollout_step: logp_stride must be >= 1");
  JAGG_CHECK_ARG(!z_model || z_model_dtype == JAGG_DTYPE_F32 || z_model_dtype == JAGG_DTYPE_BF16,
                 "jagg_rollout_step: bad z_model_dtype");
  const int64_t need = jagg_rollout_workspace_bytes(G, D);
  if ((int64_t)ws_bytes < need) {
    set_last_error("jagg_rollout_step: workspace %zu < %lld bytes", ws_bytes, (long long)need);
    return JAGG_ERR_WORKSPACE;
  }
  JAGG_CHECK_ARG(aligned16(ws), "jagg_rollout_step: workspace not 16-byte aligned");
  const int chunks = (int)((D + SIG_CHUNK - 1) / SIG_CHUNK);
  const bool vec = D % 8 == 0 && zl % 4 == 0 && yl % 8 == 0 && xl % 4 == 0 && aligned16(y_hat) && aligned16(z_cur) &&
                   aligned16(z_next) && aligned16(xi) && (!z_model || aligned16(z_model));
  RolloutStep p{y_hat, y_dtype == JAGG_DTYPE_F32, vec ? 1 : 0, z_cur, xi, z_next, z_model, z_model_dtype == JAGG_DTYPE_F32,
                D, zl, yl, xl, t_cur, t_next, sigma,
                sched ? sched[0] : 0.0, sched ? sched[1] : 0.0, sched ? sched[2] : 0.0, sched ? sched[3] : 0.0,
                sched ? 1 : 0, static_cast<double*>(ws)};
  JAGG_CUDA_TRY(launch(rollout_step_kernel, dim3(chunks, G), SIG_THREADS, 0, stream, p));
  JAGG_LAUNCHED();
  JAGG_CUDA_TRY(launch(rollout_logp_kernel, G, 32, 0, stream, static_cast<double*>(ws), chunks, sigma, D, logp,
                       logp_stride));
  JAGG_LAUNCHED();
  return JAGG_OK;
}

extern "C" int jagg_aggregate(const float* s, const double* t_window, int G, int W, int64_t D, float* cot,
                              cudaStream_t stream) {
  JAGG_CHECK_ARG(s && t_window && cot, "jagg_aggregate: null pointer");
  JAGG_CHECK_ARG(G > 0 && G <= 65535 && D > 0, "jagg_aggregate: bad G=%d or D=%lld", G, (long long)D);
  JAGG_CHECK_ARG(W >= 2, "jagg_aggregate: W=%d, the endpoints must differ (W >= 2)", W);
  JAGG_CUDA_TRY(launch(check_alpha_kernel, 1, 32, 0, stream, t_window, W));
  JAGG_LAUNCHED();
  JAGG_CUDA_TRY(launch(aggregate_kernel, dim3(ceil_div(D, 256), G), 256, 0, stream, s, t_window, G, W, D, cot));
  JAGG_LAUNCHED();
  return JAGG_OK;
}

extern "C" int jagg_aggregate_span(const float* s, int64_t s_sample_stride, const double* t_steps, double t_first,
                                   double t_last, int G, int n, int64_t D, float* cot, int accumulate,
                                   cudaStream_t stream) {
  JAGG_CHECK_ARG(s && t_steps && cot, "jagg_aggregate_span: null pointer");
  JAGG_CHECK_ARG(G > 0 && G <= 65535 && n > 0 && D > 0, "jagg_aggregate_span: bad G=%d, n=%d or D=%lld", G, n,
                 (long long)D);
  JAGG_CHECK_ARG(t_first != t_last, "jagg_aggregate_span: the window endpoints must differ");
  const int64_t ld = s_sample_stride ? s_sample_stride : (int64_t)n * D;
  JAGG_CHECK_ARG(ld >= (int64_t)n * D, "jagg_aggregate_span: sample stride %lld below n * D", (long long)ld);
  JAGG_CUDA_TRY(launch(aggregate_span_kernel, dim3(ceil_div(D, 256), G), 256, 0, stream, s, ld, t_steps, t_first,
                       t_last, G, n, D, cot,
                                                                       accumulate));
  JAGG_LAUNCHED();
  return JAGG_OK;
}

extern "C" int jagg_route(int n_windows, double jagg_frac, const double* cos, double tau, uint8_t* route,
                          double* derived_frac) {
  JAGG_CHECK_ARG(n_windows > 0 && route, "jagg_route: n_windows=%d / null route", n_windows);
  if (!cos) {
    JAGG_CHECK_ARG(jagg_frac >= 0.0 && jagg_frac <= 1.0, "jagg_route: jagg_frac %g outside [0, 1]", jagg_frac);
    int n_jagg = (int)floor(jagg_frac * n_windows + 1e-9);
    if (n_jagg > n_windows) n_jagg = n_windows;
    for (int w = 0; w < n_windows; ++w) route[w] = w < n_jagg ? 1 : 0;
    if (derived_frac) *derived_frac = (double)n_jagg / n_windows;
    return JAGG_OK;
  }
  int prefix = 0;
  bool in_prefix = true;
  for (int w = 0; w < n_windows; ++w) {
    route[w] = cos[w] >= tau ? 1 : 0;
    if (in_prefix && route[w])
      ++prefix;
    else
      in_prefix = false;
  }
  if (derived_frac) *derived_frac = (double)prefix / n_windows;
  return JAGG_OK;
}

extern "C" int64_t jagg_grad_reduce_workspace_bytes(int64_t P) {
  (void)P;
  return (int64_t)GR_BLOCKS * 3 * 8;
}

extern "C" int grad_reduce(const float* a, const float* b, int64_t P, float alpha, float* acc, double* out3, void* ws,
                           size_t ws_bytes, cudaStream_t stream) {
  JAGG_CHECK_ARG(a && P > 0, "grad_reduce: null input or P=%lld", (long long)P);
  JAGG_CHECK_ARG(aligned16(a) && (!b || aligned16(b)) && (!acc || aligned16(acc)),
                 "grad_reduce: buffers must be 16-byte aligned");
  if (!acc && !out3) return JAGG_OK;
  if (out3) {
    if (!ws || (int64_t)ws_bytes < jagg_grad_reduce_workspace_bytes(P)) {
      set_last_error("grad_reduce: workspace too small");
      return JAGG_ERR_WORKSPACE;
    }
  }
  const int tok = prof_start(stream);
  double* part = out3 ? static_cast<double*>(ws) : nullptr;
  // one wave of resident CTAs, fewer for a short vector
  const int64_t runs = (P / 4 + GR_RUN - 1) / GR_RUN;
  const int wave = gr_ctas_per_sm(b != nullptr, acc != nullptr) * sm_count();
  const int most = wave < GR_BLOCKS ? wave : GR_BLOCKS;
  const int blocks = runs < 1 ? 1 : (runs < most ? (int)runs : most);
  if (b && acc)
    JAGG_CUDA_TRY(launch(grad_reduce_kernel<true, true>, blocks, GR_THREADS, 0, stream, a, b, P, alpha, acc, part));
  else if (b)
    JAGG_CUDA_TRY(launch(grad_reduce_kernel<true, false>, blocks, GR_THREADS, 0, stream, a, b, P, alpha, acc, part));
  else if (acc)
    JAGG_CUDA_TRY(launch(grad_reduce_kernel<false, true>, blocks, GR_THREADS, 0, stream, a, b, P, alpha, acc, part));
  else
    JAGG_CUDA_TRY(launch(grad_reduce_kernel<false, false>, blocks, GR_THREADS, 0, stream, a, b, P, alpha, acc, part));
  JAGG_LAUNCHED();
  if (out3) {
    JAGG_CUDA_TRY(launch(grad_reduce_final, 1, 96, 0, stream, static_cast<const double*>(ws), blocks, out3));
    JAGG_LAUNCHED();
  }
  // algorithmic bytes: a (and b) read, acc read and written
  prof_stop(tok, stream, PROF_GRAD_REDUCE, 0.0, 4.0 * P * (1.0 + (b ? 1.0 : 0.0) + (acc ? 2.0 : 0.0)));
  return JAGG_OK;
}

// ------------------------------------------------------------------ allocation-free variant
// Scratch for grpo_step_signals_static: compiled into the library, one copy per device.
static __device__ __align__(256) unsigned char g_signals_scratch[JAGG_SIGNALS_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_ptr[kMaxDevices] = {};

// The array's device address for the device of `stream`, which must be the current device
// (the address comes from a runtime query on the current device), looked up once per device.
// In host code `g_signals_scratch` names a host-side stand-in, never the device memory itself.
int scratch_for_stream(cudaStream_t stream, void** out) {
  int dev = 0, sdev = 0;
  JAGG_CUDA_TRY(cudaGetDevice(&dev));
  JAGG_CUDA_TRY(cudaStreamGetDevice(stream, &sdev));
  JAGG_CHECK_ARG(sdev == dev, "grpo_step_signals_static: the stream belongs to device %d, the current device is %d",
                 sdev, dev);
  JAGG_CHECK_ARG(dev >= 0 && dev < kMaxDevices, "grpo_step_signals_static: device %d out of range", dev);
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    JAGG_CUDA_TRY(cudaGetSymbolAddress(&p, g_signals_scratch));
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return JAGG_OK;
}
}  // namespace

extern "C" int grpo_step_signals_static(const void* v_hat, int v_dtype, const float* z, const double* t,
                                        const double* sigma, const double* logp_old, const float* rewards, int G,
                                        int W, int64_t D, double clip_eps, double adv_clip, double adv_eps,
                                        double scale, float* s_out, float* cot_out, double* logp_new,
                                        double* ratio, uint8_t* clipped, double* adv_out, cudaStream_t stream) {
  JAGG_CHECK_ARG(G > 0 && W > 0 && D > 0, "grpo_step_signals_static: G=%d W=%d D=%lld must be positive", G, W,
                 (long long)D);
  const int64_t need = jagg_signals_workspace_bytes(G, W, D);
  if (need > (int64_t)JAGG_SIGNALS_STATIC_SCRATCH_BYTES) {
    set_last_error("grpo_step_signals_static: needs %lld scratch bytes, more than the %d compiled in",
                   (long long)need, (int)JAGG_SIGNALS_STATIC_SCRATCH_BYTES);
    return JAGG_ERR_WORKSPACE;
  }
  void* scratch = nullptr;
  JAGG_TRY(scratch_for_stream(stream, &scratch));
  return jagg::step_signals("grpo_step_signals_static", v_hat, v_dtype, z, t, nullptr, nullptr, sigma, logp_old,
                            rewards, G, W, D, clip_eps, adv_clip, adv_eps, scale, s_out, cot_out, logp_new, ratio,
                            clipped, adv_out, scratch, (size_t)JAGG_SIGNALS_STATIC_SCRATCH_BYTES, stream);
}
