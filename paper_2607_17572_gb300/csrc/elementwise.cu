// Bandwidth-bound kernels: layout transforms, embeddings, LayerNorm + adaLN modulation
// (forward and backward fused with the gated-residual backward), bias reductions,
// QK RMSNorm + 2D RoPE.
#include "elementwise.cuh"
#include "ptx.cuh"

namespace jagg {

int unit_status_elementwise(unsigned* v, int clear) { return read_unit_status(v, clear); }

namespace {

__device__ __forceinline__ float ldx(const void* p, int64_t i, int is_f32) {
  return is_f32 ? static_cast<const float*>(p)[i] : __bfloat162float(static_cast<const bf16*>(p)[i]);
}
__device__ __forceinline__ void stx(void* p, int64_t i, int is_f32, float v) {
  if (is_f32)
    static_cast<float*>(p)[i] = v;
  else
    static_cast<bf16*>(p)[i] = __float2bfloat16_rn(v);
}
__device__ __forceinline__ int64_t seg_row(int m, int seg, int seg_off, int64_t seg_stride) {
  return seg ? (int64_t)(m / seg) * seg_stride + seg_off + m % seg : (int64_t)m;
}

int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  return (int)(b < 1 ? 1 : (b > 1048576 ? 1048576 : b));
}

// ------------------------------------------------------------------ layouts
__global__ void patchify_kernel(const void* z, int in_f32, void* xp, int out_f32, int B, int C, int H, int W, int p) {
  pdl_wait();
  const int gw = W / p, gh = H / p;
  const int pd = C * p * p;
  const int64_t total = (int64_t)B * gh * gw * pd;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int f = (int)(i % pd);
    const int64_t tok = i / pd;
    const int n = (int)(tok % (gh * gw));
    const int b = (int)(tok / (gh * gw));
    const int r = n / gw, c = n % gw;
    const int ch = f / (p * p), py = (f / p) % p, px = f % p;
    const int64_t zi = (((int64_t)b * C + ch) * H + (r * p + py)) * W + (c * p + px);
    stx(xp, i, out_f32, ldx(z, zi, in_f32));
  }
}

__global__ void unpatchify_kernel(const void* xp, void* z, int is_f32, int B, int C, int H, int W, int p) {
  pdl_wait();
  const int gw = W / p, gh = H / p;
  const int pd = C * p * p;
  const int64_t total = (int64_t)B * C * H * W;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % W);
    const int y = (int)((i / W) % H);
    const int ch = (int)((i / ((int64_t)W * H)) % C);
    const int b = (int)(i / ((int64_t)W * H * C));
    const int r = y / p, py = y % p, c = x / p, px = x % p;
    const int64_t xi = ((int64_t)b * gh * gw + r * gw + c) * pd + ch * p * p + py * p + px;
    stx(z, i, is_f32, ldx(xp, xi, is_f32));
  }
}

__global__ void temb_kernel(const float* t, float* phi, int B, int dim) {
  pdl_wait();
  const int half = dim / 2;
  const int total = B * half;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int b = i / half, k = i % half;
    // w_k = 10000^(-k/half) evaluated in double so the argument 1000 t w_k is accurate
    const double w = exp(-log(10000.0) * (double)k / (double)half);
    const double a = 1000.0 * (double)t[b] * w;
    double sn, cs;
    sincos(a, &sn, &cs);  // one argument reduction for both
    phi[(int64_t)b * dim + k] = (float)cs;
    phi[(int64_t)b * dim + half + k] = (float)sn;
  }
}

__global__ void silu_kernel(const float* in, float* out, int64_t n) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = silu_f(in[i]);
}
// g *= SiLU'(x), and its copy in the storage type (an operand of the next products).
__global__ void mul_silu_grad_kernel(float* g, const float* x, void* copy, int copy_f32, int64_t n) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float v = g[i] * silu_grad_f(x[i]);
    g[i] = v;
    stx(copy, i, copy_f32, v);
  }
}

// One thread per 4 columns of one image token, added to that token of every sequence: each sine
// is evaluated once, not once per sequence (16 sequences of 256 tokens, d = 768:
// 27.2 -> 7.8 us).
__global__ void pos_embed_kernel(float* h, int B, int rows_per_seq, int row0, int gh, int gw, int d) {
  pdl_wait();
  const int q = d / 4, groups = d / 4;  // d is a multiple of 64: a group never crosses a quarter
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= gh * gw * groups) return;
  const int n = idx / groups, c = (idx % groups) * 4;
  const bool row = c < d / 2;  // the first half encodes the patch row, the second the column
  const int cc = c % (d / 2);
  const float pos = (float)(row ? n / gw : n % gw);
  float v[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    // f32 is enough here (|argument| < grid size, error ~1e-6); f64 is slow on this part
    const float a = pos * expf(-9.210340371976184f * (float)((cc + e) % q) / (float)q);  // ln(10000)
    v[e] = cc < q ? sinf(a) : cosf(a);
  }
  float* p = h + ((int64_t)row0 + n) * d + c;
#pragma unroll 4
  for (int b = 0; b < B; ++b) {
    float4* r = reinterpret_cast<float4*>(p + (int64_t)b * rows_per_seq * d);
    float4 x = *r;
    x.x += v[0]; x.y += v[1]; x.z += v[2]; x.w += v[3];
    *r = x;
  }
}

// ------------------------------------------------------------------ LayerNorm + modulation
// One warp per row; the row stays in registers (d <= 32 * 4 * LN_MAXV).
constexpr int LN_MAXV = 24;  // d <= 3072

__global__ void ln_mod_fwd_kernel(LnModFwd a) {
  pdl_wait();
  const int warps = blockDim.x / 32;
  const int m = blockIdx.x * warps + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (m >= a.M) return;
  const int nv = (a.d + 127) / 128;  // float4 slots per lane; slot (i*32 + lane) covers 4 columns
  const float* x = a.h + seg_row(m, a.seg, a.seg_off, a.seg_stride) * a.d;
  float4 v[LN_MAXV];
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < LN_MAXV; ++i) {
    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < nv && (i * 32 + lane) * 4 < a.d) {
      v[i] = reinterpret_cast<const float4*>(x)[i * 32 + lane];
      s += v[i].x + v[i].y + v[i].z + v[i].w;
    }
  }
  const float mean = warp_sum(s) / a.d;
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < LN_MAXV; ++i)
    if (i < nv && (i * 32 + lane) * 4 < a.d) {
      float dx = v[i].x - mean, dy = v[i].y - mean, dz = v[i].z - mean, dw = v[i].w - mean;
      ss += dx * dx + dy * dy + dz * dz + dw * dw;
    }
  const float rstd = rsqrtf(warp_sum(ss) / a.d + 1e-6f);
  const int b = m / a.rows_per_seq;
  const float* sh = a.shift + (int64_t)b * a.mod_stride;
  const float* sc = a.scale + (int64_t)b * a.mod_stride;
  const int is_f32 = a.dtype == JAGG_DTYPE_F32;
#pragma unroll
  for (int i = 0; i < LN_MAXV; ++i)
    if (i < nv && (i * 32 + lane) * 4 < a.d) {
      const int c = (i * 32 + lane) * 4;
      float4 s4 = *reinterpret_cast<const float4*>(sc + c);
      float4 h4 = *reinterpret_cast<const float4*>(sh + c);
      float o0 = (v[i].x - mean) * rstd * (1.f + s4.x) + h4.x;
      float o1 = (v[i].y - mean) * rstd * (1.f + s4.y) + h4.y;
      float o2 = (v[i].z - mean) * rstd * (1.f + s4.z) + h4.z;
      float o3 = (v[i].w - mean) * rstd * (1.f + s4.w) + h4.w;
      if (is_f32) {
        *reinterpret_cast<float4*>(static_cast<float*>(a.out) + (int64_t)m * a.d + c) = make_float4(o0, o1, o2, o3);
      } else {
        __nv_bfloat162 p0 = __floats2bfloat162_rn(o0, o1), p1 = __floats2bfloat162_rn(o2, o3);
        uint2 raw;
        raw.x = *reinterpret_cast<uint32_t*>(&p0);
        raw.y = *reinterpret_cast<uint32_t*>(&p1);
        *reinterpret_cast<uint2*>(static_cast<bf16*>(a.out) + (int64_t)m * a.d + c) = raw;
      }
    }
  if (lane == 0) {
    a.mean[m] = mean;
    a.rstd[m] = rstd;
  }
}

// The same with the row's 4 * 32 * NV * WPR columns split over WPR warps, NV float4 groups per
// lane, known at compile time (d = 128 NV WPR): every load of the row, its scale and its shift
// is issued before the first reduction.  Bound by DRAM once the rows fill the machine:
// 5328 rows of 768 columns 17.0 -> 7.4 us, 1225 rows 8.3 -> 3.8 us against the general kernel above
// (24 predicated groups per lane, the scale and shift loaded after the
// reductions).
template <int NV, int WPR>
__global__ void __launch_bounds__(128) ln_mod_fwd_fixed_kernel(LnModFwd a) {
  pdl_wait();
  constexpr int d = 128 * NV * WPR, ROWS = 4 / WPR;
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
  const int m = blockIdx.x * ROWS + warp / WPR;
  const int part = warp % WPR;
  if (WPR == 1 && m >= a.M) return;  // WPR > 1: one row per CTA, the grid has M CTAs
  const float* x = a.h + seg_row(m, a.seg, a.seg_off, a.seg_stride) * d;
  const int b = m / a.rows_per_seq;
  const float* sh = a.shift + (int64_t)b * a.mod_stride;
  const float* sc = a.scale + (int64_t)b * a.mod_stride;
  const int c0 = (part * NV * 32 + lane) * 4;
  float4 v[NV], s4[NV], h4[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = *reinterpret_cast<const float4*>(x + c0 + i * 128);
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    s4[i] = *reinterpret_cast<const float4*>(sc + c0 + i * 128);
    h4[i] = *reinterpret_cast<const float4*>(sh + c0 + i * 128);
  }
  __shared__ float red[2][4];
  auto row_sum = [&](float t, int slot) {  // over the row's warps
    t = warp_sum(t);
    if constexpr (WPR > 1) {
      if (lane == 0) red[slot][warp] = t;
      __syncthreads();
      t = 0.f;
#pragma unroll
      for (int w = 0; w < WPR; ++w) t += red[slot][w];
    }
    return t;
  };
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) s += (v[i].x + v[i].y) + (v[i].z + v[i].w);
  const float mean = row_sum(s, 0) / d;
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    v[i].x -= mean; v[i].y -= mean; v[i].z -= mean; v[i].w -= mean;
    ss += (v[i].x * v[i].x + v[i].y * v[i].y) + (v[i].z * v[i].z + v[i].w * v[i].w);
  }
  const float rstd = rsqrtf(row_sum(ss, 1) / d + 1e-6f);
  const int is_f32 = a.dtype == JAGG_DTYPE_F32;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int64_t o = (int64_t)m * d + c0 + i * 128;
    const float o0 = v[i].x * rstd * (1.f + s4[i].x) + h4[i].x, o1 = v[i].y * rstd * (1.f + s4[i].y) + h4[i].y;
    const float o2 = v[i].z * rstd * (1.f + s4[i].z) + h4[i].z, o3 = v[i].w * rstd * (1.f + s4[i].w) + h4[i].w;
    if (is_f32) {
      *reinterpret_cast<float4*>(static_cast<float*>(a.out) + o) = make_float4(o0, o1, o2, o3);
    } else {
      __nv_bfloat162 p0 = __floats2bfloat162_rn(o0, o1), p1 = __floats2bfloat162_rn(o2, o3);
      uint2 raw;
      raw.x = *reinterpret_cast<uint32_t*>(&p0);
      raw.y = *reinterpret_cast<uint32_t*>(&p1);
      *reinterpret_cast<uint2*>(static_cast<bf16*>(a.out) + o) = raw;
    }
  }
  if (lane == 0 && part == 0) {
    a.mean[m] = mean;
    a.rstd[m] = rstd;
  }
}

// Backward of LayerNorm + modulation and of a gated residual branch.
__device__ __forceinline__ void load4(const void* p, int64_t i, int is_f32, float (&v)[4]) {
  if (is_f32) {
    const float4 f = *reinterpret_cast<const float4*>(static_cast<const float*>(p) + i);
    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
  } else {
    const uint2 raw = *reinterpret_cast<const uint2*>(static_cast<const bf16*>(p) + i);
    const bf16* h = reinterpret_cast<const bf16*>(&raw);
    v[0] = __bfloat162float(h[0]); v[1] = __bfloat162float(h[1]);
    v[2] = __bfloat162float(h[2]); v[3] = __bfloat162float(h[3]);
  }
}
__device__ __forceinline__ void store4(void* p, int64_t i, int is_f32, const float (&v)[4]) {
  if (is_f32) {
    *reinterpret_cast<float4*>(static_cast<float*>(p) + i) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    uint2 raw;
    raw.x = *reinterpret_cast<uint32_t*>(&a);
    raw.y = *reinterpret_cast<uint32_t*>(&b);
    *reinterpret_cast<uint2*>(static_cast<bf16*>(p) + i) = raw;
  }
}

// One pass per row tile: a block of 8 warps takes LNF_ROWS rows of one sequence, each warp
// LNF_R of them.  Per row: the LayerNorm input-gradient (added to the residual gradient
// dh) and dy = gate * dh.  The per-sequence column sums (dshift, dscale, dgate, and sum dh
// for the bias gradient: sum_m dy = gate * sum_m dh) are summed over a warp's rows in
// registers, then over the block in shared memory (laid out [quantity][element][d/4] so a
// warp's atomics hit consecutive words), then flushed with one global atomic per column.
constexpr int LNF_R = 4;
constexpr int LNF_ROWS = 8 * LNF_R;

// Persistent: the grid walks the (sequence, row-chunk) units, so no wave tail.  NVT > 0
// fixes the number of float4 column groups per lane (d = 128 NVT) at compile time, so the
// column loops unroll and a warp's loads for its rows are issued together.
#ifndef LNF_MIN_BLOCKS
#define LNF_MIN_BLOCKS 3
#endif
template <int NVT>
__global__ void __launch_bounds__(256, LNF_MIN_BLOCKS) ln_gate_fused_kernel(LnGateBwd a) {
  pdl_wait();
  extern __shared__ float part[];  // [4 quantities][4][d/4]
  const int d = a.d, d4 = a.d / 4;
  const int chunks = (a.rows_per_seq + LNF_ROWS - 1) / LNF_ROWS;
  const int units = (a.M / a.rows_per_seq) * chunks;
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
  const int is_f32 = a.dtype == JAGG_DTYPE_F32;
  const int nv = NVT > 0 ? NVT : (d + 127) / 128;
  for (int unit = blockIdx.x; unit < units; unit += gridDim.x) {
    const int b = unit / chunks;
    const int r0 = (unit % chunks) * LNF_ROWS;
    for (int i = threadIdx.x; i < 4 * d; i += blockDim.x) part[i] = 0.f;
    __syncthreads();
    const float* gate = a.do_gate ? a.gate + (int64_t)b * a.mod_stride : nullptr;
    const float* sc = a.do_ln ? a.scale + (int64_t)b * a.mod_stride : nullptr;
    int mrow[LNF_R];
    int64_t hrow[LNF_R];
    bool live[LNF_R];
    float mu[LNF_R], rs[LNF_R], s1[LNF_R], s2[LNF_R];
#pragma unroll
    for (int k = 0; k < LNF_R; ++k) {
      const int r = r0 + warp * LNF_R + k;
      live[k] = r < a.rows_per_seq;
      mrow[k] = b * a.rows_per_seq + (live[k] ? r : 0);
      hrow[k] = seg_row(mrow[k], a.seg, a.seg_off, a.seg_stride);
      mu[k] = rs[k] = s1[k] = s2[k] = 0.f;
    }
    if (a.do_ln) {
#pragma unroll
      for (int k = 0; k < LNF_R; ++k) {
        if (live[k]) {
          mu[k] = a.mean[mrow[k]];
          rs[k] = a.rstd[mrow[k]];
        }
      }
#pragma unroll
      for (int i = 0; i < (NVT > 0 ? NVT : 1); ++i) {
        for (int ii = i; ii < (NVT > 0 ? i + 1 : nv); ++ii) {
          const int c = (ii * 32 + lane) * 4;
          if (c >= d) continue;
          const float4 s4 = *reinterpret_cast<const float4*>(sc + c);
          const float sv[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
          for (int k = 0; k < LNF_R; ++k) {
            if (!live[k]) continue;
            float dm[4];
            load4(a.dm, (int64_t)mrow[k] * d + c, a.dm_f32, dm);
            const float4 h4 = *reinterpret_cast<const float4*>(a.h + hrow[k] * d + c);
            const float hv[4] = {h4.x, h4.y, h4.z, h4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float dxh = dm[e] * (1.f + sv[e]);
              s1[k] += dxh;
              s2[k] += dxh * (hv[e] - mu[k]) * rs[k];
            }
          }
        }
      }
#pragma unroll
      for (int k = 0; k < LNF_R; ++k) {
        s1[k] = warp_sum(s1[k]) / d;
        s2[k] = warp_sum(s2[k]) / d;
      }
    }
#pragma unroll
    for (int i = 0; i < (NVT > 0 ? NVT : 1); ++i) {
      for (int ii = i; ii < (NVT > 0 ? i + 1 : nv); ++ii) {
        const int c = (ii * 32 + lane) * 4;
        if (c >= d) continue;
        float acc[4][4];  // [quantity][element]
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[q][e] = 0.f;
        float sv[4] = {0.f, 0.f, 0.f, 0.f}, gv[4] = {0.f, 0.f, 0.f, 0.f};
        if (a.do_ln) {
          const float4 s4 = *reinterpret_cast<const float4*>(sc + c);
          sv[0] = s4.x; sv[1] = s4.y; sv[2] = s4.z; sv[3] = s4.w;
        }
        if (gate) {
          const float4 g4 = *reinterpret_cast<const float4*>(gate + c);
          gv[0] = g4.x; gv[1] = g4.y; gv[2] = g4.z; gv[3] = g4.w;
        }
#pragma unroll
        for (int k = 0; k < LNF_R; ++k) {
          if (!live[k]) continue;
          const float4 d4v = *reinterpret_cast<const float4*>(a.dh_in + hrow[k] * d + c);
          float dh[4] = {d4v.x, d4v.y, d4v.z, d4v.w};
          if (a.do_ln) {
            float dm[4];
            load4(a.dm, (int64_t)mrow[k] * d + c, a.dm_f32, dm);
            const float4 h4 = *reinterpret_cast<const float4*>(a.h + hrow[k] * d + c);
            const float hv[4] = {h4.x, h4.y, h4.z, h4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float xh = (hv[e] - mu[k]) * rs[k];
              dh[e] += rs[k] * (dm[e] * (1.f + sv[e]) - s1[k] - xh * s2[k]);
              acc[0][e] += dm[e];
              acc[1][e] += dm[e] * xh;
            }
            *reinterpret_cast<float4*>(a.dh_out + hrow[k] * d + c) = make_float4(dh[0], dh[1], dh[2], dh[3]);
          }
          if (gate) {
            const float dy[4] = {gv[0] * dh[0], gv[1] * dh[1], gv[2] * dh[2], gv[3] * dh[3]};
            store4(a.dy, (int64_t)mrow[k] * d + c, is_f32, dy);
            float yv[4];
            load4(a.y, (int64_t)mrow[k] * d + c, is_f32, yv);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              acc[2][e] += dh[e] * yv[e];
              acc[3][e] += dh[e];
            }
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (q < 2 ? !a.do_ln : !gate) continue;
#pragma unroll
          for (int e = 0; e < 4; ++e) atomicAdd(&part[(q * 4 + e) * d4 + c / 4], acc[q][e]);
        }
      }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < d; c += blockDim.x) {
      auto P = [&](int q) { return part[(q * 4 + c % 4) * d4 + c / 4]; };
      if (a.do_ln) {
        atomicAdd(a.dshift + (int64_t)b * a.dmod_stride + c, P(0));
        atomicAdd(a.dscale + (int64_t)b * a.dmod_stride + c, P(1));
      }
      if (a.do_gate) {
        atomicAdd(a.dgate + (int64_t)b * a.dmod_stride + c, P(2));
        if (a.dbias) atomicAdd(a.dbias + c, gate[c] * P(3));
      }
    }
    __syncthreads();  // the partials are re-zeroed by the next unit
  }
}

// Row-in-registers variant for d = 128 NV <= 768, with the LayerNorm part always present and
// dm in f32 (GATE: the gate part too; YBF: y and dy in bf16).  A warp issues every load of
// one row at once (dh, dm, h, y: float4-wide groups per 128 columns), forms the row
// statistics with two warp reductions and updates the row without a second pass.  The
// sequence's scale and gate vectors sit in shared memory for the whole segment.  The
// per-sequence column sums go to a warp-private shared-memory slab ([4 quantities][d],
// plain read-modify-write, no atomics), summed over the block's 8 warps and flushed with
// atomics once per sequence segment.  Each CTA owns a contiguous, equal share of the rows
// (at most a few sequence segments), so every CTA finishes at the same time.
template <int NV, bool GATE, bool YBF>
__global__ void __launch_bounds__(256, 2) ln_gate_rowreg_kernel(LnGateBwd a) {
  pdl_wait();
  extern __shared__ float part[];  // [8 warps][4 quantities][d], then scale[d], gate[d]
  constexpr int d = 128 * NV;
  const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
  float* mine = part + warp * 4 * d;
  float* sc_s = part + 8 * 4 * d;
  float* gt_s = sc_s + d;
  const int row_begin = (int)((int64_t)a.M * blockIdx.x / gridDim.x);
  const int row_end = (int)((int64_t)a.M * (blockIdx.x + 1) / gridDim.x);
  for (int seg0 = row_begin; seg0 < row_end;) {
    const int b = seg0 / a.rows_per_seq;
    const int seg1 = min(row_end, (b + 1) * a.rows_per_seq);
    for (int i = lane; i < 4 * d; i += 32) mine[i] = 0.f;
    for (int c = threadIdx.x; c < d; c += blockDim.x) {
      sc_s[c] = 1.f + a.scale[(int64_t)b * a.mod_stride + c];
      if (GATE) gt_s[c] = a.gate[(int64_t)b * a.mod_stride + c];
    }
    __syncthreads();
#pragma unroll 1
    for (int m = seg0 + warp; m < seg1; m += 8) {
      const int64_t hr = seg_row(m, a.seg, a.seg_off, a.seg_stride);
      const float mu = a.mean[m], rs = a.rstd[m];
      float4 dh[NV], dm[NV], hv[NV];
      uint2 yb[NV];
      float4 yf[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int c = (i * 32 + lane) * 4;
        dh[i] = *reinterpret_cast<const float4*>(a.dh_in + hr * d + c);
        dm[i] = *reinterpret_cast<const float4*>(static_cast<const float*>(a.dm) + (int64_t)m * d + c);
        hv[i] = *reinterpret_cast<const float4*>(a.h + hr * d + c);
        if (GATE) {
          if (YBF)
            yb[i] = *reinterpret_cast<const uint2*>(static_cast<const bf16*>(a.y) + (int64_t)m * d + c);
          else
            yf[i] = *reinterpret_cast<const float4*>(static_cast<const float*>(a.y) + (int64_t)m * d + c);
        }
      }
      float s1 = 0.f, s2 = 0.f;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float4 sv = *reinterpret_cast<const float4*>(sc_s + (i * 32 + lane) * 4);
        hv[i].x = (hv[i].x - mu) * rs; hv[i].y = (hv[i].y - mu) * rs;  // now x-hat
        hv[i].z = (hv[i].z - mu) * rs; hv[i].w = (hv[i].w - mu) * rs;
        const float e0 = dm[i].x * sv.x, e1 = dm[i].y * sv.y, e2 = dm[i].z * sv.z, e3 = dm[i].w * sv.w;
        s1 += (e0 + e1) + (e2 + e3);
        s2 += (e0 * hv[i].x + e1 * hv[i].y) + (e2 * hv[i].z + e3 * hv[i].w);
      }
      s1 = warp_sum(s1) / d;
      s2 = warp_sum(s2) / d;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int c = (i * 32 + lane) * 4;
        const float4 sv = *reinterpret_cast<const float4*>(sc_s + c);
        dh[i].x += rs * (dm[i].x * sv.x - s1 - hv[i].x * s2);
        dh[i].y += rs * (dm[i].y * sv.y - s1 - hv[i].y * s2);
        dh[i].z += rs * (dm[i].z * sv.z - s1 - hv[i].z * s2);
        dh[i].w += rs * (dm[i].w * sv.w - s1 - hv[i].w * s2);
        *reinterpret_cast<float4*>(a.dh_out + hr * d + c) = dh[i];
        float4* q0 = reinterpret_cast<float4*>(mine + c);
        float4* q1 = reinterpret_cast<float4*>(mine + d + c);
        float4 u = *q0, w = *q1;
        u.x += dm[i].x; u.y += dm[i].y; u.z += dm[i].z; u.w += dm[i].w;
        w.x += dm[i].x * hv[i].x; w.y += dm[i].y * hv[i].y; w.z += dm[i].z * hv[i].z; w.w += dm[i].w * hv[i].w;
        *q0 = u;
        *q1 = w;
        if (GATE) {
          float y0, y1, y2, y3;
          if (YBF) {
            const bf16* h = reinterpret_cast<const bf16*>(&yb[i]);
            y0 = __bfloat162float(h[0]); y1 = __bfloat162float(h[1]);
            y2 = __bfloat162float(h[2]); y3 = __bfloat162float(h[3]);
          } else {
            y0 = yf[i].x; y1 = yf[i].y; y2 = yf[i].z; y3 = yf[i].w;
          }
          const float4 g4 = *reinterpret_cast<const float4*>(gt_s + c);
          const float dy[4] = {g4.x * dh[i].x, g4.y * dh[i].y, g4.z * dh[i].z, g4.w * dh[i].w};
          store4(a.dy, (int64_t)m * d + c, !YBF, dy);
          float4* q2 = reinterpret_cast<float4*>(mine + 2 * d + c);
          float4* q3 = reinterpret_cast<float4*>(mine + 3 * d + c);
          float4 u2 = *q2, w2 = *q3;
          u2.x += dh[i].x * y0; u2.y += dh[i].y * y1; u2.z += dh[i].z * y2; u2.w += dh[i].w * y3;
          w2.x += dh[i].x; w2.y += dh[i].y; w2.z += dh[i].z; w2.w += dh[i].w;
          *q2 = u2;
          *q3 = w2;
        }
      }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < d; c += blockDim.x) {
      float P[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int w = 0; w < 8; ++w)
#pragma unroll
        for (int q = 0; q < (GATE ? 4 : 2); ++q) P[q] += part[(w * 4 + q) * d + c];
      atomicAdd(a.dshift + (int64_t)b * a.dmod_stride + c, P[0]);
      atomicAdd(a.dscale + (int64_t)b * a.dmod_stride + c, P[1]);
      if (GATE) {
        atomicAdd(a.dgate + (int64_t)b * a.dmod_stride + c, P[2]);
        if (a.dbias) atomicAdd(a.dbias + c, gt_s[c] * P[3]);
      }
    }
    __syncthreads();  // the slabs and vectors are rewritten for the next segment
    seg0 = seg1;
  }
}

// The bf16 widths (d = 128 NV WPR): WPR warps share a row, 8 / WPR rows in work per CTA.  Bound by
// DRAM, so the loads never wait for the arithmetic: each row group has a ring of LNR_STAGES
// rows (dh, dm, h, y) that bulk copies fill ahead of the row being worked on.  The row
// statistics are warp shuffles plus, for WPR > 1, one named barrier over the group, after
// which the stage is free for the next copy.  Each CTA owns a contiguous, equal share of the rows and each
// lane the same columns for all of them, so the per-sequence column sums (dshift, dscale,
// dgate, sum dh for the bias gradient) stay in registers; at each sequence boundary the
// CTA's groups add theirs in shared memory and one 16-byte reduction per 4 columns and quantity
// leaves.
// The sums leave as 16-byte reductions: as scalar atomics 16 bytes apart, four per thread
// and column group, they took half of the kernel (5328 x 768 rows in 24.8 us, now 18.3; 1225 rows
// 17.1 -> 11.7; Flux-512's streams 42.7 -> 30.1 us on average), and loading ahead changed nothing.
constexpr int LNR_STAGES = 2;

template <int NV, int WPR, bool LN, bool GATE>
struct LnRing {
  static constexpr int D = 128 * NV * WPR, GROUPS = 8 / WPR;
  static constexpr int ROW = D * (4 + (LN ? 8 : 0) + (GATE ? 2 : 0));  // bytes of a row's operands
  static constexpr int OFF_DM = 4 * D, OFF_H = 8 * D, OFF_Y = D * (LN ? 12 : 4);
  static constexpr int OFF_VEC = GROUPS * LNR_STAGES * ROW;            // 1 + scale [D], gate [D]
  static constexpr int OFF_SUM = OFF_VEC + 8 * D;                      // [4][D] when groups share
  static constexpr int OFF_RED = OFF_SUM + (GROUPS > 1 ? 16 * D : 0);  // [GROUPS][parity][2][WPR]
  static constexpr int OFF_BAR = OFF_RED + 8 * 2 * 2 * 4;
  static constexpr int SMEM = OFF_BAR + GROUPS * LNR_STAGES * 8;
  static_assert(ROW % 16 == 0 && OFF_BAR % 8 == 0, "bulk copies and barriers are aligned");
};

template <int NV, int WPR, bool LN, bool GATE>
__global__ void __launch_bounds__(256, 2) ln_gate_ring_kernel(LnGateBwd a) {
  using C = LnRing<NV, WPR, LN, GATE>;
  constexpr int d = C::D, GROUPS = C::GROUPS, S = LNR_STAGES;
  extern __shared__ __align__(128) uint8_t lnr_sm[];
  float* sc_s = reinterpret_cast<float*>(lnr_sm + C::OFF_VEC);
  float* gt_s = sc_s + d;
  float* sum_s = reinterpret_cast<float*>(lnr_sm + C::OFF_SUM);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = warp / WPR, gw = warp % WPR;
  uint8_t* ring = lnr_sm + grp * S * C::ROW;
  float* red = reinterpret_cast<float*>(lnr_sm + C::OFF_RED) + grp * 2 * 2 * WPR;
  uint64_t* bar = reinterpret_cast<uint64_t*>(lnr_sm + C::OFF_BAR) + grp * S;
  if (tid == 0) {
    uint64_t* all = reinterpret_cast<uint64_t*>(lnr_sm + C::OFF_BAR);
    for (int i = 0; i < GROUPS * S; ++i) ptx::mbar_init(&all[i], 1);
    ptx::fence_mbar_init();
  }
  __syncthreads();
  pdl_wait();
  auto group_sync = [&]() {
    if constexpr (WPR == 1)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(32 * WPR) : "memory");
  };
  const bool leader = gw == 0 && lane == 0;
  const int col0 = (gw * NV * 32 + lane) * 4;  // columns col0 + 128 i .. + 3, i < NV
  const int row_begin = (int)((int64_t)a.M * blockIdx.x / gridDim.x);
  const int row_end = (int)((int64_t)a.M * (blockIdx.x + 1) / gridDim.x);
  auto issue = [&](int m, int st) {  // the leader: row m into stage st
    uint8_t* dst = ring + st * C::ROW;
    const int64_t hr = seg_row(m, a.seg, a.seg_off, a.seg_stride);
    ptx::mbar_arrive_expect_tx(&bar[st], C::ROW);
    ptx::bulk_load(dst, a.dh_in + hr * d, 4 * d, &bar[st]);
    if (LN) {
      ptx::bulk_load(dst + C::OFF_DM, static_cast<const float*>(a.dm) + (int64_t)m * d, 4 * d, &bar[st]);
      ptx::bulk_load(dst + C::OFF_H, a.h + hr * d, 4 * d, &bar[st]);
    }
    if (GATE) ptx::bulk_load(dst + C::OFF_Y, static_cast<const bf16*>(a.y) + (int64_t)m * d, 2 * d, &bar[st]);
  };
  int j = 0, parity = 0;  // rows this group has taken from its ring
  bool alive = true;      // false after a wait gave up: no more waiting, the status word is set
  for (int seg0 = row_begin; seg0 < row_end;) {
    const int b = seg0 / a.rows_per_seq;
    const int seg1 = min(row_end, (b + 1) * a.rows_per_seq);
    if (leader)
      for (int i = 0; i < S && seg0 + grp + i * GROUPS < seg1; ++i) issue(seg0 + grp + i * GROUPS, (j + i) % S);
    for (int c = tid * 4; c < d; c += 1024) {
      if (LN) {
        float4 v = *reinterpret_cast<const float4*>(a.scale + (int64_t)b * a.mod_stride + c);
        v.x += 1.f; v.y += 1.f; v.z += 1.f; v.w += 1.f;
        *reinterpret_cast<float4*>(sc_s + c) = v;
      }
      if (GATE) *reinterpret_cast<float4*>(gt_s + c) = *reinterpret_cast<const float4*>(a.gate + (int64_t)b * a.mod_stride + c);
    }
    float4 acc[4][NV];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int i = 0; i < NV; ++i) acc[q][i] = make_float4(0.f, 0.f, 0.f, 0.f);
    float mu_next = 0.f, rs_next = 0.f;
    if (LN && seg0 + grp < seg1) {
      mu_next = a.mean[seg0 + grp];
      rs_next = a.rstd[seg0 + grp];
    }
    __syncthreads();
#pragma unroll 1
    for (int m = seg0 + grp; m < seg1; m += GROUPS, ++j) {
      const int st = j % S;
      const uint8_t* src = ring + st * C::ROW;
      const float mu = mu_next, rs = rs_next;
      if (LN && m + GROUPS < seg1) {
        mu_next = a.mean[m + GROUPS];
        rs_next = a.rstd[m + GROUPS];
      }
      if (alive) alive = ptx::mbar_wait(&bar[st], (j / S) & 1);
      float4 dh[NV], dm[NV], hv[NV];
      uint2 yb[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int c = col0 + i * 128;
        dh[i] = *reinterpret_cast<const float4*>(src + 4 * c);
        if (LN) {
          dm[i] = *reinterpret_cast<const float4*>(src + C::OFF_DM + 4 * c);
          hv[i] = *reinterpret_cast<const float4*>(src + C::OFF_H + 4 * c);
        }
        if (GATE) yb[i] = *reinterpret_cast<const uint2*>(src + C::OFF_Y + 2 * c);
      }
      float s1 = 0.f, s2 = 0.f;
      if (LN) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          hv[i].x = (hv[i].x - mu) * rs; hv[i].y = (hv[i].y - mu) * rs;  // now x-hat
          hv[i].z = (hv[i].z - mu) * rs; hv[i].w = (hv[i].w - mu) * rs;
          const float4 sv = *reinterpret_cast<const float4*>(sc_s + col0 + i * 128);
          const float e0 = dm[i].x * sv.x, e1 = dm[i].y * sv.y, e2 = dm[i].z * sv.z, e3 = dm[i].w * sv.w;
          s1 += (e0 + e1) + (e2 + e3);
          s2 += (e0 * hv[i].x + e1 * hv[i].y) + (e2 * hv[i].z + e3 * hv[i].w);
        }
        s1 = warp_sum(s1);
        s2 = warp_sum(s2);
        if (WPR > 1 && lane == 0) {
          red[(parity * 2) * WPR + gw] = s1;
          red[(parity * 2 + 1) * WPR + gw] = s2;
        }
      }
      ptx::fence_proxy_async_smem();
      group_sync();  // every lane has read the stage: refill it
      if (leader && m + S * GROUPS < seg1) issue(m + S * GROUPS, st);
      if (LN) {
        if (WPR > 1) {
          s1 = s2 = 0.f;
#pragma unroll
          for (int w = 0; w < WPR; ++w) {
            s1 += red[(parity * 2) * WPR + w];
            s2 += red[(parity * 2 + 1) * WPR + w];
          }
          parity ^= 1;
        }
        s1 /= d;
        s2 /= d;
        float* out = a.dh_out + seg_row(m, a.seg, a.seg_off, a.seg_stride) * d + col0;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const float4 sv = *reinterpret_cast<const float4*>(sc_s + col0 + i * 128);
          dh[i].x += rs * (dm[i].x * sv.x - s1 - hv[i].x * s2);
          dh[i].y += rs * (dm[i].y * sv.y - s1 - hv[i].y * s2);
          dh[i].z += rs * (dm[i].z * sv.z - s1 - hv[i].z * s2);
          dh[i].w += rs * (dm[i].w * sv.w - s1 - hv[i].w * s2);
          *reinterpret_cast<float4*>(out + i * 128) = dh[i];
          acc[0][i].x += dm[i].x; acc[0][i].y += dm[i].y; acc[0][i].z += dm[i].z; acc[0][i].w += dm[i].w;
          acc[1][i].x += dm[i].x * hv[i].x; acc[1][i].y += dm[i].y * hv[i].y;
          acc[1][i].z += dm[i].z * hv[i].z; acc[1][i].w += dm[i].w * hv[i].w;
        }
      }
      if (GATE) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const int c = col0 + i * 128;
          const float4 g4 = *reinterpret_cast<const float4*>(gt_s + c);
          const float dy[4] = {g4.x * dh[i].x, g4.y * dh[i].y, g4.z * dh[i].z, g4.w * dh[i].w};
          store4(a.dy, (int64_t)m * d + c, 0, dy);
          const bf16* yh = reinterpret_cast<const bf16*>(&yb[i]);
          acc[2][i].x += dh[i].x * __bfloat162float(yh[0]); acc[2][i].y += dh[i].y * __bfloat162float(yh[1]);
          acc[2][i].z += dh[i].z * __bfloat162float(yh[2]); acc[2][i].w += dh[i].w * __bfloat162float(yh[3]);
          acc[3][i].x += dh[i].x; acc[3][i].y += dh[i].y; acc[3][i].z += dh[i].z; acc[3][i].w += dh[i].w;
        }
      }
    }
    // the segment's column sums: the groups in turn into shared memory, the last one (or the
    // only one) out to global memory
#pragma unroll
    for (int gi = 0; gi < GROUPS; ++gi) {
      if (grp == gi) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const int c = col0 + i * 128;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (q < 2 ? !LN : !GATE) continue;
            float4 v = acc[q][i];
            if (GROUPS > 1) {
              float4* at = reinterpret_cast<float4*>(sum_s + q * d + c);
              if (gi > 0) {
                const float4 w = *at;
                v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
              }
              if (gi < GROUPS - 1) {
                *at = v;
                continue;
              }
            }
            if (q == 3 && !a.dbias) continue;
            float* dst = q == 0   ? a.dshift + (int64_t)b * a.dmod_stride + c
                         : q == 1 ? a.dscale + (int64_t)b * a.dmod_stride + c
                         : q == 2 ? a.dgate + (int64_t)b * a.dmod_stride + c
                                  : a.dbias + c;
            if (q == 3) {
              const float4 g4 = *reinterpret_cast<const float4*>(gt_s + c);
              v.x *= g4.x; v.y *= g4.y; v.z *= g4.z; v.w *= g4.w;
            }
            ptx::red_add_v4(dst, v.x, v.y, v.z, v.w);
          }
        }
      }
      if (GROUPS > 1) __syncthreads();
    }
    if (GROUPS == 1) __syncthreads();  // the vectors are rewritten for the next segment
    seg0 = seg1;
  }
  // after a give-up, copies may still be landing: wait (bounded) for the last of every stage
  if (!alive && leader)
    for (int i = 1; i <= S && j - i >= 0; ++i) ptx::mbar_wait(&bar[(j - i) % S], ((j - i) / S) & 1);
}

template <int NV, int WPR, bool LN, bool GATE>
int launch_ln_gate_ring_t(const LnGateBwd& a, cudaStream_t s) {
  using C = LnRing<NV, WPR, LN, GATE>;
  auto kernel = ln_gate_ring_kernel<NV, WPR, LN, GATE>;
  static OncePerDevice once;
  static std::atomic<int> ctas{0};
  int per_sm = 0;
  JAGG_CUDA_TRY(allow_smem(once, kernel, C::SMEM));
  JAGG_CUDA_TRY(resident_ctas(ctas, kernel, 256, C::SMEM, &per_sm));
  // equal row shares of at least two rows per group, at most one wave of resident CTAs
  const int cap = per_sm * sm_count();
  const int want = ceil_div(a.M, 2 * C::GROUPS);
  JAGG_CUDA_TRY(launch(kernel, want < cap ? want : cap, 256, C::SMEM, s, a));
  JAGG_LAUNCHED();
  return JAGG_OK;
}

template <int NV, int WPR>
int launch_ln_gate_ring(const LnGateBwd& a, cudaStream_t s) {
  if (a.do_ln) return a.do_gate ? launch_ln_gate_ring_t<NV, WPR, true, true>(a, s)
                                : launch_ln_gate_ring_t<NV, WPR, true, false>(a, s);
  return launch_ln_gate_ring_t<NV, WPR, false, true>(a, s);
}

// What the ring kernel takes: bf16 y and dy, dm in f32, and its 16-byte accesses (8-byte stores of
// dy): every row, vector and sum aligned.
bool ln_gate_ring_serves(const LnGateBwd& a) {
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (!al(a.dh_in) || a.mod_stride % 4 || a.dmod_stride % 4) return false;
  if (a.do_ln && !(a.dm_f32 && al(a.dm) && al(a.h) && al(a.dh_out) && al(a.scale) && al(a.dshift) && al(a.dscale)))
    return false;
  return !a.do_gate || (a.dtype == JAGG_DTYPE_BF16 && al(a.y) && al(a.dy) && al(a.gate) && al(a.dgate) &&
                        (!a.dbias || al(a.dbias)));
}

// Narrow rows, d = 4 L NV <= 256 (the f32 configuration): L lanes per row, so a warp works on 32 / L
// rows at once, every operand loaded once into registers.  Bound by latency: a few hundred
// rows are one or two rounds of loads.  The column sums of a lane's rows stay in registers, meet
// in shared memory and leave as 16-byte reductions, one per 4 columns, quantity and CTA.
// 192 rows of 64 columns: 10.8 us in the general kernel (two passes over the operands, shared-memory and
// scalar global atomics); a tiny f32 training pass, with seven of them, 350 -> 323 us together with the
// launches saved around it.
template <int L, int NV>
__global__ void __launch_bounds__(256) ln_gate_narrow_kernel(LnGateBwd a, int rows_per_cta, int chunks) {
  pdl_wait();
  constexpr int d = 4 * L * NV, TEAMS = 256 / L;
  __shared__ __align__(16) float part[TEAMS][4 * L * NV];
  const int team = threadIdx.x / L, lane = threadIdx.x % L;
  const int is_f32 = a.dtype == JAGG_DTYPE_F32;
  const int b = blockIdx.x / chunks, r0 = (blockIdx.x % chunks) * rows_per_cta;
  const int r1 = min(r0 + rows_per_cta, a.rows_per_seq);
  auto vec = [&](const float* p, int i) {
    return p ? *reinterpret_cast<const float4*>(p + (int64_t)b * a.mod_stride + (i * L + lane) * 4)
             : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  float4 sc[NV], gt[NV], acc[4][NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    sc[i] = vec(a.do_ln ? a.scale : nullptr, i);
    gt[i] = vec(a.do_gate ? a.gate : nullptr, i);
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q][i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  auto team_sum = [&](float v) {
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  // every team makes the same number of rounds (the sums are warp-wide)
  for (int base = r0; base < r1; base += TEAMS) {
    const bool live = base + team < r1;
    const int m = b * a.rows_per_seq + (live ? base + team : r0);
    const int64_t hr = seg_row(m, a.seg, a.seg_off, a.seg_stride) * d, mr = (int64_t)m * d;
    float dh[NV][4], dm[NV][4], xh[NV][4], y[NV][4];
    const float mu = a.do_ln ? a.mean[m] : 0.f, rs = a.do_ln ? a.rstd[m] : 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = (i * L + lane) * 4;
      load4(a.dh_in, hr + c, 1, dh[i]);
      if (a.do_ln) {
        load4(a.dm, mr + c, a.dm_f32, dm[i]);
        load4(a.h, hr + c, 1, xh[i]);
      }
      if (a.do_gate) load4(a.y, mr + c, is_f32, y[i]);
    }
    if (a.do_ln) {
      float s1 = 0.f, s2 = 0.f;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float sv[4] = {1.f + sc[i].x, 1.f + sc[i].y, 1.f + sc[i].z, 1.f + sc[i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          xh[i][e] = (xh[i][e] - mu) * rs;
          s1 += dm[i][e] * sv[e];
          s2 += dm[i][e] * sv[e] * xh[i][e];
        }
      }
      s1 = team_sum(s1) / d;
      s2 = team_sum(s2) / d;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float sv[4] = {1.f + sc[i].x, 1.f + sc[i].y, 1.f + sc[i].z, 1.f + sc[i].w};
        float* q0 = &acc[0][i].x;
        float* q1 = &acc[1][i].x;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          dh[i][e] += rs * (dm[i][e] * sv[e] - s1 - xh[i][e] * s2);
          if (live) {
            q0[e] += dm[i][e];
            q1[e] += dm[i][e] * xh[i][e];
          }
        }
        if (live) store4(a.dh_out, hr + (i * L + lane) * 4, 1, dh[i]);
      }
    }
    if (a.do_gate && live) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const float gv[4] = {gt[i].x, gt[i].y, gt[i].z, gt[i].w};
        float dy[4];
        float* q2 = &acc[2][i].x;
        float* q3 = &acc[3][i].x;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          dy[e] = gv[e] * dh[i][e];
          q2[e] += dh[i][e] * y[i][e];
          q3[e] += dh[i][e];
        }
        store4(a.dy, mr + (i * L + lane) * 4, is_f32, dy);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (q < 2 ? !a.do_ln : !a.do_gate) continue;
    if (q == 3 && !a.dbias) continue;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) *reinterpret_cast<float4*>(&part[team][(i * L + lane) * 4]) = acc[q][i];
    __syncthreads();
    if (threadIdx.x < d / 4) {
      const int c = threadIdx.x * 4;
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < TEAMS; ++w) {
        const float4 v = *reinterpret_cast<const float4*>(&part[w][c]);
        t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
      }
      float* dst = q == 0   ? a.dshift + (int64_t)b * a.dmod_stride + c
                   : q == 1 ? a.dscale + (int64_t)b * a.dmod_stride + c
                   : q == 2 ? a.dgate + (int64_t)b * a.dmod_stride + c
                            : a.dbias + c;
      if (q == 3) {
        const float4 g4 = *reinterpret_cast<const float4*>(a.gate + (int64_t)b * a.mod_stride + c);
        t.x *= g4.x; t.y *= g4.y; t.z *= g4.z; t.w *= g4.w;
      }
      ptx::red_add_v4(dst, t.x, t.y, t.z, t.w);
    }
  }
}

template <int L, int NV>
int launch_ln_gate_narrow(const LnGateBwd& a, cudaStream_t s) {
  // two rounds of rows per CTA
  const int rows = 2 * 256 / L, chunks = ceil_div(a.rows_per_seq, rows);
  JAGG_CUDA_TRY(launch(ln_gate_narrow_kernel<L, NV>, (a.M / a.rows_per_seq) * chunks, 256, 0, s, a, rows, chunks));
  JAGG_LAUNCHED();
  return JAGG_OK;
}

// The narrow kernel's 16-byte accesses: every row, vector and sum aligned.
bool ln_gate_narrow_serves(const LnGateBwd& a) {
  auto al = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (!al(a.dh_in) || a.mod_stride % 4 || a.dmod_stride % 4) return false;
  if (a.do_ln && !(al(a.dm) && al(a.h) && al(a.dh_out) && al(a.scale) && al(a.dshift) && al(a.dscale))) return false;
  return !a.do_gate || (al(a.y) && al(a.dy) && al(a.gate) && al(a.dgate) && (!a.dbias || al(a.dbias)));
}

template <int NV, bool GATE, bool YBF>
int launch_ln_gate_rowreg_t(const LnGateBwd& a, cudaStream_t s) {
  const int smem = (8 * 4 + 2) * 128 * NV * (int)sizeof(float);
  auto kernel = ln_gate_rowreg_kernel<NV, GATE, YBF>;
  static OncePerDevice once;
  static std::atomic<int> ctas{0};
  int per_sm = 0;
  JAGG_CUDA_TRY(allow_smem(once, kernel, smem));
  JAGG_CUDA_TRY(resident_ctas(ctas, kernel, 256, smem, &per_sm));
  // equal row shares of at least 16 rows per CTA, at most one wave of resident CTAs
  const int cap = per_sm * sm_count();
  const int want = ceil_div(a.M, 16);
  JAGG_CUDA_TRY(launch(kernel, want < cap ? want : cap, 256, smem, s, a));
  JAGG_LAUNCHED();
  return JAGG_OK;
}

template <int NVT>
int launch_ln_gate_nv(const LnGateBwd& a, int smem, cudaStream_t s) {
  constexpr int most = 4 * 3072 * (int)sizeof(float);
  static OncePerDevice once;
  static std::atomic<int> ctas{0};
  int per_sm = 0;
  JAGG_CUDA_TRY(allow_smem(once, ln_gate_fused_kernel<NVT>, most));
  JAGG_CUDA_TRY(resident_ctas(ctas, ln_gate_fused_kernel<NVT>, 256, most, &per_sm));
  const int units = (a.M / a.rows_per_seq) * ceil_div(a.rows_per_seq, LNF_ROWS);
  const int cap = per_sm * sm_count();
  JAGG_CUDA_TRY(launch(ln_gate_fused_kernel<NVT>, units < cap ? units : cap, 256, smem, s, a));
  JAGG_LAUNCHED();
  return JAGG_OK;
}

// ------------------------------------------------------------------ reductions / copies
constexpr int CS_ROWS = 64;
__global__ void colsum_kernel(const void* X, int x_f32, int rows, int cols, int64_t ld, float* db) {
  pdl_wait();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int r0 = blockIdx.y * CS_ROWS;
  if (c >= cols) return;
  const int r1 = min(r0 + CS_ROWS, rows);
  float s = 0.f;
  for (int r = r0; r < r1; ++r) s += ldx(X, (int64_t)r * ld + c, x_f32);
  atomicAdd(db + c, s);
}

// Column sums of a bf16 matrix, 8 columns (one 16-byte load) per thread: block = 32 column
// groups (256 columns) x 8 row slices over rows_per_block rows; the 8 slices meet in shared memory
// and each column gets one atomic add per block.  Rows per block: as many as keep about
// CSV_BLOCKS_PER_SM blocks on every SM, at most 256: with 256 always, a few hundred rows
// left most of the machine idle and each thread a chain of 32 loads (5328 x 3072: 12.8 ->
// 9.1 us).
constexpr int CSV_MAX_ROWS = 256, CSV_BLOCKS_PER_SM = 6;
__global__ void __launch_bounds__(256) colsum_bf16x8_kernel(const bf16* X, int rows, int cols, int64_t ld,
                                                            int rows_per_block, float* db) {
  pdl_wait();
  __shared__ float part[8][257];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int c0 = (blockIdx.x * 32 + tx) * 8;
  const int r0 = blockIdx.y * rows_per_block;
  const int r1 = min(r0 + rows_per_block, rows);
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (c0 < cols) {
#pragma unroll 8
    for (int r = r0 + ty; r < r1; r += 8) {
      const uint4 raw = *reinterpret_cast<const uint4*>(X + (int64_t)r * ld + c0);
      const bf16* h = reinterpret_cast<const bf16*>(&raw);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] += __bfloat162float(h[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) part[ty][tx * 8 + i] = acc[i];
  __syncthreads();
  const int c = blockIdx.x * 256 + threadIdx.x;
  if (c < cols) {
    float t = 0.f;
#pragma unroll
    for (int y = 0; y < 8; ++y) t += part[y][threadIdx.x];
    atomicAdd(db + c, t);
  }
}

// Four columns per thread: cols a multiple of 4, 16-byte aligned rows of `in`, 8-byte aligned out.
__global__ void gather_rows_v4_kernel(const float* in, int64_t ld_in, int seg, int seg_off, int64_t seg_stride,
                                      void* out, int out_f32, int rows, int cols) {
  pdl_wait();
  const int groups = cols / 4;
  const int64_t total = (int64_t)rows * groups;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(i / groups), c = (int)(i % groups) * 4;
    const float4 f = *reinterpret_cast<const float4*>(in + seg_row(r, seg, seg_off, seg_stride) * ld_in + c);
    const float v[4] = {f.x, f.y, f.z, f.w};
    store4(out, 4 * i, out_f32, v);
  }
}

__global__ void gather_rows_kernel(const float* in, int64_t ld_in, int seg, int seg_off, int64_t seg_stride, void* out,
                                   int out_f32, int rows, int cols) {
  pdl_wait();
  const int64_t total = (int64_t)rows * cols;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(i / cols), c = (int)(i % cols);
    stx(out, i, out_f32, in[seg_row(r, seg, seg_off, seg_stride) * ld_in + c]);
  }
}

template <typename E>
__global__ void copy_rows_kernel(const E* in, int64_t ld_in, int is, int io, int64_t iss, E* out, int64_t ld_out,
                                 int os, int oo, int64_t oss, int rows, int cols) {
  pdl_wait();
  const int64_t total = (int64_t)rows * cols;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(i / cols), c = (int)(i % cols);
    out[seg_row(r, os, oo, oss) * ld_out + c] = in[seg_row(r, is, io, iss) * ld_in + c];
  }
}

// Whole rows in 16-byte vectors, a row per block iteration (row pitches, row bytes and both
// bases 16-byte aligned).
__global__ void copy_rows_v16_kernel(const uint8_t* in, int64_t ld_in_b, int is, int io, int64_t iss, uint8_t* out,
                                     int64_t ld_out_b, int os, int oo, int64_t oss, int rows, int nvec) {
  pdl_wait();
  for (int r = blockIdx.x; r < rows; r += gridDim.x) {
    const uint4* src = reinterpret_cast<const uint4*>(in + seg_row(r, is, io, iss) * ld_in_b);
    uint4* dst = reinterpret_cast<uint4*>(out + seg_row(r, os, oo, oss) * ld_out_b);
    for (int c = threadIdx.x; c < nvec; c += blockDim.x) dst[c] = __ldg(src + c);
  }
}

// ------------------------------------------------------------------ QK RMSNorm + RoPE
// One warp per (row, head) handles q and k; dh <= 128 -> up to 4 elements per lane as
// two rotated pairs.
__device__ __forceinline__ void rope_angle(int n, int n_txt, int gw, int dh, int pair, float& cs, float& sn) {
  // pair index within the head: first dh/4 pairs rotate by the patch row, the rest by the column
  const int hd = dh / 2, npair = hd / 2;
  if (n < n_txt) {
    cs = 1.f;
    sn = 0.f;
    return;
  }
  const int tok = n - n_txt;
  const int axis = pair / npair, i = pair % npair;
  // f32: the angle pos * theta (pos < grid size) is off by a few 1e-6 rad at most
  const float pos = axis == 0 ? (float)(tok / gw) : (float)(tok % gw);
  const float th = exp2f(-13.287712379549449f * 2.f * (float)i / (float)hd);  // 10000^(-2i/hd)
  sincosf(pos * th, &sn, &cs);
}

// Grid-stride over (row, head) items, one warp per item; lane j owns the rotated pairs j
// and j + 32 of the head.
constexpr int QKN_THREADS = 256, QKN_WARPS = QKN_THREADS / 32;

__global__ void __launch_bounds__(QKN_THREADS) qk_norm_rope_fwd_kernel(QkNormRope a) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int dh = a.d / a.heads;
  const int is_f32 = a.dtype == JAGG_DTYPE_F32;
  const int64_t items = (int64_t)a.M * a.heads;
  for (int64_t w = (int64_t)blockIdx.x * QKN_WARPS + threadIdx.x / 32; w < items;
       w += (int64_t)gridDim.x * QKN_WARPS) {
    const int hd = (int)(w % a.heads);
    const int m = (int)(w / a.heads);
    const int n = m % a.N;
    const bool txt = n < a.n_txt;
    for (int which = 0; which < 2; ++which) {
      const void* scl = which == 0 ? (txt ? a.qscale_txt : a.qscale_img) : (txt ? a.kscale_txt : a.kscale_img);
      const int64_t base = (int64_t)m * a.ld_qkv + which * a.d + hd * dh;
      float x[4] = {0.f, 0.f, 0.f, 0.f};
      float ss = 0.f;
      for (int j = 0; j < 2; ++j) {
        const int pair = lane + 32 * j;
        if (2 * pair < dh) {
          x[2 * j] = ldx(a.qkv, base + 2 * pair, is_f32);
          x[2 * j + 1] = ldx(a.qkv, base + 2 * pair + 1, is_f32);
          ss += x[2 * j] * x[2 * j] + x[2 * j + 1] * x[2 * j + 1];
        }
      }
      const float r = rsqrtf(warp_sum(ss) / dh + 1e-6f);
      for (int j = 0; j < 2; ++j) {
        const int pair = lane + 32 * j;
        if (2 * pair < dh) {
          const float y0 = x[2 * j] * r * ldx(scl, 2 * pair, is_f32);
          const float y1 = x[2 * j + 1] * r * ldx(scl, 2 * pair + 1, is_f32);
          float cs = 1.f, sn = 0.f;
          if (a.rope) rope_angle(n, a.n_txt, a.gw, dh, pair, cs, sn);
          const int64_t o = (int64_t)m * 2 * a.d + which * a.d + hd * dh + 2 * pair;
          stx(a.qk_out, o, is_f32, y0 * cs - y1 * sn);
          stx(a.qk_out, o + 1, is_f32, y0 * sn + y1 * cs);
        }
      }
      if (lane == 0) (which == 0 ? a.rq : a.rk)[(int64_t)m * a.heads + hd] = r;
    }
  }
}

// The scale gradients sum over every (row, head): each lane keeps its elements' partial
// sums in registers (q / k x text / image), the block adds its warps' partials in shared
// memory and issues one atomic per element.
__global__ void __launch_bounds__(QKN_THREADS) qk_norm_rope_bwd_kernel(QkNormRopeBwd b) {
  pdl_wait();
  const QkNormRope& a = b.f;
  __shared__ float part[QKN_WARPS][4][128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
  const int dh = a.d / a.heads;
  const int is_f32 = a.dtype == JAGG_DTYPE_F32;
  float acc[4][4];  // [which * 2 + stream][element]
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
  const int64_t items = (int64_t)a.M * a.heads;
  for (int64_t w = (int64_t)blockIdx.x * QKN_WARPS + warp; w < items; w += (int64_t)gridDim.x * QKN_WARPS) {
    const int hd = (int)(w % a.heads);
    const int m = (int)(w / a.heads);
    const int n = m % a.N;
    const bool txt = n < a.n_txt;
    const float* q32 = b.dq32 ? b.dq32 + ((int64_t)(m / a.N) * b.dq32_seq + b.dq32_row0 + n) * a.d + hd * dh : nullptr;
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      const void* scl = which == 0 ? (txt ? a.qscale_txt : a.qscale_img) : (txt ? a.kscale_txt : a.kscale_img);
      const float r = (which == 0 ? a.rq : a.rk)[(int64_t)m * a.heads + hd];
      const int64_t xb = (int64_t)m * a.ld_qkv + which * a.d + hd * dh;
      const int64_t gb = (int64_t)m * b.ld_dqk + which * a.d + hd * dh;
      float x[4] = {0.f, 0.f, 0.f, 0.f}, u[4] = {0.f, 0.f, 0.f, 0.f}, dsc[4] = {0.f, 0.f, 0.f, 0.f};
      float xu = 0.f;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int pair = lane + 32 * j;
        if (2 * pair < dh) {
          // undo the rotation of the incoming gradient (rotate by -angle)
          const bool wide = which == 0 && q32;
          const float g0 = wide ? q32[2 * pair] : ldx(b.dqk, gb + 2 * pair, is_f32);
          const float g1 = wide ? q32[2 * pair + 1] : ldx(b.dqk, gb + 2 * pair + 1, is_f32);
          float cs = 1.f, sn = 0.f;
          if (a.rope) rope_angle(n, a.n_txt, a.gw, dh, pair, cs, sn);
          const float dy0 = g0 * cs + g1 * sn;
          const float dy1 = -g0 * sn + g1 * cs;
          x[2 * j] = ldx(a.qkv, xb + 2 * pair, is_f32);
          x[2 * j + 1] = ldx(a.qkv, xb + 2 * pair + 1, is_f32);
          dsc[2 * j] = dy0 * x[2 * j] * r;
          dsc[2 * j + 1] = dy1 * x[2 * j + 1] * r;
          u[2 * j] = dy0 * ldx(scl, 2 * pair, is_f32);
          u[2 * j + 1] = dy1 * ldx(scl, 2 * pair + 1, is_f32);
          xu += x[2 * j] * u[2 * j] + x[2 * j + 1] * u[2 * j + 1];
        }
      }
      const int slot = which * 2 + (txt ? 0 : 1);
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[slot][e] += dsc[e];
      xu = warp_sum(xu);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int pair = lane + 32 * j;
        if (2 * pair < dh) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float dx = r * u[2 * j + e] - x[2 * j + e] * r * r * r * xu / dh;
            stx(b.dqk, gb + 2 * pair + e, is_f32, dx);
          }
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int pair = lane + 32 * j;
      if (2 * pair < dh) {
        part[warp][i][2 * pair] = acc[i][2 * j];
        part[warp][i][2 * pair + 1] = acc[i][2 * j + 1];
      }
    }
  __syncthreads();
  float* dst[4] = {b.dqs_txt, b.dqs_img, b.dks_txt, b.dks_img};
  for (int t = threadIdx.x; t < 4 * dh; t += QKN_THREADS) {
    const int i = t / dh, c = t % dh;
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < QKN_WARPS; ++w) s += part[w][i][c];
    if (s != 0.f) atomicAdd(dst[i] + c, s);
  }
}

// Head dim 128 in bf16 (the Flux and Qwen widths): lane l owns the 4 consecutive elements
// [4l, 4l + 4) of q and of k, i.e. the rotated pairs 2l and 2l + 1, so every operand moves
// in 8-byte vectors and each lane's RMSNorm scales and RoPE frequencies are fixed for the
// whole kernel.  The angles are the ones rope_angle forms (same expressions), so the forward
// rotation and its inverse in the backward agree bit for bit.  A warp walks units, rows or parts
// of their heads, two (backward) or four (forward) heads at a time: 2 KB of loads in flight per
// warp.  Bound by HBM on many rows, by latency on a few thousand: with whole rows only, 4096
// rows of 24 heads were 1.1 rounds of the resident warps (text + image of 6144 rows at d = 3072:
// backward 72 -> 65 us with dq read from attention's f32 accumulator, a pass over it less;
// forward 49 -> 45; 2973 rows 49 -> 41 and 33 -> 28).
constexpr int QKV_ITEMS = 2;      // heads per warp iteration of the backward
constexpr int QKV_ITEMS_FWD = 4;  // and of the forward (fewer live registers)

__device__ __forceinline__ void bf16x4_load(const bf16* p, float (&v)[4]) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  const bf16* h = reinterpret_cast<const bf16*>(&raw);
  v[0] = __bfloat162float(h[0]); v[1] = __bfloat162float(h[1]);
  v[2] = __bfloat162float(h[2]); v[3] = __bfloat162float(h[3]);
}
__device__ __forceinline__ void bf16x4_store(bf16* p, const float (&v)[4]) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
  uint2 raw;
  raw.x = *reinterpret_cast<uint32_t*>(&a);
  raw.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = raw;
}
// RoPE angles of head dim 128 as a table in shared memory, filled by each block: entry
// [pos][i] = (cos, sin) of pos * theta_i for the 32 frequencies of one axis, pos below the
// larger grid side; the values are rope_angle's (same expressions), so the forward rotation
// and its inverse agree bit for bit.  QKN_TABLE_MAX bounds the grid side the table serves.
constexpr int QKN_TABLE_MAX = 128;
__device__ __forceinline__ int rope_table_side(const QkNormRope& a) {
  const int gh = (a.N - a.n_txt) / a.gw;
  return gh > a.gw ? gh : a.gw;
}
__device__ __forceinline__ void rope_table_fill(const QkNormRope& a, float2* tab) {
  const int side = rope_table_side(a);
  for (int t = threadIdx.x; t < side * 32; t += blockDim.x) {
    const int pos = t / 32, i = t % 32;
    const float th = exp2f(-13.287712379549449f * 2.f * (float)i / 64.f);  // 10000^(-2i/64)
    float sn, cs;
    sincosf((float)pos * th, &sn, &cs);
    tab[t] = make_float2(cs, sn);
  }
}
// cos / sin of the lane's two pairs (2 lane, 2 lane + 1: axis lane / 16, frequencies
// 2 lane % 32 and + 1) for token n; identity for text tokens
__device__ __forceinline__ void rope_lane(const QkNormRope& a, const float2* tab, int n, int lane, float (&cs)[2],
                                          float (&sn)[2]) {
  cs[0] = cs[1] = 1.f;
  sn[0] = sn[1] = 0.f;
  if (!a.rope || n < a.n_txt) return;
  const int tok = n - a.n_txt;
  const int pos = lane < 16 ? tok / a.gw : tok % a.gw;
  const float4 v = *reinterpret_cast<const float4*>(tab + pos * 32 + ((2 * lane) & 31));
  cs[0] = v.x; sn[0] = v.y; cs[1] = v.z; sn[1] = v.w;
}

__global__ void __launch_bounds__(QKN_THREADS) qk_norm_rope_fwd_v_kernel(QkNormRope a, int heads_per_unit) {
  extern __shared__ __align__(16) float2 rope_tab[];  // [side][32] when a.rope
  if (a.rope) rope_table_fill(a, rope_tab);
  pdl_wait();
  __syncthreads();
  const int lane = threadIdx.x & 31;
  float scl[4][4];  // q txt, q img, k txt, k img: this lane's 4 elements
  bf16x4_load(static_cast<const bf16*>(a.qscale_txt) + 4 * lane, scl[0]);
  bf16x4_load(static_cast<const bf16*>(a.qscale_img) + 4 * lane, scl[1]);
  bf16x4_load(static_cast<const bf16*>(a.kscale_txt) + 4 * lane, scl[2]);
  bf16x4_load(static_cast<const bf16*>(a.kscale_img) + 4 * lane, scl[3]);
  // one unit per warp, its heads four at a time: the token's stream and angles once per unit
  const int upr = (a.heads + heads_per_unit - 1) / heads_per_unit;
  for (int unit = blockIdx.x * QKN_WARPS + threadIdx.x / 32; unit < a.M * upr; unit += gridDim.x * QKN_WARPS) {
    const int m = unit / upr, h_lo = (unit - m * upr) * heads_per_unit;
    const int h_hi = min(h_lo + heads_per_unit, a.heads);
    const int n = m % a.N;
    const bool txt = n < a.n_txt;
    float cs[2], sn[2];
    rope_lane(a, rope_tab, n, lane, cs, sn);
    const bf16* row = static_cast<const bf16*>(a.qkv) + (int64_t)m * a.ld_qkv + 4 * lane;
    bf16* out = static_cast<bf16*>(a.qk_out) + (int64_t)m * 2 * a.d + 4 * lane;
    for (int h0 = h_lo; h0 < h_hi; h0 += QKV_ITEMS_FWD) {
      float x[QKV_ITEMS_FWD][2][4];
#pragma unroll
      for (int it = 0; it < QKV_ITEMS_FWD; ++it) {
        const int hd = h0 + it < h_hi ? h0 + it : h0;
#pragma unroll
        for (int which = 0; which < 2; ++which) bf16x4_load(row + which * a.d + hd * 128, x[it][which]);
      }
#pragma unroll
      for (int it = 0; it < QKV_ITEMS_FWD; ++it) {
        const int hd = h0 + it;
        if (hd >= h_hi) break;
#pragma unroll
        for (int which = 0; which < 2; ++which) {
          float sc[4];  // selected per element: the array index stays a compile-time constant
#pragma unroll
          for (int e = 0; e < 4; ++e) sc[e] = txt ? scl[which * 2][e] : scl[which * 2 + 1][e];
          const float* xv = x[it][which];
          const float r =
              rsqrtf(warp_sum(xv[0] * xv[0] + xv[1] * xv[1] + xv[2] * xv[2] + xv[3] * xv[3]) / 128.f + 1e-6f);
          float o[4];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float y0 = xv[2 * e] * r * sc[2 * e], y1 = xv[2 * e + 1] * r * sc[2 * e + 1];
            o[2 * e] = y0 * cs[e] - y1 * sn[e];
            o[2 * e + 1] = y0 * sn[e] + y1 * cs[e];
          }
          bf16x4_store(out + which * a.d + hd * 128, o);
          if (lane == 0) (which == 0 ? a.rq : a.rk)[(int64_t)m * a.heads + hd] = r;
        }
      }
    }
  }
}

template <bool DQ32>
__global__ void __launch_bounds__(QKN_THREADS, 3) qk_norm_rope_bwd_v_kernel(QkNormRopeBwd b, int heads_per_unit) {
  const QkNormRope& a = b.f;
  __shared__ float part[QKN_WARPS][4][128];
  extern __shared__ __align__(16) float2 rope_tab[];  // [side][32] when a.rope
  if (a.rope) rope_table_fill(a, rope_tab);
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
  __shared__ __align__(16) float scl[4][128];  // q txt, q img, k txt, k img
  for (int t = threadIdx.x; t < 4 * 128; t += QKN_THREADS) {
    const void* p = t < 128 ? a.qscale_txt : t < 256 ? a.qscale_img : t < 384 ? a.kscale_txt : a.kscale_img;
    scl[t / 128][t % 128] = __bfloat162float(static_cast<const bf16*>(p)[t % 128]);
  }
  // scale gradients of the warp's units, [which * 2 + stream][element]: one read-modify-write
  // of the lane's 4 elements per unit
  float4* wpart = reinterpret_cast<float4*>(&part[warp][0][0]);
#pragma unroll
  for (int i = 0; i < 4; ++i) wpart[i * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  // one unit per warp, its heads two at a time: the token's stream and angles once per unit
  const int upr = (a.heads + heads_per_unit - 1) / heads_per_unit;
  for (int unit = blockIdx.x * QKN_WARPS + warp; unit < a.M * upr; unit += gridDim.x * QKN_WARPS) {
    const int m = unit / upr, h_lo = (unit - m * upr) * heads_per_unit;
    const int h_hi = min(h_lo + heads_per_unit, a.heads);
    const int n = m % a.N;
    const bool txt = n < a.n_txt;
    float cs[2], sn[2];
    rope_lane(a, rope_tab, n, lane, cs, sn);
    const bf16* xrow = static_cast<const bf16*>(a.qkv) + (int64_t)m * a.ld_qkv + 4 * lane;
    bf16* grow = static_cast<bf16*>(b.dqk) + (int64_t)m * b.ld_dqk + 4 * lane;
    const float* q32 = nullptr;
    if (DQ32) q32 = b.dq32 + ((int64_t)(m / a.N) * b.dq32_seq + b.dq32_row0 + n) * a.d + 4 * lane;
    float rowacc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};  // q, k scale gradients of the unit
    for (int h0 = h_lo; h0 < h_hi; h0 += QKV_ITEMS) {
      float x[QKV_ITEMS][2][4], g[QKV_ITEMS][2][4], rms[QKV_ITEMS][2];
#pragma unroll
      for (int it = 0; it < QKV_ITEMS; ++it) {
        const int hd = h0 + it < h_hi ? h0 + it : h0;
#pragma unroll
        for (int which = 0; which < 2; ++which) {
          bf16x4_load(xrow + which * a.d + hd * 128, x[it][which]);
          if (DQ32 && which == 0) {
            const float4 q = *reinterpret_cast<const float4*>(q32 + hd * 128);
            g[it][0][0] = q.x; g[it][0][1] = q.y; g[it][0][2] = q.z; g[it][0][3] = q.w;
          } else {
            bf16x4_load(grow + which * a.d + hd * 128, g[it][which]);
          }
          // with the rows: behind the first store to dqk it would be a load of its own per head
          rms[it][which] = (which == 0 ? a.rq : a.rk)[(int64_t)m * a.heads + hd];
        }
      }
#pragma unroll
      for (int it = 0; it < QKV_ITEMS; ++it) {
        const int hd = h0 + it;
        if (hd >= h_hi) break;
#pragma unroll
        for (int which = 0; which < 2; ++which) {
          const float4 sc4 = *reinterpret_cast<const float4*>(&scl[which * 2 + (txt ? 0 : 1)][4 * lane]);
          const float sc[4] = {sc4.x, sc4.y, sc4.z, sc4.w};
          const float* xv = x[it][which];
          const float r = rms[it][which];
          float u[4], dy[4];
#pragma unroll
          for (int e = 0; e < 2; ++e) {  // undo the rotation of the incoming gradient
            const float g0 = g[it][which][2 * e], g1 = g[it][which][2 * e + 1];
            dy[2 * e] = g0 * cs[e] + g1 * sn[e];
            dy[2 * e + 1] = -g0 * sn[e] + g1 * cs[e];
          }
          float xu = 0.f;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            rowacc[which][e] += dy[e] * xv[e] * r;
            u[e] = dy[e] * sc[e];
            xu += xv[e] * u[e];
          }
          xu = warp_sum(xu);
          float dx[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) dx[e] = r * u[e] - xv[e] * r * r * r * xu / 128.f;
          bf16x4_store(grow + which * a.d + hd * 128, dx);
        }
      }
    }
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      float4& q = wpart[(which * 2 + (txt ? 0 : 1)) * 32 + lane];
      q.x += rowacc[which][0]; q.y += rowacc[which][1]; q.z += rowacc[which][2]; q.w += rowacc[which][3];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 4 * 128; t += QKN_THREADS) {
    const int i = t / 128, c = t % 128;
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < QKN_WARPS; ++w) s += part[w][i][c];
    float* dst = i == 0 ? b.dqs_txt : i == 1 ? b.dqs_img : i == 2 ? b.dks_txt : b.dks_img;
    if (s != 0.f) atomicAdd(dst + c, s);
  }
}

}  // namespace

// ------------------------------------------------------------------ launchers
int launch_patchify(const void* z, int in_f32, void* xp, int out_f32, int dtype, int B, int C, int H, int W, int p,
                    cudaStream_t s) {
  (void)dtype;
  const int64_t n = (int64_t)B * C * H * W;
  JAGG_CUDA_TRY(launch(patchify_kernel, grid_for(n, 256), 256, 0, s, z, in_f32, xp, out_f32, B, C, H, W, p));
  JAGG_LAUNCHED();
  return JAGG_OK;
}
int launch_unpatchify(const void* xp, void* z, int dtype, int B, int C, int H, int W, int p, cudaStream_t s) {
  const int64_t n = (int64_t)B * C * H * W;
  JAGG_CUDA_TRY(launch(unpatchify_kernel, grid_for(n, 256), 256, 0, s, xp, z, dtype == JAGG_DTYPE_F32, B, C, H, W,
                       p));
  JAGG_LAUNCHED();
  return JAGG_OK;
}
int launch_timestep_embedding(const float* t, float* phi, int B, int dim, cudaStream_t s) {
  JAGG_CUDA_TRY(launch(temb_kernel, grid_for((int64_t)B * dim / 2, 256), 256, 0, s, t, phi, B, dim));
  JAGG_LAUNCHED();
  return JAGG_OK;
}
int launch_silu(const float* in, float* out, int64_t n, cudaStream_t s) {
  JAGG_CUDA_TRY(launch(silu_kernel, grid_for(n, 256), 256, 0, s, in, out, n));
  JAGG_LAUNCHED();
  return JAGG_OK;
}
int launch_mul_silu_grad(float* g, const float* x, void* copy, int dtype, int64_t n, cudaStream_t s) {
  JAGG_CUDA_TRY(launch(mul_silu_grad_kernel, grid_for(n, 256), 256, 0, s, g, x, copy, dtype == JAGG_DTYPE_F32, n));
  JAGG_LAUNCHED();
  return JAGG_OK;
}
int launch_add_pos_embed(float* h, int B, int rows_per_seq, int row0, int gh, int gw, int d, cudaStream_t s) {
  JAGG_CUDA_TRY(launch(pos_embed_kernel, ceil_div((int64_t)gh * gw * (d / 4), 256), 256, 0, s, h, B, rows_per_seq,
                       row0, gh, gw, d));
  JAGG_LAUNCHED();
  return JAGG_OK;
}
int launch_ln_mod_fwd(const LnModFwd& a, cudaStream_t s) {
  JAGG_CHECK_ARG(a.d % 4 == 0 && a.d <= 128 * LN_MAXV, "ln_mod: hidden %d unsupported", a.d);
  const int tok = prof_start(s);
  auto fixed = [&](auto kernel, int rows_per_cta) {
    return launch(kernel, ceil_div(a.M, rows_per_cta), 128, 0, s, a);
  };
  switch (a.d) {  // the widths of a warp per row up to 1024 columns, then of four warps per row
    case 512: JAGG_CUDA_TRY(fixed(ln_mod_fwd_fixed_kernel<4, 1>, 4)); break;
    case 768: JAGG_CUDA_TRY(fixed(ln_mod_fwd_fixed_kernel<6, 1>, 4)); break;
    case 1024: JAGG_CUDA_TRY(fixed(ln_mod_fwd_fixed_kernel<8, 1>, 4)); break;
    case 2048: JAGG_CUDA_TRY(fixed(ln_mod_fwd_fixed_kernel<4, 4>, 1)); break;
    case 3072: JAGG_CUDA_TRY(fixed(ln_mod_fwd_fixed_kernel<6, 4>, 1)); break;
    default: JAGG_CUDA_TRY(launch(ln_mod_fwd_kernel, ceil_div(a.M, 8), 256, 0, s, a));
  }
  JAGG_LAUNCHED();
  // algorithmic bytes: h read (f32), the modulated output written (storage type), statistics
  prof_stop(tok, s, PROF_LN_FWD, 0.0,
            (double)a.M * (a.d * (4.0 + (a.dtype == JAGG_DTYPE_F32 ? 4.0 : 2.0)) + 8.0));
  return JAGG_OK;
}
// The row-in-registers kernel: LayerNorm backwards with an f32 dm, with or without the gate.
template <int NV>
int launch_ln_gate_rowreg(const LnGateBwd& a, cudaStream_t s) {
  if (!a.do_gate) return launch_ln_gate_rowreg_t<NV, false, false>(a, s);
  return a.dtype == JAGG_DTYPE_F32 ? launch_ln_gate_rowreg_t<NV, true, false>(a, s)
                                   : launch_ln_gate_rowreg_t<NV, true, true>(a, s);
}

int ln_gate_route(const LnGateBwd& a) {
  switch (a.d) {
    case 64: case 128: case 256: return ln_gate_narrow_serves(a) ? LNG_NARROW : LNG_GENERAL;
    case 384: return a.do_ln && a.dm_f32 ? LNG_ROWREG : LNG_GENERAL;
    case 512: case 768: return ln_gate_ring_serves(a) ? LNG_RING : a.do_ln && a.dm_f32 ? LNG_ROWREG : LNG_GENERAL;
    case 1024: case 2048: case 3072: return ln_gate_ring_serves(a) ? LNG_RING : LNG_GENERAL;
  }
  return LNG_GENERAL;
}
int launch_ln_gate_bwd(const LnGateBwd& a, cudaStream_t s) {
  JAGG_CHECK_ARG(a.d % 4 == 0 && a.d <= 3072, "ln_gate_bwd: hidden %d unsupported", a.d);
  JAGG_CHECK_ARG(a.M % a.rows_per_seq == 0, "ln_gate_bwd: rows not a whole number of sequences");
  if (!a.do_ln && !a.do_gate) return JAGG_OK;
  const int smem = 4 * a.d * (int)sizeof(float);
  const int tok = prof_start(s);
  int st = JAGG_ERR_UNSUPPORTED;
  switch (ln_gate_route(a)) {
    case LNG_NARROW:
      st = a.d == 64 ? launch_ln_gate_narrow<16, 1>(a, s)
                     : a.d == 128 ? launch_ln_gate_narrow<32, 1>(a, s) : launch_ln_gate_narrow<32, 2>(a, s);
      break;
    case LNG_RING:
      st = a.d == 512    ? launch_ln_gate_ring<2, 2>(a, s)
           : a.d == 768  ? launch_ln_gate_ring<3, 2>(a, s)
           : a.d == 1024 ? launch_ln_gate_ring<2, 4>(a, s)
           : a.d == 2048 ? launch_ln_gate_ring<2, 8>(a, s) : launch_ln_gate_ring<3, 8>(a, s);
      break;
    case LNG_ROWREG:
      st = a.d == 384 ? launch_ln_gate_rowreg<3>(a, s)
                      : a.d == 512 ? launch_ln_gate_rowreg<4>(a, s) : launch_ln_gate_rowreg<6>(a, s);
      break;
    default:
      st = a.d == 1024   ? launch_ln_gate_nv<8>(a, smem, s)
           : a.d == 1536 ? launch_ln_gate_nv<12>(a, smem, s)
           : a.d == 3072 ? launch_ln_gate_nv<24>(a, smem, s) : launch_ln_gate_nv<0>(a, smem, s);
  }
  JAGG_TRY(st);
  // algorithmic bytes: dh read + write (f32), dm (f32), h (f32), y and dy (storage type)
  const double elem = (double)a.M * a.d;
  prof_stop(tok, s, PROF_LN_BWD, 0.0,
            elem * ((a.do_ln ? 16.0 : 4.0) + (a.do_gate ? 2.0 * (a.dtype == JAGG_DTYPE_F32 ? 4 : 2) : 0.0)));
  return JAGG_OK;
}
int launch_colsum(const void* X, int x_f32, int dtype, int rows, int cols, int64_t ld, float* db, cudaStream_t s) {
  (void)dtype;
  const int tok = prof_start(s);
  // algorithmic bytes: X read once, db read and written
  const double bytes = (double)rows * cols * (x_f32 ? 4 : 2) + 8.0 * cols;
  if (!x_f32 && cols % 8 == 0 && ld % 8 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0) {
    const int cb = ceil_div(cols, 256);
    const int want = ceil_div((int64_t)CSV_BLOCKS_PER_SM * sm_count(), cb);  // row blocks that fill the machine
    int rpb = (ceil_div(rows, want) + 7) / 8 * 8;
    rpb = rpb > CSV_MAX_ROWS ? CSV_MAX_ROWS : rpb;
    if (ceil_div(rows, rpb) > 65535) rpb = (ceil_div(rows, 65535) + 7) / 8 * 8;
    dim3 grid(cb, ceil_div(rows, rpb));
    JAGG_CUDA_TRY(launch(colsum_bf16x8_kernel, grid, 256, 0, s, static_cast<const bf16*>(X), rows, cols, ld, rpb, db));
    JAGG_LAUNCHED();
    prof_stop(tok, s, PROF_COLSUM, 0.0, bytes);
    return JAGG_OK;
  }
  dim3 grid(ceil_div(cols, 256), ceil_div(rows, CS_ROWS));
  JAGG_CUDA_TRY(launch(colsum_kernel, grid, 256, 0, s, X, x_f32, rows, cols, ld, db));
  JAGG_LAUNCHED();
  prof_stop(tok, s, PROF_COLSUM, 0.0, bytes);
  return JAGG_OK;
}
int launch_gather_rows(const float* in, int64_t ld_in, int seg, int seg_off, int64_t seg_stride, void* out,
                       int dtype, int rows, int cols, cudaStream_t s) {
  if (cols % 4 == 0 && ld_in % 4 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0 &&
      (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
    JAGG_CUDA_TRY(launch(gather_rows_v4_kernel, grid_for((int64_t)rows * (cols / 4), 256), 256, 0, s, in, ld_in, seg,
                         seg_off, seg_stride, out, dtype == JAGG_DTYPE_F32, rows, cols));
  } else {
    JAGG_CUDA_TRY(launch(gather_rows_kernel, grid_for((int64_t)rows * cols, 256), 256, 0, s, in, ld_in, seg, seg_off,
                         seg_stride, out, dtype == JAGG_DTYPE_F32, rows, cols));
  }
  JAGG_LAUNCHED();
  return JAGG_OK;
}
int launch_copy_rows(const void* in, int64_t ld_in, int in_seg, int in_seg_off, int64_t in_seg_stride, void* out,
                     int64_t ld_out, int out_seg, int out_seg_off, int64_t out_seg_stride, int rows, int cols,
                     int elem_bytes, cudaStream_t s) {
  const int tok = prof_start(s);
  const int64_t row_b = (int64_t)cols * elem_bytes;
  const bool v16 = row_b % 16 == 0 && (ld_in * elem_bytes) % 16 == 0 && (ld_out * elem_bytes) % 16 == 0 &&
                   (reinterpret_cast<uintptr_t>(in) & 15) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  const int g = grid_for((int64_t)rows * cols, 256);
  if (v16 && rows > 0) {
    const int nb = rows < 8 * sm_count() ? rows : 8 * sm_count();
    JAGG_CUDA_TRY(launch(copy_rows_v16_kernel, nb, 256, 0, s, static_cast<const uint8_t*>(in), ld_in * elem_bytes,
                         in_seg, in_seg_off,
                                            in_seg_stride, static_cast<uint8_t*>(out), ld_out * elem_bytes, out_seg,
                                            out_seg_off, out_seg_stride, rows, (int)(row_b / 16)));
  } else if (elem_bytes == 4)
    JAGG_CUDA_TRY(launch(copy_rows_kernel<float>, g, 256, 0, s, static_cast<const float*>(in), ld_in, in_seg,
                         in_seg_off, in_seg_stride,
                                             static_cast<float*>(out), ld_out, out_seg, out_seg_off, out_seg_stride,
                                             rows, cols));
  else
    JAGG_CUDA_TRY(launch(copy_rows_kernel<uint16_t>, g, 256, 0, s, static_cast<const uint16_t*>(in), ld_in, in_seg,
                         in_seg_off,
                                                in_seg_stride, static_cast<uint16_t*>(out), ld_out, out_seg,
                                                out_seg_off, out_seg_stride, rows, cols));
  JAGG_LAUNCHED();
  prof_stop(tok, s, PROF_COPY, 0.0, 2.0 * rows * cols * elem_bytes);
  return JAGG_OK;
}
// The vectorised kernels serve head dim 128 in bf16 with 8-byte aligned rows and scales.
static bool aligned8(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7) == 0; }
static int qkn_table_bytes(const QkNormRope& a) {
  if (!a.rope) return 0;
  const int gh = (a.N - a.n_txt) / a.gw;
  return (gh > a.gw ? gh : a.gw) * 32 * (int)sizeof(float2);
}
static bool qkn_vector(const QkNormRope& a) {
  if (a.rope && (a.gw <= 0 || (a.N - a.n_txt) % a.gw || (a.N - a.n_txt) / a.gw > QKN_TABLE_MAX ||
                 a.gw > QKN_TABLE_MAX))
    return false;
  return a.dtype == JAGG_DTYPE_BF16 && a.heads > 0 && a.d == 128 * a.heads && a.ld_qkv % 4 == 0 &&
         (int64_t)a.M * a.heads < (1ll << 30) &&
         aligned8(a.qkv) && aligned8(a.qk_out) && aligned8(a.qscale_txt) && aligned8(a.qscale_img) &&
         aligned8(a.kscale_txt) && aligned8(a.kscale_img);
}
// Heads per unit of the vectorised kernels (a multiple of `items`): whole rows where there are many,
// parts of a row where whole rows would leave the last round of the resident warps nearly empty.
// A unit costs its batches of heads plus about half a batch (stream, angles, scale sums).
static int qkn_heads_per_unit(const QkNormRope& a, int items, int warps) {
  int best = a.heads;
  double best_cost = 0.0;
  for (int parts = 1; parts <= ceil_div(a.heads, items); ++parts) {
    const int hu = ceil_div(ceil_div(a.heads, parts), items) * items;
    const int64_t units = (int64_t)a.M * ceil_div(a.heads, hu);
    const double cost = (double)ceil_div(units, (int64_t)warps) * (hu / items + 0.5);
    if (parts == 1 || cost < 0.97 * best_cost) {
      best_cost = cost;
      best = hu;
    }
  }
  return best;
}
int launch_qk_norm_rope_fwd(const QkNormRope& a, cudaStream_t s) {
  JAGG_CHECK_ARG(a.heads > 0 && a.d % a.heads == 0 && a.d / a.heads <= 128 && (a.d / a.heads) % 2 == 0,
                 "qk_norm: head dim unsupported");
  if (a.M <= 0) return JAGG_OK;
  const int64_t blocks = ((int64_t)a.M * a.heads + QKN_WARPS - 1) / QKN_WARPS;
  const int tok = prof_start(s);
  if (qkn_vector(a)) {
    const int cap = 3 * sm_count();  // the resident blocks (77 registers, 3 per SM)
    const int hu = qkn_heads_per_unit(a, QKV_ITEMS_FWD, cap * QKN_WARPS);
    const int64_t vb = ceil_div((int64_t)a.M * ceil_div(a.heads, hu), (int64_t)QKN_WARPS);
    JAGG_CUDA_TRY(launch(qk_norm_rope_fwd_v_kernel, (int)(vb < cap ? vb : cap), QKN_THREADS, qkn_table_bytes(a), s,
                         a, hu));
  } else {
    JAGG_CUDA_TRY(launch(qk_norm_rope_fwd_kernel, (int)(blocks < 65536 ? blocks : 65536), QKN_THREADS, 0, s, a));
  }
  JAGG_LAUNCHED();
  // algorithmic bytes: raw q, k read, transformed q, k written (storage type), 1/rms of both
  const double esz = a.dtype == JAGG_DTYPE_F32 ? 4.0 : 2.0;
  prof_stop(tok, s, PROF_QKN_FWD, 0.0, (double)a.M * (4.0 * a.d * esz + 8.0 * a.heads));
  return JAGG_OK;
}
int launch_qk_norm_rope_bwd(const QkNormRopeBwd& a, cudaStream_t s) {
  const QkNormRope& f = a.f;
  JAGG_CHECK_ARG(f.heads > 0 && f.d % f.heads == 0 && f.d / f.heads <= 128 && (f.d / f.heads) % 2 == 0,
                 "qk_norm: head dim unsupported");
  JAGG_CHECK_ARG(a.dqs_txt && a.dks_txt && a.dqs_img && a.dks_img, "qk_norm: null scale gradient");
  if (f.M <= 0) return JAGG_OK;
  // a few blocks per SM: each block ends in 4 dh atomics
  const int64_t blocks = ((int64_t)f.M * f.heads + QKN_WARPS - 1) / QKN_WARPS;
  const int cap = 4 * sm_count();
  const int tok = prof_start(s);
  if (qkn_vector(f) && a.ld_dqk % 4 == 0 && aligned8(a.dqk) && (reinterpret_cast<uintptr_t>(a.dq32) & 15) == 0) {
    // a few blocks per SM: each block ends in 4 x 128 scale-gradient atomics
    const int vcap = 3 * sm_count();  // the resident blocks (80 registers, 3 per SM)
    const int hu = qkn_heads_per_unit(f, QKV_ITEMS, vcap * QKN_WARPS);
    const int64_t vb = ceil_div((int64_t)f.M * ceil_div(f.heads, hu), (int64_t)QKN_WARPS);
    JAGG_CUDA_TRY(launch(a.dq32 ? qk_norm_rope_bwd_v_kernel<true> : qk_norm_rope_bwd_v_kernel<false>,
                         (int)(vb < vcap ? vb : vcap), QKN_THREADS, qkn_table_bytes(f), s, a, hu));
  } else {
    JAGG_CUDA_TRY(launch(qk_norm_rope_bwd_kernel, (int)(blocks < cap ? blocks : cap), QKN_THREADS, 0, s, a));
  }
  JAGG_LAUNCHED();
  // algorithmic bytes: dq, dk read and written, raw q, k read (storage type, dq in f32 if so given), 1/rms
  const double esz = f.dtype == JAGG_DTYPE_F32 ? 4.0 : 2.0;
  const double dq = a.dq32 ? 4.0 : esz;
  prof_stop(tok, s, PROF_QKN_BWD, 0.0, (double)f.M * (f.d * (dq + 5.0 * esz) + 8.0 * f.heads));
  return JAGG_OK;
}

}  // namespace jagg
