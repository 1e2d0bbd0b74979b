// Products with a handful of rows: the t-embedding MLP and the stacked modulation of B sequences.
// They are bound by streaming the weight matrix (or its gradient) once, so they run as streaming
// kernels instead of tensor-core tiles that would be nearly empty.
#include "gemm.cuh"
#include "ptx.cuh"
#include "rows.cuh"

namespace jagg {

namespace {

// ------------------------------------------------------------------ C = act(X) W^T + bias
// Each CTA keeps act(X), rounded to bf16, in shared memory (16 rows, zeros past B); a warp streams
// 8 rows of W at a time, 16 bytes per lane, into mma.m16n8k16: W is read once, straight into the
// B fragment.  A lane's 8 consecutive elements of K serve as its fragment elements of two k16
// steps; X is read from shared memory in the same order, so the sum over K is only permuted.
// Rows of X are 64 bytes more than a multiple of 128 apart: the 8 lanes of a phase read
// distinct banks.  KS warps split K where the rows of W alone would leave the machine idle.
// 4 x 43008 x 3072: 78 -> 61 us, 16 x 56832 x 768 35 -> 22, 4 x 3072 x 256 13 -> 8 against the tensor-core
// tiles (and two launches less per product: the activation and its rounding).
constexpr int RF_MAX_WARPS = 16;

template <int KS>
__global__ void __launch_bounds__(32 * RF_MAX_WARPS, 1) rows_fwd_kernel(RowsFwd a) {
  extern __shared__ __align__(16) uint8_t rf_sm[];
  __shared__ float part[KS > 1 ? RF_MAX_WARPS : 1][32][4];
  pdl_wait();
  const int pitch = a.in * 2 + 64;
#pragma unroll 4
  for (int i = threadIdx.x; i < 16 * (a.in / 4); i += blockDim.x) {
    const int b = i / (a.in / 4), c = (i % (a.in / 4)) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (b < a.B) {
      v = *reinterpret_cast<const float4*>(a.x + (int64_t)b * a.in + c);
      if (a.silu) v = make_float4(silu_f(v.x), silu_f(v.y), silu_f(v.z), silu_f(v.w));
    }
    __nv_bfloat162 p[2] = {__floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(v.z, v.w)};
    const uint2 raw = *reinterpret_cast<const uint2*>(p);
    *reinterpret_cast<uint2*>(rf_sm + b * pitch + c * 2) = raw;
    if (blockIdx.x == 0 && b < a.B) *reinterpret_cast<uint2*>(static_cast<bf16*>(a.x_act) + (int64_t)b * a.in + c) = raw;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = lane >> 2, c = lane & 3;
  const int teams = (blockDim.x >> 5) / KS, team = warp / KS, kq = warp % KS;  // a team of KS warps per 8 rows
  const int k_begin = a.in / 32 * kq / KS * 32, k_end = a.in / 32 * (kq + 1) / KS * 32;
  const uint8_t* x0 = rf_sm + row * pitch + c * 16;
  const uint8_t* x1 = x0 + 8 * pitch;
  const int groups = a.out / 8, stride = gridDim.x * teams;
  for (int g0 = 0; g0 < groups; g0 += stride) {
    const int g = g0 + team * gridDim.x + blockIdx.x;  // spread over the CTAs first
    const bool live = g < groups;
    const bf16* w = static_cast<const bf16*>(a.w) + (int64_t)((live ? g : 0) * 8 + row) * a.in + c * 8;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    if (live) {
#pragma unroll 8
      for (int k = k_begin; k < k_end; k += 32) {
        const uint4 wv = __ldcs(reinterpret_cast<const uint4*>(w + k));
        const uint4 lo = *reinterpret_cast<const uint4*>(x0 + k * 2), hi = *reinterpret_cast<const uint4*>(x1 + k * 2);
        ptx::mma_m16n8k16_bf16(acc, lo.x, hi.x, lo.y, hi.y, wv.x, wv.y);
        ptx::mma_m16n8k16_bf16(acc, lo.z, hi.z, lo.w, hi.w, wv.z, wv.w);
      }
    }
    if constexpr (KS > 1) {
      __syncthreads();
#pragma unroll
      for (int e = 0; e < 4; ++e) part[warp][lane][e] = acc[e];
      __syncthreads();
      if (kq != 0) continue;
#pragma unroll
      for (int w2 = 1; w2 < KS; ++w2)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[e] += part[warp + w2][lane][e];
    }
    if (!live) continue;
    const int n = g * 8 + 2 * c;
    const __nv_bfloat162 bb = *reinterpret_cast<const __nv_bfloat162*>(static_cast<const bf16*>(a.bias) + n);
    const float b0 = __bfloat162float(bb.x), b1 = __bfloat162float(bb.y);
    if (row < a.B) *reinterpret_cast<float2*>(a.c + (int64_t)row * a.out + n) = make_float2(acc[0] + b0, acc[1] + b1);
    if (row + 8 < a.B)
      *reinterpret_cast<float2*>(a.c + (int64_t)(row + 8) * a.out + n) = make_float2(acc[2] + b0, acc[3] + b1);
  }
}

// ------------------------------------------------------------------ G += Y^T X, few rows
// G [M, N] f32, Y [K, M] and X [K, N] bf16 with K <= KMAX: an update of rank K.  Bound by reading and
// writing G, which the L2 does: a thread keeps its 4 columns of every X row in registers, walks rows of G and
// sends each row's 4 sums as one 16-byte reduction; Y's values, uniform over the CTA, are broadcast
// from shared memory.  The reductions are atomic as in every other accumulated product, so passes
// on several streams may add into one gradient.  43008 x 3072 of rank 4: 213 -> 188 us (5.6 TB/s
// read and written), 56832 x 768 of rank 5 81 -> 68, of rank 16 68, 3072 x 3072 20 -> 19, against reduce-adds of
// nearly empty tensor-core tiles; a plain read, add and write of G, not safe beside another pass,
// takes 175, 65, 85 and 20.
constexpr int RU_THREADS = 256, RU_CHUNK = 64;

template <int KMAX>
__global__ void __launch_bounds__(RU_THREADS) rank_update_kernel(RankUpdate a) {
  __shared__ __align__(16) float ys[RU_CHUNK][KMAX];  // Y of the chunk's rows, zeros past K
  pdl_wait();
  const int n = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  const bool live = n < a.N;
  float4 x[KMAX];
#pragma unroll
  for (int k = 0; k < KMAX; ++k) {
    x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < a.K && live) {
      const uint2 raw = *reinterpret_cast<const uint2*>(a.x + (int64_t)k * a.ldx + n);
      const bf16* h = reinterpret_cast<const bf16*>(&raw);
      x[k] = make_float4(__bfloat162float(h[0]), __bfloat162float(h[1]), __bfloat162float(h[2]), __bfloat162float(h[3]));
    }
  }
  const int m_begin = (int)((int64_t)a.M * blockIdx.y / gridDim.y), m_end = (int)((int64_t)a.M * (blockIdx.y + 1) / gridDim.y);
  for (int c0 = m_begin; c0 < m_end; c0 += RU_CHUNK) {
    const int rows = min(RU_CHUNK, m_end - c0);
    __syncthreads();
    for (int t = threadIdx.x; t < RU_CHUNK * KMAX; t += blockDim.x) {
      const int k = t / RU_CHUNK, r = t % RU_CHUNK;  // neighbouring threads read neighbouring columns of Y
      ys[r][k] = k < a.K && r < rows ? __bfloat162float(a.y[(int64_t)k * a.ldy + c0 + r]) : 0.f;
    }
    __syncthreads();
    if (!live) continue;
    float* gp = a.g + (int64_t)c0 * a.ldg + n;
#pragma unroll 4
    for (int r = 0; r < rows; ++r) {
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < KMAX; k += 4) {
        const float4 y4 = *reinterpret_cast<const float4*>(&ys[r][k]);
        const float y[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          t.x = fmaf(y[e], x[k + e].x, t.x); t.y = fmaf(y[e], x[k + e].y, t.y);
          t.z = fmaf(y[e], x[k + e].z, t.z); t.w = fmaf(y[e], x[k + e].w, t.w);
        }
      }
      ptx::red_add_v4(gp + (int64_t)r * a.ldg, t.x, t.y, t.z, t.w);
    }
  }
}

bool al(const void* p, int bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

}  // namespace

bool rows_fwd_serves(const RowsFwd& a) {
  return a.B <= ROWS_MAX && a.in % 64 == 0 && a.in <= 3072 && a.out % 8 == 0 && al(a.x, 16) && al(a.w, 16) &&
         al(a.bias, 4) && al(a.c, 8) && al(a.x_act, 8);
}

int launch_rows_fwd(const RowsFwd& a, cudaStream_t s) {
  const int smem = 16 * (a.in * 2 + 64);
  constexpr int most = 16 * (3072 * 2 + 64);
  static OncePerDevice once1, once4;
  JAGG_CUDA_TRY(allow_smem(once1, rows_fwd_kernel<1>, most));
  JAGG_CUDA_TRY(allow_smem(once4, rows_fwd_kernel<4>, most));
  const int nsm = sm_count(), groups = a.out / 8;
  const int tok = prof_start(s);
  if (groups < 8 * nsm) {  // four warps per 8 rows
    // all 16 warps even where fewer teams find rows: they stage act(X)
    JAGG_CUDA_TRY(launch(rows_fwd_kernel<4>, groups < nsm ? groups : nsm, 32 * RF_MAX_WARPS, smem, s, a));
  } else {  // the number of warps (10 to 16) that leaves the last round fullest
    int warps = RF_MAX_WARPS;
    double best = 0.0;
    for (int w = RF_MAX_WARPS; w >= 10; w -= 2) {
      const double rounds = (double)groups / ((double)nsm * w);
      const double fill = rounds / ceil_div(groups, (int64_t)nsm * w);
      if (fill > best + 0.02) {
        best = fill;
        warps = w;
      }
    }
    JAGG_CUDA_TRY(launch(rows_fwd_kernel<1>, nsm, 32 * warps, smem, s, a));
  }
  JAGG_LAUNCHED();
  prof_stop(tok, s, PROF_GEMM_TC, 2.0 * a.B * a.out * (double)a.in,
            2.0 * a.out * (double)a.in + 4.0 * a.B * a.in + 4.0 * a.B * a.out, a.B, a.out, a.in);
  return JAGG_OK;
}

bool rank_update_serves(const GemmArgs& g) {
  return g.epi == EPI_ACCUM && g.a_mn && g.b_mn && g.K <= ROWS_MAX && g.tile_n == 0 && g.split_k == 0 && !g.c_trans &&
         !g.remap_rows && g.a_dtype == JAGG_DTYPE_BF16 && g.b_dtype == JAGG_DTYPE_BF16 && g.N % 4 == 0 &&
         g.ldc % 4 == 0 && al(g.C, 16) && g.ldb % 4 == 0 && al(g.B, 8) && g.M >= 64;
}

int rank_update(const GemmArgs& g, cudaStream_t s) {
  const RankUpdate a{g.M, g.N, g.K, static_cast<const bf16*>(g.A), g.lda, static_cast<const bf16*>(g.B), g.ldb,
                     static_cast<float*>(g.C), g.ldc};
  const int threads = g.N / 4 < RU_THREADS ? (g.N / 4 + 31) / 32 * 32 : RU_THREADS;
  const int gx = ceil_div(g.N, 4 * threads);
  // about 8 CTAs per SM, at least 16 rows each
  int gy = ceil_div((int64_t)8 * sm_count(), gx);
  const int most = ceil_div(g.M, 16);
  gy = gy < most ? gy : most;
  const int tok = prof_start(s);
  auto kernel = g.K <= 4 ? rank_update_kernel<4> : g.K <= 8 ? rank_update_kernel<8> : rank_update_kernel<16>;
  JAGG_CUDA_TRY(launch(kernel, dim3(gx, gy), threads, 0, s, a));
  JAGG_LAUNCHED();
  prof_stop(tok, s, PROF_GEMM_TC, 2.0 * g.M * g.N * (double)g.K, 8.0 * g.M * (double)g.N, g.M, g.N, g.K);
  return JAGG_OK;
}

}  // namespace jagg
