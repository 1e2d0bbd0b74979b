// Products with a handful of rows (the t-embedding MLP and the stacked modulation).
#pragma once

#include "gemm.cuh"

namespace jagg {

constexpr int ROWS_MAX = 16;  // rows (sequences) these kernels serve

// c[B, out] = act(x)[B, in] W[out, in]^T + bias, act the identity or SiLU; act(x) rounded to bf16
// (the product's operand) is also stored to x_act.  W and bias bf16, x and c f32.
struct RowsFwd {
  int B, out, in, silu;
  const float* x;
  void* x_act;
  const void* w;
  const void* bias;
  float* c;
};
bool rows_fwd_serves(const RowsFwd& a);
int launch_rows_fwd(const RowsFwd& a, cudaStream_t s);

// g[M, N] += y[K, M]^T x[K, N], K <= ROWS_MAX.
struct RankUpdate {
  int M, N, K;
  const bf16* y;
  int64_t ldy;
  const bf16* x;
  int64_t ldx;
  float* g;
  int64_t ldg;
};
bool rank_update_serves(const GemmArgs& g);
int rank_update(const GemmArgs& g, cudaStream_t s);

}  // namespace jagg
