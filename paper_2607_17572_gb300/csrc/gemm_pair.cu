// Dense products in tiles of 256 rows x up to 256 columns on CTA pairs (tcgen05.mma.cta_group::2).
//
// Bound by the tensor pipe on long products.  Rates in isolation, before (one CTA per 128 x 256
// tile, four or eight epilogue warps) and now, of 1923 TFLOP/s (cuBLAS): 18432 x 9216 x 3072 stored
// in bf16 1665 -> 1931, 18432 x 12288 x 3072 with GELU and its derivative 1487 -> 1840, times a
// multiplier 1530 -> 1889, 18432 x 3072 x 12288 in f32 1737 -> 1855, gated residual 1587 -> 1795,
// weight gradients of 18432 rows 1667-1735 -> 1847-1864.  Short K is bound by the epilogue: 21312 x
// 3072 x 768 with GELU 837 -> 1110, 21312 x 768 x 768 with the gated residual 368 -> 500.
//
// A cluster of two CTAs (the two SMs of a TPC) owns one tile: each CTA stages its 128 rows of A
// and its half of the columns of B, so at 256 columns a k-block of 64 moves 32 KB into each SM where
// a CTA on its own moves 48 KB for a 128 x 256 tile, and the tensor core reads 64 instead of 96
// bytes of shared memory per clock.  The leader's MMA thread issues for both; every CTA drains
// the 128 rows of the accumulator that its tensor memory holds (two 256-column accumulators:
// the next tile's products run while the epilogue works).
//
// Roles per CTA: warp 0 TMA producer (its halves, completing on the leader's barrier), warp 1
// the MMA issuer (leader only), warps 2-9 the epilogue: two warps per tensor-memory lane
// quarter on alternate column chunks, thread = output row, results through a swizzled
// shared-memory box into TMA stores (or f32 reduce-adds).  The inputs of the fused epilogues
// (the multiplier, the residual stream) arrive in the same boxes by TMA, requested before the
// accumulator is ready, and are overwritten in place by the result.
#include <cuda.h>

#include "gemm.cuh"
#include "ptx.cuh"
#include "tmap.cuh"

namespace jagg {

int unit_status_gemm_pair(unsigned* v, int clear) { return read_unit_status(v, clear); }

namespace {

enum PairEpi : int { PE_STORE_BF16 = 0, PE_STORE_F32, PE_ACCUM, PE_MUL, PE_GELU, PE_GATE };

constexpr int PT = 256;       // tile rows, and the most columns
constexpr int PK = 64;        // k-block
constexpr int P_EW = 8;       // epilogue warps
constexpr int P_THREADS = 64 + 32 * P_EW;
constexpr int P_HALF = 128 * PK * 2;      // bytes of a CTA's half of an operand tile
constexpr int P_SMEM = 232448 - 512;      // dynamic shared memory of a block
constexpr int P_FIXED = 1024 /*align*/ + 512 /*barriers*/;
constexpr int P_MAX_STAGES = 8;

template <int EPI>
struct PairCfg {
  // Staging boxes of 32 rows x 32 columns per epilogue warp: 8 KB where inputs or a second output
  // share them, 4 KB otherwise.  The rest of shared memory is operand stages, as many as fit at
  // the launch's tile width: five or six of 256 columns, six to eight of 128.  With four at 256
  // columns the products are 7 % slower (18432 x 3072 x 12288: 805 us against 748), since the
  // loads of 4 x 0.27 us of tensor work no longer cover the L2 latency under load.  At 128 columns six
  // stages cover less time, and a product of fewer units than pairs has nothing else to do: stages as
  // narrow as the tile took the pass over 5 x 245 rows (d = 768) from 2351 to 2306 us, the
  // forward of 8 x 333 rows from 1028 to 1018; wider tiles keep the ring they had.
  static constexpr bool OUT_BF16 = EPI == PE_STORE_BF16 || EPI == PE_MUL || EPI == PE_GELU;
  static constexpr int BOX = OUT_BF16 ? 2048 : 4096;
  static constexpr int BOXES = EPI == PE_STORE_BF16 ? 2 : EPI <= PE_ACCUM ? 1 : EPI == PE_GATE ? 2 : 4;
  static constexpr int WARP_BYTES = BOXES * BOX;
  static constexpr int EPI_BYTES = P_EW * WARP_BYTES;
  static_assert((2 * P_MAX_STAGES + 6 + BOXES * P_EW) * 8 + 4 <= 512, "barriers");
};

struct PairParams {
  int M, N;
  int bn;               // tile columns: a multiple of 32 from 128 to 256
  int tiles_m, tiles_n, splits, k_blocks;
  const bf16* bias;     // [N] or null
  const float* gate;    // PE_GATE
  int64_t gate_stride;
  int rows_per_seq;
  int gelu_d;           // PE_GELU: also write GELU'(u)
  float* col_sum;       // PE_MUL: column sums of the output, added, or null
  bf16* y;              // PE_GATE: the branch output before the gate, row pitch ldy
  int64_t ldy;
};

// Tensor maps: operands, C (GELU: GELU'(u)), x (PE_MUL: the multiplier; GELU: GELU(u);
// gate: the residual input), c2 (gate: the residual output).
struct PairMaps {
  CUtensorMap a, b, c, x, c2;
};

// One or two products of the same operand layout and epilogue in one launch (the text and image
// streams of a dual-stream block): the units of the second follow those of the first, so the
// small product fills the last wave of the large one instead of a wave of its own.
struct PairGroup {
  PairMaps maps[2];
  PairParams p[2];
  int total0, total;  // units of the first product, and of both
  int stages, stage_bytes;  // the operand ring: a stage holds 128 rows of A and half of the widest tile's columns of B
};

// Tiles walk groups of P_GROUP row tiles, the row tile fastest inside a group: the 76 pairs at work
// at one time cover P_GROUP x 4 tiles, so an operand panel is read from DRAM once for all of
// them.  Measured on the whole Flux-1024 forward: 42.4 ms with 4, 41.8 with 8, 41.2 with 12, 41.1
// with 19 (the rows of activations are the longer operand).
constexpr int P_GROUP = 19;
__device__ __forceinline__ void pair_decode(const PairGroup& g, int t, int& pr, int& tm, int& tn, int& ks) {
  pr = t < g.total0 ? 0 : 1;
  if (pr) t -= g.total0;
  const PairParams& p = g.p[pr];
  const int per_split = p.tiles_m * p.tiles_n;
  ks = t / per_split;
  t -= ks * per_split;
  const int per_group = P_GROUP * p.tiles_n;
  const int grp = t / per_group, in = t - grp * per_group;
  const int gm = min(P_GROUP, p.tiles_m - grp * P_GROUP);
  tm = grp * P_GROUP + in % gm;
  tn = in / gm;
}

// GELU'(u) and GELU(u) of two values (tanh from the hardware approximation, paired f32 forms).
__device__ __forceinline__ void gelu2(float2 u, float2& g, float2& dg) {
  const float c = 0.7978845608028654f, a = 0.044715f;
  auto both = [](float v) { return make_float2(v, v); };
  const float2 u2 = ptx::mul2(u, u);
  const float2 in = ptx::mul2(u, ptx::fma2(u2, both(c * a), both(c)));
  float2 t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t.x) : "f"(in.x));
  asm("tanh.approx.f32 %0, %1;" : "=f"(t.y) : "f"(in.y));
  const float2 h = ptx::mul2(u, both(0.5f));
  g = ptx::fma2(h, t, h);
  // h (1 - t^2) first: it is 0 where t has reached +-1, while h times the polynomial overflows from |u| = 1.4e13 on
  const float2 ho = ptx::mul2(h, ptx::fma2(ptx::mul2(t, both(-1.f)), t, both(1.f)));
  dg = ptx::fma2(ho, ptx::fma2(u2, both(3.f * a * c), both(c)), ptx::fma2(t, both(0.5f), both(0.5f)));
}
__device__ __forceinline__ uint32_t pack2(float x, float y) {
  __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<uint32_t*>(&v);
}
__device__ __forceinline__ float2 unpack2(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

template <bool A_MN, bool B_MN, int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(P_THREADS, 1)
    gemm_pair_kernel(const __grid_constant__ PairGroup g) {
  using Cfg = PairCfg<EPI>;
  const int stages = g.stages, ring_stage = g.stage_bytes;
  extern __shared__ uint8_t smem_pair[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_pair) + 1023) & ~uintptr_t(1023));
  uint8_t* epi_smem = smem + stages * ring_stage;
  uint64_t* full = reinterpret_cast<uint64_t*>(epi_smem + Cfg::EPI_BYTES);  // leader's: a stage landed in both CTAs
  uint64_t* empty = full + P_MAX_STAGES;     // per CTA: the products reading the stage are done
  uint64_t* tfull = empty + P_MAX_STAGES;    // [2] per CTA: an accumulator is complete
  uint64_t* tempty = tfull + 2;        // [2] leader's: both CTAs' epilogue warps have drained it
  uint64_t* auxbar = tempty + 2;       // [BOXES per epilogue warp] an epilogue input box landed
  uint64_t* drainbar = auxbar + Cfg::BOXES * P_EW;
  uint64_t* never = drainbar + 1;      // nothing arrives here: a bounded sleep after a give-up
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], 2 * P_EW);
    }
    for (int q = 0; q < Cfg::BOXES * P_EW; ++q) ptx::mbar_init(&auxbar[q], 1);
    ptx::mbar_init(drainbar, 1);
    ptx::mbar_init(never, 1);
    ptx::fence_mbar_init();
    for (int pr = 0; pr < (g.total > g.total0 ? 2 : 1); ++pr) {
      ptx::prefetch_tmap(&g.maps[pr].a);
      ptx::prefetch_tmap(&g.maps[pr].b);
      if (EPI != PE_GATE) ptx::prefetch_tmap(&g.maps[pr].c);
      if (EPI >= PE_MUL) ptx::prefetch_tmap(&g.maps[pr].x);
      if (EPI == PE_GATE) ptx::prefetch_tmap(&g.maps[pr].c2);
    }
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(tmem_slot, 512);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();  // the peer's barriers are initialised
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();

  const int total = g.total;
  const int npairs = gridDim.x >> 1;
  auto krange = [&](int pr, int ks, int& kb0, int& kb1) {
    const PairParams& p = g.p[pr];
    kb0 = (int)((long long)p.k_blocks * ks / p.splits);
    kb1 = (int)((long long)p.k_blocks * (ks + 1) / p.splits);
  };

  if (warp == 0) {
    if (ptx::elect_one()) {
      // ---------------- TMA producer: this CTA's halves of A and B
      int stage = 0;
      uint8_t* sA = smem;
      uint32_t phase = 0;
      uint32_t issued = 0, issued_parity = 0;
      for (int t = blockIdx.x >> 1; t < total && !abort_flag; t += npairs) {
        int pr, tm, tn, ks, kb0, kb1;
        pair_decode(g, t, pr, tm, tn, ks);
        krange(pr, ks, kb0, kb1);
        const PairMaps& maps = g.maps[pr];
        const int half_n = g.p[pr].bn >> 1;  // this CTA's columns of B
        const int ma = tm * PT + (int)rank * 128, nb = tn * g.p[pr].bn + (int)rank * half_n;
        // an MN-major B arrives in whole 64-column chunks (of the last, half_n % 64 are used)
        const bool two_chunks = half_n > 64;
        const uint32_t stage_bytes = 2u * (P_HALF + (B_MN ? (two_chunks ? P_HALF : P_HALF / 2) : half_n * PK * 2));
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!ptx::mbar_wait(&empty[stage], phase ^ 1)) { abort_flag = 1; break; }
          uint8_t* sB = sA + P_HALF;
          if (rank == 0) ptx::mbar_arrive_expect_tx(&full[stage], stage_bytes);
          const uint32_t bar = ptx::mapa(ptx::smem_u32(&full[stage]), 0);
          if (!A_MN) {
            ptx::tma_load_2d_pair(sA, &maps.a, bar, kb * PK, ma);
          } else {
            ptx::tma_load_2d_pair(sA, &maps.a, bar, ma, kb * PK);
            ptx::tma_load_2d_pair(sA + P_HALF / 2, &maps.a, bar, ma + 64, kb * PK);
          }
          if (!B_MN) {
            ptx::tma_load_2d_pair(sB, &maps.b, bar, kb * PK, nb);
          } else {
            ptx::tma_load_2d_pair(sB, &maps.b, bar, nb, kb * PK);
            if (two_chunks) ptx::tma_load_2d_pair(sB + P_HALF / 2, &maps.b, bar, nb + 64, kb * PK);
          }
          issued |= 1u << stage;
          issued_parity = (issued_parity & ~(1u << stage)) | (phase << stage);
          sA += ring_stage;
          if (++stage == stages) { stage = 0; phase ^= 1; sA = smem; }
        }
      }
      // After a give-up, loads already issued may still be landing: the leader waits (bounded)
      // for the last phase of every stage, the peer, whose loads complete on the leader's
      // barriers, for the length of one bounded wait.
      if (abort_flag) {
        if (rank == 0) {
          for (int s = 0; s < stages; ++s)
            if (issued & (1u << s)) ptx::mbar_wait(&full[s], (issued_parity >> s) & 1u);
        } else if (issued) {
          ptx::mbar_wait(never, 0);
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && ptx::elect_one()) {
      // ---------------- MMA issuer for both CTAs
      int stage = 0, acc = 0;
      const uint32_t a_first = ptx::smem_u32(smem);
      uint32_t a_addr = a_first;
      uint32_t phase = 0, acc_phase = 0;
      for (int t = blockIdx.x >> 1; t < total && !abort_flag; t += npairs) {
        int pr, tm, tn, ks, kb0, kb1;
        pair_decode(g, t, pr, tm, tn, ks);
        krange(pr, ks, kb0, kb1);
        if (!ptx::mbar_wait(&tempty[acc], acc_phase ^ 1)) { abort_flag = 1; break; }
        ptx::tc_fence_after();
        const uint32_t d = tmem + acc * PT;
        const uint32_t idesc = ptx::idesc_bf16(PT, g.p[pr].bn, A_MN, B_MN);
        bool ok = true;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!ptx::mbar_wait(&full[stage], phase)) { ok = false; break; }
          ptx::tc_fence_after();
          const uint32_t b_addr = a_addr + P_HALF;
          // K-major: a step of 16 elements is 32 bytes inside the swizzled 128-byte row;
          // MN-major: two 1024-byte atoms.  (The start-address field counts 16 bytes and never
          // carries: every operand lies below 2^18 bytes.)
          const uint64_t ad = A_MN ? ptx::sdesc_sw128(a_addr, 64 * PK * 2, 1024) : ptx::sdesc_sw128(a_addr, 16, 1024);
          const uint64_t bd = B_MN ? ptx::sdesc_sw128(b_addr, 64 * PK * 2, 1024) : ptx::sdesc_sw128(b_addr, 16, 1024);
#pragma unroll
          for (int k = 0; k < PK / 16; ++k)
            ptx::umma_bf16_pair(d, ad + (uint64_t)(k * (A_MN ? 128 : 2)), bd + (uint64_t)(k * (B_MN ? 128 : 2)), idesc,
                                (kb > kb0 || k > 0) ? 1u : 0u);
          ptx::umma_commit_pair(&empty[stage]);
          a_addr += ring_stage;
          if (++stage == stages) { stage = 0; phase ^= 1; a_addr = a_first; }
        }
        if (!ok) { abort_flag = 1; break; }
        ptx::umma_commit_pair(&tfull[acc]);
        if (++acc == 2) { acc = 0; acc_phase ^= 1; }
      }
      if (abort_flag) {  // products may still be running: drain them before tensor memory is freed
        ptx::umma_commit_local(drainbar);
        ptx::mbar_wait(drainbar, 0);
      }
    }
  } else {
    // ---------------- epilogue: tensor-memory lanes 32 q .. + 31 (rows of this CTA's half)
    const int q = warp & 3, half = (warp - 2) >> 2, ew = warp - 2;
    uint8_t* box = epi_smem + ew * Cfg::WARP_BYTES;
    uint64_t* aux = auxbar + Cfg::BOXES * ew;
    const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16);
    // the 16-byte piece j of this lane's row in a box: 128-byte rows (f32) or 64-byte rows (bf16),
    // swizzled as the tensor maps say
    auto piece = [&](uint8_t* bx, int j) {
      return Cfg::OUT_BF16 ? bx + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4) : bx + lane * 128 + ((j ^ (lane & 7)) << 4);
    };
    int acc = 0, sb = 0;  // sb: the box of the next store (epilogues without an input)
    uint32_t acc_phase = 0, aux_phase = 0;  // aux_phase bit b: the phase box b's barrier waits for next
    for (int t = blockIdx.x >> 1; t < total; t += npairs) {
      int pr, tm, tn, ks;
      pair_decode(g, t, pr, tm, tn, ks);
      const PairParams& p = g.p[pr];
      const PairMaps& maps = g.maps[pr];
      const int m0 = tm * PT + (int)rank * 128 + q * 32;
      const bool rows_live = m0 < p.M;
      auto col = [&](int i) { return tn * p.bn + (half + 2 * i) * 32; };
      const float* gate_row = nullptr;
      if constexpr (EPI == PE_GATE)
        gate_row = p.gate + (int64_t)(min(m0 + lane, p.M - 1) / p.rows_per_seq) * p.gate_stride;
      int live = 0;  // chunks with columns inside the output
      if (rows_live)
        for (int i = 0; (half + 2 * i) * 32 < p.bn; ++i) live += col(i) < p.N ? 1 : 0;
      // PE_MUL, PE_GATE: the first BOXES chunks' inputs, before the accumulator is waited for
      auto load_aux = [&](int i) {
        const int b = i % Cfg::BOXES;
        ptx::mbar_arrive_expect_tx(&aux[b], Cfg::BOX);
        ptx::tma_load_2d(box + b * Cfg::BOX, &maps.x, &aux[b], col(i), m0);
      };
      int loaded = 0;  // chunks whose input has been requested
      if constexpr (EPI == PE_MUL || EPI == PE_GATE) {
        loaded = live < Cfg::BOXES ? live : Cfg::BOXES;
        if (lane == 0) {
          ptx::bulk_wait_read<0>();  // the boxes' last stores have read them
          for (int i = 0; i < loaded; ++i) load_aux(i);
        }
      }
      bool ok = ptx::mbar_wait(&tfull[acc], acc_phase);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) {
        if constexpr (EPI == PE_MUL || EPI == PE_GATE)
          for (int i = 0; i < loaded; ++i) ptx::mbar_wait(&aux[i], (aux_phase >> i) & 1u);
        abort_flag = 1;
        break;
      }
      ptx::tc_fence_after();
#pragma unroll 1
      for (int i = 0; i < live; ++i) {
        const int n0 = col(i);
        // the chunk's box; PE_GELU: the box of GELU(u), that of GELU'(u) after it
        const int sl = EPI == PE_MUL || EPI == PE_GATE ? i % Cfg::BOXES : sb;
        uint8_t* slot = box + sl * Cfg::BOX;
        constexpr bool BIAS = EPI == PE_STORE_BF16 || EPI == PE_GELU || EPI == PE_GATE;
        uint4 bq[BIAS ? 4 : 1];  // the chunk's bias
        if constexpr (BIAS) {
          if (p.bias) {
#pragma unroll
            for (int j = 0; j < 4; ++j) bq[j] = *reinterpret_cast<const uint4*>(p.bias + n0 + 8 * j);
          }
        }
        uint32_t r[32];
        ptx::tmem_ld_32x32b_x32(trow + acc * PT + (half + 2 * i) * 32, r);
        float4 gq[EPI == PE_GATE ? 8 : 1];  // the gate of this lane's row
        if constexpr (EPI == PE_GATE) {
          // the next input first: into the previous chunk's box, once its store has read it
          if (i > 0 && loaded < live) {
            if (lane == 0) {
              ptx::bulk_wait_read<0>();
              load_aux(loaded);
            }
            ++loaded;
          }
          const float4* gp = reinterpret_cast<const float4*>(gate_row + n0);
#pragma unroll
          for (int j = 0; j < 8; ++j) gq[j] = gp[j];
        }
        if constexpr (EPI == PE_MUL || EPI == PE_GATE) {
          const bool got = __all_sync(0xffffffffu, ptx::mbar_wait(&aux[sl], (aux_phase >> sl) & 1u));
          aux_phase ^= 1u << sl;
          if (!got) {  // later chunks' inputs may be in flight
            for (int n = i + 1; n < loaded; ++n)
              ptx::mbar_wait(&aux[n % Cfg::BOXES], (aux_phase >> (n % Cfg::BOXES)) & 1u);
            ok = false;
            break;
          }
        } else {
          if (lane == 0) {  // the box's previous store has read it
            if constexpr (Cfg::BOXES == 1)
              ptx::bulk_wait_read<0>();
            else
              ptx::bulk_wait_read<1>();
          }
          __syncwarp();
        }
        ptx::tmem_ld_wait();
        auto add_bias = [&](int j) {  // to columns 8 j .. + 7
          if (!p.bias) return;
          const uint32_t w[4] = {bq[j].x, bq[j].y, bq[j].z, bq[j].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 v = ptx::add2(make_float2(__uint_as_float(r[8 * j + 2 * e]), __uint_as_float(r[8 * j + 2 * e + 1])),
                                       unpack2(w[e]));
            r[8 * j + 2 * e] = __float_as_uint(v.x);
            r[8 * j + 2 * e + 1] = __float_as_uint(v.y);
          }
        };
        auto f2 = [&](int c) { return make_float2(__uint_as_float(r[c]), __uint_as_float(r[c + 1])); };
        if constexpr (EPI == PE_STORE_BF16) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            add_bias(j);
            uint32_t o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = pack2(f2(8 * j + 2 * e).x, f2(8 * j + 2 * e).y);
            *reinterpret_cast<uint4*>(piece(slot, j)) = make_uint4(o[0], o[1], o[2], o[3]);
          }
        } else if constexpr (EPI == PE_STORE_F32 || EPI == PE_ACCUM) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            *reinterpret_cast<uint4*>(piece(slot, j)) = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        } else if constexpr (EPI == PE_MUL) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint4* at = reinterpret_cast<uint4*>(piece(slot, j));
            const uint4 x = *at;
            const uint32_t w[4] = {x.x, x.y, x.z, x.w};
            uint32_t o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 v = ptx::mul2(f2(8 * j + 2 * e), unpack2(w[e]));
              o[e] = pack2(v.x, v.y);
            }
            *at = make_uint4(o[0], o[1], o[2], o[3]);
          }
        } else if constexpr (EPI == PE_GELU) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            add_bias(j);
            uint32_t og[4], od[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float2 gl, dg;
              gelu2(f2(8 * j + 2 * e), gl, dg);
              og[e] = pack2(gl.x, gl.y);
              od[e] = pack2(dg.x, dg.y);
            }
            *reinterpret_cast<uint4*>(piece(slot, j)) = make_uint4(og[0], og[1], og[2], og[3]);
            if (p.gelu_d) *reinterpret_cast<uint4*>(piece(slot + Cfg::BOX, j)) = make_uint4(od[0], od[1], od[2], od[3]);
          }
        } else {  // PE_GATE: y straight to global memory (64 bytes of this lane's row), the residual in place
          bf16* yp = m0 + lane < p.M ? p.y + (int64_t)(m0 + lane) * p.ldy + n0 : nullptr;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float gv[8] = {gq[2 * j].x, gq[2 * j].y, gq[2 * j].z, gq[2 * j].w,
                                 gq[2 * j + 1].x, gq[2 * j + 1].y, gq[2 * j + 1].z, gq[2 * j + 1].w};
            add_bias(j);
            uint32_t y[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) y[e] = pack2(f2(8 * j + 2 * e).x, f2(8 * j + 2 * e).y);
            if (yp) *reinterpret_cast<uint4*>(yp + 8 * j) = make_uint4(y[0], y[1], y[2], y[3]);
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
              float4* at = reinterpret_cast<float4*>(piece(slot, 2 * j + hh));
              float4 h = *at;
              h.x = fmaf(gv[4 * hh], __uint_as_float(r[8 * j + 4 * hh]), h.x);
              h.y = fmaf(gv[4 * hh + 1], __uint_as_float(r[8 * j + 4 * hh + 1]), h.y);
              h.z = fmaf(gv[4 * hh + 2], __uint_as_float(r[8 * j + 4 * hh + 2]), h.z);
              h.w = fmaf(gv[4 * hh + 3], __uint_as_float(r[8 * j + 4 * hh + 3]), h.w);
              *at = h;
            }
          }
        }
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if constexpr (EPI == PE_ACCUM) {
            ptx::tma_reduce_add_2d(&maps.c, slot, n0, m0);
          } else if constexpr (EPI == PE_GELU) {
            ptx::tma_store_2d(&maps.x, slot, n0, m0);
            if (p.gelu_d) ptx::tma_store_2d(&maps.c, slot + Cfg::BOX, n0, m0);
          } else if constexpr (EPI == PE_GATE) {
            ptx::tma_store_2d(&maps.c2, slot, n0, m0);
          } else {
            ptx::tma_store_2d(&maps.c, slot, n0, m0);
          }
          ptx::bulk_commit();
        }
        if constexpr (EPI == PE_MUL) {
          // column sums of the box just written (rows past M are zeros): a lane sums a column pair over
          // every other row, so a step of the warp reads two whole rows
          if (p.col_sum) {
            const int cp = lane & 15, odd = lane >> 4;
            float2 sum = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const int rr = 2 * k + odd;
              sum = ptx::add2(sum, unpack2(*reinterpret_cast<const uint32_t*>(
                                       slot + rr * 64 + (((cp >> 2) ^ (k & 3)) << 4) + (cp & 3) * 4)));
            }
            sum.x += __shfl_xor_sync(0xffffffffu, sum.x, 16);
            sum.y += __shfl_xor_sync(0xffffffffu, sum.y, 16);
            if (!odd && n0 + 2 * cp < p.N) ptx::red_add_v2(p.col_sum + n0 + 2 * cp, sum.x, sum.y);
          }
        }
        sb = (sb + (EPI == PE_GELU ? 2 : 1)) % Cfg::BOXES;
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(ptx::mapa(ptx::smem_u32(&tempty[acc]), 0));
      if (!ok) { abort_flag = 1; break; }
      if (++acc == 2) { acc = 0; acc_phase ^= 1; }
    }
    pdl_trigger();  // only the stores in flight are left: the next kernel's small CTAs may come
    if (lane == 0) ptx::bulk_wait<0>();
    __syncwarp();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();  // neither CTA's shared or tensor memory is in use by the other any more
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem, 512);
  }
}

// ------------------------------------------------------------------ host side
bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

int map2d(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_cols, int box_rows, bool f32,
          CUtensorMapSwizzle swz) {
  const uint64_t dims[2] = {(uint64_t)cols, (uint64_t)rows};
  const uint64_t strides[1] = {(uint64_t)ld * (f32 ? 4 : 2)};
  const uint32_t box[2] = {(uint32_t)box_cols, (uint32_t)box_rows};
  return encode_tmap(m, f32, 2, base, dims, strides, box, swz);
}

// The epilogue that serves the product, or -1: row-major outputs, 16-byte aligned operands and
// pitches, and whole 64-column chunks where a bias or gate vector is read.
int pair_epi(const GemmArgs& g) {
  if (g.c_trans || g.bias_m || g.remap_rows || (g.C && !al16(g.C))) return -1;
  const bool c_f32 = g.c_dtype == JAGG_DTYPE_F32;
  if (g.C && (g.ldc * (c_f32 ? 4 : 2)) % 16) return -1;
  if (g.bias && (g.bias_dtype != JAGG_DTYPE_BF16 || !al16(g.bias) || g.N % 64)) return -1;
  switch (g.epi) {
    case EPI_STORE:
      if (!c_f32) return PE_STORE_BF16;
      return g.bias ? -1 : PE_STORE_F32;
    case EPI_ACCUM:
      return c_f32 ? PE_ACCUM : -1;
    case EPI_MUL_AUX:
      return !c_f32 && al16(g.aux) && g.ld_aux % 8 == 0 && (!g.col_sum || (al16(g.col_sum) && g.N % 2 == 0)) ? PE_MUL
                                                                                                             : -1;
    case EPI_GELU:
      return !c_f32 && g.C2 && al16(g.C2) && g.ldc2 % 8 == 0 ? PE_GELU : -1;
    case EPI_GATE_RESID:
      return !c_f32 && g.C && g.C2 && al16(g.C2) && g.ldc2 % 4 == 0 && al16(g.aux) && g.ld_aux % 4 == 0 &&
                     al16(g.gate) && g.gate_stride % 4 == 0 && g.N % 64 == 0
                 ? PE_GATE
                 : -1;
  }
  return -1;
}

template <bool A_MN, bool B_MN, int EPI>
int fill_pair(const GemmArgs& g, int bn, int splits, PairMaps& maps, PairParams& p) {
  const auto swz = CU_TENSOR_MAP_SWIZZLE_128B, swz_bf16 = CU_TENSOR_MAP_SWIZZLE_64B;
  JAGG_TRY(A_MN ? map2d(&maps.a, g.A, g.K, g.M, g.lda, 64, PK, false, swz)
                : map2d(&maps.a, g.A, g.M, g.K, g.lda, PK, 128, false, swz));
  JAGG_TRY(B_MN ? map2d(&maps.b, g.B, g.K, g.N, g.ldb, 64, PK, false, swz)
                : map2d(&maps.b, g.B, g.N, g.K, g.ldb, PK, bn / 2, false, swz));
  maps.c = maps.x = maps.c2 = maps.a;  // unused ones
  if (EPI == PE_STORE_BF16 || EPI == PE_MUL || (EPI == PE_GELU && g.C))
    JAGG_TRY(map2d(&maps.c, g.C, g.M, g.N, g.ldc, 32, 32, false, swz_bf16));
  if (EPI == PE_STORE_F32 || EPI == PE_ACCUM) JAGG_TRY(map2d(&maps.c, g.C, g.M, g.N, g.ldc, 32, 32, true, swz));
  if (EPI == PE_MUL) JAGG_TRY(map2d(&maps.x, g.aux, g.M, g.N, g.ld_aux, 32, 32, false, swz_bf16));
  if (EPI == PE_GELU) JAGG_TRY(map2d(&maps.x, g.C2, g.M, g.N, g.ldc2, 32, 32, false, swz_bf16));
  if (EPI == PE_GATE) {
    JAGG_TRY(map2d(&maps.x, g.aux, g.M, g.N, g.ld_aux, 32, 32, true, swz));
    JAGG_TRY(map2d(&maps.c2, g.C2, g.M, g.N, g.ldc2, 32, 32, true, swz));
  }
  p.M = g.M; p.N = g.N;
  p.tiles_m = ceil_div(g.M, PT);
  p.bn = bn;
  p.tiles_n = ceil_div(g.N, bn);
  p.splits = splits;
  p.k_blocks = ceil_div(g.K, PK);
  p.bias = static_cast<const bf16*>(g.bias);
  p.gate = g.gate;
  p.gate_stride = g.gate_stride;
  p.rows_per_seq = g.rows_per_seq > 0 ? g.rows_per_seq : 1;
  p.gelu_d = EPI == PE_GELU && g.C ? 1 : 0;
  p.col_sum = g.col_sum;
  p.y = static_cast<bf16*>(g.C);
  p.ldy = g.ldc;
  return JAGG_OK;
}

// Tile columns and K splits of one product.
struct PairPlan {
  int bn, splits;
};

// The product `a` and, when given, `b` of the same layout and epilogue.
template <bool A_MN, bool B_MN, int EPI>
int launch_pair(const GemmArgs& a, const GemmArgs* b, const PairPlan (&plan)[2], int npairs, cudaStream_t s) {
  using Cfg = PairCfg<EPI>;
  PairGroup grp;
  JAGG_TRY((fill_pair<A_MN, B_MN, EPI>(a, plan[0].bn, plan[0].splits, grp.maps[0], grp.p[0])));
  if (b) {
    JAGG_TRY((fill_pair<A_MN, B_MN, EPI>(*b, plan[1].bn, plan[1].splits, grp.maps[1], grp.p[1])));
  } else {
    grp.maps[1] = grp.maps[0];
    grp.p[1] = grp.p[0];
  }
  auto units = [](const PairParams& p) { return p.tiles_m * p.tiles_n * p.splits; };
  grp.total0 = units(grp.p[0]);
  grp.total = grp.total0 + (b ? units(grp.p[1]) : 0);
  // B arrives K-major in bn / 2 rows of 128 bytes, MN-major in whole chunks of 64 columns
  const int bn = b && plan[1].bn > plan[0].bn ? plan[1].bn : plan[0].bn;
  grp.stage_bytes = P_HALF + (B_MN ? (bn > 128 ? P_HALF : P_HALF / 2) : bn / 2 * PK * 2);
  const int fit = (P_SMEM - P_FIXED - Cfg::EPI_BYTES) / grp.stage_bytes;
  grp.stages = fit < P_MAX_STAGES ? fit : P_MAX_STAGES;
  const int smem = grp.stages * grp.stage_bytes + Cfg::EPI_BYTES + P_FIXED;
  auto kernel = gemm_pair_kernel<A_MN, B_MN, EPI>;
  static OncePerDevice once;
  JAGG_CUDA_TRY(allow_smem(once, kernel, P_SMEM));
  const int tok = prof_start(s);
  JAGG_CUDA_TRY(launch(kernel, 2 * (grp.total < npairs ? grp.total : npairs), P_THREADS, smem, s, grp));
  JAGG_LAUNCHED();
  double flops = 0.0, bytes = 0.0;
  for (const GemmArgs* g : {&a, b}) {
    if (!g) continue;
    flops += 2.0 * g->M * g->N * g->K;
    bytes += 2.0 * ((double)g->M * g->K + (double)g->N * g->K) + (double)g->M * g->N * (g->c_dtype == JAGG_DTYPE_F32 ? 4 : 2);
  }
  // a group's M (or, for weight gradients, K) is the sum over its products
  const bool sum_k = A_MN && b;
  prof_stop(tok, s, PROF_GEMM_TC, flops, bytes, a.M + (b && !sum_k ? b->M : 0), a.N, a.K + (sum_k ? b->K : 0));
  return JAGG_OK;
}

// The estimate behind the choice of tiles, in k-blocks of a 256-column tile.  A unit (a tile, or
// one K split of it) costs its k-blocks times bn / 256, a little more for narrower tiles (whose
// operand traffic per FLOP is larger), plus P_UNIT_OVERHEAD for its pipeline fill and epilogue;
// units go round-robin to the pairs, so a product takes the units of the pair that gets most.
// Narrower tiles pay where 256 columns would leave the last wave nearly empty: 4096 x 3072 x 12288 in f32 takes
// 180 us at 256 columns (192 units on 76 pairs) and 171 at 224; 633 x 3072 x 3072 19.4 -> 13.1,
// 1225 x 768 x 3072 20.7 -> 12.7, 2664 x 2304 x 768 13.6 -> 12.5.
constexpr double P_UNIT_OVERHEAD = 5.0;
constexpr int P_WIDTHS[] = {256, 224, 192, 160, 128};
constexpr double P_LAUNCH = 12.0;
constexpr double P_WIDTH_COST[] = {1.0, 1.05, 1.07, 1.10, 1.15};

struct PairUnits {
  long long n;
  double cost;
};
PairUnits pair_units(const GemmArgs& g, int w, int splits) {
  const int bn = P_WIDTHS[w];
  return {(long long)ceil_div(g.M, PT) * ceil_div(g.N, bn) * splits,
          ceil_div(ceil_div(g.K, PK), splits) * P_WIDTH_COST[w] * bn / 256.0 + P_UNIT_OVERHEAD};
}
// Duration of a's units followed by b's, dealt round-robin to np pairs.
double pair_time(PairUnits a, PairUnits b, int np) {
  const long long qa = a.n / np, ra = a.n % np, qb = b.n / np, rb = b.n % np;
  // pairs before ra take one more unit of a; b's deal starts at pair ra
  const double early = ra ? (qa + 1) * a.cost + (qb + (rb > np - ra ? 1 : 0)) * b.cost : 0.0;
  const double late = qa * a.cost + (qb + (rb > 0 ? 1 : 0)) * b.cost;
  return early > late ? early : late;
}
int most_splits(const GemmArgs& g) {
  const int kb = ceil_div(g.K, PK);
  return g.epi != EPI_ACCUM ? 1 : kb < 32 ? kb : 32;
}
double pair_plan(const GemmArgs& g, int np, PairPlan* plan) {
  double best = 0.0;
  int lo = 1, hi = most_splits(g);
  if (g.epi == EPI_ACCUM && g.split_k > 0) lo = hi = g.split_k < ceil_div(g.K, PK) ? g.split_k : ceil_div(g.K, PK);
  for (int w = 0; w < 5; ++w)
    for (int s = lo; s <= hi; ++s) {
      const double c = pair_time(pair_units(g, w, s), {0, 0.0}, np);
      if (best == 0.0 || c < 0.999 * best) {
        best = c;
        *plan = {P_WIDTHS[w], s};
      }
    }
  return best;
}

// Whether the kernel has an instance for the product.
bool pair_instance(const GemmArgs& g) {
  if (g.tile_n != 0 || g.M <= 128 || g.N < 128 || (g.a_mn && !g.b_mn)) return false;
  const int epi = pair_epi(g);
  if (epi < 0) return false;
  if (g.a_mn) return epi == PE_ACCUM;
  return g.b_mn ? epi == PE_STORE_BF16 || epi == PE_STORE_F32 || epi == PE_MUL
                : epi == PE_STORE_BF16 || epi == PE_GELU || epi == PE_GATE;
}

int dispatch_pair(const GemmArgs& a, const GemmArgs* b, const PairPlan (&plan)[2], cudaStream_t s) {
  const int np = sm_count() / 2, epi = pair_epi(a);
  if (!a.a_mn && !a.b_mn) {
    if (epi == PE_STORE_BF16) return launch_pair<false, false, PE_STORE_BF16>(a, b, plan, np, s);
    if (epi == PE_GELU) return launch_pair<false, false, PE_GELU>(a, b, plan, np, s);
    if (epi == PE_GATE) return launch_pair<false, false, PE_GATE>(a, b, plan, np, s);
  } else if (!a.a_mn) {
    if (epi == PE_STORE_BF16) return launch_pair<false, true, PE_STORE_BF16>(a, b, plan, np, s);
    if (epi == PE_STORE_F32) return launch_pair<false, true, PE_STORE_F32>(a, b, plan, np, s);
    if (epi == PE_MUL) return launch_pair<false, true, PE_MUL>(a, b, plan, np, s);
  } else if (epi == PE_ACCUM) {
    return launch_pair<true, true, PE_ACCUM>(a, b, plan, np, s);
  }
  set_last_error("gemm: the pair kernel does not serve this product");
  return JAGG_ERR_UNSUPPORTED;
}

}  // namespace

bool gemm_pair_serves(const GemmArgs& g, double* cost) {
  if (!pair_instance(g)) return false;
  PairPlan plan;
  *cost = pair_plan(g, sm_count() / 2, &plan);
  return true;
}

int gemm_pair(const GemmArgs& g, cudaStream_t s) {
  PairPlan plan[2] = {};
  pair_plan(g, sm_count() / 2, &plan[0]);
  return dispatch_pair(g, nullptr, plan, s);
}

int gemm_pair_as(const GemmArgs& x, const GemmArgs* y, const int (&bn)[2], const int (&splits)[2], cudaStream_t s) {
  PairPlan plan[2] = {};
  for (int i = 0; i < (y ? 2 : 1); ++i) {
    const GemmArgs& g = i ? *y : x;
    JAGG_TRY(gemm_validate(g));
    JAGG_CHECK_ARG(gemm_tc_eligible(g) && pair_instance(g), "gemm: the pair kernel does not serve this product");
    pair_plan(g, sm_count() / 2, &plan[i]);
    if (!bn[i]) continue;
    JAGG_CHECK_ARG(bn[i] % 32 == 0 && bn[i] >= 128 && bn[i] <= PT, "gemm: pair tiles of %d columns", bn[i]);
    JAGG_CHECK_ARG(splits[i] >= 1 && splits[i] <= (g.epi == EPI_ACCUM ? ceil_div(g.K, PK) : 1), "gemm: %d K splits",
                   splits[i]);
    plan[i] = {bn[i], splits[i]};
  }
  JAGG_CHECK_ARG(!y || (x.a_mn == y->a_mn && x.b_mn == y->b_mn && pair_epi(x) == pair_epi(*y)),
                 "gemm: a grouped launch needs one layout and epilogue");
  return dispatch_pair(x, y, plan, s);
}

int gemm_two(const GemmArgs& x, const GemmArgs& y, cudaStream_t s) {
  const bool same = x.a_mn == y.a_mn && x.b_mn == y.b_mn && x.epi == y.epi && gemm_tc_eligible(x) &&
                    gemm_tc_eligible(y) && pair_instance(x) && pair_instance(y) && pair_epi(x) == pair_epi(y);
  if (same) {
    // the longer units first, so that the short ones even out the end
    const GemmArgs& a = x.K > y.K || (x.K == y.K && x.M >= y.M) ? x : y;
    const GemmArgs& b = &a == &x ? y : x;
    const int np = sm_count() / 2;
    PairPlan plan[2] = {};
    double best = 0.0;
    const int sa_max = most_splits(a) < 8 ? most_splits(a) : 8, sb_max = most_splits(b) < 4 ? most_splits(b) : 4;
    for (int wa = 0; wa < 5; ++wa)
      for (int sa = 1; sa <= sa_max; ++sa)
        for (int wb = 0; wb < 5; ++wb)
          for (int sb = 1; sb <= sb_max; ++sb) {
            const double c = pair_time(pair_units(a, wa, sa), pair_units(b, wb, sb), np);
            if (best == 0.0 || c < 0.999 * best) {
              best = c;
              plan[0] = {P_WIDTHS[wa], sa};
              plan[1] = {P_WIDTHS[wb], sb};
            }
          }
    // against two launches of their own (the second's ramp is about P_LAUNCH k-blocks)
    const double apart = gemm_best_cost(a) + gemm_best_cost(b) + P_LAUNCH;
    if (best < apart) return dispatch_pair(a, &b, plan, s);
  }
  JAGG_TRY(gemm(x, s));
  return gemm(y, s);
}

}  // namespace jagg
