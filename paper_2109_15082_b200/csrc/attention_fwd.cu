// Fused attention forward for one (batch, head, 128-query block) per CTA on sm_100a:
//   S = Q K^T (tcgen05, fp32 accumulators in TMEM)  ->  masked softmax straight out of TMEM  ->  (student) Eq. 1 on the
//   probabilities  ->  ctx = P V with P taken from shared memory as the A operand of a second tcgen05 product.
// The scores never touch HBM.  Operands are the Q/K/V slices of the [tokens, 3*hidden] tensor
// (bf16 values for the teacher, integer codes held as bf16 for the student: every product of
// codes is exact in fp32), fetched by TMA with 128-byte swizzle.  Outputs: the probabilities
// (and their codes) for the backward pass, the context rows, and for the student the codes of
// the context (int8 for the next int8 product, bf16 for the backward).
// Head size 64, up to 128 tokens here (above: attention_fwd_long.cu).  All waits are time-bounded.
//
// What bounds it: one CTA is a serial chain (tiles by TMA, product, softmax, product, rows out) and the softmax arithmetic
// fills the issue slots only when several CTAs share an SM.  So P takes the place of Q and K in shared memory and the context that of
// the scores in TMEM, and with a thread per row, 48 KB and 128 TMEM columns four CTAs fit (two CTAs of two threads per row: 512
// CTAs were two rounds on 148 SMs and are one now).
// Keys beyond the valid length cost nothing: their chunks are neither multiplied nor exponentiated.  Instruction fetch counts too: everything runs
// once or a few times per CTA, so the loops over chunks stay rolled.
// 32 x 16 heads x 128 x 128: 20.6 -> 15 us (mean of teacher and student pass).  Since then maximum and sum in one pass over the scores and the
// context out by tiled stores instead of a row per lane: 32 x 12 heads 20.8 -> 15.1 us (student), 16.0 -> 14.1 (teacher); scalars of the context
// fetched behind the last product cost a step of 4 x 32 tokens 2 us.
#include "attention_fwd.cuh"

namespace mrem {

using namespace attf;

namespace {

// QUANT: the student pass (quantizers of the probabilities and of the context).
// Warp 0: TMA and MMA issue; warps 1 .. 4 TPR: softmax and epilogue, TPR threads per query row: one, and four CTAs per SM, or four, and one, where
// every CTA has an SM to itself: each thread then has one chunk of 32 keys and 16 columns of the context
// (figures: attention_bwd.cu).
template <int TPR, bool QUANT>
__global__ void __launch_bounds__(32 + 128 * TPR, 4 / TPR) attention_fwd_kernel(const __grid_constant__ CUtensorMap map_qkv, const __grid_constant__ CtxMaps out,
                                                               const __grid_constant__ AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_qk, bar_v, bar_s, bar_p, bar_o;
  __shared__ uint32_t tmem_slot;
  __shared__ float2 red[TPR][128];                           // [part][row]: maximum, sum
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int head = blockIdx.y, b = blockIdx.z;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  // P takes the place of Q and K once the scores are in TMEM
  const uint32_t sV = base, sP = sV + 16384, sQ = sP, sK = sQ + 16384;
  uint8_t* gP = smem_raw + (sP - smem_u32(smem_raw));        // generic pointer to the P operand tile

  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar_qk), 1);
    mbar_init(smem_u32(&bar_v), 1);
    mbar_init(smem_u32(&bar_s), 1);
    mbar_init(smem_u32(&bar_p), 128 * TPR);
    mbar_init(smem_u32(&bar_o), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(p.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  int len = p.valid_len ? p.valid_len[b] : p.S;
  len = len < 1 ? 1 : (len > p.S ? p.S : len);

  if (warp == 0) {
    if (lane == 0) {
      // ---- loads: Q block, the valid keys, the valid values (slots of the qkv tensor: head, h + head, 2h + head)
      mbar_expect_tx(smem_u32(&bar_qk), 2u * 16384u);
      tma_load_4d(sQ, &map_qkv, smem_u32(&bar_qk), 0, 0, head, b);
      tma_load_4d(sK, &map_qkv, smem_u32(&bar_qk), 0, 0, p.h + head, b);
      mbar_expect_tx(smem_u32(&bar_v), 16384u);
      tma_load_4d(sV, &map_qkv, smem_u32(&bar_v), 0, 0, 2 * p.h + head, b);
      const int n16 = (len + 15) & ~15;
      bool ok = mbar_wait(smem_u32(&bar_qk), 0, p.wait_ns);
      if (!ok) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_TMA);
      tc_fence_after();
      // ---- scores: [128 x n16] = Q [128 x 64] * K^T
      if (ok) {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n16 >> 3) << 17) | (8u << 24);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          tc_mma<0>(tmem, smem_desc(sQ + k * 32, 16u, 1024u), smem_desc(sK + k * 32, 16u, 1024u), idesc, (uint32_t)(k != 0));
      }
      tc_commit(smem_u32(&bar_s));
      // ---- context: [128 x 64] = P [128 x keys] * V [keys x 64]  (V is the MN-major operand), over the scores
      if (!mbar_wait(smem_u32(&bar_v), 0, p.wait_ns)) { if (ok) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_TMA); ok = false; }
      const bool handed = mbar_wait(smem_u32(&bar_p), 0, p.wait_ns);
      if (ok && !handed) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_EPI);
      tc_fence_after();
      if (ok && handed) {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(HD >> 3) << 17) | (8u << 24);
#pragma unroll 1
        for (int ks = 0; ks < n16 / 16; ++ks)
          tc_mma<0>(tmem, smem_desc(sP + (ks >> 2) * 16384 + (ks & 3) * 32, 16u, 1024u),
                    smem_desc(sV + ks * 2048, 8192u, 1024u), idesc, (uint32_t)(ks != 0));
      }
      tc_commit(smem_u32(&bar_o));
    }
  } else {
    const int quad = warp & 3, part = (warp - 1) >> 2;
    const int r = quad * 32 + lane;                      // row inside the block
    const bool row_ok = r < p.S;
    float alpha = p.alpha_const;
    if (p.a_p0) alpha *= *p.a_p0;
    if (p.a_p1) alpha *= *p.a_p1;
    const float ps = QUANT ? *p.p_step : 1.f, r_ps = __frcp_rn(ps);
    // (every scalar here: a load behind the last product would be waited for)
    float calpha = 1.f;
    if (p.c_p0) calpha *= *p.c_p0;
    if (p.c_p1) calpha *= *p.c_p1;
    const float cs = QUANT ? *p.c_step : 1.f;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    const int n_valid = (len + 31) / 32;                 // 32-key chunks that hold a valid key: the others are zeros
    const bool got = mbar_wait(smem_u32(&bar_s), 0, p.wait_ns);
    if (!__all_sync(0xffffffffu, got) && lane == 0) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_MMA);
    tc_fence_after();
    const float alpha2 = alpha * 1.4426950408889634f;
    RowPart row{-INFINITY, 0.f};
#pragma unroll 1
    for (int c = part; c < n_valid; c += TPR) {
      uint32_t a[32];
      tmem_ld32(trow + (uint32_t)(c * 32), a);
      join(row, chunk_part(a, len - c * 32, alpha2), alpha2);
    }
    if constexpr (TPR > 1) {                             // (TPR * 32 >= S: a chunk per thread)
      red[part][r] = make_float2(row.max, row.sum);
      asm volatile("bar.sync 1, %0;" ::"n"(128 * TPR) : "memory");
      row = RowPart{-INFINITY, 0.f};
#pragma unroll
      for (int k = 0; k < TPR; ++k)
        if (k < n_valid) join(row, RowPart{red[k][r].x, red[k][r].y}, alpha2);
    }
    const float mx2 = __fmul_rn(alpha2, row.max), sum = row.sum;
    const float inv_sum = __frcp_rn(sum);
    if (p.stats.row && part == 0) {
      if (row_ok) p.stats.row[((long long)b * p.h + head) * p.S + r] = make_float2(mx2, inv_sum);
      if (r == 0 && head == 0) { p.stats.len[b] = len; if (b == 0) *p.stats.alpha = alpha; }
    }
    const RowScale k{splat(alpha2), splat(-mx2), make_float2(inv_sum, inv_sum), splat(r_ps), splat(-ps), p.p_hi};
    const long long prow = (((long long)b * p.h + head) * p.S + r) * p.S;
    const int n_store = p.P ? (p.S + 31) / 32 : n_valid;
#pragma unroll 1
    for (int c = part; c < n_store; c += TPR) {
      uint32_t pw[16], cw[16];                            // 32 probabilities / codes packed as bf16 pairs
      if (c < n_valid) {
        uint32_t a[32];
        tmem_ld32(trow + (uint32_t)(c * 32), a);
        probabilities32<QUANT>(a, len - c * 32, k, pw, cw);
        // operand tile: block of 64 keys, row r, 16-byte chunk index XOR (r & 7)  (128-byte swizzle)
        uint8_t* rowp = gP + (c >> 1) * 16384 + r * 128;
#pragma unroll
        for (int t = 0; t < 4; ++t) store16(rowp + (((c & 1) * 4 + t) ^ (r & 7)) * 16, cw + 4 * t);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) pw[j] = cw[j] = 0u;
      }
      if (row_ok && p.P) {                                // (no P: a pass whose probabilities nobody reads)
        const int ncol = p.S - c * 32;                    // columns of this chunk inside the tensor (S % 8 == 0)
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (t * 8 < ncol) {
            store16(p.P + prow + c * 32 + t * 8, pw + 4 * t);
            if (QUANT && p.P_qt) store16(p.P_qt + prow + c * 32 + t * 8, cw + 4 * t);
          }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to the MMA
    tc_fence_before();
    mbar_arrive(smem_u32(&bar_p));
    // ---- context row, 32 columns at a time
    const bool got2 = mbar_wait(smem_u32(&bar_o), 0, p.wait_ns);
    if (!__all_sync(0xffffffffu, got2) && lane == 0) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_MMA);
    tc_fence_after();
    if (p.ctx) {                                         // (all products have run: the tiles of P and V are free)
      if constexpr (TPR == 1) {
#pragma unroll 1
        for (int hh = 0; hh < 2; ++hh) {
          uint32_t a[32];
          tmem_ld32(trow + (uint32_t)(hh * 32), a);
          context_piece<QUANT, 32>(p, a, calpha, cs, r, hh, gP, gP + 16384, gP - 16384);
        }
      } else {
        uint32_t a[16];
        tmem_ld16(trow + (uint32_t)(part * 16), a);
        context_piece<QUANT, 16>(p, a, calpha, cs, r, part, gP, gP + 16384, gP - 16384);
      }
      fence_async_shared();
      asm volatile("bar.sync 1, %0;" ::"n"(128 * TPR) : "memory");
      if (threadIdx.x == 32) {
        store_context<QUANT>(out, sP, sP + 16384, sV, 0, head, b);
        tma_store_wait_read<0>();
      }
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(p.tmem_cols) : "memory");
  }
}

template <int TPR, bool QUANT>
int launch_short(const CUtensorMap& map, const CtxMaps& out, const AttnParams& p, cudaStream_t st) {
  constexpr int smem = 1024 + 16384 * 3;
  static bool attr_set = false;
  if (!attr_set) {
    if (cudaFuncSetAttribute(attention_fwd_kernel<TPR, QUANT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return GEMM_ERR_CUDA;
    attr_set = true;
  }
  if (launch_k(attention_fwd_kernel<TPR, QUANT>, dim3(1, p.h, p.B), 32 + 128 * TPR, smem, st, map, out, p) != cudaSuccess) return GEMM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? GEMM_OK : GEMM_ERR_CUDA;
}

}  // namespace

bool attention_fwd_supported(int S, int head_dim, int dt) { return dt == 1 && head_dim == HD && S % 8 == 0 && S <= 384; }

// qkv: [B*S, 3H] storage-type tensor (values or codes).  Null p_step / c_step: no quantizer (teacher).
int launch_attention_fwd(const void* qkv, int B, int S, int h, int H, const int* valid_len, float alpha_const,
                         const float* a_p0, const float* a_p1, const float* c_p0, const float* c_p1,
                         const float* p_step, int p_lo, int p_hi, void* P, void* P_qt, void* ctx, const float* c_step,
                         int c_qmax, int8_t* ctx_q8, void* ctx_qt, int* status, cudaStream_t st, const AttentionStats* stats) {
  AttnParams p;
  p.S = S; p.h = h; p.B = B; p.H = H;
  int cols = 64;
  while (cols < S) cols *= 2;
  p.tmem_cols = cols;
  p.alpha_const = alpha_const; p.a_p0 = a_p0; p.a_p1 = a_p1; p.c_p0 = c_p0; p.c_p1 = c_p1;
  p.valid_len = valid_len;
  p.order = 0;
  p.p_step = p_step; p.p_lo = (float)p_lo; p.p_hi = (float)p_hi;
  p.c_step = c_step; p.c_qmax = (float)c_qmax;
  p.P = (bf16*)P; p.P_qt = (bf16*)P_qt; p.ctx = (bf16*)ctx; p.ctx_q8 = ctx_q8; p.ctx_qt = (bf16*)ctx_qt;
  p.stats = stats ? *stats : AttentionStats{nullptr, nullptr, nullptr};
  p.status = status;
  p.wait_ns = g_wait_limit_ns;
  Scope sc("attention_fwd_tcgen05", 4.0 * B * h * (double)S * S * HD, 1, st);
  if (S > 128) return launch_attention_fwd_long(p, qkv, st);
  // one map over the [tokens, 3H] tensor: (64 of a head, S rows, 3h head slots, B)
  OperandDesc op{qkv, 3LL * H, HD, (long long)S * 3 * H, 0};
  CUtensorMap map;
  int rc = make_operand_map(&map, op, 2, S, HD, 3 * h, B, 128, HD);
  CtxMaps out;
  if (rc == GEMM_OK) rc = make_ctx_maps(&out, p, map);
  if (rc != GEMM_OK) return rc;
  if (B * h <= 148) return p_step ? launch_short<4, true>(map, out, p, st) : launch_short<4, false>(map, out, p, st);     // a CTA per SM
  return p_step ? launch_short<1, true>(map, out, p, st) : launch_short<1, false>(map, out, p, st);
}

}  // namespace mrem
