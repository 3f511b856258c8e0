// Fused attention forward for one (batch, head, 128-query block) per CTA on sm_100a:
//   S = Q K^T (tcgen05, fp32 accumulators in TMEM)  ->  masked softmax straight out of TMEM  ->  (student) Eq. 1 on the
//   probabilities  ->  ctx = P V with P taken from shared memory as the A operand of a second tcgen05 product.
// The scores never touch HBM.  Operands are the Q/K/V slices of the [tokens, 3*hidden] tensor
// (bf16 values for the teacher, integer codes held as bf16 for the student: every product of
// codes is exact in fp32), fetched by TMA with 128-byte swizzle.  Outputs: the probabilities
// (and their codes) for the backward pass, the context rows, and for the student the codes of
// the context (int8 for the next int8 product, bf16 for the backward).
// Head size 64, sequence length up to 384.  All waits are time-bounded.
//
// What bounds it: one CTA is a serial chain (tiles by TMA, product, softmax, product, rows out) and the softmax arithmetic
// fills the issue slots only when several CTAs, or several threads per row, share an SM.  So P takes the place of Q and K
// in shared memory and the context that of the scores in TMEM, and the rest is a matter of TPR, the threads per query row:
//   S <= 128:  TPR 1, 48 KB and 128 TMEM columns: four CTAs per SM, no barrier inside the softmax (was two CTAs of two
//              threads per row: 512 CTAs were two rounds on 148 SMs and are one now);
//   S <= 256:  TPR 2, two CTAs per SM;   S <= 384:  TPR 4, one CTA per SM (384 score columns), 16 warps instead of 8.
// Keys beyond the valid length cost nothing: their chunks are neither multiplied nor exponentiated.  Instruction fetch counts too: everything runs
// once or a few times per CTA, so the loops over chunks stay rolled (67 KB of code became 35).
// 32 x 16 heads x 128 x 128: 20.6 -> 15 us (mean of teacher and student pass); 16 x 16 x 384 x 384: 98 -> 55 us.
#include "gemm.h"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace mrem {

namespace {

constexpr int HD = 64;

struct AttnParams {
  int S, h, B, H;
  int tmem_cols;             // allocation (power of two >= S, at least 64)
  float alpha_const;         // score scale = alpha_const * (*a_p0) * (*a_p1)
  const float *a_p0, *a_p1;
  const float *c_p0, *c_p1;  // context scale = (*c_p0) * (*c_p1); null = 1
  const int* valid_len;
  const float* p_step;       // quantizer of the probabilities (student), null = none
  float p_lo, p_hi;
  const float* c_step;       // symmetric quantizer of the context (student), null = none
  float c_qmax;
  bf16 *P, *P_qt;            // [B, h, S, S]
  bf16* ctx;                 // [B*S, H]
  int8_t* ctx_q8;            // [B*S, H]
  bf16* ctx_qt;              // [B*S, H]
  AttentionStats stats;      // for the backward pass (null members: none)
  int* status;
  unsigned long long wait_ns;  // limit of each wait on an mbarrier
};

__device__ __forceinline__ void store16(void* p, const uint32_t* w) {
  *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}

// TPR threads per query row; QUANT: the student pass (quantizers of the probabilities and of the context).
// Warp 0: TMA and MMA issue; warps 1 .. 4 TPR: softmax and epilogue, TPR warps per TMEM lane quadrant.
template <int TPR, bool QUANT>
__global__ void __launch_bounds__(32 + 128 * TPR, 4 / TPR) attention_fwd_kernel(const __grid_constant__ CUtensorMap map_qkv,
                                                                                const __grid_constant__ AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_qk, bar_v, bar_s, bar_p, bar_o;
  __shared__ uint32_t tmem_slot;
  __shared__ float red[2][TPR][128];                         // [max | sum][part][row]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qb = blockIdx.x, head = blockIdx.y, b = blockIdx.z;
  const int q0 = qb * 128;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int n_box = (p.S + 127) / 128;                       // 128-row TMA boxes of keys / values
  // P takes the place of Q and K once the scores are in TMEM
  const uint32_t sV = base, sP = sV + n_box * 16384, sQ = sP, sK = sQ + 16384;
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
      const int boxes = (len + 127) / 128, n16 = (len + 15) & ~15;
      mbar_expect_tx(smem_u32(&bar_qk), 16384u * (uint32_t)(1 + boxes));
      tma_load_4d(sQ, &map_qkv, smem_u32(&bar_qk), 0, q0, head, b);
#pragma unroll 1
      for (int i = 0; i < boxes; ++i) tma_load_4d(sK + i * 16384, &map_qkv, smem_u32(&bar_qk), 0, i * 128, p.h + head, b);
      mbar_expect_tx(smem_u32(&bar_v), 16384u * (uint32_t)boxes);
#pragma unroll 1
      for (int i = 0; i < boxes; ++i) tma_load_4d(sV + i * 16384, &map_qkv, smem_u32(&bar_v), 0, i * 128, 2 * p.h + head, b);
      bool ok = mbar_wait(smem_u32(&bar_qk), 0, p.wait_ns);
      if (!ok) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_TMA);
      tc_fence_after();
      // ---- scores: [128 x n16] = Q [128 x 64] * K^T, in pieces of at most 256 keys
      if (ok) {
        for (int n0 = 0; n0 < n16; n0 += 256) {
          const int n = min(256, n16 - n0);
          const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (8u << 24);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            tc_mma<0>(tmem + (uint32_t)n0, smem_desc(sQ + k * 32, 16u, 1024u), smem_desc(sK + n0 * 128 + k * 32, 16u, 1024u),
                      idesc, (uint32_t)(k != 0));
        }
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
    const int q = q0 + r;
    const bool row_ok = q < p.S;
    float alpha = p.alpha_const;
    if (p.a_p0) alpha *= *p.a_p0;
    if (p.a_p1) alpha *= *p.a_p1;
    const float ps = QUANT ? *p.p_step : 1.f, r_ps = __frcp_rn(ps);
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    const int n_valid = (len + 31) / 32;                 // 32-key chunks that hold a valid key: the others are zeros
    const bool got = mbar_wait(smem_u32(&bar_s), 0, p.wait_ns);
    if (!__all_sync(0xffffffffu, got) && lane == 0) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_MMA);
    tc_fence_after();
    // scores in units of log2(e): exp(alpha * a - max) = 2^(alpha2 * a - max2); alpha > 0, so the maximum
    // can be taken over the raw accumulators
    const float alpha2 = alpha * 1.4426950408889634f;
    float mx = -INFINITY;
#pragma unroll 1
    for (int c = part; c < n_valid; c += TPR) {
      uint32_t a[32];
      tmem_ld32(trow + (uint32_t)(c * 32), a);
      if (c * 32 + 32 <= len) {                          // all 32 keys valid (warp-uniform)
        float m4[4] = {mx, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int j = 0; j < 32; ++j) m4[j & 3] = fmaxf(m4[j & 3], __uint_as_float(a[j]));
        mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (c * 32 + j < len) mx = fmaxf(mx, __uint_as_float(a[j]));
      }
    }
    if constexpr (TPR > 1) {
      red[0][part][r] = mx;
      asm volatile("bar.sync 1, %0;" ::"n"(128 * TPR) : "memory");
#pragma unroll
      for (int k = 0; k < TPR; ++k) mx = fmaxf(mx, red[0][k][r]);
    }
    const float mx2 = alpha2 * mx;
    const float2 alpha22 = make_float2(alpha2, alpha2), nmx2 = make_float2(-mx2, -mx2);
    float2 sums[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll 1
    for (int c = part; c < n_valid; c += TPR) {
      uint32_t a[32];
      tmem_ld32(trow + (uint32_t)(c * 32), a);
      const int ncol = len - c * 32;                     // (>= 32: all keys valid)
#pragma unroll
      for (int j = 0; j < 32; j += 2) {
        const float2 t = fma2(make_float2(__uint_as_float(a[j]), __uint_as_float(a[j + 1])), alpha22, nmx2);
        float2 e = make_float2(exp2_approx(t.x), exp2_approx(t.y));
        if (ncol < 32) { e.x = j < ncol ? e.x : 0.f; e.y = j + 1 < ncol ? e.y : 0.f; }
        sums[(j >> 1) & 1] = add2(sums[(j >> 1) & 1], e);
      }
    }
    float sum = (sums[0].x + sums[0].y) + (sums[1].x + sums[1].y);
    if constexpr (TPR > 1) {
      red[1][part][r] = sum;
      asm volatile("bar.sync 1, %0;" ::"n"(128 * TPR) : "memory");
      sum = red[1][0][r];
#pragma unroll
      for (int k = 1; k < TPR; ++k) sum += red[1][k][r];
    }
    const float inv_sum = __frcp_rn(sum);
    if (p.stats.row && part == 0) {
      if (row_ok) p.stats.row[((long long)b * p.h + head) * p.S + q] = make_float2(mx2, inv_sum);
      if (r == 0 && qb == 0 && head == 0) { p.stats.len[b] = len; if (b == 0) *p.stats.alpha = alpha; }
    }
    const float2 inv2 = make_float2(inv_sum, inv_sum), r2 = make_float2(r_ps, r_ps), ns2 = make_float2(-ps, -ps);
    const float2 magic2 = make_float2(ROUND_MAGIC, ROUND_MAGIC), nmagic2 = make_float2(-ROUND_MAGIC, -ROUND_MAGIC);
    const long long prow = (((long long)b * p.h + head) * p.S + q) * p.S;
    const int n_store = p.P ? (p.S + 31) / 32 : n_valid;
#pragma unroll 1
    for (int c = part; c < n_store; c += TPR) {
      uint32_t pw[16], cw[16];                            // 32 probabilities / codes packed as bf16 pairs
      if (c < n_valid) {
        uint32_t a[32];
        tmem_ld32(trow + (uint32_t)(c * 32), a);
        const int ncol = len - c * 32;
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          // (the exponentials are formed a second time: cheaper than keeping them in TMEM)
          const float2 t = fma2(make_float2(__uint_as_float(a[j]), __uint_as_float(a[j + 1])), alpha22, nmx2);
          float2 v = mul2(make_float2(exp2_approx(t.x), exp2_approx(t.y)), inv2);
          if (ncol < 32) { v.x = j < ncol ? v.x : 0.f; v.y = j + 1 < ncol ? v.y : 0.f; }
          const __nv_bfloat162 pb = __floats2bfloat162_rn(v.x, v.y);
          pw[j >> 1] = *reinterpret_cast<const uint32_t*>(&pb);
          if constexpr (QUANT) {
            // the quotient of a bf16 value is the IEEE division of Eq. 1 (see quotient()); probabilities are not negative,
            // so only the upper bound of the code range can clip
            const float2 f = make_float2(__uint_as_float(pw[j >> 1] << 16), __uint_as_float(pw[j >> 1] & 0xffff0000u));
            const float2 z0 = mul2(f, r2);
            float2 z = fma2(fma2(z0, ns2, f), r2, z0);
            z = make_float2(fminf(z.x, p.p_hi), fminf(z.y, p.p_hi));
            const float2 k = add2(add2(z, magic2), nmagic2);
            const __nv_bfloat162 cb = __floats2bfloat162_rn(k.x, k.y);
            cw[j >> 1] = *reinterpret_cast<const uint32_t*>(&cb);
          } else {
            cw[j >> 1] = pw[j >> 1];
          }
        }
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
    float calpha = 1.f;
    if (p.c_p0) calpha *= *p.c_p0;
    if (p.c_p1) calpha *= *p.c_p1;
    const float cs = QUANT ? *p.c_step : 1.f, r_cs = __frcp_rn(cs);
    const long long crow = ((long long)b * p.S + q) * p.H + head * HD;
#pragma unroll 1
    for (int hh = part; hh < 2; hh += TPR) {
      uint32_t a[32];
      tmem_ld32(trow + (uint32_t)(hh * 32), a);
      uint32_t w[16], cq[16], c8[8];
#pragma unroll
      for (int j = 0; j < 32; j += 2) {
        const __nv_bfloat162 vb = __floats2bfloat162_rn(calpha * __uint_as_float(a[j]), calpha * __uint_as_float(a[j + 1]));
        w[j >> 1] = *reinterpret_cast<const uint32_t*>(&vb);
        if constexpr (QUANT) {
          const float2 f = __bfloat1622float2(vb);
          uint32_t b0, b1;                                 // rounding words: low byte = the 8-bit code
          const float i0 = rne_magic(fminf(fmaxf(quotient(f.x, cs, r_cs), -p.c_qmax), p.c_qmax), b0);
          const float i1 = rne_magic(fminf(fmaxf(quotient(f.y, cs, r_cs), -p.c_qmax), p.c_qmax), b1);
          const __nv_bfloat162 cb = __floats2bfloat162_rn(i0, i1);
          cq[j >> 1] = *reinterpret_cast<const uint32_t*>(&cb);
          const uint32_t two = __byte_perm(b0, b1, 0x0040) & 0xffffu;
          if ((j & 2) == 0) c8[j >> 2] = two; else c8[j >> 2] |= two << 16;
        }
      }
      if (row_ok && p.ctx) {
#pragma unroll
        for (int t = 0; t < 4; ++t) store16(p.ctx + crow + hh * 32 + t * 8, w + 4 * t);
        if constexpr (QUANT) {
#pragma unroll
          for (int t = 0; t < 4; ++t) store16(p.ctx_qt + crow + hh * 32 + t * 8, cq + 4 * t);
          store16(p.ctx_q8 + crow + hh * 32, c8);
          store16(p.ctx_q8 + crow + hh * 32 + 16, c8 + 4);
        }
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
int launch_tpr(const CUtensorMap& map, const AttnParams& p, cudaStream_t st) {
  const int n_box = (p.S + 127) / 128, n_kb = (p.S + 63) / 64;
  const int smem = 1024 + 16384 * (n_box + (n_kb > 1 + n_box ? n_kb : 1 + n_box));
  // the limit for the longest sequence of this variant, whatever this one needs: threads that get here together set the same one
  constexpr int MAX_BOX = TPR == 4 ? 3 : TPR;
  static bool attr_set = false;
  if (!attr_set) {
    if (cudaFuncSetAttribute(attention_fwd_kernel<TPR, QUANT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + 16384 * 3 * MAX_BOX) != cudaSuccess)
      return GEMM_ERR_CUDA;
    attr_set = true;
  }
  if (launch_k(attention_fwd_kernel<TPR, QUANT>, dim3((p.S + 127) / 128, p.h, p.B), 32 + 128 * TPR, smem, st, map, p) != cudaSuccess) return GEMM_ERR_CUDA;
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
  p.p_step = p_step; p.p_lo = (float)p_lo; p.p_hi = (float)p_hi;
  p.c_step = c_step; p.c_qmax = (float)c_qmax;
  p.P = (bf16*)P; p.P_qt = (bf16*)P_qt; p.ctx = (bf16*)ctx; p.ctx_q8 = ctx_q8; p.ctx_qt = (bf16*)ctx_qt;
  p.stats = stats ? *stats : AttentionStats{nullptr, nullptr, nullptr};
  p.status = status;
  p.wait_ns = g_wait_limit_ns;
  // one map over the [tokens, 3H] tensor: (64 of a head, S rows, 3h head slots, B)
  OperandDesc op{qkv, 3LL * H, HD, (long long)S * 3 * H, 0};
  CUtensorMap map;
  const int rc = make_operand_map(&map, op, 2, S, HD, 3 * h, B, 128, HD);
  if (rc != GEMM_OK) return rc;
  Scope sc("attention_fwd_tcgen05", 4.0 * B * h * (double)S * S * HD, 1, st);
  if (p_step) return S <= 128 ? launch_tpr<1, true>(map, p, st) : (S <= 256 ? launch_tpr<2, true>(map, p, st) : launch_tpr<4, true>(map, p, st));
  return S <= 128 ? launch_tpr<1, false>(map, p, st) : (S <= 256 ? launch_tpr<2, false>(map, p, st) : launch_tpr<4, false>(map, p, st));
}

}  // namespace mrem
