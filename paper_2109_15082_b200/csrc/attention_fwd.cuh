// Pieces shared by the attention forward kernels: parameters, a row's softmax pieces, a row of the context on its way out.
#pragma once
#include "gemm.h"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace mrem {
namespace attf {

constexpr int HD = 64;

struct AttnParams {
  int S, h, B, H;
  int tmem_cols;             // allocation (power of two >= S, at least 64)
  float alpha_const;         // score scale = alpha_const * (*a_p0) * (*a_p1)
  const float *a_p0, *a_p1;
  const float *c_p0, *c_p1;  // context scale = (*c_p0) * (*c_p1); null = 1
  const int* valid_len;
  int order;                 // blocks take the sequences longest first
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

__device__ __forceinline__ float max3(float a, float b, float c) {   // NaNs as fmaxf
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// A row's softmax is put together from chunks of 32 scores: maximum of a chunk, sum of its exponentials with that maximum, then the
// chunks in order.  However many threads share a row, a sequence has the same sums bit for bit.
// In units of log2(e): exp(alpha * a - max) = 2^(alpha2 * a - max2); alpha > 0, so the maximum can be taken over the raw accumulators.
// max2 is rounded (not a part of an fma): an exponential formed with it again later is the same number.
struct RowPart { float max, sum; };
// of 32 scores (accumulators a, the first ncol >= 1 of them valid)
__device__ __forceinline__ RowPart chunk_part(uint32_t* a, int ncol, float alpha2) {
  if (ncol < 32) {                                       // (warp-uniform, a row's last chunk only: nothing below tests the keys)
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j >= ncol) a[j] = 0xff800000u;                 // -inf
  }
  float m4[4] = {__uint_as_float(a[0]), __uint_as_float(a[1]), __uint_as_float(a[2]), __uint_as_float(a[3])};
#pragma unroll
  for (int j = 4; j < 32; j += 2) m4[(j >> 1) & 3] = max3(m4[(j >> 1) & 3], __uint_as_float(a[j]), __uint_as_float(a[j + 1]));
  const float m = fmaxf(max3(m4[0], m4[1], m4[2]), m4[3]);
  const float2 nmx2 = splat(m == -INFINITY ? 0.f : -__fmul_rn(alpha2, m));             // (nothing but -inf: a sum of zeros)
  float2 sums[2] = {splat(0.f), splat(0.f)};
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    const float2 t = fma2(make_float2(__uint_as_float(a[j]), __uint_as_float(a[j + 1])), splat(alpha2), nmx2);
    sums[(j >> 1) & 1] = add2(sums[(j >> 1) & 1], make_float2(exp2_approx(t.x), exp2_approx(t.y)));
  }
  return RowPart{m, (sums[0].x + sums[0].y) + (sums[1].x + sums[1].y)};
}
// row += part (a row starts as {-inf, 0})
__device__ __forceinline__ void join(RowPart& row, const RowPart& part, float alpha2) {
  const float m = fmaxf(row.max, part.max), m2 = __fmul_rn(alpha2, m);
  const float f = row.max == m ? 1.f : exp2_approx(__fmul_rn(alpha2, row.max) - m2);
  const float g = part.max == m ? 1.f : exp2_approx(__fmul_rn(alpha2, part.max) - m2);
  row = RowPart{m, __fmaf_rn(part.sum, g, __fmul_rn(row.sum, f))};
}

// 32 scores of a row (accumulators a, the first ncol of them valid) -> their probabilities as bf16 pairs (pw) and what the second
// product multiplies (cw): the codes of Eq. 1, or without a quantizer the probabilities themselves.
struct RowScale { float2 alpha2, neg_max, inv_sum, r_step, neg_step; float hi; };
template <bool QUANT>
__device__ __forceinline__ void probabilities32(const uint32_t* a, int ncol, const RowScale& k, uint32_t* pw, uint32_t* cw) {
  const float2 magic2 = make_float2(ROUND_MAGIC, ROUND_MAGIC), nmagic2 = make_float2(-ROUND_MAGIC, -ROUND_MAGIC);
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    // (the exponentials are formed a second time: cheaper than keeping them in TMEM)
    const float2 t = fma2(make_float2(__uint_as_float(a[j]), __uint_as_float(a[j + 1])), k.alpha2, k.neg_max);
    const float2 v = mul2(make_float2(exp2_approx(t.x), exp2_approx(t.y)), k.inv_sum);
    const __nv_bfloat162 pb = __floats2bfloat162_rn(v.x, v.y);
    pw[j >> 1] = *reinterpret_cast<const uint32_t*>(&pb);
    if constexpr (QUANT) {
      // the quotient of a bf16 value is the IEEE division of Eq. 1 (see quotient()); probabilities are not negative,
      // so only the upper bound of the code range can clip
      const float2 f = make_float2(__uint_as_float(pw[j >> 1] << 16), __uint_as_float(pw[j >> 1] & 0xffff0000u));
      const float2 z0 = mul2(f, k.r_step);
      float2 z = fma2(fma2(z0, k.neg_step, f), k.r_step, z0);
      z = make_float2(fminf(z.x, k.hi), fminf(z.y, k.hi));
      const float2 c = add2(add2(z, magic2), nmagic2);
      const __nv_bfloat162 cb = __floats2bfloat162_rn(c.x, c.y);
      cw[j >> 1] = *reinterpret_cast<const uint32_t*>(&cb);
    } else {
      cw[j >> 1] = pw[j >> 1];
    }
  }
  if (ncol < 32) {                                     // (warp-uniform, a row's last chunk only)
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t keep = 2 * j + 1 < ncol ? 0xffffffffu : (2 * j < ncol ? 0xffffu : 0u);
      pw[j] &= keep;
      cw[j] &= keep;
    }
  }
}

// Piece `part` of a context row, N columns (accumulators a), into operand-like tiles of 128 rows that leave by tiled stores: bf16 values, and with a
// quantizer their codes as bf16 numbers and as bytes.  (Stored from registers, a row per lane, every instruction touched 32 lines:
// 2.3 us of a CTA's 15 at 16 x 16 x 384 x 384.)
struct CtxMaps { CUtensorMap ctx, qt, q8; };
template <bool QUANT, int N>
__device__ __forceinline__ void context_piece(const AttnParams& p, const uint32_t* a, float calpha, float cs, int r, int part, uint8_t* t_ctx, uint8_t* t_qt,
                                              uint8_t* t_q8) {
  uint32_t w[N / 2], cq[N / 2], c8[N / 4];
  const float r_cs = __frcp_rn(cs);
#pragma unroll
  for (int j = 0; j < N; j += 2) {
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
  // 128-byte swizzle: 16-byte piece index XOR (row & 7); rows of 64 bytes, 64-byte swizzle: XOR (row / 2 & 3)
#pragma unroll
  for (int t = 0; t < N / 8; ++t) {
    const int at = r * 128 + ((part * (N / 8) + t) ^ (r & 7)) * 16;
    store16(t_ctx + at, w + 4 * t);
    if constexpr (QUANT) store16(t_qt + at, cq + 4 * t);
  }
  if constexpr (QUANT) {
#pragma unroll
    for (int t = 0; t < N / 16; ++t) store16(t_q8 + r * 64 + ((part * (N / 16) + t) ^ ((r >> 1) & 3)) * 16, c8 + 4 * t);
  }
}
// one thread, once every row is written and fenced: 128 rows from q0 on of (head, b); rows beyond the sequence are clipped
template <bool QUANT>
__device__ __forceinline__ void store_context(const CtxMaps& m, uint32_t t_ctx, uint32_t t_qt, uint32_t t_q8, int q0, int head, int b) {
  tma_store_4d(&m.ctx, t_ctx, 0, q0, head, b);
  if (QUANT) {
    tma_store_4d(&m.qt, t_qt, 0, q0, head, b);
    tma_store_4d(&m.q8, t_q8, 0, q0, head, b);
  }
  tma_store_commit();
}
// (no context: nothing is stored through the maps)
inline int make_ctx_maps(CtxMaps* m, const AttnParams& p, const CUtensorMap& any) {
  m->ctx = m->qt = m->q8 = any;
  if (!p.ctx) return GEMM_OK;
  auto map = [&](CUtensorMap* out, const void* ptr, int bytes) {
    return make_operand_map(out, OperandDesc{ptr, p.H, HD, (long long)p.S * p.H, 0}, bytes, p.S, HD, p.h, p.B, 128, HD);
  };
  int rc = map(&m->ctx, p.ctx, 2);
  if (rc == GEMM_OK && p.c_step) rc = map(&m->qt, p.ctx_qt, 2);
  if (rc == GEMM_OK && p.c_step) rc = map(&m->q8, p.ctx_q8, 1);
  return rc;
}

// attention_fwd_long.cu: 129 to 384 tokens
int launch_attention_fwd_long(const AttnParams& p, const void* qkv, cudaStream_t st);

}  // namespace attf
}  // namespace mrem
