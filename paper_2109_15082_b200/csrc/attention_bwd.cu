// Fused attention backward of the student on sm_100a, sequences up to 128 tokens, head size 64: one (batch, head) per CTA.
// Inputs: the gradient of the quantized context, the context and Q, K, V before quantization, the codes of Q, K, V, and per
// query row the two numbers the forward pass left of its softmax (maximum, 1 / sum).  One kernel does what otherwise takes
// five batched products, the softmax and its backward and four straight-through kernels:
//   STE of the context's quantizer: dctx (in place in its operand tile)
//   S = Q_q K_q^T and dP_hat = s_v dctx V_q^T                       (tcgen05, accumulators in TMEM)
//   P from S exactly as the forward pass formed it (bit for bit: the products of codes are exact), its codes, the STE of its
//     quantizer, dS = P * (dP - sum_j dP P): two threads per query row reading TMEM; codes of P and dS go to shared memory
//   dV_hat = s_p P_q^T dctx,  dQ_hat = s_k/sqrt(d) dS K_q,  dK_hat = s_q/sqrt(d) dS^T Q_q
//     (three tcgen05 products; the same shared-memory tile serves as K-major A operand of one product and as MN-major A
//     operand of another, so nothing is transposed)
//   STE of the Q, K, V quantizers on the way out.
// Step-size gradients leave as one partial sum per CTA and site (summed later in CTA order).  All waits are time-bounded.
//
// What bounds it: a CTA is a serial chain of small steps, so what counts is their latency.  The probabilities are recomputed
// (6 instructions per score) instead of written by the forward pass and read twice by lanes that each own a row (32 lines per
// load: 4,900 of the kernel's 40,000 cycles, and 33 MB per launch at 32 x 16 x 128 x 128); the values before quantization come
// in and the gradients go out through operand tiles that are no longer needed (TMA); tests for clipped values are made once
// per warp and chunk.  32 x 16 heads x 128 x 128: 50 + 8 us (kernel, STE of the context) -> 29 us.
// Stamps there (13 us a CTA, two rounds of two): tiles 2.4, STE 0.7, P 2.3, dS 1.4, the three gradients 3.7, sums 0.9; the sites' terms formed while the tiles
// come, K before quantization loaded into its own tile: 0.5 us less.
// Shared memory: Q, K, V, dctx tiles of 16 KB and one of 32 KB that is the context, then the codes of P, then dS; the V tile
// becomes V before quantization -> dV out, the dctx tile Q before quantization -> dQ out, the K tile K before quantization -> dK out.
// TMEM (256 columns, two CTAs per SM): dP | S; dV takes the place of S, dQ and dK that of dP.
#include "attention_bwd.cuh"

namespace mrem {

using namespace att;

namespace {

constexpr int TMEM_DP = 0, TMEM_S = 128, TMEM_DV = 128, TMEM_DQ = 0, TMEM_DK = 64, TMEM_ALLOC = 256;

struct AttnBwdParams {
  int S, h, B, H;
  float inv_sqrt_d;
  const float *s_q, *s_k, *s_v, *s_p, *s_c;
  const float* alpha;        // score scale of the forward pass
  const int* len;            // [B] valid keys (clamped)
  const float2* stat;        // [B, h, S] (alpha log2(e) max, 1 / sum)
  float q_hi;                // code range -q_hi .. q_hi of the symmetric Q / K / V / context sites
  float p_hi;                // upper end of the code range of the P site (probabilities are not negative)
  float *part_q, *part_k, *part_v, *part_p, *part_c;   // [red_slots] each: one partial per CTA, the rest zeroed
  float* col_part;           // [B, 3, H] column sums of dQ, dK, dV
  int red_slots;
  int* status;
  unsigned long long wait_ns;  // limit of each wait on an mbarrier
};

struct AttnBwdMaps { CUtensorMap codes, raw, dctx, ctx, out; };

// Warp 0: TMA + MMA issue; RW row warps: two threads per row, two CTAs per SM, or four and one.  Where every CTA has an SM to itself the
// four win: a thread's part of each link of the chain is half as long
// (step of 3 x 72 tokens, hidden 768, forward kernel alike 434 -> 423 us; of 4 x 32, hidden 128 82.4 -> 82.1).
template <int RW>
__global__ void __launch_bounds__(32 + 32 * RW, 16 / RW) attention_bwd_kernel(const __grid_constant__ AttnBwdMaps maps,
                                                                              const __grid_constant__ AttnBwdParams p) {
  constexpr int TPR = RW / 4, NC = 4 / TPR, PIECE = 8 / TPR;      // threads per row, 32-key chunks per thread, 16-byte pieces of a 64-column row
  extern __shared__ uint8_t smem_raw[];
  enum { B_CODES, B_CTX, B_STE, B_A, B_RV, B_P, B_B, B_RQ, B_S, B_O, B_RK, N_BARS };
  __shared__ __align__(8) uint64_t bars[N_BARS];
  __shared__ uint32_t tmem_slot;
  __shared__ float red_dot[TPR][128];
  __shared__ float red_part[RW][5];
  __shared__ SiteTerms sites[RW][5];                     // per warp: Q, K, V, context, P
  __shared__ __align__(8) float red_col[3][RW * 64];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int head = blockIdx.x, b = blockIdx.y;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = base, sK = sQ + 16384, sV = sK + 16384, sD = sV + 16384, sX = sD + 16384;
  uint8_t* const g0 = smem_raw + (base - smem_u32(smem_raw));
  uint8_t *const gK = g0 + (sK - base), *const gV = g0 + (sV - base), *const gD = g0 + (sD - base), *const gX = g0 + (sX - base);
  auto bar = [&](int i) { return smem_u32(&bars[i]); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < N_BARS; ++i) mbar_init(bar(i), (i == B_STE || i == B_P || i == B_S) ? 32 * RW : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TMEM_ALLOC)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  const int len = p.len[b];
  const int n_valid = (len + 31) / 32, n_chunks = (p.S + 31) / 32;        // 32-key chunks with a valid key, with any key
  const int q_steps = (p.S + 15) / 16, k_steps = (len + 15) / 16;

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(bar(B_CTX), 2u * 16384u);
      tma_load_4d(sD, &maps.dctx, bar(B_CTX), 0, 0, head, b);
      tma_load_4d(sX, &maps.ctx, bar(B_CTX), 0, 0, head, b);
      mbar_expect_tx(bar(B_CODES), 3u * 16384u);
      tma_load_4d(sQ, &maps.codes, bar(B_CODES), 0, 0, head, b);
      tma_load_4d(sK, &maps.codes, bar(B_CODES), 0, 0, p.h + head, b);
      tma_load_4d(sV, &maps.codes, bar(B_CODES), 0, 0, 2 * p.h + head, b);
      bool ok = mbar_wait(bar(B_CODES), 0, p.wait_ns);
      if (!ok) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_TMA);
      tc_fence_after();
      const uint32_t f32 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
      const uint32_t id_s = f32 | ((uint32_t)(n_valid * 32 >> 3) << 17);
      if (ok)        // S [queries x keys] = Q_q [q x d] * K_q^T
#pragma unroll
        for (int k = 0; k < 4; ++k)
          tc_mma<0>(tmem + TMEM_S, smem_desc(sQ + k * 32, 16u, 1024u), smem_desc(sK + k * 32, 16u, 1024u), id_s, (uint32_t)(k != 0));
      ok = mbar_wait(bar(B_STE), 0, p.wait_ns) && ok;
      tc_fence_after();
      if (ok)        // dP_hat [queries x keys] = dctx [q x d] * V_q^T
#pragma unroll
        for (int k = 0; k < 4; ++k)
          tc_mma<0>(tmem + TMEM_DP, smem_desc(sD + k * 32, 16u, 1024u), smem_desc(sV + k * 32, 16u, 1024u), id_s, (uint32_t)(k != 0));
      tc_commit(bar(B_A));
      ok = mbar_wait(bar(B_A), 0, p.wait_ns) && ok;
      mbar_expect_tx(bar(B_RV), 16384u);                       // the V tile is free: V before quantization
      tma_load_4d(sV, &maps.raw, bar(B_RV), 0, 0, 2 * p.h + head, b);
      const uint32_t f = f32 | ((uint32_t)(HD >> 3) << 17);
      const uint32_t id_tt = f | (1u << 15) | (1u << 16);     // A and B MN-major
      const uint32_t id_nt = f | (1u << 16);                  // A K-major, B MN-major
      ok = mbar_wait(bar(B_P), 0, p.wait_ns) && ok;
      tc_fence_after();
      if (ok)
#pragma unroll 1
        for (int ks = 0; ks < q_steps; ++ks)      // dV_hat [keys x d] = P_q^T [keys x q] * dctx [q x d]
          tc_mma<0>(tmem + TMEM_DV, smem_desc(sX + ks * 2048, 16384u, 1024u), smem_desc(sD + ks * 2048, 8192u, 1024u), id_tt, (uint32_t)(ks != 0));
      tc_commit(bar(B_B));
      ok = mbar_wait(bar(B_B), 0, p.wait_ns) && ok;
      mbar_expect_tx(bar(B_RQ), 16384u);                       // the dctx tile is free: Q before quantization
      tma_load_4d(sD, &maps.raw, bar(B_RQ), 0, 0, head, b);
      ok = mbar_wait(bar(B_S), 0, p.wait_ns) && ok;
      if (!ok) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_EPI);
      tc_fence_after();
      if (ok) {
#pragma unroll 1
        for (int ks = 0; ks < k_steps; ++ks)      // dQ_hat [q x d] = dS [q x keys] * K_q [keys x d]
          tc_mma<0>(tmem + TMEM_DQ, smem_desc(sX + (ks >> 2) * 16384 + (ks & 3) * 32, 16u, 1024u), smem_desc(sK + ks * 2048, 8192u, 1024u), id_nt, (uint32_t)(ks != 0));
#pragma unroll 1
        for (int ks = 0; ks < q_steps; ++ks)      // dK_hat [keys x d] = dS^T [keys x q] * Q_q [q x d]
          tc_mma<0>(tmem + TMEM_DK, smem_desc(sX + ks * 2048, 16384u, 1024u), smem_desc(sQ + ks * 2048, 8192u, 1024u), id_tt, (uint32_t)(ks != 0));
      }
      tc_commit(bar(B_O));
      ok = mbar_wait(bar(B_O), 0, p.wait_ns) && ok;
      mbar_expect_tx(bar(B_RK), 16384u);                       // the codes of K have been multiplied: K before quantization
      tma_load_4d(sK, &maps.raw, bar(B_RK), 0, 0, p.h + head, b);
    }
  } else {
    const int quad = warp & 3, part = (warp - 1) >> 2;
    const int r = quad * 32 + lane;                       // row of the tile: a query for S / dP / dS / dQ, a key for dK / dV
    const bool row_ok = r < p.S;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    const float s_p = *p.s_p, s_v = *p.s_v, s_q = *p.s_q, s_k = *p.s_k, s_c = *p.s_c;
    float2 st = make_float2(0.f, 0.f);                    // rows beyond the sequence: P = 0
    if (row_ok) st = p.stat[((long long)b * p.h + head) * p.S + r];
    const float alpha2 = *p.alpha * 1.4426950408889634f;
    if (lane < 5) {
      const float step = lane == 0 ? s_q : (lane == 1 ? s_k : (lane == 2 ? s_v : (lane == 3 ? s_c : s_p)));
      sites[warp - 1][lane] = site_terms(step, lane == 4 ? p.p_hi : p.q_hi);
    }
    if (head == 0 && b == 0)             // the slots no CTA owns
      for (int i = p.B * p.h + (int)threadIdx.x - 32; i < p.red_slots; i += 32 * RW) {
        p.part_p[i] = 0.f; p.part_q[i] = 0.f; p.part_k[i] = 0.f; p.part_v[i] = 0.f; p.part_c[i] = 0.f;
      }
    __syncwarp();
    bool got = mbar_wait(bar(B_CTX), 0, p.wait_ns);
    // ---- STE of the context's quantizer, this thread's part of the row's 64 columns, in place
    float ds_c;
    {
      uint32_t d[4 * PIECE], x[4 * PIECE];
      piece_load<PIECE>(gD, r, part, d);
      piece_load<PIECE>(gX, r, part, x);
      ds_c = ste_pairs<4 * PIECE>(x, [&](int j) { return unpack2(d[j]); }, s_c, p.q_hi, sites[warp - 1][3]);
      piece_store<PIECE>(gD, r, part, x);                 // (bf16 gradients pass or become zero: nothing is rounded again)
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive(bar(B_STE));
    got = mbar_wait(bar(B_A), 0, p.wait_ns) && got;
    tc_fence_after();
    // ---- pass A: P as the forward pass formed it, its codes into the operand tile, STE of its quantizer, row dot product
    const float2 alpha22 = both(alpha2), nmx2 = both(-st.x), inv2 = both(st.y), sv2 = both(s_v), r2 = both(sites[warp - 1][4].r), ns2 = both(-s_p),
                 magic2 = both(ROUND_MAGIC), nmagic2 = both(-ROUND_MAGIC), m1 = both(-1.f);
    const float lim_p = sites[warp - 1][4].lim;
    // one test per warp tells whether anything can be clipped
    const bool clips = !__all_sync(0xffffffffu, probability_bound(st.x, st.y) <= lim_p);
    // this thread's probabilities, one or two chunks of 32; the loops over them stay rolled, the chunks rotate through the registers
    // (the kernel's code is executed once per CTA: with everything unrolled it was 130 KB, and a third of the stalls were
    //  instruction fetches)
    uint32_t pw0[16], pw1[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) pw1[j] = 0u;
    float2 dot2 = both(0.f), dsp2 = both(0.f);
#pragma unroll 1
    for (int i = 0; i < NC; ++i) {
      const int c = part + TPR * i;
#pragma unroll
      for (int j = 0; j < 16; ++j) pw0[j] = pw1[j];
      if (c >= n_chunks) continue;                        // (warp-uniform: TMEM accesses are warp-collective)
      uint32_t cw[16];
      if (c < n_valid) {
        const int ncol = len - c * 32;                    // below 32 only in the last chunk
        {
          uint32_t a[32];
          tmem_ld32(trow + TMEM_S + (uint32_t)(c * 32), a);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float2 t = fma2(acc2(a, j), alpha22, nmx2);
            float2 v = mul2(make_float2(exp2_approx(t.x), exp2_approx(t.y)), inv2);
            if (ncol < 32) { v.x = 2 * j < ncol ? v.x : 0.f; v.y = 2 * j + 1 < ncol ? v.y : 0.f; }
            pw1[j] = pack2(v);
          }
        }
        uint32_t a[32];
        tmem_ld32(trow + TMEM_DP + (uint32_t)(c * 32), a);
        if (!clips) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float2 pv = unpack2(pw1[j]), d = mul2(acc2(a, j), sv2);
            const float2 z0 = mul2(pv, r2), z = fma2(fma2(z0, ns2, pv), r2, z0);
            const float2 q = add2(add2(z, magic2), nmagic2);
            dsp2 = fma2(d, fma2(z, m1, q), dsp2);
            dot2 = fma2(d, pv, dot2);
            cw[j] = pack2(q);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float2 pv = unpack2(pw1[j]);
            float2 d = mul2(acc2(a, j), sv2);
            const float2 z0 = mul2(pv, r2), z = fma2(fma2(z0, ns2, pv), r2, z0);
            const bool in0 = pv.x <= lim_p, in1 = pv.y <= lim_p;
            const float2 q = add2(add2(make_float2(fminf(z.x, p.p_hi), fminf(z.y, p.p_hi)), magic2), nmagic2);
            dsp2 = fma2(d, make_float2(in0 ? q.x - z.x : q.x, in1 ? q.y - z.y : q.y), dsp2);
            d = make_float2(in0 ? d.x : 0.f, in1 ? d.y : 0.f);
            dot2 = fma2(d, pv, dot2);
            cw[j] = pack2(q);
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) pw1[j] = cw[j] = 0u;
      }
      tile_store(gX + (c >> 1) * 16384, r, c & 1, cw);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    mbar_arrive(bar(B_P));
    red_dot[part][r] = dot2.x + dot2.y;
    asm volatile("bar.sync 1, %0;" ::"n"(32 * RW) : "memory");
    float dot = red_dot[0][r] + red_dot[1][r];
    if (TPR == 4) dot += red_dot[2 % TPR][r] + red_dot[3 % TPR][r];
    const float2 ndot2 = both(-dot);
    // ---- pass B: dS = P * (dP - dot), in place of P, held in registers until the dV product has consumed the codes of P
#pragma unroll 1
    for (int i = 0; i < NC; ++i) {
      const int c = part + TPR * i;
      uint32_t (&pw)[16] = NC == 1 ? pw1 : pw0;            // (one chunk: it did not rotate on)
      if (c < n_valid) {
        uint32_t a[32];
        tmem_ld32(trow + TMEM_DP + (uint32_t)(c * 32), a);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 pv = unpack2(pw[j]);
          float2 d = mul2(acc2(a, j), sv2);
          if (clips) d = make_float2(pv.x <= lim_p ? d.x : 0.f, pv.y <= lim_p ? d.y : 0.f);
          pw[j] = pack2(mul2(pv, add2(d, ndot2)));
        }
      }
      if (NC > 1) {
#pragma unroll
        for (int j = 0; j < 16; ++j) { const uint32_t t = pw0[j]; pw0[j] = pw1[j]; pw1[j] = t; }
      }
    }
    const float w_p = warp_sum(dsp2.x + dsp2.y), w_c = warp_sum(ds_c);      // (beside the dV product)
    got = mbar_wait(bar(B_B), 0, p.wait_ns) && got;
    tc_fence_after();
    if (NC == 1) {
      if (part < n_chunks) tile_store(gX + (part >> 1) * 16384, r, part & 1, pw1);
    } else {
      if (part < n_chunks) tile_store(gX, r, part, pw0);
      if (part + 2 < n_chunks) tile_store(gX + 16384, r, part, pw1);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    mbar_arrive(bar(B_S));
    // ---- the three gradients: STE of the Q, K, V quantizers, this thread's part of the 64 head columns, in place in the tile
    // that holds the values before quantization, then one tiled store (rows beyond the sequence are clipped)
    float ds_v = 0.f, ds_q = 0.f, ds_k = 0.f;
#pragma unroll 1
    for (int g = 0; g < 3; ++g) {                          // V, Q, K
      const float step = g == 0 ? s_v : (g == 1 ? s_q : s_k), scale = g == 0 ? s_p : p.inv_sqrt_d * (g == 1 ? s_k : s_q);
      uint8_t* const tile = g == 0 ? gV : (g == 1 ? gD : gK);
      got = mbar_wait(bar(g == 0 ? B_RV : (g == 1 ? B_RQ : B_RK)), 0, p.wait_ns) && got;
      if (g == 1) { got = mbar_wait(bar(B_O), 0, p.wait_ns) && got; tc_fence_after(); }
      uint32_t a[8 * PIECE], x[4 * PIECE];
      const uint32_t at = trow + (uint32_t)((g == 0 ? TMEM_DV : (g == 1 ? TMEM_DQ : TMEM_DK)) + part * 8 * PIECE);
      if constexpr (PIECE == 4) tmem_ld32(at, a); else tmem_ld16(at, a);
      piece_load<PIECE>(tile, r, part, x);
      const float2 sc2 = both(scale);
      float ds = ste_pairs<4 * PIECE>(x, [&](int j) { return mul2(acc2(a, j), sc2); }, step, p.q_hi, sites[warp - 1][g == 0 ? 2 : g - 1]);
      piece_store<PIECE>(tile, r, part, x);
      fence_async_shared();
      asm volatile("bar.sync 1, %0;" ::"n"(32 * RW) : "memory");
      ds = row_ok ? ds : 0.f;
      ds_v = g == 0 ? ds : ds_v; ds_q = g == 1 ? ds : ds_q; ds_k = g == 2 ? ds : ds_k;
      if (threadIdx.x == 32) {
        tma_store_4d(&maps.out, g == 0 ? sV : (g == 1 ? sD : sK), 0, 0, (g == 0 ? 2 * p.h : (g == 1 ? 0 : p.h)) + head, b);
        tma_store_commit();
      }
      tile_col_sums<RW>(tile, p.S, warp - 1, lane, red_col[g]);
    }
    tc_fence_before();
    if (!__all_sync(0xffffffffu, got) && lane == 0) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_MMA);
    // ---- one partial per CTA and site, added in a fixed order
    const float w[5] = {w_p, warp_sum(ds_q), warp_sum(ds_k), warp_sum(ds_v), w_c};
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < 5; ++i) red_part[warp - 1][i] = w[i];
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * RW) : "memory");
    if (warp == 1 && lane < 5) {
      float t = 0.f;
#pragma unroll
      for (int k = 0; k < RW; ++k) t += red_part[k][lane];
      float* dst = lane == 0 ? p.part_p : (lane == 1 ? p.part_q : (lane == 2 ? p.part_k : (lane == 3 ? p.part_v : p.part_c)));
      dst[b * p.h + head] = t;
    }
    if (const int i = (int)threadIdx.x - 32; i < 192) {      // V, Q, K as above
      const int g = i >> 6, plane = g == 0 ? 2 : g - 1;
      p.col_part[((long long)b * 3 + plane) * p.H + head * HD + (i & 63)] = add_col_sums<RW>(red_col[g], i & 63);
    }
    if (threadIdx.x == 32) tma_store_wait_read<0>();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_ALLOC) : "memory");
  }
}

}  // namespace

bool attention_bwd_supported(int S, int head_dim, int dt, int batch_heads) {
  return dt == 1 && head_dim == HD && S % 8 == 0 && S <= 384 && batch_heads <= RED_BLOCKS;
}

int launch_attention_bwd(const AttentionBwd& a, cudaStream_t st) {
  if (a.S > 128) return launch_attention_bwd_long(a, st);
  AttnBwdParams p;
  p.S = a.S; p.h = a.h; p.B = a.B; p.H = a.H;
  p.inv_sqrt_d = 1.f / sqrtf((float)HD);
  p.s_q = a.s_q; p.s_k = a.s_k; p.s_v = a.s_v; p.s_p = a.s_p; p.s_c = a.s_c;
  p.alpha = a.alpha; p.len = a.len; p.stat = a.stat;
  p.q_hi = (float)a.q_hi; p.p_hi = (float)a.p_hi;
  p.part_q = a.part_q; p.part_k = a.part_k; p.part_v = a.part_v; p.part_p = a.part_p; p.part_c = a.part_c;
  p.red_slots = RED_BLOCKS;
  p.col_part = a.col_part;
  p.status = a.status;
  p.wait_ns = g_wait_limit_ns;
  // tensor maps over [tokens, 3H] and [tokens, H] tensors: (64 of a head, S rows, head slots, B)
  AttnBwdMaps m;
  const long long S = a.S;
  auto map = [&](CUtensorMap* out, const void* ptr, int slots) {
    return make_operand_map(out, OperandDesc{ptr, (long long)slots * HD, HD, S * slots * HD, 0}, 2, a.S, HD, slots, a.B, 128, HD);
  };
  int rc = map(&m.codes, a.qkv_codes, 3 * a.h);
  if (rc == GEMM_OK) rc = map(&m.raw, a.qkv, 3 * a.h);
  if (rc == GEMM_OK) rc = map(&m.out, a.dqkv, 3 * a.h);
  if (rc == GEMM_OK) rc = map(&m.dctx, a.dctx, a.h);
  if (rc == GEMM_OK) rc = map(&m.ctx, a.ctx, a.h);
  if (rc != GEMM_OK) return rc;
  const int smem = 1024 + 4 * 16384 + 32768;
  static bool attr_set = false;
  if (!attr_set) {
    if (cudaFuncSetAttribute(attention_bwd_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaFuncSetAttribute(attention_bwd_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
      return GEMM_ERR_CUDA;
    attr_set = true;
  }
  Scope sc("attention_bwd_tcgen05", 10.0 * a.B * a.h * (double)S * S * HD, 1, st);
  const bool alone = a.B * a.h <= 148;              // a CTA per SM
  if (launch_k(alone ? attention_bwd_kernel<16> : attention_bwd_kernel<8>, dim3(a.h, a.B), alone ? 544 : 288, smem, st, m, p) != cudaSuccess) return GEMM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? GEMM_OK : GEMM_ERR_CUDA;
}

}  // namespace mrem
