// Fused attention backward of the student for 129 to 384 tokens (head size 64), two kernels:
//   attention_bwd_q_kernel   one 128-query block of one head per CTA: STE of the context's quantizer (the masked gradient is
//                            also written for the second kernel), P from the scores, the row sums of dP P, dQ
//   attention_bwd_kv_kernel  one 128-key block of one head per CTA: dK and dV, accumulated in TMEM over the queries in chunks of
//                            64, from TRANSPOSED score tiles (keys in the lanes), so that the codes of P^T and dS^T are
//                            plain K-major operands
// The probabilities are formed again from the codes of Q and K and the forward pass's row statistics in both (bit for bit
// what the forward pass used), so nothing of size seq x seq is ever written: the kernel-per-operation path moves eleven such
// tensors through memory (75 MB each at 16 x 16 x 384 x 384).  The products are far from the limit.
// All waits are time-bounded.
//
// What bounds them: about 14 (queries) and 10 (keys) issue slots a score, and the latency of a CTA's chain of loads, products and row
// arithmetic: two CTAs share an SM (192 and 256 TMEM columns, 97 and 102 KB), and within one the scores of the next chunk are formed as
// soon as the row warps have read this one's.  The query kernel goes over the keys twice in chunks of 64, for the row sums and for dQ,
// and forms scores and dP anew the second time: whole rows of scores in TMEM and probabilities in registers meant one CTA of 544
// threads per SM, 38 issue slots a score for rotating registers and all warps waiting at the same time.  The key kernel starts its loads
// before it fetches the rows' statistics, which it keeps by pairs of queries (two loads a pair instead of four).  Both take long sequences
// first.  16 x 16 heads x 384 x 384 inside the step: 97 -> 56 us and 83 -> 64 us; 11 x 12 heads x 200 28 -> 18 us (queries).
#include "attention_bwd.cuh"

namespace mrem {

using namespace att;

namespace {

struct LongParams {
  int S, h, B;
  int order;                 // blocks take the sequences longest first
  int clustered;             // the CTAs of a head are a cluster and share a slot of the step-size partials (else a slot per CTA)
  float inv_sqrt_d;
  const float *s_q, *s_k, *s_v, *s_p, *s_c;
  const float* alpha;
  const int* len;
  const float2* stat;
  float* dot;                // [B, h, S] row sums of dP P
  float q_hi, p_hi;
  float *part_q, *part_k, *part_v, *part_p, *part_c;
  int red_slots;
  int* status;
  unsigned long long wait_ns;
};

// Step-size partials: a slot per CTA as long as there are that many.  Beyond (more than RED_BLOCKS CTAs) the CTAs of a head form a cluster and
// theirs go to its first CTA.  A CTA may touch another one's shared memory once that one is known to have started: every thread
// arrives on the cluster's barrier after its CTA's set-up and waits on it just before the remote store.  Clusters cost time because a
// cluster starts only where all its CTAs fit at once: 16 x 16 heads x 384 x 384 65 and
// 74 us as clusters, 56 and 64 without.
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void store_remote(float* local, uint32_t rank, float v) {
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_u32(local)), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// ------------------------------------------------------------------ queries
constexpr int Q_THREADS = 288;            // warp 0: TMA + MMA issue; 8 warps, two threads per query row, 32 of a chunk's 64 keys each
constexpr int Q_SLOTS = 3;                // pieces of 64 keys (codes of K | codes of V) in flight
struct QMaps { CUtensorMap codes, codes64, raw, dctx, ctx, dctx_out, out; };

__global__ void __launch_bounds__(Q_THREADS, 2) attention_bwd_q_kernel(const __grid_constant__ QMaps maps, const __grid_constant__ LongParams p) {
  extern __shared__ uint8_t smem_raw[];
  // A: scores and dP of a chunk, FREE: read, S: a chunk of dS written, W: multiplied
  enum { B_CTX, B_Q, B_F0, B_F1, B_F2, B_STE, B_A, B_FREE, B_S, B_W, B_RAW, N_BARS };
  __shared__ __align__(8) uint64_t bars[N_BARS];
  __shared__ uint32_t tmem_slot;
  __shared__ float red_dot[2][128];
  __shared__ float red_part[8][3];
  __shared__ SiteTerms sites[8][3];                        // per warp: Q, context, P (attention_bwd.cuh)
  __shared__ float cta_part[3][3];                         // [cluster rank][site]
  constexpr int TMEM_S = 0, TMEM_DP = 64, TMEM_DQ = 128;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qb = blockIdx.x, head = blockIdx.y, q0 = qb * 128;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  // X: the context, then a chunk of dS; the last slot of the ring: Q before quantization, then dQ
  const uint32_t sQ = base, sD = sQ + 16384, sX = sD + 16384, sC = sX + 16384;
  uint8_t* const g0 = smem_raw + (base - smem_u32(smem_raw));
  uint8_t *const gD = g0 + (sD - base), *const gX = g0 + (sX - base), *const gC = g0 + (sC - base);
  auto bar = [&](int i) { return smem_u32(&bars[i]); };
  if (threadIdx.x == 0) {
    for (int i = 0; i < N_BARS; ++i) mbar_init(bar(i), (i == B_STE || i == B_FREE || i == B_S) ? 8 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(256) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (p.clustered) cluster_arrive();                       // (see store_remote)
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  const Sequence sq = p.order ? longest_first(p.len, p.B, (int)blockIdx.z) : Sequence{(int)blockIdx.z, p.len[blockIdx.z]};
  const int b = sq.b, len = sq.len, n = (len + 63) / 64, raw_slot = 2 * n % Q_SLOTS;       // chunks with a valid key; steps: twice as many
  float share = 0.f;                                       // this CTA's step-size partials, one per lane of warp 1

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(bar(B_CTX), 2u * 16384u);
      tma_load_4d(sD, &maps.dctx, bar(B_CTX), 0, q0, head, b);
      tma_load_4d(sX, &maps.ctx, bar(B_CTX), 0, q0, head, b);
      mbar_expect_tx(bar(B_Q), 16384u);
      tma_load_4d(sQ, &maps.codes, bar(B_Q), 0, q0, head, b);
      auto load = [&](int s) {                             // of step s; behind the last one Q before quantization
        const uint32_t dst = sC + (uint32_t)(s % Q_SLOTS) * 16384u;
        if (s < 2 * n) {
          const uint32_t fb = bar(B_F0 + s % Q_SLOTS);
          const int k0 = (s < n ? s : s - n) * 64;
          mbar_expect_tx(fb, 16384u);
          tma_load_4d(dst, &maps.codes64, fb, 0, k0, p.h + head, b);
          tma_load_4d(dst + 8192, &maps.codes64, fb, 0, k0, 2 * p.h + head, b);
        } else {
          mbar_expect_tx(bar(B_RAW), 16384u);
          tma_load_4d(dst, &maps.raw, bar(B_RAW), 0, q0, head, b);
        }
      };
#pragma unroll 1
      for (int s = 0; s < Q_SLOTS && s <= 2 * n; ++s) load(s);
      const uint32_t f32 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 17) | (8u << 24);      // 128 x 64
      int code = 0;                                        // what the first wait that ran out was waiting for
      auto wait = [&](int i, int round, int what) {
        if (code == 0 && !mbar_wait(bar(i), (uint32_t)(round & 1), p.wait_ns)) { code = what; atomicCAS(p.status, 0, what); }
      };
      wait(B_Q, 0, DEV_TIMEOUT_TMA);
#pragma unroll 1
      for (int s = 0; s <= 2 * n; ++s) {
        if (s < 2 * n) {                                   // S = Q_q K_q^T and dP_hat = dctx V_q^T of a chunk: [128 queries x 64 keys]
          const uint32_t k = sC + (uint32_t)(s % Q_SLOTS) * 16384u;
          if (s > 0) wait(B_FREE, s - 1, DEV_TIMEOUT_EPI);
          wait(B_F0 + s % Q_SLOTS, s / Q_SLOTS, DEV_TIMEOUT_TMA);
          tc_fence_after();
          if (code == 0)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              tc_mma<0>(tmem + TMEM_S, smem_desc(sQ + i * 32, 16u, 1024u), smem_desc(k + i * 32, 16u, 1024u), f32, (uint32_t)(i != 0));
          if (s == 0) {
            wait(B_STE, 0, DEV_TIMEOUT_EPI);
            tc_fence_after();
            if (code == 0) tma_store_4d(&maps.dctx_out, sD, 0, q0, head, b);      // the masked context gradient, for the key kernel
            tma_store_commit();
          }
          if (code == 0)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              tc_mma<0>(tmem + TMEM_DP, smem_desc(sD + i * 32, 16u, 1024u), smem_desc(k + 8192 + i * 32, 16u, 1024u), f32, (uint32_t)(i != 0));
          tc_commit(bar(B_A));
        }
        if (s > n) {                                       // dQ_hat [q x d] += dS [q x 64 keys] * K_q [keys x d] of the step before
          const int c = s - 1 - n, steps = min(4, (len - c * 64 + 15) / 16);
          const uint32_t k = sC + (uint32_t)((s - 1) % Q_SLOTS) * 16384u;
          wait(B_S, c, DEV_TIMEOUT_EPI);
          tc_fence_after();
          if (code == 0)
#pragma unroll 1
            for (int ks = 0; ks < steps; ++ks)
              tc_mma<0>(tmem + TMEM_DQ, smem_desc(sX + ks * 32, 16u, 1024u), smem_desc(k + ks * 2048, 8192u, 1024u), f32 | (1u << 16), (uint32_t)(c > 0 || ks != 0));
          tc_commit(bar(B_W));
        }
        if (s > 0 && s + 2 >= Q_SLOTS && s + 2 <= 2 * n) { // the slot of the step before is free once its products have run
          if (s > n) wait(B_W, s - 1 - n, DEV_TIMEOUT_MMA);
          load(s + 2);
        }
      }
      tma_store_wait_read<0>();
    }
  } else {
    const int quad = warp & 3, half = (warp - 1) >> 2;
    const int r = quad * 32 + lane, q = q0 + r;
    const bool row_ok = q < p.S;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 32);
    const float s_p = *p.s_p, s_v = *p.s_v, s_q = *p.s_q, s_k = *p.s_k, s_c = *p.s_c;
    const long long srow = ((long long)b * p.h + head) * p.S + q;
    float2 st = make_float2(0.f, 0.f);                     // rows beyond the sequence: P = 0
    if (row_ok) st = p.stat[srow];
    const float alpha2 = *p.alpha * 1.4426950408889634f;
    bool got = true;
    auto wait = [&](int i, int round) { got = got && mbar_wait(bar(i), (uint32_t)(round & 1), p.wait_ns); __syncwarp(); };
    auto signal = [&](int i) { __syncwarp(); if (lane == 0) mbar_arrive(bar(i)); };
    if (lane < 3) sites[warp - 1][lane] = site_terms(lane == 0 ? s_q : (lane == 1 ? s_c : s_p), lane == 2 ? p.p_hi : p.q_hi);
    wait(B_CTX, 0);
    float ds_c, ds_q;
    {                                                      // STE of the context's quantizer, 32 columns per thread, in place
      uint32_t d[16], x[16];
      tile_load(gD, r, half, d);
      tile_load(gX, r, half, x);
      ds_c = ste32(x, [&](int j) { return unpack2(d[j]); }, s_c, p.q_hi, sites[warp - 1][1]);
      tile_store(gD, r, half, x);
    }
    fence_async_shared();
    signal(B_STE);
    const float2 alpha22 = both(alpha2), nmx2 = both(-st.x), inv2 = both(st.y), sv2 = both(s_v), r2 = both(sites[warp - 1][2].r), ns2 = both(-s_p),
                 magic2 = both(ROUND_MAGIC), nmagic2 = both(-ROUND_MAGIC), m1 = both(-1.f);
    const float lim_p = sites[warp - 1][2].lim;
    const bool clips = !__all_sync(0xffffffffu, probability_bound(st.x, st.y) <= lim_p);   // (see attention_bwd.cu)
    // this thread's 32 probabilities of step s, as the forward pass formed them, and dP beside them; the accumulators go back
    // as soon as the warp has read them
    auto fetch = [&](int s, int ncol, uint32_t* pw, uint32_t* a) {
      wait(B_A, s);
      tc_fence_after();
      tmem_ld32(trow + TMEM_S, a);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 t = fma2(acc2(a, j), alpha22, nmx2);
        pw[j] = pack2(mul2(make_float2(exp2_approx(t.x), exp2_approx(t.y)), inv2));
      }
      if (ncol < 32) {                                     // (a row's last chunk only)
#pragma unroll
        for (int j = 0; j < 16; ++j) pw[j] &= 2 * j + 1 < ncol ? 0xffffffffu : (2 * j < ncol ? 0xffffu : 0u);
      }
      tmem_ld32(trow + TMEM_DP, a);
      tc_fence_before();
      signal(B_FREE);
    };
    // ---- pass 1: STE of P's quantizer and the row sums of dP P
    float2 dot2[2] = {both(0.f), both(0.f)}, dsp2[2] = {both(0.f), both(0.f)};
#pragma unroll 1
    for (int c = 0; c < n; ++c) {
      const int ncol = len - c * 64 - half * 32;
      uint32_t pw[16], a[32];
      fetch(c, ncol, pw, a);
      if (ncol <= 0) continue;
      if (!clips) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 pv = unpack2(pw[j]), d = mul2(acc2(a, j), sv2);
          const float2 z0 = mul2(pv, r2), z = fma2(fma2(z0, ns2, pv), r2, z0);
          const float2 qv = add2(add2(z, magic2), nmagic2);
          dsp2[j & 1] = fma2(d, fma2(z, m1, qv), dsp2[j & 1]);
          dot2[j & 1] = fma2(d, pv, dot2[j & 1]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 pv = unpack2(pw[j]);
          float2 d = mul2(acc2(a, j), sv2);
          const float2 z0 = mul2(pv, r2), z = fma2(fma2(z0, ns2, pv), r2, z0);
          const bool in0 = pv.x <= lim_p, in1 = pv.y <= lim_p;
          const float2 qv = add2(add2(make_float2(fminf(z.x, p.p_hi), fminf(z.y, p.p_hi)), magic2), nmagic2);
          dsp2[j & 1] = fma2(d, make_float2(in0 ? qv.x - z.x : qv.x, in1 ? qv.y - z.y : qv.y), dsp2[j & 1]);
          d = make_float2(in0 ? d.x : 0.f, in1 ? d.y : 0.f);
          dot2[j & 1] = fma2(d, pv, dot2[j & 1]);
        }
      }
    }
    red_dot[half][r] = (dot2[0].x + dot2[0].y) + (dot2[1].x + dot2[1].y);
    asm volatile("bar.sync 1, 256;" ::: "memory");
    const float dot = red_dot[0][r] + red_dot[1][r];
    if (half == 0 && row_ok) p.dot[srow] = dot;
    const float2 ndot2 = both(-dot);
    // ---- pass 2: dS = P * (dP - dot), chunk by chunk into the operand tile (the context, there before, has been read)
#pragma unroll 1
    for (int c = 0; c < n; ++c) {
      const int ncol = len - c * 64 - half * 32;
      uint32_t pw[16], a[32];
      fetch(n + c, ncol, pw, a);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 pv = unpack2(pw[j]);
        float2 d = mul2(acc2(a, j), sv2);
        if (clips) d = make_float2(pv.x <= lim_p ? d.x : 0.f, pv.y <= lim_p ? d.y : 0.f);
        pw[j] = pack2(mul2(pv, add2(d, ndot2)));
      }
      if (c > 0) wait(B_W, c - 1);                         // the chunk before has been multiplied
      tile_store(gX, r, half, pw);
      fence_async_shared();
      signal(B_S);
    }
    // ---- dQ: STE of Q's quantizer, in place in the tile that holds Q before quantization
    wait(B_RAW, 0);
    wait(B_W, n - 1);
    tc_fence_after();
    uint8_t* const gR = gC + raw_slot * 16384;
    {
      uint32_t a[32], x[16];
      tmem_ld32(trow + TMEM_DQ, a);
      tile_load(gR, r, half, x);
      const float2 sc2 = both(p.inv_sqrt_d * s_k);
      ds_q = ste32(x, [&](int j) { return mul2(acc2(a, j), sc2); }, s_q, p.q_hi, sites[warp - 1][0]);
      tile_store(gR, r, half, x);
      if (!row_ok) ds_q = 0.f;
    }
    fence_async_shared();
    tc_fence_before();
    if (!__all_sync(0xffffffffu, got) && lane == 0) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_MMA);
    const float w[3] = {warp_sum((dsp2[0].x + dsp2[0].y) + (dsp2[1].x + dsp2[1].y)), warp_sum(ds_q), warp_sum(ds_c)};
    if (lane == 0) { red_part[warp - 1][0] = w[0]; red_part[warp - 1][1] = w[1]; red_part[warp - 1][2] = w[2]; }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (threadIdx.x == 32) { tma_store_4d(&maps.out, sC + (uint32_t)raw_slot * 16384u, 0, q0, head, b); tma_store_commit(); }
    if (warp == 1 && lane < 3) {
#pragma unroll
      for (int k = 0; k < 8; ++k) share += red_part[k][lane];
    }
    if (threadIdx.x == 32) tma_store_wait_read<0>();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
  }
  int slot = (b * p.h + head) * (int)gridDim.x + qb, n_slots = p.B * p.h * (int)gridDim.x;
  if (p.clustered) {
    cluster_wait();
    if (warp == 1 && lane < 3) store_remote(&cta_part[cluster_rank()][lane], 0, share);
    cluster_arrive();                                      // the share is there
    if (qb > 0) return;                                    // (nobody reads this CTA's shared memory)
    cluster_wait();
    share = 0.f;
    if (warp == 1 && lane < 3)
      for (int k = 0; k < (int)gridDim.x; ++k) share += cta_part[k][lane];
    slot = b * p.h + head;
    n_slots = p.B * p.h;
  }
  if (warp == 1 && lane < 3) (lane == 0 ? p.part_p : (lane == 1 ? p.part_q : p.part_c))[slot] = share;
  if (qb == 0 && head == 0 && blockIdx.z == 0)             // the slots nobody owns
    for (int i = n_slots + (int)threadIdx.x; i < p.red_slots; i += Q_THREADS) { p.part_p[i] = 0.f; p.part_q[i] = 0.f; p.part_c[i] = 0.f; }
}

// ------------------------------------------------------------------ keys and values
constexpr int KV_THREADS = 288;           // warp 0: TMA + MMA issue; 8 warps, two threads per key, 32 of a chunk's 64 queries each
struct KvMaps { CUtensorMap codes, codes64, raw, dctx64, out; };

__global__ void __launch_bounds__(KV_THREADS, 2) attention_bwd_kv_kernel(const __grid_constant__ KvMaps maps, const __grid_constant__ LongParams p) {
  extern __shared__ uint8_t smem_raw[];
  enum { B_KV, B_F0, B_F1, B_A, B_FREE, B_P, B_W, B_RAW, N_BARS };
  __shared__ __align__(8) uint64_t bars[N_BARS];
  __shared__ uint32_t tmem_slot;
  __shared__ float red_part[8][2];
  __shared__ SiteTerms sites[8][2];                        // per warp: V, K (attention_bwd.cuh)
  __shared__ float cta_part[3][2];
  constexpr int TMEM_S = 0, TMEM_DP = 64, TMEM_DV = 128, TMEM_DK = 192;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kb = blockIdx.x, head = blockIdx.y, k0 = kb * 128;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sK = base, sV = sK + 16384, sC = sV + 16384 /* two buffers of Q | dctx chunks */, sP = sC + 32768, sS = sP + 16384;
  uint8_t* const g0 = smem_raw + (base - smem_u32(smem_raw));
  uint8_t *const gK = g0, *const gV = g0 + (sV - base), *const gP = g0 + (sP - base), *const gS = g0 + (sS - base);
  // per pair of queries: -max and 1 / sum, -dot
  float4* const qstat = reinterpret_cast<float4*>(g0 + (sS - base) + 16384);
  float2* const qdot = reinterpret_cast<float2*>(qstat + (p.S + 63) / 64 * 32);
  auto bar = [&](int i) { return smem_u32(&bars[i]); };
  if (threadIdx.x == 0) {
    for (int i = 0; i < N_BARS; ++i) mbar_init(bar(i), i == B_P || i == B_FREE ? 8 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(256) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (p.clustered) cluster_arrive();                       // (see store_remote)
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  const Sequence sq = p.order ? longest_first(p.len, p.B, (int)blockIdx.z) : Sequence{(int)blockIdx.z, p.len[blockIdx.z]};
  const int b = sq.b, len = sq.len, n_q = (p.S + 63) / 64;
  float share = 0.f;                                       // (as in the query kernel)
  const bool active = k0 < len;                            // a block of padded keys has zero gradients
  auto load_chunk = [&](int c) {
    const uint32_t dst = sC + (c & 1) * 16384, fb = bar(B_F0 + (c & 1));
    mbar_expect_tx(fb, 16384u);
    tma_load_4d(dst, &maps.codes64, fb, 0, c * 64, head, b);
    tma_load_4d(dst + 8192, &maps.dctx64, fb, 0, c * 64, head, b);
  };
  if (threadIdx.x == 0 && active) {
    mbar_expect_tx(bar(B_KV), 2u * 16384u);
    tma_load_4d(sK, &maps.codes, bar(B_KV), 0, k0, p.h + head, b);
    tma_load_4d(sV, &maps.codes, bar(B_KV), 0, k0, 2 * p.h + head, b);
    load_chunk(0);
    if (n_q > 1) load_chunk(1);
  }
  const float s_p = *p.s_p, lim_p = range_limit(s_p, p.p_hi);
  bool over = false;
  if (active)
    for (int i = threadIdx.x; i < n_q * 64; i += KV_THREADS) {
      float2 st = make_float2(0.f, 0.f);                   // queries beyond the sequence: P = 0
      float dot = 0.f;
      if (i < p.S) {
        const long long at = ((long long)b * p.h + head) * p.S + i;
        st = p.stat[at];
        dot = p.dot[at];
      }
      over = over || !(probability_bound(-st.x, st.y) <= lim_p);
      float* const v = reinterpret_cast<float*>(qstat + (i >> 1)) + (i & 1);
      v[0] = -st.x;
      v[2] = st.y;
      reinterpret_cast<float*>(qdot)[i] = -dot;
    }
  const bool clips = __syncthreads_or(over);

  if (warp == 0) {
    if (lane == 0 && active) {
      const uint32_t f32 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
      const uint32_t id_s = f32 | (8u << 17), id_g = f32 | (8u << 17) | (1u << 16);     // N = 64; B K-major / MN-major
      bool ok = mbar_wait(bar(B_KV), 0, p.wait_ns);
#pragma unroll 1
      for (int c = 0; c <= n_q; ++c) {
        if (c < n_q) {                                     // S^T and dP^T of chunk c: [128 keys x 64 queries]
          if (c > 0) ok = mbar_wait(bar(B_FREE), (uint32_t)((c - 1) & 1), p.wait_ns) && ok;
          ok = mbar_wait(bar(B_F0 + (c & 1)), (uint32_t)((c >> 1) & 1), p.wait_ns) && ok;
          tc_fence_after();
          const uint32_t q = sC + (c & 1) * 16384, d = q + 8192;
          if (ok)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              tc_mma<0>(tmem + TMEM_S, smem_desc(sK + k * 32, 16u, 1024u), smem_desc(q + k * 32, 16u, 1024u), id_s, (uint32_t)(k != 0));
              tc_mma<0>(tmem + TMEM_DP, smem_desc(sV + k * 32, 16u, 1024u), smem_desc(d + k * 32, 16u, 1024u), id_s, (uint32_t)(k != 0));
            }
          tc_commit(bar(B_A));
        }
        if (c > 0) { ok = mbar_wait(bar(B_P), (uint32_t)((c - 1) & 1), p.wait_ns) && ok; tc_fence_after(); }
        if (c > 0) {                                       // dV += P_q^T dctx, dK += dS^T Q_q of chunk c - 1
          const uint32_t q = sC + ((c - 1) & 1) * 16384, d = q + 8192;
          if (ok)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              tc_mma<0>(tmem + TMEM_DV, smem_desc(sP + ks * 32, 16u, 1024u), smem_desc(d + ks * 2048, 8192u, 1024u), id_g, (uint32_t)(c > 1 || ks != 0));
              tc_mma<0>(tmem + TMEM_DK, smem_desc(sS + ks * 32, 16u, 1024u), smem_desc(q + ks * 2048, 8192u, 1024u), id_g, (uint32_t)(c > 1 || ks != 0));
            }
          tc_commit(bar(B_W));
          if (c + 1 < n_q) {                               // the buffer of chunk c - 1 is free once those products have run
            ok = mbar_wait(bar(B_W), (uint32_t)((c - 1) & 1), p.wait_ns) && ok;
            load_chunk(c + 1);
          }
        }
        if (c == n_q - 1) {                                // the codes of K and V are not needed any more: the values before quantization
          ok = mbar_wait(bar(B_A), (uint32_t)(c & 1), p.wait_ns) && ok;
          mbar_expect_tx(bar(B_RAW), 2u * 16384u);
          tma_load_4d(sV, &maps.raw, bar(B_RAW), 0, k0, 2 * p.h + head, b);
          tma_load_4d(sK, &maps.raw, bar(B_RAW), 0, k0, p.h + head, b);
        }
      }
      if (!ok) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_EPI);
    }
  } else {
    const int quad = warp & 3, half = (warp - 1) >> 2;
    const int r = quad * 32 + lane, key = k0 + r;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    float ds_v = 0.f, ds_k = 0.f;
    if (active) {
      const float s_v = *p.s_v, s_q = *p.s_q, s_k = *p.s_k;
      const float alpha2 = *p.alpha * 1.4426950408889634f;
      const uint32_t keep = key < len ? 0xffffffffu : 0u;
      const float2 alpha22 = both(alpha2), sv2 = both(s_v), r2 = both(__frcp_rn(s_p)), ns2 = both(-s_p), magic2 = both(ROUND_MAGIC),
                   nmagic2 = both(-ROUND_MAGIC);
      if (lane < 2) sites[warp - 1][lane] = site_terms(lane == 0 ? s_v : s_k, p.q_hi);
      __syncwarp();
      bool got = true;
#pragma unroll 1
      for (int c = 0; c < n_q; ++c) {
        got = mbar_wait(bar(B_A), (uint32_t)(c & 1), p.wait_ns) && got;
        __syncwarp();
        tc_fence_after();
        uint32_t pw[16], w[16];
        const float4* const st = qstat + c * 32 + half * 16;
        const float2* const nd = qdot + c * 32 + half * 16;
        uint32_t a[32];
        tmem_ld32(trow + (uint32_t)(TMEM_S + half * 32), a);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float4 s4 = st[j];
          const float2 t = fma2(acc2(a, j), alpha22, make_float2(s4.x, s4.y));
          pw[j] = pack2(mul2(make_float2(exp2_approx(t.x), exp2_approx(t.y)), make_float2(s4.z, s4.w))) & keep;
        }
        tmem_ld32(trow + (uint32_t)(TMEM_DP + half * 32), a);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_FREE));             // the next chunk's scores may come
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 pv = unpack2(pw[j]);
          float2 d = mul2(acc2(a, j), sv2);
          const float2 z0 = mul2(pv, r2);
          float2 z = fma2(fma2(z0, ns2, pv), r2, z0);
          if (clips) {
            d = make_float2(pv.x <= lim_p ? d.x : 0.f, pv.y <= lim_p ? d.y : 0.f);
            z = make_float2(fminf(z.x, p.p_hi), fminf(z.y, p.p_hi));
          }
          w[j] = pack2(mul2(pv, add2(d, nd[j])));
          pw[j] = pack2(add2(add2(z, magic2), nmagic2));
        }
        if (c > 0) {                                       // the products of the chunk before have read the two tiles
          got = mbar_wait(bar(B_W), (uint32_t)((c - 1) & 1), p.wait_ns) && got;
          tc_fence_after();
        }
        tile_store(gP, r, half, pw);
        tile_store(gS, r, half, w);
        fence_async_shared();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_P));
      }
      got = mbar_wait(bar(B_W), (uint32_t)((n_q - 1) & 1), p.wait_ns) && got;
      got = mbar_wait(bar(B_RAW), 0, p.wait_ns) && got;
      tc_fence_after();
#pragma unroll 1
      for (int g = 0; g < 2; ++g) {                        // V, K: in place in the tile that holds the values before quantization
        const float step = g == 0 ? s_v : s_k;
        uint8_t* const tile = g == 0 ? gV : gK;
        uint32_t a[32], x[16];
        tmem_ld32(trow + (uint32_t)((g == 0 ? TMEM_DV : TMEM_DK) + half * 32), a);
        tile_load(tile, r, half, x);
        const float2 sc2 = both(g == 0 ? s_p : p.inv_sqrt_d * s_q);
        float ds = ste32(x, [&](int j) { return mul2(acc2(a, j), sc2); }, step, p.q_hi, sites[warp - 1][g]);
        tile_store(tile, r, half, x);
        ds = key < p.S ? ds : 0.f;
        if (g == 0) ds_v = ds; else ds_k = ds;
      }
      tc_fence_before();
      if (!__all_sync(0xffffffffu, got) && lane == 0) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_MMA);
    } else {
      uint32_t z[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) z[j] = 0u;
      tile_store(gV, r, half, z);
      tile_store(gK, r, half, z);
    }
    fence_async_shared();
    const float w0 = warp_sum(ds_v), w1 = warp_sum(ds_k);
    if (lane == 0) { red_part[warp - 1][0] = w0; red_part[warp - 1][1] = w1; }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    if (threadIdx.x == 32) {
      tma_store_4d(&maps.out, sV, 0, k0, 2 * p.h + head, b);
      tma_store_4d(&maps.out, sK, 0, k0, p.h + head, b);
      tma_store_commit();
    }
    if (warp == 1 && lane < 2) {
#pragma unroll
      for (int k = 0; k < 8; ++k) share += red_part[k][lane];
    }
    if (threadIdx.x == 32) tma_store_wait_read<0>();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
  }
  int slot = (b * p.h + head) * (int)gridDim.x + kb, n_slots = p.B * p.h * (int)gridDim.x;
  if (p.clustered) {
    if (!active) return;                                   // (no shares; the barrier counts the threads that are left)
    cluster_wait();
    if (warp == 1 && lane < 2) store_remote(&cta_part[cluster_rank()][lane], 0, share);
    cluster_arrive();
    if (kb > 0) return;
    cluster_wait();
    share = 0.f;
    if (warp == 1 && lane < 2)
      for (int k = 0; k * 128 < len; ++k) share += cta_part[k][lane];
    slot = b * p.h + head;
    n_slots = p.B * p.h;
  }
  if (warp == 1 && lane < 2) (lane == 0 ? p.part_v : p.part_k)[slot] = share;
  if (kb == 0 && head == 0 && blockIdx.z == 0)
    for (int i = n_slots + (int)threadIdx.x; i < p.red_slots; i += KV_THREADS) { p.part_v[i] = 0.f; p.part_k[i] = 0.f; }
}

}  // namespace

int launch_attention_bwd_long(const AttentionBwd& a, cudaStream_t st) {
  LongParams p;
  p.S = a.S; p.h = a.h; p.B = a.B;
  p.order = a.B <= 32 && (a.S + 127) / 128 * a.h * a.B > 2 * 148;      // more CTAs than run at the same time
  p.inv_sqrt_d = 1.f / sqrtf((float)HD);
  p.s_q = a.s_q; p.s_k = a.s_k; p.s_v = a.s_v; p.s_p = a.s_p; p.s_c = a.s_c;
  p.alpha = a.alpha; p.len = a.len; p.stat = a.stat; p.dot = a.dot;
  p.q_hi = (float)a.q_hi; p.p_hi = (float)a.p_hi;
  p.part_q = a.part_q; p.part_k = a.part_k; p.part_v = a.part_v; p.part_p = a.part_p; p.part_c = a.part_c;
  p.red_slots = RED_BLOCKS;
  p.status = a.status;
  p.wait_ns = g_wait_limit_ns;
  const long long S = a.S;
  auto map = [&](CUtensorMap* out, const void* ptr, int slots, int rows) {     // (64 of a head, S rows, head slots, B)
    return make_operand_map(out, OperandDesc{ptr, (long long)slots * HD, HD, S * slots * HD, 0}, 2, a.S, HD, slots, a.B, rows, HD);
  };
  QMaps mq;
  KvMaps mk;
  int rc = map(&mq.codes, a.qkv_codes, 3 * a.h, 128);
  if (rc == GEMM_OK) rc = map(&mq.raw, a.qkv, 3 * a.h, 128);
  if (rc == GEMM_OK) rc = map(&mq.dctx, a.dctx, a.h, 128);
  if (rc == GEMM_OK) rc = map(&mq.ctx, a.ctx, a.h, 128);
  if (rc == GEMM_OK) rc = map(&mq.dctx_out, a.dctx_masked, a.h, 128);
  if (rc == GEMM_OK) rc = map(&mq.out, a.dqkv, 3 * a.h, 128);
  if (rc == GEMM_OK) rc = map(&mq.codes64, a.qkv_codes, 3 * a.h, 64);
  if (rc == GEMM_OK) rc = map(&mk.dctx64, a.dctx_masked, a.h, 64);
  if (rc != GEMM_OK) return rc;
  mk.codes = mq.codes; mk.codes64 = mq.codes64; mk.raw = mq.raw; mk.out = mq.out;
  const int n_box = (a.S + 127) / 128, n_kb = (a.S + 63) / 64;
  const int smem_q = 1024 + 16384 * (3 + Q_SLOTS), smem_k = 1024 + 6 * 16384 + n_kb * 32 * (int)(sizeof(float4) + sizeof(float2));
  static bool attr_set = false;
  if (!attr_set) {
    if (cudaFuncSetAttribute(attention_bwd_q_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_q) != cudaSuccess ||
        cudaFuncSetAttribute(attention_bwd_kv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + 6 * 16384 + 6 * 32 * 24) != cudaSuccess)
      return GEMM_ERR_CUDA;
    attr_set = true;
  }
  const dim3 grid(n_box, a.h, a.B);
  p.clustered = n_box * a.h * a.B > RED_BLOCKS;
  const int cluster = p.clustered ? n_box : 1;
  Scope sc("attention_bwd_tcgen05", 14.0 * a.B * a.h * (double)S * S * HD, 1, st);
  if (launch_cluster(attention_bwd_q_kernel, grid, Q_THREADS, smem_q, st, cluster, mq, p) != cudaSuccess) return GEMM_ERR_CUDA;
  if (launch_cluster(attention_bwd_kv_kernel, grid, KV_THREADS, smem_k, st, cluster, mk, p) != cudaSuccess) return GEMM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? GEMM_OK : GEMM_ERR_CUDA;
}

}  // namespace mrem
