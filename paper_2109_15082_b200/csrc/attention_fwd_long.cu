// Fused attention forward for 129 to 384 tokens (head size 64): one (batch, head, 128-query block) per CTA, the keys in chunks of 64.
//   pass 1: S = Q K^T of a chunk (tcgen05, fp32 accumulators in TMEM), its maximum and sum of exponentials joined to the row's
//   pass 2: S of the chunk again, probabilities with the row's maximum and sum, (student) Eq. 1 on them, ctx += P V
// Same operands, outputs and arithmetic on a score as attention_fwd.cu; only the sum over a row is taken chunk by chunk (a chunk with
// a new maximum rescales what has been added up so far).  All waits are time-bounded.
//
// What bounds it: about 4 + 7 (teacher) or 4 + 11 issue slots a score, of which two exponentials (16 a clock and SM).  Whole rows of
// scores in TMEM (the kernel before: 384 of 512 columns, P behind them in shared memory) leave room for one CTA per SM, whose warps
// all wait for the same loads, products and barriers: 0.32 of the issue slots used.  Forming the scores twice costs the idle tensor
// pipe 260 clocks a chunk and buys a CTA of 192 TMEM columns and at most 105 KB, so that two share an SM, and within a CTA the product of a chunk
// runs beside the arithmetic of the one before (two score buffers, given back as soon as they have been read).
// Then: fewer issue slots a score (one pass for maximum and sum, three-input maxima, no tests of keys but in a row's last chunk), the
// context out by tiled stores, long sequences first.  Inside the step of 16 x 384 tokens, hidden 1024: 68 -> 47 us (student), 52 -> 39 (teacher).
// A CTA there takes 13.7 us (stamps): 3 until its first scores, 3 in pass 1, 5 in pass 2, 2 for the context; 5.2 CTAs per SM.
// Shared memory: Q, all keys, a ring of three 64-row pieces of V, the operand tile of one chunk's P.  TMEM: scores 2 x 64, context 64.
#include "attention_fwd.cuh"

namespace mrem {

using namespace attf;

namespace {

constexpr int LONG_THREADS = 288;         // warp 0: TMA + MMA issue; warps 1..8: two threads per query row, 32 of a chunk's 64 keys each
constexpr int LONG_ROUND = 2 * 148;       // CTAs that run at the same time: more take the sequences longest first
constexpr int TMEM_O = 128, TMEM_ALLOC = 256, V_SLOTS = 3;

template <bool QUANT>
__global__ void __launch_bounds__(LONG_THREADS, 2) attention_fwd_long_kernel(const __grid_constant__ CUtensorMap map_qkv, const __grid_constant__ CUtensorMap map_v,
                                                                             const __grid_constant__ CtxMaps out, const __grid_constant__ AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  enum { B_K0, B_K1, B_K2, B_V0, B_V1, B_V2, B_S0, B_S1, B_F0, B_F1, B_P, B_PV, N_BARS };   // F: score buffer read, P: chunk of P written
  __shared__ __align__(8) uint64_t bars[N_BARS];
  __shared__ uint32_t tmem_slot;
  __shared__ float2 red[2][128];                             // [half][row]: maximum, sum
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qb = blockIdx.x, head = blockIdx.y, q0 = qb * 128;
  const int n_box = (p.S + 127) / 128;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = base, sP = sQ + 16384, sK = sP + 16384, sV = sK + n_box * 16384;
  uint8_t* const gP = smem_raw + (sP - smem_u32(smem_raw));
  auto bar = [&](int i) { return smem_u32(&bars[i]); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < N_BARS; ++i) mbar_init(bar(i), (i == B_F0 || i == B_F1 || i == B_P) ? 8 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TMEM_ALLOC) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  const Sequence sq = p.order ? longest_first(p.valid_len, p.B, (int)blockIdx.z) : Sequence{(int)blockIdx.z, p.valid_len ? p.valid_len[blockIdx.z] : p.S};
  const int b = sq.b;
  int len = sq.len;
  len = len < 1 ? 1 : (len > p.S ? p.S : len);
  const int n = (len + 63) / 64;                             // chunks with a valid key

  if (warp == 0) {
    if (lane == 0) {
      auto load_v = [&](int c) {
        mbar_expect_tx(bar(B_V0 + c % V_SLOTS), 8192u);
        tma_load_4d(sV + (uint32_t)(c % V_SLOTS) * 8192u, &map_v, bar(B_V0 + c % V_SLOTS), 0, c * 64, 2 * p.h + head, b);
      };
      mbar_expect_tx(bar(B_K0), 2u * 16384u);
      tma_load_4d(sQ, &map_qkv, bar(B_K0), 0, q0, head, b);
      tma_load_4d(sK, &map_qkv, bar(B_K0), 0, 0, p.h + head, b);
      const int boxes = (len + 127) / 128;
#pragma unroll 1
      for (int i = 1; i < boxes; ++i) {
        mbar_expect_tx(bar(B_K0 + i), 16384u);
        tma_load_4d(sK + i * 16384, &map_qkv, bar(B_K0 + i), 0, i * 128, p.h + head, b);
      }
#pragma unroll 1
      for (int c = 0; c < min(n, V_SLOTS); ++c) load_v(c);
      const uint32_t f32 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 17) | (8u << 24);      // 128 x 64
      int code = 0;                                          // what the first wait that ran out was waiting for
      auto wait = [&](int i, int round, int what) {
        if (code == 0 && !mbar_wait(bar(i), (uint32_t)(round & 1), p.wait_ns)) { code = what; atomicCAS(p.status, 0, what); }
      };
#pragma unroll 1
      for (int s = 0; s <= 2 * n; ++s) {
        if (s < 2 * n) {                                     // scores of chunk s mod n: [128 x 64] = Q K^T
          const int c = s < n ? s : s - n;
          if (s >= 2) wait(B_F0 + (s & 1), (s >> 1) - 1, DEV_TIMEOUT_EPI);
          if (s < n && (s & 1) == 0) wait(B_K0 + (s >> 1), 0, DEV_TIMEOUT_TMA);
          tc_fence_after();
          if (code == 0)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              tc_mma<0>(tmem + (uint32_t)((s & 1) * 64), smem_desc(sQ + k * 32, 16u, 1024u), smem_desc(sK + c * 8192 + k * 32, 16u, 1024u), f32, (uint32_t)(k != 0));
          tc_commit(bar(B_S0 + (s & 1)));
        }
        if (s > n) {                                         // ctx += P V of chunk c  (V is the MN-major operand)
          const int c = s - n - 1, steps = min(4, (len - c * 64 + 15) / 16);
          if (c > 0 && c + 2 < n) {                          // the slot of the chunk before is free once its product has run
            wait(B_PV, c - 1, DEV_TIMEOUT_MMA);
            load_v(c + 2);
          }
          wait(B_V0 + c % V_SLOTS, c / V_SLOTS, DEV_TIMEOUT_TMA);
          wait(B_P, c, DEV_TIMEOUT_EPI);
          tc_fence_after();
          if (code == 0)
#pragma unroll 1
            for (int ks = 0; ks < steps; ++ks)
              tc_mma<0>(tmem + TMEM_O, smem_desc(sP + ks * 32, 16u, 1024u), smem_desc(sV + (uint32_t)(c % V_SLOTS) * 8192u + ks * 2048, 8192u, 1024u),
                        f32 | (1u << 16), (uint32_t)(c > 0 || ks != 0));
          tc_commit(bar(B_PV));
        }
      }
    }
  } else {
    const int quad = warp & 3, half = (warp - 1) >> 2;
    const int r = quad * 32 + lane, q = q0 + r;              // row inside the block, query
    const bool row_ok = q < p.S;
    float alpha = p.alpha_const;
    if (p.a_p0) alpha *= *p.a_p0;
    if (p.a_p1) alpha *= *p.a_p1;
    const float ps = QUANT ? *p.p_step : 1.f;
    // (every scalar here: a load behind the last product would be waited for)
    float calpha = 1.f;
    if (p.c_p0) calpha *= *p.c_p0;
    if (p.c_p1) calpha *= *p.c_p1;
    const float cs = QUANT ? *p.c_step : 1.f;
    const uint32_t trow = tmem + ((uint32_t)(quad * 32) << 16);
    bool got = true;
    auto wait = [&](int i, int round) { got = got && mbar_wait(bar(i), (uint32_t)(round & 1), p.wait_ns); };
    // this thread's 32 scores of step s; the buffer goes back as soon as the warp has read it
    auto fetch = [&](int s, uint32_t* a) {
      wait(B_S0 + (s & 1), s >> 1);
      __syncwarp();
      tc_fence_after();
      tmem_ld32(trow + (uint32_t)((s & 1) * 64 + half * 32), a);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_F0 + (s & 1)));
    };
    const float alpha2 = alpha * 1.4426950408889634f;
    RowPart row{-INFINITY, 0.f};
#pragma unroll 1
    for (int c = 0; c < n; ++c) {
      uint32_t a[32];
      fetch(c, a);
      const int ncol = len - c * 64 - half * 32;             // (>= 32: all keys valid)
      if (ncol > 0) join(row, chunk_part(a, ncol, alpha2), alpha2);
    }
    red[half][r] = make_float2(row.max, row.sum);
    asm volatile("bar.sync 1, 256;" ::: "memory");
    row = RowPart{red[0][r].x, red[0][r].y};
    // (a sequence of up to 32 tokens has no key in the second half of its chunk)
    if (len > 32) join(row, RowPart{red[1][r].x, red[1][r].y}, alpha2);
    const float mx2 = __fmul_rn(alpha2, row.max), sum = row.sum;
    const float inv_sum = __frcp_rn(sum);
    if (p.stats.row && half == 0) {
      if (row_ok) p.stats.row[((long long)b * p.h + head) * p.S + q] = make_float2(mx2, inv_sum);
      if (r == 0 && qb == 0 && head == 0) { p.stats.len[b] = len; if (b == 0) *p.stats.alpha = alpha; }
    }
    const RowScale k{splat(alpha2), make_float2(-mx2, -mx2), make_float2(inv_sum, inv_sum), splat(__frcp_rn(ps)), splat(-ps), p.p_hi};
    const long long prow = (((long long)b * p.h + head) * p.S + q) * p.S;
    const int n_store = p.P ? (p.S + 63) / 64 : n;           // (no P: a pass whose probabilities nobody reads)
#pragma unroll 1
    for (int c = 0; c < n_store; ++c) {
      uint32_t pw[16], cw[16];                               // 32 probabilities / codes packed as bf16 pairs
      const int ncol = len - c * 64 - half * 32;
      if (c < n) {
        uint32_t a[32];
        fetch(n + c, a);
        if (ncol > 0) probabilities32<QUANT>(a, ncol, k, pw, cw);
      }
      if (c >= n || ncol <= 0) {
#pragma unroll
        for (int j = 0; j < 16; ++j) pw[j] = cw[j] = 0u;
      }
      if (c < n) {
        if (c > 0) wait(B_PV, c - 1);                        // the chunk before has been multiplied
        // operand tile: row r, 16-byte piece index XOR (r & 7)  (128-byte swizzle)
        uint8_t* const rowp = gP + r * 128;
#pragma unroll
        for (int t = 0; t < 4; ++t) store16(rowp + ((half * 4 + t) ^ (r & 7)) * 16, cw + 4 * t);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to the MMA
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B_P));
      }
      if (row_ok && p.P) {
        const int left = p.S - c * 64 - half * 32;           // columns of this chunk inside the tensor (S % 8 == 0)
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (t * 8 < left) {
            store16(p.P + prow + c * 64 + half * 32 + t * 8, pw + 4 * t);
            if (QUANT && p.P_qt) store16(p.P_qt + prow + c * 64 + half * 32 + t * 8, cw + 4 * t);
          }
      }
    }
    // ---- context row, 32 columns per thread
    wait(B_PV, n - 1);
    __syncwarp();
    if (!__all_sync(0xffffffffu, got) && lane == 0) atomicCAS(p.status, 0, (int)DEV_TIMEOUT_MMA);
    tc_fence_after();
    // (all products have run: the tiles of Q, K and P are free)
    uint32_t a[32];
    tmem_ld32(trow + (uint32_t)(TMEM_O + half * 32), a);
    if (p.ctx) {
      context_piece<QUANT, 32>(p, a, calpha, cs, r, half, gP - 16384, gP, gP + 16384);
      fence_async_shared();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (threadIdx.x == 32) {
        store_context<QUANT>(out, sQ, sP, sK, q0, head, b);
        tma_store_wait_read<0>();
      }
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_ALLOC) : "memory");
  }
}

template <bool QUANT>
int launch_long(const CUtensorMap& map, const CUtensorMap& map_v, const CtxMaps& out, const AttnParams& p, cudaStream_t st) {
  const int n_box = (p.S + 127) / 128, smem = 1024 + 16384 * (2 + n_box) + 8192 * V_SLOTS;
  static bool attr_set = false;
  if (!attr_set) {
    if (cudaFuncSetAttribute(attention_fwd_long_kernel<QUANT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + 16384 * 5 + 8192 * V_SLOTS) != cudaSuccess)
      return GEMM_ERR_CUDA;
    attr_set = true;
  }
  if (launch_k(attention_fwd_long_kernel<QUANT>, dim3(n_box, p.h, p.B), LONG_THREADS, smem, st, map, map_v, out, p) != cudaSuccess) return GEMM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? GEMM_OK : GEMM_ERR_CUDA;
}

}  // namespace

int attf::launch_attention_fwd_long(const AttnParams& params, const void* qkv, cudaStream_t st) {
  AttnParams p = params;
  p.order = p.valid_len && p.B <= 32 && (p.S + 127) / 128 * p.h * p.B > LONG_ROUND;
  // one tensor, two boxes: (64 of a head, S rows, 3h head slots, B), 128 and 64 rows at a time
  const OperandDesc op{qkv, 3LL * p.H, HD, (long long)p.S * 3 * p.H, 0};
  CUtensorMap map, map_v;
  int rc = make_operand_map(&map, op, 2, p.S, HD, 3 * p.h, p.B, 128, HD);
  if (rc == GEMM_OK) rc = make_operand_map(&map_v, op, 2, p.S, HD, 3 * p.h, p.B, 64, HD);
  CtxMaps out;
  if (rc == GEMM_OK) rc = make_ctx_maps(&out, p, map);
  if (rc != GEMM_OK) return rc;
  return p.p_step ? launch_long<true>(map, map_v, out, p, st) : launch_long<false>(map, map_v, out, p, st);
}

}  // namespace mrem
