// Products with few output tiles and a long inner dimension (sm_100a): the CTAs of a cluster share one tile.
//
// A CTA takes operand tiles in at the rate one SM can read (about 0.29 us per 128-byte deep block of a 128 x 64 tile), so a
// product of 216 x 768 x 3072, 24 tiles, spent 17.5 us on a sixth of the chip.  Here `splits` CTAs (a cluster) each run the main
// loop of tc_gemm_kernel over their share of the inner dimension; then every CTA finishes a part of the tile's rows: the others
// leave their accumulators of those rows in their own shared memory (where the operand stages were), the owner adds
// them to its own in rank order (the sum does not depend on which CTA is first) and runs the usual epilogue on the total.
// Integer accumulators are added as integers.  One tile per CTA, whole 32-column chunks only.
#include <cuda.h>

#include "gemm_epi.cuh"

namespace mrem {

using namespace tc;

namespace {

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t peer_address(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t ld_peer(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_own(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }

// MODE as in tc_gemm_kernel: bf16 output with the terms of its bits 0 to 3, fp32 with bit 4; -1: int32 as accumulated.
template <int KIND, int MODE>
__global__ void __maxnreg__(128)
tc_gemm_split_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                     const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_d, const __grid_constant__ TcParams p, int splits) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t tfull_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ __align__(16) float col_terms[EPI_WARPS][2 * COLVEC];

  constexpr bool CODES = MODE >= 0 && (MODE & 32) != 0;
  __shared__ float2 code_terms[CODES ? EPI_WARPS : 1][3];
  constexpr int OUT = MODE < 0 ? OUT_I32 : (MODE & 16 ? OUT_F32 : OUT_BF16);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int rank = (int)cluster_rank();
  const TileCoord t = decode_tile(p, blockIdx.x / splits);
  const int kb0 = p.k_blocks * rank / splits, kb1 = p.k_blocks * (rank + 1) / splits;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.num_stages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&tfull_bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(p.block_n)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  auto load_b = [&](int kb, int stage) {
    const uint32_t bar = smem_u32(&full_bar[stage]), sb = tiles_base + stage * p.stage_bytes + A_STAGE_BYTES;
    const int k0 = kb * p.block_k;
    if (!p.b_mn) tma_load_4d(sb, &map_b, bar, k0, t.n0, t.b0, t.b1);
    else if (p.b_mn == 2) tma_load_5d(sb, &map_b, bar, 0, k0, t.n0 >> 6, t.b0, t.b1);
    else for (int j = 0; j < p.block_n / 64; ++j) tma_load_4d(sb + j * 8192, &map_b, bar, t.n0 + 64 * j, k0, t.b0, t.b1);
  };
  const int prefetched = p.b_static ? min(kb1 - kb0, p.num_stages) : 0;      // see tc_gemm_kernel
  if (threadIdx.x == 0) {
    for (int i = 0; i < prefetched; ++i) {
      mbar_expect_tx(smem_u32(&full_bar[i]), (uint32_t)p.stage_bytes);
      load_b(kb0 + i, i);
    }
  }
  pdl_wait();
  const uint32_t tmem_d = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  volatile int* vabort = &abort_flag;

  // rows of quadrant q (32 of them) are finished by CTA q * splits / 4 of the cluster
  const int quad = warp & 3, half = (warp - 2) >> 2, owner = quad * splits / 4;
  const int chunks = p.block_n >> 6;                       // 32-column chunks per epilogue warp
  const Epilogue& e = p.epi;
  // the partials' place: per (quadrant, half, chunk) 32 columns x 32 rows of 4 bytes, a row per lane
  const uint32_t part = tiles_base + (uint32_t)((quad * 2 + half) * chunks) * 4096u + 4u * (uint32_t)lane;
  float alpha = e.alpha_const, rb = 0.f;
  float* const cv = col_terms[warp < 2 ? 0 : warp - 2];
  const int row = t.m0 + quad * 32 + lane, c_begin = half * 32 * chunks, col_begin = t.n0 + c_begin;
  const bool row_ok = row < p.M;
  const long long row_off = (long long)t.b0 * e.c_b0 + (long long)t.b1 * e.c_b1 + (long long)row * e.ldc;
  const int nfull = col_begin < p.N ? min((p.N - col_begin) >> 5, chunks) : 0;
  bool got = true;

  if (warp == 0) {
    const bool leader = elect_one();     // see tc_gemm_kernel
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait_warp(smem_u32(&empty_bar[stage]), phase ^ 1u, vabort, p.wait_ns)) {
        if (leader && !*vabort) fail(p, DEV_TIMEOUT_MMA, vabort);
        ok = false;
        break;
      }
      if (leader) {
        const uint32_t bar = smem_u32(&full_bar[stage]), sa = tiles_base + stage * p.stage_bytes;
        const bool b_done = kb - kb0 < prefetched;
        if (!b_done) mbar_expect_tx(bar, (uint32_t)p.stage_bytes);
        const int k0 = kb * p.block_k;
        if (!p.a_mn) tma_load_4d(sa, &map_a, bar, k0, t.m0, t.b0, t.b1);
        else if (p.a_mn == 2) tma_load_5d(sa, &map_a, bar, 0, k0, t.m0 >> 6, t.b0, t.b1);
        else for (int j = 0; j < BLOCK_M / 64; ++j) tma_load_4d(sa + j * 8192, &map_a, bar, t.m0 + 64 * j, k0, t.b0, t.b1);
        if (!b_done) load_b(kb, stage);
      }
      __syncwarp();
      if (++stage == p.num_stages) { stage = 0; phase ^= 1u; }
    }
    if (leader) {
      pdl_trigger();
      if (!ok) {
        // let the copies already in flight land before the CTA may exit
        for (int s = 0; s < p.num_stages; ++s) {
          const unsigned long long t0 = global_ns();
          while (global_ns() - t0 < 1000000ull) { }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    const bool leader = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    const uint32_t adv_a = (p.a_mn ? 2048u : 32u) >> 4, adv_b = (p.b_mn ? 2048u : 32u) >> 4;
    const uint64_t proto_a = smem_desc(tiles_base, p.a_mn ? 8192u : 16u, 1024u);
    const uint64_t proto_b = smem_desc(tiles_base + A_STAGE_BYTES, p.b_mn ? 8192u : 16u, 1024u);
    const uint32_t a_hi = (uint32_t)(proto_a >> 32), b_hi = (uint32_t)(proto_b >> 32), stage_adv = (uint32_t)p.stage_bytes >> 4;
    uint32_t a_lo = (uint32_t)proto_a, b_lo = (uint32_t)proto_b;
    bool ok = true;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait_warp(smem_u32(&full_bar[stage]), phase, vabort, p.wait_ns)) {
        if (leader && !*vabort) fail(p, DEV_TIMEOUT_TMA, vabort);
        ok = false;
        break;
      }
      tc_fence_after();
      if (leader) {
        tc_mma_lohi<KIND>(tmem_d, a_lo, a_hi, b_lo, b_hi, p.idesc, (uint32_t)(kb != kb0));
        tc_mma_lohi<KIND>(tmem_d, a_lo + adv_a, a_hi, b_lo + adv_b, b_hi, p.idesc, 1u);
        tc_mma_lohi<KIND>(tmem_d, a_lo + 2 * adv_a, a_hi, b_lo + 2 * adv_b, b_hi, p.idesc, 1u);
        tc_mma_lohi<KIND>(tmem_d, a_lo + 3 * adv_a, a_hi, b_lo + 3 * adv_b, b_hi, p.idesc, 1u);
        tc_commit(smem_u32(&empty_bar[stage]));
      }
      __syncwarp();
      a_lo += stage_adv; b_lo += stage_adv;
      if (++stage == p.num_stages) { stage = 0; phase ^= 1u; a_lo = (uint32_t)proto_a; b_lo = (uint32_t)proto_b; }
    }
    if (ok && leader) tc_commit(smem_u32(&tfull_bar));
    __syncwarp();
  } else {
    if (e.alpha_p0) alpha *= *e.alpha_p0;
    if (e.alpha_p1) alpha *= *e.alpha_p1;
    if (owner == rank) {
      if (row_ok) rb = row_term(e, row);
      if (nfull > 0) stage_col_terms<MODE>(e, cv, alpha, col_begin, 32 * chunks, p.N, lane);
      if constexpr (CODES) stage_code_terms(e, code_terms[warp - 2], lane);
    }
    got = mbar_wait_or_abort(smem_u32(&tfull_bar), 0u, vabort, p.wait_ns);
    got = __all_sync(0xffffffffu, got);
    if (!got && lane == 0 && !*vabort) fail(p, DEV_TIMEOUT_MMA, vabort);
    tc_fence_after();
    if (got && owner != rank) {
#pragma unroll 1
      for (int c = 0; c < nfull; ++c) {
        uint32_t acc[32];
        tmem_ld32(tmem_d + ((uint32_t)(quad * 32) << 16) + (uint32_t)(c_begin + 32 * c), acc);
#pragma unroll
        for (int j = 0; j < 32; ++j) st_own(part + 4096u * c + 128u * j, acc[j]);
      }
    }
  }
  cluster_arrive();                                        // every CTA's partials are in its shared memory (or it has given up)
  cluster_wait();
  if (warp >= 2 && got && owner == rank) {
    StoreCtx sx{p.c_tma ? &map_c : nullptr, tiles_base + (uint32_t)(p.num_stages * p.stage_bytes) + (uint32_t)((warp - 2) * OUT_BOX_BYTES),
                t.m0 + quad * 32, t.b0, t.b1, lane, &map_d, code_terms[CODES ? warp - 2 : 0]};
#pragma unroll 1
    for (int c = 0; c < nfull; ++c) {
      uint32_t own[32], acc[32], res[16];
      tmem_ld32_issue(tmem_d + ((uint32_t)(quad * 32) << 16) + (uint32_t)(c_begin + 32 * c), own);
      if (OUT == OUT_BF16 && EpiFlags<MODE>(e).res) fetch_res_bf16(e, row_off + col_begin + 32 * c, row_ok, res);
      tmem_ld_wait();
      tmem_ld_pin(own);
#pragma unroll
      for (int j = 0; j < 32; ++j) acc[j] = 0u;
#pragma unroll 1
      for (int r = 0; r < splits; ++r) {
        const uint32_t from = peer_address(part + 4096u * c, (uint32_t)r);
        uint32_t v[32];
        if (r == rank) {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = own[j];
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = ld_peer(from + 128u * j);
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = KIND == 1 ? acc[j] + v[j] : __float_as_uint(__uint_as_float(acc[j]) + __uint_as_float(v[j]));
      }
      finish_chunk<KIND, OUT, OUT == OUT_I32 ? 0 : MODE>(e, acc, res, alpha, rb, cv + 32 * c, row_off + col_begin + 32 * c, row_ok, sx, col_begin + 32 * c);
    }
    if (p.c_tma && lane == 0) tma_store_wait_read<0>();
    __syncwarp();
  }
  tc_fence_before();
  cluster_arrive();                                        // no CTA leaves while another one reads its partials
  cluster_wait();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(p.block_n) : "memory");
  }
}

typedef void (*SplitKern)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const TcParams, int);
const struct { int kind, mode; SplitKern fn; } kVariants[] = {
    {0, 0, tc_gemm_split_kernel<0, 0>}, {0, 2, tc_gemm_split_kernel<0, 2>}, {0, 6, tc_gemm_split_kernel<0, 6>},
    {0, 10, tc_gemm_split_kernel<0, 10>}, {0, 16, tc_gemm_split_kernel<0, 16>}, {1, -1, tc_gemm_split_kernel<1, -1>}, {1, 1, tc_gemm_split_kernel<1, 1>}, {1, 3, tc_gemm_split_kernel<1, 3>}, {1, 7, tc_gemm_split_kernel<1, 7>}, {1, 35, tc_gemm_split_kernel<1, 35>}};
constexpr int kNumVariants = sizeof(kVariants) / sizeof(kVariants[0]);
constexpr int SPLIT_STAGES = 6;                          // one fewer where a second box per epilogue warp holds codes

int variant_of(int kind, const Epilogue& e) {
  const int mode = epilogue_mode(kind, e);
  if (mode < 0 && e.out_kind != OUT_I32) return -1;
  for (int i = 0; i < kNumVariants; ++i)
    if (kVariants[i].kind == kind && kVariants[i].mode == mode) return i;
  return -1;
}
int split_smem(int block_n, bool codes) {
  return (SPLIT_STAGES - codes) * (A_STAGE_BYTES + block_n * 128) + 1024 + EPI_WARPS * OUT_BOX_BYTES * (1 + codes);
}

}  // namespace

// an output and terms that are compiled, rows and column vectors on the boundaries of the vector path
bool tc_gemm_split_eligible(int kind, const GemmShape& g, const Epilogue& e) {
  auto al = [](const void* p, uintptr_t n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1)) == 0; };
  return variant_of(kind, e) >= 0 && g.N % 32 == 0 && e.ldc % 16 == 0 && e.c_b0 % 16 == 0 && e.c_b1 % 16 == 0 && al(e.out, 32) && al(e.residual, 32) &&
         al(e.col_scale, 16) && al(e.col_bias, 16);
}

int tc_gemm_split_launch(int kind, const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mc, const CUtensorMap& md, const TcParams& params, int splits,
                         cudaStream_t stream) {
  const int vi = variant_of(kind, params.epi);
  if (vi < 0) return GEMM_ERR_ARG;
  TcParams p = params;
  const bool codes = p.epi.codes != nullptr;
  p.num_stages = SPLIT_STAGES - codes;
  static bool attr_set[kNumVariants] = {};
  if (!attr_set[vi]) {
    if (cudaFuncSetAttribute(kVariants[vi].fn, cudaFuncAttributeMaxDynamicSharedMemorySize, split_smem(128, codes)) != cudaSuccess) return GEMM_ERR_CUDA;
    attr_set[vi] = true;
  }
  if (launch_cluster(kVariants[vi].fn, p.num_tiles * splits, GEMM_THREADS, split_smem(p.block_n, codes), stream, splits, ma, mb, mc, md, p, splits) != cudaSuccess)
    return GEMM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? GEMM_OK : GEMM_ERR_CUDA;
}

}  // namespace mrem
