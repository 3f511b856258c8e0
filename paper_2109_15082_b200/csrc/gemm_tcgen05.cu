// Tensor-core GEMM for sm_100a: C[b][m][n] = epilogue( sum_k A[b][m][k] * B[b][n][k] ).
//
// One persistent CTA per SM.  Warp 0 streams operand tiles into a ring of shared-memory
// stages with TMA (128-byte swizzle), warp 1 issues tcgen05.mma (bf16 -> fp32, or
// int8 -> int32 with exact accumulation) into one of two TMEM accumulator buffers, and
// warps 2..9 drain the other buffer with tcgen05.ld, apply the epilogue (column scale and
// bias staged in shared memory before the accumulator is ready) and write their rows: bf16
// through a 2 KB shared-memory box per warp and tiled stores, anything else straight from
// registers with 32-byte vector stores.  The epilogue of tile i overlaps the main loop of
// tile i+1.
// The student's QKV product also writes the codes of its stored output (MODE bit 5): a quantizer launch between it and the attention
// read 25 MB and wrote 25 at 32 x 128 tokens, hidden 1024, and was 3.5 us of a small step's chain a layer.  Passes timed in turn: 32 x 128,
// hidden 768, forward of both modules 556 -> 547 us; 8 x 256 936 -> 919; 11 x 200 with gradients 356 -> 353; 3 x 72 422.5 -> 419.6; 4 x 32, hidden 128
// 82.4 -> 81.0; beside the teacher's pass with many tokens (32 x 128, two streams) unchanged.
// Either operand may be stored k-contiguous ("K-major") or m/n-contiguous ("MN-major");
// the second form serves the backward products (dX = dY * W_hat, dW = dY^T * X_hat) and
// the attention products without any transposed copy.
//
// Every wait on an mbarrier is bounded in time; when one runs out the kernel records a
// code in the status word, stops issuing work, frees its TMEM and returns.
#include <cuda.h>

#include <cstdio>

#include "gemm_epi.cuh"

namespace mrem {

using namespace tc;

namespace {

// ------------------------------------------------------------------ the kernel
// (Two blocks' worth of registers: a second CTA never fits the shared memory, but 96 registers a thread instead of 168 leave
// room for three blocks of the other stream's row and update kernels beside a product.  8 x 256 tokens, hidden 768: step 1048 ->
// 1037 us; 32 x 128, hidden 1024: 3660 -> 3643.)
template <int KIND, int MODE>
__global__ void __launch_bounds__(GEMM_THREADS, 2)
tc_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_d, const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t tfull_bar[2];
  __shared__ __align__(8) uint64_t tempty_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ __align__(16) float col_terms[EPI_WARPS][2 * COLVEC];
  constexpr bool CODES = MODE >= 0 && (MODE & 32) != 0;
  __shared__ float2 code_terms[CODES ? EPI_WARPS : 1][3];

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.num_stages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&tfull_bar[a]), 1);
      mbar_init(smem_u32(&tempty_bar[a]), EPI_WARPS);
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // A B operand that the preceding kernel does not write (weights): the producer fetches the B tiles of its first
  // stages now, while that kernel is still finishing; the matching A tiles follow after the wait.
  const int prefetched = p.b_static && (int)blockIdx.x < p.num_tiles ? (p.k_blocks < p.num_stages ? p.k_blocks : p.num_stages) : 0;
  if (threadIdx.x == 0 && prefetched > 0) {
    const TileCoord t = decode_tile(p, blockIdx.x);
    for (int kb = 0; kb < prefetched; ++kb) {
      const uint32_t bar = smem_u32(&full_bar[kb]);
      const uint32_t sb = tiles_base + kb * p.stage_bytes + A_STAGE_BYTES;
      mbar_expect_tx(bar, (uint32_t)p.stage_bytes);
      const int k0 = kb * p.block_k;
      if (!p.b_mn) {
        tma_load_4d(sb, &map_b, bar, k0, t.n0, t.b0, t.b1);
      } else if (p.b_mn == 2) {
        tma_load_5d(sb, &map_b, bar, 0, k0, t.n0 >> 6, t.b0, t.b1);
      } else {
        for (int j = 0; j < p.block_n / 64; ++j) tma_load_4d(sb + j * 8192, &map_b, bar, t.n0 + 64 * j, k0, t.b0, t.b1);
      }
    }
  }
  pdl_wait();                            // set-up done; from here on the predecessor's results are needed
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  volatile int* vabort = &abort_flag;

  if (warp == 0) {
    // ---------------- TMA producer: like the issuer, the whole warp walks the loop and one elected lane issues (see elect_one).  Its chain
    // of instructions sets the pace of every tile below 256 columns: 0.287 us per block of the inner dimension whatever the
    // width (0.21 in a copy that loads nothing); from the whole warp 0.276.  2048 x 768 x 3072 17.9 -> 17.3 us, 1500 x 1024 x 4096 22.7 ->
    // 22.4, int8 2200 x 768 x 3072 11.8 -> 11.45.  (Looking at the next stage's barrier before this stage's loads: 0.265, but 256-wide tiles
    // slower; step of 32 x 128 tokens, hidden 1024 3484 -> 3510 us.  The same in the issuer's loop: 1 % slower at every width.)
    const bool leader = elect_one();
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < p.num_tiles && ok; tile += gridDim.x) {
      const TileCoord t = decode_tile(p, tile);
      for (int kb = 0; kb < p.k_blocks; ++kb) {
        if (!mbar_wait_warp(smem_u32(&empty_bar[stage]), phase ^ 1u, vabort, p.wait_ns)) {
          if (leader && !*vabort) fail(p, DEV_TIMEOUT_MMA, vabort);
          ok = false;
          break;
        }
        if (leader) {
          const uint32_t bar = smem_u32(&full_bar[stage]);
          const uint32_t sa = tiles_base + stage * p.stage_bytes, sb = sa + A_STAGE_BYTES;
          const bool b_done = tile == (int)blockIdx.x && kb < prefetched;     // fetched (and announced) before the wait
          if (!b_done) mbar_expect_tx(bar, (uint32_t)p.stage_bytes);
          const int k0 = kb * p.block_k;
          if (!p.a_mn) {
            tma_load_4d(sa, &map_a, bar, k0, t.m0, t.b0, t.b1);
          } else if (p.a_mn == 2) {
            tma_load_5d(sa, &map_a, bar, 0, k0, t.m0 >> 6, t.b0, t.b1);
          } else {
            for (int j = 0; j < BLOCK_M / 64; ++j) tma_load_4d(sa + j * 8192, &map_a, bar, t.m0 + 64 * j, k0, t.b0, t.b1);
          }
          if (b_done) {
          } else if (!p.b_mn) {
            tma_load_4d(sb, &map_b, bar, k0, t.n0, t.b0, t.b1);
          } else if (p.b_mn == 2) {
            tma_load_5d(sb, &map_b, bar, 0, k0, t.n0 >> 6, t.b0, t.b1);
          } else {
            for (int j = 0; j < p.block_n / 64; ++j) tma_load_4d(sb + j * 8192, &map_b, bar, t.n0 + 64 * j, k0, t.b0, t.b1);
          }
        }
        __syncwarp();
        if (++stage == p.num_stages) { stage = 0; phase ^= 1u; }
      }
    }
    if (leader) {
      pdl_trigger();                     // the last tiles are on their way: the next kernel's launch hides behind their products
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
    // ---------------- MMA issuer: the whole warp walks the loop, one elected lane issues (see elect_one)
    const bool leader = elect_one();
    int stage = 0, acc = 0;
    uint32_t phase = 0, acc_phase = 0;
    // descriptor words: high word fixed (stride between 8-row groups, version, 128-byte swizzle); low word =
    // address >> 4 plus the leading-dimension offset field, advanced per 16-deep step and per stage
    const uint32_t adv_a = (p.a_mn ? 2048u : 32u) >> 4, adv_b = (p.b_mn ? 2048u : 32u) >> 4;
    const uint64_t proto_a = smem_desc(tiles_base, p.a_mn ? 8192u : 16u, 1024u);
    const uint64_t proto_b = smem_desc(tiles_base + A_STAGE_BYTES, p.b_mn ? 8192u : 16u, 1024u);
    const uint32_t a_hi = (uint32_t)(proto_a >> 32), b_hi = (uint32_t)(proto_b >> 32);
    const uint32_t a_lo0 = (uint32_t)proto_a, b_lo0 = (uint32_t)proto_b, stage_adv = (uint32_t)p.stage_bytes >> 4;
    uint32_t a_lo = a_lo0, b_lo = b_lo0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < p.num_tiles && ok; tile += gridDim.x) {
      if (!mbar_wait_warp(smem_u32(&tempty_bar[acc]), acc_phase ^ 1u, vabort, p.wait_ns)) {
        if (leader && !*vabort) fail(p, DEV_TIMEOUT_EPI, vabort);
        break;
      }
      tc_fence_after();
      const uint32_t tmem_d = tmem_base + (uint32_t)(acc * p.block_n);
      for (int kb = 0; kb < p.k_blocks; ++kb) {
        if (!mbar_wait_warp(smem_u32(&full_bar[stage]), phase, vabort, p.wait_ns)) {
          if (leader && !*vabort) fail(p, DEV_TIMEOUT_TMA, vabort);
          ok = false;
          break;
        }
        tc_fence_after();
        if (leader) {
          tc_mma_lohi<KIND>(tmem_d, a_lo, a_hi, b_lo, b_hi, p.idesc, (uint32_t)(kb != 0));
          tc_mma_lohi<KIND>(tmem_d, a_lo + adv_a, a_hi, b_lo + adv_b, b_hi, p.idesc, 1u);
          tc_mma_lohi<KIND>(tmem_d, a_lo + 2 * adv_a, a_hi, b_lo + 2 * adv_b, b_hi, p.idesc, 1u);
          tc_mma_lohi<KIND>(tmem_d, a_lo + 3 * adv_a, a_hi, b_lo + 3 * adv_b, b_hi, p.idesc, 1u);
          tc_commit(smem_u32(&empty_bar[stage]));
        }
        __syncwarp();
        a_lo += stage_adv; b_lo += stage_adv;
        if (++stage == p.num_stages) { stage = 0; phase ^= 1u; a_lo = a_lo0; b_lo = b_lo0; }
      }
      if (!ok) break;
      if (leader) tc_commit(smem_u32(&tfull_bar[acc]));
      __syncwarp();
      acc ^= 1;
      if (acc == 0) acc_phase ^= 1u;
    }
  } else {
    // ---------------- epilogue warps: TMEM lane quadrant = warp % 4, two warps per quadrant, each draining
    // its 32 rows over one half of the tile's columns
    const int quad = warp & 3, half = (warp - 2) >> 2;
    const Epilogue& e = p.epi;
    float alpha = e.alpha_const;
    if (e.alpha_p0) alpha *= *e.alpha_p0;
    if (e.alpha_p1) alpha *= *e.alpha_p1;
    const bool direct = direct_epilogue_ok(e);
    const bool res_bf16 = e.residual != nullptr && e.out_kind == OUT_BF16;
    const int cols_per_warp = p.block_n >> 1, c_begin = half * cols_per_warp;
    // bf16 rows leave through this warp's shared-memory box (behind the operand stages) and tiled stores
    const bool boxed = direct && p.c_tma;
    StoreCtx sx{boxed ? &map_c : nullptr, tiles_base + (uint32_t)(p.num_stages * p.stage_bytes) + (uint32_t)((warp - 2) * OUT_BOX_BYTES),
                0, 0, 0, lane, &map_d, code_terms[CODES ? warp - 2 : 0]};
    if constexpr (CODES) stage_code_terms(e, code_terms[warp - 2], lane);
    int acc = 0;
    uint32_t acc_phase = 0;
    for (int tile = blockIdx.x; tile < p.num_tiles; tile += gridDim.x) {
      const TileCoord t = decode_tile(p, tile);
      const int row = t.m0 + quad * 32 + lane, col_begin = t.n0 + c_begin;
      const bool row_ok = row < p.M;
      const long long row_off = (long long)t.b0 * e.c_b0 + (long long)t.b1 * e.c_b1 + (long long)row * e.ldc;
      // whole 32-column chunks of this warp's range that lie inside N take the vector path
      int nfull = 0;
      if (direct && col_begin < p.N) nfull = min((p.N - col_begin) >> 5, cols_per_warp >> 5);
      uint32_t res0[16];
      if (nfull > 0 && res_bf16) fetch_res_bf16(e, row_off + col_begin, row_ok, res0);   // in flight during the wait
      const float rb = row_ok ? row_term(e, row) : 0.f;
      float* cv = col_terms[warp - 2];
      if (nfull > 0) stage_col_terms<MODE>(e, cv, alpha, col_begin, cols_per_warp, p.N, lane);   // before the wait as well
      // every lane polls; the decision is made warp-uniform before any .sync.aligned instruction
      const bool got = mbar_wait_or_abort(smem_u32(&tfull_bar[acc]), acc_phase, vabort, p.wait_ns);
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0 && !*vabort) fail(p, DEV_TIMEOUT_MMA, vabort);
        break;
      }
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * p.block_n);
      sx.row0 = t.m0 + quad * 32; sx.b0 = t.b0; sx.b1 = t.b1;
      if (nfull > 0) drain_dispatch<KIND, MODE>(e, taddr + (uint32_t)c_begin, nfull, alpha, rb, cv, row_off + col_begin, row_ok, res0, sx, col_begin);
      for (int c = c_begin + 32 * nfull; c < c_begin + cols_per_warp && t.n0 + c < p.N; c += 32) {   // ragged or unaligned rest
        uint32_t r[32];
        tmem_ld32(taddr + (uint32_t)c, r);
        epilogue_chunk<KIND>(p, r, alpha, row_off, row, t.n0 + c, row_ok, false);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&tempty_bar[acc]));
      acc ^= 1;
      if (acc == 0) acc_phase ^= 1u;
    }
    if (boxed && lane == 0) tma_store_wait_read<0>();      // the boxes are read before the CTA ends
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// One thread waits, with the library's bounded wait, on an mbarrier that nothing ever arrives at; when the limit runs
// out it reports through the same status word and code as a product whose operand tile never landed, and returns.
__global__ void wait_probe_kernel(int* status, unsigned long long limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait_or_abort(smem_u32(&bar), 0u, &abort_flag, limit_ns)) atomicCAS(status, 0, (int)DEV_TIMEOUT_TMA);
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// The encoder is a driver call: it fails in a thread that has made no runtime call yet (and so has no current context).  The
// current device's context is then made current, as the first runtime call would, and the call repeated.
template <typename... Args>
CUresult encode_tiled(Args... args) {
  const EncodeTiledFn fn = encode_fn();
  if (!fn) return CUDA_ERROR_NOT_FOUND;
  CUresult r = fn(args...);
  int device = 0;
  if (r == CUDA_ERROR_INVALID_CONTEXT && cudaGetDevice(&device) == cudaSuccess && cudaSetDevice(device) == cudaSuccess) r = fn(args...);
  return r;
}

}  // namespace

// Tensor map of one operand: 4-D (contiguous index, strided index, batch0, batch1).  128-byte swizzle; rows of 64 bytes have a 64-byte one.
int make_operand_map(CUtensorMap* map, const OperandDesc& op, int elem_bytes, int mn_extent, int K, int nb0, int nb1,
             int tile_mn, int block_k, int* chunked) {
  if (chunked) *chunked = 0;
  if (chunked && op.mn_contig && elem_bytes == 2 && mn_extent % 64 == 0 && tile_mn % 64 == 0) {
    // (64 contiguous, k rows, chunk of 64, batch0, batch1): one box = every 64-wide piece of the tile, piece after piece
    const cuuint64_t s1 = (cuuint64_t)op.ld * 2, rows = (cuuint64_t)K;
    const cuuint64_t s3 = nb0 > 1 ? (cuuint64_t)op.s_b0 * 2 : s1 * rows;
    const cuuint64_t s4 = nb1 > 1 ? (cuuint64_t)op.s_b1 * 2 : s3 * (cuuint64_t)nb0;
    if ((reinterpret_cast<uintptr_t>(op.ptr) & 15) || (s1 & 15) || (s3 & 15) || (s4 & 15)) return GEMM_ERR_ALIGN;
    if (s1 < (cuuint64_t)mn_extent * 2) return GEMM_ERR_ARG;
    cuuint64_t dims[5] = {64, rows, (cuuint64_t)(mn_extent / 64), (cuuint64_t)nb0, (cuuint64_t)nb1};
    cuuint64_t strides[4] = {s1, 128, s3, s4};
    cuuint32_t box[5] = {64, (cuuint32_t)block_k, (cuuint32_t)(tile_mn / 64), 1, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    CUresult r = encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(op.ptr), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return GEMM_ERR_CUDA;
    *chunked = 1;
    return GEMM_OK;
  }
  const cuuint64_t inner = op.mn_contig ? (cuuint64_t)mn_extent : (cuuint64_t)K;
  const cuuint64_t rows = op.mn_contig ? (cuuint64_t)K : (cuuint64_t)mn_extent;
  cuuint64_t dims[4] = {inner, rows, (cuuint64_t)nb0, (cuuint64_t)nb1};
  cuuint64_t s1 = (cuuint64_t)op.ld * elem_bytes;
  cuuint64_t s2 = nb0 > 1 ? (cuuint64_t)op.s_b0 * elem_bytes : s1 * rows;
  cuuint64_t s3 = nb1 > 1 ? (cuuint64_t)op.s_b1 * elem_bytes : s2 * (cuuint64_t)nb0;
  if ((reinterpret_cast<uintptr_t>(op.ptr) & 15) || (s1 & 15) || (s2 & 15) || (s3 & 15)) return GEMM_ERR_ALIGN;
  if (s1 < inner * elem_bytes) return GEMM_ERR_ARG;
  cuuint64_t strides[3] = {s1, s2, s3};
  cuuint32_t box[4];
  if (op.mn_contig) {
    box[0] = 128 / elem_bytes;
    box[1] = (cuuint32_t)block_k;
  } else {
    box[0] = (cuuint32_t)block_k;
    box[1] = (cuuint32_t)tile_mn;
  }
  box[2] = box[3] = 1;
  cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUtensorMapDataType dt = elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8;
  CUresult r = encode_tiled(map, dt, 4, const_cast<void*>(op.ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  box[0] * elem_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? GEMM_OK : GEMM_ERR_CUDA;
}

namespace {

// `splits` > 1: that many CTAs share each tile's inner dimension (tc_gemm_split_kernel), worth the exchange of partial sums where
// the tiles are few and the inner dimension is long.  Alone / shared, us: 216 x 768 x 3072 17.0 / 9.5 (int8 codes 10.4 / 7.4),
// 216 x 768 x 2304 13.5 / 8.6, 512 x 768 x 3072 17.3 / 11.8, 1024 x 1024 x 4096 22.9 / 17.1, 128 x 1024 x 1024 7.8 / 6.9,
// 216 x 768 x 768 6.7 / 6.3; on the other side of the line 512 x 1024 x 1024 8.2 / 9.2, 1024 x 1024 x 1024 8.5 / 8.8.
// The figures of both sides below are of the loops before the loads were issued from a whole warp.  Judged by tc_pick_block_n's newer ones
// the sharing would end earlier at 1.1 % of the products of 128 to 1024 wide layers (fewer than 2400 tokens): there it is still the better one,
// alone (best width) / shared: 1160 x 512 x 1536 10.1 / 9.7, 1664 x 512 x 2048 12.5 / 11.1, 1280 x 768 x 2304 13.7 / 11.6, 768 x 256 x 768
// 6.55 / 6.3, int8 256 x 512 x 1536 6.9 / 6.1, 896 x 768 x 3072 10.7 / 9.5, 1152 x 1024 x 4096 13.0 / 10.9.
// No more tiles than all clusters can hold at once: cudaOccupancyMaxActiveClusters gives 74 clusters of two and 33 of four for
// every variant on an idle chip; the limits, 72 and 32, lie below that (no product of a 768 or 1024 wide layer has one of the
// few tile counts between).  Returns the tile width of the shared form (at most 128), or 0 with *splits = 1.
int pick_split(int M, int N, int k_blocks, int batches, int sm_count, int* splits) {
  const int m_tiles = (M + BLOCK_M - 1) / BLOCK_M;
  int best = 64;
  double best_cost = 1e30;
  *splits = 1;
  for (int bn = 64; bn <= 256; bn *= 2) {
    if (bn > 64 && bn / 2 >= N) break;
    const long long tiles = (long long)m_tiles * ((N + bn - 1) / bn) * batches;
    const long long waves = (tiles + sm_count - 1) / sm_count;
    const double step_us = bn == 64 ? 0.32 : (bn == 128 ? 0.43 : 0.50);
    const double epi_us = bn == 64 ? 0.5 : (bn == 128 ? 1.0 : 2.0);
    const double cost = (double)waves * (k_blocks * step_us + epi_us);
    if (cost < best_cost - 1e-9) { best_cost = cost; best = bn; *splits = 1; }
    for (int s = 2; s <= 4 && bn <= 128; s *= 2) {
      if (tiles * s > (s == 2 ? sm_count - 4 : sm_count - 20) || k_blocks < 4 * s) continue;
      const double exchange_us = 1.5 + 0.012 * (double)(tiles * s);
      const double split_cost = (double)((k_blocks + s - 1) / s) * step_us + epi_us / s + exchange_us;
      if (split_cost < best_cost - 1e-9) { best_cost = split_cost; best = bn; *splits = s; }
    }
  }
  return *splits > 1 ? best : 0;
}

}  // namespace

// Tile width by a cost model fitted to event timings (us): a persistent CTA works through `waves` tiles one after the other; a block of
// the inner dimension takes nearly the same time at any width (the producer's pace), a tile's epilogue is hidden by the next tile's
// main loop if that is longer, and the last one's, with launch, set-up and pipeline fill, is not.  So the widest tile that leaves no wave
// nearly empty wins: 192 columns where 256 do.  Widths 256 / 192 alone, us: 6144 x 1024 x 4096 46 / 44, 6144 x 1024 x 1024
// 14.8 / 13.8, 4096 x 768 x 3072 19.1 / 18.0, 4096 x 768 x 768 8.2 / 7.7, 2048 x 3072 x 768 12.4 / 11.7, int8 2200 x 2304 x 768
// 8.6 / 8.0; on the other side 4096 x 4096 x 1024 27 / 30, 4096 x 1024 x 4096 25 / 41.  Forward of both modules, one after the other, 32 x
// 128 tokens, hidden 768: 602 -> 577 us; 11 x 200 tokens with gradients 387 -> 376.  But those SMs are not idle when another stream's
// kernels run `beside` the launch, and 192 columns take more SM time in all (step of 16 x 384 tokens, hidden 1024: 5850 -> 5974
// us; 32 x 128, hidden 768: 1198 -> 1202): then not.  That holds for a step's teacher pass, its backward pass with the update under it and
// the per-product step, whichever streams they are issued to.  Not for the student's pass, whose int8 products are half as long (without
// 192 columns 8 x 256, hidden 768 976 -> 981 us, 16 x 384 and 32 x 128 within 0.1 %), nor for gradients alone, which leave little
// to the other stream (32 x 128, hidden 768 441 -> 448 us, 11 x 200 377 -> 383, hidden 1024 within 0.5 %).  `wide_out`: a group's fp32
// outputs, which take longer to store (single products' are costed as bf16).
int tc_pick_block_n(const int* M, const int* N, const int* k_blocks, int n, int batches, int sm_count, bool wide_out, bool beside) {
  static const struct { int bn; double step, tile, fixed, fixed_f32; } widths[] = {
      {64, 0.29, 0.8, 2.8, 3.5}, {128, 0.30, 1.5, 3.4, 4.4}, {192, 0.31, 2.2, 3.7, 5.3}, {256, 0.345, 2.8, 4.3, 6.4}};
  int best = 64;
  double best_cost = 1e30;
  for (const auto& w : widths) {
    if ((wide_out && w.bn == 64) || (beside && w.bn == 192)) continue;       // (groups: measured from 128 on)
    int widest = 0, kb = 0;
    long long tiles = 0;
    for (int i = 0; i < n; ++i) {
      tiles += (long long)((M[i] + BLOCK_M - 1) / BLOCK_M) * ((N[i] + w.bn - 1) / w.bn) * batches;
      widest = N[i] > widest ? N[i] : widest;
      kb = k_blocks[i] > kb ? k_blocks[i] : kb;
    }
    if (w.bn > 64 && w.bn / 2 >= widest && best_cost < 1e30) break;
    const long long waves = (tiles + sm_count - 1) / sm_count;
    const double loop = kb * w.step, hidden = loop > w.tile ? loop : w.tile;
    const double cost = loop + (double)(waves - 1) * hidden + (wide_out ? w.fixed_f32 : w.fixed);
    if (cost < best_cost - 1e-9) { best_cost = cost; best = w.bn; }
  }
  return best;
}

int tc_gemm(int kind, int a_unsigned, const OperandDesc& A, const OperandDesc& B, const GemmShape& g,
            const Epilogue& epi, int block_n, int* d_status, int sm_count, cudaStream_t stream, bool beside) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0 || g.nb0 <= 0 || g.nb1 <= 0) return GEMM_ERR_ARG;
  const int es = kind == 0 ? 2 : 1;
  if (kind == 1 && (A.mn_contig || B.mn_contig)) return GEMM_ERR_ARG;
  TcParams p;
  p.M = g.M; p.N = g.N; p.K = g.K; p.nb0 = g.nb0; p.nb1 = g.nb1;
  int splits = 1;
  p.block_n = block_n;
  if (block_n <= 0) {
    const int kb = (g.K + 128 / es - 1) / (128 / es), batches = g.nb0 * g.nb1;
    p.block_n = tc_gemm_split_eligible(kind, g, epi) ? pick_split(g.M, g.N, kb, batches, sm_count, &splits) : 0;
    if (p.block_n == 0) p.block_n = tc_pick_block_n(&g.M, &g.N, &kb, 1, batches, sm_count, false, beside);
    // With codes a tile of 256 columns has three stages only, and its long epilogue is hidden by the next tile's main loop or not at all: 192
    // where there is no next tile.  Steps / passes with 256 and with 192: 8 x 256, hidden 768 (144 tiles) 929 and 919 us; 32 x 128, hidden 768
    // (288 tiles) 547 and 554, hidden 1024 (384 tiles) the same.
    if (epi.codes && p.block_n == 256 && (long long)((g.M + BLOCK_M - 1) / BLOCK_M) * ((g.N + 255) / 256) * batches <= sm_count) p.block_n = 192;
  } else if (block_n != 64 && block_n != 128 && block_n != 256) {
    return GEMM_ERR_ARG;
  }
  p.block_k = 128 / es;
  p.m_tiles = (g.M + BLOCK_M - 1) / BLOCK_M;
  p.n_tiles = (g.N + p.block_n - 1) / p.block_n;
  p.k_blocks = (g.K + p.block_k - 1) / p.block_k;
  p.num_tiles = p.m_tiles * p.n_tiles * g.nb0 * g.nb1;
  p.stage_bytes = A_STAGE_BYTES + p.block_n * 128;
  const int code_boxes = epi.codes ? EPI_WARPS * OUT_BOX_BYTES : 0;         // (a second box per epilogue warp: fewer stages)
  p.num_stages = (SINGLE_CTA_SMEM_BUDGET - code_boxes) / p.stage_bytes;
  if (p.num_stages > MAX_STAGES) p.num_stages = MAX_STAGES;
  p.a_mn = A.mn_contig; p.b_mn = B.mn_contig;
  p.b_static = B.is_static;
  p.epi = epi;
  p.status = d_status;
  p.wait_ns = g_wait_limit_ns;
  // instruction descriptor: D format, A/B formats, majors, N >> 3, M >> 4
  uint32_t idesc = 0;
  if (kind == 0) {
    idesc |= 1u << 4;                          // fp32 accumulate
    idesc |= 1u << 7;                          // A = bf16
    idesc |= 1u << 10;                         // B = bf16
  } else {
    idesc |= 2u << 4;                          // int32 accumulate
    idesc |= (a_unsigned ? 0u : 1u) << 7;      // A = u8 / s8
    idesc |= 1u << 10;                         // B = s8
  }
  idesc |= (uint32_t)(A.mn_contig ? 1 : 0) << 15;
  idesc |= (uint32_t)(B.mn_contig ? 1 : 0) << 16;
  idesc |= (uint32_t)(p.block_n >> 3) << 17;
  idesc |= (uint32_t)(BLOCK_M >> 4) << 24;
  p.idesc = idesc;

  CUtensorMap ma, mb;
  int a_chunked = 0, b_chunked = 0;           // MN-major operands: one 5-D load per stage where the extent allows it
  int rc = make_operand_map(&ma, A, es, g.M, g.K, g.nb0, g.nb1, BLOCK_M, p.block_k, &a_chunked);
  if (rc != GEMM_OK) return rc;
  rc = make_operand_map(&mb, B, es, g.N, g.K, g.nb0, g.nb1, p.block_n, p.block_k, &b_chunked);
  if (rc != GEMM_OK) return rc;
  if (a_chunked) p.a_mn = 2;
  if (b_chunked) p.b_mn = 2;
  // bf16 output whose rows and batches start on 16-byte boundaries: tiled stores of 32 x 32 boxes
  CUtensorMap mc = ma, md = ma;
  p.c_tma = 0;
  if (epi.out_kind == OUT_BF16 && (reinterpret_cast<uintptr_t>(epi.out) & 15) == 0 && epi.ldc % 8 == 0 && epi.ldc >= g.N &&
      (g.nb0 == 1 || epi.c_b0 % 8 == 0) && (g.nb1 == 1 || epi.c_b1 % 8 == 0)) {
    const cuuint64_t s1 = (cuuint64_t)epi.ldc * 2;
    const cuuint64_t s2 = g.nb0 > 1 ? (cuuint64_t)epi.c_b0 * 2 : s1 * (cuuint64_t)g.M;
    const cuuint64_t s3 = g.nb1 > 1 ? (cuuint64_t)epi.c_b1 * 2 : s2 * (cuuint64_t)g.nb0;
    cuuint64_t dims[4] = {(cuuint64_t)g.N, (cuuint64_t)g.M, (cuuint64_t)g.nb0, (cuuint64_t)g.nb1};
    cuuint64_t strides[3] = {s1, s2, s3};
    cuuint32_t box[4] = {32, 32, 1, 1}, estr[4] = {1, 1, 1, 1};
    auto out_map = [&](CUtensorMap* m, void* ptr) {
      return encode_tiled(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    if (out_map(&mc, epi.out)) p.c_tma = 1;
    if (epi.codes && ((reinterpret_cast<uintptr_t>(epi.codes) & 15) || !p.c_tma || !out_map(&md, epi.codes))) return GEMM_ERR_ALIGN;
  } else if (epi.codes) {
    return GEMM_ERR_ALIGN;
  }
  if (epi.codes && (g.N % 32 || epi.code_cols % 32 || epi.code_cols * 3 < g.N || epi.ldc % 16 || (reinterpret_cast<uintptr_t>(epi.out) & 31) ||
                    (reinterpret_cast<uintptr_t>(epi.col_scale) & 15) || (reinterpret_cast<uintptr_t>(epi.col_bias) & 15)))
    return GEMM_ERR_ALIGN;

  const int smem = p.num_stages * p.stage_bytes + 1024 + EPI_WARPS * OUT_BOX_BYTES + code_boxes;
  typedef void (*Kern)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const TcParams);
  static const struct { int kind, mode; Kern fn; } variants[] = {
      {0, -1, tc_gemm_kernel<0, -1>}, {0, 0, tc_gemm_kernel<0, 0>}, {0, 2, tc_gemm_kernel<0, 2>}, {0, 6, tc_gemm_kernel<0, 6>},
      {0, 10, tc_gemm_kernel<0, 10>}, {0, 16, tc_gemm_kernel<0, 16>}, {1, -1, tc_gemm_kernel<1, -1>}, {1, 1, tc_gemm_kernel<1, 1>}, {1, 3, tc_gemm_kernel<1, 3>}, {1, 7, tc_gemm_kernel<1, 7>}, {1, 35, tc_gemm_kernel<1, 35>}};
  constexpr int n_variants = sizeof(variants) / sizeof(variants[0]);
  static bool attr_set[n_variants] = {};
  const int mode = epilogue_mode(kind, epi);
  int vi = 0;
  while (vi < n_variants && !(variants[vi].kind == kind && variants[vi].mode == mode)) ++vi;
  if (vi == n_variants) return GEMM_ERR_ARG;
  Kern kern = variants[vi].fn;
  if (!attr_set[vi]) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SINGLE_CTA_SMEM_BUDGET + 1024 + EPI_WARPS * OUT_BOX_BYTES) != cudaSuccess)
      return GEMM_ERR_CUDA;
    attr_set[vi] = true;
  }
  const int grid = p.num_tiles < sm_count ? p.num_tiles : sm_count;
  Scope sc([&] {
    char buf[40];                          // (shape, operand layouts, batches, tile width, thread blocks per tile)
    int len = snprintf(buf, sizeof(buf), "%s %dx%dx%d%s%s b%d w%d", kind == 0 ? "gemm_bf16" : "gemm_i8", g.M, g.N, g.K,
                       A.mn_contig ? "T" : "N", B.mn_contig ? "N" : "T", g.nb0 * g.nb1, p.block_n);
    if (splits > 1 && len < (int)sizeof(buf)) snprintf(buf + len, sizeof(buf) - len, "/%d", splits);
    return std::string(buf);
  }, 2.0 * g.M * g.N * (double)g.K * g.nb0 * g.nb1, 1, stream, 0);
  if (splits > 1) return tc_gemm_split_launch(kind, ma, mb, mc, md, p, splits, stream);
  if (launch_k(kern, grid, GEMM_THREADS, smem, stream, ma, mb, mc, md, p) != cudaSuccess) return GEMM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? GEMM_OK : GEMM_ERR_CUDA;
}

cudaError_t launch_wait_probe(int* d_status, unsigned long long limit_ns, cudaStream_t stream) {
  return launch_k(wait_probe_kernel, 1, 32, 0, stream, d_status, limit_ns);
}

}  // namespace mrem
