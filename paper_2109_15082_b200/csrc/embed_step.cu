// Embedding layers of the first module (Sec. 4.1: besides the grouped Transformer layers the MSE of the
// Transformer embedding is minimised; Sec. 3.1: embeddings are quantized symmetrically like weights).
//   teacher  e     = LayerNorm(word[ids] + pos[0..S) + type[type_ids])
//   student  e_hat = LayerNorm(Q(word)[ids] + pos + type),  Q = Eq. 1 on the word table, one step per row
//   loss     c * || e_hat - e ||^2,  straight-through backward, AdamW on the student's tables, the word
//            table's row steps and the LayerNorm parameters; the update re-quantizes the word table.
// The word table is treated as a weight matrix with `vocab` output rows: its quantizer, straight-through
// mask and fused AdamW + re-quantization are the kernels of the encoder matrices; of rows wider than the kernel
// below takes, LayerNorm and loss likewise.  New here: everything per token (both gathers, both LayerNorms, the loss, its
// gradient through the LayerNorm) in one kernel, and everything that adds up the token gradients (rows of the
// word table, sums over the batch for the position and token-type tables) in a second one, with fixed
// summation orders.  Nothing is allocated: the caller brings every tensor and one workspace.
#include <cmath>

#include "../../include/mrem.h"
#include "row_update.cuh"
#include "vec.cuh"

namespace mrem {

namespace {

// The first and the last token of every id and their number (atomicMin / atomicMax of an index, atomicAdd of 1: no dependence on
// scheduling); they say which table rows were gathered at all, who adds up a row's gradients, and how far to look.  A launch of
// its own, so that the rows nobody gathered can be updated beside the token kernels.  One block more than the tokens need prepares
// the optimizer's scalars.
__global__ void __launch_bounds__(256) embed_mark_kernel(const int* __restrict__ ids, int M, int vocab, unsigned* __restrict__ row_first,
                                                         int* __restrict__ row_last, int* __restrict__ row_count, const OptimArgs optim) {
  pdl_wait();
  pdl_trigger();
  const int t = (int)blockIdx.x * 256 + (int)threadIdx.x;
  if (t < M) {
    const int id = min(max(ids[t], 0), vocab - 1);
    atomicMin(row_first + id, (unsigned)t);
    atomicMax(row_last + id, t);
    atomicAdd(row_count + id, 1);                                   // (starts at -1)
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0 && optim.out) optim_prepare(optim);
}

// y[t, :] = row(ids[t]) + pos[t % S, :] + type[type_ids[t], :], rounded as stored; one block of 128 threads per token.
// With codes the row is scale[id] * codes[id, :] (the quantized table), else word[id, :].
template <typename T>
__global__ void __launch_bounds__(128) embed_sum_kernel(const float* __restrict__ word, const int8_t* __restrict__ codes,
                                                        const float* __restrict__ scale, const float* __restrict__ pos,
                                                        const float* __restrict__ type, const int* __restrict__ ids,
                                                        const int* __restrict__ type_ids, int S, int H, int vocab, int n_types,
                                                        T* __restrict__ y, int* __restrict__ status) {
  pdl_wait();
  pdl_trigger();
  const long long t = blockIdx.x;
  int id = ids[t], tt = type_ids ? type_ids[t] : 0;
  if (id < 0 || id >= vocab || tt < 0 || tt >= n_types) {          // recorded, then clamped: no out-of-range access
    if (threadIdx.x == 0) atomicCAS(status, 0, (int)DEV_BAD_INDEX);
    id = min(max(id, 0), vocab - 1);
    tt = min(max(tt, 0), n_types - 1);
  }
  const int s = (int)(t % S);
  const float sc = codes ? scale[id] : 0.f;
  for (int c = threadIdx.x; c < H; c += blockDim.x) {
    const float w = codes ? sc * (float)codes[(long long)id * H + c] : word[(long long)id * H + c];
    y[t * H + c] = from_f<T>(w + pos[(long long)s * H + c] + type[(long long)tt * H + c]);
  }
}

// Everything that happens to one token, W warps per token and one vector of V columns per thread (rows up to 32 * V * MAX_W
// wide): both gathers, both LayerNorms, the squared error, its gradient and the LayerNorm's backward: the operations of the
// separate kernels (embed_sum, ln_fwd, loss, ln_bwd) in their order, without their intermediates' round trips through memory
// and without six of their seven launches.  Latency bounds it: with one vector per thread a token is one round of loads and three block sums
// (both modules' means together, both variances, the two sums of the backward), and eight blocks share an SM.
// (One warp per token with the whole row in its 128 registers: 22 % of the warps active, 29 us; the step of 30522 x 1024, 32 x 128
// tokens 204 -> 200 us, of 30522 x 768, 5 x 56 tokens 154 -> 150.)
// (Rows of the table updated by blocks behind those of the tokens gained less than the same rows beside the sums.)
constexpr int MAX_W = 4;
struct EmbedRow {
  const float *t_word, *t_pos, *t_type, *t_g, *t_b;           // teacher tables and LayerNorm
  const float *pos, *type, *ln_g, *ln_b;
  const int8_t* codes; const float* scale;
  const int *ids, *type_ids;
  int S, H, vocab, n_types; long long M;
  float eps, c;                                               // c: loss scale
  int* status; unsigned* ticket;                              // (the ticket starts as 0xffffffff)
  float *mean, *rstd, *loss_partial, *loss;
  int row_blocks;
};

template <int V>
__device__ __forceinline__ void load_f32(const float* p, float* v) {
#pragma unroll
  for (int j = 0; j < V; j += 4) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p + j));
    v[j] = t.x; v[j + 1] = t.y; v[j + 2] = t.z; v[j + 3] = t.w;
  }
}

// Sums of two values over the W warps of a token, in warp order; every thread gets them.  `part`: one place per warp of the block.
template <int W>
__device__ __forceinline__ float2 token_sums(float a, float b, float2* part, int warp) {
  a = warp_sum(a);
  b = warp_sum(b);
  if (W == 1) return make_float2(a, b);
  if ((threadIdx.x & 31) == 0) part[warp] = make_float2(a, b);
  __syncthreads();
  const int first = warp / W * W;
  float2 r = part[first];
#pragma unroll
  for (int k = 1; k < W; ++k) { r.x += part[first + k].x; r.y += part[first + k].y; }
  return r;
}

__host__ __device__ constexpr int tokens_per_block(int W) { return W == 3 ? 1 : 4 / W; }

template <typename T, int V, int W>
__global__ void __launch_bounds__(32 * W * tokens_per_block(W), 8)
embed_row_kernel(const __grid_constant__ EmbedRow p, const T* __restrict__ extra, T* __restrict__ e_t, T* __restrict__ e_s,
                 T* __restrict__ y_s, T* __restrict__ dsum, T* __restrict__ dy) {
  pdl_wait();
  pdl_trigger();
  constexpr int TPB = tokens_per_block(W);
  __shared__ float sh[32];
  __shared__ float2 part[3][W * TPB];                         // one set per sum: the next token's first is behind this one's last
  __shared__ int last;
  const int wid = threadIdx.x >> 5, H = p.H, c = (int)(threadIdx.x % (32 * W)) * V;
  float err = 0.f;
  int next_id = 0, next_tt = 0;                               // (a token's ids are fetched one token ahead of its rows)
  auto fetch = [&](long long t) {
    next_id = t < p.M ? p.ids[t] : 0;
    next_tt = t < p.M && p.type_ids ? p.type_ids[t] : 0;
  };
  fetch((long long)blockIdx.x * TPB + wid / W);
  for (long long t0 = (long long)blockIdx.x * TPB; t0 < p.M; t0 += (long long)p.row_blocks * TPB) {
    const long long t = t0 + wid / W;
    const bool live = t < p.M, on = live && c < H;
    int id = next_id, tt = next_tt;
    fetch(t + (long long)p.row_blocks * TPB);
    if (id < 0 || id >= p.vocab || tt < 0 || tt >= p.n_types) {   // recorded, then clamped: no out-of-range access
      if (c == 0) atomicCAS(p.status, 0, (int)DEV_BAD_INDEX);
      id = min(max(id, 0), p.vocab - 1);
      tt = min(max(tt, 0), p.n_types - 1);
    }
    const long long row = (long long)id * H, prow = (t % p.S) * (long long)H, trow = (long long)tt * H, base = t * H;
    float et[V], y[V];                                        // teacher row, student row, as stored before the LayerNorm
#pragma unroll
    for (int j = 0; j < V; ++j) et[j] = y[j] = 0.f;
    if (on) {
      const float sc = p.scale[id];
      float a[V], b[V];
      load_f32<V>(p.t_word + row + c, et);
      load_f32<V>(p.t_pos + prow + c, a);
      load_f32<V>(p.t_type + trow + c, b);
      // (the student's position and token-type rows are written by a later kernel of this step: no read-only loads)
#pragma unroll
      for (int j = 0; j < V; j += 4) {
        const float4 pa = *reinterpret_cast<const float4*>(p.pos + prow + c + j), ta = *reinterpret_cast<const float4*>(p.type + trow + c + j);
        const char4 q = *reinterpret_cast<const char4*>(p.codes + row + c + j);
        y[j] = stored<T>(sc * (float)q.x + pa.x + ta.x);
        y[j + 1] = stored<T>(sc * (float)q.y + pa.y + ta.y);
        y[j + 2] = stored<T>(sc * (float)q.z + pa.z + ta.z);
        y[j + 3] = stored<T>(sc * (float)q.w + pa.w + ta.w);
      }
#pragma unroll
      for (int j = 0; j < V; ++j) et[j] = stored<T>(et[j] + a[j] + b[j]);
      store_vec<T, V>(y_s + base + c, y);
    }
    float sum_t = 0.f, sum_s = 0.f;
#pragma unroll
    for (int j = 0; j < V; ++j) { sum_t += et[j]; sum_s += y[j]; }
    float2 r = token_sums<W>(sum_t, sum_s, part[0], wid);
    const float mu_t = r.x / (float)H, mu = r.y / (float)H;
    sum_t = sum_s = 0.f;
    if (on) {
#pragma unroll
      for (int j = 0; j < V; ++j) { sum_t += (et[j] - mu_t) * (et[j] - mu_t); sum_s += (y[j] - mu) * (y[j] - mu); }
    }
    r = token_sums<W>(sum_t, sum_s, part[1], wid);
    const float rs_t = 1.f / sqrtf(r.x / (float)H + p.eps), rs = 1.f / sqrtf(r.y / (float)H + p.eps);
    if (live && c == 0) { p.mean[t] = mu; p.rstd[t] = rs; }
    // both outputs, the squared error, its gradient and what of it enters the LayerNorm: et becomes that gradient times
    // gamma, y the normalised row
    float s1 = 0.f, s2 = 0.f;
    if (on) {
      float g[V], d[V];
      load_f32<V>(p.t_g + c, g);
      load_f32<V>(p.t_b + c, d);
#pragma unroll
      for (int j = 0; j < V; ++j) et[j] = (et[j] - mu_t) * rs_t * g[j] + d[j];
      store_vec<T, V>(e_t + base + c, et);
      load_f32<V>(p.ln_g + c, g);
      load_f32<V>(p.ln_b + c, d);
#pragma unroll
      for (int j = 0; j < V; ++j) {
        y[j] = (y[j] - mu) * rs;
        d[j] = y[j] * g[j] + d[j];
      }
      store_vec<T, V>(e_s + base + c, d);
#pragma unroll
      for (int j = 0; j < V; ++j) {
        const float diff = stored<T>(d[j]) - stored<T>(et[j]);
        err += diff * diff;
        d[j] = stored<T>(2.f * p.c * diff);
      }
      if (extra) {
        float x[V];
        load_vec<T, V>(extra + base + c, x);
#pragma unroll
        for (int j = 0; j < V; ++j) d[j] = stored<T>(d[j] + x[j]);
      }
      store_vec<T, V>(dsum + base + c, d);
#pragma unroll
      for (int j = 0; j < V; ++j) {
        et[j] = d[j] * g[j];
        s1 += et[j];
        s2 += et[j] * y[j];
      }
    }
    r = token_sums<W>(s1, s2, part[2], wid);
    if (on) {
      s1 = r.x / (float)H;
      s2 = r.y / (float)H;
#pragma unroll
      for (int j = 0; j < V; ++j) et[j] = rs * (et[j] - s1 - y[j] * s2);
      store_vec<T, V>(dy + base + c, et);
    }
  }
  // per-block errors, added in block order by the last block to arrive
  err = block_sum(err, sh);
  if (threadIdx.x == 0) {
    p.loss_partial[blockIdx.x] = err;
    if (!isfinite(err)) atomicCAS(p.status, 0, (int)DEV_NONFINITE);
    __threadfence();
    last = atomicAdd(p.ticket, 1u) + 2u == (unsigned)p.row_blocks;   // (starts at 0xffffffff)
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  float a = 0.f;
  for (int i = threadIdx.x; i < p.row_blocks; i += blockDim.x) a += __ldcg(p.loss_partial + i);
  a = block_sum(a, sh);
  if (threadIdx.x == 0) *p.loss = a * p.c;
}

// Every sum over the token gradients dy in one launch (256 threads a block), and AdamW on the small tensors as their sums
// become complete:
//   (in the order ln_chunks, token types, word table, positions: the longest chains first)
//   max_pos blocks: one position each, two half sums over the batch (even and odd sequences), then that row's update.
//   TYPE_CHUNKS blocks per token type: one chunk of tokens each; the last chunk to finish adds the chunks in index order
//     and updates the row.
//   ln_chunks blocks: the LayerNorm's parameters, the same way.
//   one warp per token and group of TAB_COLS columns: word table.  The warp of the FIRST token with an id adds the gradients of all tokens with
//     it in token order: it compares 128 ids at a time up to the last one and keeps four rows' loads in flight.  A row
//     gathered by more than WARP_MAX tokens is left to the whole block, its warps taking consecutive eighths of the tokens and
//     the eight sums being added in warp order.  Warp w of block i has token w * blocks + i: frequent ids first appear among
//     the first tokens, and would otherwise all meet in one block.
//   Before all of these, up to two blocks per SM walk through idle rows of the word table, a warp per row, and do not wait for the token
//     kernel: they stream through memory that its last tokens and the sums leave idle.
// The sums are chains of dependent loads.  The longest were the last chunks' totals (a column per thread, eight chunks at a time; now
// four columns and sixteen chunks) and the walk over the ids (the next 128 are on their way now): step 217 -> 192 us at 32 x 128
// tokens, 136 -> 125 at 5 x 56.  Three blocks: four spill, 200 -> 207 us there although 280 tokens take 148 instead of 150.
constexpr int IDLE_BLOCKS = 148;                              // one per SM
constexpr int TYPE_CHUNKS = 64;
// Chunks of the LayerNorm's sums: above 4096 tokens twice as many, or their chains are the longest of the launch (table 1000 x 512, 48 x 128
// tokens 67.0 -> 65.6 us; 30522 x 768, 5 x 56 tokens 125 with 48, 130 with 96).
constexpr int LN_CHUNKS_MAX = 96;
inline int ln_chunks(long long tokens) { return tokens <= 4096 ? LN_CHUNKS_MAX / 2 : LN_CHUNKS_MAX; }
static_assert(TYPE_CHUNKS % 4 == 0 && LN_CHUNKS_MAX % 8 == 0, "see sum_chunks4");
constexpr int TAB_COLS = 512;                                 // columns a word-table block works on
constexpr int WARP_MAX = 16;                                  // tokens of one id that a single warp adds up
struct EmbedTables {
  const int *ids, *type_ids; const unsigned* row_first; const int *row_last, *row_count; unsigned* type_ticket;      // (n_types + 1 tickets)
  int B, S, H, vocab, n_types, max_pos, M;
  const float *mean, *rstd;
  float *g_word, *g_pos, *g_type, *type_partial, *ln_partial;
  const OptimScalars* sc;                                     // null: gradients only
  AdamEntry pos, type, ln_g, ln_b;
  bool vec;                                                   // these tensors start on 16-byte boundaries
  int ln_chunks, sum_blocks;                                  // blocks of the sums; those before take idle rows
  IdleRows idle;
};

__device__ __forceinline__ void adam_at(const AdamEntry& e, const OptimScalars& o, long long i, float g) {
  float m = e.m[i], v = e.v[i];
  e.p[i] = adam_one(e.p[i], g, m, v, o, e.wd, e.min_value);
  e.m[i] = m;
  e.v[i] = v;
}

// the same of four consecutive elements from i on (16-byte aligned)
__device__ __forceinline__ void adam4_at(const AdamEntry& e, const OptimScalars& o, long long i, float4 g) {
  float4 p = *reinterpret_cast<const float4*>(e.p + i), m = *reinterpret_cast<const float4*>(e.m + i), v = *reinterpret_cast<const float4*>(e.v + i);
  p.x = adam_one(p.x, g.x, m.x, v.x, o, e.wd, e.min_value);
  p.y = adam_one(p.y, g.y, m.y, v.y, o, e.wd, e.min_value);
  p.z = adam_one(p.z, g.z, m.z, v.z, o, e.wd, e.min_value);
  p.w = adam_one(p.w, g.w, m.w, v.w, o, e.wd, e.min_value);
  *reinterpret_cast<float4*>(e.p + i) = p;
  *reinterpret_cast<float4*>(e.m + i) = m;
  *reinterpret_cast<float4*>(e.v + i) = v;
}
// Gradients and tensors of the caller: 16-byte accesses where they allow them (`vec`).
__device__ __forceinline__ void store4(float* p, float4 g, bool vec) {
  if (vec) { *reinterpret_cast<float4*>(p) = g; return; }
  p[0] = g.x; p[1] = g.y; p[2] = g.z; p[3] = g.w;
}
__device__ __forceinline__ void update4(const AdamEntry& e, const OptimScalars& o, long long i, float4 g, bool vec) {
  if (vec) { adam4_at(e, o, i, g); return; }
  adam_at(e, o, i, g.x); adam_at(e, o, i + 1, g.y); adam_at(e, o, i + 2, g.z); adam_at(e, o, i + 3, g.w);
}
// Sums over `n` chunks (a multiple of 4) of part[ch * stride + c .. + 4): every fourth chunk's in order, then the four sums, sixteen
// chunks' loads in flight.  (In one chain the LayerNorm's gradients were 1.1e-7 from the exact sums, a column reduction of their own 0.7 to 0.9e-7,
// now 0.5 to 0.6e-7.  In 64 bits 0.3 to 0.4e-7, but 194.4 us instead of 193.2 a step of 32 x 128 tokens.)
__device__ __forceinline__ float4 sum_chunks4(const float* part, int n, long long stride, int c) {
  float4 a[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) a[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int ch = 0; ch < n; ch += 4)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 t = __ldcg(reinterpret_cast<const float4*>(part + (ch + k) * stride + c));
      a[k].x += t.x; a[k].y += t.y; a[k].z += t.z; a[k].w += t.w;
    }
  return make_float4((a[0].x + a[1].x) + (a[2].x + a[3].x), (a[0].y + a[1].y) + (a[2].y + a[3].y), (a[0].z + a[1].z) + (a[2].z + a[3].z),
                     (a[0].w + a[1].w) + (a[2].w + a[3].w));
}

// acc += the rows dy[t, c0 ..] of the tokens t in [b0, b1) whose (clamped) id is `id`, in token order, by one warp.
template <typename T, int V, int NV>
__device__ __forceinline__ void add_rows_of_id(const EmbedTables& p, const T* __restrict__ dy, int id, int b0, int b1, int c0, int lane,
                                               float (&acc)[NV][V]) {
  constexpr int FLY = sizeof(T) == 2 ? 4 : 2;                 // rows in flight
  const int H = p.H;
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int j = 0; j < V; ++j) acc[i][j] = 0.f;
  int next[4];                                                // ids of the next 128 tokens, on their way while these are compared
  auto fetch = [&](int b) {
#pragma unroll
    for (int k = 0; k < 4; ++k) next[k] = b + 32 * k + lane < b1 ? p.ids[b + 32 * k + lane] : -1;
  };
  fetch(b0);
  for (int b = b0; b < b1; b += 128) {
    int mine[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) mine[k] = b + 32 * k + lane < b1 ? min(max(next[k], 0), p.vocab - 1) : -1;
    fetch(b + 128);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      unsigned hits = __ballot_sync(0xffffffffu, mine[k] == id);
      while (hits) {
        uint32_t r[FLY][NV][RawWords<T, V>::N];
        const int n = min(__popc(hits), FLY);
#pragma unroll
        for (int f = 0; f < FLY; ++f) {
          if (f < n) {
            const T* src = dy + (long long)(b + 32 * k + __ffs(hits) - 1) * H;
            hits &= hits - 1;
#pragma unroll
            for (int i = 0; i < NV; ++i) {
              const int c = c0 + (lane + 32 * i) * V;
              if (c < H) load_raw<T, V>(src + c, r[f][i]);
            }
          }
        }
#pragma unroll
        for (int f = 0; f < FLY; ++f) {
          if (f < n) {
#pragma unroll
            for (int i = 0; i < NV; ++i) {
              if (c0 + (lane + 32 * i) * V < H) {
                float v[V];
                widen_raw<T, V>(r[f][i], v);
#pragma unroll
                for (int j = 0; j < V; ++j) acc[i][j] += v[j];
              }
            }
          }
        }
      }
    }
  }
}

template <typename T, int V>
__global__ void __launch_bounds__(256, 3) embed_tables_kernel(const __grid_constant__ EmbedTables p, const T* __restrict__ dy, const T* __restrict__ dsum,
                                                              const T* __restrict__ y_s) {
  const int idle_blocks = (int)gridDim.x - p.sum_blocks;
  if ((int)blockIdx.x < idle_blocks) {
    pdl_trigger();
    update_idle_rows<2>(p.idle, (int)blockIdx.x * 8 + (int)(threadIdx.x >> 5), idle_blocks * 8);
    return;
  }
  pdl_wait();
  pdl_trigger();
  __shared__ float red[8][TAB_COLS];
  __shared__ int flag, group[8];
  constexpr int NV = TAB_COLS / (32 * V);                     // vectors per lane in a pass
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, H = p.H;
  OptimScalars o{};
  if (p.sc) o = *p.sc;
  int blk = (int)blockIdx.x - idle_blocks;
  if (blk < p.ln_chunks) {
    // gradients of the LayerNorm's gain and bias: sums over the tokens of d * (y - mean) * rstd and of d
    const int tx = threadIdx.x & 127, ty = threadIdx.x >> 7, per = (p.M + p.ln_chunks - 1) / p.ln_chunks, t0 = blk * per, t1 = min(p.M, t0 + per);
    for (int c0 = 0; c0 < H; c0 += 128 * V) {
      const int c = c0 + tx * V;
      float ab[V], ag[V];
#pragma unroll
      for (int j = 0; j < V; ++j) ab[j] = ag[j] = 0.f;
      if (c < H) {
#pragma unroll 4
        for (int t = t0 + ty; t < t1; t += 2) {
          const float mu = p.mean[t], rs = p.rstd[t];
          float d[V], y[V];
          load_vec<T, V>(dsum + (long long)t * H + c, d);
          load_vec<T, V>(y_s + (long long)t * H + c, y);
#pragma unroll
          for (int j = 0; j < V; ++j) { ab[j] += d[j]; ag[j] += d[j] * ((y[j] - mu) * rs); }
        }
      }
      for (int k = 0; k < 2; ++k) {
        float* dst = p.ln_partial + ((long long)blk * 2 + k) * H;
        if (ty == 1) {
#pragma unroll
          for (int j = 0; j < V; ++j) red[j][tx] = k ? ag[j] : ab[j];
        }
        __syncthreads();
        if (ty == 0) {
#pragma unroll
          for (int j = 0; j < V; ++j) red[j][tx] += k ? ag[j] : ab[j];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 128 * V && c0 + i < H; i += 256) dst[c0 + i] = red[i % V][i / V];
        __syncthreads();
      }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) flag = atomicAdd(p.type_ticket + p.n_types, 1u) + 2u == (unsigned)p.ln_chunks;
    __syncthreads();
    if (!flag) return;
    __threadfence();
    for (int c = 4 * threadIdx.x; c < 2 * H; c += 1024) {      // (H is a multiple of 16: no group of four crosses the two)
      const float4 acc = sum_chunks4(p.ln_partial, p.ln_chunks, 2ll * H, c);
      const AdamEntry& e = c < H ? p.ln_b : p.ln_g;
      const int i = c < H ? c : c - H;
      store4(e.g + i, acc, p.vec);
      if (p.sc) update4(e, o, i, acc, p.vec);
    }
    return;
  }
  blk -= p.ln_chunks;
  const int n_type = TYPE_CHUNKS * p.n_types, nb = (p.M + 7) / 8, n_word = nb * ((p.H + TAB_COLS - 1) / TAB_COLS);
  if (blk < n_type || blk >= n_type + n_word) {
    // sums over rows of dy: threads 0..127 take the even rows of the set, 128..255 the odd ones
    const int tx = threadIdx.x & 127, ty = threadIdx.x >> 7;
    const bool is_pos = blk >= n_type;
    if (is_pos) blk -= n_type + n_word;
    const int s = blk, k = blk / TYPE_CHUNKS, chunk = blk % TYPE_CHUNKS;
    const int per = (p.M + TYPE_CHUNKS - 1) / TYPE_CHUNKS, t0 = chunk * per, t1 = min(p.M, t0 + per);
    float* dst = is_pos ? p.g_pos + (long long)s * H : p.type_partial + ((long long)chunk * p.n_types + k) * H;
    for (int c0 = 0; c0 < H; c0 += 128 * V) {
      const int c = c0 + tx * V;
      float acc[V];
#pragma unroll
      for (int j = 0; j < V; ++j) acc[j] = 0.f;
      if (c < H && is_pos && s < p.S) {
#pragma unroll 8
        for (int b = ty; b < p.B; b += 2) {
          float v[V];
          load_vec<T, V>(dy + ((long long)b * p.S + s) * H + c, v);
#pragma unroll
          for (int j = 0; j < V; ++j) acc[j] += v[j];
        }
      } else if (c < H && !is_pos) {
#pragma unroll 8
        for (int t = t0 + ty; t < t1; t += 2) {
          const int tt = p.type_ids ? min(max(p.type_ids[t], 0), p.n_types - 1) : 0;
          float v[V];
          load_vec<T, V>(dy + (long long)t * H + c, v);
#pragma unroll
          for (int j = 0; j < V; ++j) acc[j] += tt == k ? v[j] : 0.f;
        }
      }
      if (ty == 1) {
#pragma unroll
        for (int j = 0; j < V; ++j) red[j][tx] = acc[j];
      }
      __syncthreads();
      if (ty == 0) {
#pragma unroll
        for (int j = 0; j < V; ++j) red[j][tx] += acc[j];
      }
      __syncthreads();
      for (int i = 4 * threadIdx.x; i < 128 * V && c0 + i < H; i += 1024) {
        const float4 g = make_float4(red[i % V][i / V], red[i % V + 1][i / V], red[i % V + 2][i / V], red[i % V + 3][i / V]);
        store4(dst + c0 + i, g, p.vec || !is_pos);
        if (is_pos && p.sc) update4(p.pos, o, (long long)s * H + c0 + i, g, p.vec);
      }
      __syncthreads();
    }
    if (is_pos) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) flag = atomicAdd(p.type_ticket + k, 1u) + 2u == (unsigned)TYPE_CHUNKS;   // (starts at 0xffffffff)
    __syncthreads();
    if (!flag) return;
    __threadfence();
    for (int c = 4 * threadIdx.x; c < H; c += 1024) {
      const float4 acc = sum_chunks4(p.type_partial + (long long)k * H, TYPE_CHUNKS, (long long)p.n_types * H, c);
      store4(p.g_type + (long long)k * H + c, acc, p.vec);
      if (p.sc) update4(p.type, o, (long long)k * H + c, acc, p.vec);
    }
    return;
  }
  blk -= n_type;
  const int c0 = (blk / nb) * TAB_COLS;
  blk = blk % nb;
  const int tok = wid * nb + blk;
  int mine = -1, count = 0;                                   // id whose row this warp's token is the first to gather
  if (tok < p.M) {
    const int id = min(max(p.ids[tok], 0), p.vocab - 1);
    if (p.row_first[id] == (unsigned)tok) { mine = id; count = p.row_count[id] + 1; }
  }
  if (lane == 0) group[wid] = count > WARP_MAX ? mine : -1;
  if (mine >= 0 && count <= WARP_MAX) {
    const int end = count == 1 ? tok + 1 : p.row_last[mine] + 1;
    float acc[NV][V];
    add_rows_of_id<T, V, NV>(p, dy, mine, tok, end, c0, lane, acc);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = c0 + (lane + 32 * i) * V;
      if (c < H) {
#pragma unroll
        for (int j = 0; j < V; j += 4)
          *reinterpret_cast<float4*>(p.g_word + (long long)mine * H + c + j) = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
      }
    }
  }
  __syncthreads();
  for (int k = 0; k < 8; ++k) {
    const int id = group[k];
    if (id < 0) continue;
    const int t0 = k * nb + blk, end = p.row_last[id] + 1, seg = (end - t0 + 7) / 8;
    const int b0 = t0 + wid * seg, b1 = min(end, b0 + seg);
    float acc[NV][V];
    add_rows_of_id<T, V, NV>(p, dy, id, b0, b1, c0, lane, acc);
#pragma unroll
    for (int i = 0; i < NV; ++i)
#pragma unroll
      for (int j = 0; j < V; ++j) red[wid][(lane + 32 * i) * V + j] = acc[i][j];
    __syncthreads();
    for (int c = threadIdx.x; c < TAB_COLS && c0 + c < H; c += 256) {
      float a = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) a += red[w][c];
      p.g_word[(long long)id * H + c0 + c] = a;
    }
    __syncthreads();
  }
}

struct Carve {                         // the workspace, cut the same way by the sizing call and by the step
  char* base; size_t off = 0;
  explicit Carve(void* b) : base((char*)b) {}
  void* take(size_t bytes) { off = (off + 255) & ~size_t(255); void* p = base ? base + off : nullptr; off += bytes; return p; }
};
struct EmbedScratch {
  void *y_t, *y_s, *dE, *dy, *dsum;
  float *mean, *rstd, *ln_partial, *loss_partial;
  int8_t* codes; int32_t* rowsum; float* scale;
  OptimScalars* optim_sc;
  unsigned* marks; size_t mark_bytes;      // first and last token of every id and their number, then the tickets of the loss, the token types and the LayerNorm
  float* type_partial;
  size_t bytes;
};
// What one call leaves for the next (the quantized table) comes first and whatever depends on the number of tokens last: calls of
// any size find the table at the same place.
EmbedScratch carve(const mrem_embed_desc& d, long long max_tokens, void* base) {
  Carve A(base);
  EmbedScratch s;
  s.codes = (int8_t*)A.take((size_t)d.vocab * d.hidden);
  s.rowsum = (int32_t*)A.take(sizeof(int32_t) * d.vocab);
  s.scale = (float*)A.take(sizeof(float) * d.vocab);
  s.optim_sc = (OptimScalars*)A.take(sizeof(OptimScalars));
  s.ln_partial = (float*)A.take(sizeof(float) * 2 * LN_CHUNKS_MAX * d.hidden);
  s.loss_partial = (float*)A.take(sizeof(float) * RED_BLOCKS);
  s.mark_bytes = sizeof(unsigned) * (3 * (size_t)d.vocab + 2 + d.n_types);
  s.marks = (unsigned*)A.take(s.mark_bytes);
  s.type_partial = (float*)A.take(sizeof(float) * (size_t)TYPE_CHUNKS * d.n_types * d.hidden);
  const size_t es = d.act_dtype == MREM_BF16 ? 2 : 4;
  const size_t MH = (size_t)max_tokens * d.hidden;
  s.y_t = A.take(MH * es); s.y_s = A.take(MH * es); s.dE = A.take(MH * es); s.dy = A.take(MH * es); s.dsum = A.take(MH * es);
  s.mean = (float*)A.take(4 * max_tokens); s.rstd = (float*)A.take(4 * max_tokens);
  s.bytes = (A.off + 255) & ~size_t(255);
  return s;
}

int check_desc(const mrem_embed_desc* d) {
  if (!d || d->struct_size != sizeof(mrem_embed_desc)) return MREM_ERR_ARG;
  if (d->vocab < 1 || d->hidden < 16 || d->hidden % 16 || d->max_pos < 1 || d->n_types < 1) return MREM_ERR_SHAPE;
  if (d->e_bits != 2 && d->e_bits != 4 && d->e_bits != 8) return MREM_ERR_UNSUPPORTED;
  if (d->act_dtype != MREM_F32 && d->act_dtype != MREM_BF16) return MREM_ERR_ARG;
  return MREM_OK;
}

}  // namespace
}  // namespace mrem

using namespace mrem;

extern "C" {

int32_t mrem_embed_workspace_bytes(const mrem_embed_desc* d, int32_t max_tokens, size_t* out_bytes) {
  const int rc = check_desc(d);
  if (rc != MREM_OK) return rc;
  if (!out_bytes || max_tokens < 1) return MREM_ERR_ARG;
  *out_bytes = carve(*d, max_tokens, nullptr).bytes;
  return MREM_OK;
}

int32_t mrem_embed_step(const mrem_embed_desc* d, const mrem_embed_tensors* x, void* workspace, size_t workspace_bytes,
                        const int32_t* d_ids, const int32_t* d_type_ids, int32_t batch, int32_t seq, int32_t requantize,
                        void* d_e_teacher, void* d_e_student, const void* d_extra_grad, const mrem_optim* o, float* d_loss,
                        int32_t* d_status, void* cuda_stream) {
  int rc = check_desc(d);
  if (rc != MREM_OK) return rc;
  if (!x || !workspace || !d_ids || !d_e_teacher || !d_e_student || !d_loss || !d_status) return MREM_ERR_ARG;
  if (batch < 1 || seq < 1 || seq > d->max_pos) return MREM_ERR_SHAPE;
  const float* need[] = {x->t_word, x->t_pos, x->t_type, x->t_ln_g, x->t_ln_b, x->word, x->pos, x->type, x->ln_g, x->ln_b,
                         x->word_step, x->g_word, x->g_word_step, x->g_pos, x->g_type, x->g_ln_g, x->g_ln_b};
  for (const float* p : need) if (!p) return MREM_ERR_ARG;
  if (o && (!x->m_word || !x->v_word || !x->m_word_step || !x->v_word_step || !x->m_pos || !x->v_pos || !x->m_type || !x->v_type ||
            !x->m_ln_g || !x->v_ln_g || !x->m_ln_b || !x->v_ln_b || !x->d_step_counter))
    return MREM_ERR_ARG;
  const long long M = (long long)batch * seq;
  const int H = d->hidden, V = d->vocab, dt = d->act_dtype == MREM_BF16 ? 1 : 0;
  const EmbedScratch s = carve(*d, M, workspace);
  if (s.bytes > workspace_bytes) return MREM_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255) || (reinterpret_cast<uintptr_t>(d_e_teacher) & 15) ||
      (reinterpret_cast<uintptr_t>(d_e_student) & 15) || (reinterpret_cast<uintptr_t>(x->word) & 15) ||
      (reinterpret_cast<uintptr_t>(x->g_word) & 15))
    return MREM_ERR_ALIGN;
  cudaStream_t st = (cudaStream_t)cuda_stream;

  // Eq. 1 on the word table (only when the caller changed it or its steps since the last update)
  if (requantize) launch_quantize_weight(x->word, V, H, x->word_step, 1, d->e_bits, 0, s.codes, s.rowsum, s.scale, nullptr, dt, st);
  const long long n = M * H;
  const float cc = d->loss_mean ? 1.f / (float)n : 1.f;
  if (d_extra_grad && (reinterpret_cast<uintptr_t>(d_extra_grad) & 15)) return MREM_ERR_ALIGN;
  if (cudaMemsetAsync(s.marks, 0xff, s.mark_bytes, st) != cudaSuccess) return MREM_ERR_CUDA;
  unsigned* row_first = s.marks;
  int *row_last = (int*)(s.marks + V), *row_count = row_last + V;
  unsigned *loss_ticket = s.marks + 3 * (size_t)V, *type_ticket = loss_ticket + 1;
  bool aligned = true;                                     // 16-byte accesses of the tables' rows
  const float* const rows[] = {x->t_word, x->t_pos, x->t_type, x->t_ln_g, x->t_ln_b, x->pos, x->type, x->ln_g, x->ln_b};
  for (const float* q : rows) aligned = aligned && (reinterpret_cast<uintptr_t>(q) & 15) == 0;
  void* dsum = s.dsum;                                     // the gradient the LayerNorm sees
  OptimArgs oa{};
  if (o) oa = OptimArgs{s.optim_sc, x->d_step_counter, o->step, o->lr, o->decay_total_steps, o->beta1, o->beta2, o->eps, o->weight_decay};
  launch_k(embed_mark_kernel, (unsigned)((M + 255) / 256 + (o ? 1 : 0)), 256, 0, st, d_ids, (int)M, V, row_first, row_last, row_count, oa);
  // Update of the word table: mask + step gradient + AdamW on the steps and the table + Eq. 1 with the new values in one pass (the
  // small tensors are updated by the launch that adds up their gradients, the other embedding tables decayed like weight matrices,
  // LayerNorm not).  The rows that no token gathered need nothing of this step but the marks and the optimizer's scalars, which are complete
  // before the token kernel lets its successors start.  So the launch of the sums begins with a few blocks that walk through such rows
  // without waiting for the token kernel, and the last launch, whose blocks keep more bytes in flight, begins with the rest and does
  // not wait for the sums.  30522 x 1024 with 32 x 128 tokens 194.5 -> 181.6 us, 30522 x 768 with 5 x 56 125.4 -> 119.2, with 48 x 128 170.7 ->
  // 160.1, 21128 x 512 with 8 x 64 74.4 -> 68.1 (before: blocks behind those of the token kernel and of the sums, everything waiting).
  // The share of the sums' launch, a number of rows that grows with the tokens, whose chains last that long, and 145 MB at 29 bytes a weight
  // (half as many: 184.7, 121.3, 165.2, 71.3), and its blocks, one of three per SM or with few tokens two (two with many: 185.5, 166.4; one with
  // few: 121.7, 74.0; as many as it takes: 186.6, 121.4, 166.5, 71.4), were fitted at these sizes.
  const RowUpdate table{x->word, x->g_word, x->m_word, x->v_word, x->word_step, x->m_word_step, x->v_word_step, nullptr,
                        s.codes, s.rowsum, s.scale, nullptr, V, H};
  int idle_at = o ? 0 : V;                                   // the next idle row to hand out
  auto take_idle = [&](long long n) {
    const int first = idle_at;
    idle_at = (int)(first + n < V ? first + n : V);
    return IdleRows{table, s.optim_sc, row_first, d->e_bits, first, idle_at};
  };
  const int row_warps = (H + 32 * (dt == 1 ? 8 : 4) - 1) / (32 * (dt == 1 ? 8 : 4));
  if (row_warps <= MAX_W && aligned) {
    // one vector per thread: everything per token in one kernel
    const int tpb = tokens_per_block(row_warps);
    const long long want = (M + tpb - 1) / tpb;
    const int row_blocks = (int)(want < RED_BLOCKS ? want : RED_BLOCKS);
    const EmbedRow er{x->t_word, x->t_pos, x->t_type, x->t_ln_g, x->t_ln_b, x->pos, x->type, x->ln_g, x->ln_b, s.codes, s.scale, d_ids, d_type_ids,
                      (int)seq, H, V, (int)d->n_types, M, d->ln_eps, cc, d_status, loss_ticket,
                      s.mean, s.rstd, s.loss_partial, d_loss, row_blocks};
    Scope sc("embed_row", (double)M * H * (8.0 + 1.0 + (dt == 1 ? 2.0 : 4.0) * (d_extra_grad ? 6 : 5)), 0, st);
#define MREM_ROW(T, V, W) launch_k(embed_row_kernel<T, V, W>, row_blocks, 32 * W * tokens_per_block(W), 0, st, er, (const T*)d_extra_grad, (T*)d_e_teacher, (T*)d_e_student, (T*)s.y_s, (T*)s.dsum, (T*)s.dy)
#define MREM_ROWS(T, V) do { if (row_warps == 1) MREM_ROW(T, V, 1); else if (row_warps == 2) MREM_ROW(T, V, 2); else if (row_warps == 3) MREM_ROW(T, V, 3); else MREM_ROW(T, V, 4); } while (0)
    if (dt == 1) MREM_ROWS(bf16, 8); else MREM_ROWS(float, 4);
#undef MREM_ROWS
#undef MREM_ROW
  } else {
    // wide rows: both embedding sums, the two LayerNorms, the loss and the LayerNorm backward as kernels of their own
#define MREM_EMB(T) do { \
    launch_k(embed_sum_kernel<T>, (unsigned)M, 128, 0, st, x->t_word, (const int8_t*)nullptr, (const float*)nullptr, x->t_pos, x->t_type, d_ids, d_type_ids, (int)seq, H, V, (int)d->n_types, (T*)s.y_t, d_status); \
    launch_k(embed_sum_kernel<T>, (unsigned)M, 128, 0, st, (const float*)x->word, (const int8_t*)s.codes, (const float*)s.scale, (const float*)x->pos, (const float*)x->type, d_ids, d_type_ids, (int)seq, H, V, (int)d->n_types, (T*)s.y_s, d_status); } while (0)
    if (dt == 1) MREM_EMB(bf16); else MREM_EMB(float);
#undef MREM_EMB
    launch_layernorm_fwd(s.y_t, x->t_ln_g, x->t_ln_b, d->ln_eps, M, H, d_e_teacher, nullptr, nullptr, nullptr, 0, nullptr, nullptr, dt, st);
    launch_layernorm_fwd(s.y_s, x->ln_g, x->ln_b, d->ln_eps, M, H, d_e_student, s.mean, s.rstd, nullptr, 0, nullptr, nullptr, dt, st);
    launch_loss(d_e_student, d_e_teacher, 1, n, cc, s.dE, s.loss_partial, d_status, dt, st);
    launch_loss_finalize(s.loss_partial, 1, cc, d_loss, nullptr, st);
    // (with a gradient arriving from the layers the embedding feeds, the LayerNorm sees the sum of the two)
    launch_layernorm_bwd(s.dE, d_extra_grad, s.y_s, s.mean, s.rstd, x->ln_g, M, H, s.dy, d_extra_grad ? s.dsum : nullptr, dt, st);
    if (!d_extra_grad) dsum = s.dE;
  }
  // word, position and token-type tables: sums of the token gradients.  Rows of the word table that no token gathered are
  // cleared by the update (row_first says which they are), without one here.
  if (!o && cudaMemsetAsync(x->g_word, 0, sizeof(float) * (size_t)V * H, st) != cudaSuccess) return MREM_ERR_CUDA;
  const int n_sum = (int)(d->max_pos + (long long)TYPE_CHUNKS * d->n_types + ln_chunks(M) + ((M + 7) / 8) * ((H + TAB_COLS - 1) / TAB_COLS));
  bool vec = true;
  const float* const small[] = {x->pos, x->type, x->ln_g, x->ln_b, x->g_pos, x->g_type, x->g_ln_g, x->g_ln_b};
  for (const float* q : small) vec = vec && (reinterpret_cast<uintptr_t>(q) & 15) == 0;
  if (o) {
    const float* const moments[] = {x->m_pos, x->v_pos, x->m_type, x->v_type, x->m_ln_g, x->v_ln_g, x->m_ln_b, x->v_ln_b};
    for (const float* q : moments) vec = vec && (reinterpret_cast<uintptr_t>(q) & 15) == 0;
  }
  const EmbedTables tb{d_ids, d_type_ids, row_first, row_last, row_count, type_ticket, (int)batch, (int)seq, H, V, (int)d->n_types,
                       (int)d->max_pos, (int)M, s.mean, s.rstd, x->g_word, x->g_pos, x->g_type, s.type_partial, s.ln_partial, o ? s.optim_sc : nullptr,
                       {x->pos, x->g_pos, x->m_pos, x->v_pos, 0, 1.f, -INFINITY}, {x->type, x->g_type, x->m_type, x->v_type, 0, 1.f, -INFINITY},
                       {x->ln_g, x->g_ln_g, x->m_ln_g, x->v_ln_g, 0, 0.f, -INFINITY}, {x->ln_b, x->g_ln_b, x->m_ln_b, x->v_ln_b, 0, 0.f, -INFINITY},
                       vec, ln_chunks(M), n_sum, take_idle(M + 5000000 / H)};
  const int idle_rows = tb.idle.end - tb.idle.first, idle_limit = M <= 1024 ? 2 * IDLE_BLOCKS : IDLE_BLOCKS,
            idle_blocks = (idle_rows + 7) / 8 < idle_limit ? (idle_rows + 7) / 8 : idle_limit;
  const unsigned tgrid = (unsigned)(n_sum + idle_blocks);
  {
    Scope sc("embed_tables", (double)M * H * 5.0 * (dt == 1 ? 2.0 : 4.0) + 29.0 * H * (tb.idle.end - tb.idle.first), 0, st);
    if (dt == 1) launch_k(embed_tables_kernel<bf16, 8>, tgrid, 256, 0, st, tb, (const bf16*)s.dy, (const bf16*)dsum, (const bf16*)s.y_s);
    else launch_k(embed_tables_kernel<float, 4>, tgrid, 256, 0, st, tb, (const float*)s.dy, (const float*)dsum, (const float*)s.y_s);
  }
  if (!o) {
    // gradients only: the word table's straight-through mask and its row-step gradients, left in g_word / g_word_step
    launch_ste_weight(x->word, x->word_step, 1, d->e_bits, 0, x->g_word, V, H, x->g_word_step, st);
    return cudaGetLastError() == cudaSuccess ? MREM_OK : MREM_ERR_CUDA;
  }
  launch_table_update(take_idle(V), TokenRows{d_ids, row_first, (int)M}, dt, st);
  return cudaGetLastError() == cudaSuccess ? MREM_OK : MREM_ERR_CUDA;
}

}  // extern "C"
