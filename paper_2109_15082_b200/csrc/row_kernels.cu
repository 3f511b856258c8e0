// Row-wise kernels: LayerNorm forward/backward, attention softmax forward/backward (with the
// quantizer of the probabilities), and column sums over rows (bias / LayerNorm-parameter
// gradients).  One warp owns one row and keeps it in registers (one read of each input,
// 8- or 16-byte vector accesses, warp-shuffle reductions); a slower re-reading form covers
// rows too long for the register cache or views that are not vector aligned.
#include "kernels.h"
#include "vec.cuh"

namespace mrem {

namespace {

constexpr int MAXNV = 4;     // vectors per lane held in registers

__device__ __forceinline__ float qz(float x, float s, float off, bool has_off) {
  return __fdiv_rn(has_off ? __fsub_rn(x, off) : x, s);
}
__device__ __forceinline__ int qcode(float z, float lo, float hi) { return __float2int_rn(fminf(fmaxf(z, lo), hi)); }

// 4 consecutive values
template <typename T> __device__ __forceinline__ void load4(const T* p, float* v);
template <> __device__ __forceinline__ void load4<float>(const float* p, float* v) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <> __device__ __forceinline__ void load4<bf16>(const bf16* p, float* v) {
  const uint2 t = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&t);
  const float2 a = __bfloat1622float2(h[0]), b = __bfloat1622float2(h[1]);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
template <typename T> __device__ __forceinline__ void store4(T* p, const float* v);
template <> __device__ __forceinline__ void store4<float>(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
template <> __device__ __forceinline__ void store4<bf16>(bf16* p, const float* v) {
  uint2 t;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&t);
  h[0] = __floats2bfloat162_rn(v[0], v[1]);
  h[1] = __floats2bfloat162_rn(v[2], v[3]);
  *reinterpret_cast<uint2*>(p) = t;
}

// V consecutive floats of a per-column vector (16-byte aligned when V % 4 == 0: the vector paths guarantee it)
template <int V>
__device__ __forceinline__ void load_cols(const float* __restrict__ p, float* v) {
  if constexpr (V % 4 == 0) {
#pragma unroll
    for (int j = 0; j < V; j += 4) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(p + j));
      v[j] = t.x; v[j + 1] = t.y; v[j + 2] = t.z; v[j + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < V; ++j) v[j] = p[j];
  }
}

// ------------------------------------------------------------------ LayerNorm forward
// CACHED: the row sits in registers (cols <= 32 * V * MAXNV, cols % V == 0); else V == 1 and
// the row is re-read from L1/L2 in each of the three passes.
template <typename T, int V, bool CACHED>
__global__ void __launch_bounds__(128) ln_fwd_kernel(const T* __restrict__ y, const float* __restrict__ gamma,
                                                     const float* __restrict__ beta, float eps, long long rows,
                                                     int cols, T* __restrict__ out, float* __restrict__ mean,
                                                     float* __restrict__ rstd, const float* __restrict__ step,
                                                     float qmax, int8_t* __restrict__ q8, T* __restrict__ qt) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const long long row = blockIdx.x * 4ll + (threadIdx.x >> 5);
  if (row >= rows) return;
  const T* yr = y + row * cols;
  float v[CACHED ? MAXNV : 1][V];
  float sum = 0.f;
  if constexpr (CACHED) {
#pragma unroll
    for (int i = 0; i < MAXNV; ++i) {
      const int c = (lane + 32 * i) * V;
      if (c < cols) {
        load_vec<T, V>(yr + c, v[i]);
#pragma unroll
        for (int j = 0; j < V; ++j) sum += v[i][j];
      }
    }
  } else {
    for (int c = lane; c < cols; c += 32) sum += to_f<T>(yr[c]);
  }
  const float mu = warp_sum(sum) / (float)cols;
  float sq = 0.f;
  if constexpr (CACHED) {
#pragma unroll
    for (int i = 0; i < MAXNV; ++i)
      if ((lane + 32 * i) * V < cols) {
#pragma unroll
        for (int j = 0; j < V; ++j) sq += (v[i][j] - mu) * (v[i][j] - mu);
      }
  } else {
    for (int c = lane; c < cols; c += 32) { const float d = to_f<T>(yr[c]) - mu; sq += d * d; }
  }
  const float rs = 1.f / sqrtf(warp_sum(sq) / (float)cols + eps);
  if (lane == 0) {
    if (mean) mean[row] = mu;
    if (rstd) rstd[row] = rs;
  }
  const float s = step ? *step : 1.f, r_s = __frcp_rn(s);
  auto emit = [&](int c, float* o) {
    float gm[V], bt[V];
    load_cols<V>(gamma + c, gm);
    load_cols<V>(beta + c, bt);
#pragma unroll
    for (int j = 0; j < V; ++j) o[j] = (o[j] - mu) * rs * gm[j] + bt[j];
    store_vec<T, V>(out + row * cols + c, o);
    if (step) {
      uint32_t b[V];
#pragma unroll
      for (int j = 0; j < V; ++j) o[j] = stored<T>(o[j]);
      codes_of<sizeof(T) == 2, V>(o, s, r_s, -qmax, qmax, b);                   // bfloat16-valued numerators are exact
      if (q8) store_code_bytes<V>(q8 + row * cols + c, b);
      if (qt) store_vec<T, V>(qt + row * cols + c, o);
    }
  };
  if constexpr (CACHED) {
#pragma unroll
    for (int i = 0; i < MAXNV; ++i) {
      const int c = (lane + 32 * i) * V;
      if (c < cols) emit(c, v[i]);
    }
  } else {
    for (int c = lane; c < cols; c += 32) {
      float o[V];
      o[0] = to_f<T>(yr[c]);
      emit(c, o);
    }
  }
}

// ------------------------------------------------------------------ LayerNorm backward
template <typename T, int V, bool CACHED>
__global__ void __launch_bounds__(128) ln_bwd_kernel(const T* __restrict__ dout, const T* __restrict__ dout2,
                                                     const T* __restrict__ y, const float* __restrict__ mean,
                                                     const float* __restrict__ rstd, const float* __restrict__ gamma,
                                                     long long rows, int cols, T* __restrict__ dy,
                                                     T* __restrict__ dsum) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const long long row = blockIdx.x * 4ll + (threadIdx.x >> 5);
  if (row >= rows) return;
  const float mu = mean[row], rs = rstd[row];
  const long long base = row * cols;
  float d[CACHED ? MAXNV : 1][V], xn[CACHED ? MAXNV : 1][V];
  float s1 = 0.f, s2 = 0.f;
  // total incoming gradient of one vector; written to dsum (rounded to storage) when requested
  auto fetch = [&](int c, float* dv, float* xv) {
    load_vec<T, V>(dout + base + c, dv);
    if (dout2) {
      float e[V];
      load_vec<T, V>(dout2 + base + c, e);
#pragma unroll
      for (int j = 0; j < V; ++j) dv[j] += e[j];
      if (dsum) {
        store_vec<T, V>(dsum + base + c, dv);
#pragma unroll
        for (int j = 0; j < V; ++j) dv[j] = stored<T>(dv[j]);
      }
    }
    load_vec<T, V>(y + base + c, xv);
    float gm[V];
    load_cols<V>(gamma + c, gm);
#pragma unroll
    for (int j = 0; j < V; ++j) {
      xv[j] = (xv[j] - mu) * rs;
      dv[j] *= gm[j];
    }
  };
  if constexpr (CACHED) {
#pragma unroll
    for (int i = 0; i < MAXNV; ++i) {
      const int c = (lane + 32 * i) * V;
      if (c < cols) {
        fetch(c, d[i], xn[i]);
#pragma unroll
        for (int j = 0; j < V; ++j) { s1 += d[i][j]; s2 += d[i][j] * xn[i][j]; }
      }
    }
  } else {
    for (int c = lane; c < cols; c += 32) {
      fetch(c, d[0], xn[0]);
      s1 += d[0][0];
      s2 += d[0][0] * xn[0][0];
    }
  }
  s1 = warp_sum(s1) / (float)cols;
  s2 = warp_sum(s2) / (float)cols;
  if constexpr (CACHED) {
#pragma unroll
    for (int i = 0; i < MAXNV; ++i) {
      const int c = (lane + 32 * i) * V;
      if (c < cols) {
#pragma unroll
        for (int j = 0; j < V; ++j) d[i][j] = rs * (d[i][j] - s1 - xn[i][j] * s2);
        store_vec<T, V>(dy + base + c, d[i]);
      }
    }
  } else {
    const T* dsrc = (dout2 && dsum) ? dsum : dout;
    for (int c = lane; c < cols; c += 32) {
      float dv = to_f<T>(dsrc[base + c]);
      if (dout2 && !dsum) dv += to_f<T>(dout2[base + c]);
      const float x = (to_f<T>(y[base + c]) - mu) * rs;
      dy[base + c] = from_f<T>(rs * (dv * gamma[c] - s1 - x * s2));
    }
  }
}

// ------------------------------------------------------------------ LayerNorm backward with its column sums
// The gradient that enters the LayerNorm, with STE assembled on the fly:
//   dv = dout (when given) + 1[lo <= x / step <= hi] * dxhat + add,
// i.e. the straight-through pass of the activation quantizer that saw x (Sec. 3.1.1) followed by the skip connection; without it
// dv = dout.  dv, rounded as stored, goes into the LayerNorm backward; the quantizer's step-size gradient leaves as one partial sum
// per block (fixed order; slots beyond the grid are zeroed).
// The gradients of the LayerNorm's bias and gain and of the bias of the product before it are sums over the rows of dv, of
// dv * (y - mean) * rstd and of dy: a thread keeps one vector of columns and adds its rows in row order, and every group of the W
// warps that share a row leaves 3 * cols partial sums; col_finish_kernel adds the groups' in index order.
// No more than 128 threads a block and no shared memory to speak of, so that blocks fit beside a product of the other stream (with
// 256 threads and the groups added up in shared memory they did not).  Two rows in flight per group.
// One warp per row with the row in its registers, dv written out, and a launch that read dv, y and dy again for the sums: the steps
// of 32 x 128 tokens, hidden 1024, 3512 us (now 3465), of 8 x 256, hidden 768, 995 (984), of 3 x 72 461 (456); 16 x 384, hidden 1024 within
// the 0.8 % by which two runs differ.
__host__ __device__ constexpr int ln_groups(int W) { return W >= 3 ? 1 : 4 / W; }
constexpr int LN_ROWS = 2;                                     // rows a group has in flight
template <typename T, int V, int W, bool STE>
__global__ void __launch_bounds__(32 * W * ln_groups(W), 4)
ln_bwd_cols_kernel(const T* __restrict__ dout, const T* __restrict__ x, const T* __restrict__ dxhat, const T* __restrict__ add,
                   const float* __restrict__ step, float lo, float hi, const T* __restrict__ y, const float* __restrict__ mean,
                   const float* __restrict__ rstd, const float* __restrict__ gamma, long long rows, int cols, T* __restrict__ dy,
                   float* __restrict__ part_s, int n_slots, float* __restrict__ col_part) {
  pdl_wait();
  pdl_trigger();
  constexpr int G = ln_groups(W), R = LN_ROWS, NW = W * G, RW = RawWords<T, V>::N;
  __shared__ float2 sums[2][NW][R];
  __shared__ float sh[NW];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = wid / W, tc = (int)threadIdx.x - grp * 32 * W, c = tc * V;
  const bool on = c < cols;
  const float s = STE ? *step : 1.f, r_s = __frcp_rn(s);
  float a0[V], a1[V], a2[V], gm[V];
#pragma unroll
  for (int j = 0; j < V; ++j) a0[j] = a1[j] = a2[j] = gm[j] = 0.f;
  if (on) load_cols<V>(gamma + c, gm);
  float ds = 0.f;
  int flip = 0;
  for (long long r0 = (long long)blockIdx.x * (G * R); r0 < rows; r0 += (long long)gridDim.x * (G * R), flip ^= 1) {
    uint32_t wo[R][RW], wx[R][RW], wd[R][RW], wa[R][RW], wy[R][RW];
    float mu[R], rs[R];
    bool live[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {                              // all loads first
      const long long r = r0 + k * G + grp, i = r * cols + c;
      live[k] = r < rows;
      mu[k] = rs[k] = 0.f;
      if (live[k]) { mu[k] = mean[r]; rs[k] = rstd[r]; }
      live[k] = live[k] && on;
      if (!live[k]) continue;
      if (STE) {
        load_raw<T, V>(x + i, wx[k]);
        load_raw<T, V>(dxhat + i, wd[k]);
        load_raw<T, V>(add + i, wa[k]);
      }
      if (!STE || dout) load_raw<T, V>(dout + i, wo[k]);
      load_raw<T, V>(y + i, wy[k]);
    }
    float d[R][V], xn[R][V];
    float2 t[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
      t[k] = make_float2(0.f, 0.f);
      if (!live[k]) continue;
      if (STE) {
        float e[V];
        widen_raw<T, V>(wx[k], e);
        widen_raw<T, V>(wd[k], d[k]);
#pragma unroll
        for (int j = 0; j < V; ++j) {
          const float z = quotient(e[j], s, r_s);
          const bool in = z >= lo && z <= hi;
          ds += d[k][j] * (rne_magic(fminf(fmaxf(z, lo), hi)) - (in ? z : 0.f));
          d[k][j] = in ? d[k][j] : 0.f;
        }
        widen_raw<T, V>(wa[k], e);
#pragma unroll
        for (int j = 0; j < V; ++j) d[k][j] += e[j];
        if (dout) {
          widen_raw<T, V>(wo[k], e);
#pragma unroll
          for (int j = 0; j < V; ++j) d[k][j] += e[j];
        }
#pragma unroll
        for (int j = 0; j < V; ++j) d[k][j] = stored<T>(d[k][j]);
      } else {
        widen_raw<T, V>(wo[k], d[k]);
      }
      widen_raw<T, V>(wy[k], xn[k]);
#pragma unroll
      for (int j = 0; j < V; ++j) {
        xn[k][j] -= mu[k];
        a0[j] += d[k][j];
        a1[j] += d[k][j] * xn[k][j] * rs[k];
        xn[k][j] *= rs[k];
        d[k][j] *= gm[j];
        t[k].x += d[k][j];
        t[k].y += d[k][j] * xn[k][j];
      }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
      t[k].x = warp_sum(t[k].x);
      t[k].y = warp_sum(t[k].y);
      if (W > 1 && lane == 0) sums[flip][wid][k] = t[k];
    }
    if constexpr (W > 1) {
      __syncthreads();                                         // (the other set is behind the next iteration's barrier)
#pragma unroll
      for (int k = 0; k < R; ++k) {
        t[k] = sums[flip][grp * W][k];
#pragma unroll
        for (int w = 1; w < W; ++w) { t[k].x += sums[flip][grp * W + w][k].x; t[k].y += sums[flip][grp * W + w][k].y; }
      }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
      if (!live[k]) continue;
      const float s1 = t[k].x / (float)cols, s2 = t[k].y / (float)cols;
#pragma unroll
      for (int j = 0; j < V; ++j) d[k][j] = rs[k] * (d[k][j] - s1 - xn[k][j] * s2);
      store_vec<T, V>(dy + (r0 + k * G + grp) * cols + c, d[k]);
#pragma unroll
      for (int j = 0; j < V; ++j) a2[j] += stored<T>(d[k][j]);
    }
  }
  if (on) {
    float* dst = col_part + ((long long)blockIdx.x * G + grp) * 3 * cols + c;
#pragma unroll
    for (int j = 0; j < V; j += 4) {
      *reinterpret_cast<float4*>(dst + j) = make_float4(a0[j], a0[j + 1], a0[j + 2], a0[j + 3]);
      *reinterpret_cast<float4*>(dst + cols + j) = make_float4(a1[j], a1[j + 1], a1[j + 2], a1[j + 3]);
      *reinterpret_cast<float4*>(dst + 2 * cols + j) = make_float4(a2[j], a2[j + 1], a2[j + 2], a2[j + 3]);
    }
  }
  if (STE) {
    ds = warp_sum(ds);
    if (lane == 0) sh[wid] = ds;
    __syncthreads();
  }
  if (STE) {
    if (threadIdx.x == 0) {
      float v = sh[0];
#pragma unroll
      for (int w = 1; w < NW; ++w) v += sh[w];
      part_s[blockIdx.x] = v;
    }
    if (blockIdx.x == 0)
      for (int i = gridDim.x + threadIdx.x; i < n_slots; i += blockDim.x) part_s[i] = 0.f;
  }
}

// out_k[c] = sum over n parts of part[i][k][c], in index order within 32 runs of them and the runs in order; 32 columns a block.  Added
// in 64 bits, so that the sums are as exact as the parts: in 32 bits these two chains (19 and 32 long at 592 parts) were most of the error.
__global__ void __launch_bounds__(256) col_finish_kernel(const float* __restrict__ part, int n, int cols, float* __restrict__ out0,
                                                         float* __restrict__ out1, float* __restrict__ out2) {
  pdl_wait();
  pdl_trigger();
  __shared__ double red[32][33];
  const int run = threadIdx.x >> 3, k4 = threadIdx.x & 7, width = 3 * cols;
  const int i = ((int)blockIdx.x * 8 + k4) * 4, per = (n + 31) / 32, k0 = run * per, k1 = min(n, k0 + per);
  double v[4] = {0., 0., 0., 0.};
  if (i < width) {
#pragma unroll 5
    for (int k = k0; k < k1; k += 2) {                        // (pairs in 32 bits: half the conversions)
      const float4 e = *reinterpret_cast<const float4*>(part + (long long)k * width + i);
      const float4 f = k + 1 < k1 ? *reinterpret_cast<const float4*>(part + (long long)(k + 1) * width + i) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[0] += e.x + f.x; v[1] += e.y + f.y; v[2] += e.z + f.z; v[3] += e.w + f.w;
    }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) red[run][4 * k4 + j] = v[j];
  __syncthreads();
  const int c = (int)threadIdx.x, o = (int)blockIdx.x * 32 + c;
  if (c >= 32 || o >= width) return;
  double t = red[0][c];
#pragma unroll
  for (int w = 1; w < 32; ++w) t += red[w][c];
  const int pl = o / cols;
  (pl == 0 ? out0 : (pl == 1 ? out1 : out2))[o - pl * cols] = (float)t;
}

// ------------------------------------------------------------------ column sums over rows
// out0[c] = sum_r a[r,c];  with y and a2 also out1[c] = sum_r a[r,c] * (y[r,c] - mean[r]) * rstd[r] and out2[c] = sum_r a2[r,c].
// A block of 8 x 32 threads owns 8*V columns (one 128-byte line per row for 16-byte vectors) of
// one chunk of rows (gridDim.y chunks): a thread keeps NB rows' loads in flight (as many as the registers hold for one
// or three tensors: latency bounds this kernel) and adds them in row
// order, the block adds its 32 row groups in index order; the last block to finish a column group (ticket
// counter) adds the chunks' partials in index order, so the result does not depend on scheduling.
// Four rows at a time whatever the tensors, and eight chunks at a time in the last block: 11 x 200 tokens, hidden 768, gradients 394 -> 391 us;
// 32 x 128, hidden 1024, six layers 3559 -> 3540 (both before the sums of three tensors joined the LayerNorm backward, which leaves
// this kernel those of rows too wide for it and those of one tensor).
constexpr int COLRED_CT = 8, COLRED_RT = 32;
template <typename T, int V, bool ALL, int NB>
__global__ void __launch_bounds__(256, 2) col_reduce_kernel(const T* __restrict__ a, long long ld_a,
                                                            const T* __restrict__ y, const float* __restrict__ mean,
                                                            const float* __restrict__ rstd, const T* __restrict__ a2,
                                                            long long ld_a2, long long rows, int cols,
                                                            float* __restrict__ out0, float* __restrict__ out1,
                                                            float* __restrict__ out2, float* __restrict__ scratch,
                                                            long long plane, int* __restrict__ counters) {
  pdl_wait();
  pdl_trigger();
  constexpr int BC = COLRED_CT * V;                        // columns per block
  constexpr int PLANES = ALL ? 3 : 1;
  __shared__ float sh[PLANES][COLRED_RT][BC + 1];
  __shared__ int is_last;
  const int tx = threadIdx.x % COLRED_CT, ty = threadIdx.x / COLRED_CT;
  const int c = blockIdx.x * BC + tx * V;
  const int chunks = gridDim.y;
  const long long per = (rows + chunks - 1) / chunks;
  const long long r0 = blockIdx.y * per, r1 = r0 + per < rows ? r0 + per : rows;
  float a0[V], a1[V], a2s[V];
#pragma unroll
  for (int j = 0; j < V; ++j) a0[j] = a1[j] = a2s[j] = 0.f;
  if (c < cols) {
    constexpr int RW = RawWords<T, V>::N;
    for (long long rb = r0 + ty; rb < r1; rb += NB * COLRED_RT) {
      uint32_t v[NB][RW], w[ALL ? NB : 1][RW], u[ALL ? NB : 1][RW];
      float mu[NB], rs[NB];
#pragma unroll
      for (int k = 0; k < NB; ++k) {                      // all loads of NB rows first (raw words: few registers)
        const long long r = rb + COLRED_RT * k;
        if (r < r1) {
          load_raw<T, V>(a + r * ld_a + c, v[k]);
          if (ALL) {
            load_raw<T, V>(y + r * cols + c, w[k]);
            mu[k] = mean[r]; rs[k] = rstd[r];
            load_raw<T, V>(a2 + r * ld_a2 + c, u[k]);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        if (rb + COLRED_RT * k < r1) {
          float fv[V], fw[V];
          widen_raw<T, V>(v[k], fv);
#pragma unroll
          for (int j = 0; j < V; ++j) a0[j] += fv[j];
          if (ALL) {
            widen_raw<T, V>(w[k], fw);
#pragma unroll
            for (int j = 0; j < V; ++j) a1[j] += fv[j] * (fw[j] - mu[k]) * rs[k];
            widen_raw<T, V>(u[k], fw);
#pragma unroll
            for (int j = 0; j < V; ++j) a2s[j] += fw[j];
          }
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < V; ++j) {
    sh[0][ty][tx * V + j] = a0[j];
    if constexpr (ALL) { sh[1][ty][tx * V + j] = a1[j]; sh[2][ty][tx * V + j] = a2s[j]; }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < PLANES * BC; i += 256) {
    const int pl = i / BC, col = i - pl * BC, cc = blockIdx.x * BC + col;
    if (cc >= cols) continue;
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < COLRED_RT; ++k) t += sh[pl][k][col];
    scratch[pl * plane + (long long)blockIdx.y * cols + cc] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(&counters[blockIdx.x], 1) == chunks - 1;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  for (int i = threadIdx.x; i < PLANES * BC; i += 256) {
    const int pl = i / BC, col = i - pl * BC, cc = blockIdx.x * BC + col;
    if (cc >= cols) continue;
    const float* src = scratch + pl * plane + cc;
    float t = 0.f;
    for (int k0 = 0; k0 < chunks; k0 += 24) {              // up to 24 loads in flight, added in index order
      float q[24];
#pragma unroll
      for (int k = 0; k < 24; ++k) q[k] = k0 + k < chunks ? src[(long long)(k0 + k) * cols] : 0.f;
#pragma unroll
      for (int k = 0; k < 24; ++k) t += q[k];
    }
    float* out = pl == 0 ? out0 : (pl == 1 ? out1 : out2);
    out[cc] = t;
  }
  if (threadIdx.x == 0) counters[blockIdx.x] = 0;         // ready for the next launch on this stream
}

// ------------------------------------------------------------------ softmax forward
// CACHED: S % 4 == 0 and S <= 128 * MAXNV; the row of scores stays in registers.
template <typename T, bool CACHED>
__global__ void __launch_bounds__(128) softmax_fwd_kernel(const float* __restrict__ scores,
                                                          const int* __restrict__ valid_len, int h, int S,
                                                          long long rows, T* __restrict__ P,
                                                          const float* __restrict__ step,
                                                          const float* __restrict__ offset, float lo, float hi,
                                                          T* __restrict__ qt) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const long long row = blockIdx.x * 4ll + (threadIdx.x >> 5);
  if (row >= rows) return;
  const int b = (int)(row / ((long long)h * S));
  int len = valid_len ? valid_len[b] : S;
  len = len < 1 ? 1 : (len > S ? S : len);
  const float* sr = scores + row * S;
  const float s = step ? *step : 1.f;
  const bool has_off = offset != nullptr;
  const float off = has_off ? *offset : 0.f;
  if constexpr (CACHED) {
    float e[MAXNV][4];
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < MAXNV; ++i) {
      const int c = (lane + 32 * i) * 4;
      if (c < S) {
        load4<float>(sr + c, e[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) if (c + j < len) mx = fmaxf(mx, e[i][j]);
      }
    }
    mx = warp_max(mx);
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < MAXNV; ++i) {
      const int c = (lane + 32 * i) * 4;
      if (c < S) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          e[i][j] = c + j < len ? expf(e[i][j] - mx) : 0.f;
          sum += e[i][j];
        }
      }
    }
    sum = warp_sum(sum);
#pragma unroll
    for (int i = 0; i < MAXNV; ++i) {
      const int c = (lane + 32 * i) * 4;
      if (c < S) {
#pragma unroll
        for (int j = 0; j < 4; ++j) e[i][j] = __fdiv_rn(e[i][j], sum);
        store4<T>(P + row * S + c, e[i]);
        if (qt) {
#pragma unroll
          for (int j = 0; j < 4; ++j) e[i][j] = (float)qcode(qz(stored<T>(e[i][j]), s, off, has_off), lo, hi);
          store4<T>(qt + row * S + c, e[i]);
        }
      }
    }
  } else {
    float mx = -INFINITY;
    for (int j = lane; j < len; j += 32) mx = fmaxf(mx, sr[j]);
    mx = warp_max(mx);
    float sum = 0.f;
    for (int j = lane; j < len; j += 32) sum += expf(sr[j] - mx);
    sum = warp_sum(sum);
    for (int j = lane; j < S; j += 32) {
      const float p = j < len ? __fdiv_rn(expf(sr[j] - mx), sum) : 0.f;
      P[row * S + j] = from_f<T>(p);
      if (qt) qt[row * S + j] = from_f<T>((float)qcode(qz(stored<T>(p), s, off, has_off), lo, hi));
    }
  }
}

// ------------------------------------------------------------------ softmax backward with the STE of the P quantizer
template <typename T, bool CACHED>
__global__ void __launch_bounds__(256) softmax_bwd_kernel(const T* __restrict__ P, const T* __restrict__ dphat,
                                                          T* __restrict__ dS, long long rows, int S,
                                                          const float* __restrict__ step, float lo, float hi,
                                                          int quantized, float* __restrict__ part_s) {
  pdl_wait();
  pdl_trigger();
  __shared__ float sh[32];
  const int lane = threadIdx.x & 31;
  const long long warp0 = blockIdx.x * 8ll + (threadIdx.x >> 5), nwarps = gridDim.x * 8ll;
  const float s = quantized ? *step : 1.f, r_s = __frcp_rn(s);
  float ds = 0.f;
  for (long long row = warp0; row < rows; row += nwarps) {
    const long long base = row * S;
    if constexpr (CACHED) {
      float p[MAXNV][4], d[MAXNV][4];
      float dot = 0.f;
#pragma unroll
      for (int i = 0; i < MAXNV; ++i) {
        const int c = (lane + 32 * i) * 4;
        if (c < S) {
          load4<T>(P + base + c, p[i]);
          load4<T>(dphat + base + c, d[i]);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (quantized) {
              const float z = quotient(p[i][j], s, r_s);
              const bool in = z >= lo && z <= hi;
              ds += d[i][j] * ((float)qcode(z, lo, hi) - (in ? z : 0.f));
              d[i][j] = in ? d[i][j] : 0.f;
            }
            dot += d[i][j] * p[i][j];
          }
        }
      }
      dot = warp_sum(dot);
#pragma unroll
      for (int i = 0; i < MAXNV; ++i) {
        const int c = (lane + 32 * i) * 4;
        if (c < S) {
#pragma unroll
          for (int j = 0; j < 4; ++j) d[i][j] = p[i][j] * (d[i][j] - dot);
          store4<T>(dS + base + c, d[i]);
        }
      }
    } else {
      float dot = 0.f;
      for (int j = lane; j < S; j += 32) {
        const float p = to_f<T>(P[base + j]);
        float d = to_f<T>(dphat[base + j]);
        if (quantized) {
          const float z = quotient(p, s, r_s);
          const bool in = z >= lo && z <= hi;
          ds += d * ((float)qcode(z, lo, hi) - (in ? z : 0.f));
          d = in ? d : 0.f;
        }
        dot += d * p;
      }
      dot = warp_sum(dot);
      for (int j = lane; j < S; j += 32) {
        const float p = to_f<T>(P[base + j]);
        float d = to_f<T>(dphat[base + j]);
        if (quantized) {
          const float z = quotient(p, s, r_s);
          d = (z >= lo && z <= hi) ? d : 0.f;
        }
        dS[base + j] = from_f<T>(p * (d - dot));
      }
    }
  }
  ds = block_sum(ds, sh);
  if (threadIdx.x == 0 && part_s) part_s[blockIdx.x] = ds;
}

inline bool al16(const void* p) { return p == nullptr || (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

#define MREM_DT(dt, T, ...)            \
  do {                                 \
    if ((dt) == 1) { using T = bf16; __VA_ARGS__; } else { using T = float; __VA_ARGS__; } \
  } while (0)

void launch_layernorm_fwd(const void* y, const float* gamma, const float* beta, float eps, long long rows, int cols,
                          void* out, float* mean, float* rstd, const float* step, int qmax, int8_t* q8, void* qt,
                          int dt, cudaStream_t st) {
  if (rows <= 0) return;
  Scope sc("layernorm_fwd", (double)rows * cols * ((dt == 1 ? 2.0 : 4.0) * (qt ? 3 : 2) + (q8 ? 1 : 0)), 0, st);
  const int grid = (int)((rows + 3) / 4);
  MREM_DT(dt, T, {
    constexpr int V = 16 / (int)sizeof(T);
    const bool v = cols % V == 0 && cols <= 32 * V * MAXNV && al16(y) && al16(out) && al16(qt) && al16(gamma) && al16(beta) &&
                   (reinterpret_cast<uintptr_t>(q8) % V) == 0;
    if (v) launch_k(ln_fwd_kernel<T, V, true>, grid, 128, 0, st, (const T*)y, gamma, beta, eps, rows, cols, (T*)out, mean, rstd, step, (float)qmax, q8, (T*)qt);
    else launch_k(ln_fwd_kernel<T, 1, false>, grid, 128, 0, st, (const T*)y, gamma, beta, eps, rows, cols, (T*)out, mean, rstd, step, (float)qmax, q8, (T*)qt);
  });
}

void launch_layernorm_bwd(const void* dout, const void* dout2, const void* y, const float* mean, const float* rstd,
                          const float* gamma, long long rows, int cols, void* dy, void* dsum, int dt,
                          cudaStream_t st) {
  if (rows <= 0) return;
  Scope sc("layernorm_bwd", (double)rows * cols * (dt == 1 ? 2.0 : 4.0) * (3 + (dout2 ? 1 : 0) + (dsum ? 1 : 0)), 0, st);
  const int grid = (int)((rows + 3) / 4);
  MREM_DT(dt, T, {
    constexpr int V = 16 / (int)sizeof(T);
    const bool v = cols % V == 0 && cols <= 32 * V * MAXNV && al16(dout) && al16(dout2) && al16(y) && al16(dy) && al16(dsum) && al16(gamma);
    if (v) launch_k(ln_bwd_kernel<T, V, true>, grid, 128, 0, st, (const T*)dout, (const T*)dout2, (const T*)y, mean, rstd, gamma, rows, cols, (T*)dy, (T*)dsum);
    else launch_k(ln_bwd_kernel<T, 1, false>, grid, 128, 0, st, (const T*)dout, (const T*)dout2, (const T*)y, mean, rstd, gamma, rows, cols, (T*)dy, (T*)dsum);
  });
}

// Warps that share a row of the kernel with column sums; 0: rows it does not take.
static int ln_cols_warps(int cols, int dt) {
  const int V = dt == 1 ? 8 : 4;
  return cols % V == 0 && cols <= 32 * V * MAXNV ? (cols + 32 * V - 1) / (32 * V) : 0;
}
bool layernorm_bwd_cols_supported(int cols, int dt) { return ln_cols_warps(cols, dt) > 0; }
// groups: two rows each while there are fewer rows than that takes.  Narrow rows have more groups, as many as the bytes of LN_PARTS partial
// sums 512 wide: with LN_PARTS a few warps per SM walked ten rows each, and a step of 48 x 128 tokens took 489 us at hidden 128 (now 459;
// 463 with the sums in a launch of their own) and 606 at hidden 256 (582; 593), but 612 with four times LN_PARTS.
static int ln_cols_grid(long long rows, int cols, int W) {
  const int per = ln_groups(W) * LN_ROWS;
  int parts = LN_PARTS * 512 / cols;
  parts = parts < LN_PARTS ? LN_PARTS : (parts > 4 * LN_PARTS ? 4 * LN_PARTS : parts);
  const long long want = (rows + per - 1) / per, limit = parts / ln_groups(W);
  return (int)(want < limit ? want : limit);
}
size_t layernorm_bwd_cols_floats(long long rows, int cols, int dt) {
  const int W = ln_cols_warps(cols, dt);
  return W == 0 ? 0 : (size_t)ln_cols_grid(rows, cols, W) * ln_groups(W) * 3 * cols;
}

int launch_layernorm_bwd_cols(const void* dout, const void* x, const void* dxhat, const void* add, const float* step, int lo, int hi,
                              const void* y, const float* mean, const float* rstd, const float* gamma, long long rows, int cols,
                              void* dy, float* part_s, float* col_part, int dt, cudaStream_t st) {
  const int W = ln_cols_warps(cols, dt);
  if (rows <= 0 || W == 0 || !(al16(dout) && al16(x) && al16(dxhat) && al16(add) && al16(y) && al16(dy) && al16(gamma))) return 0;
  Scope sc(x ? "layernorm_bwd_ste" : "layernorm_bwd", (double)rows * cols * (dt == 1 ? 2.0 : 4.0) * (x ? (dout ? 6 : 5) : 3), 0, st);
  const int grid = ln_cols_grid(rows, cols, W);
#define MREM_LN(T, V, W, STE) launch_k(ln_bwd_cols_kernel<T, V, W, STE>, grid, 32 * W * ln_groups(W), 0, st, (const T*)dout, (const T*)x, (const T*)dxhat, (const T*)add, step, (float)lo, (float)hi, (const T*)y, mean, rstd, gamma, rows, cols, (T*)dy, part_s, RED_BLOCKS, col_part)
#define MREM_LNS(T, V, STE) do { if (W == 1) MREM_LN(T, V, 1, STE); else if (W == 2) MREM_LN(T, V, 2, STE); else if (W == 3) MREM_LN(T, V, 3, STE); else MREM_LN(T, V, 4, STE); } while (0)
  if (dt == 1) { if (x) MREM_LNS(bf16, 8, true); else MREM_LNS(bf16, 8, false); }
  else { if (x) MREM_LNS(float, 4, true); else MREM_LNS(float, 4, false); }
#undef MREM_LNS
#undef MREM_LN
  return grid * ln_groups(W);
}

void launch_col_finish(const float* col_part, int n, int cols, float* out0, float* out1, float* out2, cudaStream_t st) {
  Scope sc("col_reduce", (double)n * cols * 12.0, 0, st);
  launch_k(col_finish_kernel, (3 * cols + 31) / 32, 256, 0, st, col_part, n, cols, out0, out1, out2);
}

void launch_col_reduce(const void* a, long long ld_a, const void* y, const float* mean, const float* rstd,
                       const void* a2, long long ld_a2, long long rows, int cols, float* out0, float* out1,
                       float* out2, float* scratch, long long plane_floats, int* counters, int dt, cudaStream_t st) {
  Scope sc("col_reduce", (double)rows * cols * (dt == 1 ? 2.0 : 4.0) * (y ? 3 : 1), 0, st);
  // (y and a2 come together)
  // as many row chunks as one plane of the scratch holds, up to two blocks per SM (one wave) and 128 rows per chunk
#define MREM_COLRED(T, V) do { const int col_blocks = (cols + COLRED_CT * V - 1) / (COLRED_CT * V); \
    long long chunks = plane_floats / cols; \
    if (chunks > 288 / col_blocks) chunks = 288 / col_blocks; \
    if (chunks > (rows + 4 * COLRED_RT - 1) / (4 * COLRED_RT)) chunks = (rows + 4 * COLRED_RT - 1) / (4 * COLRED_RT); \
    if (chunks < 1) chunks = 1; \
    dim3 grid(col_blocks, (unsigned)chunks); \
    if (y) MREM_COLRED_K(T, V, true, 4); \
    else MREM_COLRED_K(T, V, false, 12); } while (0)
#define MREM_COLRED_K(T, V, ALL, NB) launch_k(col_reduce_kernel<T, V, ALL, NB>, grid, 256, 0, st, (const T*)a, ld_a, (const T*)y, mean, rstd, (const T*)a2, ld_a2, rows, cols, out0, out1, out2, scratch, plane_floats, counters)
  const bool vec_ok = cols % 8 == 0 && ld_a % 8 == 0 && ld_a2 % 8 == 0 && al16(a) && al16(y) && al16(a2);
  if (dt == 1) { if (vec_ok) MREM_COLRED(bf16, 8); else MREM_COLRED(bf16, 1); }
  else { if (vec_ok) MREM_COLRED(float, 4); else MREM_COLRED(float, 1); }
#undef MREM_COLRED_K
#undef MREM_COLRED
}

void launch_softmax_fwd(const float* scores, const int* valid_len, int B, int h, int S, void* P, const float* step,
                        const float* offset, int lo, int hi, void* qt, int dt, cudaStream_t st) {
  const long long rows = (long long)B * h * S;
  if (rows <= 0) return;
  Scope sc("softmax_fwd", (double)rows * S * (4.0 + (dt == 1 ? 2.0 : 4.0) * (qt ? 2 : 1)), 0, st);
  const int grid = (int)((rows + 3) / 4);
  const bool cached = S % 4 == 0 && S <= 128 * MAXNV && al16(scores) && al16(P) && al16(qt);
  MREM_DT(dt, T, {
    if (cached) launch_k(softmax_fwd_kernel<T, true>, grid, 128, 0, st, scores, valid_len, h, S, rows, (T*)P, step, offset, (float)lo, (float)hi, (T*)qt);
    else launch_k(softmax_fwd_kernel<T, false>, grid, 128, 0, st, scores, valid_len, h, S, rows, (T*)P, step, offset, (float)lo, (float)hi, (T*)qt);
  });
}

void launch_softmax_bwd(const void* P, const void* dphat, void* dS, long long rows, int S, const float* step,
                        int lo, int hi, int quantized, float* part_s, int dt, cudaStream_t st) {
  Scope sc("softmax_bwd", (double)rows * S * 3 * (dt == 1 ? 2.0 : 4.0), 0, st);
  const bool cached = S % 4 == 0 && S <= 128 * MAXNV && al16(P) && al16(dphat) && al16(dS);
  MREM_DT(dt, T, {
    if (cached) launch_k(softmax_bwd_kernel<T, true>, RED_BLOCKS, 256, 0, st, (const T*)P, (const T*)dphat, (T*)dS, rows, S, step, (float)lo, (float)hi, quantized, part_s);
    else launch_k(softmax_bwd_kernel<T, false>, RED_BLOCKS, 256, 0, st, (const T*)P, (const T*)dphat, (T*)dS, rows, S, step, (float)lo, (float)hi, quantized, part_s);
  });
}

}  // namespace mrem
