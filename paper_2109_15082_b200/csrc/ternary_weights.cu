// Weight codes whose scale is recomputed from the weights instead of learnt (Sec. 5.1 names one such rule for 2-bit
// and one for 4-bit weights), one block per output row.
//
// Ternary rule (2-bit):  delta = 0.7 * mean|w|,  t = sign(w) * 1[|w| > delta],  alpha = mean of |w| over the kept
// entries (0 when none is kept),  w_hat = alpha * t.  Nothing is learnt about the scale: the update is
// AdamW on the latent weights with the gradient of w_hat passed through unchanged, followed by the same
// rule on the new weights.  Both means are accumulated in float64 in a fixed order and the comparison
// |w| > delta is made in float32 on float32(delta), so the codes are a function of the stored weights
// alone.  Two kernels share the row routine: the stand-alone quantizer and the fused update.
//
// Refitted scale (b-bit, the loss-aware rule read with unit curvature weights): minimise ||w - alpha q||^2 over
// alpha and q in Omega(b)^n by alternating the two exact half-steps  q = Pi_Omega(b)(w / alpha)  (Eq. 1, float32
// division)  and  alpha = <q, w> / <q, q>  (alpha rounded to float32), LAQ_ROUNDS times from
// alpha_0 = min(3 mean|w|, max|w|) / qmax; a row of zeros keeps alpha = 0 and codes 0.  A round is a function of alpha
// alone, so a round that returns the alpha it was given ends the loop: all later rounds would repeat it (Gaussian rows
// 768 wide need 10 rounds on average, 1024 wide 11, 3072 wide 14 of the 15).
#include "optim.cuh"

namespace mrem {

namespace {

// Ternary rule: 256 threads per row, up to 4 float4 vectors per thread in registers (rows up to 4096 wide).  Refitted
// scale: two vectors per thread and as many threads as that takes (rows up to 4096 wide; 96 threads for 768, 384 for
// 3072: no idle lanes at the encoder's widths).  Wider rows are re-read by 256 threads.
constexpr int TW_THREADS = 256;
constexpr int TW_MAXV = 4;
constexpr int LAQ_V = 2;
constexpr int LAQ_MAX_WARPS = 16;

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum_d(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double r = (lane < nw) ? sh[lane] : 0.0;
  return warp_sum_d(r);
}
__device__ __forceinline__ int block_sum_i(int v, int* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum_i(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  int r = (lane < nw) ? sh[lane] : 0;
  return warp_sum_i(r);
}

template <typename T>
__device__ __forceinline__ void store4(T* p, float a, float b, float c, float d);
template <>
__device__ __forceinline__ void store4<float>(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
template <>
__device__ __forceinline__ void store4<bf16>(bf16* p, float a, float b, float c, float d) {
  uint2 t;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&t);
  h[0] = __floats2bfloat162_rn(a, b);
  h[1] = __floats2bfloat162_rn(c, d);
  *reinterpret_cast<uint2*>(p) = t;
}

__device__ __forceinline__ int tern(float w, float delta) { return fabsf(w) > delta ? (w > 0.f ? 1 : -1) : 0; }

// The rule on one row.  `cached`: the row sits in wr[] (vector c = threadIdx.x + i * NT), else it is re-read
// from w_row.  Writes codes, row sum, scale and the dequantized row.
template <typename T, int NT, int MAXV>
__device__ __forceinline__ void ternary_row(const float4* wr, bool cached, const float* w_row, int cols, int row,
                                            int8_t* codes_row, int32_t* rowsum, float* scale, T* what_row,
                                            double* shd, int* shi) {
  const int nvec = cols / 4;
  double s = 0.0;
  if (cached) {
#pragma unroll
    for (int i = 0; i < MAXV; ++i) {
      const int c = threadIdx.x + i * NT;
      if (c < nvec) s += (double)fabsf(wr[i].x) + (double)fabsf(wr[i].y) + (double)fabsf(wr[i].z) + (double)fabsf(wr[i].w);
    }
  } else {
    for (int c = threadIdx.x; c < nvec; c += NT) {
      const float4 v = reinterpret_cast<const float4*>(w_row)[c];
      s += (double)fabsf(v.x) + (double)fabsf(v.y) + (double)fabsf(v.z) + (double)fabsf(v.w);
    }
  }
  s = block_sum_d(s, shd);
  const float delta = (float)(0.7 * (s / (double)cols));
  double ks = 0.0;
  int cnt = 0;
  auto acc = [&](float4 v) {
    if (fabsf(v.x) > delta) { ks += (double)fabsf(v.x); ++cnt; }
    if (fabsf(v.y) > delta) { ks += (double)fabsf(v.y); ++cnt; }
    if (fabsf(v.z) > delta) { ks += (double)fabsf(v.z); ++cnt; }
    if (fabsf(v.w) > delta) { ks += (double)fabsf(v.w); ++cnt; }
  };
  if (cached) {
#pragma unroll
    for (int i = 0; i < MAXV; ++i) {
      const int c = threadIdx.x + i * NT;
      if (c < nvec) acc(wr[i]);
    }
  } else {
    for (int c = threadIdx.x; c < nvec; c += NT) acc(reinterpret_cast<const float4*>(w_row)[c]);
  }
  ks = block_sum_d(ks, shd);
  cnt = block_sum_i(cnt, shi);
  const float alpha = (float)(ks / (double)(cnt > 0 ? cnt : 1));
  int sum = 0;
  auto emit = [&](int c, float4 v) {
    const int q0 = tern(v.x, delta), q1 = tern(v.y, delta), q2 = tern(v.z, delta), q3 = tern(v.w, delta);
    *reinterpret_cast<uint32_t*>(codes_row + 4 * c) =
        (uint32_t)(q0 & 0xff) | ((uint32_t)(q1 & 0xff) << 8) | ((uint32_t)(q2 & 0xff) << 16) | ((uint32_t)(q3 & 0xff) << 24);
    if (what_row) store4<T>(what_row + 4 * c, alpha * (float)q0, alpha * (float)q1, alpha * (float)q2, alpha * (float)q3);
    sum += q0 + q1 + q2 + q3;
  };
  if (cached) {
#pragma unroll
    for (int i = 0; i < MAXV; ++i) {
      const int c = threadIdx.x + i * NT;
      if (c < nvec) emit(c, wr[i]);
    }
  } else {
    for (int c = threadIdx.x; c < nvec; c += NT) emit(c, reinterpret_cast<const float4*>(w_row)[c]);
  }
  sum = block_sum_i(sum, shi);
  if (threadIdx.x == 0) {
    rowsum[row] = sum;
    scale[row] = alpha;
  }
}

constexpr int LAQ_ROUNDS = 16;

__device__ __forceinline__ int laq_code(float w, float alpha, float qmax) {
  return __float2int_rn(fminf(fmaxf(__fdiv_rn(w, alpha), -qmax), qmax));
}
// The same code from RN(1 / alpha): quotient() differs from the division only where w / alpha lies within 2^-48
// (relative) of the midpoint of two floats, and the code differs only if that quotient is also next to a half-integer.
// Used in the rounds that only feed the two sums; the codes that are written out come from the division.
__device__ __forceinline__ int laq_code_fast(float w, float alpha, float r_alpha, float qmax) {
  return __float2int_rn(fminf(fmaxf(quotient(w, alpha, r_alpha), -qmax), qmax));
}
// (double)q for |q| < 2^31 without the conversion unit: 2^52 + 2^31 + q is exact in the low word of a double.
__device__ __forceinline__ double int_as_double(int q) {
  return __hiloint2double(0x43300000, (int)(0x80000000u ^ (unsigned)q)) - 4503601774854144.0;
}

// Block-wide sum of a double and of an int in one pass.  Every thread gets the results.
__device__ __forceinline__ void block_sum_di(double& a, int& n, double* shd, int* shi) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  a = warp_sum_d(a);
  n = __reduce_add_sync(0xffffffffu, n);
  __syncthreads();
  if (lane == 0) { shd[w] = a; shi[w] = n; }
  __syncthreads();
  a = warp_sum_d(lane < nw ? shd[lane] : 0.0);
  n = __reduce_add_sync(0xffffffffu, lane < nw ? shi[lane] : 0);
}

// The alternating rule on a row too wide for registers, re-read in every round.
template <typename T, int NT>
__device__ __forceinline__ void laq_row(const float* w_row, int cols, int row, int bits, int8_t* codes_row, int32_t* rowsum,
                                        float* scale, T* what_row, double* shd, int* shi, float* shf) {
  const int nvec = cols / 4;
  const float qmax = (float)((1 << (bits - 1)) - 1);
  auto for_row = [&](auto&& f) {
    for (int c = threadIdx.x; c < nvec; c += NT) f(c, reinterpret_cast<const float4*>(w_row)[c]);
  };
  double s = 0.0;
  float mx = 0.f;
  for_row([&](int, float4 v) {
    s += (double)fabsf(v.x) + (double)fabsf(v.y) + (double)fabsf(v.z) + (double)fabsf(v.w);
    mx = fmaxf(fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
  });
  s = block_sum_d(s, shd);
  mx = block_max(mx, shf);
  float alpha = (float)(fmin(3.0 * (s / (double)cols), (double)mx) / (double)qmax);
  for (int r = 0; r + 1 < LAQ_ROUNDS; ++r) {
    double qw = 0.0, qw1 = 0.0, qw2 = 0.0, qw3 = 0.0;
    int qq = 0;
    auto sums = [&](auto code) {
      for_row([&](int, float4 v) {
        const int q0 = code(v.x), q1 = code(v.y), q2 = code(v.z), q3 = code(v.w);
        qw = fma(int_as_double(q0), (double)v.x, qw);              // four independent chains
        qw1 = fma(int_as_double(q1), (double)v.y, qw1);
        qw2 = fma(int_as_double(q2), (double)v.z, qw2);
        qw3 = fma(int_as_double(q3), (double)v.w, qw3);
        qq += q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3;
      });
    };
    if (alpha > 1e-30f) {                                  // 1 / alpha and the residual stay in the normal range
      const float r_alpha = __frcp_rn(alpha);
      sums([&](float w) { return laq_code_fast(w, alpha, r_alpha, qmax); });
    } else if (alpha > 0.f) {
      sums([&](float w) { return laq_code(w, alpha, qmax); });
    }
    qw = (qw + qw1) + (qw2 + qw3);
    block_sum_di(qw, qq, shd, shi);
    const float next = qq > 0 ? (float)(qw / (double)qq) : 0.f;
    if (next == alpha) break;
    alpha = next;
  }
  // last round: the codes of this alpha (by the division of Eq. 1) go out with the scale refitted to them
  double qw = 0.0;
  int qq = 0, sum = 0;
  for_row([&](int c, float4 v) {
    int q0 = 0, q1 = 0, q2 = 0, q3 = 0;
    if (alpha > 0.f) {
      q0 = laq_code(v.x, alpha, qmax); q1 = laq_code(v.y, alpha, qmax);
      q2 = laq_code(v.z, alpha, qmax); q3 = laq_code(v.w, alpha, qmax);
    }
    qw += (double)q0 * (double)v.x + (double)q1 * (double)v.y + (double)q2 * (double)v.z + (double)q3 * (double)v.w;
    qq += q0 * q0 + q1 * q1 + q2 * q2 + q3 * q3;
    sum += q0 + q1 + q2 + q3;
    *reinterpret_cast<uint32_t*>(codes_row + 4 * c) =
        (uint32_t)(q0 & 0xff) | ((uint32_t)(q1 & 0xff) << 8) | ((uint32_t)(q2 & 0xff) << 16) | ((uint32_t)(q3 & 0xff) << 24);
  });
  block_sum_di(qw, qq, shd, shi);
  const float next = qq > 0 ? (float)(qw / (double)qq) : 0.f;
  if (what_row) {
    auto unpack = [](uint32_t pk, int j) { return (float)(int)(int8_t)(pk >> (8 * j)); };
    for (int c = threadIdx.x; c < nvec; c += NT) {        // this thread's own codes, written above
      const uint32_t pk = *reinterpret_cast<const uint32_t*>(codes_row + 4 * c);
      store4<T>(what_row + 4 * c, next * unpack(pk, 0), next * unpack(pk, 1), next * unpack(pk, 2), next * unpack(pk, 3));
    }
  }
  sum = block_sum_i(sum, shi);
  if (threadIdx.x == 0) {
    rowsum[row] = sum;
    scale[row] = next;
  }
}

// The rule on a row held in registers, LAQ_V vectors per thread (missing ones are zeros: their code is 0 and they add
// nothing).  The rounds that only feed the two sums get them without float64 arithmetic per weight: w / 2^(e - 23), e = the
// exponent of max|w|, is split once into two integers of 12 bits and a rest of at most 1/2,
//   w = (4096 nh + nm + nl) 2^(e - 23),
// so that sums of q nh and q nm over a thread's weights are exact in float32 (below 2^24 for codes of up to 4 bits) and, as
// integers, over the block; the rest enters at 2^-39 of max|w|.  7 instructions per weight and round instead of 38, four
// integer warp reductions instead of a float64 butterfly, one barrier instead of two.
// BERT-base module of three layers: step 1801 -> 1693 us.
struct LaqShared { int4 sums[2][LAQ_MAX_WARPS]; double d[32]; int i[64]; float f[32]; };

template <typename T>
__device__ __forceinline__ void laq_row_cached(const float4 (&wr)[LAQ_V], int cols, int row, int bits, int8_t* codes_row,
                                               int32_t* rowsum, float* scale, T* what_row, LaqShared& sh) {
  constexpr int NW = 4 * LAQ_V;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, nvec = cols / 4;
  const float qmax = (float)((1 << (bits - 1)) - 1);
  float2 w[NW / 2];
#pragma unroll
  for (int i = 0; i < LAQ_V; ++i) { w[2 * i] = make_float2(wr[i].x, wr[i].y); w[2 * i + 1] = make_float2(wr[i].z, wr[i].w); }
  double s = 0.0;
  float mx = 0.f;
#pragma unroll
  for (int e = 0; e < NW / 2; ++e) {
    s += (double)fabsf(w[e].x) + (double)fabsf(w[e].y);
    mx = fmaxf(mx, fmaxf(fabsf(w[e].x), fabsf(w[e].y)));
  }
  s = block_sum_d(s, sh.d);
  mx = block_max(mx, sh.f);
  float alpha = (float)(fmin(3.0 * (s / (double)cols), (double)mx) / (double)qmax);
  const bool split = bits <= 4 && mx > 1e-30f && mx < 1e30f;
  const int ex = (int)((__float_as_uint(mx) >> 23) & 255u) - 127;
  float2 nh[NW / 2], nm[NW / 2], nl[NW / 2];
  double unit = 0.0;                                       // 2^(ex - 23)
  if (split) {
    const float inv_u = __uint_as_float((uint32_t)(127 + 11 - ex) << 23);
    unit = (double)__uint_as_float((uint32_t)(127 - 23 + ex) << 23);
#pragma unroll
    for (int e = 0; e < NW / 2; ++e) {
      const float tx = w[e].x * inv_u, ty = w[e].y * inv_u;     // exact, below 2^12
      nh[e] = make_float2(rne_magic(tx), rne_magic(ty));
      const float ux = (tx - nh[e].x) * 4096.f, uy = (ty - nh[e].y) * 4096.f;
      nm[e] = make_float2(rne_magic(ux), rne_magic(uy));
      nl[e] = make_float2(ux - nm[e].x, uy - nm[e].y);
    }
  }
  for (int r = 0; r + 1 < LAQ_ROUNDS; ++r) {
    float next;
    if (split && alpha > 1e-30f) {                         // 1 / alpha and the residual stay in the normal range
      const float r_alpha = __frcp_rn(alpha);
      const float2 r2 = make_float2(r_alpha, r_alpha), na2 = make_float2(-alpha, -alpha), magic2 = make_float2(ROUND_MAGIC, ROUND_MAGIC),
                   nmagic2 = make_float2(-ROUND_MAGIC, -ROUND_MAGIC);
      float2 ah = make_float2(0.f, 0.f), am = ah, al = ah, aq = ah;
#pragma unroll
      for (int e = 0; e < NW / 2; ++e) {                   // (quotient() and the rounding on pairs)
        const float2 z0 = mul2(w[e], r2), z = fma2(fma2(z0, na2, w[e]), r2, z0);
        const float2 q = add2(add2(make_float2(fminf(fmaxf(z.x, -qmax), qmax), fminf(fmaxf(z.y, -qmax), qmax)), magic2), nmagic2);
        ah = fma2(q, nh[e], ah);
        am = fma2(q, nm[e], am);
        al = fma2(q, nl[e], al);
        aq = fma2(q, q, aq);
      }
      const int4 mine = make_int4(__reduce_add_sync(0xffffffffu, __float2int_rn(ah.x + ah.y)), __reduce_add_sync(0xffffffffu, __float2int_rn(am.x + am.y)),
                                  __reduce_add_sync(0xffffffffu, __float2int_rn((al.x + al.y) * 65536.f)), __reduce_add_sync(0xffffffffu, __float2int_rn(aq.x + aq.y)));
      if (lane == 0) sh.sums[r & 1][wid] = mine;
      __syncthreads();
      int4 t = make_int4(0, 0, 0, 0);
      if (nw <= 4) {
        for (int k = 0; k < nw; ++k) {
          const int4 v = sh.sums[r & 1][k];
          t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
        }
      } else {
        if (lane < nw) t = sh.sums[r & 1][lane];
        t = make_int4(__reduce_add_sync(0xffffffffu, t.x), __reduce_add_sync(0xffffffffu, t.y), __reduce_add_sync(0xffffffffu, t.z),
                      __reduce_add_sync(0xffffffffu, t.w));
      }
      // <q, w> / <q, q>: float32 quotient and one correction from the float64 residual (2^-46 before the rounding to float32)
      const double qw = fma((double)t.z, 1.52587890625e-05, fma((double)t.x, 4096.0, (double)t.y)) * unit;
      const float rq = __frcp_rn((float)t.w), a0 = (float)qw * rq;
      next = t.w > 0 ? (float)fma(fma(-(double)a0, (double)t.w, qw), (double)rq, (double)a0) : 0.f;
    } else {
      double qw = 0.0;
      int qq = 0;
      if (alpha > 0.f) {
#pragma unroll
        for (int e = 0; e < NW / 2; ++e) {
          const int qx = laq_code(w[e].x, alpha, qmax), qy = laq_code(w[e].y, alpha, qmax);
          qw += (double)qx * (double)w[e].x + (double)qy * (double)w[e].y;
          qq += qx * qx + qy * qy;
        }
      }
      block_sum_di(qw, qq, sh.d, sh.i);
      next = qq > 0 ? (float)(qw / (double)qq) : 0.f;
    }
    if (next == alpha) break;
    alpha = next;
  }
  // last round: the codes of this alpha (by the division of Eq. 1) go out with the scale refitted to them (float64)
  double qw = 0.0;
  int qq = 0, sum = 0;
  float q[NW];
  const bool normal = alpha > 1e-30f && alpha < 1e30f;
  const float r_alpha = __frcp_rn(alpha);
#pragma unroll
  for (int i = 0; i < LAQ_V; ++i) {
    const int c = threadIdx.x + i * blockDim.x;
    uint32_t b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int e = 4 * i + j;
      const float we = (j & 1) ? w[e >> 1].y : w[e >> 1].x;
      int k = 0;
      q[e] = 0.f;
      if (normal) {
        q[e] = code_f<false>(we, alpha, r_alpha, -qmax, qmax, b[j]);
        k = (int)(int8_t)(b[j] & 0xffu);
      } else if (alpha > 0.f) {
        k = laq_code(we, alpha, qmax);
        q[e] = (float)k;
        b[j] = (uint32_t)k;
      }
      qw += int_as_double(k) * (double)we;
      qq += k * k;
      sum += k;
    }
    if (c < nvec) *reinterpret_cast<uint32_t*>(codes_row + 4 * c) = pack_low_bytes(b[0], b[1], b[2], b[3]);
  }
  qw = warp_sum_d(qw);
  qq = __reduce_add_sync(0xffffffffu, qq);
  sum = __reduce_add_sync(0xffffffffu, sum);
  __syncthreads();
  if (lane == 0) { sh.d[wid] = qw; sh.i[wid] = qq; sh.i[32 + wid] = sum; }
  __syncthreads();
  qw = warp_sum_d(lane < nw ? sh.d[lane] : 0.0);
  qq = __reduce_add_sync(0xffffffffu, lane < nw ? sh.i[lane] : 0);
  const float next = qq > 0 ? (float)(qw / (double)qq) : 0.f;
  if (what_row) {
#pragma unroll
    for (int i = 0; i < LAQ_V; ++i) {
      const int c = threadIdx.x + i * blockDim.x;
      if (c < nvec) store4<T>(what_row + 4 * c, next * q[4 * i], next * q[4 * i + 1], next * q[4 * i + 2], next * q[4 * i + 3]);
    }
  }
  if (wid == 0) {
    sum = __reduce_add_sync(0xffffffffu, lane < nw ? sh.i[32 + lane] : 0);
    if (lane == 0) {
      rowsum[row] = sum;
      scale[row] = next;
    }
  }
}

// The two kernels of the refitted scale on rows held in registers; NT: upper bound of the block size.
template <typename T, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) laq_quantize_kernel(const float* __restrict__ w, int cols, int bits,
                                                                     int8_t* __restrict__ codes, int32_t* __restrict__ rowsum,
                                                                     float* __restrict__ scale, T* __restrict__ what) {
  pdl_wait();
  pdl_trigger();
  __shared__ LaqShared sh;
  const long long base = (long long)blockIdx.x * cols;
  const float4* w4 = reinterpret_cast<const float4*>(w + base);
  float4 wr[LAQ_V];
#pragma unroll
  for (int i = 0; i < LAQ_V; ++i) {
    const int c = threadIdx.x + i * blockDim.x;
    wr[i] = c < cols / 4 ? w4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  laq_row_cached<T>(wr, cols, blockIdx.x, bits, codes + base, rowsum, scale, what ? what + base : nullptr, sh);
}

template <typename T, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) laq_update_kernel(float* __restrict__ w, const float* __restrict__ g,
                                                                   float* __restrict__ m, float* __restrict__ v,
                                                                   const OptimScalars* __restrict__ sc, int cols, int train_w,
                                                                   int bits, int8_t* __restrict__ codes,
                                                                   int32_t* __restrict__ rowsum, float* __restrict__ scale,
                                                                   T* __restrict__ what) {
  pdl_wait();
  pdl_trigger();
  __shared__ LaqShared sh;
  const OptimScalars o = *sc;
  const long long base = (long long)blockIdx.x * cols;
  const int nvec = cols / 4;
  float4* w4 = reinterpret_cast<float4*>(w + base);
  const float4* g4 = reinterpret_cast<const float4*>(g + base);
  float4* m4 = reinterpret_cast<float4*>(m + base);
  float4* v4 = reinterpret_cast<float4*>(v + base);
  float4 wr[LAQ_V], gr[LAQ_V], mr[LAQ_V], vr[LAQ_V];
#pragma unroll
  for (int i = 0; i < LAQ_V; ++i) {                        // all loads in flight first
    const int c = threadIdx.x + i * blockDim.x;
    wr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < nvec) {
      wr[i] = w4[c];
      if (train_w) { gr[i] = g4[c]; mr[i] = m4[c]; vr[i] = v4[c]; }
    }
  }
  if (train_w) {
#pragma unroll
    for (int i = 0; i < LAQ_V; ++i) {
      const int c = threadIdx.x + i * blockDim.x;
      if (c < nvec) {
        wr[i].x = adam_one(wr[i].x, gr[i].x, mr[i].x, vr[i].x, o, 1.f, -INFINITY);
        wr[i].y = adam_one(wr[i].y, gr[i].y, mr[i].y, vr[i].y, o, 1.f, -INFINITY);
        wr[i].z = adam_one(wr[i].z, gr[i].z, mr[i].z, vr[i].z, o, 1.f, -INFINITY);
        wr[i].w = adam_one(wr[i].w, gr[i].w, mr[i].w, vr[i].w, o, 1.f, -INFINITY);
        w4[c] = wr[i];
        m4[c] = mr[i];
        v4[c] = vr[i];
      }
    }
  }
  laq_row_cached<T>(wr, cols, blockIdx.x, bits, codes + base, rowsum, scale, what ? what + base : nullptr, sh);
}

// Block size of the two kernels above, or 0 when the row does not fit.
inline int laq_threads(int cols) {
  const int warps = (cols / 4 + 32 * LAQ_V - 1) / (32 * LAQ_V);
  return warps <= LAQ_MAX_WARPS ? 32 * warps : 0;
}

template <typename T, int RULE, int NT, int MAXV>
__device__ __forceinline__ void closed_form_row(const float4* wr, bool cached, const float* w_row, int cols,
                                                int row, int bits, int8_t* codes_row, int32_t* rowsum, float* scale,
                                                T* what_row, double* shd, int* shi, float* shf) {
  if (RULE == 3) laq_row<T, NT>(w_row, cols, row, bits, codes_row, rowsum, scale, what_row, shd, shi, shf);
  else ternary_row<T, NT, MAXV>(wr, cached, w_row, cols, row, codes_row, rowsum, scale, what_row, shd, shi);
}

template <typename T, int RULE, int NT, int MAXV>
__global__ void __launch_bounds__(NT, RULE == 2 ? 5 : 4) closed_form_quantize_kernel(const float* __restrict__ w, int cols,
                                                                      int bits,
                                                                      int8_t* __restrict__ codes,
                                                                      int32_t* __restrict__ rowsum,
                                                                      float* __restrict__ scale, T* __restrict__ what) {
  pdl_wait();
  pdl_trigger();
  __shared__ double shd[64];
  __shared__ int shi[32];
  __shared__ float shf[32];
  const int row = blockIdx.x;
  const long long base = (long long)row * cols;
  const int nvec = cols / 4;
  const bool cached = RULE == 2 && nvec <= MAXV * NT;
  float4 wr[MAXV];
  if (cached) {
#pragma unroll
    for (int i = 0; i < MAXV; ++i) {
      const int c = threadIdx.x + i * NT;
      if (c < nvec) wr[i] = reinterpret_cast<const float4*>(w + base)[c];
    }
  }
  closed_form_row<T, RULE, NT, MAXV>(wr, cached, w + base, cols, row, bits, codes + base, rowsum, scale,
                     what ? what + base : nullptr, shd, shi, shf);
}

// AdamW on the row (gradient of w_hat passed through unchanged), then the rule on the new weights.
template <typename T, int RULE, int NT, int MAXV>
__global__ void __launch_bounds__(NT, RULE == 2 ? 5 : 4) closed_form_update_kernel(float* __restrict__ w, const float* __restrict__ g,
                                                                    float* __restrict__ m, float* __restrict__ v,
                                                                    const OptimScalars* __restrict__ sc, int cols,
                                                                    int train_w, int bits,
                                                                    int8_t* __restrict__ codes,
                                                                    int32_t* __restrict__ rowsum,
                                                                    float* __restrict__ scale, T* __restrict__ what) {
  pdl_wait();
  pdl_trigger();
  __shared__ double shd[64];
  __shared__ int shi[32];
  __shared__ float shf[32];
  const int row = blockIdx.x;
  const OptimScalars o = *sc;
  const long long base = (long long)row * cols;
  const int nvec = cols / 4;
  const bool cached = RULE == 2 && nvec <= MAXV * NT;
  float4* w4 = reinterpret_cast<float4*>(w + base);
  const float4* g4 = reinterpret_cast<const float4*>(g + base);
  float4* m4 = reinterpret_cast<float4*>(m + base);
  float4* v4 = reinterpret_cast<float4*>(v + base);
  float4 wr[MAXV];
  auto upd = [&](int c) {
    float4 wv = w4[c];
    if (train_w) {
      const float4 d = g4[c];
      float4 mm = m4[c], vv = v4[c];
      wv.x = adam_one(wv.x, d.x, mm.x, vv.x, o, 1.f, -INFINITY);
      wv.y = adam_one(wv.y, d.y, mm.y, vv.y, o, 1.f, -INFINITY);
      wv.z = adam_one(wv.z, d.z, mm.z, vv.z, o, 1.f, -INFINITY);
      wv.w = adam_one(wv.w, d.w, mm.w, vv.w, o, 1.f, -INFINITY);
      w4[c] = wv;
      m4[c] = mm;
      v4[c] = vv;
    }
    return wv;
  };
  if (cached) {
#pragma unroll
    for (int i = 0; i < MAXV; ++i) {
      const int c = threadIdx.x + i * NT;
      if (c < nvec) wr[i] = upd(c);
    }
  } else {
    for (int c = threadIdx.x; c < nvec; c += NT) upd(c);
    __syncthreads();                     // the row is re-read below by other threads of the block
  }
  closed_form_row<T, RULE, NT, MAXV>(wr, cached, w + base, cols, row, bits, codes + base, rowsum, scale,
                     what ? what + base : nullptr, shd, shi, shf);
}

}  // namespace

void launch_closed_form_quantize(const float* w, int rows, int cols, int rule, int bits, int8_t* codes, int32_t* rowsum,
                                 float* scale, void* what, int dt, cudaStream_t st) {
  Scope sc("quantize_weight", (double)rows * cols * (5.0 + (what ? (dt == 1 ? 2.0 : 4.0) : 0.0)) + rows * 8.0, 0, st);
  auto go = [&](auto kernel, int nt, auto* out) { launch_k(kernel, rows, nt, 0, st, w, cols, bits, codes, rowsum, scale, out); };
  const int nt = rule == 3 ? laq_threads(cols) : 0;
  if (dt == 1) {
    if (nt > 128) go(laq_quantize_kernel<bf16, 512>, nt, (bf16*)what);
    else if (nt) go(laq_quantize_kernel<bf16, 128>, nt, (bf16*)what);
    else if (rule == 3) go(closed_form_quantize_kernel<bf16, 3, TW_THREADS, TW_MAXV>, TW_THREADS, (bf16*)what);
    else go(closed_form_quantize_kernel<bf16, 2, TW_THREADS, TW_MAXV>, TW_THREADS, (bf16*)what);
  } else {
    if (nt > 128) go(laq_quantize_kernel<float, 512>, nt, (float*)what);
    else if (nt) go(laq_quantize_kernel<float, 128>, nt, (float*)what);
    else if (rule == 3) go(closed_form_quantize_kernel<float, 3, TW_THREADS, TW_MAXV>, TW_THREADS, (float*)what);
    else go(closed_form_quantize_kernel<float, 2, TW_THREADS, TW_MAXV>, TW_THREADS, (float*)what);
  }
}

void launch_closed_form_update(float* w, const float* g, float* m, float* v, const OptimScalars* sc, int rows, int cols,
                               int train_w, int rule, int bits, int8_t* codes, int32_t* rowsum, float* scale, void* what,
                               int dt, cudaStream_t st) {
  Scope scope("fused_weight_update", (double)rows * cols * (29.0 + (what ? (dt == 1 ? 2.0 : 4.0) : 0.0)), 0, st);
  auto go = [&](auto kernel, int nt, auto* out) {
    launch_k(kernel, rows, nt, 0, st, w, g, m, v, sc, cols, train_w, bits, codes, rowsum, scale, out);
  };
  const int nt = rule == 3 ? laq_threads(cols) : 0;
  if (dt == 1) {
    if (nt > 128) go(laq_update_kernel<bf16, 512>, nt, (bf16*)what);
    else if (nt) go(laq_update_kernel<bf16, 128>, nt, (bf16*)what);
    else if (rule == 3) go(closed_form_update_kernel<bf16, 3, TW_THREADS, TW_MAXV>, TW_THREADS, (bf16*)what);
    else go(closed_form_update_kernel<bf16, 2, TW_THREADS, TW_MAXV>, TW_THREADS, (bf16*)what);
  } else {
    if (nt > 128) go(laq_update_kernel<float, 512>, nt, (float*)what);
    else if (nt) go(laq_update_kernel<float, 128>, nt, (float*)what);
    else if (rule == 3) go(closed_form_update_kernel<float, 3, TW_THREADS, TW_MAXV>, TW_THREADS, (float*)what);
    else go(closed_form_update_kernel<float, 2, TW_THREADS, TW_MAXV>, TW_THREADS, (float*)what);
  }
}

}  // namespace mrem
