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
#include "row_update.cuh"

namespace mrem {

namespace {

// Ternary rule: 256 threads per row, up to 4 float4 vectors per thread in registers (rows up to 4096 wide).  Refitted
// scale: two to eight vectors per thread and as many warps as that takes (rows up to 4096 wide).  Wider rows are re-read by
// 256 threads.
constexpr int TW_THREADS = 256;
constexpr int TW_MAXV = 4;
constexpr int LAQ_MAX_WARPS = 4;

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

// The rule on a row held in registers, V vectors of four per thread (missing ones are zeros: their code is 0 and they add
// nothing), up to LAQ_MAX_WARPS warps a row.  Everything but the codes that go out is the same for w and |w|: <q, w> =
// <|q|, |w|>, so the rounds work on |w| and need one bound.  The two sums of a round get neither float64 arithmetic nor
// conversions per weight: with e = the exponent of max|w|, |w| in units of 2^(e - 31) is a whole number of 32 bits for every
// weight of at least 2^(e - 8), and the others have code 0 while alpha >= 2^(e - 6); its four bytes, each kept beside those of the
// three neighbouring weights, meet the four codes in byte dot products, and the sums are exact (a byte sum of a block is below
// 2^23, two of them 8 bits apart below 2^31: codes of up to 4 bits).  Other rows, and more bits, take float64 sums.
// Bound by instruction issue and latency: 5 instructions per weight and round and about 70 per warp for the sums, so a warp takes a
// row of up to 1024 alone (no barrier) and three or four take wider ones.  A layer's four matrices, hidden 768, with the update: 145 us
// with 8 weights a thread (3 warps for 768, 12 for 3072) and float32 sums of two 12-bit parts and a rest, now 107 (75 in shared launches, below); the step of three
// layers, 32 x 128 tokens, 1347 -> 1263 us (rows of 768 on three, two, one warp 1324, 1285, 1263).
template <int V> struct LaqRow { float2 a[2 * V]; uint32_t limb[V][4], neg[V]; };   // |w|; bytes of four; ff where negative
struct LaqShared { uint4 sums[2][LAQ_MAX_WARPS]; double d[32]; int i[64]; float f[32]; };

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {     // (0x8 in a nibble: the byte's sign, eight times)
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
__device__ __forceinline__ double uint_as_double(uint32_t x) { return __hiloint2double(0x43300000, (int)x) - 4503599627370496.0; }

template <int V>
__device__ __forceinline__ void laq_take(LaqRow<V>& rw, int i, float4 w) {
  rw.a[2 * i] = make_float2(fabsf(w.x), fabsf(w.y));
  rw.a[2 * i + 1] = make_float2(fabsf(w.z), fabsf(w.w));
  rw.neg[i] = prmt(prmt(__float_as_uint(w.x), __float_as_uint(w.y), 0x00fb), prmt(__float_as_uint(w.z), __float_as_uint(w.w), 0x00fb), 0x5410);
}

// The codes of four |w| by the division of Eq. 1, one per byte.  (A call: the few weights next to a rounding boundary, and rows
// without byte sums; inlined at every vector it filled the instruction cache.)
__device__ __noinline__ uint32_t laq_codes_exact(float4 a, float alpha, float qmax) {
  return (uint32_t)laq_code(a.x, alpha, qmax) | ((uint32_t)laq_code(a.y, alpha, qmax) << 8) | ((uint32_t)laq_code(a.z, alpha, qmax) << 16) |
         ((uint32_t)laq_code(a.w, alpha, qmax) << 24);
}
// The same without the division but where it decides (code_f); alpha in (1e-30, 1e30).
__device__ __forceinline__ uint32_t laq_codes(float4 a, float alpha, float r_alpha, float qmax) {
  const float2 z = quotient2(make_float2(a.x, a.y), splat(-alpha), splat(r_alpha)), y = quotient2(make_float2(a.z, a.w), splat(-alpha), splat(r_alpha));
  const float2 zc = make_float2(fminf(z.x, qmax), fminf(z.y, qmax)), yc = make_float2(fminf(y.x, qmax), fminf(y.y, qmax));
  uint32_t k[4];
  const float2 t = rne_magic2(zc, k[0], k[1]), u = rne_magic2(yc, k[2], k[3]);
  if (fmaxf(fmaxf(fabsf(zc.x - t.x), fabsf(zc.y - t.y)), fmaxf(fabsf(yc.x - u.x), fabsf(yc.y - u.y))) > 0.5f - HALF_WINDOW)
    return laq_codes_exact(a, alpha, qmax);
  return pack_low_bytes(k[0], k[1], k[2], k[3]);
}
__device__ __forceinline__ double laq_dot(uint32_t q, float4 a) {
  return (uint_as_double(q & 0xffu) * (double)a.x + uint_as_double((q >> 8) & 0xffu) * (double)a.y) +
         (uint_as_double((q >> 16) & 0xffu) * (double)a.z + uint_as_double(q >> 24) * (double)a.w);
}

// Sums over the block of v.x, v.y, v.z (and v.w): every thread gets them.  `slot` alternates from call to call.
template <bool W>
__device__ __forceinline__ uint4 block_sum_u4(uint4 v, uint4* slot, int wid, int nw) {
  v.x = __reduce_add_sync(0xffffffffu, v.x);
  v.y = __reduce_add_sync(0xffffffffu, v.y);
  v.z = __reduce_add_sync(0xffffffffu, v.z);
  if (W) v.w = __reduce_add_sync(0xffffffffu, v.w);
  if (nw == 1) return v;
  if ((threadIdx.x & 31) == 0) slot[wid] = v;
  __syncthreads();
  v = slot[0];
  for (int k = 1; k < nw; ++k) {
    const uint4 e = slot[k];
    v.x += e.x; v.y += e.y; v.z += e.z; v.w += e.w;
  }
  return v;
}

template <typename T, int V>
__device__ __forceinline__ void laq_row_cached(LaqRow<V>& rw, int cols, int row, int bits, int8_t* codes_row, int32_t* rowsum,
                                               float* scale, T* what_row, LaqShared& sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, nvec = cols / 4;
  const float qmax = (float)((1 << (bits - 1)) - 1);
  double s = 0.0;
  float mx = 0.f;
#pragma unroll
  for (int e = 0; e < 2 * V; ++e) {
    s += (double)rw.a[e].x + (double)rw.a[e].y;
    mx = fmaxf(mx, fmaxf(rw.a[e].x, rw.a[e].y));
  }
  s = warp_sum_d(s);
  mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
  if (nw > 1) {
    if (lane == 0) { sh.d[wid] = s; sh.f[wid] = mx; }
    __syncthreads();
    s = sh.d[0];
    mx = sh.f[0];
    for (int k = 1; k < nw; ++k) { s += sh.d[k]; mx = fmaxf(mx, sh.f[k]); }
    __syncthreads();
  }
  float alpha = (float)(fmin(3.0 * (s / (double)cols), (double)mx) / (double)qmax);
  const bool split = bits <= 4 && mx > 1e-30f && mx < 1e30f;
  const int eb = (int)(__float_as_uint(mx) >> 23);         // e + 127
  const float lowest = split ? fmaxf(1e-30f, __uint_as_float((uint32_t)(eb - 6) << 23)) : INFINITY;
  const double unit = __hiloint2double((eb - 127 - 31 + 1023) << 20, 0);
#pragma unroll
  for (int i = 0; i < V; ++i) {
    uint32_t x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t u = __float_as_uint((j & 1) ? rw.a[2 * i + (j >> 1)].y : rw.a[2 * i + (j >> 1)].x);
      x[j] = __funnelshift_rc((u << 8) | 0x80000000u, 0u, (uint32_t)eb - (u >> 23));   // (32 places or more: 0)
    }
    const uint32_t l0 = prmt(x[0], x[1], 0x5140), l1 = prmt(x[2], x[3], 0x5140), h0 = prmt(x[0], x[1], 0x7362), h1 = prmt(x[2], x[3], 0x7362);
    rw.limb[i][0] = prmt(l0, l1, 0x5410);
    rw.limb[i][1] = prmt(l0, l1, 0x7632);
    rw.limb[i][2] = prmt(h0, h1, 0x5410);
    rw.limb[i][3] = prmt(h0, h1, 0x7632);
  }
  int it = 0;
  for (int r = 0; r + 1 < LAQ_ROUNDS; ++r) {
    float next = 0.f;
    if (alpha >= lowest) {
      const float r_alpha = __frcp_rn(alpha);
      uint32_t b0 = 0u, b1 = 0u, b2 = 0u, b3 = 0u, qq = 0u;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const float2 z = quotient2(rw.a[2 * i], splat(-alpha), splat(r_alpha)), y = quotient2(rw.a[2 * i + 1], splat(-alpha), splat(r_alpha));
        const float2 t = add2(make_float2(fminf(z.x, qmax), fminf(z.y, qmax)), splat(ROUND_MAGIC));
        const float2 u = add2(make_float2(fminf(y.x, qmax), fminf(y.y, qmax)), splat(ROUND_MAGIC));
        const uint32_t q = pack_low_bytes(__float_as_uint(t.x), __float_as_uint(t.y), __float_as_uint(u.x), __float_as_uint(u.y));
        b0 = __dp4a(rw.limb[i][0], q, b0);
        b1 = __dp4a(rw.limb[i][1], q, b1);
        b2 = __dp4a(rw.limb[i][2], q, b2);
        b3 = __dp4a(rw.limb[i][3], q, b3);
        qq = __dp4a(q, q, qq);
      }
      const uint4 t = block_sum_u4<false>(make_uint4(b0 + (b1 << 8), b2 + (b3 << 8), qq, 0u), sh.sums[it++ & 1], wid, nw);
      // <q, w> / <q, q>: float32 quotient and one correction from the float64 residual (2^-46 before the rounding to float32)
      const double qw = fma(uint_as_double(t.y), 65536.0, uint_as_double(t.x)) * unit, n = uint_as_double(t.z);
      const float rq = __frcp_rn((float)t.z), a0 = (float)qw * rq;
      if (t.z) next = (float)fma(fma(-(double)a0, n, qw), (double)rq, (double)a0);
    } else {
      double qw = 0.0;
      int qq = 0;
      if (alpha > 0.f) {
        const bool normal = alpha > 1e-30f && alpha < 1e30f;
        const float r_alpha = __frcp_rn(alpha);
#pragma unroll
        for (int i = 0; i < V; ++i) {
          const float4 a4 = make_float4(rw.a[2 * i].x, rw.a[2 * i].y, rw.a[2 * i + 1].x, rw.a[2 * i + 1].y);
          const uint32_t q = normal ? laq_codes(a4, alpha, r_alpha, qmax) : laq_codes_exact(a4, alpha, qmax);
          qw += laq_dot(q, a4);
          qq += (int)__dp4a(q, q, 0u);
        }
      }
      block_sum_di(qw, qq, sh.d, sh.i);
      next = qq > 0 ? (float)(qw / (double)qq) : 0.f;
    }
    if (next == alpha) break;
    alpha = next;
  }
  // last round: the codes of this alpha (by the division of Eq. 1) go out with the scale refitted to them
  const bool whole = alpha >= lowest, normal = alpha > 1e-30f && alpha < 1e30f;
  const float r_alpha = __frcp_rn(alpha);
  double qw = 0.0;
  uint32_t b0 = 0u, b1 = 0u, b2 = 0u, b3 = 0u, qq = 0u, code[V];
  int sum = 0;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int c = threadIdx.x + i * blockDim.x;
    const float4 a4 = make_float4(rw.a[2 * i].x, rw.a[2 * i].y, rw.a[2 * i + 1].x, rw.a[2 * i + 1].y);
    const uint32_t q = normal ? laq_codes(a4, alpha, r_alpha, qmax) : (alpha > 0.f ? laq_codes_exact(a4, alpha, qmax) : 0u);
    if (!whole) qw += laq_dot(q, a4);
    b0 = __dp4a(rw.limb[i][0], q, b0);
    b1 = __dp4a(rw.limb[i][1], q, b1);
    b2 = __dp4a(rw.limb[i][2], q, b2);
    b3 = __dp4a(rw.limb[i][3], q, b3);
    qq = __dp4a(q, q, qq);
    code[i] = (q & ~rw.neg[i]) | (((0x80808080u - q) ^ 0x80808080u) & rw.neg[i]);    // (no borrow: codes are at most 127)
    sum = __dp4a((int)code[i], 0x01010101, sum);
    if (c < nvec) *reinterpret_cast<uint32_t*>(codes_row + 4 * c) = code[i];
  }
  const uint4 t = block_sum_u4<true>(make_uint4(b0 + (b1 << 8), b2 + (b3 << 8), qq, (uint32_t)sum), sh.sums[it & 1], wid, nw);
  if (whole) {
    qw = fma(uint_as_double(t.y), 65536.0, uint_as_double(t.x)) * unit;
  } else {
    int none = 0;
    block_sum_di(qw, none, sh.d, sh.i);
  }
  float next = t.z ? (float)(qw / uint_as_double(t.z)) : 0.f;
  if (!(s == s)) next = (float)s;                          // a weight that is not a number has no byte sums, and no scale either
  if (what_row) {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int c = threadIdx.x + i * blockDim.x;
      const uint32_t u = code[i] ^ 0x80808080u;            // code + 128, then 2^23 + code + 128 as a float
      auto value = [&](uint32_t sel) { return next * (__uint_as_float(prmt(u, 0x4b000000u, sel)) - 8388736.f); };
      if (c < nvec) store4<T>(what_row + 4 * c, value(0x7650), value(0x7651), value(0x7652), value(0x7653));
    }
  }
  if (threadIdx.x == 0) {
    rowsum[row] = (int)t.w;
    scale[row] = next;
  }
}

// Blocks of the two kernels below that an SM is to hold (registers: about 9 V and 35)
constexpr int laq_blocks(int V) { return V == 8 ? 4 : (V == 6 ? 5 : (V == 4 ? 6 : 8)); }

// The matrices of a layer whose rows take the same kernel are updated by one launch: a launch each left the chip half idle at every
// matrix' last rows and first loads (three layers of hidden 768 with refitted scales, 32 x 128 tokens: 1263 -> 1235 us).
struct ClosedUpdate {
  RowUpdate mat[MAX_ROW_UPDATES];
  int row_end[MAX_ROW_UPDATES];        // running row count: matrix i owns the blocks [row_end[i - 1], row_end[i])
  int n, bits, train_w;
  int wait_last;                       // the launch before is this one's twin of another width: wait for it at the end only
  const OptimScalars* sc;
};
// What the matrices need is complete when the blocks of the first of two launches have passed their wait, which is when the second's may start.
__device__ __forceinline__ void closed_wait(const ClosedUpdate& P) {
  if (P.wait_last) load_acquire(reinterpret_cast<const unsigned*>(P.sc)); else pdl_wait();
  pdl_trigger();
}
__device__ __forceinline__ const RowUpdate& matrix_of_block(const ClosedUpdate& P, int& row) {
  int i = 0;
  while (i + 1 < P.n && (int)blockIdx.x >= P.row_end[i]) ++i;
  row = (int)blockIdx.x - (i ? P.row_end[i - 1] : 0);
  return P.mat[i];
}

// The two kernels of the refitted scale on rows held in registers.
template <typename T, int V>
__global__ void __launch_bounds__(32 * LAQ_MAX_WARPS, laq_blocks(V)) laq_quantize_kernel(const float* __restrict__ w, int cols, int bits,
                                                                                       int8_t* __restrict__ codes, int32_t* __restrict__ rowsum,
                                                                                       float* __restrict__ scale, T* __restrict__ what) {
  pdl_wait();
  pdl_trigger();
  __shared__ LaqShared sh;
  const long long base = (long long)blockIdx.x * cols;
  const float4* w4 = reinterpret_cast<const float4*>(w + base);
  LaqRow<V> rw;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int c = threadIdx.x + i * blockDim.x;
    laq_take(rw, i, c < cols / 4 ? w4[c] : make_float4(0.f, 0.f, 0.f, 0.f));
  }
  laq_row_cached<T, V>(rw, cols, blockIdx.x, bits, codes + base, rowsum, scale, what ? what + base : nullptr, sh);
}

template <typename T, int V>
__global__ void __launch_bounds__(32 * LAQ_MAX_WARPS, laq_blocks(V)) laq_update_kernel(const __grid_constant__ ClosedUpdate P) {
  closed_wait(P);
  __shared__ LaqShared sh;
  const OptimScalars o = *P.sc;
  int row;
  const RowUpdate& M = matrix_of_block(P, row);
  const int cols = M.cols, nvec = cols / 4, train_w = P.train_w;
  const long long base = (long long)row * cols;
  float4* w4 = reinterpret_cast<float4*>(M.w + base);
  const float4* g4 = reinterpret_cast<const float4*>(M.g + base);    // (not __restrict__: the non-coherent path knows no acquire)
  float4* m4 = reinterpret_cast<float4*>(M.m + base);
  float4* v4 = reinterpret_cast<float4*>(M.v + base);
  constexpr int N = V <= 4 ? 2 : V / 2;                    // vectors whose loads are in flight together
  LaqRow<V> rw;
#pragma unroll
  for (int i0 = 0; i0 < V; i0 += N) {
    float4 wr[N], gr[N], mr[N], vr[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int c = threadIdx.x + (i0 + i) * blockDim.x;
      wr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c < nvec) {
        wr[i] = w4[c];
        if (train_w) { gr[i] = g4[c]; mr[i] = m4[c]; vr[i] = v4[c]; }
      }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int c = threadIdx.x + (i0 + i) * blockDim.x;
      if (train_w && c < nvec) {
        wr[i].x = adam_one(wr[i].x, gr[i].x, mr[i].x, vr[i].x, o, 1.f, -INFINITY);
        wr[i].y = adam_one(wr[i].y, gr[i].y, mr[i].y, vr[i].y, o, 1.f, -INFINITY);
        wr[i].z = adam_one(wr[i].z, gr[i].z, mr[i].z, vr[i].z, o, 1.f, -INFINITY);
        wr[i].w = adam_one(wr[i].w, gr[i].w, mr[i].w, vr[i].w, o, 1.f, -INFINITY);
        w4[c] = wr[i];
        m4[c] = mr[i];
        v4[c] = vr[i];
      }
      laq_take(rw, i0 + i, wr[i]);
    }
  }
  laq_row_cached<T, V>(rw, cols, row, P.bits, M.codes + base, M.rowsum, M.scale, M.what ? reinterpret_cast<T*>(M.what) + base : nullptr, sh);
  if (P.wait_last) pdl_wait();
}

// Vectors per thread (2, 4, 6 or 8) and warps of the two kernels above: the fewest instructions a round, the sums of a warp
// counted as those of three vectors; 0 warps when the row does not fit.
inline int laq_warps(int cols, int& V) {
  const int n = (cols / 4 + 31) / 32;
  int warps = 0;
  for (int t = 2; t <= 8; t += 2) {
    const int k = (n + t - 1) / t;
    if (k <= LAQ_MAX_WARPS && (!warps || k * (t + 3) < warps * (V + 3))) { warps = k; V = t; }
  }
  return warps;
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
__global__ void __launch_bounds__(NT, RULE == 2 ? 5 : 4) closed_form_update_kernel(const __grid_constant__ ClosedUpdate P) {
  closed_wait(P);
  __shared__ double shd[64];
  __shared__ int shi[32];
  __shared__ float shf[32];
  const OptimScalars o = *P.sc;
  int row;
  const RowUpdate& M = matrix_of_block(P, row);
  const int cols = M.cols, nvec = cols / 4, train_w = P.train_w;
  const long long base = (long long)row * cols;
  const bool cached = RULE == 2 && nvec <= MAXV * NT;
  float4* w4 = reinterpret_cast<float4*>(M.w + base);
  const float4* g4 = reinterpret_cast<const float4*>(M.g + base);
  float4* m4 = reinterpret_cast<float4*>(M.m + base);
  float4* v4 = reinterpret_cast<float4*>(M.v + base);
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
  closed_form_row<T, RULE, NT, MAXV>(wr, cached, M.w + base, cols, row, P.bits, M.codes + base, M.rowsum, M.scale,
                     M.what ? reinterpret_cast<T*>(M.what) + base : nullptr, shd, shi, shf);
  if (P.wait_last) pdl_wait();
}

}  // namespace

void launch_closed_form_quantize(const float* w, int rows, int cols, int rule, int bits, int8_t* codes, int32_t* rowsum,
                                 float* scale, void* what, int dt, cudaStream_t st) {
  Scope sc("quantize_weight", (double)rows * cols * (5.0 + (what ? (dt == 1 ? 2.0 : 4.0) : 0.0)) + rows * 8.0, 0, st);
  auto go = [&](auto kernel, int nt, auto* out) { launch_k(kernel, rows, nt, 0, st, w, cols, bits, codes, rowsum, scale, out); };
  int V = 0;
  const int warps = rule == 3 ? laq_warps(cols, V) : 0;
  if (dt == 1) {
    if (warps && V == 2) go(laq_quantize_kernel<bf16, 2>, 32 * warps, (bf16*)what);
    else if (warps && V == 4) go(laq_quantize_kernel<bf16, 4>, 32 * warps, (bf16*)what);
    else if (warps && V == 6) go(laq_quantize_kernel<bf16, 6>, 32 * warps, (bf16*)what);
    else if (warps) go(laq_quantize_kernel<bf16, 8>, 32 * warps, (bf16*)what);
    else if (rule == 3) go(closed_form_quantize_kernel<bf16, 3, TW_THREADS, TW_MAXV>, TW_THREADS, (bf16*)what);
    else go(closed_form_quantize_kernel<bf16, 2, TW_THREADS, TW_MAXV>, TW_THREADS, (bf16*)what);
  } else {
    if (warps && V == 2) go(laq_quantize_kernel<float, 2>, 32 * warps, (float*)what);
    else if (warps && V == 4) go(laq_quantize_kernel<float, 4>, 32 * warps, (float*)what);
    else if (warps && V == 6) go(laq_quantize_kernel<float, 6>, 32 * warps, (float*)what);
    else if (warps) go(laq_quantize_kernel<float, 8>, 32 * warps, (float*)what);
    else if (rule == 3) go(closed_form_quantize_kernel<float, 3, TW_THREADS, TW_MAXV>, TW_THREADS, (float*)what);
    else go(closed_form_quantize_kernel<float, 2, TW_THREADS, TW_MAXV>, TW_THREADS, (float*)what);
  }
}

namespace {
// The kernel that takes the rows of a matrix: warps * 16 + vectors per thread of the refitted scale, 0 the general one.
inline int closed_variant(int cols, int rule) {
  int V = 0;
  const int warps = rule == 3 ? laq_warps(cols, V) : 0;
  return warps ? warps * 16 + V : 0;
}
template <typename T>
void launch_closed_variant(int variant, int rule, int rows, const ClosedUpdate& p, cudaStream_t st) {
  auto go = [&](auto kernel, int nt) { launch_k(kernel, rows, nt, 0, st, p); };
  const int nt = 32 * (variant >> 4);
  switch (variant & 15) {
    case 2: return go(laq_update_kernel<T, 2>, nt);
    case 4: return go(laq_update_kernel<T, 4>, nt);
    case 6: return go(laq_update_kernel<T, 6>, nt);
    case 8: return go(laq_update_kernel<T, 8>, nt);
  }
  if (rule == 3) go(closed_form_update_kernel<T, 3, TW_THREADS, TW_MAXV>, TW_THREADS);
  else go(closed_form_update_kernel<T, 2, TW_THREADS, TW_MAXV>, TW_THREADS);
}
}  // namespace

void launch_closed_form_update(const RowUpdate* mats, int n, const OptimScalars* sc, int train_w, int rule, int bits, int dt, cudaStream_t st) {
  // The widest rows first: theirs are the longest chains, and the next launch's blocks fill the SMs as they leave.
  unsigned done = 0;
  bool first = true;
  while (done != (1u << n) - 1u) {
    int lead = -1;
    for (int j = 0; j < n; ++j)
      if (!(done >> j & 1u) && (lead < 0 || mats[j].cols > mats[lead].cols)) lead = j;
    const int variant = closed_variant(mats[lead].cols, rule);
    ClosedUpdate p = {};
    p.bits = bits; p.train_w = train_w; p.sc = sc; p.wait_last = !first;
    double bytes = 0;
    int rows = 0;
    for (int j = 0; j < n; ++j) {
      if ((done >> j & 1u) || closed_variant(mats[j].cols, rule) != variant) continue;
      done |= 1u << j;
      p.mat[p.n] = mats[j];
      p.row_end[p.n++] = rows += mats[j].rows;
      bytes += (double)mats[j].rows * mats[j].cols * (29.0 + (mats[j].what ? (dt == 1 ? 2.0 : 4.0) : 0.0));
    }
    Scope scope("fused_weight_update", bytes, 0, st);
    if (dt == 1) launch_closed_variant<bf16>(variant, rule, rows, p, st); else launch_closed_variant<float>(variant, rule, rows, p, st);
    first = false;
  }
}

}  // namespace mrem
