// Pieces shared by the attention backward kernels: pairs of values, rows of swizzled operand tiles, the straight-through
// pass of a symmetric quantizer over 32 values of a row.
#pragma once
#include "gemm.h"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace mrem {
namespace att {

constexpr int HD = 64;                    // head size

__device__ __forceinline__ void ld16(const void* p, uint32_t* w) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  w[0] = u.x; w[1] = u.y; w[2] = u.z; w[3] = u.w;
}
__device__ __forceinline__ void st16(void* p, const uint32_t* w) {
  *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ float2 unpack2(uint32_t w) { return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ __forceinline__ uint32_t pack2(float2 v) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 acc2(const uint32_t* a, int j) { return make_float2(__uint_as_float(a[2 * j]), __uint_as_float(a[2 * j + 1])); }

// The largest non-negative bfloat16 value whose quotient by `step` is within the code range (quotient() is monotonic, and
// for bfloat16 values the IEEE division): |x| <= this is the straight-through mask.
__device__ __forceinline__ float range_limit(float step, float hi) {
  const float r = __frcp_rn(step);
  const uint32_t b = __float_as_uint(hi * step) >> 16;
  float lim = __uint_as_float((b - 1u) << 16);
  if (quotient(__uint_as_float(b << 16), step, r) <= hi) lim = __uint_as_float(b << 16);
  if (quotient(__uint_as_float((b + 1u) << 16), step, r) <= hi) lim = __uint_as_float((b + 1u) << 16);
  return lim;
}

// What the straight-through pass of a site needs besides its step.  The two take a dependent chain of some 200 clocks to form, so they are
// formed while the first tiles are on their way, and wait in shared memory (a copy per warp: no barrier).
struct SiteTerms { float lim, r; };
__device__ __forceinline__ SiteTerms site_terms(float step, float hi) { return SiteTerms{range_limit(step, hi), __frcp_rn(step)}; }

// No stored probability of a row is above this (m = RN(alpha log2(e) max), inv = 1 / sum, both as the forward pass left them).
// The largest one is not 2^0 inv: its exponent fma(max, alpha log2(e), -m) is the rounding error of m, up to 2^-24 |m|, and where
// that is positive the probability can be stored one bf16 spacing above the stored inv.  The last factor covers the two
// approximate exponentials and the roundings of the products.  Only whether a tile tests its elements one by one depends on this.
__device__ __forceinline__ float probability_bound(float m, float inv) {
  return __bfloat162float(__float2bfloat16_rn(inv * exp2_approx(fabsf(m) * 5.9604645e-8f) * (1.f + 9.5367432e-7f)));
}

// Straight-through pass of one symmetric quantizer over 2 NP values of a row: x (bf16 pairs before quantization, replaced by the
// masked gradient as bf16 pairs), g(j) = the incoming gradient of pair j.  Returns the sum of the step-size terms.  A NaN is
// outside every range (its code is the lowest): the test for clipped values keeps it (max.NaN).
template <int NP, class G>
__device__ __forceinline__ float ste_pairs(uint32_t* x, G&& g, float step, float hi, SiteTerms site) {
  const float lim = site.lim;
  const float2 r2 = both(site.r), ns2 = both(-step), magic2 = both(ROUND_MAGIC), nmagic2 = both(-ROUND_MAGIC), m1 = both(-1.f);
  __nv_bfloat162 mx = __habs2(*reinterpret_cast<const __nv_bfloat162*>(&x[0]));
#pragma unroll
  for (int j = 1; j < NP; ++j) mx = __hmax2_nan(mx, __habs2(*reinterpret_cast<const __nv_bfloat162*>(&x[j])));
  const float2 m = __bfloat1622float2(mx);
  float2 ds = both(0.f);
  if (__all_sync(0xffffffffu, m.x <= lim && m.y <= lim)) {       // nothing clipped in the whole warp
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const float2 xv = unpack2(x[j]), gv = g(j);
      const float2 z0 = mul2(xv, r2), z = fma2(fma2(z0, ns2, xv), r2, z0);
      const float2 q = add2(add2(z, magic2), nmagic2);
      ds = fma2(gv, fma2(z, m1, q), ds);
      x[j] = pack2(gv);
    }
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const float2 xv = unpack2(x[j]);
      float2 gv = g(j);
      const float2 z0 = mul2(xv, r2), z = fma2(fma2(z0, ns2, xv), r2, z0);
      const bool in0 = fabsf(xv.x) <= lim, in1 = fabsf(xv.y) <= lim;
      const float2 c = make_float2(fminf(fmaxf(z.x, -hi), hi), fminf(fmaxf(z.y, -hi), hi));
      const float2 q = add2(add2(c, magic2), nmagic2);
      ds = fma2(gv, make_float2(in0 ? q.x - z.x : q.x, in1 ? q.y - z.y : q.y), ds);
      x[j] = pack2(make_float2(in0 ? gv.x : 0.f, in1 ? gv.y : 0.f));
    }
  }
  return ds.x + ds.y;
}

template <class G>
__device__ __forceinline__ float ste32(uint32_t* x, G&& g, float step, float hi, SiteTerms site) { return ste_pairs<16>(x, g, step, hi, site); }

// Piece `part` of a row of a 128-byte-swizzled tile of 128 rows x 128 bytes: 8 NW columns (16 NW bytes)
template <int NW>
__device__ __forceinline__ void piece_load(const uint8_t* tile, int r, int part, uint32_t* w) {
#pragma unroll
  for (int t = 0; t < NW; ++t) ld16(tile + r * 128 + (((part * NW + t) ^ (r & 7)) * 16), w + 4 * t);
}
template <int NW>
__device__ __forceinline__ void piece_store(uint8_t* tile, int r, int part, const uint32_t* w) {
#pragma unroll
  for (int t = 0; t < NW; ++t) st16(tile + r * 128 + (((part * NW + t) ^ (r & 7)) * 16), w + 4 * t);
}
__device__ __forceinline__ void tile_load(const uint8_t* tile, int r, int half, uint32_t* w) { piece_load<4>(tile, r, half, w); }
__device__ __forceinline__ void tile_store(uint8_t* tile, int r, int half, const uint32_t* w) { piece_store<4>(tile, r, half, w); }

// Sums over the first `rows` rows of such a tile of bf16 values, for the bias gradient of the product that made Q, K and V: a warp
// of NW takes 128 / NW rows and a lane two columns (a row per load, all banks), its sums go to red[warp][64].  The tile is read as
// stored, so the sums are those of the stored gradients.  Instead of a launch that read them again from memory: step of 3 x 72
// tokens, hidden 768, 455 -> 442 us, of 32 x 128 tokens, hidden 1024, 3464 -> 3453.  The kernels for longer sequences leave theirs
// to that launch: with the sums inside 11 x 200 and 16 x 384 tokens gained nothing and 8 x 256 took 993 us instead of 982.
template <int NW>
__device__ __forceinline__ void tile_col_sums(const uint8_t* tile, int rows, int warp, int lane, float* red) {
  float2 t[4] = {both(0.f), both(0.f), both(0.f), both(0.f)};      // (four short chains: a quarter of one long one's rounding)
#pragma unroll 8
  for (int i = 0; i < 128 / NW; ++i) {
    const int r = warp * (128 / NW) + i;
    const uint32_t w = *reinterpret_cast<const uint32_t*>(tile + r * 128 + (((lane >> 2) ^ (r & 7)) * 16) + (lane & 3) * 4);
    const float2 v = unpack2(w);
    if (r < rows) t[i & 3] = add2(t[i & 3], v);
  }
  *reinterpret_cast<float2*>(red + warp * 64 + 2 * lane) = add2(add2(t[0], t[1]), add2(t[2], t[3]));
}
// the warps' sums of one column, neighbours first
template <int NW>
__device__ __forceinline__ float add_col_sums(const float* red, int col) {
  float t[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) t[w] = red[w * 64 + col];
#pragma unroll
  for (int d = 1; d < NW; d *= 2)
#pragma unroll
    for (int w = 0; w < NW; w += 2 * d) t[w] += t[w + d];
  return t[0];
}

}  // namespace att
}  // namespace mrem
