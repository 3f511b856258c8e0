// Pieces of the per-row weight update (weight_update.cu has the whole of it) that other kernels share: AdamW on pairs of weights, and
// the update of the rows of a table that got no gradient.
#pragma once
#include "optim.cuh"

namespace mrem {

struct Adam2 { float2 b1, ob1, b2, ob2, rsq, eps, neg_lr, decay; };
__device__ __forceinline__ Adam2 make_adam2(const OptimScalars& o) {
  return Adam2{splat(o.beta1), splat(__fsub_rn(1.f, o.beta1)), splat(o.beta2), splat(__fsub_rn(1.f, o.beta2)),
               splat(o.rsqrt_bc2), splat(o.eps), splat(-o.lr_bc1), splat(__fsub_rn(1.f, __fmul_rn(o.lr, o.weight_decay)))};
}
__device__ __forceinline__ float2 adam2(float2 p, float2 g, float2& m, float2& v, const Adam2& a) {      // adam_one of both
  m = fma2(a.b1, m, mul2(a.ob1, g));
  v = fma2(a.b2, v, mul2(mul2(a.ob2, g), g));
  const float2 denom = fma2(make_float2(sqrt_approx(v.x), sqrt_approx(v.y)), a.rsq, a.eps), num = mul2(a.neg_lr, m);
  return add2(mul2(p, a.decay), make_float2(__fdividef(num.x, denom.x), __fdividef(num.y, denom.y)));
}

// A word that a launch before the one before wrote, read by a block that has not waited for the one before: the word is in memory, and the
// acquire keeps this thread's later loads (of the step's scalars) from what its SM's L1 held before.
__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// The rows in [first, end) of a table of which `used` says 0xffffffff: no token gathered them, so their gradient is zero (written
// as such), their step gradient too, and nothing but the optimizer's scalars is needed to update them.  A warp updates a row by
// itself, without a barrier and whatever its block does besides: blocks of these rows run beside those of launches that wait on
// latency, not on memory, and may do so before the launch before their own has ended.  The same arithmetic as the fused update's, integer grid.
struct IdleRows {
  RowUpdate m;
  const OptimScalars* sc;
  const unsigned* used;
  int bits, first, end;
};
// `warp` of `n_warps` takes every n_warps-th row; U vectors of w, m and v in flight per lane.
template <int U>
__device__ __forceinline__ void update_idle_rows(const IdleRows& r, int warp, int n_warps) {
  const int lane = threadIdx.x & 31, nvec = r.m.cols / 4;
  const float qmax = (float)((1 << (r.bits - 1)) - 1);
  if (r.first < r.end) load_acquire(r.used + r.first);
  const OptimScalars o = *r.sc;
  const Adam2 ad = make_adam2(o);
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int row = r.first + warp; row < r.end; row += n_warps) {
    if (__ldcg(r.used + row) != 0xffffffffu) continue;
    const long long base = (long long)row * r.m.cols;
    float4* w4 = reinterpret_cast<float4*>(r.m.w + base);
    float4* g4 = reinterpret_cast<float4*>(r.m.g + base);
    float4* m4 = reinterpret_cast<float4*>(r.m.m + base);
    float4* v4 = reinterpret_cast<float4*>(r.m.v + base);
    uint32_t* codes = reinterpret_cast<uint32_t*>(r.m.codes + base);
    float ms = r.m.m_s[row], vs = r.m.v_s[row];
    const float s = adam_one(r.m.steps[row], 0.f, ms, vs, o, 0.f, 1e-8f), r_s = __frcp_rn(s);
    float2 sum2 = splat(0.f);                                  // codes are whole numbers: exact in any order
#pragma unroll 1
    for (int c0 = lane; c0 < nvec; c0 += 32 * U) {
      float4 wv[U], mv[U], vv[U];
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const int c = c0 + 32 * i;
        if (c < nvec) { wv[i] = w4[c]; mv[i] = m4[c]; vv[i] = v4[c]; }
      }
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const int c = c0 + 32 * i;
        if (c >= nvec) continue;
        float2 ma = make_float2(mv[i].x, mv[i].y), mb = make_float2(mv[i].z, mv[i].w), va = make_float2(vv[i].x, vv[i].y),
               vb = make_float2(vv[i].z, vv[i].w);
        const float2 wa = adam2(make_float2(wv[i].x, wv[i].y), splat(0.f), ma, va, ad);
        const float2 wb = adam2(make_float2(wv[i].z, wv[i].w), splat(0.f), mb, vb, ad);
        w4[c] = make_float4(wa.x, wa.y, wb.x, wb.y);
        m4[c] = make_float4(ma.x, ma.y, mb.x, mb.y);
        v4[c] = make_float4(va.x, va.y, vb.x, vb.y);
        g4[c] = zero4;
        float q[4] = {wa.x, wa.y, wb.x, wb.y};
        uint32_t b[4];
        codes_f<false, 4>(q, s, r_s, -qmax, qmax, b);
        codes[c] = pack_low_bytes(b[0], b[1], b[2], b[3]);
        sum2 = add2(sum2, add2(make_float2(q[0], q[1]), make_float2(q[2], q[3])));
      }
    }
    const int sum = __reduce_add_sync(0xffffffffu, (int)sum2.x + (int)sum2.y);
    __syncwarp();                                              // every lane has read the row's step and moments
    if (lane == 0) {
      r.m.rowsum[row] = sum;
      r.m.scale[row] = s;
      r.m.m_s[row] = ms;
      r.m.v_s[row] = vs;
      r.m.steps[row] = s;
    }
  }
}

}  // namespace mrem
