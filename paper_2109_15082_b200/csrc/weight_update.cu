// Fused update of weight matrices and their per-row quantization steps (Algorithm 2:
// Update(w), Update(s)), one block per output row and ONE pass over the row's state:
//   1. straight-through factors of the weight quantizer at the old (w, s): the step
//      gradient ds = sum_k dW_hat * d w_hat / d s (fixed-order block sum),
//   2. AdamW on the row's step (clamped to stay positive),
//   3. AdamW on the latent weights with the masked gradient dW = dW_hat * 1[inside],
//   4. Eq. 1 on the new weights with the new step: int8 codes, row sum, dequantization
//      scale and the dequantized row for the next step's products.
// The row's weights and gradients are read once with 16-byte loads and held in registers
// (rows up to 4096 wide; longer rows are re-read).  Traffic per weight: read w, g, m, v
// (16 B), write w, m, v (12 B), codes (1 B) and the dequantized value (2 or 4 B); the separate
// passes it replaces move about twice that.
#include "row_update.cuh"

namespace mrem {

namespace {

template <typename T>
__device__ __forceinline__ void store_what4(T* p, float a, float b, float c, float d);
template <>
__device__ __forceinline__ void store_what4<float>(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
template <>
__device__ __forceinline__ void store_what4<bf16>(bf16* p, float a, float b, float c, float d) {
  uint2 t;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&t);
  h[0] = __floats2bfloat162_rn(a, b);
  h[1] = __floats2bfloat162_rn(c, d);
  *reinterpret_cast<uint2*>(p) = t;
}

// Pairs of weights: the arithmetic below is the scalar one of optim.cuh and code_f, two elements per instruction where the
// hardware has the form.
// The step gradient's terms of two elements (step_grad_acc), and which gradients pass.
template <int GRID>
__device__ __forceinline__ float2 step_grad2(float2 acc, float2 w, float2 d, float2 neg_s, float2 r_s, float qmax, bool& in0, bool& in1) {
  const float2 z = quotient2(w, neg_s, r_s);
  float2 level;
  if (GRID == 0) {
    const float2 zc = clamp2(z, -qmax, qmax);
    in0 = zc.x == z.x; in1 = zc.y == z.y;
    level = add2(add2(zc, splat(RINT_MAGIC)), splat(-RINT_MAGIC));
  } else {                                                     // clamp(floor(z), -2, 1) + 0.5 without the conversion unit
    in0 = z.x >= -2.f && z.x < 2.f; in1 = z.y >= -2.f && z.y < 2.f;
    level.x = z.x < 0.f ? (z.x < -1.f ? -1.5f : -0.5f) : (z.x >= 1.f ? 1.5f : 0.5f);
    level.y = z.y < 0.f ? (z.y < -1.f ? -1.5f : -0.5f) : (z.y >= 1.f ? 1.5f : 0.5f);
  }
  const float2 inside = make_float2(in0 ? -z.x : 0.f, in1 ? -z.y : 0.f);
  return fma2(d, add2(level, inside), acc);
}
struct UpdateParams {
  RowUpdate mat[MAX_ROW_UPDATES];
  int row_end[MAX_ROW_UPDATES];        // running row count: matrix i owns the blocks [row_end[i - 1], row_end[i])
  int n, bits, train_w, train_s;
  int wait_last;                       // the launch before is this one's twin of another width: wait for it at the end only
  const OptimScalars* sc;
  TokenRows tokens;
  IdleRows idle;
};

// One block of NT threads per row, NV float4 vectors of w, g, m and v per thread in registers; rows wider than the widest
// variant holds are re-read by it.  The matrices of a layer whose rows take the same variant go in one launch.
// The kernel moves 31 bytes a weight and should be bound by that, but was bound by the issue slots (71 % busy, DRAM at 39 %):
// with one float4 per thread, the two block sums, the step's own update behind a barrier and the scalars cost each thread as
// much as its four weights.  So: few threads per row, every thread forms the row's new step itself, and the arithmetic runs
// on pairs.  Measured: a layer of 1024 x 4096 shapes 87 -> 74 us (floor 59), its three 1024-wide matrices 56 -> 47 us in one
// launch; a whole table in one launch, 30522 x 1024 165 -> 136 us (7.1 TB/s), 30522 x 768 128 -> 116 us (today the launches before take
// part of its rows: embed_step.cu).
// Variants (X(index, NT, NV, blocks per SM)), by the widest row they hold: 16 weights a thread keep the most bytes in flight
// (1024 wide: 64 x 4 vectors 136 us, 128 x 2 144 us, 256 x 1 152 us for that table), but 64 x 3 for 768 wide rows, with
// the same ten blocks on an SM, does not (128 us; 96 x 2 at 62 registers 116 us).
#define UPD_VARIANTS(X) X(0, 96, 2, 10) X(1, 64, 4, 10) X(2, 128, 4, 5) X(3, 192, 4, 3) X(4, 256, 4, 2)
constexpr int UPD_WIDEST = 4;
// GRID (the weight grid, 0: Eq. 1's integers, 1: half-integer 2-bit levels) is a template parameter: the per-weight code
// then holds one of the two rules, not both under predicates.  SPARSE: an embedding table, one matrix per launch (its pointers
// stay at fixed places of the parameters, 235 -> 204 us for the step).  The first blocks have an idle row each: g is not read, and is cleared
// here instead of by a pass before.  They need the marks and the optimizer's scalars, which are complete before the launch before this one
// lets it start, and do not wait for its sums (embedding step of 30522 x 1024, 32 x 128 tokens 195 -> 190 us, 30522 x 768, 5 x 56 125.7 -> 121.7).
// The last blocks have a token each and update the row it gathered, if it is the first to gather it; they wait for the sums.
template <typename T, int NV, int NT, int BLOCKS, int GRID, bool SPARSE>
__global__ void __launch_bounds__(NT, BLOCKS) fused_weight_update_kernel(const __grid_constant__ UpdateParams P) {
  if (!SPARSE) {
    if (P.wait_last) load_acquire(reinterpret_cast<const unsigned*>(P.sc)); else pdl_wait();
    pdl_trigger();
  }
  constexpr int NW = NT / 32;
  constexpr bool WIDE = NT == 256;                             // the variant that also takes rows beyond its registers
  __shared__ float ds_sh[NW];
  __shared__ int sum_sh[NW];
  int mi = 0;
  int block_row = (int)blockIdx.x;
  bool no_grad = false;
  if (SPARSE) {
    const int n_idle = P.idle.end - P.idle.first, token = block_row - n_idle;
    no_grad = token < 0;
    if (!no_grad) pdl_wait();
    pdl_trigger();
    const int id = no_grad ? P.idle.first + block_row : min(max(P.tokens.ids[token], 0), P.mat[0].rows - 1);
    if (load_acquire(P.tokens.row_first + id) != (no_grad ? 0xffffffffu : (unsigned)token)) return;
    block_row = id;
  }
  if (!SPARSE)
    while (mi + 1 < P.n && (int)blockIdx.x >= P.row_end[mi]) ++mi;
  const RowUpdate& M = P.mat[mi];
  const int row = block_row - (mi ? P.row_end[mi - 1] : 0), t = threadIdx.x;
  const int train_w = P.train_w, train_s = P.train_s;
  const long long base = (long long)row * M.cols;
  const int nvec = M.cols / 4;                                 // cols is a multiple of 16
  const bool cached = !WIDE || nvec <= NV * NT;
  float4* w4 = reinterpret_cast<float4*>(M.w + base);
  float4* g4 = reinterpret_cast<float4*>(M.g + base);
  float4* m4 = reinterpret_cast<float4*>(M.m + base);
  float4* v4 = reinterpret_cast<float4*>(M.v + base);
  T* const what = M.what ? reinterpret_cast<T*>(M.what) + base : nullptr;
  int8_t* const codes = M.codes + base;
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 wr[NV], gr[NV], mr[NV], vr[NV];
  // everything is fetched before the first use: the moments' latency hides behind the reduction and the step's update
  if (cached) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = t + i * NT;
      wr[i] = gr[i] = mr[i] = vr[i] = zero4;
      if (c < nvec) {
        wr[i] = w4[c];
        if (no_grad) g4[c] = zero4; else gr[i] = g4[c];
        if (train_w) { mr[i] = m4[c]; vr[i] = v4[c]; }
      }
    }
  }
  const OptimScalars o = *P.sc;
  const float s_old = M.steps[row];
  float ms = 0.f, vs = 0.f;
  if (train_s) { ms = M.m_s[row]; vs = M.v_s[row]; }
  const float qmax = (float)((1 << (P.bits - 1)) - 1);
  const bool masked = M.ds_in != nullptr;                      // gradients were masked and reduced before (same arithmetic)
  // 1. step gradient of this row; the masked gradient is kept for step 3
  const float2 ns_old = splat(-s_old), r_old = splat(__frcp_rn(s_old));
  float2 ds2 = splat(0.f);
  auto ste = [&](float4 wv, float4 d) {
    bool a, b, e, f;
    ds2 = step_grad2<GRID>(ds2, make_float2(wv.x, wv.y), make_float2(d.x, d.y), ns_old, r_old, qmax, a, b);
    ds2 = step_grad2<GRID>(ds2, make_float2(wv.z, wv.w), make_float2(d.z, d.w), ns_old, r_old, qmax, e, f);
    return make_float4(a || masked ? d.x : 0.f, b || masked ? d.y : 0.f, e || masked ? d.z : 0.f, f || masked ? d.w : 0.f);
  };
  if (cached) {
#pragma unroll
    for (int i = 0; i < NV; ++i) gr[i] = ste(wr[i], gr[i]);    // (a vector beyond the row has a zero gradient)
  } else {
    for (int c = t; c < nvec; c += NT) {
      if (no_grad) g4[c] = zero4;
      ste(w4[c], no_grad ? zero4 : g4[c]);
    }
  }
  float ds = warp_sum(ds2.x + ds2.y);
  if ((threadIdx.x & 31) == 0) ds_sh[threadIdx.x >> 5] = ds;
  __syncthreads();
  ds = ds_sh[0];
#pragma unroll
  for (int i = 1; i < NW; ++i) ds += ds_sh[i];
  if (masked) ds = M.ds_in[row];
  // 2. the row's step, formed by every thread
  const float s_new = train_s ? adam_one(s_old, ds, ms, vs, o, 0.f, 1e-8f) : s_old;
  const float sc_new = GRID == 0 ? s_new : 0.5f * s_new;
  // 3 + 4. weights, then their new codes
  const float2 ns_new = splat(-s_new), r_new = splat(__frcp_rn(s_new));
  const Adam2 ad = make_adam2(o);
  const float vanishes = __fmul_rd(0.5f * s_new, 1.401298464e-45f);    // s 2^-150 in whole units of 2^-149 (GRID 1)
  float2 sum2 = splat(0.f);                                    // codes are whole numbers: exact in any order
  auto update = [&](int c, float4 wv, float4 d, float4 mm, float4 vv) {
    float2 wa = make_float2(wv.x, wv.y), wb = make_float2(wv.z, wv.w);
    if (train_w) {
      float2 ma = make_float2(mm.x, mm.y), mb = make_float2(mm.z, mm.w), va = make_float2(vv.x, vv.y), vb = make_float2(vv.z, vv.w);
      wa = adam2(wa, make_float2(d.x, d.y), ma, va, ad);
      wb = adam2(wb, make_float2(d.z, d.w), mb, vb, ad);
      w4[c] = make_float4(wa.x, wa.y, wb.x, wb.y);
      m4[c] = make_float4(ma.x, ma.y, mb.x, mb.y);
      v4[c] = make_float4(va.x, va.y, vb.x, vb.y);
    }
    float2 fa, fb;
    uint32_t b0, b1, b2, b3;
    if (GRID == 0) {      // codes_f, written out: as a call the loads of a row were scheduled worse (30522 x 1024 table, step 205 -> 232 us)
      auto code_quotient = [&](float2 x) {                     // (a first product that overflows ends on its sign's bound)
        const float2 z0 = clamp2(mul2(x, r_new), -qmax - 1.f, qmax + 1.f);
        return clamp2(fma2(fma2(z0, ns_new, x), r_new, z0), -qmax, qmax);
      };
      float2 za = code_quotient(wa), zb = code_quotient(wb);
      fa = rne_magic2(za, b0, b1); fb = rne_magic2(zb, b2, b3);
      const float2 ea = fma2(fa, splat(-1.f), za), eb = fma2(fb, splat(-1.f), zb);
      if (fmaxf(fmaxf(fabsf(ea.x), fabsf(ea.y)), fmaxf(fabsf(eb.x), fabsf(eb.y))) > 0.5f - HALF_WINDOW) {
        za = clamp2(make_float2(exact_quotient(wa.x, s_new), exact_quotient(wa.y, s_new)), -qmax, qmax);
        zb = clamp2(make_float2(exact_quotient(wb.x, s_new), exact_quotient(wb.y, s_new)), -qmax, qmax);
        fa = rne_magic2(za, b0, b1); fb = rne_magic2(zb, b2, b3);
      }
    } else {
      // 2 clamp(floor(w / s), -2, 1) + 1: a quotient of floats rounds to 1 or more exactly when w >= s, and to less than -1
      // exactly when -w > s (the neighbours of s are further than half an ulp of 1 away from it, relatively); it underflows to
      // -0, whose level is that of 0, when -w <= s 2^-150.  A NaN takes the lowest level.
      auto level = [&](float x) { return x >= -vanishes ? (x >= s_new ? 3.f : 1.f) : (-x <= s_new ? -1.f : -3.f); };
      fa = make_float2(level(wa.x), level(wa.y)); fb = make_float2(level(wb.x), level(wb.y));
      const float2 ta = add2(fa, splat(ROUND_MAGIC)), tb = add2(fb, splat(ROUND_MAGIC));
      b0 = __float_as_uint(ta.x); b1 = __float_as_uint(ta.y); b2 = __float_as_uint(tb.x); b3 = __float_as_uint(tb.y);
    }
    *reinterpret_cast<uint32_t*>(codes + 4 * c) = pack_low_bytes(b0, b1, b2, b3);
    const float2 ha = mul2(splat(sc_new), fa), hb = mul2(splat(sc_new), fb);
    if (what) store_what4<T>(what + 4 * c, ha.x, ha.y, hb.x, hb.y);
    sum2 = add2(sum2, add2(fa, fb));
  };
  if (cached) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = t + i * NT;
      if (c < nvec) update(c, wr[i], gr[i], mr[i], vr[i]);
    }
  } else {
    for (int c = t; c < nvec; c += NT) {
      const float4 wv = w4[c];
      update(c, wv, ste(wv, no_grad ? zero4 : g4[c]), train_w ? m4[c] : zero4, train_w ? v4[c] : zero4);
    }
  }
  const int sum = __reduce_add_sync(0xffffffffu, (int)sum2.x + (int)sum2.y);
  if ((threadIdx.x & 31) == 0) sum_sh[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (t == 0) {
    int total = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i) total += sum_sh[i];
    M.rowsum[row] = total;
    M.scale[row] = sc_new;
    if (train_s) {
      M.m_s[row] = ms;
      M.v_s[row] = vs;
      M.steps[row] = s_new;
    }
  }
  if (!SPARSE && P.wait_last) pdl_wait();
}

template <typename T, int NV, int NT, int BLOCKS>
void launch_rows(const UpdateParams& p, int grid, cudaStream_t st) {
  const int rows = p.row_end[p.n - 1];
  if (grid != 0) launch_k(fused_weight_update_kernel<T, NV, NT, BLOCKS, 1, false>, rows, NT, 0, st, p);
  else if (p.tokens.ids)
    launch_k(fused_weight_update_kernel<T, NV, NT, BLOCKS, 0, true>, p.tokens.n + p.idle.end - p.idle.first, NT, 0, st, p);
  else launch_k(fused_weight_update_kernel<T, NV, NT, BLOCKS, 0, false>, rows, NT, 0, st, p);
}
template <typename T>
void launch_variant(int variant, const UpdateParams& p, int grid, cudaStream_t st) {
#define MREM_UPD(I, NT, NV, BLOCKS) case I: launch_rows<T, NV, NT, BLOCKS>(p, grid, st); break;
  switch (variant) { UPD_VARIANTS(MREM_UPD) }
#undef MREM_UPD
}
int variant_of(int cols) {
#define MREM_UPD(I, NT, NV, BLOCKS) if (cols <= NT * NV * 4) return I;
  UPD_VARIANTS(MREM_UPD)
#undef MREM_UPD
  return UPD_WIDEST;
}

}  // namespace

void launch_fused_weight_update(const RowUpdate* mats, int n, const OptimScalars* sc, int bits, int grid, int train_w, int train_s,
                                int dt, cudaStream_t st, bool twins) {
  // One launch per variant.  `twins`: the widest rows first (their blocks are large, and the next launch's fill the SMs as they leave), and
  // the next launch does not wait for the first to end before it loads, only before it ends itself, so that whoever waits for it has
  // waited for both: what the matrices need is complete when the first launch's blocks have passed their wait, which is when the second's
  // may start.  Step of 8 x 256 tokens, hidden 768 932 -> 925 us, 3 x 72 the same; not where a layer's four matrices are updated at once
  // beside longer products (32 x 128, hidden 768 1153 -> 1158).
  bool first = true;
  for (int k = 0; k <= UPD_WIDEST; ++k) {
    const int variant = twins ? UPD_WIDEST - k : k;
    UpdateParams p = {};
    p.bits = bits; p.train_w = train_w; p.train_s = train_s; p.sc = sc; p.wait_last = twins && !first;
    double bytes = 0;
    int rows = 0;
    for (int j = 0; j < n; ++j) {                              // the matrices of one variant go in one launch
      if (variant_of(mats[j].cols) != variant) continue;
      p.mat[p.n] = mats[j];
      p.row_end[p.n++] = rows += mats[j].rows;
      bytes += (double)mats[j].rows * mats[j].cols * (29.0 + (mats[j].what ? (dt == 1 ? 2.0 : 4.0) : 0.0));
    }
    if (p.n == 0) continue;
    Scope scope("fused_weight_update", bytes, 0, st);
    if (dt == 1) launch_variant<bf16>(variant, p, grid, st); else launch_variant<float>(variant, p, grid, st);
    first = false;
  }
}

void launch_table_update(const IdleRows& idle, const TokenRows& tokens, int dt, cudaStream_t st) {
  UpdateParams p = {};
  p.bits = idle.bits; p.train_w = p.train_s = 1; p.sc = idle.sc; p.tokens = tokens; p.idle = idle;
  p.mat[0] = idle.m;
  p.row_end[0] = idle.m.rows;
  p.n = 1;
  // (bytes: the rows without a gradient only; how many have one the host does not know)
  Scope scope("fused_weight_update", (double)(idle.end - idle.first) * idle.m.cols * 29.0, 0, st);
  if (dt == 1) launch_variant<bf16>(variant_of(idle.m.cols), p, 0, st); else launch_variant<float>(variant_of(idle.m.cols), p, 0, st);
}

}  // namespace mrem
