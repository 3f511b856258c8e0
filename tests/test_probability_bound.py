"""The bound by which the attention backward kernels decide whether a row's probabilities can be clipped, emulated in numpy:
no stored probability lies above it, and it is the stored 1 / sum unless that is next to a rounding boundary."""
import numpy as np

from oracle import mrem_oracle as O

f32 = np.float32


def test_no_stored_probability_is_above_its_rows_bound():
    rng = np.random.default_rng(0)
    rows, keys = 40_000, 24
    alpha2 = (10.0 ** rng.uniform(-4, 0, (rows, 1))).astype(f32)
    score = np.rint(rng.standard_normal((rows, keys)) * 10.0 ** rng.uniform(1, 5, (rows, 1))).astype(f32)   # sums of codes' products
    score[: rows // 4] = score[: rows // 4, :1]                               # equal scores: the residual weighs most
    m = (alpha2 * score.max(1, keepdims=True)).astype(f32)
    t = (alpha2.astype(np.float64) * score - m).astype(f32)                   # fma: one rounding
    for off in (-2.0 ** -22, 0.0, 2.0 ** -22):                                # the approximate exponential's relative error
        e = np.exp2(t.astype(np.float64))
        total = e.astype(f32).sum(1, keepdims=True, dtype=f32)
        inv = (f32(1.0) / total).astype(f32)
        p = ((e * (1 + off)).astype(f32) * inv).astype(f32)
        stored = O.round_bf16(p).max(1)
        up = np.exp2(np.abs(m).astype(np.float64) * 2.0 ** -24) * (1 - abs(off))
        bound = O.round_bf16((inv * up.astype(f32) * f32(1 + 2.0 ** -20)).astype(f32))[:, 0]
        plain = O.round_bf16(inv)[:, 0]
        assert np.all(stored <= bound)
        small = np.abs(m)[:, 0] < 64
        assert (stored > plain).any() and (bound[small] > plain[small]).mean() < 1e-2
