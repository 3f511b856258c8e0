"""Bias and LayerNorm gradients, the sums over the tokens that ride along with other kernels: every form of the LayerNorm backward at
the widths and row counts where it changes, the separate kernels for rows too wide for it, and the attention backward's."""
import numpy as np
import pytest
import torch

from oracle import mrem_oracle as O
from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem, compare_grads, loss_gradients_apart, rel, traced

pytestmark = pytest.mark.gpu


# One to four warps share a row (a thread keeps 8 bf16 or 4 float32 columns), the last one whole or not; wider rows take the
# separate kernels.  Rows: fewer than a block's eight, a few blocks, more than all groups take in one round (2368 at 256
# columns, 1894 at 320, 1184 from 512 on).
@pytest.mark.parametrize("dtype,hidden,ffn,batch,seq", [
    ("bf16", 64, 128, 1, 8), ("bf16", 256, 128, 20, 120), ("bf16", 320, 128, 1, 8), ("bf16", 320, 64, 16, 120), ("bf16", 512, 64, 3, 40),
    ("bf16", 576, 2304, 3, 72), ("bf16", 832, 64, 10, 120), ("bf16", 1088, 64, 3, 40),
    ("f32", 192, 64, 3, 7), ("f32", 256, 64, 1, 2), ("f32", 320, 64, 9, 133), ("f32", 384, 64, 5, 11), ("f32", 512, 64, 3, 7),
    ("f32", 576, 64, 3, 7)])
def test_gradients_of_layers_of_every_row_width(dtype, hidden, ffn, batch, seq):
    """Two layers, so that the LayerNorm backward runs on the loss gradient alone, with a straight-through pass inside and with both.
    Tolerances of the module tests (scalars of the deeper layer: tests/test_scalar_noise_floor.py), and the distance of the loss
    gradients themselves.  The offset's gradient, a sum over the clipped values alone, has too few of them at these sizes."""
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=2, hidden=hidden, n_heads=hidden // 64, ffn=ffn, seq=seq, batch=batch,
                      len_lo=max(1, seq // 3), len_hi=seq, act_dtype=dtype)
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        got = p.run_gpu()
        # (the straight-through pass inside the LayerNorm backward is traced under this name, the separate kernels under others)
        assert ("layernorm_bwd_ste" in traced(p.m, p.run_gpu)) == (hidden <= (1024 if dtype == "bf16" else 512))
        r = p.run_oracle()
        apart = loss_gradients_apart(got, r)
        assert apart < 5e-2, apart                         # (a few flipped roundings; a wrong row or column would be of order 1)
        worst = compare_grads(got["grads"], r["grads"], 2e-2 + apart, check_offset=False, deep_scalar_floor=0.05, deep_group_tol=0.05 + apart)
        print(dtype, hidden, batch, seq, "loss gradients apart", apart, "worst gradient", worst)
    finally:
        p.close()


# one round of rows and two; one, two and three warps a row
@pytest.mark.parametrize("dtype,hidden,batch,seq", [("f32", 256, 5, 64), ("f32", 128, 9, 133), ("f32", 384, 3, 50), ("bf16", 768, 16, 128)])
def test_column_sums_are_those_of_64_bits_but_for_their_last_rounding(dtype, hidden, batch, seq):
    """The gradient of the last LayerNorm's bias is the sum over the tokens of the loss gradient, 2 c (student - teacher) rounded as
    stored.  Rounding the sum to float32 is at most 2^-24 of it and 0.4 of that in the 2-norm over many columns; the few 32-bit
    additions before the 64-bit ones add less than the rest (0.45 2^-24 seen; all additions in 32 bits: 1.4 2^-24)."""
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=hidden, n_heads=hidden // 64, ffn=64, seq=seq, batch=batch,
                      len_lo=max(1, seq // 3), len_hi=seq, act_dtype=dtype)
    p = Problem(wl, student_noise=0.002)
    try:
        m, n = p.m, batch * seq * hidden
        m.quantize_weights()
        t, s = m.forward_teacher(p.xd, p.vld, batch, seq).float(), m.forward_student(p.xd, p.vld, batch, seq).float()
        m.recon_loss()
        m.backward()
        c2 = 2 * (torch.ones((), device=m.device) / torch.full((), float(n), device=m.device))
        d = (c2 * (s - t)).to(m.tdtype).view(-1, hidden).double()
        assert rel(m.grad(0, B.LN2_B, (hidden,)).cpu().numpy(), d.sum(0).cpu().numpy()) < 2.0 ** -24
        assert m.poll_status() == 0
    finally:
        p.close()


# one kernel up to 128 tokens, whole and partly filled tiles; two kernels and a launch for the sums above
@pytest.mark.parametrize("batch,seq", [(3, 8), (2, 72), (3, 120), (5, 128), (35, 128), (3, 136)])
def test_bias_gradient_of_the_qkv_projection_is_the_sum_of_what_the_matrix_gradient_sums(batch, seq):
    """Where a column of the layer's input is one number in every token, its codes are one whole number q: the matrix's gradient in
    that column is step * q times the sum over the tokens of the same stored values that the bias's gradient sums.  Both are float32
    sums of n terms of either sign (the products by q are exact): a few 2^-24 of the sum of their magnitudes, about sqrt(n) times
    the sum itself, apart: at most sqrt(n) 1e-6, where one token too few or too many is 1 / sqrt(n)."""
    H = 128
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=H, n_heads=2, ffn=256, seq=seq, batch=batch, len_lo=max(1, seq // 3),
                      len_hi=seq)
    p = Problem(wl, student_noise=0.002)
    try:
        m = p.m
        p.xd[:, :, 5] = 1.5
        m.quantize_weights()
        m.forward_teacher(p.xd, p.vld, batch, seq)
        m.forward_student(p.xd, p.vld, batch, seq)
        m.recon_loss()
        m.backward()
        step = np.float32(m.get_steps()[1][0, 0])
        q = np.rint(np.float32(1.5) / step)
        assert 1 <= abs(q) <= 127
        # (rows whose weight in that column lies inside the quantizer's range: its gradient is not masked)
        inside = np.abs(p.student[0]["Wqkv"][:, 5] / p.ws[0]["Wqkv"].reshape(-1)) < 6.9
        w = m.grad(0, B.WQKV, (3 * H, H)).cpu().numpy()[:, 5].astype(np.float64) / (float(step) * q)
        b = m.grad(0, B.BQKV, (3 * H,)).cpu().numpy().astype(np.float64)
        for plane in (0, 2):                               # (a key's bias moves all scores of a row alike: its gradient is rounding)
            rows = np.flatnonzero(inside[plane * H:(plane + 1) * H]) + plane * H
            assert len(rows) > H // 2 and np.abs(b[rows]).max() > 0
            assert rel(w[rows], b[rows]) < 1e-6 * np.sqrt(batch * seq), rel(w[rows], b[rows])
        rows = np.flatnonzero(inside[H:2 * H]) + H
        assert np.abs(w[rows] - b[rows]).max() < 1e-6 * batch * seq * np.abs(b[:H]).max()
    finally:
        p.close()
