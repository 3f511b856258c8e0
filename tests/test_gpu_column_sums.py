"""Bias and LayerNorm gradients: the sums over the tokens that ride along with other kernels."""
import pytest
import torch

from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem, rel

pytestmark = pytest.mark.gpu


# one round of rows and two; two, three and four warps a row
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
