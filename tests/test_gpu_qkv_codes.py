"""The codes of Q, K and V that the QKV product's epilogue writes against the quantizer's own launch on the values it stored."""
import pytest
import torch

from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem

pytestmark = pytest.mark.gpu


# one head (a tile of 192 columns holds all three segments), segments that end inside a tile, tiles of 64 to 256 columns; ragged
# rows; few rows of a wide layer (several thread blocks share a tile); codes of 8 and 4 bits, steps small enough to clip
@pytest.mark.parametrize("hidden,batch,seq,a_bits", [(64, 1, 8, 8), (64, 5, 40, 4), (128, 3, 40, 8), (192, 7, 56, 8), (320, 9, 64, 4), (768, 8, 256, 8),
                                                     (1024, 3, 40, 8), (1024, 32, 128, 4), (2048, 1, 40, 8)])
def test_codes_from_the_epilogue_are_the_quantizer_s(hidden, batch, seq, a_bits):
    wl = synth.shrink(synth.workloads()["large6_w4a8"], n_layers=1, hidden=hidden, n_heads=hidden // 64, ffn=2 * hidden, seq=seq, batch=batch,
                      len_lo=max(1, seq // 4), len_hi=seq)
    p = Problem(wl, step_shrink=0.3, student_noise=0.002, a_bits=a_bits)
    try:
        m = p.m
        m.quantize_weights()
        m.forward_student(p.xd, p.vld, batch, seq)
        ptr, n = B.mrem_get_activation(m.ctx, B.STUDENT, 0, B.ACT_QKV), batch * seq * 3 * hidden
        values = m._ws_view(ptr, n, torch.bfloat16).view(-1, 3, hidden)
        # the codes lie behind the values in the workspace (pieces of 256 bytes)
        codes = m._ws_view(ptr + (2 * n + 255) // 256 * 256, n, torch.bfloat16).view(-1, 3, hidden)
        hi, clipped = 2 ** (a_bits - 1) - 1, 0
        for seg in range(3):
            x = values[:, seg].contiguous()
            want = torch.empty_like(x)
            B.mrem_quantize_act(x, B.BF16, x.numel(), m.a_steps[0, 1 + seg], None, -hi, hi, None, want, m.stream)
            torch.cuda.synchronize()
            assert torch.equal(codes[:, seg], want), seg
            clipped += int((want.abs() == hi).sum())
        assert clipped > 0
    finally:
        p.close()
