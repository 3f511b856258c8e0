"""The fused attention kernels at the edges of their tiles: sequence lengths around 128, 256 and 384 (where threads per row,
shared-memory layout and the number of kernels change), valid lengths of one key and around multiples of 16, 32 and 128."""
import numpy as np
import pytest
import torch

from oracle import mrem_oracle as O
from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem
from tests.test_gpu_module import compare_grads

pytestmark = pytest.mark.gpu


# (seq, valid lengths of the three sequences); 2e-2 against the oracle's gradients: the module tests' tolerance
@pytest.mark.parametrize("seq,lens", [(8, (1, 8, 5)), (64, (64, 33, 1)), (120, (120, 97, 16)), (128, (128, 127, 64)), (136, (136, 128, 1)),
                                      (192, (192, 129, 31)), (256, (256, 255, 65)), (264, (264, 257, 130)), (384, (384, 353, 96))])
def test_attention_at_the_edges_of_its_tiles(seq, lens):
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=len(lens))
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        p.vl = np.array(lens, np.int32)
        p.vld = torch.from_numpy(p.vl).to(p.m.device)
        r = p.run_oracle()
        fused = p.run_gpu()
        compare_grads(fused["grads"], r["grads"], 2e-2, check_offset=True)
        # the probabilities, which the fused path forms again when they are asked for, are those the kernel-per-operation
        # path stores, bit for bit
        m = p.m
        shape = (wl.batch, wl.n_heads, seq, seq)

        def probabilities():
            m.quantize_weights()
            m.forward_student(p.xd, p.vld, wl.batch, seq)
            return m.activation(B.STUDENT, 0, B.ACT_P, shape)

        a = probabilities()
        m.set_fused_attention_backward(False)
        b = probabilities()
        assert torch.equal(a, b)
        for i, n in enumerate(lens):
            assert not a[i, :, :, n:].any() and torch.allclose(a[i].float().sum(-1), torch.ones((), device=m.device), atol=2 ** -8 * 2)
    finally:
        p.close()


# one kernel, two kernels
@pytest.mark.parametrize("seq", [72, 200])
def test_reading_the_probabilities_leaves_the_backward_pass_alone(seq):
    """The fused path forms the probabilities when they are read, without their codes: the gradients that follow are the same bits."""
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=2)
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        m = p.m

        def gradient(read):
            m.quantize_weights()
            m.forward_teacher(p.xd, p.vld, wl.batch, seq)
            m.forward_student(p.xd, p.vld, wl.batch, seq)
            if read:
                m.activation(B.STUDENT, 0, B.ACT_P, (wl.batch, wl.n_heads, seq, seq))
            m.recon_loss()
            m.backward()
            return m.grad(0, B.WQKV, (3 * wl.hidden, wl.hidden)).clone()

        a = gradient(False)
        assert a.any() and torch.equal(a, gradient(True))
    finally:
        p.close()
