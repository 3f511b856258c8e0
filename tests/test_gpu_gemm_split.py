"""Products with few tiles and a long inner dimension, which several thread blocks share."""
import numpy as np
import pytest
import torch

from oracle import mrem_oracle as O
from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem, compare_grads, rel
from tests.test_gpu_full_width import teacher_layer_stage_by_stage
from tests.test_gpu_module import rem_step_of_one_product

pytestmark = pytest.mark.gpu
DEV = "cuda"


# one row, full and just beyond a tile; one, two and three 32-column chunks, many tiles; the fewest 128-byte deep blocks that
# are shared (8), an odd number of them with a ragged last one, and many
@pytest.mark.parametrize("M", [1, 128, 129, 216])
@pytest.mark.parametrize("N", [32, 96, 768])
@pytest.mark.parametrize("blocks,ragged", [(8, 0), (11, 3), (33, 1), (48, 0)])
def test_shared_products_are_exact(M, N, blocks, ragged):
    """Whole numbers small enough that every partial sum is exact (|sum| <= 3072 * 16 < 2^24): equal in any order, bit for bit."""
    rng = np.random.default_rng(M + N + blocks)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    stream = torch.cuda.current_stream().cuda_stream
    K = 64 * blocks - 16 * ragged
    a, b = rng.integers(-4, 5, (M, K)), rng.integers(-4, 5, (N, K))
    ref = O.int_matmul(a, b)
    for a_mn, b_mn in ((0, 0), (0, 1), (1, 1)):
        if a_mn and M % 8:
            continue                                       # the strides of an operand are multiples of 16 bytes
        ad = torch.from_numpy(np.ascontiguousarray(a.T if a_mn else a)).to(DEV).to(torch.bfloat16)
        bd = torch.from_numpy(np.ascontiguousarray(b.T if b_mn else b)).to(DEV).to(torch.bfloat16)
        out = torch.full((M, N), 0.5, device=DEV)
        B.mrem_gemm(B.BF16, ad, a_mn, M if a_mn else K, 0, bd, b_mn, N if b_mn else K, 0, M, N, K, 1, 1.0, out, N, 0, 0, status, stream)
        assert np.array_equal(out.cpu().numpy().astype(np.int64), ref), (a_mn, b_mn)
    K *= 2
    a, b = rng.integers(-127, 128, (M, K)), rng.integers(-127, 128, (N, K))
    acc = torch.full((M, N), -1, dtype=torch.int32, device=DEV)
    B.mrem_gemm_i8(torch.from_numpy(a.astype(np.int8)).to(DEV), 0, torch.from_numpy(b.astype(np.int8)).to(DEV), M, N, K, acc, 0, status, stream)
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), O.int_matmul(a, b))
    assert int(status[0]) == 0


# The cost model splits these products.  At 3 x 40 tokens and BERT-large widths: all four of the full-precision pass (bias; bias
# and residual; bias and GELU), FFN2 of the quantized pass, all input gradients.  At 3 x 72: output projection and FFN2, FFN2, all
# input gradients but FFN2's.  At hidden and FFN 2048, 40 or 120 tokens: all of the quantized pass but QKV.

def test_shared_products_of_the_full_precision_pass_stage_by_stage():
    """Bias, bias + residual, bias + GELU: every stored tensor against the oracle's arithmetic for that stage."""
    teacher_layer_stage_by_stage(synth.shrink(synth.workloads()["large6_w4a8"], n_layers=1, seq=40, batch=3, len_lo=10, len_hi=40))


@pytest.mark.parametrize("seq", [40, 72])
def test_gradients_through_shared_products(seq):
    wl = synth.shrink(synth.workloads()["large6_w4a8"], n_layers=1, seq=seq, batch=3, len_lo=10, len_hi=seq)
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        g, r = p.run_gpu(), p.run_oracle()
        assert rel(g["f_s"], r["f_s"]) < 1e-3 and abs(g["loss"] - r["loss"]) <= 2e-2 * r["loss"]
        compare_grads(g["grads"], r["grads"], 2e-2, check_offset=True)
    finally:
        p.close()


@pytest.mark.parametrize("hidden,ffn", [(1024, 4096), (2048, 2048)])
def test_a_sequence_alone_and_in_a_batch_give_the_same_bits(hidden, ffn):
    """The quantized pass multiplies whole numbers and treats rows independently: a sequence whose products are shared between
    thread blocks has the outputs, bit for bit, that it has among 32, whose products are not."""
    wl = synth.shrink(synth.workloads()["large6_w4a8"], n_layers=1, hidden=hidden, n_heads=hidden // 64, ffn=ffn, seq=40, batch=32, len_lo=10,
                      len_hi=40)
    p = Problem(wl, student_noise=0.002)
    try:
        m = p.m
        m.quantize_weights()
        many = m.forward_student(p.xd, p.vld, 32, 40).clone()
        for i in (0, 31):
            one = m.forward_student(p.xd[i:i + 1].contiguous(), p.vld[i:i + 1].clone(), 1, 40)
            assert torch.equal(one[:, 0], many[:, i]), i
        three = m.forward_student(p.xd[5:8].contiguous(), p.vld[5:8].clone(), 3, 40)
        assert torch.equal(three, many[:, 5:8])
    finally:
        p.close()


# W2 with its offset as a column bias and without one (scale only), and the output projection
@pytest.mark.parametrize("name,asym", [("W2", 3), ("W2", 1), ("Wo", 3)])
def test_per_product_step_on_shared_products(name, asym):
    rem_step_of_one_product(synth.shrink(synth.workloads()["large6_w4a8"], n_layers=1, seq=72, batch=3, len_lo=10, len_hi=72), name, asym)
