"""The fused attention kernels at the edges of their tiles: sequence lengths around 128, 256 and 384 (where threads per row,
shared-memory layout and the number of kernels change), valid lengths of one key and around multiples of 16, 32 and 128."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from oracle import mrem_oracle as O
from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem, rel
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


# above 128 tokens more blocks than run at once: they take the sequences longest first (equal lengths, one key, whole chunks and
# one more among them); up to 128 tokens more blocks than SMs: a thread per row instead of four
@pytest.mark.parametrize("seq,batch", [(136, 12), (320, 8), (136, 32), (8, 32), (72, 12), (104, 12), (128, 18)])
def test_sequences_of_a_large_batch_are_those_of_a_small_one(seq, batch):
    """The quantized pass treats sequences independently (whole numbers, and row sums in the same order): bit for bit the outputs
    of the same sequences two at a time, which are few blocks."""
    wl = synth.shrink(synth.workloads()["large6_w4a8"], n_layers=1, seq=seq, batch=batch, len_lo=1, len_hi=seq)
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        m = p.m
        lens = np.array(([seq, 1, 64, 65, seq, 128, 129, seq - 1, 64, 33, 32, 97] * 3)[:batch], np.int32).clip(1, seq)
        vld = torch.from_numpy(lens).to(m.device)
        m.quantize_weights()
        many = m.forward_student(p.xd, vld, batch, seq).clone()
        for i in range(0, batch, 6):
            two = m.forward_student(p.xd[i:i + 2].contiguous(), vld[i:i + 2].clone(), 2, seq)
            assert torch.equal(two, many[:, i:i + 2]), i
    finally:
        p.close()


# above 128 tokens a slot of step-size partials per block, and one more block than there are slots (the blocks of a head share one);
# up to 128 tokens as many blocks as SMs (four threads per row), and more (two)
@pytest.mark.parametrize("seq,batch", [(136, 295), (136, 297), (40, 74), (40, 75), (128, 75)])
def test_gradients_on_both_sides_of_the_number_of_blocks(seq, batch):
    """Against the kernel-per-operation path: the weight and bias gradients by a few bf16 roundings of dS and dQKV (2^-9 each, averaged
    over thousands of rows: 1e-2 leaves a factor of two for each), the step gradients as everywhere within 2e-2 of the largest."""
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=batch, len_lo=1, len_hi=seq)
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        got = []
        for fused in (True, False):
            p.m.set_fused_attention_backward(fused)
            got.append(p.run_gpu()["grads"][0])
        assert rel(got[0]["Wqkv"], got[1]["Wqkv"]) < 1e-2 and rel(got[0]["bqkv"], got[1]["bqkv"]) < 1e-2
        a, b = got[0]["a"], got[1]["a"]
        assert np.isfinite(a).all() and np.abs(a - b).max() < 2e-2 * np.abs(b).max(), (a, b)
    finally:
        p.close()


def _rounded_up_case(a_bits, lo_len, hi_len):
    """A step s, codes cq and ck, a number of keys n and a step s_p such that n equal scores alpha 64 cq ck have probabilities
    1 / n that are stored one bf16 spacing ABOVE the stored 1 / sum, with the upper end of P's range between the two: the
    kernels' exponent of the largest score is the rounding error r of alpha log2(e) score, so their sum is n 2^r."""
    f32 = np.float32
    p_hi, cq, ck = (255, 120, 121) if a_bits == 8 else (15, 5, 6)
    r, s = -1.0, None
    for t in np.sqrt(np.linspace(7e3, 1e4, 200) / (8 * cq * ck)).astype(f32):        # scores of 7,000 to 10,000
        alpha2 = f32(f32(f32(0.125) * t) * t) * f32(1.4426950408889634)
        score = f32(64 * cq * ck)
        err = float(alpha2) * float(score) - float(f32(alpha2 * score))
        if err > r:
            r, s = err, t
    for n in range(lo_len, hi_len + 1):
        up, low = float(O.round_bf16(np.array(1.0 / n))), float(O.round_bf16(np.array(2.0 ** -r / n)))
        middle = (low + up) / 2
        if low < up and 1.0 / n > (1 + 2e-5) * middle and 2.0 ** -r / n < (1 - 2e-5) * middle:
            return s, cq, ck, n, f32((low + 0.25 * (up - low)) / p_hi), up
    raise AssertionError("no such case")


# one kernel and two, 8- and 4-bit codes
@pytest.mark.parametrize("seq,a_bits", [(64, 8), (128, 4), (264, 8), (384, 4)])
def test_probabilities_stored_above_the_reciprocal_sum_are_clipped(seq, a_bits):
    """Every probability is one bf16 spacing beyond its quantizer's range although the row's 1 / sum, as stored, is not.  All of
    them are then clipped: no gradient reaches Q, K and their steps, and the value gradients see the highest code.  The step
    gradient of P is a sum of d times the highest code, 2e-2 from the oracle's as everywhere; the value gradients differ from
    the kernel-per-operation path's by a few bf16 roundings (2^-9 each), where one code more would be 1 / 255 or 1 / 15."""
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=2)
    H = wl.hidden
    s, cq, ck, n, s_p, stored = _rounded_up_case(a_bits, seq // 2, seq)
    p = Problem(wl, step_shrink=0.8, student_noise=0.002, a_bits=a_bits)
    try:
        m = p.m
        p.vl = np.array([n, n], np.int32)
        p.vld = torch.from_numpy(p.vl).to(m.device)
        p.student[0]["Wqkv"][:2 * H] = 0
        p.student[0]["bqkv"][:H], p.student[0]["bqkv"][H:2 * H] = cq * s, ck * s
        p.a[0, 1], p.a[0, 2], p.a[0, 4] = s, s, s_p
        m.load_student(p.student)
        m.set_steps(p.ws, p.a, p.off)
        r = p.run_oracle()["grads"][0]
        got = []
        for fused in (True, False):
            m.set_fused_attention_backward(fused)
            got.append(p.run_gpu()["grads"][0])
            P = m.activation(B.STUDENT, 0, B.ACT_P, (2, wl.n_heads, seq, seq)).float()
            assert (P[..., :n] == stored).all() and not P[..., n:].any()
        g, per_op = got
        assert not g["bqkv"][:2 * H].any() and not g["Wqkv"][:2 * H].any() and g["a"][1] == 0 and g["a"][2] == 0
        assert abs(g["a"][4] - r["a"][4]) <= 2e-2 * abs(r["a"][4])
        assert rel(g["bqkv"][2 * H:], per_op["bqkv"][2 * H:]) < 2e-3 and rel(g["Wqkv"][2 * H:], per_op["Wqkv"][2 * H:]) < 2e-3
    finally:
        p.close()


# clusters of two and three blocks in which all but the first hold padding only
@pytest.mark.parametrize("seq,lens", [(256, (1, 128, 60)), (384, (1, 77, 128))])
def test_step_gradients_of_sequences_that_are_mostly_padding(seq, lens):
    """The blocks of a head whose keys are all padding have nothing to do before they hand in their share of the step
    gradients: against the oracle, and the same bits every time.  (Not the offset gradient, which does not pass through
    these kernels: at 384 tokens it is 2 % of the sum of its 23 terms' sizes, and the oracle itself moves by 13 to 29 % when
    its stored tensors are perturbed by 3e-6.)"""
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=len(lens))
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        p.vl = np.array(lens, np.int32)
        p.vld = torch.from_numpy(p.vl).to(p.m.device)
        first = p.run_gpu()["grads"]
        compare_grads(first, p.run_oracle()["grads"], 2e-2, check_offset=False)
        for _ in range(20):
            assert np.array_equal(p.run_gpu()["grads"][0]["a"], first[0]["a"])
    finally:
        p.close()


# the quantized site the value belongs to, one kernel and two
@pytest.mark.parametrize("seq", [72, 200])
@pytest.mark.parametrize("site", ["q", "k", "v"])
def test_a_value_that_is_not_a_number_takes_no_gradient(seq, site):
    """Eq. 1's comparisons are false for a NaN: its code is the lowest one and the straight-through mask stops its gradient, in
    the fused kernels as in the kernel-per-operation path; the step gradients of the others stay numbers."""
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=2)
    p = Problem(wl, step_shrink=1.5, student_noise=0.002)            # (nothing else is clipped)
    try:
        m, at = p.m, 70 + wl.hidden * "qkv".index(site)
        p.student[0]["bqkv"][at] = np.nan
        m.load_student(p.student)
        m.set_steps(p.ws, p.a, p.off)
        got = []
        for fused in (True, False):
            m.set_fused_attention_backward(fused)
            got.append(p.run_gpu()["grads"][0])
        g, per_op = got
        assert np.isfinite(g["a"]).all() and g["bqkv"][at] == 0 and per_op["bqkv"][at] == 0
        assert np.abs(g["a"] - per_op["a"]).max() <= 2e-2 * np.abs(per_op["a"]).max()
        assert rel(g["bqkv"], per_op["bqkv"]) < 2e-2 and rel(g["Wqkv"], per_op["Wqkv"]) < 2e-2
    finally:
        p.close()


# longer than the fused kernels take; more heads than there are slots for their partial sums
@pytest.mark.parametrize("seq,batch", [(392, 2), (16, 600)])
def test_sizes_beyond_the_fused_backward_kernels(seq, batch):
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=batch, len_lo=seq // 4, len_hi=seq)
    p = Problem(wl, step_shrink=0.8, student_noise=0.002)
    try:
        compare_grads(p.run_gpu()["grads"], p.run_oracle()["grads"], 2e-2, check_offset=True)
    finally:
        p.close()


def test_contexts_of_different_lengths_make_their_first_pass_together():
    """Contexts are independent: threads whose sequences take the same variants of the kernels with different amounts of shared
    memory (and other variants) start at the same moment in a fresh process; every pass equals the same one made alone."""
    code = """
import threading
import torch
from tests.gpu_util import Problem
from paper_2109_15082_b200 import synth
lengths = (256, 136, 384, 264, 200, 328)
ps, outs, errs = [], {}, []
for seq in lengths:
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        p = Problem(synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=128, n_heads=2, ffn=256, seq=seq, batch=2))
        ps.append((seq, p, st))
torch.cuda.synchronize()
gate = threading.Barrier(len(ps))
def run(seq, p, st, key, wait):
    try:
        if wait:
            gate.wait()
        with torch.cuda.stream(st):
            p.m.quantize_weights()
            t = p.m.forward_teacher(p.xd, p.vld, 2, seq).clone()
            s = p.m.forward_student(p.xd, p.vld, 2, seq).clone()
        st.synchronize()
        outs[key, seq] = (t, s)
    except Exception as e:
        errs.append((seq, repr(e)))
threads = [threading.Thread(target=run, args=(*x, "together", True)) for x in ps]
for t in threads: t.start()
for t in threads: t.join()
assert not errs, errs
for x in ps: run(*x, "alone", False)
assert not errs, errs
for seq, p, st in ps:
    assert all(torch.equal(a, b) for a, b in zip(outs["together", seq], outs["alone", seq])), seq
    assert p.m.poll_status() == 0
    p.close()
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
