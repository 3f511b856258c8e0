"""The refitted weight scale at every width of its row kernel, and at rows whose weights lie far apart."""
import numpy as np
import pytest
import torch

from oracle import mrem_oracle as O
from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem

pytestmark = pytest.mark.gpu
MATRICES = ((B.WQKV, "Wqkv"), (B.WO, "Wo"), (B.W1, "W1"), (B.W2, "W2"))


def _scales(m, layer, pid):
    """The dequantization scales, which lie behind the row sums in the workspace (pieces of 256 bytes)."""
    rows = m.shapes[pid][0]
    _, rowsum = B.mrem_get_weight_codes(m.ctx, layer, pid)
    return m._ws_view(rowsum + (4 * rows + 255) // 256 * 256, rows, torch.float32).cpu().numpy()


def _far_apart(w, rng):
    """Rows of zeros, of one value, below and above the range of the byte sums, and with one weight 2^1 to 2^24 times the others'."""
    w[0] = 0.0
    w[1] = np.float32(-0.03)
    w[2] *= np.float32(1e-32)
    w[3] *= np.float32(1e32)
    w[4] *= np.float32(1e-37)
    for i in range(5, 29):
        w[i, int(rng.integers(w.shape[1]))] = np.float32(0.02 * 2.0 ** (i - 4) * (-1) ** i)
    w[29, ::2] = -0.0


def _check(m, w, bits):
    for pid, name in MATRICES:
        codes, rowsum = m.weight_codes(0, pid)
        ref, alpha, _ = O.quantize_weight_laq(w[name], bits, True)
        assert np.array_equal(codes.cpu().numpy().astype(np.int64), ref), name
        assert np.array_equal(rowsum.cpu().numpy().astype(np.int64), ref.sum(-1)), name
        # both sums are good to 2^-46 or better: the scales are equal but for a quotient that close to the middle of two floats
        got, want = _scales(m, 0, pid), alpha[:, 0].astype(np.float32)
        assert np.all(np.abs(got.astype(np.float64) - want) <= np.spacing(want)) and np.mean(got != want) < 0.01, name


# widths of 16 to 4096 (2, 4, 6 and 8 vectors a thread, one to four warps, last vectors missing); 8 bits take float64 sums
@pytest.mark.parametrize("hidden,ffn,bits", [(64, 80, 4), (64, 272, 2), (128, 400, 4), (320, 640, 4), (768, 3072, 4), (768, 1040, 2),
                                             (1024, 4096, 4), (128, 1536, 8), (64, 2064, 4)])
def test_refitted_scales_and_codes_are_the_oracle_s(hidden, ffn, bits):
    wl = synth.shrink(synth.workloads()["base3_w4a8"], n_layers=1, hidden=hidden, n_heads=hidden // 64, ffn=ffn, seq=8, batch=1, len_lo=8, len_hi=8,
                      w_grid=3, w_bits=bits)
    p = Problem(wl, student_noise=0.002)
    try:
        m = p.m
        p.run_gpu()
        _check(m, p.student[0], bits)
        m.step(B.make_optim(step=1, lr=0.0, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.01))   # the update's own copy of the rule
        torch.cuda.synchronize()
        after = m.student_numpy()
        assert all(np.array_equal(after[0][n], p.student[0][n]) for _, n in MATRICES)
        _check(m, after[0], bits)
        rng = np.random.default_rng(hidden + ffn)
        for _, n in MATRICES:
            _far_apart(p.student[0][n], rng)
        m.load_student(p.student)
        m.quantize_weights()
        _check(m, p.student[0], bits)
        p.student[0]["W2"][7, ffn - 1] = np.nan                      # no scale for a row that holds something else than numbers
        p.student[0]["W2"][8, 0] = -np.inf
        m.load_student(p.student)
        m.quantize_weights()
        bad = ~np.isfinite(_scales(m, 0, B.W2))
        assert bad[7] and bad.sum() <= 2
    finally:
        p.close()
