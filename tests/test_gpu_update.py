"""The fused update of a layer's matrices against the oracle's AdamW and quantizer, at the edges of its variants."""
import numpy as np
import pytest
import torch

from oracle import mrem_oracle as O
from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200 import synth
from tests.gpu_util import Problem

pytestmark = pytest.mark.gpu


# widths of W2's rows: one vector slot unused, full and just beyond each variant (768, 1024, 2048, 3072, 4096 wide)
@pytest.mark.parametrize("grid,ffn", [(0, 16), (1, 752), (0, 768), (1, 784), (0, 1024), (0, 1040), (1, 2048), (0, 2064), (0, 3072),
                                      (1, 3088), (0, 4096), (0, 4112), (1, 4112)])
def test_fused_update_at_the_edges_of_its_row_variants(grid, ffn):
    """One step from the raw gradients (unmasked inside the update), and one from gradients masked beforehand.

    Bounds: one step from zero moments moves every value by lr g / (|g| + eps), formed with a dozen roundings and two
    approximate instructions (2 ulp): lr 2^-20, plus the value's own rounding.  A step's gradient is a sum of n terms
    d (level - z), each off by at most the roundings of n additions and one ulp of z; relative to the sum that is what its
    direction can be wrong by.  Codes and row sums are whole numbers formed from the stored weights and steps: exact."""
    wl = synth.shrink(synth.workloads()["base3_w2a8" if grid else "base3_w4a8"], n_layers=1, hidden=64, n_heads=1, ffn=ffn, seq=24,
                      batch=2, len_lo=5, len_hi=24)
    lr, wd = 1e-3, 0.01
    opt = B.make_optim(lr=lr, step=1, weight_decay=wd)
    f32 = lambda x: float(np.float32(x))
    for masked in (False, True):
        p, q = Problem(wl, step_shrink=0.8, student_noise=0.002), Problem(wl, step_shrink=0.8, student_noise=0.002)
        try:
            m = p.m
            for a in (p, q):
                a.m.quantize_weights()
                a.m.forward_teacher(a.xd, a.vld, wl.batch, wl.seq)
                a.m.forward_student(a.xd, a.vld, wl.batch, wl.seq)
                a.m.recon_loss()
                a.m.backward()
            base, n = B.mrem_grad_bucket(m.ctx, 0)
            raw = m._ws_view(base, n, torch.float32).cpu().numpy().copy()
            base_q, _ = B.mrem_grad_bucket(q.m.ctx, 0)
            w0, s0 = m.student_numpy()[0], m.get_steps()[0][0]
            offsets = {pid: (B.mrem_get_grad(q.m.ctx, 0, pid) - base_q) // 4 for pid in (B.WQKV, B.WO, B.W1, B.W2)}   # (masks q's)
            if masked:
                B.mrem_get_grad(m.ctx, 0, B.W2)
            m.step(opt)
            torch.cuda.synchronize()
            w1, s1 = m.student_numpy()[0], m.get_steps()[0][0]
            for pid in (B.WQKV, B.WO, B.W1, B.W2):
                name = B.PARAM_NAMES[pid]
                w, s = w0[name], np.asarray(s0[name], np.float32).reshape(-1, 1)
                d = raw[offsets[pid]:offsets[pid] + w.size].reshape(w.shape).astype(np.float64)
                z = (w / s).astype(np.float64)
                if grid:
                    inside, level = (z >= -2) & (z < 2), np.clip(np.floor(z), -2, 1) + 0.5
                else:
                    qmax = 2 ** (wl.w_bits - 1) - 1
                    inside, level = np.abs(z) <= qmax, np.rint(np.clip(z, -qmax, qmax))
                terms = d * (level - np.where(inside, z, 0.0))
                ds = terms.sum(1)
                ds_err = 2.0 ** -24 * ((w.shape[1] + 4) * np.abs(terms).sum(1) + 2 * np.abs(d * z).sum(1))
                kw = dict(beta1=f32(0.9), beta2=f32(0.999), eps=f32(1e-8))
                ref_s = np.maximum(O.adamw_update(s[:, 0], ds, 0 * ds, 0 * ds, 1, f32(lr), **kw)[0], 1e-8)
                got_s = np.asarray(s1[name], np.float64).reshape(-1)
                wrong = np.minimum(2.0, 2 * ds_err / np.maximum(np.abs(ds), 1e-300))
                assert np.all(np.abs(got_s - ref_s) <= lr * (2.0 ** -20 + wrong) + 2.0 ** -23 * s[:, 0]), (masked, name)
                ref_w = O.adamw_update(w, d * inside, 0 * d, 0 * d, 1, f32(lr), weight_decay=f32(wd), **kw)[0]
                assert np.all(np.abs(w1[name] - ref_w) <= lr * 2.0 ** -20 + 2.0 ** -23 * np.abs(w)), (masked, name)
                codes, rowsum = m.weight_codes(0, pid)
                ref_q = O.quantize_weight(w1[name], np.asarray(s1[name], np.float32).reshape(-1, 1), wl.w_bits, grid, "f32")[0]
                assert np.array_equal(codes.cpu().numpy(), ref_q), (masked, name)
                assert np.array_equal(rowsum.cpu().numpy(), ref_q.sum(1)), (masked, name)
        finally:
            p.close()
            q.close()


def test_half_integer_codes_of_the_update_are_those_of_the_quantizer():
    """A learning rate of zero leaves the weights as they are, so the update has to leave the codes that the quantizer made of
    them (by the division of Eq. 1): around the levels' ends, where the quotient underflows, and for values that are no numbers."""
    wl = synth.shrink(synth.workloads()["base3_w2a8"], n_layers=1, hidden=64, n_heads=1, ffn=128, seq=24, batch=2, len_lo=5, len_hi=24)
    p = Problem(wl)
    try:
        m, f32 = p.m, np.float32
        w, s = p.student[0]["W1"], np.asarray(p.ws[0]["W1"], f32).reshape(-1)
        s[:] = np.exp2(np.linspace(-12, 12, s.size)).astype(f32) * np.linspace(1, 2, s.size, endpoint=False).astype(f32)
        edges = [0.0, 1e-45, 1e-44, 1e-42, 1e-38, np.inf]
        for r, step in enumerate(s):
            near = [np.nextafter(step, f32(0)), step, np.nextafter(step, f32(np.inf)), 2 * step]
            tie = [f32(k) * f32(1e-45) for k in (np.floor(step / 2) + np.arange(-1, 3)) if k > 0]
            row = np.array(edges + near + tie, f32)
            row = np.concatenate([row, -row, [f32(np.nan)]])
            w[r, :row.size] = row
        m.load_student(p.student)
        m.set_steps(p.ws, p.a, p.off)
        m.quantize_weights()
        before = [x.clone() for x in m.weight_codes(0, B.W1)]
        m.forward_teacher(p.xd, p.vld, wl.batch, wl.seq)
        m.forward_student(p.xd, p.vld, wl.batch, wl.seq)
        m.recon_loss()
        m.backward()
        m.step(B.make_optim(lr=0.0, step=1, weight_decay=0.0))
        assert np.array_equal(m.get_steps()[0][0]["W1"].reshape(-1), s)
        after = m.weight_codes(0, B.W1)
        assert set(after[0].unique().tolist()) == {-3, -1, 1, 3}
        assert torch.equal(after[0], before[0]) and torch.equal(after[1], before[1])
    finally:
        p.close()
