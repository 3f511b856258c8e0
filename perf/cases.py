"""Performance cases: the calls a user of this framework makes, over the range of sizes it is used at.

Six kinds of call, each through the public classes of the package (`session`, `dist`, `embedding`) and `binding`:

  step    one reconstruction step the way `ModuleSweep.run_module` takes it: gather the next calibration batch (and its
          valid lengths) from the device, replay the captured step.  Returns the loss and every updated parameter and
          step size.
  grads   one data-parallel step of one rank (`DataParallelModule.step`, no process group): the eager call sequence with
          separate backward and update.  Returns the same, both modules' layer outputs and the gradient buckets.
  cache   both modules forward over one batch, the way `ModuleSweep.cache_outputs` prepares the next module's inputs.
          Returns both sets of layer outputs.
  host    one step from pinned host buffers (`mrem_recon_step_host`), blocking until the loss is back.
  rem     one step of the per-product objective on one weight matrix (`ReconModule.rem_step`).
  embed   one step of the first module's embedding layers (`EmbeddingStep.step`).

Inputs follow the synthetic workloads of `synth.py`: weights N(0, 0.02^2), hidden states N(0, 1) with a few channels
scaled by 20, valid lengths uniform between a quarter of the sequence length and all of it.
"""
import math

import numpy as np
import torch

from paper_2109_15082_b200 import binding as B
from paper_2109_15082_b200.dist import DataParallelModule
from paper_2109_15082_b200.embedding import EmbeddingStep
from paper_2109_15082_b200.session import MATRICES, ReconModule

VECTORS = tuple(p for p in range(12) if p not in MATRICES)
BATCHES = 4                    # calibration batches a state holds and walks through
HEAD = 64                      # head size of every configuration
_stream = None


def _rate(case):
    """The workloads' learning rate; a tenth of it for 8-bit weights, whose steps are that much smaller; for the gradient
    case the rate near the end of the decay (so that its second pass differentiates at the first one's weights)."""
    if case["kind"] == "grads":
        return 1e-6
    return 1e-5 if case.get("w_bits") == 8 else 1e-4


def _module(name, kind, layers, hidden, seq, batch, w_bits=4, w_grid=0, a_bits=8, lam=0.0):
    return dict(name=name, kind=kind, layers=layers, hidden=hidden, ffn=4 * hidden, seq=seq, batch=batch, w_bits=w_bits,
                w_grid=w_grid, a_bits=a_bits, lam=lam)


def listed():
    return [
        # the benchmark's workload: a BERT-large module of six layers, 4-bit weights
        _module("step_large_w4a8", "step", 6, 1024, 128, 32),
        # reading comprehension: 384 tokens, 2-bit weights on the half-integer grid; the largest step
        _module("step_large_w2a8_s384", "step", 6, 1024, 384, 16, w_bits=2, w_grid=1),
        # a BERT-base module of three layers, teacher forcing half way through its annealing
        _module("step_base_w4a8_mix", "step", 3, 768, 128, 32, lam=0.5),
        # the 4-bit scales refitted from the weights in every step
        _module("step_base_refit", "step", 3, 768, 128, 32, w_grid=3),
        # few short ragged sequences: weights and launches outweigh the tokens
        _module("step_base_w2a8_small", "step", 3, 768, 72, 3, w_bits=2, w_grid=1),
        # the smallest module: launches and latency only
        _module("step_tiny", "step", 1, 128, 32, 4),
        # one rank's share of a data-parallel step on a one-layer module, an odd length, 4-bit activations
        _module("grads_base_w4a4_s200", "grads", 1, 768, 200, 11, a_bits=4),
        # caching the next module's inputs
        _module("cache_base_w4a8", "cache", 3, 768, 128, 32),
        # batches that live in host memory, BERT-base at 256 tokens
        _module("host_base_w4a8_s256", "host", 3, 768, 256, 8),
        # the per-product baseline: the widest matrix of BERT-large on 32 x 128 tokens
        dict(_module("rem_large_w1", "rem", 1, 1024, 128, 32), tensor=B.W1),
        # the first module's embedding layers: BERT-large table, 32 x 128 tokens; and a BERT-base table, few tokens
        dict(name="embed_large", kind="embed", vocab=30522, hidden=1024, seq=128, batch=32, e_bits=4),
        dict(name="embed_base_small", kind="embed", vocab=30522, hidden=768, seq=56, batch=5, e_bits=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "grads", "cache", "host", "rem", "embed"])
    hidden = rng.choice([128, 256, 512, 768, 768, 1024, 1024])
    seq = 8 * _log_int(rng, 2, 48)
    # never more tokens than the largest listed step, nor more scores per head than 2^21 (16 x 384 x 384)
    batch = _log_int(rng, 1, max(1, min(64, 6144 // seq, (1 << 21) // (seq * seq))))
    if kind == "embed":
        return dict(kind="embed", vocab=rng.choice([1000, 21128, 28996, 30522]), hidden=hidden, seq=seq, batch=batch,
                    e_bits=rng.choice([2, 4, 8]))
    layers = 1 if kind in ("rem", "grads") else rng.choice([1, 2, 3, 4] if kind == "cache" else [1, 2, 3, 4, 6])
    w_bits, w_grid = rng.choice([(4, 0), (4, 0), (4, 0), (2, 1), (2, 1), (2, 0), (2, 2), (4, 3)] + [(8, 0)] * (kind != "grads"))
    a_bits = rng.choice([8, 8, 8, 4]) if kind != "cache" else 8
    lam = rng.choice([0.0, 0.0, 0.0, round(rng.uniform(0.1, 0.9), 2)]) if kind in ("step", "host") else 0.0
    case = _module("", kind, layers, hidden, seq, batch, w_bits, w_grid, a_bits, lam)
    del case["name"]
    if kind == "rem":
        case["tensor"] = rng.choice(list(MATRICES))
    return case


# ----------------------------------------------------------------------------- states

class _State:
    """What a program keeps between calls; closes the module's context when it is dropped."""

    def __init__(self, case):
        self.case, self.t, self.m = case, 0, None

    def __del__(self):
        if self.m is not None:
            self.m.close()


def _work_stream():
    """One stream for all states, as a program has: a captured step cannot live on the legacy default stream."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _hidden_states(gen, n, seq, hidden, dtype):
    x = torch.randn(n, seq, hidden, device="cuda", generator=gen)
    outliers = torch.randperm(hidden, device="cuda", generator=gen)[:4]
    x[:, :, outliers] *= 20.0
    return x.to(dtype)


def _new_module(case, gen, rule):
    m = ReconModule(case["layers"], case["hidden"], case["hidden"] // HEAD, case["ffn"], case["seq"], case["batch"],
                    case["w_bits"], case["a_bits"], case["w_grid"], stream=_work_stream())
    # the vectors and the weight steps of all layers in one allocation each (their sizes are multiples of 256 bytes)
    pieces = [(l, p) for l in range(m.L) for p in VECTORS]
    m.vectors = torch.zeros(sum(m.student[l][p].numel() for l, p in pieces), device=m.device)
    off = 0
    for l, p in pieces:
        n = m.student[l][p].numel()
        m.student[l][p] = m.vectors[off:off + n].view_as(m.student[l][p])
        B.mrem_bind_param(m.ctx, B.STUDENT, l, p, m.student[l][p], B.F32)
        off += n
    m.flat_w_steps = torch.ones(sum(s.numel() for ws in m.w_steps for s in ws), device=m.device)
    off = 0
    for l in range(m.L):
        for k in range(len(MATRICES)):
            n = m.w_steps[l][k].numel()
            m.w_steps[l][k] = m.flat_w_steps[off:off + n]
            B.mrem_bind_steps(m.ctx, l, k, m.w_steps[l][k], None)
            off += n
    for l in range(m.L):
        for p in range(12):
            w = m.teacher[l][p]
            if p in MATRICES:
                w.copy_(torch.randn(w.shape, device="cuda", generator=gen) * 0.02)
            else:
                w.copy_(torch.randn(w.shape, device="cuda", generator=gen) * 0.02 + (1.0 if p in (B.LN1_G, B.LN2_G) else 0.0))
    m.init_student_from_teacher()
    m.init_weight_steps(rule)
    return m


def _prepare_module(case, seed):
    s = _State(case)
    kind, batch, seq, hidden = case["kind"], case["batch"], case["seq"], case["hidden"]
    stream = _work_stream()
    with torch.cuda.stream(stream):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        s.m = m = _new_module(case, gen, 1 if case["w_bits"] == 2 else 0)
        s.optim = B.make_optim(lr=_rate(case), step=0, decay_total_steps=100000)
        n = BATCHES * batch
        calib = _hidden_states(gen, n, seq, hidden, m.tdtype)
        lens = torch.randint(max(1, seq // 4), seq + 1, (n,), device="cuda", generator=gen, dtype=torch.int32)
        s.order = torch.randperm(n, device="cuda", generator=gen).to(torch.int32)
        s.calib = calib
        # the batches' valid lengths as rows of whole 16-byte pieces, so that one gather fetches a batch's
        s.lens = torch.zeros(BATCHES, (batch + 3) // 4 * 4, dtype=torch.int32, device="cuda")
        s.lens[:, :batch] = lens[s.order.long()].view(BATCHES, batch)
        s.batch_ids = torch.arange(BATCHES, dtype=torch.int32, device="cuda")
        s.x = torch.empty(batch, seq, hidden, dtype=m.tdtype, device="cuda")
        s.xs = s.x
        s.len = torch.zeros(max(64, s.lens.shape[1]), dtype=torch.int32, device="cuda")
        if case["lam"]:                       # under teacher forcing the student's inputs are its own
            s.calib_s = (calib.float() + 0.05 * torch.randn(calib.shape, device="cuda", generator=gen)).to(m.tdtype)
            s.xs = torch.empty_like(s.x)
        _stage(s)
        m.init_act_steps(s.xs, s.len, batch, seq)
        if kind == "step":
            B.mrem_graph_capture_step(m.ctx, s.x, s.xs, case["lam"], s.len, batch, seq, m.t_out, m.s_out, m.loss, s.optim)
        elif kind == "grads":
            s.dp = DataParallelModule(m)
        elif kind == "host":
            pick = s.order.long().view(BATCHES, batch)
            host = lambda c: [c[pick[t]].cpu().pin_memory() for t in range(BATCHES)]
            s.h_x = host(calib)
            s.h_xs = host(s.calib_s) if case["lam"] else s.h_x
            s.h_len = [s.lens[t, :batch].cpu().pin_memory() for t in range(BATCHES)]
    stream.synchronize()
    return s


def _prepare_rem(case, seed):
    s = _State(case)
    rows, hidden, ffn = case["batch"] * case["seq"], case["hidden"], case["ffn"]
    stream = _work_stream()
    with torch.cuda.stream(stream):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        s.m = m = _new_module(case, gen, 1 if case["w_bits"] == 2 else 0)
        s.optim = B.make_optim(lr=_rate(case), step=0, decay_total_steps=100000)
        x = _hidden_states(gen, case["batch"], case["seq"], hidden, m.tdtype)
        m.init_act_steps(x, None, case["batch"], case["seq"])
        if case["tensor"] == B.W2:            # that product's input is a GELU output
            u = torch.randn(BATCHES * rows, ffn, device="cuda", generator=gen)
            s.a = torch.nn.functional.gelu(u).to(m.tdtype)
        else:
            s.a = _hidden_states(gen, BATCHES, rows, hidden, m.tdtype).view(BATCHES * rows, hidden)
        s.a = s.a.view(BATCHES, rows, -1)
    stream.synchronize()
    return s


def _prepare_embed(case, seed):
    s = _State(case)
    V, H, seq, batch = case["vocab"], case["hidden"], case["seq"], case["batch"]
    stream = _work_stream()
    with torch.cuda.stream(stream):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        randn = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)
        teacher = dict(word=(0.05 * randn(V, H)).cpu().numpy(), pos=(0.02 * randn(512, H)).cpu().numpy(),
                       type=(0.02 * randn(2, H)).cpu().numpy(), ln_g=np.ones(H, np.float32), ln_b=np.zeros(H, np.float32))
        s.emb = EmbeddingStep(teacher, case["e_bits"], batch * seq, stream=stream)
        q = max(1.0, 2.0 ** (case["e_bits"] - 1) - 1)
        s.emb.set_student(None, np.abs(teacher["word"]).max(1) / q)
        s.optim = B.make_optim(lr=_rate(case), step=0, decay_total_steps=100000)
        # word frequencies fall like 1 / rank, as in text
        u = torch.rand(BATCHES, batch, seq, device="cuda", generator=gen)
        s.ids = (torch.exp(u * math.log(V)) - 1.0).to(torch.int32).clamp_(0, V - 1)
        turn = torch.randint(1, seq + 1, (BATCHES, batch, 1), device="cuda", generator=gen)
        s.types = (torch.arange(seq, device="cuda") >= turn).to(torch.int32)      # first and second segment of each pair
    stream.synchronize()
    return s


def prepare(case, seed):
    if case["kind"] == "embed":
        return _prepare_embed(case, seed)
    if case["kind"] == "rem":
        return _prepare_rem(case, seed)
    return _prepare_module(case, seed)


# ----------------------------------------------------------------------------- one pass

def _stage(s):
    """The next batch of the calibration set and its valid lengths into the step's input buffers."""
    c, st = s.case, _work_stream().cuda_stream
    b = s.t % BATCHES
    s.t += 1
    rows = s.order[b * c["batch"]:(b + 1) * c["batch"]]
    row_bytes = c["seq"] * c["hidden"] * s.x.element_size()
    B.mrem_gather_rows(s.calib, rows, c["batch"], row_bytes, s.x, st)
    if s.xs is not s.x:
        B.mrem_gather_rows(s.calib_s, rows, c["batch"], row_bytes, s.xs, st)
    B.mrem_gather_rows(s.lens, s.batch_ids[b:b + 1], 1, s.lens.shape[1] * 4, s.len, st)


def _updated(m, loss):
    out = dict(loss=loss, vectors=m.vectors, w_steps=m.flat_w_steps, a_steps=m.a_steps[:, :, 0], a_off=m.a_off[:, :, 0])
    for l in range(m.L):
        for p in MATRICES:
            out["%s_%d" % (B.PARAM_NAMES[p], l)] = m.student[l][p]
    return out


def run(s):
    c = s.case
    kind = c["kind"]
    with torch.cuda.stream(_work_stream()):
        if kind == "embed":
            b = s.t % BATCHES
            s.t += 1
            e = s.emb
            loss = e.step(s.ids[b], s.types[b], s.optim)
            e_t, e_s = e.outputs(c["batch"], c["seq"])
            return dict(loss=loss, e_teacher=e_t, e_student=e_s, word_step=e.word_step, **e.s)
        m = s.m
        if kind == "rem":
            b = s.t % BATCHES
            s.t += 1
            loss = m.rem_step(0, c["tensor"], s.a[b], s.optim)
            k = MATRICES.index(c["tensor"])
            return dict(loss=loss, w=m.student[0][c["tensor"]], w_steps=m.w_steps[0][k], a_steps=m.a_steps[:, :, 0], a_off=m.a_off[:, :, 0])
        if kind == "host":
            b = s.t % BATCHES
            s.t += 1
            loss = B.mrem_recon_step_host(m.ctx, s.h_x[b], s.h_xs[b], s.h_len[b], c["batch"], c["seq"], c["lam"], s.optim)
            return _updated(m, loss)
        _stage(s)
        if kind == "step":
            B.mrem_graph_launch(m.ctx)
            return _updated(m, m.loss[:1])
        if kind == "grads":
            loss = s.dp.step(s.x, s.xs, s.len, c["batch"], c["batch"], c["seq"], s.optim)
            out = _updated(m, loss)
            out["teacher"], out["student"] = m.t_out, m.s_out
            for l, g in enumerate(s.dp.buckets):
                out["grad_%d" % l] = g
            return out
        m.quantize_weights()
        f_t = m.forward_teacher(s.x, s.len, c["batch"], c["seq"])
        f_s = m.forward_student(s.xs, s.len, c["batch"], c["seq"])
        return dict(teacher=f_t, student=f_s)


# ----------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    kind, H, M = case["kind"], case["hidden"], case["batch"] * case["seq"]
    if kind == "embed":
        V = case["vocab"]
        rows = min(V, M)                                  # table rows the batch gathers, at most
        params = (V + 512 + 2 + 2) * H + V
        # latent values and both moments read and written; the teacher's rows read; both outputs written
        return {"bytes": 24.0 * params + 4.0 * H * rows + 2.0 * 2 * M * H + 8.0 * M, "flops": 30.0 * params + 60.0 * M * H}
    F = case["ffn"]
    per_layer = 4 * H * H + 2 * H * F
    if kind == "rem":
        n_out, n_in = {B.WQKV: (3 * H, H), B.WO: (H, H), B.W1: (F, H), B.W2: (H, F)}[case["tensor"]]
        n = n_out * n_in
        return {"bytes": 2.0 * n + 24.0 * n + 2.0 * M * n_in, "flops": 4 * 2.0 * M * n}
    L = case["layers"]
    n = L * per_layer
    products, attention = 2.0 * M * n, 4.0 * M * case["seq"] * H * L
    inputs = 2.0 * M * H * (2 if case["lam"] else 1)
    outputs = 2 * 2.0 * M * H * L
    if kind == "cache":                                   # teacher matrices and student codes read, layer outputs written
        return {"bytes": 2.0 * n + 1.0 * n + inputs + outputs, "flops": 2 * products + 2 * attention}
    # teacher read; latent weights and both moments read and written; two forward and two backward products
    grads = 4.0 * n if kind == "grads" else 0.0
    returned = outputs if kind != "host" else 0.0
    return {"bytes": 2.0 * n + 24.0 * n + inputs + returned + grads, "flops": 4 * products + 4 * attention}


def tolerance(case):
    """About four times what the same state shows when every LayerNorm parameter is one float32 ulp off.  A last-bit
    difference flips bf16 roundings and integer codes, which spread through the layers above, and Adam's first steps move
    a weight by the whole learning rate (half a percent of its size) in the direction of its gradient's sign."""
    kind = case["kind"]
    if kind == "embed":                       # seen: 6e-5, single bf16 outputs by one spacing
        return {"rel": 3e-4, "max": 5e-2}
    if kind == "rem":                         # seen: 1e-3; a flipped sign is 2e-2 of a weight
        return {"rel": 4e-3, "max": 0.16}
    if kind == "cache":                       # seen: 3e-3 after three layers, 1.2e-2 after six
        return {"rel": 1.2e-2 if case["layers"] <= 3 else 3e-2, "max": 0.9}
    if kind == "grads":                       # seen: 1e-2 of a gradient bucket, single bias gradients 0.4
        return {"rel": 3e-2, "max": 0.99}
    # seen: 1.1e-3 of the parameters (4e-3 with 4-bit activations); the loss of a few hundred tokens 9e-3
    few = case["a_bits"] == 4 or case["batch"] * case["seq"] < 1024
    return {"rel": 2e-2 if few else 4e-3, "max": 0.5 if few else 0.16}
