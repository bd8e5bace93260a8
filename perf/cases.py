"""The work that users of this library have it do, as cases that can be timed and compared.

Every case goes through the public binding (`meq.MeqMuon`, `meq.ns_cv_trajectory`,
`meq.row_col_stats_noalloc`). A case is a dict of plain values:

  call       "step": one optimizer step (`step`); "split": the same step as
             `step_prepare` and `step_apply`, as a training loop that overlaps work on
             the parameters calls it; "inspect": what an analysis or a checkpoint reads
             back after a step (momentum, NS output, update, statistics); "replay": the CV
             trajectory of the NS iterates; "stats": the allocation-free statistics.
  layers, hidden, ffn, vocab
             a Llama-style model: its hidden weights, and with vocab > 0 every other
             parameter too (embedding, LM head, norm weights). layers = 0: `shapes`.
  shapes     hidden weights as text, "rowsxcols,rowsxcols".
  imbalance  row / column imbalance of the gradients: "row_col" (each matrix one of
             the two), "both", "heavy" (Student-t scales on both sides). With both, one
             side of each matrix is the more uneven one: where the two are alike, rounding
             decides Eq. (11), and two correct results differ.
  rule       "meqmuon" or "muon"; nesterov: the look-ahead momentum;
  ns         "fp16" (default) or "bf16" Newton-Schulz operands.
  rows, cols, steps
             the matrix of "replay" and "stats", and the replay's length.

The parameters of a case lie in one flat buffer (each at a 64-element boundary), as a
trainer with flat parameter buffers keeps them; the step updates them in place and they
are its output. The momentum holds the history of one earlier step taken at learning
rate 0 (which leaves the parameters as they are), so that it takes part in the result.
"""
import math

import numpy as np
import torch

from paper_2609_35701_gb300 import meq

LR, MU, WD, EPS, RHO = 0.02, 0.95, 0.1, 1e-7, 0.2
NS_A, NS_B, NS_C, NS_STEPS = 3.4445, -4.7750, 2.0315, 5
TIE_ATOL = 1e-6

HIDDEN, REMAINING_2D, VECTOR = 0, 1, 2

# flops of one pass above which no 64-bit result is computed (it would take over 20 s)
EXACT_FLOPS = 1.6e13


def _model(call="step", layers=0, hidden=0, ffn=0, vocab=0, shapes="", imbalance="row_col", rule="meqmuon",
           nesterov=False, ns="fp16", name=None):
    c = {"call": call, "layers": layers, "hidden": hidden, "ffn": ffn, "vocab": vocab, "shapes": shapes,
         "imbalance": imbalance, "rule": rule, "nesterov": nesterov, "ns": ns}
    return c if name is None else dict(c, name=name)


def _matrix(call, rows, cols, steps=0, name=None):
    c = {"call": call, "rows": rows, "cols": cols, "steps": steps}
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # One small weight: a unit test, a toy model, a bias-free probe. Latency and launches count.
        _model(shapes="256x256", imbalance="both", name="one 256x256"),
        # A small network whose widths are no multiples of anything: seven shapes, all ragged.
        _model(shapes="300x177,177x300,1000x64,64x500,333x77,130x70,200x333", imbalance="both", name="ragged small set"),
        # Every parameter of a 60M model: embeddings and norm weights weigh more than the hidden weights.
        _model(layers=8, hidden=512, ffn=1376, vocab=32000, name="60m whole model"),
        # The hidden weights of a 60M model under the comparison rule and in bf16, as an ablation runs them.
        _model(layers=8, hidden=512, ffn=1376, rule="muon", ns="bf16", name="60m hidden muon bf16"),
        # The hidden weights of a 130M model: 84 matrices, the ordinary pretraining step.
        _model(layers=12, hidden=768, ffn=2048, name="130m hidden"),
        # Every parameter of a 130M model, the step in two calls.
        _model(call="split", layers=12, hidden=768, ffn=2048, vocab=32000, name="130m whole model split"),
        # The hidden weights of a 350M model with look-ahead momentum.
        _model(layers=24, hidden=1024, ffn=2736, nesterov=True, name="350m hidden nesterov"),
        # Four layers of a 1B-class model: an odd FFN width, heavy-tailed gradients.
        _model(layers=4, hidden=2048, ffn=5461, imbalance="heavy", name="1b four layers"),
        # Two layers of a 7B-class model: the largest matrices, bound by the tensor cores and by power.
        _model(layers=2, hidden=4096, ffn=11008, name="7b two layers"),
        # What an analysis of one 350M layer reads back after a step, and what a checkpoint saves.
        _model(call="inspect", layers=1, hidden=1024, ffn=2736, name="inspect a 350m layer"),
        # The CV trajectory of one 350M FFN matrix over 20 iterations.
        _matrix("replay", 1024, 2736, steps=20, name="replay 1024x2736"),
        # The statistics of one 7B-class FFN matrix without allocation.
        _matrix("stats", 4096, 11008, name="stats 4096x11008"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "step", "split", "split", "inspect", "replay", "stats"])
    if call in ("replay", "stats"):
        rows, cols = _log_uniform(rng, 48, 4096), _log_uniform(rng, 48, 4096)
        if rng.random() < 0.5:  # widths of real layers: a multiple of 16 and a tall or wide partner
            rows = 16 * max(3, rows // 16)
            cols = min(11008, int(rows * rng.choice([1, 2, 2.67, 4])))
            if rng.random() < 0.5:
                rows, cols = cols, rows
        return _matrix(call, rows, cols, steps=rng.randint(4, 24) if call == "replay" else 0)
    opts = {
        "call": call,
        "imbalance": rng.choice(["row_col", "row_col", "both", "heavy"]),
        "rule": "meqmuon",
        "nesterov": rng.random() < 0.3,
        "ns": rng.choice(["fp16", "fp16", "fp16", "bf16"]),
    }
    if rng.random() < 0.3 and call != "inspect":  # a small network: a handful of matrices of any shape
        n = rng.randint(1, 12)
        text = ",".join("%dx%d" % (_log_uniform(rng, 24, 1400), _log_uniform(rng, 24, 1400)) for _ in range(n))
        return _model(shapes=text, **opts)
    hidden = _log_uniform(rng, 96, 4096 if call != "inspect" else 1536)
    if rng.random() < 0.75:
        hidden = 64 * max(2, hidden // 64)
    ffn = int(hidden * rng.uniform(2.0, 4.0))
    if rng.random() < 0.6:
        ffn = 16 * max(1, ffn // 16)
    ffn = min(ffn, 11008)
    most = max(_flops(c) for c in listed() if "layers" in c)
    layers = 1 if call == "inspect" else rng.randint(1, 24)
    while layers > 1 and _flops(_model(layers=layers, hidden=hidden, ffn=ffn)) > most:
        layers -= 1
    vocab = rng.choice([0, 0, rng.randint(1000, 50000)]) if call != "inspect" and hidden <= 1024 else 0
    if vocab == 0 and call != "inspect" and rng.random() < 0.2:
        opts["rule"] = "muon"
    return _model(layers=layers, hidden=hidden, ffn=ffn, vocab=vocab, **opts)


# ------------------------------------------------------------------- inputs
def _entries(case):
    """(rows, cols, kind) of every parameter, in order."""
    if case["layers"] == 0:
        return [tuple(int(x) for x in t.split("x")) + (HIDDEN,) for t in case["shapes"].split(",")]
    d, f, v, out = case["hidden"], case["ffn"], case["vocab"], []
    for _ in range(case["layers"]):
        out += [(d, d, HIDDEN)] * 4 + [(f, d, HIDDEN)] * 2 + [(d, f, HIDDEN)]
    if v:
        out += [(v, d, REMAINING_2D)] * 2 + [(1, d, VECTOR)] * (2 * case["layers"] + 1)
    return out


def _views(flat, entries):
    out, at = [], 0
    for m, n, _ in entries:
        out.append(flat[at:at + m * n].view(m, n))
        at += -(-m * n // 64) * 64
    return out


def _flat_size(entries):
    return sum(-(-m * n // 64) * 64 for m, n, _ in entries)


def _generator(device, seed):
    g = torch.Generator(device=device)
    g.manual_seed(1000003 * int(seed) + 17)
    return g


def _scale(n, heavy, mild, g, device):
    if heavy:  # |t_3|
        z = torch.randn(n, generator=g, device=device)
        v = torch.randn(3, n, generator=g, device=device).square().sum(0)
        s = (z / torch.sqrt(v / 3.0)).abs()
    else:  # 0.1 .. 10
        s = torch.exp(torch.rand(n, generator=g, device=device) * math.log(100.0) + math.log(0.1))
    return s.pow(0.3) if mild else s


def _inputs(case, seed, device):
    """Flat parameters, and the flat gradients of an earlier step and of this one."""
    entries, g = _entries(case), _generator(device, seed)
    size = _flat_size(entries)
    flats = [torch.zeros(size, device=device) for _ in range(3)]
    views = [_views(f, entries) for f in flats]
    for i, (m, n, _) in enumerate(entries):
        views[0][i].normal_(0.0, 0.02, generator=g)
        heavy, one = case["imbalance"] == "heavy", case["imbalance"] == "row_col"
        rs = _scale(m, heavy, i % 2 == 1, g, device) if not one or i % 2 == 0 else None
        cs = _scale(n, heavy, i % 2 == 0, g, device) if not one or i % 2 == 1 else None
        for v in views[1:]:
            v[i].normal_(0.0, 0.01, generator=g)
            if rs is not None:
                v[i].mul_(rs[:, None])
            if cs is not None:
                v[i].mul_(cs[None, :])
    return entries, flats, views


def _input_matrix(case, seed, device):
    """The matrix of "replay" (a gradient-like one) and of "stats" (an NS-output-like one)."""
    m, n, g = case["rows"], case["cols"], _generator(device, seed)
    x = torch.randn(m, n, generator=g, device=device)
    if case["call"] == "replay":
        return x.mul_(0.01).mul_(_scale(m, False, False, g, device)[:, None])
    x.mul_(1.0 / math.sqrt(max(m, n)))
    return x.mul_(torch.exp(0.3 * torch.randn(m, generator=g, device=device))[:, None]) \
            .mul_(torch.exp(0.1 * torch.randn(n, generator=g, device=device))[None, :])


def prepare(case, seed):
    device = torch.device("cuda")
    if case["call"] in ("replay", "stats"):
        x = _input_matrix(case, seed, device)
        state = {"case": case, "x": x}
        if case["call"] == "stats":
            state["out"] = (torch.empty(case["rows"], device=device), torch.empty(case["cols"], device=device),
                            torch.empty(2, dtype=torch.float64, device=device),
                            torch.empty(1, dtype=torch.int32, device=device))
        return state
    entries, flats, views = _inputs(case, seed, device)
    opt = meq.MeqMuon([(m, n) for m, n, _ in entries], kinds=[k for _, _, k in entries],
                      nesterov=int(case["nesterov"]), ns_fp16_mask=0xFFFFFFFF if case["ns"] == "fp16" else 0,
                      update_rule=meq.RULE_MUON if case["rule"] == "muon" else meq.RULE_MEQMUON)
    opt.step(views[0], views[1], lr=0.0, momentum=MU, weight_decay=0.0, eps=EPS)
    if case["call"] == "inspect":
        opt.step(views[0], views[2], lr=LR, momentum=MU, weight_decay=WD, eps=EPS)
    return {"case": case, "opt": opt, "flat": flats[0], "params": views[0], "grads": views[2]}


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "step":
        state["opt"].step(state["params"], state["grads"], lr=LR, momentum=MU, weight_decay=WD, eps=EPS)
        return state["flat"]
    if call == "split":
        state["opt"].step_prepare(state["grads"], lr=LR, momentum=MU, weight_decay=WD, eps=EPS)
        state["opt"].step_apply(state["params"])
        return state["flat"]
    if call == "inspect":
        opt, out = state["opt"], []
        for i in range(len(opt.shapes)):
            out.append({"momentum": opt.read_momentum(i), "ns_output": opt.read_ns_output(i),
                        "update": opt.read_update(i), "stats": opt.read_stats(i)})
        return out
    if call == "replay":
        return meq.ns_cv_trajectory(state["x"], steps=case["steps"], eps=EPS)
    status = meq.row_col_stats_noalloc(state["x"], *state["out"], eps=EPS)
    if status != meq.MEQ_OK:
        raise RuntimeError("row_col_stats_noalloc: status %d" % status)
    return state["out"]


# --------------------------------------------------------------------- work
def _ns_flops(m, n, steps):
    """Eq. (5) on the smaller side: the symmetric halves of X X^T and A A, and P X."""
    s, l = min(m, n), max(m, n)
    return steps * (float(s) * (s + 1) * l + float(s) * s * (s + 1) + 2.0 * s * s * l)


def _flops(case):
    if case["call"] == "inspect":
        return 0.0
    if case["call"] == "replay":
        return _ns_flops(case["rows"], case["cols"], case["steps"])
    if case["call"] == "stats":
        return 0.0
    return sum(_ns_flops(m, n, NS_STEPS) for m, n, k in _entries(case) if k == HIDDEN)


def work(case):
    if case["call"] in ("replay", "stats"):
        return {"bytes": 4.0 * case["rows"] * case["cols"] + 4.0 * (case["rows"] + case["cols"]), "flops": _flops(case)}
    numel = float(sum(m * n for m, n, _ in _entries(case)))
    if case["call"] == "inspect":  # momentum and U (2 bytes) read, three fp32 matrices delivered
        return {"bytes": 18.0 * numel, "flops": 0.0}
    # gradients read, momentum and parameters read and written
    return {"bytes": 20.0 * numel, "flops": _flops(case)}


def tolerance(case):
    """About four times what the results differ by from `exact` over the declared ranges."""
    if case["call"] == "stats":
        return {"rel": 2e-6, "differ": 0.0}
    if case["call"] == "replay":
        return {"rel": 1.8e-2}
    bf16, heavy = case["ns"] == "bf16", case["imbalance"] == "heavy"
    if case["call"] == "inspect":
        return {"rel": 2.8e-2 if bf16 else 1.2e-2, "max": 0.6 if heavy else 0.3 if bf16 else 0.12, "differ": 0.0}
    # the parameters: the update (relative error as above) is a fifth of them
    return {"rel": 6e-3 if bf16 else 2.4e-3, "max": 0.3 if heavy else 0.1 if bf16 else 0.06}


# -------------------------------------------------------------------- 64 bits
def _ns_iterates(H, steps):
    """X_0 .. X_steps of Eq. (5), taken on the smaller side."""
    tall = H.shape[0] > H.shape[1]
    X = H.T.contiguous() if tall else H
    X = X / torch.linalg.norm(X)
    for k in range(steps + 1):
        yield X.T if tall else X
        if k < steps:
            A = X @ X.T
            X = NS_A * X + (NS_B * A + NS_C * (A @ A)) @ X


def _rms(X):
    return X.square().mean(1).sqrt(), X.square().mean(0).sqrt()


def _cv(v):
    v = v[v > EPS]
    return float((v - v.mean()).square().mean().sqrt() / v.mean()) if v.numel() else 0.0


def _inv(v):
    return torch.where(v > EPS, 1.0 / v, torch.zeros_like(v))


def _update(case, kind, B, G):
    """The normalised update of one parameter and, for a hidden weight, U and its statistics."""
    if kind == VECTOR:
        rms = B.square().mean().sqrt()
        return B * _inv(rms), None
    if kind == REMAINING_2D:
        N = B * _inv(_rms(B)[0])[:, None]
        return N * _inv(_rms(N)[1])[None, :], None
    for U in _ns_iterates(G + MU * B if case["nesterov"] else B, NS_STEPS):
        pass
    r, c = _rms(U)
    gr, gc = _cv(r), _cv(c)
    if case["rule"] == "muon":
        return math.sqrt(max(U.shape)) * U, (U, r, c, gr, gc, 4)
    row = gr >= gc - TIE_ATOL
    return (U * _inv(r)[:, None] if row else U * _inv(c)[None, :]), (U, r, c, gr, gc, 0 if row else 1)


def exact(case, seed):
    device = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["call"] in ("replay", "stats"):
        if 3 * _flops(case) > EXACT_FLOPS:
            return None
        X = _input_matrix(case, seed, device).double()
        if case["call"] == "stats":
            r, c = _rms(X)
            gr, gc = _cv(r), _cv(c)
            return (r, c, torch.tensor([gr, gc], dtype=torch.float64),
                    torch.tensor([0 if gr >= gc - TIE_ATOL else 1], dtype=torch.int32))
        stats = [_rms(x) for x in _ns_iterates(X, case["steps"])]
        return np.array([_cv(r) for r, _ in stats]), np.array([_cv(c) for _, c in stats])
    if 2 * _flops(case) > EXACT_FLOPS:
        return None
    entries, flats, views = _inputs(case, seed, device)
    W = flats[0].double()
    out, Ws = [], _views(W, entries)
    for i, (_, _, kind) in enumerate(entries):
        G = views[2][i].double()
        B = MU * views[1][i].double() + G
        Ut, hidden = _update(case, kind, B, G)
        if case["call"] == "inspect":
            U, r, c, gr, gc, d = hidden
            out.append({"momentum": B, "ns_output": U, "update": Ut,
                        "stats": {"r": r, "c": c, "gamma_r": gr, "gamma_c": gc, "direction": d}})
        else:
            Ws[i].copy_((1.0 - LR * WD) * Ws[i] - RHO * LR * Ut)
    return out if case["call"] == "inspect" else W
