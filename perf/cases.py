"""The work that a user of this library has it do, as cases that can be timed: stacked-LSTM and H-LSTM inference
through the public binding, over the sizes of the paper's two models (Section 5.1: a language model of two stacked
layers of width 1500 or 200; Section 5.2: a speech model of five bidirectional layers of width 800; Table 1 and Table 4:
their pruned and H-LSTM forms, measured at batch 16) and over ragged sizes between them.

A case is a dict: ``cell`` "lstm" or "hlstm", ``layers``, ``bidir``, ``in_dim``, ``hidden``, ``gate_hidden`` (H-LSTM only,
else 0), ``T`` and ``B`` of the call, ``max_T`` the handle was made for, ``dtype`` "bf16" (bf16 weights, fp32 state) or
"fp32", ``density`` of the Bernoulli keep-masks (1.0: dense), ``state``: the call continues from carried h0, c0;
``host``: the call takes and fills pinned host buffers.
"""
import math

import torch

import paper_1901_10997_b200 as lib


def _case(name, layers, in_dim, hidden, T, B, *, bidir=False, cell="lstm", gate_hidden=0, max_T=0, dtype="bf16", density=1.0,
          state=False, host=False):
    c = {"cell": cell, "layers": layers, "bidir": bidir, "in_dim": in_dim, "hidden": hidden, "gate_hidden": gate_hidden,
         "T": T, "B": B, "max_T": max(max_T, T), "dtype": dtype, "density": density, "state": state, "host": host}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # language model, one sentence scored while its author waits: the paper's baseline shape at batch 1
        _case("lm_single", 2, 1500, 1500, 35, 1),
        # the same from and to host memory, as a program without a GPU pipeline of its own calls it
        _case("lm_single_host", 2, 1500, 1500, 35, 1, host=True),
        # generation: one word per call, the state carried from call to call; the smallest call there is
        _case("lm_step", 2, 1500, 1500, 1, 1, max_T=35, state=True),
        # the language model at the batch it is usually evaluated with
        _case("lm_batch20", 2, 1500, 1500, 35, 20),
        # scoring a corpus offline: as many sentences at once as there are
        _case("lm_bulk", 2, 1500, 1500, 35, 100),
        # a small model of odd widths for a few requests at a time
        _case("lm_narrow", 2, 301, 517, 23, 3, state=True),
        # the small language model in full fp32
        _case("fp32_batch20", 2, 200, 200, 35, 20, dtype="fp32"),
        # the pruned language model, for one sentence and at the paper's batch
        _case("pruned_single", 2, 1500, 1500, 35, 1, density=0.1),
        _case("pruned_batch16", 2, 1500, 1500, 35, 16, density=0.1),
        # the speech model on one utterance and at the paper's batch
        _case("speech_single", 5, 1312, 800, 400, 1, bidir=True),
        _case("speech_batch16", 5, 1312, 800, 400, 16, bidir=True),
        # the paper's compressed language model (Table 1 step (c)): an H-LSTM layer of 1200 with gate layers of 320,
        # sentences of length 70 at batch 16
        _case("hlstm_batch16", 1, 1500, 1200, 70, 16, cell="hlstm", gate_hidden=320),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["lm", "lm", "lm", "pruned", "speech", "fp32", "hlstm_lm", "hlstm_speech"])
    state = rng.random() < 0.5
    if kind == "lm":
        hidden = rng.randint(500, 1500)
        in_dim = hidden if rng.random() < 0.5 else rng.randint(300, 1500)
        B = log_int(1, 100)
        T = min(log_int(1, 70), 3500 // B)
        return _case("", 2, in_dim, hidden, T, B, max_T=rng.choice([T, 70]), state=state, host=rng.random() < 0.25)
    if kind == "pruned":
        hidden = rng.randint(800, 1500)
        return _case("", 2, hidden, hidden, log_int(2, 70), log_int(1, 16), density=rng.choice([0.05, 0.1]), state=state)
    if kind == "speech":
        return _case("", rng.randint(3, 5), rng.randint(161, 1312), rng.randint(400, 800), rng.randint(50, 400), log_int(1, 16), bidir=True)
    if kind == "fp32":
        hidden = rng.randint(64, 256)
        return _case("", 2, hidden, hidden, log_int(4, 70), log_int(1, 32), dtype="fp32", state=state)
    if kind == "hlstm_lm":
        return _case("", 1, rng.randint(300, 1500), rng.randint(800, 1500), log_int(1, 70), log_int(1, 16), cell="hlstm",
                     gate_hidden=rng.randint(300, 1500), state=state)
    return _case("", 3, rng.randint(161, 1312), rng.randint(400, 800), rng.randint(50, 150), log_int(1, 8), bidir=True, cell="hlstm",
                 gate_hidden=rng.randint(200, 800))


def _in_l(c, layer):
    return c["in_dim"] if layer == 0 else (2 if c["bidir"] else 1) * c["hidden"]


def prepare(case, seed):
    c = case
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    dirs = 2 if c["bidir"] else 1
    H, Hh = c["hidden"], c["gate_hidden"]

    def uniform(a, *shape):
        return (torch.rand(shape, generator=g, device=dev) * 2 - 1) * a

    def keep(*shape):
        return (torch.rand(shape, generator=g, device=dev) < c["density"]).to(torch.uint8)

    weights = []
    for layer in range(c["layers"]):
        for _ in range(dirs):
            n = _in_l(c, layer)
            if c["cell"] == "hlstm":
                a, a_out = 1 / math.sqrt(H), 1.5 / math.sqrt(Hh)
                weights.append({"ux": uniform(a, 4 * Hh, n), "uh": uniform(a, 4 * Hh, H), "a": uniform(a, 4 * Hh),
                                "w": uniform(a_out, 4 * H, Hh), "b": uniform(a_out, 4 * H)})
                continue
            a = 1 / math.sqrt(H * c["density"])
            w = {"wx": uniform(a, 4 * H, n), "wh": uniform(a, 4 * H, H), "b": uniform(a, 4 * H)}
            if c["density"] < 1:
                w["mask_x"], w["mask_h"] = keep(4 * H, n), keep(4 * H, H)
            weights.append(w)
    shape = {"layers": c["layers"], "in_dim": c["in_dim"], "hidden": H, "bidir": c["bidir"], "dtype": c["dtype"],
             "max_T": c["max_T"], "max_B": c["B"]}
    if c["cell"] == "hlstm":
        model = lib.HLSTM(weights, gate_hidden=Hh, **shape)
    else:
        model = lib.LSTM(weights, exec_mode="csr" if c["density"] < 1 else "dense", **shape)

    x = torch.randn((c["T"], c["B"], c["in_dim"]), generator=g, device=dev)
    h0 = c0 = None
    if c["state"]:
        h0 = uniform(0.9, c["layers"] * dirs, c["B"], H)
        c0 = 0.5 * torch.randn((c["layers"] * dirs, c["B"], H), generator=g, device=dev)
    s = {"model": model, "x": x, "h0": h0, "c0": c0, "out": None}
    if c["host"]:
        # pinned buffers that such a program keeps from call to call
        s["x"], s["h0"], s["c0"] = (t if t is None else t.cpu().pin_memory() for t in (x, h0, c0))
        s["out"] = (torch.empty((c["T"], c["B"], dirs * H), pin_memory=True),
                    torch.empty((c["layers"] * dirs, c["B"], H), pin_memory=True),
                    torch.empty((c["layers"] * dirs, c["B"], H), pin_memory=True))
    return s


def run(state):
    s = state
    if s["out"] is not None:
        y, hT, cT = s["out"]
        return s["model"].forward_host(s["x"], s["h0"], s["c0"], y=y, hT=hT, cT=cT)
    return s["model"].forward(s["x"], s["h0"], s["c0"])


def work(case):
    c = case
    dirs = 2 if c["bidir"] else 1
    H, Hh, M = c["hidden"], c["gate_hidden"], c["T"] * c["B"]
    entries = biases = 0.0
    for layer in range(c["layers"]):
        n = _in_l(c, layer)
        if c["cell"] == "hlstm":
            entries += dirs * (4 * Hh * (n + H) + 4 * H * Hh)
            biases += dirs * 4 * (Hh + H)
        else:
            entries += dirs * 4 * H * (n + H) * c["density"]
            biases += dirs * 4 * H
    # a surviving weight of a pruned matrix comes with its 16-bit column
    weight = (4 if c["dtype"] == "fp32" else 2) + (2 if c["density"] < 1 else 0)
    states = c["layers"] * dirs * c["B"] * H * (4 if c["state"] else 2)
    return {"bytes": entries * weight + 4 * (biases + M * (c["in_dim"] + dirs * H) + states), "flops": 2.0 * M * entries}


def tolerance(case):
    # Activations enter the bf16 products as two terms of 8 bits each (relative error 2^-17 an element) and sums are fp32;
    # fp32 storage sums in fp64 and rounds h, c and the stored projection to fp32.  Against a float64 evaluation of the same
    # weights the outputs of these cases are off by at most 4e-6 (bf16) and 4.3e-8 (fp32) in the 2-norm, and by 5e-5 and
    # 2e-7 in the worst element; four times that.
    return {"rel": 2e-7, "max": 8e-7} if case["dtype"] == "fp32" else {"rel": 1.6e-5, "max": 2e-4}
