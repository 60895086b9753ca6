"""The workloads by which this library's speed is measured.

Each case is one call (or one training step) of the kind a user's program
makes: a whole beam dedispersed, a chunk pushed into a stream, a batch of
uneven beams, the adjoint, the detection loss, one step of learning the
channel weights.  Sizes are those of the library's own setups (tiny,
Apertif-like, LOFAR-like and the uneven batch) and generic ones between them.

``prepare`` makes what such a program holds before the call (plan, device
buffers, seeded data with dispersed pulses), ``run`` makes the call, ``work``
counts the bytes and operations the call cannot do without, and ``exact``
states the result in 64-bit torch arithmetic without the library's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1601_01165_gb300 import autograd, binding

# Observing bands: lowest frequency and bandwidth in MHz, sampling time in s,
# DM step (the Apertif- and LOFAR-like surveys of the library's setups).
BANDS = {"apertif": (1420.0, 300.0, 50e-6, 0.25), "lofar": (138.0, 6.25, 5e-6, 0.01),
         "tiny": (1400.0, 64.0, 1e-3, 1.0)}
BOX = 8  # boxcar length of the detection loss


def listed():
    return [
        # the smallest call: a quick look at a short stretch of a narrow band
        {"name": "tiny_f32", "op": "forward", "dtype": "f32", "band": "tiny", "C": 64, "n_dm": 32, "n_out": 1024,
         "padded": True},
        # a second of one Apertif-like beam, float samples: the headline
        {"name": "apertif_f32", "op": "forward", "dtype": "f32", "band": "apertif", "C": 1024, "n_dm": 2048,
         "n_out": 20000, "padded": True},
        # the same beam as the telescope delivers it, 8-bit samples
        {"name": "apertif_u8", "op": "forward", "dtype": "u8", "band": "apertif", "C": 1024, "n_dm": 2048,
         "n_out": 20000, "padded": True},
        # a second of one LOFAR-like beam: few channels, steep delays, a large output
        {"name": "lofar_f32", "op": "forward", "dtype": "f32", "band": "lofar", "C": 32, "n_dm": 4096,
         "n_out": 200000, "padded": True},
        # a narrow DM search around a known source
        {"name": "narrow_f32", "op": "forward", "dtype": "f32", "band": "apertif", "C": 1024, "n_dm": 64,
         "n_out": 20000, "padded": True},
        # sizes as they come, and an input tensor without any row padding
        {"name": "ragged_f32", "op": "forward", "dtype": "f32", "band": "apertif", "C": 509, "n_dm": 301,
         "n_out": 7777, "padded": False},
        # a low-frequency beam of the uneven batch, 8-bit samples
        {"name": "lofar256_u8", "op": "forward", "dtype": "u8", "band": "lofar", "C": 256, "n_dm": 1024,
         "n_out": 50000, "padded": True},
        # real-time operation: the next second of a beam pushed into its stream
        {"name": "stream_u8", "op": "stream", "dtype": "u8", "band": "apertif", "C": 1024, "n_dm": 2048,
         "n_out": 20000},
        # several beams of different sizes and sample types in one call
        {"name": "batch_6", "op": "batch", "beams": 6, "batch_seed": 5},
        # gradients of a dedispersed block with respect to its input and the channel weights
        {"name": "adjoint_f32", "op": "adjoint", "band": "apertif", "C": 1024, "n_dm": 2048, "n_out": 20000},
        # the detection loss of a dedispersed block, and its gradient
        {"name": "snr_loss", "op": "loss", "n_dm": 2048, "n_out": 20000},
        # one step of learning the channel weights: weighted forward, loss, backward
        {"name": "train_step", "op": "train", "band": "apertif", "C": 1024, "n_dm": 2048, "n_out": 20000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forward"] * 6 + ["stream", "adjoint", "loss", "train"])
    band = rng.choice(["apertif", "apertif", "lofar"])
    while True:
        C, n_dm = _log(rng, 32, 1024), _log(rng, 16, 4096)
        n_out = _log(rng, 1000, 20000 if op in ("adjoint", "train") else 200000)
        if C * n_dm * n_out <= 25e9 and n_dm * n_out <= 500e6:
            break
    case = {"op": op, "band": band, "C": C, "n_dm": n_dm, "n_out": n_out}
    if op == "forward":
        case |= {"dtype": rng.choice(["f32", "u8"]), "padded": rng.random() < 0.75}
    elif op == "stream":
        case["dtype"] = rng.choice(["f32", "u8"])
    elif op == "loss":
        return {"op": op, "n_dm": n_dm, "n_out": n_out}
    elif op in ("adjoint", "train"):
        case["band"] = "apertif"
    return case


# ------------------------------------------------------------------ inputs
def _geometry(case):
    """Plan arguments: channels, lowest frequency, channel width, sampling time, first DM, DM step, trials, samples."""
    f_low, bw, t_samp, step = BANDS[case["band"]]
    return case["C"], f_low, bw / case["C"], t_samp, 0.0, step, case["n_dm"], case["n_out"]


def _beams(case):
    """The beams of a batch: sizes and sample types as uneven as a survey's, fixed by the case."""
    rng = np.random.default_rng(case["batch_seed"])
    beams = []
    for k in range(case["beams"]):
        beams.append({"op": "forward", "dtype": "f32" if k % 2 == 0 else "u8",
                      "band": "lofar" if k % 3 == 2 else "apertif", "C": (32, 256, 1024)[k % 3],
                      "n_dm": int(rng.choice([256, 1024])), "n_out": int(rng.integers(10000, 40001))})
    return beams


def _noise(shape, dtype, gen):
    if dtype == "f32":
        return torch.randn(shape, generator=gen, device="cuda")
    x = torch.randn(shape, generator=gen, device="cuda")
    return x.mul_(16.0).add_(128.0).round_().clamp_(0, 255).to(torch.uint8)


def _beam_input(case, seed, plan, padded=True):
    """Receiver noise with two dispersed pulses, in rows as the plan likes them or exactly n_in long."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = plan.alloc_input(plan.padded_in_stride() if padded else plan.n_in)
    x[:, :plan.n_in] = _noise((plan.channels, plan.n_in), plan.dtype, gen)
    rng = np.random.default_rng(seed)
    delays = plan.delays()
    rows = torch.arange(plan.channels, device="cuda")
    for _ in range(2):
        i, t = int(rng.integers(plan.n_dm)), int(rng.integers(0, plan.n_out - 3))
        at = torch.from_numpy(delays[i].astype(np.int64) + t).cuda()
        for k in range(3):
            if plan.dtype == "u8":
                v = x[rows, at + k].to(torch.int32) + 40
                x[rows, at + k] = v.clamp_(0, 255).to(torch.uint8)
            else:
                x[rows, at + k] += 5.0
    return x


def _weights(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    return torch.rand(case["C"], generator=gen, device="cuda") + 0.5


def _block(case, seed):
    """A dedispersed block: noise of a channel sum's size and one burst."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((case["n_dm"], case["n_out"]), generator=gen, device="cuda").mul_(32.0)
    rng = np.random.default_rng(seed)
    i, t = int(rng.integers(case["n_dm"])), int(rng.integers(0, case["n_out"] - BOX))
    x[i, t:t + 3] += 320.0
    return x


def prepare(case, seed):
    op = case["op"]
    state = {"case": case}
    if op == "loss":
        state["x"] = _block(case, seed)
        return state
    if op == "batch":
        plans = [binding.Plan(*_geometry(b), dtype=b["dtype"]) for b in _beams(case)]
        state["ins"] = [_beam_input(b, seed + k, p) for k, (b, p) in enumerate(zip(_beams(case), plans))]
        state["outs"] = [torch.empty((p.n_dm, p.n_out), dtype=p.out_dtype, device="cuda") for p in plans]
        state["batch"] = binding.Batch(plans)
        return state
    plan = binding.Plan(*_geometry(case), dtype=case.get("dtype", "f32"))
    state["plan"] = plan
    if op == "stream":
        state["stream"] = binding.Stream(plan, case["n_out"])
        gen = torch.Generator(device="cuda").manual_seed(seed)
        state["chunk"] = _noise((case["C"], case["n_out"]), plan.dtype, gen)
        # the seconds already received: the tail of the stream is full of samples
        for _ in range(-(-plan.max_delay // case["n_out"])):
            state["stream"].push(state["chunk"])
        state["out"] = torch.empty((plan.n_dm, case["n_out"]), dtype=plan.out_dtype, device="cuda")
        return state
    state["x"] = _beam_input(case, seed, plan, case.get("padded", True))
    if op == "forward":
        state["out"] = torch.empty((plan.n_dm, plan.n_out), dtype=plan.out_dtype, device="cuda")
    elif op == "adjoint":
        gen = torch.Generator(device="cuda").manual_seed(seed + 2)
        state["w"] = _weights(case, seed)
        state["g"] = torch.randn((plan.n_dm, plan.n_out), generator=gen, device="cuda")
        state["grad_in"] = torch.empty((plan.channels, plan.n_in), device="cuda")
    elif op == "train":
        state["w"] = _weights(case, seed).requires_grad_()
    return state


def run(state):
    op = state["case"]["op"]
    if op == "forward":
        return state["plan"].forward(state["x"], out=state["out"])
    if op == "stream":
        return state["stream"].push(state["chunk"], out=state["out"])[0]
    if op == "batch":
        return state["batch"].run(state["ins"], state["outs"])
    if op == "adjoint":
        gi, gw = state["plan"].adjoint(state["g"], w=state["w"], x=state["x"], grad_in=True, grad_w=True,
                                       grad_in_out=state["grad_in"])
        return {"grad_in": gi, "grad_w": gw}
    if op == "loss":
        raw, g = binding.boxcar_snr(state["x"], grad=True)
        # the result's four doubles (loss, S/N, mean, deviation), then its sample, row and flag
        return {"stats": raw[:32].view(torch.float64), "best_t": raw[32:40].view(torch.int64),
                "best_row": raw[40:].view(torch.int32), "grad": g}
    w = state["w"]
    w.grad = None
    out = autograd.dedisperse(state["x"], w, state["plan"])
    loss = autograd.boxcar_snr_loss(out)
    loss.backward()
    return {"loss": loss.detach(), "out": out.detach(), "grad_w": w.grad}


# -------------------------------------------------------------------- work
def _delays(case):
    """Eq. 1 of Sclocco et al. in double, rounded half up: [n_dm][C] int64."""
    C, f_low, bw, t_samp, dm0, step, n_dm, _ = _geometry(case)
    f = f_low + np.arange(C) * bw
    dm = dm0 + np.arange(n_dm) * step
    return np.floor((4150.0 * dm)[:, None] * (1.0 / (f * f) - 1.0 / (f[-1] * f[-1]))[None, :] / t_samp + 0.5).astype(np.int64)


def _max_delay(case):
    return int(_delays(case)[-1, 0])


def _beam_work(case):
    elem = 1 if case["dtype"] == "u8" else 4
    n_in = case["n_out"] + _max_delay(case)
    return {"bytes": elem * case["C"] * n_in + 4 * case["n_dm"] * case["n_out"],
            "flops": case["C"] * case["n_dm"] * case["n_out"]}


def work(case):
    op = case["op"]
    if op == "loss":  # read the block, write its gradient; boxcar sums, moments, maximum
        n = case["n_dm"] * case["n_out"]
        return {"bytes": 8 * n, "flops": 12 * n}
    if op == "batch":
        w = [_beam_work(b) for b in _beams(case)]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    if op == "forward":
        return _beam_work(case)
    C, n_dm, n_out, tail = case["C"], case["n_dm"], case["n_out"], _max_delay(case)
    if op == "stream":  # read the chunk and the kept tail, write the output and the next tail
        elem = 1 if case["dtype"] == "u8" else 4
        return {"bytes": elem * C * (n_out + 2 * tail) + 4 * n_dm * n_out, "flops": C * n_dm * n_out}
    n_in = n_out + tail
    if op == "adjoint":  # read grad_out and the input, write both gradients
        return {"bytes": 4 * (n_dm * n_out + 2 * C * n_in), "flops": C * n_dm * n_out + 3 * C * n_in}
    # train: the input, the output block, and its gradient read back through the channels
    return {"bytes": 4 * (C * n_in + 2 * n_dm * n_out), "flops": 4 * C * n_dm * n_out}


# ------------------------------------------------------------------- exact
def _forward64(x, delays, n_out, w=None):
    """sum_c w[c] x[c][t + delays[i][c]] in double, a block of trials at a time."""
    n_dm, C = delays.shape
    out = torch.zeros((n_dm, n_out), dtype=torch.float64, device="cuda")
    step = max(1, int(2e8 // n_out))
    for i0 in range(0, n_dm, step):
        block = out[i0:i0 + step]
        for c in range(C):
            rows = x[c].double().unfold(0, n_out, 1)[delays[i0:i0 + step, c]]
            block.add_(rows, alpha=1.0 if w is None else float(w[c]))
    return out


def _loss64(x):
    """Best boxcar S/N of a block and the gradient of minus it: (loss, S/N, mean, sd, t, row, gradient of that row)."""
    nb = x.shape[1] - BOX + 1
    best = None
    for i0 in range(0, x.shape[0], 512):
        b = x[i0:i0 + 512].double().unfold(1, BOX, 1).sum(2)
        mean, sd = b.mean(1, keepdim=True), b.std(1, correction=0, keepdim=True)
        z = (b - mean) / sd
        k = int(z.argmax())
        if best is None or float(z.flatten()[k]) > best[1]:
            r, t = divmod(k, nb)
            best = (-float(z[r, t]), float(z[r, t]), float(mean[r]), float(sd[r]), t, i0 + r, z[r].clone())
    loss, snr, mean, sd, t, row, z = best
    db = -(1.0 / nb + snr * z / nb) / sd
    db[t] += 1.0 / sd
    g = torch.zeros(x.shape[1], dtype=torch.float64, device="cuda")
    for k in range(BOX):
        g[k:k + nb] -= db
    return loss, snr, mean, sd, t, row, g


def exact(case, seed):
    op = case["op"]
    if op == "batch":  # integer beams are compared sample for sample
        s = prepare(case, seed)
        return [_forward64(x, torch.from_numpy(_delays(b)).cuda(), b["n_out"]) if b["dtype"] == "f32" else None
                for b, x in zip(_beams(case), s["ins"])]
    if case.get("dtype") == "u8":
        return None
    s = prepare(case, seed)
    if op == "loss":
        loss, snr, mean, sd, t, row, g = _loss64(s["x"])
        grad = torch.zeros_like(s["x"], dtype=torch.float64)
        grad[row] = g
        return {"stats": torch.tensor([loss, snr, mean, sd], dtype=torch.float64), "best_t": None, "best_row": None,
                "grad": grad}
    delays = torch.from_numpy(_delays(case)).cuda()
    n_out = case["n_out"]
    if op == "forward":
        return _forward64(s["x"], delays, n_out)
    if op == "stream":  # the same chunk over and over, the oldest samples from the last of them that fit
        tail = int(delays.max())
        chunk = s["chunk"]
        x = chunk.repeat(1, -(-tail // n_out) + 1)[:, -(tail + n_out):]
        return _forward64(x, delays, n_out)
    if op == "adjoint":
        tail = int(delays.max())
        n_in = n_out + tail
        pad = torch.nn.functional.pad(s["g"].double(), (tail, tail))
        flat, width = pad.flatten(), pad.shape[1]
        first = torch.arange(case["n_dm"], device="cuda") * width + tail
        gi = torch.empty((case["C"], n_in), dtype=torch.float64, device="cuda")
        gw = torch.empty(case["C"], dtype=torch.float64, device="cuda")
        spans = flat.unfold(0, n_in, 1)
        for c in range(case["C"]):
            g = spans[first - delays[:, c]].sum(0)
            gw[c] = (g * s["x"][c, :n_in].double()).sum()
            gi[c] = g * float(s["w"][c])
        return {"grad_in": gi, "grad_w": gw}
    w = s["w"].detach()
    out = _forward64(s["x"], delays, n_out, w.tolist())
    loss, _, _, _, _, row, g = _loss64(out)
    gw = torch.stack([(g * s["x"][c].double()[int(delays[row, c]):][:n_out]).sum() for c in range(case["C"])])
    return {"loss": torch.tensor(loss, dtype=torch.float64), "out": out, "grad_w": gw}
