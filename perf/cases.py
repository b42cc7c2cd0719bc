"""What a user of this framework has it do, as timed cases: Algorithm 1 and Algorithm 2 of Flora through the public calls.

A case is one optimizer-side pass over the weight matrices of a program: the gradients are on the GPU, the weights and
the sketches too, and the pass makes the calls that compress the gradients, keep the sketches and update the weights.
Two manners of calling are covered, as the package offers them: the single-matrix calls (`calls` = "single": an
optimizer that loops over its parameters) and the weight sets driven by the host classes of the two algorithms (`calls`
= "set").  `mode` says which algorithm a pass belongs to:

    accumulate           Algorithm 1: one cycle of `tau` compressions, then the weights take the mean (a new seed per cycle)
    momentum             Algorithm 2: one step, M <- beta M + (1-beta) G A^T, then W <- W - lr M A
    resample             Algorithm 2 where the projection is resampled: one step that starts M, and one that carries it
                         over to a new projection (transfer), each followed by the weight update
    accumulate+momentum  Algorithm 1 feeding Algorithm 2: a cycle, the transfer of its sketch into M, the weight update

`shapes` names the matrices: "512x512", a list "130x70,1000x515", "gpt2:768x12" (twelve transformer blocks of width 768:
fused attention input, attention output and the two feed-forward matrices) or "gated:1024,2816,24" (24 encoder and 24
decoder blocks with gated feed-forward).  Gradients are N(0, 1e-3) (N(0, 1e-2) in fp32), with 1 % of the entries
multiplied by 100 where `outliers` is set; weights are N(0, 0.02^2).  The step size moves a weight by some per cent of
its size, so that every pass shows in it.
"""
from __future__ import annotations

import torch

from paper_2402_03293_b200 import binding as fb
from paper_2402_03293_b200 import hostlogic
from paper_2402_03293_b200 import workloads as wl

BETA = 0.9
KAPPA = 200             # Algorithm 2 resamples every KAPPA steps in the modes that keep M over many passes


def listed():
    return [
        # the smallest use: one small fp32 matrix, low rank, a cycle of four micro-steps; all latency and launches
        {"name": "f32_512x512_r8_cycle", "shapes": "512x512", "dtype": "f32", "r": 8, "mode": "accumulate", "tau": 4, "calls": "single"},
        # an ordinary fp32 layer with compressed momentum (fp32 is what a program has that does not train in bf16)
        {"name": "f32_1024x4096_r64_momentum", "shapes": "1024x4096", "dtype": "f32", "r": 64, "mode": "momentum", "tau": 1, "calls": "single"},
        # a whole small model in fp32, gradient accumulation
        {"name": "f32_gpt2_small_set_r32_cycle", "shapes": "gpt2:768x12", "dtype": "f32", "r": 32, "mode": "accumulate", "tau": 4, "calls": "set"},
        # a small bf16 matrix: the lowest latency the bf16 calls have, with the projection resampled
        {"name": "bf16_256x384_r32_resample", "shapes": "256x384", "dtype": "bf16", "r": 32, "mode": "resample", "tau": 1, "calls": "single"},
        # odd sizes: rows that start at no aligned address
        {"name": "bf16_1000x4097_r64_momentum", "shapes": "1000x4097", "dtype": "bf16", "r": 64, "mode": "momentum", "tau": 1, "calls": "single"},
        # a ragged set: small, tall, wide and odd matrices together, accumulation feeding momentum
        {"name": "bf16_ragged_set_r32_both", "shapes": "130x70,1000x515,257x4097,128x64,4000x129,768x768,10x768,50x3072", "dtype": "bf16", "r": 32,
         "mode": "accumulate+momentum", "tau": 4, "calls": "set"},
        # an optimizer that loops over a model's parameters with the single-matrix calls
        {"name": "bf16_gpt2_small_loop_r16_momentum", "shapes": "gpt2:768x12", "dtype": "bf16", "r": 16, "mode": "momentum", "tau": 1, "calls": "single"},
        # a small model as a set, gradient accumulation; every micro-step's gradients are new tensors
        {"name": "bf16_gpt2_small_set_r32_cycle", "shapes": "gpt2:768x12", "dtype": "bf16", "r": 32, "mode": "accumulate", "tau": 8, "calls": "set",
         "rebind": True},
        # a large set of medium matrices with compressed momentum
        {"name": "bf16_t5_large_set_r64_momentum", "shapes": "gated:1024,2816,24", "dtype": "bf16", "r": 64, "mode": "momentum", "tau": 1, "calls": "set"},
        # one large feed-forward matrix at a low rank and at the highest
        {"name": "bf16_4096x11008_r8_momentum", "shapes": "4096x11008", "dtype": "bf16", "r": 8, "mode": "momentum", "tau": 1, "calls": "single"},
        {"name": "bf16_4096x11008_r256_resample", "shapes": "4096x11008", "dtype": "bf16", "r": 256, "mode": "resample", "tau": 1, "calls": "single"},
        # the largest: a 1.5 billion element model at the highest rank, 16 micro-steps feeding compressed momentum
        {"name": "bf16_gpt2_xl_set_r256_both", "shapes": "gpt2:1600x48", "dtype": "bf16", "r": 256, "mode": "accumulate+momentum", "tau": 16,
         "calls": "set", "outliers": True},
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def _size(rng, lo, hi):
    """A size spread over the logarithm of lo..hi: any whole number, or one rounded to 8, 64 or 128."""
    to = rng.choice((1, 1, 8, 64, 128))
    return int(min(hi, max(lo, to, round(_log(rng, lo, hi) / to) * to)))


def draw(rng):
    while True:
        dtype = rng.choice(("bf16", "bf16", "f32"))
        r = int(round(_log(rng, 4, 256))) if rng.random() < 0.5 else rng.choice((8, 16, 32, 64, 128, 256))
        mode = rng.choice(("accumulate", "momentum", "resample", "accumulate+momentum"))
        kind = rng.choice(("matrix", "matrix", "loop", "blocks", "gated", "ragged"))
        calls = "single" if kind in ("matrix", "loop") else "set"
        if kind == "matrix":
            shapes = "%dx%d" % (_size(rng, 64, 8192), _size(rng, 64, 16384))
        elif kind == "gated":
            shapes = "gated:%d,%d,%d" % (64 * rng.randint(4, 16), 64 * rng.randint(8, 44), int(round(_log(rng, 1, 24))))
        elif kind == "ragged":
            shapes = ",".join("%dx%d" % (_size(rng, 16, 4096), _size(rng, 64, 8192)) for _ in range(rng.randint(2, 12)))
        else:
            shapes = "gpt2:%dx%d" % (8 * rng.randint(32, 200), int(round(_log(rng, 1, 12 if kind == "loop" else 48))))
        if mode == "accumulate+momentum" and calls == "single":
            mode = "accumulate"
        if mode == "resample" and calls == "set":
            mode = "momentum"
        tau = int(round(_log(rng, 2, 16))) if mode.startswith("accumulate") else 1
        case = {"shapes": shapes, "dtype": dtype, "r": r, "mode": mode, "tau": tau, "calls": calls}
        if mode == "accumulate" and calls == "set" and rng.random() < 0.5:
            case["rebind"] = True
        if rng.random() < 0.2:
            case["outliers"] = True
        cost = _cost(case)
        # fp32 contractions and odd sizes have no matrix instructions of full rate to rely on: they get an eighth of the largest case's work
        if cost <= _cost(listed()[-1]) * (0.125 if dtype == "f32" or kind in ("ragged", "matrix") else 1.0):
            return case


def _shapes(text):
    if text.startswith("gpt2:"):
        d, blocks = (int(v) for v in text[5:].split("x"))
        return [(d, 3 * d), (d, d), (d, 4 * d), (4 * d, d)] * blocks
    if text.startswith("gated:"):
        d, ff, blocks = (int(v) for v in text[6:].split(","))
        ffn = [(d, ff), (d, ff), (ff, d)]
        return ([(d, d)] * 4 + ffn) * blocks + ([(d, d)] * 8 + ffn) * blocks
    return [tuple(int(v) for v in s.split("x")) for s in text.split(",")]


def _flat(shapes, dtype):
    """Matrices as views of one buffer (as a program keeps the parameters of a model), each at a 256-byte boundary."""
    pad = 256 // torch.empty(0, dtype=dtype).element_size()
    offsets, total = [], 0
    for n, m in shapes:
        offsets.append(total)
        total += -(-n * m // pad) * pad
    buf = torch.zeros(total, dtype=dtype, device="cuda")
    return buf, [buf[o:o + n * m].view(n, m) for o, (n, m) in zip(offsets, shapes)]


def _fill(mats, std, gen, outliers=False):
    for x in mats:
        v = torch.randn(x.shape, generator=gen, device="cuda") * std
        if outliers:
            v = torch.where(torch.rand(x.shape, generator=gen, device="cuda") < 0.01, v * 100.0, v)
        x.copy_(v)


class State:
    pass


def prepare(case, seed):
    s = State()
    shapes = _shapes(case["shapes"])
    dtype, r = wl.torch_dtype(case["dtype"]), case["r"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s.case, s.r, s.tau, s.base = case, r, case["tau"], seed
    # gradients: two sets where micro-steps bring new tensors or the matrices are few, one otherwise (a program's fixed .grad buffers)
    sets = 2 if case.get("rebind") or case["calls"] == "single" else 1
    var = 1e-2 if case["dtype"] == "f32" else 1e-3
    s.G = []
    for _ in range(sets):
        _, g = _flat(shapes, dtype)
        _fill(g, var ** 0.5, gen, bool(case.get("outliers")))
        s.G.append(g)
    s.W_all, s.W = _flat(shapes, dtype)
    _fill(s.W, 0.02, gen)
    sketches = [(n, r) for n, _ in shapes]
    s.C_all, s.C = _flat(sketches, torch.float32)
    s.M_all, s.M = (_flat(sketches, torch.float32) if case["mode"] == "accumulate+momentum" else (None, None))
    s.lr = {"accumulate": 1e-2, "momentum": 3e-2, "resample": 3e-3, "accumulate+momentum": 3e-2}[case["mode"]]
    if case.get("outliers"):
        s.lr *= 0.1
    s.epoch = 0
    if case["calls"] == "set":
        count = len(shapes)
        if case["mode"] == "accumulate":
            s.set = fb.FloraSet(s.G[0], s.W, s.C)
            s.algo = hostlogic.AccumulationCycle(s.set, count, s.tau, base_seed=seed)
        elif case["mode"] == "momentum":
            s.set = fb.FloraSet(s.G[0], s.W, s.C)
            s.algo = hostlogic.MomentumState(s.set, count, BETA, KAPPA, base_seed=seed)
        else:
            s.acc, s.mom = fb.FloraSet(s.G[0], None, s.C), fb.FloraSet(None, s.W, s.M)
            s.algo = hostlogic.AccumulatedMomentum(s.acc, s.mom, count, s.tau, BETA, KAPPA, base_seed=seed)
    return s


def run(s):
    case, mode = s.case, s.case["mode"]
    if case["calls"] == "set":
        if mode == "momentum":
            s.algo.step(s.lr)
        else:
            for k in range(s.tau):
                if case.get("rebind"):
                    s.set.rebind_gradients(s.G[k % 2])
                s.algo.accumulate()
            s.algo.apply(s.lr)
    else:
        for i, (W, C) in enumerate(zip(s.W, s.C)):
            if mode == "accumulate":
                seed = fb.flora_derive_seed(s.base, i, s.epoch)
                fb.flora_momentum_step(s.G[0][i], C, 0.0, seed)                     # the first compression of a cycle overwrites C
                for k in range(1, s.tau):
                    fb.flora_compress_accumulate(s.G[k % 2][i], C, seed, s.r)
                fb.flora_decompress_apply(W, C, seed, s.lr, 1.0 / s.tau)
            elif mode == "momentum":
                seed = fb.flora_derive_seed(s.base, i, 0)
                fb.flora_momentum_step(s.G[s.epoch % 2][i], C, BETA, seed)
                fb.flora_decompress_apply(W, C, seed, s.lr, 1.0)
            else:
                old, new = fb.flora_derive_seed(s.base, i, s.epoch), fb.flora_derive_seed(s.base, i, s.epoch + 1)
                fb.flora_momentum_step(s.G[0][i], C, 0.0, old)                      # M starts anew
                fb.flora_decompress_apply(W, C, old, s.lr, 1.0)
                fb.flora_momentum_step_resampled(s.G[1][i], C, BETA, old, new)
                fb.flora_decompress_apply(W, C, new, s.lr, 1.0)
        s.epoch += 1
    out = {"W": s.W_all, "C": s.C_all}
    if s.M_all is not None:
        out["M"] = s.M_all
    return out


def work(case):
    """Each pass reads every gradient once per compression, the weights once, and writes the weights and the state once per
    operation that changes them; a projection costs no bytes (it is a function of its seed)."""
    shapes, r, tau, mode = _shapes(case["shapes"]), case["r"], case["tau"], case["mode"]
    eb = 4 if case["dtype"] == "f32" else 2
    elements = sum(n * m for n, m in shapes)
    state = sum(n * r * 4 for n, _ in shapes)
    product = 2 * elements * r
    transfer = sum(2 * r * r * m + 2 * n * r * r for n, m in shapes)
    update = 2 * elements * eb + state                       # W read and written, the sketch read
    if mode == "accumulate":
        return {"bytes": tau * elements * eb + (2 * tau - 1) * state + update, "flops": (tau + 1) * product}
    if mode == "momentum":
        return {"bytes": elements * eb + 2 * state + update, "flops": 2 * product}
    if mode == "resample":
        return {"bytes": 2 * elements * eb + state + 2 * state + 2 * update, "flops": 4 * product + transfer}
    return {"bytes": tau * elements * eb + (2 * tau - 1) * state + 3 * state + update, "flops": (tau + 1) * product + transfer}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def tolerance(case):
    # fp32: sums of up to m + r terms in fp32.  bf16: the weights are stored in bf16 (half a spacing is 2^-9 of the value),
    # and the update is computed from a sketch read with 8 to 11 significant bits.
    return {"rel": 1e-5, "max": 2e-4} if case["dtype"] == "f32" else {"rel": 5e-3, "max": 5e-2}
