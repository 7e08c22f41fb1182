"""The work a training run has the delayed rotated-Adam step do, as cases that can be timed and compared.

A case is a set of weight matrices with its options; one pass is `calls` calls of
`BasisRotation.step`, from gradients on the device to updated weights on the device.  Two kinds:

* a whole refresh period (`calls` = `freq`): the steady steps and the one refresh of every basis that
  fall due between two refreshes, in the proportion in which a training run meets them;
* a single step between two refreshes (`calls` = 1, no refresh due): the latency of one call.

`power` cases are the stand-alone Power() entry point (`br_power_static`), for callers that own all of
the device's memory.

The state a pass starts from is a run some way in: the delay ring is full, the factors have seen
several gradients and, for single steps, the bases have been refreshed once.  Gradients cycle through a
pool of different ones whose ranks add up to more than the largest dimension, so that the factors keep
full rank, as they do in training (one gradient over and over would leave them rank-deficient).
"""
import math

import torch

import paper_2602_03515_b200 as br
from workloads.configs import LayerSpec

GEOMS = {"none": br.BR_GEOM_NONE, "uni": br.BR_GEOM_UNILATERAL, "bi": br.BR_GEOM_BILATERAL}
SOURCES = {"1st": br.BR_SRC_FIRST, "2nd": br.BR_SRC_SECOND}
NEVER = 1 << 30        # a refresh period that no pass reaches
BASE = {"kind": "step", "block": "", "d": 0, "ffn": 0, "blocks": 1, "vocab": 0, "shapes": "", "geom": "bi", "source": "2nd",
        "grad": "bf16", "values": "lowrank", "noise": 0.1, "rank": 16, "prec": "bf16", "tau": 4, "freq": 10, "calls": 10,
        "decay": 0.0, "clip": 0.0, "pool": 6}


def listed():
    def case(name, **kw):
        return dict(BASE, name=name, **kw)
    return [
        # the smallest set there is, one 64x32 fp32 matrix (toy problems, tests, a single head): the latency of one call
        case("f32 64x32 call", shapes="64x32", grad="f32", values="normal", noise=0.01, prec="f32", tau=2, freq=NEVER, calls=1),
        # the same matrix through a whole refresh period of five calls
        case("f32 64x32 period", shapes="64x32", grad="f32", values="normal", noise=0.01, prec="f32", tau=2, freq=5, calls=5),
        # odd and ragged shapes that no tile divides, in full fp32 (layers the tensor-core path does not take)
        case("f32 ragged period", shapes="37x53,130x130,333x257,96x515", grad="f32", values="normal", noise=0.05, prec="f32", tau=1),
        # the smallest decoder the paper trains (emb 384, one pipeline stage of 4 blocks): small matrices, many of them
        case("decoder d384 x4 period", block="fused", d=384, ffn=1536, blocks=4),
        # one GPT-style block at d = 1024, both sides rotated, factor EMAs of the gradient
        case("block d1024 bi period", block="fused", d=1024, ffn=4096),
        # the same block rotated on the smaller side only, bases from the momentum
        case("block d1024 uni 1st period", block="fused", d=1024, ffn=4096, geom="uni", source="1st", tau=8),
        # the same block with global-norm clipping and weight decay, one step between refreshes
        case("block d1024 clip call", block="fused", d=1024, ffn=4096, freq=NEVER, calls=1, clip=1.0, decay=0.1),
        # a LLaMA-style block at d = 2048 with its embedding, heavy-tailed gradients, long delay
        case("decoder d2048 period", block="gated", d=2048, ffn=5632, vocab=32000, values="student", noise=1e-3, tau=16, freq=20, calls=20),
        # the ~3B layer set's block with its embedding over its refresh period of 50 steps: the headline, per block
        case("decoder d2560 period", block="gated", d=2560, ffn=6912, vocab=32000, noise=0.05, rank=32, freq=50, calls=50, pool=4),
        # four such blocks and the embedding, one steady step: the largest grouped launches
        case("decoder d2560 x4 call", block="gated", d=2560, ffn=6912, blocks=4, vocab=32000, noise=0.05, rank=32, freq=NEVER, calls=1, pool=4),
        # parameters that are not rotated (embeddings, plain Adam), through the delay ring
        case("plain 32000x2560 call", shapes="32000x2560", geom="none", freq=NEVER, calls=1, pool=2),
        # stand-alone Power() within the fixed scratch
        dict(name="power k384", kind="power", k=384, noise=0.1, rank=16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["f32", "block", "block", "block", "plain", "power"])
    if kind == "power":
        return {"kind": "power", "k": int(_log(rng, 16, 513)), "noise": round(rng.uniform(0.05, 0.5), 3), "rank": rng.randint(2, 16)}
    period = rng.random() < 0.6
    freq = rng.choice([5, 10, 20]) if period else NEVER
    c = dict(BASE, freq=freq, calls=freq if period else 1, tau=rng.choice([0, 1, 2, 4, 8]),
             decay=rng.choice([0.0, 0.1]), clip=rng.choice([0.0, 0.0, 1.0]))
    if kind == "plain":
        m, n = int(_log(rng, 16, 32000)), int(_log(rng, 16, 2560))
        return dict(c, shapes="%dx%d" % (m, n), geom="none", grad=rng.choice(["bf16", "f32"]), freq=NEVER, calls=1, pool=2)
    c.update(geom=rng.choice(["bi", "bi", "uni"]), source=rng.choice(["2nd", "2nd", "1st"]), noise=round(rng.uniform(0.05, 0.5), 3))
    if kind == "f32":
        # (a bilateral layer whose basis comes from the momentum is short of rank on its larger side: its period ends with
        # completed bases, which say little about the arithmetic; square enough matrices avoid that)
        if c["geom"] == "bi":
            c["source"] = "2nd"
        shapes = []
        for _ in range(rng.randint(1, 4)):
            m = int(_log(rng, 16, 400))
            shapes.append("%dx%d" % (m, max(16, min(640, int(m * _log(rng, 0.34, 3.0))))))
        return dict(c, shapes=",".join(shapes), grad=rng.choice(["f32", "bf16"]), values="normal", prec="f32")
    d = 8 * int(_log(rng, 16, 321))                 # 128 .. 2560, multiples of 8
    gated = rng.random() < 0.5
    if c["geom"] == "bi":
        c["source"] = "2nd"
    return dict(c, block="gated" if gated else "fused", d=d, ffn=8 * int(d * rng.uniform(2.5, 4.0 if d <= 2048 else 2.7) / 8),
                blocks=rng.randint(1, 4) if d <= 768 else 1, vocab=rng.choice([0, 0, 8 * int(_log(rng, 500, 4000))]),
                values=rng.choice(["lowrank", "student", "normal"]))


def _shapes(case):
    """[(m, n, geometry)] of the case's weight matrices."""
    if case["shapes"]:
        return [tuple(int(v) for v in s.split("x")) + (case["geom"],) for s in case["shapes"].split(",")]
    d, f = case["d"], case["ffn"]
    one = [(d, 3 * d), (d, d), (d, f), (f, d)] if case["block"] == "fused" else [(d, d)] * 4 + [(d, f)] * 2 + [(f, d)]
    out = [s + (case["geom"],) for _ in range(case["blocks"]) for s in one]
    if case["vocab"]:
        out.append((case["vocab"], d, "uni"))       # the embedding is rotated on the model dimension only
    return out


def _rotated(m, n, geom):
    """Orders of the bases of a matrix: (left or 0, right or 0)."""
    if geom == "bi":
        return m, n
    return (0, 0) if geom == "none" else (m, 0) if m <= n else (0, n)


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)

    def randn(*shape):
        return torch.randn(*shape, device=dev, generator=gen)

    if case["kind"] == "power":
        k = case["k"]
        A = randn(k, case["rank"])
        G = A @ randn(case["rank"], 4 * k) + case["noise"] * randn(k, 4 * k)
        Q = torch.linalg.qr(randn(k, k))[0].contiguous()
        return {"kind": "power", "k": k, "F": (G @ G.T / (4 * k)).contiguous(), "Q": Q,
                "flag": torch.zeros(1, dtype=torch.int32, device=dev)}
    shapes = _shapes(case)
    specs = [LayerSpec("w%d" % i, m, n, GEOMS[g], SOURCES[case["source"]], case["tau"]) for i, (m, n, g) in enumerate(shapes)]
    weights = [0.02 * randn(m, n) for m, n, _ in shapes]
    dtype = torch.bfloat16 if case["grad"] == "bf16" else torch.float32
    pool = [[None] * len(shapes) for _ in range(case["pool"])]
    for i, (m, n, _) in enumerate(shapes):
        # a persistent low-rank signal under fresh noise, independent entries, or heavy tails
        signal = randn(m, case["rank"]) @ randn(case["rank"], n) if case["values"] == "lowrank" else None
        for p in range(case["pool"]):
            g = case["noise"] * randn(m, n)
            if case["values"] == "lowrank":
                g += signal
            elif case["values"] == "student":       # Student t with three degrees of freedom
                chi = randn(m, n).square_()
                chi += randn(m, n).square_()
                chi += randn(m, n).square_()
                g *= (chi / 3).rsqrt_()
            pool[p][i] = g.to(dtype)
    opt = br.BasisRotation(specs, weights, grad_dtype=case["grad"], lr=1e-3, weight_decay=case["decay"], freq=case["freq"],
                           clip_norm=case["clip"], gemm_prec=br.BR_GEMM_FP32 if case["prec"] == "f32" else br.BR_GEMM_BF16)
    state = {"kind": "step", "opt": opt, "weights": weights, "pool": pool, "calls": case["calls"], "at": 0}
    # fill the ring; then half a period (the refresh falls into the middle of the first pass), or several
    # updates and one refresh of every basis
    period = case["freq"] != NEVER
    _steps(state, case["tau"] + (case["freq"] // 2 if period else case["pool"]))
    if not period and any(g != "none" for _, _, g in shapes):
        opt.refresh_basis()
    return state


def _steps(state, calls):
    opt, pool, at = state["opt"], state["pool"], state["at"]
    for _ in range(calls):
        opt.step(pool[at % len(pool)])
        at += 1
    state["at"] = at


def run(state):
    if state["kind"] == "power":
        br.br_power_static(torch.cuda.current_stream().cuda_stream, state["F"].data_ptr(), state["Q"].data_ptr(), state["k"],
                           state["flag"].data_ptr())
        return [state["Q"], state["flag"]]
    _steps(state, state["calls"])
    return state["weights"]


def work(case):
    """Per call: each gradient in (through the ring when there is a delay: stored once and read once more), every
    piece of state in and out once, each basis in; the factor products on one triangle, the rotation of the
    gradient and the rotation of the update back.  Per refresh: F Q and a Gram-Schmidt of k columns, factor and
    basis in and basis out, and the momentum carried from the old basis to the new one."""
    if case["kind"] == "power":
        k = case["k"]
        return {"bytes": 12.0 * k * k, "flops": 4.0 * k ** 3}
    g = 2 if case["grad"] == "bf16" else 4
    step_b = step_f = fresh_b = fresh_f = 0.0
    for m, n, geom in _shapes(case):
        step_b += m * n * (24 + g * (3 if case["tau"] else 1))
        for k in _rotated(m, n, geom):
            if not k:
                continue
            second = case["source"] == "2nd"
            step_f += m * n * k * (5.0 if second else 4.0)
            step_b += k * k * (12.0 if second else 4.0)
            other = m * n // k
            fresh_f += 2.0 * k ** 3 + (2.0 * k ** 3 if second else 4.0 * k * k * other) + 4.0 * m * n * k
            fresh_b += (8.0 + (4.0 if second else 0.0)) * k * k + 8.0 * m * n
    fresh = 1 if case["freq"] != NEVER else 0
    return {"bytes": case["calls"] * step_b + fresh * fresh_b, "flops": case["calls"] * step_f + fresh * fresh_f}


def tolerance(case):
    """About four times what a change in the order of the sums moves the outputs by (measured)."""
    if case["kind"] == "power" or case["prec"] == "f32":
        return {"rel": 1e-5}                        # fp32 sums, and fp64 ones rounded to fp32: 1e-7 measured
    if case["geom"] == "none":
        return {"rel": 1e-6}                        # element-wise fp32
    if case["values"] == "lowrank" and case["d"] > 20000 * case["noise"]:
        # a strong signal over weak noise: the trailing basis vectors come out of a cancellation, and factor products summed
        # in chunks of one k-block instead of four move the weights by 1.2e-3 (largest entry 0.055 of the root mean square)
        return {"rel": 5e-3, "max": 0.25}
    return {"rel": 5e-4, "max": 3e-2}               # the same change: at most 1.3e-4 and 8.6e-3 over sixty drawn cases
