"""The calls by which this library is measured: what programs that use it have it do, at the sizes they do it.

A case names one `op` and its sizes; side lists are written as text ("1,2,3,4").
  step    one masked sub-step of one scale at inference (hmar_attn_scale_step)
  sweep   one attention layer of a sampler: every scale of a schedule, several sub-steps each, keys and values of the
          previous and the current scale adjacent in one ring (hmar_attn_scale_step_strided)
  fwd     the training forward alone, as evaluation runs it (hmar_attn_fwd)
  train   forward and backward of one attention layer (hmar_attn_fwd, hmar_attn_bwd), or, with layout "packed", on the
          projections' own layouts (hmar_attn_fwd_packed, hmar_attn_bwd_packed)
  recon   the sampler's steps next to the attention: per scale the running reconstruction brought down to the scale's
          resolution, then the scale's selected tokens looked up, enlarged and added (hmar_recon_downsample,
          hmar_recon_accumulate); without `sample` the additions alone, which is the decoding of given token maps
"""
import math

import torch

import paper_2506_04421_b200 as hmar

SIDES_256 = "1,2,3,4,5,6,8,10,13,16"
SIDES_512 = "1,2,3,4,6,9,13,18,24,32"
SIDES_1024 = "1,2,3,4,5,7,9,12,16,21,27,36,48,64"
D = 64
SCALE = 0.125
WINDOWS = {"markov": hmar.HMAR_WINDOW_MARKOV, "causal": hmar.HMAR_WINDOW_CAUSAL}


def _sides(case):
    return [int(s) for s in case["sides"].split(",")]


def listed():
    return [
        # one image, a coarse scale: a call's own latency is all there is; a sampler makes hundreds of these per image
        {"name": "step_coarse_b1", "op": "step", "B": 1, "H": 16, "prev": 2, "cur": 3, "lse": False},
        # a middle scale of the 512 x 512 schedule at a serving batch: a short window, bound by memory
        {"name": "step_mid_b64", "op": "step", "B": 64, "H": 24, "prev": 13, "cur": 18, "lse": False},
        # a whole layer of sampling at the paper's inference batch, four sub-steps per scale: from the launch-bound
        # scales to the last, which holds most of the arithmetic
        {"name": "sweep_512_b16", "op": "sweep", "B": 16, "H": 24, "sides": SIDES_512, "sub_steps": 4},
        # evaluation of the 256 x 256 model of depth 16
        {"name": "fwd_256_b8", "op": "fwd", "B": 8, "H": 16, "sides": SIDES_256, "window": "markov"},
        # training of the 256 x 256 model of depth 30
        {"name": "train_256_b32", "op": "train", "B": 32, "H": 30, "sides": SIDES_256, "window": "markov", "dtype": "bf16", "layout": "heads"},
        # training of the 512 x 512 model of depth 24: the benchmark's shape
        {"name": "train_512_b16", "op": "train", "B": 16, "H": 24, "sides": SIDES_512, "window": "markov", "dtype": "bf16", "layout": "heads"},
        # the same schedule on the QKV projection's own layouts, a smaller batch and model, as a fine-tuning run has it
        {"name": "train_512_packed_b6", "op": "train", "B": 6, "H": 16, "sides": SIDES_512, "window": "markov", "dtype": "bf16", "layout": "packed"},
        # a schedule of odd sides, an odd batch and an odd number of heads: no tile is full
        {"name": "train_ragged_b3", "op": "train", "B": 3, "H": 13, "sides": "1,3,5,7,11,15,21,27", "window": "markov", "dtype": "bf16", "layout": "heads"},
        # a long sequence (1024 x 1024): the largest call
        {"name": "train_1024_b8", "op": "train", "B": 8, "H": 24, "sides": SIDES_1024, "window": "markov", "dtype": "bf16", "layout": "heads"},
        # the fp32 build on a small batch: the pass that a bf16 run is checked against
        {"name": "train_256_f32_b2", "op": "train", "B": 2, "H": 16, "sides": SIDES_256, "window": "markov", "dtype": "f32", "layout": "heads"},
        # the sampler's other steps at a serving batch: twenty small calls per image batch
        {"name": "recon_sampler_b16", "op": "recon", "B": 16, "C": 32, "V": 4096, "sides": SIDES_512, "sample": True},
        # decoding of token maps in bulk: a reconstruction larger than the caches, ten additions
        {"name": "recon_decode_b2048", "op": "recon", "B": 2048, "C": 32, "V": 4096, "sides": SIDES_512, "sample": False},
    ]


# Bounds of what draw() gives: the largest listed case of each kind.
MOST_PAIRS = 38444026 * 8 * 24            # (query, key) pairs of a pass, bf16
MOST_ROWS = 9451 * 8 * 24                 # tokens times heads
MOST_PAIRS_F32 = 180820 * 2 * 16
MOST_RECON = 2048 * 32 * 32 * 32 * 10     # elements added to in a pass


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def _schedule(rng, most):
    """A rising list of sides from 1 to something between 6 and `most`, about evenly spaced in their logarithm."""
    last = _log_int(rng, 6, most)
    count = rng.randint(4, min(14, last))
    sides = {1, last}
    for i in range(1, count - 1):
        sides.add(max(2, min(last - 1, round(last ** (i / (count - 1)) * rng.uniform(0.85, 1.15)))))
    return sorted(sides)


def draw(rng):
    kind = rng.choices(["step", "sweep", "fwd", "train", "f32", "recon"], [5, 2, 3, 6, 2, 3])[0]
    if kind == "step":
        case = {"op": "step", "B": _log_int(rng, 1, 64), "H": rng.randint(4, 30), "cur": _log_int(rng, 1, 48), "lse": rng.random() < 0.25}
        case["prev"] = min(case["cur"] - 1, max(1, round(case["cur"] * rng.uniform(0.55, 0.85)))) if case["cur"] > 1 else 0
        while _pairs(case) > MOST_PAIRS // 8:
            case["B"] = (case["B"] + 1) // 2
        return case
    if kind == "recon":
        sides = _schedule(rng, 64)
        case = {"op": "recon", "B": _log_int(rng, 1, 2048), "C": rng.choice([16, 32, 32, 64]), "V": rng.choice([1024, 4096, 8192]),
                "sides": ",".join(map(str, sides)), "sample": rng.random() < 0.5}
        while case["B"] * case["C"] * sides[-1] ** 2 * len(sides) > MOST_RECON // (2 if case["sample"] else 1):
            case["B"] = (case["B"] + 1) // 2
        return case
    sides = _schedule(rng, 24 if kind == "f32" else 64)
    case = {"op": kind if kind in ("sweep", "fwd") else "train", "B": _log_int(rng, 1, 32), "H": rng.randint(4, 30), "sides": ",".join(map(str, sides))}
    if kind == "sweep":
        case["sub_steps"] = rng.randint(1, 4)
    else:
        case["window"] = "causal" if rng.random() < 0.2 else "markov"
    if case["op"] == "train":
        case["dtype"] = "f32" if kind == "f32" else "bf16"
        case["layout"] = "packed" if kind == "train" and case["window"] == "markov" and rng.random() < 0.3 else "heads"
    most = MOST_PAIRS_F32 if kind == "f32" else MOST_PAIRS
    while _pairs(case) > most or _rows(case) > MOST_ROWS:
        if case["B"] > 1:
            case["B"] = (case["B"] + 1) // 2
        else:
            case["H"] = (case["H"] + 1) // 2
    return case


def _rows(case):
    return case["B"] * case["H"] * sum(s * s for s in _sides(case))


def _pairs(case):
    """(query, key) pairs of one pass, over all heads."""
    if case["op"] == "step":
        n = case["cur"] ** 2
        return case["B"] * case["H"] * n * (n + case["prev"] ** 2)
    n = [s * s for s in _sides(case)]
    causal = case.get("window") == "causal"
    pairs = sum(n[i] * (sum(n[:i + 1]) if causal else n[i] + (n[i - 1] if i else 0)) for i in range(len(n)))
    return case["B"] * case["H"] * pairs * case.get("sub_steps", 1)


def _randn(g, *shape, dtype=torch.bfloat16):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32).to(dtype)


def prepare(case, seed):
    """Activations behind a normalised QKV projection are close to N(0, 1); token ids are uniform and a sub-step's mask
    takes half of the positions."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    state = {"case": dict(case)}
    if case["op"] == "step":
        B, H, cur, prev = case["B"], case["H"], case["cur"] ** 2, case["prev"] ** 2
        state["q"], state["k_cur"], state["v_cur"] = (_randn(g, B, H, cur, D) for _ in range(3))
        state["k_prev"], state["v_prev"] = (_randn(g, B, H, prev, D) for _ in range(2)) if prev else (None, None)
    elif case["op"] == "sweep":
        B, H, scales, before = case["B"], case["H"], [], 0
        for side in _sides(case):
            n, m = side * side, before * before
            k, v = (_randn(g, B, H, m + n, D) for _ in range(2))
            views = (k[:, :, :m], v[:, :, :m]) if m else (None, None)
            queries = [_randn(g, B, H, n, D) for _ in range(case["sub_steps"])]
            scales.append((before, side, *views, k[:, :, m:], v[:, :, m:], queries))
            before = side
        state["scales"] = scales
    elif case["op"] == "recon":
        B, sides = case["B"], _sides(case)
        state["sides"] = sides
        state["codebook"] = _randn(g, case["V"], case["C"], dtype=torch.float32)
        ids = lambda s: torch.randint(0, case["V"], (B, s, s), generator=g, device="cuda", dtype=torch.int32)  # noqa: E731
        state["new"] = [ids(s) for s in sides]
        if case["sample"]:
            state["old"] = [ids(s) for s in sides]
            state["mask"] = [torch.randint(0, 2, (B, s, s), generator=g, device="cuda", dtype=torch.uint8) for s in sides]
            state["selected"] = [torch.empty_like(t) for t in state["new"]]
    else:
        B, H, sides = case["B"], case["H"], _sides(case)
        L = sum(s * s for s in sides)
        state["sides"] = sides
        if case.get("layout") == "packed":
            state["qkv"], state["dout"] = _randn(g, B, L, 3, H, D), _randn(g, B, L, H, D)
        else:
            dtype = torch.float32 if case.get("dtype") == "f32" else torch.bfloat16
            state["q"], state["k"], state["v"] = (_randn(g, B, H, L, D, dtype=dtype) for _ in range(3))
            if case["op"] == "train":
                state["dout"] = _randn(g, B, H, L, D, dtype=dtype)
    return state


def run(state):
    case = state["case"]
    if case["op"] == "step":
        out, lse = hmar.hmar_attn_scale_step(state["q"], state["k_prev"], state["v_prev"], state["k_cur"], state["v_cur"],
                                             case["prev"], case["cur"], SCALE, want_lse=case["lse"])
        return (out, lse) if case["lse"] else (out,)
    if case["op"] == "sweep":
        outs = []
        for before, side, k_prev, v_prev, k_cur, v_cur, queries in state["scales"]:
            for q in queries:
                outs.append(hmar.hmar_attn_scale_step_strided(q, k_prev, v_prev, k_cur, v_cur, before, side, SCALE, want_lse=False)[0])
        return outs
    if case["op"] == "recon":
        sides = state["sides"]
        xhat = torch.zeros((case["B"], case["C"], sides[-1], sides[-1]), device="cuda")
        small = []
        for i, side in enumerate(sides):
            if case["sample"]:
                if i:
                    small.append(hmar.hmar_recon_downsample(xhat, side))
                hmar.hmar_recon_accumulate(xhat, state["codebook"], state["new"][i], state["old"][i], state["mask"][i], state["selected"][i])
            else:
                hmar.hmar_recon_accumulate(xhat, state["codebook"], state["new"][i])
        return {"xhat": xhat, "small": small, "selected": state.get("selected", [])}
    sides = state["sides"]
    if case.get("layout") == "packed":
        out, lse = hmar.hmar_attn_fwd_packed(state["qkv"], sides, SCALE)
        return out, lse, hmar.hmar_attn_bwd_packed(state["qkv"], out, lse, state["dout"], sides, SCALE)
    window = WINDOWS[case["window"]]
    q, k, v = state["q"], state["k"], state["v"]
    out, lse = hmar.hmar_attn_fwd(q, k, v, sides, SCALE, window=window)
    if case["op"] == "fwd":
        return out, lse
    return (out, lse, *hmar.hmar_attn_bwd(q, k, v, out, lse, state["dout"], sides, SCALE, window=window))


def work(case):
    """Inputs read once and outputs written once; 4 D operations per pair forward and 10 D backward (the masked pairs do
    not count); 2 operations per tap of a separable bicubic enlargement and 1 per pixel of a mean."""
    if case["op"] == "recon":
        B, C, sides = case["B"], case["C"], _sides(case)
        image, maps = B * C * sides[-1] ** 2, B * sum(s * s for s in sides)
        work_bytes, flops = len(sides) * 2 * 4 * image + 4 * maps, 0
        for s in sides:
            flops += B * C * (8 * s * sides[-1] + 8 * sides[-1] ** 2 + sides[-1] ** 2)
        if case["sample"]:
            work_bytes += (4 + 1 + 4) * maps + (len(sides) - 1) * 4 * image + 4 * C * (maps - B)
            flops += (len(sides) - 1) * image
        return {"bytes": work_bytes + 4 * case["V"] * C, "flops": flops}
    BH, pairs = case["B"] * case["H"], _pairs(case)
    if case["op"] == "step":
        n, m = case["cur"] ** 2, case["prev"] ** 2
        return {"bytes": BH * (2 * D * (2 * n + 2 * (n + m)) + (4 * n if case["lse"] else 0)), "flops": 4 * D * pairs}
    if case["op"] == "sweep":
        n = [s * s for s in _sides(case)]
        rows = sum(2 * n[i] + 2 * (n[i] + (n[i - 1] if i else 0)) for i in range(len(n)))
        return {"bytes": case["sub_steps"] * BH * rows * 2 * D, "flops": 4 * D * pairs}
    element = 4 if case.get("dtype") == "f32" else 2
    tensors, per_pair = (4, 4 * D) if case["op"] == "fwd" else (8, 14 * D)
    return {"bytes": _rows(case) * (tensors * D * element + 4), "flops": per_pair * pairs}


def tolerance(case):
    """About four times what was seen.  bf16 against the fp32 build on the same values: out 2.3e-3, dq, dk, dv 2.5e-3 (the
    rounding of P, dS and of the results), largest single difference 0.16 of the root mean square (in the 1024 x 1024
    gradients).  fp32 against fp64: 4.1e-7 and 4.4e-6; the reconstruction 4.3e-7 and 3.1e-6."""
    if case["op"] == "recon" or case.get("dtype") == "f32":
        return {"rel": 2e-6, "max": 2e-5}
    return {"rel": 1e-2, "max": 0.6}
