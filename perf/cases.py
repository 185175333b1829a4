"""The work that programs have this library do, as cases that can be timed and compared.

Calls (the public entry points of paper_2609_38095_gb300):
  perturb    one in-place perturbation pass over a parameter list
  perturb2   a probe's restore and the next probe's +eps in one pass
  pair       the out-of-place pair: theta + eps z and theta - eps z into two other lists
  update     the fused K-probe update on given coefficients, with (pre) or without the last probe's restore in it
  step       the whole in-place step on given losses: perturb, K perturb passes with the K - 1 perturb2 passes
             between them, the preconditioner and the update that carries the last restore
  quad_step  a step of the small quadratic workload (QuadraticStep, schedule "onepass"), losses computed on the device

Parameter lists: the tensor shapes of OPT and Qwen3 decoders (workloads.opt_shapes, workloads.qwen3_shapes) at several
widths and depths, or "ragged": many tensors of unequal, mostly odd sizes (small multilayer models, adapters). Layout
"own": every tensor starts on a 256-byte boundary, as its own allocation would; "flat": the tensors lie back to back in
one buffer, from its second element on, so most of them start off every vector boundary. Either way they are views of
one buffer, which is what run() returns.
"""
import math
import random

import numpy as np
import torch

import paper_2609_38095_gb300 as zo
from paper_2609_38095_gb300 import workloads
from paper_2609_38095_gb300.quadratic import QuadraticStep

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
SIZE = {"f32": 4, "bf16": 2, "f16": 2}
EPS = 1e-3
LR = 1e-3           # the paper ties the step size to eps
QUAD_LR = 1e-5      # a step size at which the quadratic workload stays stable however often it is stepped
WEIGHT_SCALE = 0.02


def listed():
    return [
        # smallest calls: one pass over a small fp32 model of uneven tensors, where launches and host work are the cost
        {"name": "mlp_perturb", "call": "perturb", "shape": "ragged", "tensors": 12, "d": 270_001, "dtype": "f32",
         "layout": "own", "packing": 1},
        # a whole step of a small model or an adapter: 18 calls on a few million weights
        {"name": "mlp_step_k8", "call": "step", "shape": "ragged", "tensors": 24, "d": 1_600_003, "dtype": "bf16",
         "layout": "own", "packing": 1, "K": 8},
        # the benchmark's small workload: every forward point on the device, d = 2^20, K = 8
        {"name": "quad_step_k8", "call": "quad_step", "d": 1 << 20, "K": 8},
        # the passes between the forwards of a billion-weight model (the OPT-1.3B-shaped bf16 set)
        {"name": "opt_perturb", "call": "perturb", "shape": "opt", "layers": 24, "width": 2048, "vocab": 50272,
         "dtype": "bf16", "layout": "own", "packing": 1},
        # restore and next probe in one pass: eight Qwen3-8B-shaped layers, with their 128-element norms
        {"name": "qwen_perturb2", "call": "perturb2", "shape": "qwen", "layers": 8, "width": 4096, "vocab": 32000,
         "dtype": "bf16", "layout": "own", "packing": 1, "probe": 3},
        # out of place, for programs with room for two copies: an OPT-30B-shaped layer and its embedding
        {"name": "opt_pair", "call": "pair", "shape": "opt", "layers": 1, "width": 7168, "vocab": 50272,
         "dtype": "f16", "layout": "own", "packing": 1},
        # the updates at the probe counts these sets are trained with: few probes (bound by memory) ...
        {"name": "opt_update_k16", "call": "update", "shape": "opt", "layers": 24, "width": 2048, "vocab": 50272,
         "dtype": "bf16", "layout": "own", "packing": 1, "K": 16, "pre": True},
        # ... a middling number ...
        {"name": "qwen_update_k64", "call": "update", "shape": "qwen", "layers": 8, "width": 4096, "vocab": 32000,
         "dtype": "bf16", "layout": "own", "packing": 1, "K": 64, "pre": True},
        # ... and many (bound by arithmetic): two OPT-30B-shaped layers
        {"name": "opt_update_k256", "call": "update", "shape": "opt", "layers": 2, "width": 7168, "vocab": 2048,
         "dtype": "f16", "layout": "own", "packing": 1, "K": 256, "pre": True},
        # a model whose parameters are slices of one flat buffer: tensors at odd offsets
        {"name": "flat_update_k32", "call": "update", "shape": "ragged", "tensors": 200, "d": 400_000_007,
         "dtype": "bf16", "layout": "flat", "packing": 1, "K": 32, "pre": True},
        # full-precision weights
        {"name": "f32_update_k16", "call": "update", "shape": "opt", "layers": 12, "width": 1024, "vocab": 50272,
         "dtype": "f32", "layout": "own", "packing": 1, "K": 16, "pre": True},
        # one generated byte per weight and probe instead of one bit
        {"name": "packing8_update_k64", "call": "update", "shape": "opt", "layers": 12, "width": 1024, "vocab": 50272,
         "dtype": "bf16", "layout": "own", "packing": 8, "K": 64, "pre": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# A drawn case does at most this much: weights, and weights times probes of an update (fewer where each probe costs
# a Philox call of its own).
MOST_D = 1_200_000_000
MOST_PAIRS = 300_000_000_000


def draw(rng):
    call = rng.choice(["perturb", "perturb2", "pair", "update", "update", "update", "update", "update", "step",
                       "quad_step"])
    if call == "quad_step":
        return {"call": call, "d": _log(rng, 1 << 12, 1 << 22), "K": _log(rng, 1, 32)}
    c = {"call": call, "dtype": rng.choice(["bf16", "bf16", "f16", "f32"]),
         "layout": rng.choice(["own", "own", "own", "flat"]), "packing": rng.choice([1, 1, 1, 1, 8])}
    if call in ("update", "step"):
        c["K"] = _log(rng, 1, 24 if call == "step" else 512)
    if call == "update":
        c["pre"] = rng.random() < 0.7
    if call in ("perturb", "perturb2"):
        c["probe"] = rng.randrange(256)
    most = MOST_D // (2 if c["dtype"] == "f32" else 1)
    if call == "update":
        most = min(most, MOST_PAIRS // (c["K"] * (6 if c["packing"] == 8 else 1)))
    if call == "step":
        most = min(most, 3_000_000_000 // c["K"])
    shape = rng.choice(["ragged", "opt", "qwen"])
    if shape == "ragged":
        d = _log(rng, 10_000, most)
        c.update(shape=shape, tensors=max(1, min(d // 64, _log(rng, 1, 400))), d=d)
        return c
    for _ in range(100):
        c.update(shape=shape, layers=_log(rng, 1, 32), width=128 * _log(rng, 1, 56), vocab=_log(rng, 1000, 60_000))
        if sum(_numels(c)) <= most:
            return c
    c.update(layers=1, width=256, vocab=1000)
    return c


def _numels(case):
    """Sizes of the list's tensors, in order."""
    if case["shape"] == "opt":
        w = case["width"]
        return [n for _, n in workloads.opt_shapes(case["layers"], w, 4 * w, vocab=case["vocab"])]
    if case["shape"] == "qwen":
        w = case["width"]
        return [n for _, n in workloads.qwen3_shapes(case["layers"], w, 3 * w, n_q=w // 128, n_kv=max(1, w // 512),
                                                     vocab=case["vocab"])]
    rng = random.Random(case["d"] * 1009 + case["tensors"])
    part = [math.exp(rng.uniform(0.0, math.log(256.0))) for _ in range(case["tensors"])]
    out = [max(1, int(case["d"] * p / sum(part))) for p in part]
    out[-1] += max(0, case["d"] - sum(out))
    return out


def _starts(case):
    """(first element of every tensor in the buffer, elements of the buffer)."""
    step = 256 // SIZE[case["dtype"]] if case["layout"] == "own" else 1
    at, out = 0 if case["layout"] == "own" else 1, []
    for n in _numels(case):
        out.append(at)
        at = (at + n + step - 1) // step * step
    return out, at


def _views(case, flat):
    return [flat[s:s + n] for s, n in zip(_starts(case)[0], _numels(case))]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _weights(case, seed):
    flat = torch.empty(_starts(case)[1], dtype=DTYPES[case["dtype"]], device="cuda")
    return flat.normal_(0.0, WEIGHT_SCALE, generator=_generator(seed))


def _coefficients(losses):
    """c_k of the loss triples (Eqs. 3-5 at alpha = 0.1, lambda_reg = 1), fp64."""
    lp, lm, l0 = losses[:, 0], losses[:, 1], losses[:, 2]
    w = 1.0 / np.maximum(1.0, np.abs((lp - 2.0 * l0 + lm) / (EPS * EPS)) ** 0.1)
    return w * (lp - lm) / (2.0 * EPS)


def _quad_inputs(case, seed):
    g = _generator(seed)
    theta = torch.empty(case["d"], dtype=torch.float32, device="cuda").normal_(0.0, WEIGHT_SCALE, generator=g)
    a = torch.empty(case["d"], dtype=torch.float32, device="cuda").uniform_(-2.0, 2.0, generator=g)
    return theta, torch.pow(10.0, a)


def prepare(case, seed):
    s = {"case": case, "seed": workloads.step_seed(seed)}
    if case["call"] == "quad_step":
        theta, a = _quad_inputs(case, seed)
        s["quad"] = QuadraticStep(theta, a, case["K"], EPS, QUAD_LR, schedule="onepass")
        return s
    s["flat"] = _weights(case, seed)
    s["params"] = zo.ParamList(_views(case, s["flat"]), packing=case["packing"])
    if case["call"] == "pair":
        s["plus"], s["minus"] = s["flat"].clone(), s["flat"].clone()
        s["plus_list"] = zo.ParamList(_views(case, s["plus"]), packing=case["packing"])
        s["minus_list"] = zo.ParamList(_views(case, s["minus"]), packing=case["packing"])
    if case["call"] in ("update", "step"):
        losses = workloads.synthetic_losses(case["K"], seed)
        if case["call"] == "update":
            s["c"] = torch.from_numpy(_coefficients(losses)).cuda()
            s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        else:
            s["losses"] = torch.from_numpy(losses).cuda()
            s["out"] = (torch.empty(case["K"], dtype=torch.float64, device="cuda"),
                        torch.empty(1, dtype=torch.int32, device="cuda"))
    return s


def run(state):
    case, seed, call = state["case"], state["seed"], state["case"]["call"]
    if call == "quad_step":
        q = state["quad"]
        q.step(seed)
        return {"theta": q.theta, "losses": q.losses, "c": q.c}
    p = state["params"]
    k = case.get("probe", 0)
    if call == "perturb":
        zo.perturb(p, seed, k, EPS)
    elif call == "perturb2":
        zo.perturb2(p, seed, k, EPS, k + 1, EPS)
    elif call == "pair":
        zo.perturb_pair(p, state["plus_list"], state["minus_list"], seed, k, EPS)
        return {"plus": state["plus"], "minus": state["minus"]}
    elif call == "update":
        zo.update(p, seed, state["c"], LR, status=state["status"],
                  pre=(case["K"] - 1, EPS) if case["pre"] else None)
    else:
        K = case["K"]
        zo.perturb(p, seed, 0, EPS)
        for j in range(K):
            zo.perturb(p, seed, j, -2.0 * EPS)
            if j + 1 < K:
                zo.perturb2(p, seed, j, EPS, j + 1, EPS)
        c, status = zo.precondition(state["losses"], EPS, out=state["out"])
        zo.update(p, seed, c, LR, status=status, pre=(K - 1, EPS))
        return {"theta": state["flat"], "c": c}
    return {"theta": state["flat"]}


def work(case):
    """One read and one write of the weights per pass, and per weight and probe one addition (perturbations too)."""
    call = case["call"]
    if call == "quad_step":  # theta and the curvatures in, theta out; 2 K + 1 forward points of three operations
        d, K = case["d"], case["K"]
        return {"bytes": 12 * d, "flops": d * (3 * (2 * K + 1) + 4 * K)}
    d, size = sum(_numels(case)), SIZE[case["dtype"]]
    if call == "pair":
        return {"bytes": 3 * d * size, "flops": 2 * d}
    if call == "update":
        return {"bytes": 2 * d * size, "flops": d * (case["K"] + (1 if case["pre"] else 0))}
    if call == "step":       # 2 K passes between forwards, then the update
        return {"bytes": (2 * case["K"] + 1) * 2 * d * size, "flops": d * 4 * case["K"]}
    return {"bytes": 2 * d * size, "flops": d * (2 if call == "perturb2" else 1)}


def tolerance(case):
    """Perturbations are one fp32 addition and one rounding each: nothing is left open. The fused update's fp32 sum has
    an order: another one moves about 1e-5 of 16-bit weights (bf16; 7e-5 of fp16 ones) by a unit in the last place, and
    fp32 ones by a few 1e-8 of the sum. The losses of the quadratic workload are fp64 sums."""
    if case["call"] in ("perturb", "perturb2", "pair"):
        return "exact"
    if case["call"] == "quad_step":
        return {"rel": 1e-6, "max": 1e-5}
    return {"bf16": {"rel": 1e-4, "max": 1.6e-2}, "f16": {"rel": 4e-5, "max": 2e-3},
            "f32": {"rel": 5e-7, "max": 5e-6}}[case["dtype"]]


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch: no rounding of the weights in between.
# ---------------------------------------------------------------------------
_LOW = 0xFFFFFFFF


def _philox_bytes(first, count, word, seed):
    """Philox4x32-10 of the counters (block, word, 0) for `count` blocks from `first`: 16 bytes a block."""
    b = torch.arange(first, first + count, dtype=torch.int64, device="cuda")
    c = [b & _LOW, b >> 32, torch.full_like(b, word), torch.zeros_like(b)]
    k0, k1 = seed & _LOW, (seed >> 32) & _LOW
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57     # modulo 2^64, which keeps both halves
        c = [((p1 >> 32) & _LOW) ^ c[1] ^ k0, p1 & _LOW, ((p0 >> 32) & _LOW) ^ c[3] ^ k1, p0 & _LOW]
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    words = torch.stack([torch.where(w >= 1 << 31, w - (1 << 32), w) for w in c], dim=1).to(torch.int32)
    return words.view(torch.uint8).reshape(-1)


def _signs(first, count, probe, packing, seed):
    """z of one probe for the 16 * count weights of a range of blocks, fp64."""
    word, bit = (probe // 8, probe % 8) if packing == 1 else (probe, 0)
    return ((_philox_bytes(first, count, word, seed) >> bit) & 1).double() * 2.0 - 1.0


def _add_probes(x, first, coefficients, packing, seed):
    """x + sum_k coefficients[k] z_k over a range of weights whose first block is `first`."""
    n = x.numel()
    count = (n + 15) // 16
    if packing == 8:
        for k, v in coefficients.items():
            x = x + v * _signs(first, count, k, packing, seed)[:n]
        return x
    for q in sorted({k // 8 for k in coefficients}):
        at = np.arange(256)
        table = sum((((at >> (k % 8)) & 1) * 2.0 - 1.0) * v for k, v in coefficients.items() if k // 8 == q)
        x = x + torch.from_numpy(table).cuda()[_philox_bytes(first, count, q, seed)[:n].int()]
    return x


def _exact_list(case, flat, coefficients, seed):
    out = flat.double()
    chunk = 1 << 26
    block = 0
    for s, n in zip(_starts(case)[0], _numels(case)):
        for at in range(0, n, chunk):
            m = min(chunk, n - at)
            out[s + at:s + at + m] = _add_probes(out[s + at:s + at + m], block + at // 16, coefficients,
                                                 case["packing"], seed)
        block += (n + 15) // 16
    return out


def exact(case, seed):
    call, philox_seed = case["call"], workloads.step_seed(seed)
    if call == "quad_step":
        theta, a = (t.double() for t in _quad_inputs(case, seed))
        d, K = case["d"], case["K"]
        losses = torch.empty(K, 3, dtype=torch.float64, device="cuda")
        losses[:, 2] = 0.5 * (a * theta * theta).sum()
        for k in range(K):
            z = _signs(0, (d + 15) // 16, k, 1, philox_seed)[:d]
            for j, sign in enumerate((1.0, -1.0)):
                losses[k, j] = 0.5 * (a * (theta + sign * EPS * z) ** 2).sum()
        c = _coefficients(losses.cpu().numpy())
        theta = _add_probes(theta, 0, {k: -(QUAD_LR / K) * float(c[k]) for k in range(K)}, 1, philox_seed)
        return {"theta": theta, "losses": losses, "c": torch.from_numpy(c)}
    flat = _weights(case, seed)
    k = case.get("probe", 0)
    if call == "perturb":
        return {"theta": _exact_list(case, flat, {k: EPS}, philox_seed)}
    if call == "perturb2":
        return {"theta": _exact_list(case, flat, {k: EPS, k + 1: EPS}, philox_seed)}
    if call == "pair":
        return {name: _exact_list(case, flat, {k: sign * EPS}, philox_seed)
                for name, sign in (("plus", 1.0), ("minus", -1.0))}
    K = case["K"]
    c = _coefficients(workloads.synthetic_losses(K, seed))
    total = {j: -(LR / K) * float(c[j]) for j in range(K)}
    if call == "step":
        return {"theta": _exact_list(case, flat, total, philox_seed), "c": torch.from_numpy(c)}
    if case["pre"]:
        total[K - 1] += EPS
    return {"theta": _exact_list(case, flat, total, philox_seed)}
