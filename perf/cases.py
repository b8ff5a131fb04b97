"""The work a program has this library do, as cases to be timed: one pass each through the public entry points.

A case is a dict of plain values: what is called ("kind"), the layer shapes ("shapes" and their own sizes), the
code width, the number of workers, the norm order and scope, the step-size rule.  Five kinds:

  step       one QODA iteration: ENCODE of all workers' dual vectors (lq_quantize_pack, against the previous
             message), then DECODE + mean + update (qoda_step).
  levels     an iteration at which the levels are renewed: histograms are collected while encoding, the levels
             refitted, the probabilities of the new levels read off, then the update.
  aggregate  lq_decode_aggregate alone: the mean of K received messages.
  encode     the entropy stage on one message: fixed-width words -> Huffman streams.
  decode     its inverse, with the run offsets.

The gradients of two successive iterations are kept in memory and taken in turn, as a training program fills its
buffers anew each iteration: another draw, other embedding rows untouched.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2505_14371_b200 as lq
from paper_2505_14371_b200 import workloads as W

BITS_OF_MIXED = (2, 3, 4, 8)


def listed():
    return [
        # The smallest: 2000 iterations of a bilinear game on the joint 8192-vector.  Latency and launches only.
        dict(name="bilinear-step", kind="step", shapes="bilinear", bits=4, workers=8, q=2, scope="layer", fitted=True),
        # One gradient set of a 784-256-10 perceptron, uniform 3-bit levels, four workers.
        dict(name="mlp-step", kind="step", shapes="mlp", bits=3, workers=4, q=2, scope="layer", fitted=False),
        # DCGAN-style generator and discriminator, one norm per layer, fitted 3-bit levels.
        dict(name="wgan-step", kind="step", shapes="wgan", width=128, bits=3, workers=8, q=2, scope="layer", fitted=True),
        # The same networks as the paper's own runs have them: 5 bits, one norm per bucket of 128 coordinates.
        dict(name="wgan-bucket-step", kind="step", shapes="wgan", width=128, bits=5, workers=8, q=2, scope="bucket",
             fitted=True),
        # An iteration at which the levels are renewed (histograms, fit, probabilities of the new levels).
        dict(name="wgan-levels", kind="levels", shapes="wgan", width=128, bits=4, workers=8, q=2, scope="layer",
             fitted=True),
        # Low-rank factors of a Transformer-XL's matrices: 306 layers of a few thousand to eight million values.
        dict(name="factors-step", kind="step", shapes="factors", rank=32, blocks=16, vocab=267735, bits=4, workers=8, q=2,
             scope="layer", fitted=True),
        # The headline: all gradients of a Transformer-XL-base, 90 % of the embedding's rows untouched.
        dict(name="transformer-step", kind="step", shapes="transformer", blocks=16, vocab=267735, bits=4, workers=8, q=2,
             scope="layer", fitted=True),
        # One dense layer of odd size at the widest code, max norm: 256 levels.
        dict(name="flat-8bit-max-step", kind="step", shapes="flat", coords=50331653, bits=8, workers=4, q=0, scope="layer",
             fitted=False),
        # 512 layers of 64 to four million values, code widths 2, 3, 4 and 8 side by side.
        dict(name="ragged-mixed-step", kind="step", shapes="ragged", layers=512, low=64, high=4 << 20, shape_seed=5,
             bits=0, workers=4, q=2, scope="layer", fitted=False),
        # A receiver that only wants the mean of 16 workers' 2-bit messages.
        dict(name="flat-2bit-mean-of-16", kind="aggregate", shapes="flat", coords=33554477, bits=2, workers=16, q=2,
             scope="layer", fitted=False),
        # Storing or sending the headline's message entropy-coded, and getting it back.
        dict(name="transformer-encode", kind="encode", shapes="transformer", blocks=16, vocab=267735, bits=4, workers=8,
             q=2, scope="layer", fitted=True),
        dict(name="transformer-decode", kind="decode", shapes="transformer", blocks=16, vocab=267735, bits=4, workers=8,
             q=2, scope="layer", fitted=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: 2^13 to 2^30 worker-coordinates, every kind, width, scope and step-size rule."""
    kind = rng.choice(["step", "step", "step", "step", "step", "levels", "aggregate", "encode", "decode"])
    shapes = rng.choice(["flat", "flat", "ragged", "ragged", "wgan", "transformer", "factors"])
    workers = rng.choice([1, 2, 3, 4, 8, 8, 12, 16])
    case = dict(kind=kind, shapes=shapes, workers=workers, q=rng.choice([2, 2, 2, 0, 1]),
                scope=rng.choice(["layer", "layer", "layer", "bucket", "global"]) if kind in ("step", "levels") else "layer",
                fitted=rng.random() < 0.6)
    case["bits"] = rng.choice([2, 3, 4, 5, 8])
    coords = max(1024, _log_uniform(rng, 1 << 13, 1 << 30) // workers)
    if kind == "levels":
        case.update(bits=rng.choice([2, 3, 4, 5]), fitted=True)
        coords = min(coords, (1 << 27) // workers)
    if shapes == "flat":
        case["coords"] = coords
    elif shapes == "ragged":
        high = min(4 << 20, max(256, coords // 4))
        mean = (high - 64) / math.log(high / 64)
        case.update(low=64, high=high, layers=max(1, min(64 if kind == "levels" else 1024, int(coords / mean))),
                    shape_seed=rng.randrange(1 << 20))
        if kind == "step" and rng.random() < 0.5:
            case["bits"] = 0                                 # a width of its own for every layer
    elif shapes == "wgan":
        case["width"] = max(4, min(320, int(math.sqrt(coords / 386))))
    elif shapes == "transformer":
        blocks = rng.choice([b for b in (1, 2, 4, 8, 16) if b == 1 or 5300000 * b <= coords])
        case.update(blocks=blocks, vocab=max(1000, min(267735, (coords - 2650000 * blocks) // 410)))
        case["workers"] = max(1, min(workers, (1 << 30) // (case["vocab"] * 410 + 2650000 * blocks)))
    else:
        blocks = rng.choice([1, 2, 4, 8, 16])
        case.update(blocks=blocks, rank=rng.choice([4, 8, 16, 32, 64]), vocab=_log_uniform(rng, 1000, 267735))
    if kind == "step" and rng.random() < 0.25:
        case["alt"] = rng.choice([0.25, 0.1])                # the alternative step sizes
    if kind == "step" and rng.random() < 0.2:
        case["average"] = True                               # the running sum of the half iterates
    return case


# ---- shapes and inputs -------------------------------------------------------------------------------------

def _layers(case):
    """(layer sizes, bits of each, distribution, scale exponents, length of the rows of layer 0 that may be zero or 0)"""
    s = case["shapes"]
    rows = 0
    if s == "bilinear":
        sizes, dist, exps = W.bilinear_workload().layer_sizes, "normal", (0.0, 0.0)
    elif s == "mlp":
        sizes, dist, exps = W.mlp_workload().layer_sizes, "normal", (-4.0, -1.0)
    elif s == "wgan":
        w = case["width"]
        g = [128 * 64 * w, 64 * w, 4 * w * 2 * w * 16, 2 * w * w * 16, w * 3 * 16]
        d = [3 * w * 16, w * 2 * w * 16, 2 * w * 4 * w * 16, 64 * w]
        sizes, dist, exps = g + d, "laplace", (-4.0, -1.0)
    elif s == "transformer":
        sizes = W.transformer_xl_workload(case["blocks"], case["vocab"]).layer_sizes
        dist, exps, rows = "student3", (-5.0, -2.0), 410
    elif s == "factors":
        sizes = W.powersgd_factor_workload(case["rank"], case["blocks"], case["vocab"]).layer_sizes
        dist, exps, rows = "normal", (-4.0, -1.0), case["rank"]
    elif s == "flat":
        sizes, dist, exps = [case["coords"]], "normal", (0.0, 0.0)
    else:
        r = random.Random(case["shape_seed"])
        sizes = [_log_uniform(r, case["low"], case["high"]) for _ in range(case["layers"])]
        dist, exps = "normal", (0.0, 0.0)
    if case["bits"]:
        bits = [case["bits"]] * len(sizes)
    else:
        bits = [BITS_OF_MIXED[i % len(BITS_OF_MIXED)] for i in range(len(sizes))]
    return sizes, bits, dist, exps, rows


def _values(dist, n, gen):
    z = torch.randn(n, generator=gen, device="cuda")
    if dist == "laplace":
        u = torch.rand(n, generator=gen, device="cuda").clamp_(min=1e-7)
        return z.sign_().mul_(u.log_())
    if dist == "student3":
        c = torch.zeros(n, device="cuda")
        for _ in range(3):
            r = torch.randn(n, generator=gen, device="cuda")
            c.addcmul_(r, r)
        return z.div_(c.div_(3.0).sqrt_().clamp_(min=1e-6))
    return z


def _gradients(plan, case, scale, gen):
    sizes, _, dist, _, rows = _layers(case)
    grads = torch.empty((plan.num_workers, plan.padded_elems), device="cuda")
    for k in range(plan.num_workers):
        torch.mul(_values(dist, plan.padded_elems, gen), scale, out=grads[k])
        if rows:
            n = sizes[0] // rows
            keep = torch.rand((n, 1), generator=gen, device="cuda") >= 0.9
            grads[k, plan.elem_offsets[0]: plan.elem_offsets[0] + n * rows].view(n, rows).mul_(keep)
    return grads


# ---- one case ----------------------------------------------------------------------------------------------

def prepare(case, seed):
    sizes, bits, _, exps, _ = _layers(case)
    kind = case["kind"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    host = random.Random(seed)
    plan = lq.Plan(sizes, bits, case["q"], case["workers"], seed=0x5EED0DA + seed)
    plan.lq_set_norm_scope(case["scope"])
    if case.get("alt"):
        plan.qoda_set_alt_rates(case["alt"])
    scale = torch.zeros(plan.padded_elems, device="cuda")     # the padding between layers stays zero
    for off, n in zip(plan.elem_offsets, sizes):
        scale[off: off + n] = 10.0 ** host.uniform(*exps)
    s = dict(case=case, plan=plan, t=1)
    grads = [_gradients(plan, case, scale, gen)]
    s["packed"] = [plan.empty_packed(), plan.empty_packed()]
    s["norms"] = [plan.empty_norms(), plan.empty_norms()]
    iterating = kind in ("step", "levels")
    if iterating:
        grads.append(_gradients(plan, case, scale, gen))
        s["X1"] = torch.randn(plan.padded_elems, generator=gen, device="cuda").mul_(0.05)
        s["Y"], s["Xhalf"] = torch.empty_like(s["X1"]), torch.empty_like(s["X1"])
        if case.get("average"):
            s["xsum"] = torch.zeros(plan.padded_elems, dtype=torch.float64, device="cuda")
            plan.qoda_set_average(s["xsum"])
        plan.qoda_init(s["X1"], s["Y"], s["Xhalf"])
        s["grads"] = grads
    # the first iteration, with the level fit that precedes the steady state
    hist = plan.zero_hist() if case["fitted"] or kind == "levels" else None
    plan.lq_quantize_pack(grads[0], 1, s["packed"][1], s["norms"][1], hist=hist)
    if case["fitted"]:
        plan.lq_fit_levels(hist, s["norms"][1], plan.num_workers)
    if iterating:
        plan.qoda_step(s["packed"][1], s["norms"][1], s["X1"], s["Y"], s["Xhalf"])
    if kind == "levels":
        s["hist"] = hist
        s["probs"] = torch.zeros((plan.num_layers, 256), dtype=torch.float64, device="cuda")
    if iterating:
        return s
    # the other kinds work on the second message, encoded with the levels as fitted
    plan.lq_quantize_pack(grads[0], 2, s["packed"][0], s["norms"][0])
    s["message"], s["message_norms"] = s.pop("packed")[0], s.pop("norms")[0]
    if kind == "aggregate":
        s["gbar"] = torch.zeros(plan.padded_elems, device="cuda")
        return s
    counts = torch.zeros((plan.num_workers, plan.num_layers, 256), dtype=torch.int32, device="cuda")
    plan.lq_symbol_counts(s["message"], counts)
    for m, c in enumerate(counts.sum(dim=0).tolist()):
        plan.lq_code_set(m, lq.lq_code_build([x + 1e-9 for x in c[: 1 << bits[m]]]))
    s["stream"] = torch.zeros((plan.num_workers, plan.packed_words), dtype=torch.int32, device="cuda")
    s["offsets"] = torch.zeros((plan.num_workers, plan.lq_plan_blocks() + 1), dtype=torch.int32, device="cuda")
    s["runs"] = plan.empty_run_offsets()
    if kind == "decode":
        plan.lq_entropy_encode(s["message"], s["stream"], s["offsets"], s["runs"])
        s["back"] = torch.empty_like(s["message"])
    return s


def run(s):
    plan, kind = s["plan"], s["case"]["kind"]
    if kind == "aggregate":
        plan.lq_decode_aggregate(s["message"], s["message_norms"], s["gbar"])
        return s["gbar"]
    if kind == "encode":
        plan.lq_entropy_encode(s["message"], s["stream"], s["offsets"], s["runs"])
        return {"stream": s["stream"], "offsets": s["offsets"], "runs": s["runs"]}
    if kind == "decode":
        plan.lq_entropy_decode(s["stream"], s["offsets"], s["back"], s["runs"])
        return s["back"]
    s["t"] += 1
    t = s["t"]
    c, p = t % 2, (t + 1) % 2
    out = {"packed": s["packed"][c], "norms": s["norms"][c], "Y": s["Y"], "Xhalf": s["Xhalf"]}
    if kind == "levels":
        s["hist"].zero_()
        plan.lq_quantize_pack(s["grads"][p], t, s["packed"][c], s["norms"][c], hist=s["hist"],
                              prev_packed=s["packed"][p], prev_norms=s["norms"][p])
        plan.lq_fit_levels(s["hist"], s["norms"][c], plan.num_workers)
        plan.lq_level_probabilities(s["hist"], s["norms"][c], plan.num_workers, s["probs"], staged=True)
        out["hist"], out["probs"] = s["hist"], s["probs"]
    else:
        plan.lq_quantize_pack(s["grads"][p], t, s["packed"][c], s["norms"][c],
                              prev_packed=s["packed"][p], prev_norms=s["norms"][p])
    plan.qoda_step(s["packed"][c], s["norms"][c], s["X1"], s["Y"], s["Xhalf"])
    if "xsum" in s:
        out["xsum"] = s["xsum"]
    return out


def work(case):
    """Bytes: every input read once and every output written once; a message that one call of the pass hands to the
    next counts once, as the output it is.  flops: the floating-point operations of the definition."""
    sizes, bits, _, _, _ = _layers(case)
    K = case["workers"]
    D = float(sum(sizes))
    message = K * sum(n * (b + 1) / 8.0 for n, b in zip(sizes, bits))
    norms = 4.0 * K * (D / 128.0 if case["scope"] == "bucket" else len(sizes))
    if case["kind"] == "aggregate":
        return {"bytes": message + norms + 4.0 * D, "flops": 2.0 * K * D}
    if case["kind"] in ("encode", "decode"):
        # the stream's length depends on the values: about two bits per coordinate
        return {"bytes": message + 0.25 * K * D, "flops": 0.0}
    # norm (2), normalise, subtract, scale the uniform, compare, decode now and before, difference and its square (4)
    moved = 4.0 * K * D + 2.0 * (message + norms) + 16.0 * D
    if case["kind"] == "levels":
        moved += 2.0 * 4.0 * K * len(sizes) * lq.NUM_BINS + 8.0 * 256 * len(sizes)
    if case.get("average"):
        moved += 16.0 * D
    return {"bytes": moved, "flops": 10.0 * K * D + (K + 6.0) * D}


def tolerance(case):
    """Integers of the entropy stage are exact.  Norms and sums are fp32 values of fp64 accumulations; one unit in a
    norm's last place moves a few in 10^7 coordinates across their rounding threshold."""
    if case["kind"] in ("encode", "decode"):
        return "exact"
    if case["kind"] == "aggregate":
        return {"rel": 1e-6}
    return {"rel": 1e-5, "differ": 1e-6}
