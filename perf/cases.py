"""Timing cases of the ZGR step: the calls that a program which trains with it makes, over the sizes it makes them at.

Four kinds of pass, all through ``paper_2601_12917_b200.zgr``:

  step       one optimiser step on the weights: per query perturb(+eps), perturb(-2 eps), restore_update
  round      a step whose guided payload arrives from the host, layer by layer under the first sweep, with the
             norms of the perturbation kept by that sweep, read back, and used to move the mixing ratio
  aggregate  the server's side: the updates of several clients' seeds in one pass over the weights
  basis      the cloud's side: an orthonormal basis from collected gradient directions, for every matrix of a model

A model is described by its width, feed-forward width, vocabulary and depth ("gated": three feed-forward
matrices and no biases, otherwise two and biases); every matrix has a subspace of the same rank.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2601_12917_b200 import zgr

EPS, LR = 1e-3, 1e-4
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BUCKET = 1 << 30            # weights are kept in flat buckets of at most about this many elements


def _case(name, kind, d, ffn, vocab, layers, dtype, rank, *, gated=False, head=False, bits=16, alpha=0.5, queries=1, payload="seed", seeds=0):
    c = {"kind": kind, "d": d, "ffn": ffn, "vocab": vocab, "layers": layers, "gated": gated, "head": head, "dtype": dtype, "rank": rank,
         "bits": bits, "alpha": alpha, "queries": queries, "payload": payload, "seeds": seeds}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a handful of small layers (adapters, a classification head): launches and latency are all there is
        _case("step_tiny_f32_r4", "step", 256, 0, 0, 1, "f32", 4, bits=32),
        # fine-tuning a RoBERTa-large-shaped encoder in fp32, the ordinary small-rank subspace
        _case("step_roberta_f32_r8", "step", 1024, 4096, 50265, 24, "f32", 8),
        # fp32 weights with a wide subspace (a quarter of the same encoder): better guidance, no 16-bit storage
        _case("step_roberta_f32_r32", "step", 1024, 4096, 50265, 6, "f32", 32, bits=32),
        # OPT-1.3B-shaped decoder in fp16
        _case("step_opt_f16_r16", "step", 2048, 8192, 50272, 24, "f16", 16),
        # the headline: LLaMA-7B-shaped bf16, four queries averaged per step
        _case("step_llama7b_bf16_r32_q4", "step", 4096, 11008, 32000, 32, "bf16", 32, gated=True, head=True, queries=4),
        # the widest subspace, coefficients delivered as int8 codes: ten of the 40 layers of a LLaMA-13B-shaped set
        _case("step_llama13b_bf16_r64_int8", "step", 5120, 13824, 32000, 10, "bf16", 64, gated=True, head=True, payload="int8"),
        # every normal from 32 random bits instead of 16 (the binding's default), four layers of the 7B shape
        _case("step_llama7b_bf16_r32_bits32", "step", 4096, 11008, 32000, 4, "bf16", 32, gated=True, head=True, bits=32),
        # plain zeroth-order training without a subspace (alpha = 1), the method's own baseline
        _case("step_opt_bf16_plain", "step", 2048, 8192, 50272, 6, "bf16", 0, alpha=1.0),
        # widths that are no multiple of eight elements: pruned or transposed layers
        _case("step_ragged_bf16_r16", "step", 1234, 4937, 8003, 6, "bf16", 16),
        # a guided round: new subspaces stream in from pinned host memory, norms are kept and read, alpha adapts
        _case("round_llama7b_bf16_r32", "round", 4096, 11008, 32000, 8, "bf16", 32, gated=True, head=True, payload="subspace"),
        # eight clients' projected gradients applied in one pass
        _case("aggregate8_opt_f16_r16", "aggregate", 2048, 8192, 50272, 24, "f16", 16, seeds=8),
        # bases for all matrices of the OPT-1.3B-shaped decoder
        _case("basis_opt_r16", "basis", 2048, 8192, 50272, 24, "f16", 16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "round", "aggregate", "basis"])
    d = int(_log(rng, 96, 5200))
    width = rng.random()
    unit = 128 if width < 0.4 else (8 if width < 0.75 else 1)      # most widths are multiples of 128, some of 8, some of nothing
    d = max(unit, d // unit * unit)
    gated = rng.random() < 0.5
    ffn = int(d * (2.7 if gated else 4.0) * rng.uniform(0.9, 1.1)) // unit * unit
    dtype = rng.choice(["f32", "f16", "bf16", "bf16"])
    rank = rng.choice([4, 8, 16, 32, 64, rng.randint(1, 64)])
    rank = min(rank, d)
    bits = 32 if rng.random() < 0.3 else 16
    alpha = 1.0 if kind == "step" and rng.random() < 0.1 else rng.choice([0.5, 0.5, 0.25, 0.8])
    if alpha == 1.0:
        rank = 0
    queries = rng.choice([1, 1, 1, 2, 4]) if kind == "step" else 1
    seeds = rng.randint(2, 8) if kind == "aggregate" else 0
    payload = "seed"
    if kind == "round":
        payload = rng.choice(["subspace", "int8", "int4"])
    elif kind == "step" and rank > 0 and rng.random() < 0.25:
        payload = rng.choice(["int8", "int4"])
    vocab = int(_log(rng, 2000, 50000))
    most = _log(rng, 3e5, 1.2e9 / queries)                         # weights of the model
    if (unit == 1 or dtype == "f32") and rank > 8:                 # (these take several times as long per weight)
        most /= 4
    per_layer = 4 * d * d + (3 if gated else 2) * d * ffn
    vocab = min(vocab, max(0, int(most / 2 / d)))
    layers = max(1, min(40, int((most - vocab * d) / per_layer)))
    if kind == "basis":
        layers = min(layers, 24)
    head = gated and vocab > 0 and rng.random() < 0.5
    return _case(None, kind, d, ffn, vocab, layers, dtype, rank, gated=gated, head=head, bits=bits, alpha=alpha, queries=queries, payload=payload, seeds=seeds)


def _model(case):
    """(rows, cols, rank) of every tensor, and the index one past each layer."""
    d, f, r = case["d"], case["ffn"], case["rank"]
    t, ends = [], []
    if case["vocab"]:
        t.append((case["vocab"], d, r))
        ends.append(len(t))
    for _ in range(case["layers"]):
        t += [(d, d, r)] * 4
        if f:
            t += [(f, d, r)] * (2 if case["gated"] else 1) + [(d, f, r)]
        if case["gated"]:
            t += [(1, d, 0)] * 2
        elif f:
            t += [(1, d, 0)] * 4 + [(1, f, 0)] + [(1, d, 0)] * 5
        else:
            t += [(1, d, 0)] * 4
        ends.append(len(t))
    if case["head"]:
        t += [(1, d, 0), (case["vocab"], d, r)]
        ends.append(len(t))
    return [(m, n, min(k, m)) for m, n, k in t], ends


def _flat(sizes, dtype, device="cuda", pin=False):
    """One view per size in flat buffers, each starting on a 512-byte boundary, and the buffers."""
    step = 512 // torch.empty(0, dtype=dtype).element_size()
    starts, lengths = [], [0]
    for n in sizes:
        if lengths[-1] and lengths[-1] + n > BUCKET:
            lengths.append(0)
        starts.append((len(lengths) - 1, lengths[-1]))
        lengths[-1] += -(-n // step) * step
    buckets = [torch.zeros(n, dtype=dtype, device=device, pin_memory=pin) for n in lengths]
    return [buckets[b][s:s + n] for (b, s), n in zip(starts, sizes)], buckets


def _orthonormal(views, shapes, gen):
    """Fill the views with orthonormal columns (Cholesky QR of a Gaussian), tensors of one shape together."""
    by_shape = {}
    for v, s in zip(views, shapes):
        by_shape.setdefault(s, []).append(v)
    for (m, r), vs in by_shape.items():
        for v in vs:
            g = torch.randn(m, r, generator=gen, device="cuda")
            for _ in range(2 if m < 8 * r else 1):
                low = torch.linalg.cholesky((g.T.double() @ g.double()))
                g = torch.linalg.solve_triangular(low, g.T.double(), upper=False).T.float()
            v.copy_(g.reshape(-1))


def prepare(case, seed):
    shapes, ends = _model(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dtype = DTYPES[case["dtype"]]
    flat, buckets = _flat([m * n for m, n, _ in shapes], dtype)
    for b in buckets:                                   # weights are N(0, 0.02^2)
        for at in range(0, b.numel(), 1 << 28):
            b[at:at + (1 << 28)].normal_(0.0, 0.02, generator=gen)
    weights = [w.view(m, n) if m > 1 else w for w, (m, n, _) in zip(flat, shapes)]
    guided = [l for l, (_, _, r) in enumerate(shapes) if r]
    ur = [(shapes[l][0], shapes[l][2]) for l in guided]
    u_flat, u_buckets = _flat([m * r for m, r in ur], torch.float32) if guided else ([], [])
    _orthonormal(u_flat, ur, gen)
    U = [None] * len(shapes)
    for l, u, (m, r) in zip(guided, u_flat, ur):
        U[l] = u.view(m, r)
    s = {"kind": case["kind"], "weights": buckets, "bases": u_buckets, "queries": case["queries"], "ends": ends, "step": 0, "seed": 1_000_003 * (seed % (1 << 40))}
    z = s["zgr"] = zgr.Zgr(weights, U, case["alpha"], EPS, zgr.SCALE_UNIT, case["bits"])
    rng = random.Random(seed)
    s["losses"] = [(rng.uniform(1.5, 2.5), rng.uniform(1.5, 2.5)) for _ in range(256)]
    codes, scales, zeros = {}, {}, {}
    if case["payload"] in ("int8", "int4"):
        for l in guided:
            _, n, r = shapes[l]
            g = torch.randn(r, n, generator=gen, device="cuda")
            wobble = 1 + 0.1 * (2 * torch.rand(r, generator=gen, device="cuda") - 1)
            if case["payload"] == "int8":               # unit Gaussian coefficients quantised over +-4.2 sigma
                codes[l] = (g * (127 / 4.2)).round().clamp(-127, 127).to(torch.int8)
                scales[l], zeros[l] = wobble * (4.2 / 127), None
                z.set_coeffs_dtc(l, codes[l], scales[l])
            else:                                       # unsigned 4-bit codes, two to a byte, with a zero point
                q = (g * (15 / 6.0) + 7.5).round().clamp(0, 15).to(torch.uint8)
                q = torch.nn.functional.pad(q, (0, n & 1))
                codes[l] = (q[:, 0::2] | (q[:, 1::2] << 4)).contiguous().view(torch.int8)
                scales[l], zeros[l] = wobble * (6.0 / 15), torch.full((r,), 7.5, device="cuda")
                z.set_coeffs_dtc(l, codes[l], scales[l], zeros[l], bits=4)
    if case["kind"] == "round":                         # what arrives from the cloud, in pinned host memory
        s["copies"] = torch.cuda.Stream()
        if case["payload"] == "subspace":
            new = [torch.empty_like(u) for u in u_flat]
            _orthonormal(new, ur, gen)
            host, s["host"] = _flat([m * r for m, r in ur], torch.float32, "cpu", True)
            for h, u in zip(host, new):
                h.copy_(u)
            s["deliveries"] = [(l, None, None, None, h.view(m, r)) for l, h, (m, r) in zip(guided, host, ur)]
        else:
            s["codes"] = list(codes.values())
            s["deliveries"] = [(l, codes[l].cpu().pin_memory(), scales[l].cpu().pin_memory(), None if zeros[l] is None else zeros[l].cpu().pin_memory())
                               for l in guided]
        z.enable_stats(True)
    if case["kind"] == "aggregate":
        s["seeds"] = case["seeds"]
    if case["kind"] == "basis":                         # gradient directions: mixed Gaussian columns of different sizes
        s["grads"] = []
        for l in guided:
            m, _, r = shapes[l]
            g = torch.randn(m, r, generator=gen, device="cuda")
            g = g @ (torch.eye(r, device="cuda") + 0.3 / math.sqrt(r) * torch.randn(r, r, generator=gen, device="cuda"))
            s["grads"].append((l, (g * torch.logspace(0, -2, r, device="cuda")).contiguous()))
    torch.cuda.synchronize()
    return s


def run(s):
    z, t = s["zgr"], s["step"]
    s["step"] = t + 1
    losses = s["losses"]
    if s["kind"] == "basis":
        for l, g in s["grads"]:
            z.build_subspace(l, g)
        return s["bases"]
    if s["kind"] == "aggregate":
        n = s["seeds"]
        pairs = [losses[(n * t + i) % len(losses)] for i in range(n)]
        z.restore_update_multi([s["seed"] + 1000 * t + i for i in range(n)], [p[0] for p in pairs], [p[1] for p in pairs], LR / n)
        return s["weights"]
    if s["kind"] == "round":
        seed = s["seed"] + 1000 * t
        plus, minus = losses[t % len(losses)]
        z.perturb_layers(seed, EPS, s["ends"], s["deliveries"], copy_stream=s["copies"])
        z.perturb(seed, -2 * EPS)
        z.restore_update(seed, plus, minus, LR)
        norms = z.get_stats(seed)
        return {"weights": s["weights"], "norms": norms, "alpha": z.adapt_alpha(norms)}
    q = s["queries"]
    for i in range(q):
        seed = s["seed"] + 1000 * t + i
        plus, minus = losses[(q * t + i) % len(losses)]
        z.perturb(seed, EPS)
        z.perturb(seed, -2 * EPS)
        z.restore_update(seed, plus, minus, LR / q)
    return s["weights"]


def work(case):
    shapes, _ = _model(case)
    eb = torch.empty(0, dtype=DTYPES[case["dtype"]]).element_size()
    weights = sum(m * n for m, n, _ in shapes)
    basis = sum(m * r for m, _, r in shapes)
    if case["kind"] == "basis":       # directions in, basis out; one Gram matrix and one triangular product
        return {"bytes": 8.0 * basis, "flops": float(sum(2 * m * r * r for m, _, r in shapes))}
    guided = sum(m * n * r for m, n, r in shapes)
    coeffs = sum(n * r for _, n, r in shapes)
    code_bytes = {"int8": 1.0, "int4": 0.5}.get(case["payload"], 0.0) * coeffs
    sweeps = 1 if case["kind"] == "aggregate" else 3 * case["queries"]
    terms = max(1, case["seeds"])
    each = 2.0 * eb * weights + 4.0 * basis + code_bytes
    extra = 4.0 * basis if case["payload"] == "subspace" else code_bytes if case["kind"] == "round" else 0.0
    return {"bytes": sweeps * each + extra, "flops": sweeps * (2.0 * guided + 2.0 * terms * weights)}


# Measured on 4.7 million weights against the same passes in 64 bits with one rounding to the storage type per sweep:
# fp32 rel 5e-8 to 8e-8, max 7e-7 (four queries); fp16 rel 1.0e-5 to 2.7e-5, max 1.5e-3 (one unit in the last place);
# bf16 rel 2.7e-5 to 7.5e-5, max 7e-3 to 2.1e-2 (up to three units in the last place after twelve sweeps), where a
# weight lands next to a rounding boundary; norms rel 5e-7; bases rel 2.6e-8, max 6e-8.
def tolerance(case):
    if case["kind"] == "basis":
        return {"rel": 1e-7, "max": 5e-7}
    return {"f32": {"rel": 4e-7, "max": 3e-6}, "f16": {"rel": 1e-4, "max": 6e-3}, "bf16": {"rel": 3e-4, "max": 5e-2}}[case["dtype"]]
