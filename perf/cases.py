"""Measured cases: what a program that serves or prepares a mixed-bitwidth sparse-MoE model has this library do.

forward   one pass of a batch through a stack of MoE layers (MoELayer.forward_device, one call per layer), weights
          resident on the GPU: decoding one request or a batch of them, and prefill with even or Zipf-like expert loads
pack      quantise and pack the fp32 matrices of one expert (the offline stage)
requant   move the stored matrices of one expert to a narrower width (bitwidth selection)
cached    decode steps of a stack whose experts live in pinned host memory behind the HBM expert cache

Shapes are those of the repository's workloads (inputs.WORKLOADS) and the ranges around them.  Weights ~ N(0, 0.02^2),
activations ~ N(0, 1); the experts of a layer are 2, 4 and 8 bits wide in the proportion 1:2:1.
"""
import math
import random

import torch

from paper_2308_14352_b200 import binding as B, cached_stack, inputs, layer

STD = 0.02
_SCALE_DTYPE = {"f32": B.DTYPE_F32, "f16": B.DTYPE_F16}


def _forward(name, layers, tokens, d_model, d_ff, experts, top_k=1, act="relu", gate="softmax", group=128, scales="f16",
             acts="bf16", zipf=0.0):
    case = {"work": "forward", "layers": layers, "tokens": tokens, "d_model": d_model, "d_ff": d_ff, "experts": experts,
            "top_k": top_k, "act": act, "gate": gate, "group": group, "scales": scales, "acts": acts, "zipf": zipf}
    return dict(case, name=name) if name else case


def _gated(name, layers, tokens, d_model, d_ff, experts=8):
    return _forward(name, layers, tokens, d_model, d_ff, experts, 2, "swiglu", "softmax_renorm")


def _pack(name, rows, cols, act, bits, group, scales="f16"):
    case = {"work": "pack", "d_ff": rows, "d_model": cols, "act": act, "bits": bits, "group": group, "scales": scales}
    return dict(case, name=name) if name else case


def _requant(name, rows, cols, act, bits, bits_out, group, scales="f16"):
    case = dict(_pack(None, rows, cols, act, bits, group, scales), work="requant", bits_out=bits_out)
    return dict(case, name=name) if name else case


def _cached(name, layers, steps, tokens, d_model, d_ff, experts, slots):
    case = {"work": "cached", "layers": layers, "steps": steps, "tokens": tokens, "d_model": d_model, "d_ff": d_ff,
            "experts": experts, "slots": slots}
    return dict(case, name=name) if name else case


def listed():
    return [
        # one request decoding on a Switch-base stack: the paper's own target, where latency and launches count
        _forward("base_decode_t1", 12, 1, 768, 3072, 32),
        # a served batch on the same stack: about two tokens per activated expert (the benchmark's default)
        _forward("base_decode_t64", 12, 64, 768, 3072, 32),
        # several prompts at once on that stack, an odd number of tokens, some 24 per expert
        _forward("base_prefill_t777", 12, 777, 768, 3072, 32),
        # full-precision activations and per-channel fp32 scales (the accuracy reference configuration), eight layers
        _forward("tiny_fp32_t16", 8, 16, 768, 3072, 8, group=0, scales="f32", acts="f32"),
        # prefill over 128 experts with Zipf-like loads: a few experts with hundreds of tokens, many with a handful
        _forward("large_prefill_zipf_t2048", 1, 2048, 1024, 4096, 128, zipf=1.1),
        # one request, a few requests and an odd batch of them decoding on a Mixtral-like layer: weight streaming
        _gated("mixtral_decode_t1", 1, 1, 4096, 14336),
        _gated("mixtral_decode_t4", 1, 4, 4096, 14336),
        _gated("mixtral_decode_t23", 1, 23, 4096, 14336),
        # a long prompt on that layer: about 512 tokens per expert, a dense contraction
        _gated("mixtral_prefill_t2048", 1, 2048, 4096, 14336),
        # the offline stage on one Mixtral-like expert
        _pack("pack_mixtral_int4", 14336, 4096, "swiglu", 4, 128),
        # bitwidth selection: that expert moved from 8 to 4 bits
        _requant("requant_mixtral_8to4", 14336, 4096, "swiglu", 8, 4, 128),
        # decoding with a quarter of the experts resident: routing, prediction, loads and the forward of every layer
        _cached("cached_decode_t1", 6, 16, 1, 768, 3072, 32, 48),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, lo, hi, ratio_lo, ratio_hi, step):
    """d_model from lo to hi and d_ff from ratio_lo to ratio_hi times that, both multiples of step."""
    d = step * _log_int(rng, lo / step, hi / step)
    return d, step * max(1, int(round(d * rng.uniform(ratio_lo, ratio_hi) / step)))


def draw(rng: random.Random):
    kind = rng.choice(["small_decode", "small_decode", "prefill", "prefill", "fp32", "gated_decode", "gated_decode",
                       "gated_prefill", "pack", "requant", "cached"])
    if kind == "small_decode":
        d, f = _dims(rng, 512, 1280, 2.0, 4.5, 128)
        experts = rng.choice([8, 16, 32, 64])
        if rng.random() < 0.25:
            return _gated(None, rng.randint(2, 8), _log_int(rng, 1, 96), d, f, experts)
        return _forward(None, rng.randint(3, 12), _log_int(rng, 1, 128), d, f, experts, group=rng.choice([0, 128, 128, 128]))
    if kind == "prefill":
        d, f = _dims(rng, 512, 1536, 3.0, 4.0, rng.choice([128, 512]))
        experts = rng.choice([16, 32, 64, 128])
        layers = rng.randint(1, 4)
        return _forward(None, layers, _log_int(rng, 192, 2048), d, f, experts, zipf=rng.choice([0.0, 1.1]))
    if kind == "fp32":
        d, f = _dims(rng, 256, 1024, 2.0, 4.0, 64)
        return _forward(None, rng.randint(2, 8), _log_int(rng, 1, 64), d, f, rng.choice([4, 8, 16]), rng.choice([1, 2]),
                        group=rng.choice([0, 0, 64]), scales=rng.choice(["f32", "f16"]), acts="f32")
    if kind == "gated_decode":
        d, f = _dims(rng, 2048, 4096, 2.5, 3.5, 128)
        return _gated(None, 1, _log_int(rng, 1, 64), d, f)
    if kind == "gated_prefill":
        d, f = _dims(rng, 1024, 4096, 2.5, 3.5, 512)
        return _gated(None, 1, _log_int(rng, 256, 2048), d, f)
    d, f = _dims(rng, 512, 4096, 2.0, 3.5, 128)
    act = rng.choice(["relu", "swiglu"])
    if kind == "pack":
        return _pack(None, f, d, act, rng.choice([2, 4, 8]), rng.choice([0, 64, 128, 128, 128]))
    if kind == "requant":
        bits, bits_out = rng.choice([(8, 4), (8, 4), (8, 2), (4, 2)])
        return _requant(None, f, d, act, bits, bits_out, rng.choice([0, 64, 128, 128, 128]))
    d, f = _dims(rng, 512, 1024, 2.0, 4.0, 128)
    layers, experts = rng.randint(2, 6), rng.choice([8, 16, 32])
    return _cached(None, layers, rng.randint(4, 16), rng.randint(1, 4), d, f, experts, max(8, layers * experts // 4))


def _shape(case):
    if case["work"] == "forward":
        return inputs.LayerShape(case["d_model"], case["d_ff"], case["experts"], case["top_k"], case["act"], case["gate"],
                                 case["group"], case["scales"], case["acts"])
    if case["work"] == "cached":
        return inputs.LayerShape(case["d_model"], case["d_ff"], case["experts"], 1, "relu", "softmax", 128, "f16", "bf16")
    return inputs.LayerShape(case["d_model"], case["d_ff"], 1, 1, case["act"], "softmax", case["group"], case["scales"], "bf16")


def _widths(n, rng):
    widths = ([4, 2, 4, 8] * n)[:n]
    rng.shuffle(widths)
    return widths


class _State:
    """Holds what a program keeps between calls; gives the library's context back when it goes."""

    def __init__(self, case):
        self.case, self.shape = case, _shape(case)
        self.gen = torch.Generator(device="cuda")
        self.owner = None  # whose close() frees the context

    def normal(self, *size, std=1.0):
        return torch.randn(*size, generator=self.gen, device="cuda") * std

    def __del__(self):
        if getattr(self, "owner", None) is not None:
            self.owner.close()


def prepare(case, seed):
    s = _State(case)
    sh = s.shape
    s.gen.manual_seed(seed)
    rng = random.Random(seed)
    if case["work"] == "cached":
        s.stack = s.owner = cached_stack.CachedStack(sh, case["layers"], _widths(sh.n_experts, rng), case["slots"],
                                                     max_tokens=case["tokens"], seed=seed)
        s.xs = [[s.normal(case["tokens"], sh.d_model).to(torch.bfloat16) for _ in range(case["layers"])]
                for _ in range(case["steps"])]
    elif case["work"] == "forward":
        tokens = case["tokens"]
        s.layers, s.x, s.router, s.bias, s.y = [], [], [], [], []
        for _ in range(case["layers"]):
            moe = layer.MoELayer(sh, _widths(sh.n_experts, rng), max_tokens=tokens, ctx=s.owner.ctx if s.owner else None)
            s.owner = s.owner or moe
            for e in range(sh.n_experts):
                for m in range(sh.n_matrices):
                    moe.pack_matrix(e, m, s.normal(*sh.matrix_shape(m), std=STD))
            s.layers.append(moe)
            x = s.normal(tokens, sh.d_model)
            s.x.append(x.to(torch.bfloat16) if sh.act_dtype == "bf16" else x)
            s.router.append(s.normal(sh.d_model, sh.n_experts, std=STD))
            s.bias.append(_zipf_bias(sh, case["zipf"]) if case["zipf"] else None)
            s.y.append(torch.empty(tokens, sh.d_model, device="cuda"))
    else:
        bits = case["bits"]
        s.moe = s.owner = layer.MoELayer(sh, [bits])
        s.weights = [s.normal(*sh.matrix_shape(m), std=STD) for m in range(sh.n_matrices)]
        if case["work"] == "requant":
            for m, w in enumerate(s.weights):
                s.moe.pack_matrix(0, m, w)
            del s.weights
            s.out = [(torch.empty(t.numel() * case["bits_out"] // bits, dtype=torch.uint8, device="cuda"),
                      torch.empty_like(sc)) for t, sc in zip(s.moe.packed[0], s.moe.scales[0])]
    torch.cuda.synchronize()
    return s


def _zipf_bias(sh, exponent):
    """Additive router bias that makes the loads fall off about as Zipf's law: the logarithm of the target shares, scaled
    from the spread of Gumbel noise (for which it would be exact) to that of the logits, N(0, d_model * STD^2)."""
    spread = STD * math.sqrt(sh.d_model) / (math.pi / math.sqrt(6.0))
    shares = torch.from_numpy(inputs.zipf_targets(sh.n_experts, exponent))
    return (shares.log() * spread).to(torch.float32).cuda()


def run(s):
    work = s.case["work"]
    if work == "forward":
        for moe, x, router, bias, y in zip(s.layers, s.x, s.router, s.bias, s.y):
            moe.forward_device(x, router, bias, y)
        return s.y
    if work == "cached":
        outputs, picks = [], []
        for xs in s.xs:
            picks.append(s.stack.forward_stack(xs, outputs=outputs))
        s.stack.compute.synchronize()  # the step's tokens are read by the host
        return {"picks": torch.tensor([[p.tolist() for p in step] for step in picks]),
                "gates": torch.stack([g for g, _ in outputs]), "y": torch.stack([y for _, y in outputs])}
    if work == "pack":
        for m, w in enumerate(s.weights):
            s.moe.pack_matrix(0, m, w)
        return {"packed": s.moe.packed[0], "scales": s.moe.scales[0]}
    sh, c = s.shape, s.case
    for m, (packed, scales) in enumerate(s.out):
        rows, cols = sh.matrix_shape(m)
        B.emoe_requantize_expert(s.moe.ctx, s.moe.packed[0][m].data_ptr(), s.moe.scales[0][m].data_ptr(), rows, cols,
                                 c["bits"], c["bits_out"], sh.group, _SCALE_DTYPE[sh.scale_dtype], packed.data_ptr(),
                                 scales.data_ptr())
    return {"packed": [p for p, _ in s.out], "scales": [sc for _, sc in s.out]}


def _expert_weights(sh):
    return sum(r * c for r, c in (sh.matrix_shape(m) for m in range(sh.n_matrices)))


def _expert_scale_bytes(sh):
    size = 2 if sh.scale_dtype == "f16" else 4
    return size * sum(r * (c // (sh.group or c)) for r, c in (sh.matrix_shape(m) for m in range(sh.n_matrices)))


def _activated(sh, tokens, zipf):
    """Expected number of distinct experts that the tokens of one call activate."""
    shares = inputs.zipf_targets(sh.n_experts, zipf) if zipf else [1.0 / sh.n_experts] * sh.n_experts
    return float(sum(1.0 - (1.0 - min(1.0, sh.top_k * p)) ** tokens for p in shares))


def work(case):
    sh = _shape(case)
    weights, scale_bytes = _expert_weights(sh), _expert_scale_bytes(sh)
    if case["work"] == "pack":
        return {"bytes": weights * (4 + case["bits"] / 8) + scale_bytes, "flops": 0}
    if case["work"] == "requant":
        return {"bytes": weights * (case["bits"] + case["bits_out"]) / 8 + 2 * scale_bytes, "flops": 0}
    widths = _widths(sh.n_experts, random.Random(0))
    per_expert = weights * sum(widths) / len(widths) / 8 + scale_bytes
    tokens, act_size = case["tokens"], 2 if sh.act_dtype == "bf16" else 4
    per_call = (_activated(sh, tokens, case.get("zipf", 0.0)) * per_expert + tokens * sh.d_model * (act_size + 4) +
                4 * sh.d_model * sh.n_experts)
    flops = 2.0 * tokens * (sh.top_k * weights + sh.d_model * sh.n_experts)
    calls = case["layers"] * case.get("steps", 1)
    return {"bytes": calls * per_call, "flops": calls * flops}


def tolerance(case):
    if case["work"] in ("pack", "requant"):
        return "exact"  # codes and scales are defined bit for bit
    if _shape(case).act_dtype == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    # the hidden vector is rounded to bf16: sums in another order move some of its values by one unit in the last place
    return {"rel": 5e-3, "max": 5e-2}
