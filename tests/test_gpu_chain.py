"""Layers one behind the other on one stream, each taking what the one in front leaves: with dependent launches the
first kernel of a call may be running while the last one of the call in front still stores y, so it must not
read x before that kernel is done.  Bit-identical with the same layers run one at a time."""
import pytest
import torch

from paper_2308_14352_b200 import binding as B, inputs, layer

pytestmark = pytest.mark.gpu

LAYERS, ROUNDS = 6, 8
CASES = [
    # activations, tokens, experts, router + Top-K + permutation in one launch: one for each form of the router's product
    ("f32", 3, 4, False),       # inside the one-launch layer
    ("f32", 40, 8, False),      # one token per CTA
    ("f32", 40, 6, False),      # ... one expert per thread
    ("f32", 600, 6, False),     # eight tokens per CTA, one expert per thread
    ("f32", 200, 8, False),     # register-tiled, eight tokens per CTA
    ("f32", 1600, 8, False),    # ... sixteen
    ("bf16", 4, 8, False),
    ("bf16", 40, 8, False),
    ("bf16", 40, 8, True),
    ("bf16", 200, 8, False),
    ("bf16", 300, 48, False),   # the streaming kernel in front of two tcgen05 launches that find nobody
    ("bf16", 300, 4, False),    # ... of the rounded tcgen05 form for most experts, whose second projection starts early
    ("bf16", 600, 2, False),    # the rounded form alone
]


@pytest.mark.parametrize("acts,T,E,fused_routing", CASES)
def test_layers_chained_through_one_stream(acts, T, E, fused_routing):
    d = 512 if acts == "bf16" else 256
    shape = inputs.LayerShape(d, d, E, 1, "relu", "softmax_renorm", 128, "f16", acts)  # one pick, renormalised: its gate is 1
    gen = torch.Generator(device="cuda")
    gen.manual_seed(61)
    stream = torch.cuda.Stream()
    moe = []
    try:
        for _ in range(LAYERS):
            moe.append(layer.MoELayer(shape, ([8, 4, 2, 4] * E)[:E], max_tokens=T, ctx=moe[0].ctx if moe else None))
            for e in range(E):
                for m in range(2):
                    # a layer keeps its inputs' size
                    moe[-1].pack_matrix(e, m, torch.randn(d, d, generator=gen, device="cuda") * (2.0 / d) ** 0.5 * (1.4 if m else 1.0))
        Wr = [torch.randn(d, E, generator=gen, device="cuda") * 0.1 for _ in range(LAYERS)]
        B.emoe_set_fused_routing(moe[0].ctx, fused_routing)

        def chain(x0, one_at_a_time):
            B.emoe_set_dependent_launch(moe[0].ctx, not one_at_a_time)
            ys = [torch.full((T, d), float("nan"), device="cuda") for _ in range(LAYERS)]
            xs = [x0] + [torch.full_like(x0, float("nan")) for _ in range(LAYERS - 1)] if acts == "bf16" else [x0] + ys[:-1]
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                for l in range(LAYERS):
                    if l and acts == "bf16":
                        xs[l].copy_(ys[l - 1])  # a kernel of the caller's in front
                    moe[l].forward_device(xs[l], Wr[l], None, ys[l], stream=stream.cuda_stream)
                    if one_at_a_time:
                        torch.cuda.synchronize()
            torch.cuda.synchronize()
            assert B.emoe_device_status(moe[0].ctx, stream.cuda_stream) == B.OK
            return ys

        for _ in range(ROUNDS):
            x0 = torch.randn(T, d, generator=gen, device="cuda").to(torch.bfloat16 if acts == "bf16" else torch.float32)
            want, got = chain(x0, True), chain(x0, False)
            for l in range(LAYERS):
                assert torch.isfinite(want[l]).all() and want[l].abs().max() > 1e-2
                assert torch.equal(got[l], want[l]), l
    finally:
        torch.cuda.synchronize()
        for m in reversed(moe):
            m.close()
