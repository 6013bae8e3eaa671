"""A stack of MoE layers whose packed experts live in pinned host memory and are staged into the
library's HBM expert cache: the predict-then-prefetch pipeline of the paper's Section 3.3
("Preloading and pipeline", "Cache eviction policy") on a B200.  Everything here is plumbing
(memory, streams, the order of the library calls); the arithmetic runs in the library's kernels
and the cache decisions in its host code.

Per layer and token batch, one call (emoe_cached_layer):
  ids, gates = emoe_router_topk(x, Wr, bias)           # bias ties the routing to the prior
  emoe_prefetch_experts(ranked experts of the next layer)   # copy stream, overlaps this layer
  emoe_cache_acquire(activated experts)                # compute stream waits on the device
  emoe_moe_forward_routed(...); emoe_cache_release(...)
"""
from __future__ import annotations

from typing import List, Optional, Sequence

import numpy as np
import torch

from . import binding as B
from .inputs import LayerShape
from .layer import make_desc

_SDT = {"f32": B.DTYPE_F32, "f16": B.DTYPE_F16}


class CachedStack:
    def __init__(self, shape: LayerShape, n_layers: int, bits: Sequence[int], n_slots: int, device: int = 0,
                 max_tokens: int = 1, seed: int = 4, policy: int = B.EVICT_FORWARD, beta: float = 4.0,
                 n_prefetch: Optional[int] = None):
        if not torch.cuda.is_available():
            raise RuntimeError("CachedStack needs a CUDA device: there is no CPU path")
        assert shape.act_dtype == "bf16"
        self.shape, self.n_layers, self.bits = shape, n_layers, list(bits)
        self.dev = torch.device("cuda", device)
        torch.cuda.set_device(self.dev)
        self.desc = make_desc(shape)
        self.max_tokens = max_tokens
        self.beta = beta
        self.n_prefetch = shape.top_k if n_prefetch is None else n_prefetch
        self.ctx = B.emoe_create(device, B.emoe_workspace_bytes(self.desc, max_tokens))
        self.compute = torch.cuda.Stream(device=self.dev)
        self.copy = torch.cuda.Stream(device=self.dev)
        E = shape.n_experts
        self.seed = seed
        self._gen = torch.Generator(device=self.dev)
        sdt = torch.float16 if shape.scale_dtype == "f16" else torch.float32
        # experts: seeded N(0, 0.02^2) fp32 on the device -> packed by the library -> pinned host memory
        self.host: List[List[tuple]] = []
        self.expert_bytes = 0
        slot_bytes = 0
        for l in range(n_layers):
            row = []
            for e in range(E):
                pm, sm = [], []
                for m in range(shape.n_matrices):
                    N, K = shape.matrix_shape(m)
                    G = shape.group if shape.group > 0 else K
                    W = self.draw_matrix(l, e, m)
                    p = torch.empty(N * K * self.bits[e] // 8, dtype=torch.uint8, device=self.dev)
                    s = torch.empty(N * (K // G), dtype=sdt, device=self.dev)
                    B.emoe_pack_expert(self.ctx, W.data_ptr(), N, K, self.bits[e], shape.group, _SDT[shape.scale_dtype],
                                       p.data_ptr(), s.data_ptr(), 0)
                    pm.append(p)
                    sm.append(s)
                    del W
                nb = self._nbytes(pm, sm)
                pm, sm = self._pin(pm, sm, nb)
                row.append((pm, sm))
                self.expert_bytes += sum(nb)
                slot_bytes = max(slot_bytes, sum((b + 255) // 256 * 256 for b in nb))
            self.host.append(row)
        self.slot_bytes = slot_bytes
        self.n_slots = n_slots
        B.emoe_cache_create(self.ctx, n_slots, slot_bytes, n_layers, policy)
        for l in range(n_layers):
            for e in range(E):
                pm, sm = self.host[l][e]
                pad = [0] * (3 - len(pm))
                B.emoe_register_expert(self.ctx, self.expert_id(l, e), l, self.bits[e], [t.data_ptr() for t in pm] + pad,
                                       [t.data_ptr() for t in sm] + pad, self._nbytes(pm, sm))
        # routers and the layer-transition prior (row-stochastic, seeded)
        rng = np.random.default_rng(seed)
        self.Wr = [torch.from_numpy((rng.standard_normal((shape.d_model, E)) * 0.02).astype(np.float32)).to(self.dev)
                   for _ in range(n_layers)]
        self._Wr_ptrs = [w.data_ptr() for w in self.Wr]
        prior = rng.random((E, E)) ** 4          # peaked rows: a few likely successors per expert
        self.prior = (prior / prior.sum(axis=1, keepdims=True)).astype(np.float32)
        self._exposed_ns_seen = 0
        self.ids = torch.empty(max_tokens, shape.top_k, dtype=torch.int32, device=self.dev)
        self.gates = torch.empty(max_tokens, shape.top_k, dtype=torch.float32, device=self.dev)
        self.bias = torch.zeros(max_tokens, E, dtype=torch.float32, device=self.dev)
        self.y = torch.empty(max_tokens, shape.d_model, dtype=torch.float32, device=self.dev)
        # picks of a layer and the router bias on their way to and from the device
        self._pin_ids = torch.empty(max_tokens, shape.top_k, dtype=torch.int32, pin_memory=True)
        self._pin_bias = torch.empty(max_tokens, E, dtype=torch.float32, pin_memory=True)
        # one previous pick per token: the bias is a row of a fixed table
        self._bias_rows = (beta * np.log(self.prior[:, None].mean(axis=1) + 1e-9)).astype(np.float32)
        self._bias_rows_dev = torch.from_numpy(self._bias_rows).to(self.dev)
        torch.cuda.synchronize(self.dev)

    def draw_matrix(self, l: int, e: int, m: int) -> torch.Tensor:
        """The fp32 weight matrix m of expert e of layer l (seeded N(0, 0.02^2), drawn on the device)."""
        N, K = self.shape.matrix_shape(m)
        self._gen.manual_seed((self.seed << 32) ^ (l << 16) ^ (e << 4) ^ m)
        return torch.randn(N, K, generator=self._gen, device=self.dev, dtype=torch.float32) * 0.02

    @staticmethod
    def _pin(pm, sm, nb):
        """Copies of the matrices and scales in one pinned block, at the 256-byte boundaries they will have in a cache slot
        (the library then loads an expert with one copy)."""
        at, total = [], 0
        for b in nb:
            at.append(total)
            total += (b + 255) // 256 * 256
        block = torch.empty(total, dtype=torch.uint8, pin_memory=True)

        def put(t, o):
            v = block[o:o + t.numel() * t.element_size()].view(t.dtype)
            v.copy_(t)
            return v

        return [put(t, at[m]) for m, t in enumerate(pm)], [put(t, at[3 + m]) for m, t in enumerate(sm)]

    @staticmethod
    def _nbytes(pm, sm):
        nb = [t.numel() * t.element_size() for t in pm] + [0] * (3 - len(pm))
        return nb + [t.numel() * t.element_size() for t in sm] + [0] * (3 - len(sm))

    def expert_id(self, layer: int, e: int) -> int:
        return layer * self.shape.n_experts + e

    def close(self):
        if self.ctx is not None:
            torch.cuda.synchronize(self.dev)
            B.emoe_destroy(self.ctx)
            self.ctx = None

    def h2d_rate_gbs(self) -> float:
        """Pinned host -> device copy rate of this machine, on one expert's largest matrix."""
        src = max((t for t in self.host[0][0][0]), key=lambda t: t.numel())
        dst = torch.empty(src.numel(), dtype=torch.uint8, device=self.dev)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(self.copy):
            dst.copy_(src, non_blocking=True)
            e0.record()
            for _ in range(4):
                dst.copy_(src, non_blocking=True)
            e1.record()
        e1.synchronize()
        return 4 * src.numel() / (e0.elapsed_time(e1) * 1e-3) / 1e9

    def forward_stack(self, xs: Sequence[torch.Tensor], measure: bool = False, prefetch: bool = True,
                      outputs: Optional[list] = None):
        """One pass of the token batch through all layers.  xs[l]: [T][d] bf16 on the device.
        Returns the picks of every layer (host arrays).  With measure=True the library brackets
        every acquire by two events on the compute stream (emoe_cache_set_timing): their distance is
        the time the compute stream stood still for a load (the exposed copy time).  If `outputs` is a list, every
        layer appends (gates, y) of the batch to it (device tensors of their own)."""
        sh, E = self.shape, self.shape.n_experts
        T = xs[0].shape[0]
        cs, cps = self.compute.cuda_stream, self.copy.cuda_stream
        picks = []
        prev = None
        B.emoe_cache_set_timing(self.ctx, measure)
        host_ids, host_bias = self._pin_ids.numpy()[:T], self._pin_bias.numpy()
        # a batch never needs more of the next layer than every token's share; preloading the whole layer for a few tokens kept
        # the link busy with experts nobody used.  8 steps on inputs the stack has not seen, whole layer -> share, a quarter / half of the
        # experts resident: 6 layers 768 x 3072, 32 experts, 2 tokens 71.0 -> 6.6 / 45.3 -> 4.5 ms, 4 tokens 72.4 -> 11.1 / 45.4 -> 7.6;
        # 4 layers 512 x 1024, 16 experts, 4 tokens 7.4 -> 2.5 / 5.0 -> 2.2; 4 layers 1024 x 3072, 8 experts, 4 tokens 17.6 -> 8.2 / 10.9 -> 4.2
        n_prefetch = min(E, T * self.n_prefetch) if prefetch else 0
        ids_ptr, pin_ids_ptr, prior_ptr = self.ids.data_ptr(), self._pin_ids.data_ptr(), self.prior.ctypes.data
        gates_ptr, y_ptr, gates_step, y_step = self.gates.data_ptr(), self.y.data_ptr(), 0, 0
        with torch.cuda.stream(self.compute):
            if outputs is not None:  # straight into the tensors that are handed out
                gates = torch.empty((self.n_layers, T, sh.top_k), dtype=torch.float32, device=self.dev)
                y = torch.empty((self.n_layers, T, sh.d_model), dtype=torch.float32, device=self.dev)
                outputs.extend(zip(gates.unbind(), y.unbind()))
                gates_ptr, y_ptr, gates_step, y_step = gates.data_ptr(), y.data_ptr(), T * sh.top_k * 4, T * sh.d_model * 4
            for l in range(self.n_layers):
                bias_ptr, stride = None, 0
                if prev is not None:
                    # routing follows the prior: bias[t] = beta * log(mean of the prior rows of t's previous picks)
                    if T == 1 and sh.top_k == 1:
                        bias_ptr, stride = self._bias_rows_dev.data_ptr() + int(prev[0, 0]) * E * 4, E
                    else:
                        if sh.top_k == 1:
                            host_bias[:T] = self._bias_rows[prev[:, 0]]
                        else:
                            host_bias[:T] = self.beta * np.log(self.prior[prev].mean(axis=1) + 1e-9)
                        self.bias[:T].copy_(self._pin_bias[:T], non_blocking=True)
                        bias_ptr, stride = self.bias.data_ptr(), E
                more = l + 1 < self.n_layers
                B.emoe_cached_layer(self.ctx, self.desc, l, xs[l].data_ptr(), T, self._Wr_ptrs[l], bias_ptr, stride,
                                    self.expert_id(l, 0), prior_ptr if more else None, n_prefetch, self.expert_id(l + 1, 0),
                                    ids_ptr, gates_ptr + l * gates_step, y_ptr + l * y_step, pin_ids_ptr, cs, cps)
                prev = host_ids.copy()
                picks.append(prev)
        return picks

    def exposed_ms(self) -> float:
        """Sum of the compute-stream stalls the library measured since the last call (synchronises)."""
        self.compute.synchronize()
        ns = B.emoe_cache_get_stats(self.ctx)["exposed_copy_ns"]
        ms = (ns - self._exposed_ns_seen) * 1e-6
        self._exposed_ns_seen = ns
        return ms
