"""The decode workloads whose speed this library is judged by.

A case names a model shape, where its experts are (`slots` cache slots per layer; `slots` >= `experts`
means that everything fits into HBM), how many sequences are decoded together and which entry point is
called. One pass is one decode step: `batch` hidden rows through all layers of the model. The shapes are
the ones of `synth.gen.CONFIGS` with fewer layers (a layer costs the same wherever it stands), so that a
model is built in about a second.

Weights are N(0, 0.02), hidden rows N(0, 1) rounded to the weight type: rows of an embedding table, one per
distinct token, for token ids drawn from Zipf(1.1) over the vocabulary, so popular tokens repeat within a
batch and from one step to the next.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_24787_b200.model import OffloadedMoE, PinnedStore, pack_experts_q4

VOCAB, ZIPF_A = 151936, 1.1
STEPS = 16          # distinct decode steps a state holds; pass i takes step i % STEPS
BUDGET = 1          # prefetches per layer: what the profiled window gives on this machine

QWEN3 = dict(hidden=2048, experts=128, inter=768, top_k=8, shared=0)
DSVL2 = dict(hidden=1280, experts=64, inter=896, top_k=6, shared=2)
TINY = dict(hidden=256, experts=16, inter=128, top_k=2, shared=0)


def _case(name, shape, dtype, layers, slots, batch, policy, entry):
    return dict(name=name, **shape, dtype=dtype, layers=layers, slots=slots, batch=batch, policy=policy, entry=entry)


def listed():
    return [
        # the fp32 parity model, one sequence, host rows in and out: nothing but latency
        _case("tiny_offload", TINY, "fp32", 2, 4, 1, "adapter", "host"),
        # the headline: one sequence, experts in pinned host memory, adapter-guided prefetch, host rows in and out
        _case("qwen3_offload", QWEN3, "bf16", 4, 16, 1, "adapter", "host"),
        # the on-device setting of the method: 4-bit experts, two shared ones, a small cache
        _case("dsvl2_q4_offload", DSVL2, "q4", 12, 8, 1, "adapter", "device"),
        # a serving batch whose demand exceeds the cache: every layer runs in waves
        _case("batch64_offload", QWEN3, "bf16", 2, 32, 64, "adapter", "device"),
        # one sequence with every expert in HBM: what latency-bound serving does when the model fits
        _case("qwen3_resident", QWEN3, "bf16", 12, 128, 1, "adapter", "device"),
        _case("dsvl2_resident", DSVL2, "bf16", 12, 64, 1, "on_demand", "device"),
        _case("qwen3_q4_resident", QWEN3, "q4", 12, 128, 1, "adapter", "device"),
        # serving batches with every expert in HBM: a few sequences (odd), the full batch, both weight types
        _case("batch5_resident", QWEN3, "bf16", 6, 128, 5, "adapter", "device"),
        _case("batch64_resident", QWEN3, "bf16", 6, 128, 64, "adapter", "device"),
        _case("batch64_q4_resident", QWEN3, "q4", 6, 128, 64, "on_demand", "device"),
        # a batch of the shape with shared experts
        _case("dsvl2_batch16_resident", DSVL2, "bf16", 6, 64, 16, "on_demand", "device"),
        # the stand-alone calls layer by layer, as a calibration pass or a custom serving loop makes them
        _case("dsvl2_layer_calls", DSVL2, "bf16", 12, 64, 1, "adapter", "calls"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the listed shapes or odd ones, any cache size, 1 to 64 sequences, every weight type."""
    base = rng.choice((QWEN3, DSVL2, TINY, None, None))
    if base is None:
        hidden = 256 * rng.randint(1, 8)
        experts = rng.choice((12, 24, 60, 64, 96, 128))
        top_k = rng.randint(1, min(8, experts))
        # intermediate sizes that tile by 128 and ones that do not
        inter = 128 * rng.randint(1, 8) if rng.random() < 0.6 else rng.randint(96, 1000)
        base = dict(hidden=hidden, experts=experts, inter=inter, top_k=top_k, shared=rng.choice((0, 0, 0, 1, 2)))
    dtype = "fp32" if base is TINY else rng.choice(("bf16", "bf16", "q4", "q4", "fp32"))
    if base["hidden"] > 1024 and dtype == "fp32":
        dtype = "bf16"
    batch = _log_int(rng, 1, 64) if rng.random() < 0.6 else 1
    offload = rng.random() < 0.35
    slots = base["experts"] if not offload else rng.randint(base["top_k"], max(base["top_k"], base["experts"] // 2))
    layers = rng.randint(2, 8)
    entry = rng.choice(("device", "device", "host", "calls")) if batch <= 16 else "device"
    c = dict(**base, dtype=dtype, layers=layers, slots=slots, batch=batch,
             policy=rng.choice(("adapter", "adapter", "on_demand", "naive")), entry=entry)
    if entry == "calls":
        c["policy"] = "adapter"
    # no dearer than the largest listed case: an offloaded step moves at most two layers of the large shape
    limit = 2.4e9 if offload else 8e9
    while c["layers"] > 2 and c["layers"] * c["experts"] * _blob_bytes(c) > limit:
        c["layers"] -= 1
    return c


# ---- sizes -------------------------------------------------------------------
def _blob_bytes(c):
    per_row = c["hidden"] // 2 + c["hidden"] // 16 if c["dtype"] == "q4" else c["hidden"] * (4 if c["dtype"] == "fp32" else 2)
    return 3 * c["inter"] * per_row


def _zipf_p():
    p = np.arange(1, VOCAB + 1, dtype=np.float64) ** -ZIPF_A
    return p / p.sum()


def _distinct_experts(c):
    """Expected number of distinct routed experts of a layer: distinct tokens of the batch, each with its own top_k."""
    tokens = float(np.sum(1.0 - (1.0 - _zipf_p()) ** c["batch"]))
    return c["experts"] * (1.0 - (1.0 - c["top_k"] / c["experts"]) ** tokens)


def work(case):
    """Every weight a step needs once (experts, gate, adapters), the rows in and out; two operations per weight and row."""
    c = case
    e = 4 if c["dtype"] == "fp32" else 2
    rank = 16
    weights = 3 * c["inter"] * c["hidden"]
    per_layer = (_distinct_experts(c) + c["shared"]) * _blob_bytes(c) + c["experts"] * c["hidden"] * e
    adapters = (rank * c["hidden"] + c["experts"] * rank) * e * (c["layers"] - 1) if c["policy"] == "adapter" else 0
    rows = c["batch"] * c["hidden"] * 4 * 2
    flops = 2 * c["batch"] * c["layers"] * ((c["top_k"] + c["shared"]) * weights + c["experts"] * c["hidden"])
    return {"bytes": c["layers"] * per_layer + adapters + rows, "flops": flops}


def _bf16_activations(c):
    """Whether the step runs on the tensor-core path, which rounds activations to bf16 (spm_set_batched_path)."""
    return (c["batch"] > 1 and c["shared"] == 0 and c["dtype"] != "fp32" and c["inter"] % 128 == 0
            and c["hidden"] % (256 if c["dtype"] == "q4" else 128) == 0)


def tolerance(case):
    """fp32 activations: four times what another summation order shows (4e-7 of what the layers add, 1e-6 at the worst
    element), with room for the sums of wider models. bf16 activations against fp32 ones: 4e-4 to 7e-4, and up to 1e-2
    (0.2 at one element) where the rounding tips one token's last expert."""
    if _bf16_activations(case):
        return {"rel": 1e-2, "max": 0.4, "differ": 0.005}
    return {"rel": 1e-5, "max": 4e-4}


# ---- inputs ------------------------------------------------------------------
def _randn(gen, shape, dtype, scale):
    return torch.randn(shape, generator=gen, device="cuda", dtype=dtype).mul_(scale)


def _quantize(w):
    """Symmetric 4 bit along the last dimension, groups of 32: value = scale * (q - 8)."""
    g = w.float().reshape(*w.shape[:-1], -1, 32)
    scale = (g.abs().amax(-1) / 7.0).half()
    q = (torch.round(g / scale.float().unsqueeze(-1)) + 8).clamp_(0, 15).to(torch.uint8)
    return q.reshape(w.shape), scale


def _experts(gen, c, count):
    """`count` packed expert blobs, flat bytes."""
    shape = (count, c["inter"], c["hidden"])
    if c["dtype"] == "q4":
        parts = [_quantize(_randn(gen, shape, torch.bfloat16, 0.02)) for _ in range(3)]
        return pack_experts_q4(*parts).reshape(-1)
    dtype = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    return _randn(gen, (count, c["inter"], 3, c["hidden"]), dtype, 0.02).view(torch.uint8).reshape(-1)


class _State:
    pass


def prepare(case, seed):
    """The model with its expert store filled (and, where it fits, its experts in HBM) and the rows of STEPS decode steps."""
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    L, n, D, rank = c["layers"], c["experts"], c["hidden"], 16
    # one layer of experts on the host serves all layers (host_store_layers): sizes and traffic are those of a full store
    store = PinnedStore(n * _blob_bytes(c))
    chunk = 16
    for e0 in range(0, n, chunk):
        blobs = _experts(gen, c, min(chunk, n - e0))
        at = e0 * _blob_bytes(c)
        store.tensor[at:at + blobs.numel()].copy_(blobs, non_blocking=True)
    s = _State()
    shared = torch.cat([_experts(gen, c, c["shared"]) for _ in range(L)]) if c["shared"] else None
    s.m = OffloadedMoE(n_layers=L, hidden=D, n_experts=n, inter=c["inter"], top_k=c["top_k"], n_shared=c["shared"],
                       adapter_rank=rank, dtype={"fp32": torch.float32, "bf16": "bf16", "q4": "q4"}[c["dtype"]],
                       renormalize=1, rms_eps=1e-6, max_batch=c["batch"], slots=c["slots"], budget=BUDGET,
                       gamma=1.0 + _randn(gen, (L, D), torch.float32, 0.1), router_w=_randn(gen, (L, n, D), dtype, 0.02),
                       adapter_a=_randn(gen, (L - 1, rank, D), dtype, 0.02), adapter_b=_randn(gen, (L - 1, n, rank), dtype, 0.02),
                       shared_blobs=shared, store=store, store_layers=1)
    s.m.set_policy(c["policy"])
    if c["slots"] >= n:
        for l in range(L):
            s.m.prefetch_async(l, np.arange(n, dtype=np.int32))
    s.m.synchronize()
    ids = np.searchsorted(np.cumsum(_zipf_p()), np.random.default_rng(seed).random(STEPS * c["batch"]))
    _, inverse = np.unique(ids, return_inverse=True)
    table = _randn(gen, (int(inverse.max()) + 1, D), dtype, 1.0).float()
    s.rows = table[torch.from_numpy(inverse.reshape(-1)).cuda()].view(STEPS, c["batch"], D).contiguous()
    s.out = torch.empty(c["batch"], D, device="cuda")
    s.entry, s.at = c["entry"], 0
    if s.entry == "host":
        s.rows, s.out = s.rows.cpu().pin_memory(), torch.empty(c["batch"], D).pin_memory()
    torch.cuda.synchronize()
    return s


def run(state):
    s, m = state, state.m
    rows = s.rows[s.at % STEPS]
    s.at += 1
    if s.entry == "host":
        return m.decode_step_host(rows, s.out)
    # the rows come from, and the result goes to, work on the caller's stream (embedding, output head)
    stream = torch.cuda.current_stream()
    if s.entry == "device":
        m.compute.wait_stream(stream)
        m.decode_step(rows, s.out)
        stream.wait_stream(m.compute)
        return s.out
    s.out.copy_(rows)
    m.compute.wait_stream(stream)
    all_ids, all_scores, last = [], [], None
    for l in range(m.L):
        x, ids, w, last = m.router_topk(l, s.out, want_logits=True)
        m.moe_ffn(l, x, ids, w, s.out)
        if l + 1 < m.L:
            scores, order = m.adapter_predict(l, x)
            m.prefetch_async(l + 1, m.budget_select(l + 1, order))
            all_scores.append(scores)
        all_ids.append(np.sort(ids, axis=1))
    stream.wait_stream(m.compute)
    return {"h": s.out, "ids": np.stack(all_ids), "scores": np.stack(all_scores), "logits": last}
