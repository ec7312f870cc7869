"""Calls on one stream see what the calls before them wrote, also where the kernels in between overlap: the weights of one context are the
output of another one's expert kernels, whose combine kernel lets its successor start before it has written."""
import numpy as np
import pytest
import torch

import synth
from paper_2607_24787_b200 import binding as B
from test_gpu_edges import build

pytestmark = pytest.mark.gpu


def writer(hidden):
    """A context whose moe_ffn adds an expert's output to a row of `hidden` floats, and such a call."""
    cfg = synth.get_config("tiny", n_layers=1, hidden=hidden, n_experts=4, inter=300, top_k=1, slots=4)
    m = build(cfg)
    x, ids, w = torch.randn(1, hidden, device="cuda"), np.zeros((1, 1), np.int32), torch.ones(1, 1, device="cuda")
    m.moe_ffn(0, x, ids, w, torch.zeros(1, hidden, device="cuda"))      # (the expert is in HBM from here on)
    m.synchronize()
    return m, lambda row: m.moe_ffn(0, x, ids, w, row)


def on_stream_of(other, cfg):
    """A context on `other`'s compute stream, and its weights [gamma, router_w, adapter_a, adapter_b, shared experts]."""
    m = build(cfg)
    ptr = [t.data_ptr() if t is not None else None for t in m._keep[:5]]
    B.spm_destroy(m.ctx)
    m.compute = other.compute
    m.ctx = B.spm_init(m.cfg, m.slots, 0, B.Buffers(*ptr, m.store.ptr, (m.arena.data_ptr() + 255) // 256 * 256, m.arena.numel() - 256,
                                                    m.compute.cuda_stream, m.copy.cuda_stream, 0))
    return m, m._keep[:5]


def same_as_after_a_pause(call, row, a, write):
    """call() right behind a call that writes `row`, and again when all is quiet."""
    for _ in range(5):
        row.zero_()
        torch.cuda.synchronize()
        call()
        a.synchronize()
        write(row)
        first = call()
        a.synchronize()
        second = call()
        a.synchronize()
        for p, q in zip(first, second):
            assert torch.equal(p.view(torch.int32), q.view(torch.int32)) if torch.is_tensor(p) else np.array_equal(p, q)


def test_router_and_adapter_read_weights_written_just_before():
    a, write = writer(256)
    m, (gamma, router_w, adapter_a, _, _) = on_stream_of(a, synth.get_config("tiny", n_layers=2, hidden=256))
    h = torch.randn(1, 256, device="cuda")
    torch.cuda.synchronize()
    x = m.router_topk(0, h)[0]

    def route():
        x2, ids, w, logits = m.router_topk(0, h, want_logits=True)
        return [x2, w, logits, ids]

    same_as_after_a_pause(route, gamma[0:1], a, write)
    gamma.fill_(1)
    same_as_after_a_pause(route, router_w[0, 3:4], a, write)
    same_as_after_a_pause(lambda: [x.new_tensor(t) if t.dtype == np.float32 else t for t in m.adapter_predict(0, x)], adapter_a[0, 2:3], a, write)
    m.close()
    a.close()


def test_4bit_shared_experts_written_just_before():
    a, write = writer(256)
    cfg = synth.get_config("dsvl2_q4", n_layers=1, hidden=256, n_experts=4, inter=64, top_k=1, n_shared=2, slots=4, batch=1, budget=0, adapter_rank=2)
    m, weights = on_stream_of(a, cfg)
    blobs = weights[4].view(-1)
    x, ids, w = torch.randn(1, 256, device="cuda"), np.zeros((1, 1), np.int32), torch.ones(1, 1, device="cuda")
    m.prefetch_async(0, ids[0])
    m.synchronize()

    outs = iter(torch.zeros(15, 1, 256, device="cuda"))

    def ffn():
        out = next(outs)
        m.moe_ffn(0, x, ids, w, out)
        return [out]

    half = blobs.numel() // 2 // 16 * 16            # in the second shared expert: the rows of the last CTAs
    same_as_after_a_pause(ffn, blobs[half:half + 1024].view(torch.float32).view(1, 256), a, write)
    m.close()
    a.close()
