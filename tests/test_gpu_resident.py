"""Batch-1 host-free steps as one cooperative kernel: the bits, events and statistics of host-driven steps at the edges of its
exchanges (owned columns, rows over all CTAs, more experts than threads) and of its shared-memory layouts."""
import threading

import numpy as np
import pytest
import torch

import synth
from paper_2607_24787_b200 import binding as B
from paper_2607_24787_b200.binding import SpmError
from test_gpu_host_free import build, preload, rows, run

pytestmark = pytest.mark.gpu

# hidden: one 16-column owner a 16 columns, 8 to 128 of them; inter * top_k: CTAs without a row, with one, with ragged shares; n_experts:
# ranked by two threads each, from 3 to more than the threads, and more rows than warps of all CTAs; odd adapter ranks.
CASES = {
    "fp32_smallest": dict(base="tiny", hidden=128, n_experts=3, inter=7, top_k=1, adapter_rank=1),
    "fp32_widest": dict(base="tiny", hidden=1024, n_experts=20, inter=331, top_k=4, adapter_rank=7),
    "fp32_shared": dict(base="tiny", hidden=640, n_experts=37, inter=50, top_k=3, n_shared=2, adapter_rank=5),
    "bf16_widest": dict(base="qwen3", hidden=2048, n_experts=24, inter=129, top_k=8, adapter_rank=16),
    "bf16_many_experts": dict(base="qwen3", hidden=256, n_experts=600, inter=24, top_k=16, adapter_rank=3),
    "bf16_row_in_ring": dict(base="qwen3", hidden=2048, n_experts=513, inter=10, top_k=2, adapter_rank=63),
    "bf16_nine_warps": dict(base="dsvl2", hidden=1280, n_experts=16, inter=224, top_k=6, n_shared=2, adapter_rank=16),
    "q4_narrow": dict(base="qwen3_q4", hidden=256, n_experts=12, inter=96, top_k=3, adapter_rank=4),
    "q4_shared": dict(base="dsvl2_q4", hidden=1280, n_experts=16, inter=224, top_k=6, n_shared=2, adapter_rank=16),
    "q4_widest": dict(base="qwen3_q4", hidden=2048, n_experts=20, inter=450, top_k=8, adapter_rank=16),
    "q4_many_experts": dict(base="qwen3_q4", hidden=768, n_experts=300, inter=33, top_k=10, adapter_rank=2),
    # owners of columns, and the CTA that ranks the adapter's logits, without a row
    "q4_fewer_rows_than_ctas": dict(base="qwen3_q4", hidden=2048, n_experts=128, inter=9, top_k=3, adapter_rank=16),
    "q4_one_row": dict(base="qwen3_q4", hidden=512, n_experts=100, inter=1, top_k=1, adapter_rank=40),
    "q4_ring_of_three": dict(base="qwen3_q4", hidden=2048, n_experts=12, inter=896, top_k=8, adapter_rank=16),       # (three and four tiles)
    "q4_ring_of_three_full": dict(base="qwen3_q4", hidden=2048, n_experts=128, inter=1024, top_k=8, adapter_rank=16),
    "q4_ring_of_three_shared": dict(base="qwen3_q4", hidden=2048, n_experts=12, inter=768, top_k=8, n_shared=2, adapter_rank=16),
    "q4_ring_of_three_long": dict(base="qwen3_q4", hidden=2048, n_experts=9, inter=1600, top_k=8, adapter_rank=16),
    "q4_ring_of_five": dict(base="qwen3_q4", hidden=1536, n_experts=10, inter=1517, top_k=8, adapter_rank=16),
    "q4_ring_of_seven": dict(base="qwen3_q4", hidden=1024, n_experts=9, inter=2202, top_k=8, adapter_rank=16),
    "bf16_raw_weights": dict(base="qwen3", hidden=1792, n_experts=9, inter=100, top_k=3, renormalize=0, adapter_rank=4),
}


def config(name, **over):
    kw = dict(CASES[name], **over)
    n = kw["n_experts"]
    return synth.get_config(kw.pop("base"), n_layers=3, slots=n, budget=2, batch=1, **kw)


@pytest.mark.parametrize("policy", ["adapter", "on_demand"])
@pytest.mark.parametrize("name", list(CASES))
def test_one_kernel_gives_the_bits_of_host_driven_steps(name, policy):
    cfg = config(name)
    steps = 10                      # more than the trace ring holds
    H = rows(cfg, steps)
    results = []
    for host_free in (1, 0):
        m = build(cfg, store_layers=1)
        m.set_host_free(host_free)
        m.set_policy(policy)
        preload(cfg, m)
        m.reset_stats()
        outs = run(m, H, sync_every=0 if host_free else 1)
        st = m.stats()
        assert st["host_free_steps"] == (steps if host_free else 0) and st["ffn_launches"] == steps * cfg.n_layers
        assert st["kernel_launches"] == (steps if host_free else steps * (2 * cfg.n_layers + 1))
        results.append((outs, m.events(), {k: st[k] for k in ("hits", "touches", "steps", "tokens", "recall_sum", "ready_sum")}))
        m.close()
    (a, ev_a, st_a), (b, ev_b, st_b) = results
    for s in range(steps):
        assert np.array_equal(a[s], b[s]), s
    assert ev_a == ev_b and st_a == st_b


@pytest.mark.parametrize("base,n,k", [("tiny", 3, 3), ("tiny", 32, 2), ("bf16_nine_warps", 97, 6), ("q4_widest", 128, 8), ("tiny", 129, 4),
                                      ("tiny", 33, 3), ("tiny", 64, 4), ("tiny", 65, 2), ("bf16_nine_warps", 64, 6), ("q4_widest", 63, 5), ("q4_widest", 65, 8),
                                      ("fp32_widest", 128, 4), ("fp32_widest", 129, 4), ("bf16_nine_warps", 65, 2)])
def test_equal_logits_go_to_the_lower_id(base, n, k):
    """Experts with one and the same router row, on both sides of the number that a warp ranks by itself: the lowest ids of the largest logit,
    in order, as in host-driven steps."""
    if base == "tiny":
        cfg = synth.get_config("tiny", n_layers=3, n_experts=n, top_k=k, slots=n, budget=2, batch=1)
    else:
        cfg = config(base, n_experts=n, top_k=k, inter=64)
    H = rows(cfg, 3)
    results = []
    for host_free in (1, 0):
        m = build(cfg, store_layers=1)
        w = m._keep[1]
        w[:, 1::2] = w[:, 1:2].clone()                # every second expert like expert 1, ...
        w[2] = w[2, :1].clone()                       # ... and all of the last layer's alike
        torch.cuda.synchronize()
        m.set_host_free(host_free)
        preload(cfg, m)
        outs = run(m, H)
        _, ids, _, logits = m.router_topk(2, torch.as_tensor(H[0], dtype=torch.float32).cuda(), want_logits=True)
        assert list(ids[0]) == list(range(k))
        results.append((outs, m.events()))
        m.close()
    (a, ev_a), (b, ev_b) = results
    for s in range(3):
        assert np.array_equal(a[s], b[s]), s
    assert ev_a == ev_b


def test_other_launches_in_between_and_rows_from_anywhere():
    """The exchange words share memory with other kernels' partial rows: steps before and after such kernels, in place, from rows
    at any float and from pinned host rows."""
    cfg = config("bf16_nine_warps")
    H = torch.as_tensor(rows(cfg, 4), dtype=torch.float32).cuda()
    m = build(cfg, store_layers=1)
    preload(cfg, m)
    torch.cuda.synchronize()
    want = [m.decode_step(H[s]) for s in range(4)]
    m.synchronize()
    want = [w.clone() for w in want]
    x, ids, w, _ = m.router_topk(0, H[0])
    scratch = H[0].clone()
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, scratch)            # writes partial rows
    in_place = H[1].clone()
    odd = torch.empty(cfg.hidden + 1, device="cuda")
    odd[1:].copy_(H[2][0])
    torch.cuda.synchronize()
    third = torch.empty_like(H[2])
    got = [m.decode_step(H[0]), m.decode_step(in_place, in_place), m.decode_step(odd[1:].view(1, -1), third)]
    m.set_timing(1)                             # the separate launches
    timed = m.decode_step(H[3])
    m.set_timing(0)
    got.append(m.decode_step(H[3]))
    host = torch.empty(1, cfg.hidden).pin_memory()
    m.decode_step_host(H[3].cpu().pin_memory(), host)
    m.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert torch.equal(timed, want[3]) and torch.equal(host.cuda(), want[3])
    m.close()


def test_non_finite_logits_are_reported_once():
    cfg = config("fp32_shared")
    m = build(cfg, store_layers=1)
    preload(cfg, m)
    h = torch.as_tensor(rows(cfg, 1)[0], dtype=torch.float32).cuda()
    torch.cuda.synchronize()
    want = m.decode_step(h)
    m.synchronize()
    want = want.clone()
    bad = h.clone()
    bad[0, 3] = float("nan")
    torch.cuda.synchronize()
    m.decode_step(bad)
    with pytest.raises(SpmError) as e:
        m.synchronize()
    assert e.value.code == -7
    got = m.decode_step(h)
    m.synchronize()
    assert torch.equal(got, want)
    m.close()


def test_two_contexts_at_once():
    """Two threads, each with a context and streams of its own: both kernels want every SM, one waits for the other."""
    cfg = config("bf16_nine_warps")
    H = rows(cfg, 24)
    ms = [build(cfg, store_layers=1) for _ in range(2)]
    for m in ms:
        preload(cfg, m)
    want = run(ms[0], H)
    outs = [None, None]

    def work(i):
        outs[i] = run(ms[i], H)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for o in outs:
        for a, b in zip(o, want):
            assert np.array_equal(a, b)
    for m in ms:
        m.close()


@pytest.mark.parametrize("name", ["fp32_widest", "bf16_nine_warps", "q4_widest", "q4_shared"])
def test_expert_without_a_slot_is_reported(name):
    """A slot map that names no slot for a routed expert (written over here, where the step reads it) is a bad slot, not a shared expert."""
    cfg = config(name)
    m = build(cfg, store_layers=1)
    preload(cfg, m)
    h = torch.as_tensor(rows(cfg, 1)[0], dtype=torch.float32).cuda()
    torch.cuda.synchronize()
    want = m.decode_step(h)
    m.synchronize()
    used = m.router_topk(0, h)[1][0]
    m.synchronize()
    table = np.full((cfg.n_layers, cfg.n_experts), -1, np.int16)
    for l in range(cfg.n_layers):
        in_slot = m.slot_table(l)
        for slot, e in enumerate(in_slot):
            if e >= 0:
                table[l, e] = slot
    at = m.arena.cpu().numpy().tobytes().rindex(table.tobytes())
    entry = m.arena[at + 2 * int(used[-1]):at + 2 * int(used[-1]) + 2]
    saved = entry.clone()
    entry.fill_(255)                    # -1
    torch.cuda.synchronize()
    m.decode_step(h)
    with pytest.raises(SpmError) as e:
        m.synchronize()
    assert e.value.code == -5
    entry.copy_(saved)
    torch.cuda.synchronize()
    got = m.decode_step(h)
    m.synchronize()
    assert torch.equal(got, want)
    m.close()


def test_compute_stream_that_may_not_use_all_sms():
    """Where the CTAs of the one-kernel step cannot all be running at once, the step is separate launches with the same bits."""
    cu = pytest.importorskip("cuda.bindings.driver")

    def ok(result):
        if result[0] != cu.CUresult.CUDA_SUCCESS:
            pytest.skip(f"no green contexts here: {result[0]}")
        return result[1] if len(result) > 1 else None

    cfg = config("bf16_nine_warps")
    H = torch.as_tensor(rows(cfg, 3), dtype=torch.float32).cuda()
    m = build(cfg, store_layers=1)
    preload(cfg, m)
    torch.cuda.synchronize()
    want = [m.decode_step(h) for h in H]
    m.synchronize()
    assert m.stats()["kernel_launches"] == 3
    dev = ok(cu.cuDeviceGet(torch.cuda.current_device()))
    sms = ok(cu.cuDeviceGetDevResource(dev, cu.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    part = ok(cu.cuDevSmResourceSplitByCount(1, sms, 0, 72))
    green = ok(cu.cuGreenCtxCreate(ok(cu.cuDevResourceGenerateDesc(part, 1)), dev, cu.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream = ok(cu.cuGreenCtxStreamCreate(green, cu.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    ptr = [t.data_ptr() if t is not None else None for t in m._keep[:5]]
    B.spm_destroy(m.ctx)
    m.ctx = B.spm_init(m.cfg, m.slots, 0, B.Buffers(*ptr, m.store.ptr, (m.arena.data_ptr() + 255) // 256 * 256, m.arena.numel() - 256,
                                                    int(stream), m.copy.cuda_stream, 1))
    preload(cfg, m)
    got = [m.decode_step(h) for h in H]
    m.synchronize()
    st = m.stats()
    assert st["host_free_steps"] == 3 and st["kernel_launches"] == 3 * (2 * cfg.n_layers + 1)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    m.close()
    ok(cu.cuStreamDestroy(stream))
    ok(cu.cuGreenCtxDestroy(green))


# many experts of a few rows: with the routing weights in host memory a layer's logits take tens of microseconds to arrive
SLOW = {
    "fp32": dict(base="tiny", hidden=1024, n_experts=900, inter=8, top_k=4, adapter_rank=16),
    "bf16_shared": dict(base="dsvl2", hidden=1280, n_experts=900, inter=40, top_k=4, n_shared=2, adapter_rank=16),
    "bf16_widest": dict(base="qwen3", hidden=2048, n_experts=700, inter=16, top_k=8, adapter_rank=16),
    "q4": dict(base="qwen3_q4", hidden=2048, n_experts=700, inter=64, top_k=8, adapter_rank=16),
}


@pytest.mark.parametrize("name", list(SLOW))
def test_exchange_that_runs_out(name):
    """A limit of a microsecond, and logits that take longer: the CTAs give up, with rows of shared experts on their way in one case, the host reads
    the time-out once, and the next step has the bits of any other."""
    kw = dict(SLOW[name])
    cfg = synth.get_config(kw.pop("base"), n_layers=3, slots=kw["n_experts"], budget=2, batch=1, **kw)
    m = build(cfg, store_layers=1)
    preload(cfg, m)
    h = torch.as_tensor(rows(cfg, 1)[0], dtype=torch.float32).cuda()
    torch.cuda.synchronize()
    want = m.decode_step(h)
    m.synchronize()
    slow = m._keep[1].cpu().pin_memory()
    ptr = [t.data_ptr() if t is not None else None for t in m._keep[:5]]
    B.spm_destroy(m.ctx)
    m.ctx = B.spm_init(m.cfg, m.slots, 0, B.Buffers(ptr[0], slow.data_ptr(), *ptr[2:], m.store.ptr, (m.arena.data_ptr() + 255) // 256 * 256,
                                                    m.arena.numel() - 256, m.compute.cuda_stream, m.copy.cuda_stream, 1))
    preload(cfg, m)
    for _ in range(2):
        got = m.decode_step(h)
        m.synchronize()
        assert torch.equal(got, want)
        m.set_device_wait_limit_us(1)
        m.decode_step(h)
        with pytest.raises(SpmError) as e:
            m.synchronize()
        assert e.value.code == -4 and "another of its CTAs" in str(e.value)
        m.synchronize()                         # reported once
        m.set_device_wait_limit_us(0)
    got = m.decode_step(h)
    m.synchronize()
    assert torch.equal(got, want) and m.stats()["kernel_launches"] == 5
    m.close()


def test_clock_slots_and_exchange_share_memory():
    """More timed launches than there are clock slots ahead of the exchange, then one-kernel steps, and both again: no window is lost to the
    other's words and no word to a window."""
    cfg = config("fp32_smallest")
    m = build(cfg, store_layers=1)
    preload(cfg, m)
    h = torch.as_tensor(rows(cfg, 1)[0], dtype=torch.float32).cuda()
    torch.cuda.synchronize()
    want = m.decode_step(h)
    m.synchronize()
    steps = 8192 // (2 * cfg.n_layers + 1) + 100
    m.reset_stats()
    for done in (1, 2):
        m.set_timing(1)
        for _ in range(steps):
            m.decode_step(h)
        m.set_timing(0)
        got = m.decode_step(h)
        m.synchronize()
        assert torch.equal(got, want)
        st = m.stats()
        assert st["kernel_launches"] == done * (steps * (2 * cfg.n_layers + 1) + 1)
        for key in ("ffn_window_us", "router_window_us"):
            assert 0.5 < st[key] / (done * steps * cfg.n_layers) < 100, key
    m.close()
