"""The several-sequences expert kernel with fp32 activations (fp32 weights, shared experts, sizes that do not tile by
128) at the edges of its blocks, token runs and column groups, each against the CPU oracle."""
import time

import numpy as np
import pytest
import torch

import synth
from paper_2607_24787_b200 import binding as B
from paper_2607_24787_b200.binding import SpmError
from test_gpu_edges import build, compare_run
from test_gpu_host_free import preload, rows, run

pytestmark = pytest.mark.gpu

# Tokens of an expert: runs of eight, one MMA per tile up to two tokens of a run and three above. Rows: blocks of eight.
# Columns: groups of 32 over eight warps. The kernel takes over where enough weights are not read again (takes_kernel),
# hence few experts and many tokens.
CASES = {
    # every expert in every token: 64 = 8 full runs; 17 = two runs and one token; 10 = one run and two; 11 = ... and three
    "fp32_all_experts": dict(base="tiny", hidden=256, n_experts=3, inter=463, top_k=3, slots=3, batch=64),
    "fp32_run_of_one": dict(base="tiny", hidden=1024, n_experts=4, inter=460, top_k=4, slots=4, batch=17),
    "fp32_idle_last_group": dict(base="tiny", hidden=384, n_experts=6, inter=511, top_k=3, slots=6, batch=48),
    "fp32_half_the_warps": dict(base="tiny", hidden=128, n_experts=12, inter=461, top_k=8, slots=12, batch=64),       # four groups of columns
    "bf16_run_of_two": dict(base="qwen3", hidden=2048, n_experts=4, inter=401, top_k=4, slots=4, batch=10),
    "bf16_run_of_three": dict(base="qwen3", hidden=1280, n_experts=4, inter=601, top_k=4, slots=4, batch=11),
    "bf16_shared_waves": dict(base="dsvl2", hidden=1280, n_experts=12, inter=250, top_k=3, slots=5, batch=29),
    "bf16_narrow": dict(base="qwen3", hidden=256, n_experts=9, inter=743, top_k=2, slots=9, batch=64),
    "q4_narrow": dict(base="qwen3_q4", hidden=256, n_experts=7, inter=777, top_k=2, slots=7, batch=64),
    "q4_shared": dict(base="dsvl2_q4", hidden=1280, n_experts=6, inter=263, top_k=2, slots=6, batch=23),
    "q4_widest_waves": dict(base="qwen3_q4", hidden=2048, n_experts=9, inter=129, top_k=3, slots=4, batch=32),
}


def takes_kernel(cfg, nb):
    """The rule by which a batch that keeps fp32 activations is given to this kernel."""
    expert = 3 * cfg.inter * cfg.hidden
    distinct = min(nb * cfg.top_k, cfg.n_experts) + cfg.n_shared
    reads, computed = nb * (cfg.top_k + cfg.n_shared) * expert, distinct * expert
    if reads - computed < 64 << 20:
        return False
    if cfg.dtype == "bf16":
        return reads - computed >= (59 << 20) + cfg.hidden * 8192
    if cfg.dtype == "q4":
        return reads - computed >= computed // 4096 * cfg.hidden
    cols = -(-cfg.hidden // 256) * 256
    return 4 * reads >= 5 * computed // cfg.hidden * (cols + 256) + 4 * ((12 << 20) + 3 * cols * 16384)


def config(name):
    kw = dict(CASES[name])
    cfg = synth.get_config(kw.pop("base"), n_layers=2, budget=1, **kw)
    assert takes_kernel(cfg, cfg.batch), "this shape would take the other kernel"
    return cfg


@pytest.mark.parametrize("name", list(CASES))
def test_several_sequences_match_the_oracle(name):
    # fp32 sums of at most 2048 terms, in blocks of 16 or 32: some 1e-6 of the largest element, as on the batch-1 path
    compare_run(config(name), steps=2, tol=4e-5 if name.startswith("fp32") else 4e-4)


@pytest.mark.parametrize("name", ["fp32_run_of_one", "bf16_shared_waves", "q4_shared", "q4_narrow"])
def test_several_sequences_equal_one_at_a_time(name):
    """Same weights and rows through the batch-1 kernel: both keep activations and sums in fp32. The sums are taken in
    another order, so they differ by the roundings of some hundred additions: 5e-6 of the largest element is ample."""
    cfg = config(name)
    m = build(cfg, slots=cfg.n_experts)
    tok = synth.zipf_tokens(cfg, steps=1)
    h = synth.embedding_rows(cfg, tok.reshape(-1)).float().cuda()
    torch.cuda.synchronize()
    m.set_batched_path(1)
    x, ids, w, _ = m.router_topk(0, h)
    both = torch.zeros(2, *h.shape, device="cuda")
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, both[0])
    for t in range(cfg.batch):
        m.moe_ffn(0, x[t:t + 1], ids[t:t + 1], w[t:t + 1].contiguous(), both[1, t:t + 1])
    m.synchronize()
    assert (both[0] - both[1]).abs().max() <= 5e-6 * both[1].abs().max()
    m.close()


SPLITS = [("tiny", d) for d in (128, 256, 384, 512, 640, 768, 896, 1024)] + [(b, d) for b in ("qwen3", "qwen3_q4") for d in range(256, 2049, 256)]


@pytest.mark.parametrize("base,hidden", SPLITS)
def test_every_split_of_the_columns_over_warps(base, hidden):
    """17 tokens of all four experts: two full runs and one token, against the batch-1 kernel's sums with the bound of the test above. One or two
    rows in the last block."""
    for inter in (1202, 1201) if hidden == 1280 else (1201 * 128 // hidden * 8 + 1,):
        cfg = synth.get_config(base, n_layers=1, budget=1, hidden=hidden, n_experts=4, inter=inter, top_k=4, slots=4, batch=17)
        assert takes_kernel(cfg, cfg.batch)
        m = build(cfg)
        gen = torch.Generator(device="cuda").manual_seed(hidden)
        x = torch.randn(17, hidden, generator=gen, device="cuda")
        torch.cuda.synchronize()
        m.set_batched_path(1)
        _, ids, w, _ = m.router_topk(0, x)
        both = torch.zeros(2, 17, hidden, device="cuda")
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, both[0])
        for t in range(17):
            m.moe_ffn(0, x[t:t + 1], ids[t:t + 1], w[t:t + 1].contiguous(), both[1, t:t + 1])
        m.synchronize()
        assert (both[0] - both[1]).abs().max() <= 5e-6 * both[1].abs().max()
        m.close()


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_hidden_rows_may_start_at_any_float(offset):
    """spm_moe_ffn updates h_inout in place wherever it lies: an offset slice has the alignment of a float only. Same sums
    in the same order, hence the bits of the aligned call."""
    cfg = config("bf16_narrow")
    m = build(cfg, slots=cfg.n_experts)
    h = torch.randn(cfg.batch, cfg.hidden, device="cuda")
    x, ids, w, _ = m.router_topk(0, h)
    want = h.clone()
    buf = torch.empty(h.numel() + 4, device="cuda")
    at = buf[offset:offset + h.numel()].view_as(h)
    at.copy_(h)
    torch.cuda.synchronize()
    assert at.data_ptr() % 16 == 4 * offset
    m.moe_ffn(0, x, ids, w, want)
    m.moe_ffn(0, x, ids, w, at)
    m.synchronize()
    assert torch.equal(at, want) and not torch.equal(want, h)
    m.close()


@pytest.mark.parametrize("name", ["fp32_all_experts", "bf16_narrow", "q4_shared"])
@pytest.mark.parametrize("bad", [-1, 30000])
def test_a_slot_outside_the_pool_ends_the_launch_with_an_error(name, bad):
    """The kernel checks the slot numbers that it reads on the device. One that names no slot (planted in the slot map of a
    host-free step) stops the CTAs that meet it: no access, no long wait, an error status, and the context goes on."""
    cfg = config(name).replace(slots=config(name).n_experts)
    H = rows(cfg, 3)
    m = build(cfg)
    preload(cfg, m)
    good = run(m, H)
    assert m.stats()["host_free_steps"] == 3
    slot_map = np.full((cfg.n_layers, cfg.n_experts), -1, np.int16)
    for l in range(cfg.n_layers):
        for s, e in enumerate(m.slot_table(l)):
            slot_map[l, e] = s
    # the map follows the pools in the arena: [layer][expert], 16-bit, 256-byte aligned
    arena = m.arena.cpu().numpy()
    base = (-m.arena.data_ptr()) % 256
    first = base + -(-cfg.n_layers * cfg.slots * cfg.expert_bytes // 256) * 256
    at = [i for i in range(first, arena.size - slot_map.nbytes, 256) if arena[i:i + slot_map.nbytes].tobytes() == slot_map.tobytes()]
    assert len(at) == 1
    e = 1
    m.arena[at[0] + 2 * e:at[0] + 2 * e + 2] = torch.from_numpy(np.array([bad], np.int16).view(np.uint8)).cuda()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    with pytest.raises(SpmError) as err:
        run(m, H[:1])
    assert err.value.code == -5 and time.perf_counter() - t0 < 1.5
    m.cache_reset()
    preload(cfg, m)
    for a, b in zip(run(m, H), good):
        assert np.array_equal(a, b)
    m.close()


def plant_infinity(cfg, m, expert, part, row, col):
    """An infinite weight (4-bit: an infinite scale of the column's group) in one expert of layer 0 of the host store."""
    if cfg.dtype == "q4":
        part_bytes, at, raw = cfg.hidden // 2 + cfg.hidden // 16, cfg.hidden // 2 + col // 32 * 2, np.float16(np.inf).tobytes()
    else:
        part_bytes, at = cfg.hidden * cfg.elem_bytes, col * cfg.elem_bytes
        raw = np.float32(np.inf).tobytes()[-cfg.elem_bytes:]
    at += expert * cfg.expert_bytes + (row * 3 + part) * part_bytes
    m.store.tensor[at:at + len(raw)] = torch.from_numpy(np.frombuffer(raw, np.uint8).copy())


@pytest.mark.parametrize("what", ["activation_inf", "activation_nan", "gate_inf", "down_inf"])
@pytest.mark.parametrize("name", ["fp32_run_of_one", "bf16_narrow", "q4_shared"])
def test_infinities_and_nans_are_those_of_one_sequence_at_a_time(name, what):
    """Activations with eight significant bits (the lower parts of their split are zero: an infinite weight times those
    would be NaN) and a NaN that its upper half alone would turn into an infinity. Where the batch-1 kernel has a number, an
    infinity or a NaN, so has this one; sequences that have nothing to do with it keep their bits."""
    cfg = config(name)
    gen = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn(cfg.batch, cfg.hidden, generator=gen, device="cuda").bfloat16().float()
    x[:, 40] = 1.0
    outs = {}
    for planted in (False, True):
        m = build(cfg, slots=cfg.n_experts)
        m.set_batched_path(1)
        _, ids, w, _ = m.router_topk(0, x)
        if planted and what == "gate_inf":
            plant_infinity(cfg, m, 1, 0, cfg.inter // 2, 40)
        elif planted and what == "down_inf":
            plant_infinity(cfg, m, 1, 2, cfg.inter - 1, 40)
        elif planted:
            x[3, 40] = float("inf")
            if what == "activation_nan":
                x[3, 40:41].copy_(torch.tensor([0x7f800001], dtype=torch.int32, device="cuda").view(torch.float32))
        both = torch.zeros(2, cfg.batch, cfg.hidden, device="cuda")
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, both[0])
        for t in range(cfg.batch):
            m.moe_ffn(0, x[t:t + 1], ids[t:t + 1], w[t:t + 1].contiguous(), both[1, t:t + 1])
        m.synchronize()
        outs[planted] = both.cpu()
        m.close()
    got, want = outs[True]
    hit = (ids == 1).any(1) if what.endswith("_inf") and not what.startswith("act") else np.arange(cfg.batch) == 3
    assert hit.any() and not torch.isfinite(want[torch.from_numpy(hit)]).all()
    assert torch.equal(got[torch.from_numpy(~hit)], outs[False][0][torch.from_numpy(~hit)])
    assert torch.equal(got.isnan(), want.isnan())
    assert torch.equal(got.isposinf(), want.isposinf()) and torch.equal(got.isneginf(), want.isneginf())
    ok = want.isfinite()
    assert not ok.any() or (got[ok] - want[ok]).abs().max() <= 5e-6 * want[ok].abs().max()


def test_an_arena_without_room_for_the_kernel_is_accepted(monkeypatch):
    """An arena of the size that the model needed without this kernel: one GEMV per sequence serves the batch."""
    cfg = config("bf16_shared_waves").replace(slots=12)
    H = rows(cfg, 2)
    outs = []
    ask = B.spm_query_arena
    rows_of = lambda n: n * cfg.hidden * 4
    entries = min(cfg.batch * cfg.top_k, cfg.n_experts) + cfg.batch * cfg.top_k // 8 + cfg.n_shared * -(-cfg.batch // 8)
    extra = rows_of((148 + entries) * 8) - rows_of(296 + cfg.batch)          # partial rows beyond the GEMV's
    for less in (0, extra):
        monkeypatch.setattr(B, "spm_query_arena", lambda c, s: ask(c, s) - less // 256 * 256)
        m = build(cfg)
        outs.append(run(m, H))
        m.close()
    for a, b in zip(*outs):
        assert not np.array_equal(a, b) and np.abs(a - b).max() <= 1e-5 * np.abs(b).max()


# kernels of a layer and of the end of a step: routing + GEMV (folded by the next routing kernel) and one combine kernel; routing,
# gather, grouped FFN, combine; routing, several-sequences FFN, combine
COUNTS = {
    "one_sequence": (synth.get_config("tiny", slots=16), 2, 1),
    "gemv_per_sequence": (synth.get_config("tiny", slots=16, batch=3), 2, 1),
    "tensor_cores": (synth.get_config("qwen3", n_layers=3, hidden=256, n_experts=8, inter=128, top_k=2, slots=8, budget=1, batch=5), 4, 0),
    "several_sequences": (config("bf16_run_of_three"), 3, 0),
    "several_sequences_shared": (config("q4_shared"), 3, 0),
}


@pytest.mark.parametrize("host_free", [0, 1])
@pytest.mark.parametrize("name", list(COUNTS))
def test_kernels_of_a_step_are_counted_once(name, host_free):
    """spm_stats.kernel_launches says what was launched, whichever way a step is enqueued (12 steps: replayed captures among
    them); it also tells which expert kernel a batch ran."""
    cfg, a_layer, at_the_end = COUNTS[name]
    m = build(cfg)
    m.set_host_free(host_free)
    preload(cfg, m)
    m.reset_stats()
    run(m, rows(cfg, 12))
    st = m.stats()
    assert st["host_free_steps"] == (12 if host_free else 0)
    assert st["ffn_launches"] == 12 * cfg.n_layers
    assert st["kernel_launches"] == 12 * (a_layer * cfg.n_layers + at_the_end)
    m.close()


# around the line of each weight type: (shape, sequences below it, sequences above it)
LINES = {
    "bf16_wide": (dict(base="dsvl2", hidden=1280, n_experts=24, inter=653, top_k=7, slots=24, adapter_rank=8), 6, 8),
    "q4_one_token_each": (dict(base="dsvl2_q4", hidden=2048, n_experts=30, inter=906, top_k=2, n_shared=1, slots=30, adapter_rank=8), 15, 18),
    "fp32": (dict(base="tiny", hidden=1024, n_experts=24, inter=250, top_k=4, n_shared=1, slots=24), 24, 32),
}


@pytest.mark.parametrize("name", list(LINES))
def test_the_line_between_the_kernels(name):
    """Where this kernel was measured slower than one GEMV per sequence, the batch runs the GEMV: seen in the launches of a
    step (routing and GEMV a layer and one combine kernel; routing, FFN and combine kernel a layer)."""
    kw, below, above = LINES[name]
    kw = dict(kw)
    cfg = synth.get_config(kw.pop("base"), n_layers=2, budget=1, batch=above, **kw)
    assert not takes_kernel(cfg, below) and takes_kernel(cfg, above)
    m = build(cfg, store_layers=1)
    preload(cfg, m)
    H = torch.as_tensor(rows(cfg, 1)[0], dtype=torch.float32).cuda()
    for nb, launches in ((below, 2 * cfg.n_layers + 1), (above, 3 * cfg.n_layers)):
        h = H[:nb].contiguous()
        torch.cuda.synchronize()
        m.reset_stats()
        m.decode_step(h)
        m.synchronize()
        assert m.stats()["kernel_launches"] == launches, nb
    m.close()


HOST_FREE = ["fp32_all_experts", "fp32_idle_last_group", "bf16_run_of_three", "bf16_shared_waves", "q4_shared", "q4_widest_waves"]


@pytest.mark.parametrize("name", HOST_FREE)
def test_host_free_steps_equal_host_driven_ones(name):
    """The routing read on the device (launch by launch, then replayed from captures) against the routing in the launch
    arguments: same bits, events and statistics. The launch counts say that both ran this kernel."""
    cfg = config(name).replace(slots=config(name).n_experts)
    steps = 20                      # every slot of the trace ring is captured and replayed
    H = rows(cfg, steps)
    results = []
    for host_free in (1, 0):
        m = build(cfg)
        m.set_host_free(host_free)
        m.set_policy("adapter")
        preload(cfg, m)
        m.reset_stats()
        outs = run(m, H, sync_every=0 if host_free else 1)
        st = m.stats()
        assert st["host_free_steps"] == (steps if host_free else 0) and st["misses"] == 0
        assert st["kernel_launches"] == 3 * cfg.n_layers * steps
        results.append((outs, m.events(), {k: st[k] for k in ("hits", "touches", "steps", "tokens", "recall_sum", "ready_sum")}))
        m.close()
    (a, ev_a, st_a), (b, ev_b, st_b) = results
    for s in range(steps):
        assert np.array_equal(a[s], b[s]), s
    assert ev_a == ev_b and st_a == st_b


@pytest.mark.parametrize("name", ["fp32_all_experts", "bf16_shared_waves", "q4_narrow"])
def test_fewer_sequences_than_the_context_was_made_for(name):
    """One context over both sides of the rule: which kernel a call takes follows its own number of sequences, and the
    results are those of one sequence at a time either way (5e-6: the roundings of some hundred additions)."""
    cfg = config(name).replace(slots=config(name).n_experts)
    first = next(nb for nb in range(1, cfg.batch + 1) if takes_kernel(cfg, nb))
    m = build(cfg)
    preload(cfg, m)
    H = torch.as_tensor(rows(cfg, 1)[0], dtype=torch.float32).cuda()
    for nb in sorted({2, first - 1, first, cfg.batch - 1}):
        h = H[:nb].contiguous()
        torch.cuda.synchronize()
        x, ids, w, _ = m.router_topk(0, h)
        both = torch.zeros(2, *h.shape, device="cuda")
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, both[0])
        for t in range(nb):
            m.moe_ffn(0, x[t:t + 1], ids[t:t + 1], w[t:t + 1].contiguous(), both[1, t:t + 1])
        m.synchronize()
        assert (both[0] - both[1]).abs().max() <= 5e-6 * both[1].abs().max()
        m.reset_stats()
        m.decode_step(h)
        m.synchronize()
        assert m.stats()["kernel_launches"] == (3 * cfg.n_layers if nb >= first else 2 * cfg.n_layers + 1), nb
    m.close()


def test_error_against_64_bits_is_that_of_fp32_sums():
    """Distance of one layer's output from 64-bit arithmetic, this kernel against one GEMV (fp32 multiply-adds) per sequence.
    Products are exact in both and both round some hundred partial sums: neither is better in general, so a shape may
    favour one by a quarter, and all shapes together by a tenth at most."""
    ratios = {}
    for name in ("fp32_all_experts", "fp32_run_of_one", "fp32_idle_last_group", "bf16_run_of_two", "bf16_shared_waves", "bf16_narrow", "q4_narrow", "q4_shared"):
        cfg = config(name)
        m = build(cfg, slots=cfg.n_experts)
        h = torch.randn(cfg.batch, cfg.hidden, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
        torch.cuda.synchronize()
        x, ids, w, _ = m.router_topk(0, h)
        both = torch.zeros(2, *h.shape, device="cuda")
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, both[0])
        for t in range(cfg.batch):
            m.moe_ffn(0, x[t:t + 1], ids[t:t + 1], w[t:t + 1].contiguous(), both[1, t:t + 1])
        m.synchronize()
        m.close()
        want = torch.zeros_like(h, dtype=torch.float64)
        for e in range(cfg.n_experts + cfg.n_shared):
            gate, up, down = (a[0].double() for a in synth.expert_matrices(cfg, 0, [e], device="cuda"))
            part = torch.from_numpy(ids).cuda() == e if e < cfg.n_experts else torch.zeros(cfg.batch, cfg.top_k, device="cuda")
            weight = (w.double() * part).sum(1) if e < cfg.n_experts else torch.ones(cfg.batch, dtype=torch.float64, device="cuda")
            xd = x.double()
            want += weight[:, None] * ((torch.nn.functional.silu(xd @ gate.T) * (xd @ up.T)) @ down.T)
        err = [((b.double() - want).norm() / want.norm()).item() for b in both]
        assert err[0] <= 4e-7, (name, err)
        ratios[name] = err[0] / err[1]
    assert max(ratios.values()) <= 1.25 and np.exp(np.mean(np.log(list(ratios.values())))) <= 1.1, ratios
