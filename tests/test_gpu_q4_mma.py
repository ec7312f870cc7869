"""4-bit experts through mma.sync operands: the one-token kernel at the edges of its tiles against 64-bit sums, the batched kernels at the edges
of their runs of tokens against the one-token kernel and against their roundings restated in 64 bits."""
import time

import numpy as np
import pytest
import torch

import synth
from paper_2607_24787_b200.binding import SpmError
from test_gpu_edges import build
from test_gpu_multi import takes_kernel

pytestmark = pytest.mark.gpu


def make(hidden, inter, n, k, shared=0, batch=1, layers=1):
    return synth.get_config("qwen3_q4", n_layers=layers, hidden=hidden, inter=inter, n_experts=n, top_k=k, n_shared=shared, slots=n,
                            batch=batch, budget=1, adapter_rank=4)


def exact(cfg, x, ids, w):
    """The layer's expert sum of every row in 64 bits."""
    out = torch.zeros_like(x, dtype=torch.float64)
    for e in range(cfg.n_experts + cfg.n_shared):
        wt = (w.double() * (torch.from_numpy(ids).cuda() == e)).sum(1) if e < cfg.n_experts else torch.ones(len(x), dtype=torch.float64, device="cuda")
        gate, up, down = (a[0].double() for a in synth.expert_matrices(cfg, 0, [e], device="cuda"))
        out += wt[:, None] * ((torch.nn.functional.silu(x.double() @ gate.T) * (x.double() @ up.T)) @ down.T)
    return out


# rows of a CTA (148 of them): none or one; 15 to 17; several tiles; more than the ring holds. Every split of the columns over warps.
GEMV = [(256, 37, 4, 1, 0), (512, 148, 4, 3, 0), (768, 592, 4, 4, 0), (1024, 629, 5, 4, 0), (1280, 896, 8, 6, 2), (1536, 333, 6, 5, 1),
        (1792, 200, 6, 3, 0), (2048, 768, 9, 8, 0), (2048, 1000, 12, 12, 2)]


@pytest.mark.parametrize("shape", GEMV)
def test_one_token(shape):
    """Products are exact and sums of at most 2048 terms are rounded in fp32: 1e-6 of the result, whatever the scale of the operands."""
    cfg = make(*shape)
    m = build(cfg)
    gen = torch.Generator(device="cuda").manual_seed(1)
    for scale in (1.0, 1e-6, 3e4, 1e9):         # the last two: activations beyond 2^15 and 2^60
        x = torch.randn(1, cfg.hidden, generator=gen, device="cuda") * scale
        x[0, 5] *= 100
        torch.cuda.synchronize()
        _, ids, w, _ = m.router_topk(0, torch.randn(1, cfg.hidden, generator=gen, device="cuda"))
        got = torch.zeros_like(x)
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, got)
        m.synchronize()
        want = exact(cfg, x, ids, w)
        assert (got.double() - want).norm() <= 1e-6 * want.norm(), scale
    m.close()


def test_infinite_operands_reach_the_result():
    """Columns whose value lies beyond fp32 are not finite, as with fp32 multiply-adds."""
    cfg = make(512, 128, 4, 1)
    m = build(cfg)
    x = torch.full((1, 512), 1e25, device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, torch.randn(1, 512, device="cuda"))
    got = torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    m.synchronize()
    want = exact(cfg, x, ids, w)                # finite in 64 bits, beyond fp32
    big = want.abs() > 1e39
    assert big.any() and not got[big].isfinite().any()
    m.close()


# Rounds of tiles: 8, 9 and 17 rows a CTA (blocks of eight), 33 and 49 (a last tile of one row), 65 and 70 (five tiles, rings of four), 144 (nine, a ring of
# eight). (hidden, inter, experts, top-k)
ROUNDS = [(1024, 148, 9, 8), (512, 148, 10, 9), (1536, 148 * 17, 3, 1), (768, 148 * 3, 12, 11), (1280, 148 * 7, 8, 7), (1792, 148 * 13, 6, 5),
          (2048, 1480, 8, 7), (256, 148 * 12, 13, 12)]


@pytest.mark.parametrize("shape", ROUNDS)
def test_rounds_of_tiles(shape):
    """Against 64 bits, with the bound of test_one_token, and beyond fp32, where every tile's activations are infinite."""
    hidden, inter, n, k = shape
    cfg = make(hidden, inter, n, k)
    m = build(cfg)
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(1, hidden, generator=gen, device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, x)
    got, huge = torch.zeros_like(x), torch.zeros_like(x)
    big = x * 1e25                              # gate * up beyond fp32
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    m.moe_ffn(0, big, ids, w, huge)
    m.synchronize()
    want = exact(cfg, x, ids, w)
    assert (got.double() - want).norm() <= 1e-6 * want.norm()
    far = exact(cfg, big, ids, w).abs() > 1e39
    assert far.any() and not huge[far].isfinite().any()
    m.close()


# Rings of an odd number of stages, and more tiles: (hidden, rows of an expert, stages), an expert a CTA; one tile more than stages, one row either side of a
# tile, two and three times the ring, and several hundred tiles. (tests/test_abi_cpu.py holds the stages against the kernel's own rule.)
ODD_RINGS = [(1536, 81, 5), (1536, 96, 5), (1536, 97, 5), (1536, 161, 5), (1536, 240, 5), (1536, 5000, 5),
             (1024, 113, 7), (1024, 128, 7), (1024, 129, 7), (1024, 180, 7), (1024, 336, 7), (1024, 5000, 7)]


@pytest.mark.parametrize("hidden,inter,stages", ODD_RINGS)
def test_odd_rings(hidden, inter, stages):
    """Against 64 bits, with the bound of test_one_token_long_shares."""
    cfg = make(hidden, inter, 5, 4, 1)
    m = build(cfg)
    m.set_ffn_ctas(5)
    x = torch.randn(1, hidden, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, x)
    got = torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    m.synchronize()
    want = exact(cfg, x, ids, w)
    assert (got.double() - want).norm() <= 5e-7 * want.norm()
    m.close()


# (hidden, inter, experts, top-k, shared, sequences, stages): one GEMV a sequence, on 296 CTAs over the sequences
ODD_RINGS_BATCHED = [(1536, 600, 40, 8, 0, 5, 5), (1536, 1000, 24, 8, 0, 3, 5), (1536, 768, 24, 6, 2, 4, 5), (1024, 550, 40, 8, 0, 8, 7), (1024, 768, 36, 6, 2, 6, 7)]


@pytest.mark.parametrize("hidden,inter,n,k,shared,nb,stages", ODD_RINGS_BATCHED)
def test_odd_rings_of_several_sequences(hidden, inter, n, k, shared, nb, stages):
    cfg = make(hidden, inter, n, k, shared, nb)
    assert not takes_kernel(cfg, nb) and (shared or inter % 128)           # (neither of the batched kernels)
    m = build(cfg)
    x = torch.randn(nb, hidden, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, x)
    got = torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    m.synchronize()
    want = exact(cfg, x, ids, w)
    assert ((got.double() - want).norm(dim=1) <= 5e-7 * want.norm(dim=1)).all()
    m.close()


# tokens of an expert: runs of eight (every expert in every token), one short and one over; few and many tasks a CTA; every split of the columns
BATCHED = {
    "one_run": (2048, 128, 3, 3, 8), "run_and_one": (2048, 256, 3, 3, 9), "run_short": (1792, 384, 2, 2, 15), "eight_runs": (1536, 128, 2, 2, 64),
    "narrow": (512, 2048, 12, 2, 3), "wide_spread": (1280, 768, 60, 6, 24), "many_tasks": (1024, 1152, 128, 8, 5), "three_segments": (768, 768, 9, 3, 4),
    "one_segment": (256, 256, 2, 1, 2),
}


@pytest.mark.parametrize("name", list(BATCHED))
def test_batched(name):
    """bf16 activations against the one-token kernel's fp32 ones, on either side of the line between the two batched kernels: both operands
    that are rounded carry 2^-9, over all terms some 3e-3 of a row. A row keeps its bits in another place of the batch."""
    hidden, inter, n, k, nb = BATCHED[name]
    cfg = make(hidden, inter, n, k, batch=nb)
    m = build(cfg)
    gen = torch.Generator(device="cuda").manual_seed(2)
    for scale in (1.0, 2e4):
        x = torch.randn(nb, hidden, generator=gen, device="cuda") * scale
        torch.cuda.synchronize()
        _, ids, w, _ = m.router_topk(0, torch.randn(nb, hidden, generator=gen, device="cuda"))
        got, turned, rows = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
        x2, w2 = x.roll(1, 0), w.roll(1, 0)
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, got)
        m.moe_ffn(0, x2, np.roll(ids, 1, 0), w2, turned)
        for t in range(nb):
            m.moe_ffn(0, x[t:t + 1], ids[t:t + 1], w[t:t + 1].contiguous(), rows[t:t + 1])
        m.synchronize()
        assert torch.equal(turned.roll(-1, 0), got)
        assert ((got - rows).norm(dim=1) <= 1e-2 * rows.norm(dim=1)).all()
    m.close()


# (sequences, top-k), every pair an expert of its own: as many tasks as CTAs, one less, up to one a CTA more, two a CTA and either side of it, three
# and a few; three tasks an expert in rows of other widths
SPLIT = [(512, 128, 21, 7), (512, 128, 37, 4), (512, 128, 50, 3), (512, 128, 31, 5), (512, 128, 59, 5), (512, 128, 37, 8), (512, 128, 33, 9), (512, 128, 64, 7),
         (1280, 384, 25, 2), (2048, 384, 64, 3)]


@pytest.mark.parametrize("hidden,inter,nb,k", SPLIT)
def test_tasks_split_between_two_ctas_keep_their_bits(hidden, inter, nb, k):
    """Against the same rows in calls so small that no task is split."""
    cfg = make(hidden, inter, nb * k, k, batch=nb)
    m = build(cfg)
    m.test_grouped_q4(2)
    x = torch.randn(nb, hidden, generator=torch.Generator(device="cuda").manual_seed(4), device="cuda")
    ids = np.random.default_rng(5).permutation(nb * k).astype(np.int32).reshape(nb, k)
    w = torch.rand(nb, k, device="cuda")
    got, want = torch.zeros_like(x), torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    few = max(2, 140 // (k * (inter // 128)))
    for t in range(0, nb, few):
        t = min(t, nb - 2)
        want[t:t + few] = 0
        torch.cuda.synchronize()
        m.moe_ffn(0, x[t:t + few], ids[t:t + few], w[t:t + few].contiguous(), want[t:t + few])
        m.synchronize()
    assert m.test_grouped_q4(0)[0] == 0
    assert got.abs().min(1).values.max() > 0 and torch.equal(got, want)
    m.close()


def rounded(cfg, x, ids, w, parts=None):
    """The layer's expert sum with what the batched kernels round rounded to bf16 (token rows, scales, scale * (q - 8), activations), all
    sums in 64 bits. parts(e): the expert's ((q, scale), (q, scale), (q, scale)) where they are not the configuration's."""
    out = torch.zeros_like(x, dtype=torch.float64)
    rows = x.bfloat16().double()
    for e in range(cfg.n_experts):
        hit = torch.from_numpy(ids).cuda() == e
        on = hit.any(1)
        if not on.any():
            continue
        wt = (w.double() * hit).sum(1)
        mats = parts(e) if parts else [(q[0], s[0]) for q, s in synth.expert_q4(cfg, 0, [e], device="cuda")]
        gate, up, down = (((q.float() - 8) * s.bfloat16().float().repeat_interleave(32, -1)).bfloat16().double() for q, s in mats)
        act = (torch.nn.functional.silu(rows[on] @ gate.T) * (rows[on] @ up.T) * wt[on, None]).bfloat16().double()
        out[on] += act @ down
    return out


@pytest.mark.parametrize("name", list(BATCHED) + ["tcgen05"])
def test_batched_kernels_round_alike(name):
    """Outputs of batched 4-bit experts are the same numbers whichever kernel a batch size leads to: both round what `rounded` does. Sums in
    fp32 against 64 bits, 1e-6 of a gate, tip one activation in 2^12 to its other bf16 neighbour, 2^-8 of it: 6e-5 of the whole on
    average, and five times that with few and uneven activations. An operand rounded elsewhere shows at 2e-3."""
    hidden, inter, n, k, nb = dict(BATCHED, tcgen05=(2048, 768, 24, 8, 64))[name]
    cfg = make(hidden, inter, n, k, batch=nb)
    m = build(cfg)
    gen = torch.Generator(device="cuda").manual_seed(3)
    for scale in (1.0, 2e4):
        x = torch.randn(nb, hidden, generator=gen, device="cuda") * scale
        torch.cuda.synchronize()
        _, ids, w, _ = m.router_topk(0, torch.randn(nb, hidden, generator=gen, device="cuda"))
        got = torch.zeros_like(x)
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, got)
        m.synchronize()
        want, whole = rounded(cfg, x, ids, w), exact(cfg, x, ids, w)
        assert (got.double() - want).norm() <= 3e-4 * want.norm(), scale
        # all four roundings carry 2^-9 at most, three of them on independent terms: some 4e-3 of a row
        assert ((got.double() - whole).norm(dim=1) <= 8e-3 * whole.norm(dim=1)).all(), scale
    m.close()


def test_batch_mates_do_not_change_a_row():
    """Rows that are not finite, or as large as fp32 goes, beside ordinary rows of the same experts."""
    cfg = make(1024, 256, 3, 3, batch=9)
    m = build(cfg)
    gen = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randn(9, 1024, generator=gen, device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, torch.randn(9, 1024, generator=gen, device="cuda"))
    odd = x.clone()
    odd[1, 7], odd[2], odd[4, 0], odd[5] = float("inf"), x[2] * 1e19, float("nan"), x[5] * 1e37
    clean, mixed = torch.zeros_like(x), torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, clean)
    m.moe_ffn(0, odd, ids, w, mixed)
    m.synchronize()
    same = [0, 3, 6, 7, 8]
    assert torch.equal(mixed[same], clean[same])
    assert not mixed[[1, 4]].isfinite().any()
    m.close()


def test_scales_that_are_not_finite():
    """An infinite or NaN scale of W_down makes infinities and NaNs of its columns, where the products say so, and of no others."""
    cfg = make(1280, 256, 2, 2, batch=3)
    m = build(cfg)
    part = cfg.hidden // 2 + cfg.hidden // 16
    blobs = m.store.tensor.view(cfg.n_experts, cfg.inter, 3, part)
    bad = {(0, 5, 3): 0x7c00, (0, 130, 39): 0xfc00, (1, 255, 17): 0x7e01}         # (expert, row, group): fp16 bits
    for (e, j, grp), bits in bad.items():
        at = cfg.hidden // 2 + 2 * grp
        blobs[e, j, 2, at], blobs[e, j, 2, at + 1] = bits & 255, bits >> 8

    def parts(e):
        mats = [(q[0], s[0].clone()) for q, s in synth.expert_q4(cfg, 0, [e], device="cuda")]
        for (e2, j, grp), bits in bad.items():
            if e2 == e:
                mats[2][1].view(torch.int16)[j, grp] = bits - 65536 if bits > 32767 else bits
        return mats

    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(3, cfg.hidden, generator=gen, device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, x)
    got = torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    m.synchronize()
    want = rounded(cfg, x, ids, w, parts)
    assert torch.equal(got.isnan(), want.isnan()) and torch.equal(got.isposinf(), want.isposinf()) and torch.equal(got.isneginf(), want.isneginf())
    ok = want.isfinite()
    assert (~ok).sum() == 3 * 96 and ((got.double() - want)[ok].norm() <= 3e-4 * want[ok].norm())
    m.close()


def test_silu_of_negative_gates():
    """One row, one column that is not zero: gate and up are exact, so what is left is exp (two units in the last place at most), a sum, a
    quotient, three products and the split sum of the result, 2^-24 each: 6e-7 of an element. The fast exponential is off by more the
    larger the gate."""
    cfg = make(256, 1, 2, 1)
    m = build(cfg)
    (gq, gs), (uq, us), _ = synth.expert_q4(cfg, 0, [0], device="cuda")
    gate = ((gq[0, 0].float() - 8) * gs[0, 0].float().repeat_interleave(32)).cpu()
    up = ((uq[0, 0].float() - 8) * us[0, 0].float().repeat_interleave(32)).cpu()
    col = int((gate + 1e3 * (up == 0)).argmin())
    ids, w = np.zeros((1, 1), np.int32), torch.ones(1, 1, device="cuda")
    m.prefetch_async(0, ids[0])
    for target in np.linspace(1, 40, 40):
        x = torch.zeros(1, 256, device="cuda")
        x[0, col] = round(target / -float(gate[col]) * 4) / 4            # few bits: its products with the weights are exact
        got = torch.zeros_like(x)
        torch.cuda.synchronize()
        m.moe_ffn(0, x, ids, w, got)
        m.synchronize()
        want = exact(cfg, x, ids, w)
        assert ((got.double() - want).abs() <= 6e-7 * want.abs()).all(), target
    m.close()


@pytest.mark.parametrize("shape", [(256, 96, 8, 2, 0), (768, 333, 16, 4, 0), (1280, 896, 16, 6, 2), (1792, 128, 16, 4, 1), (2048, 768, 24, 8, 0)])
def test_one_token_rows_of_one_sign_and_heavy_tails(shape):
    """Rows whose sum is large beside the result (all of one sign) or that a few elements rule: no more error than fp32 multiply-adds,
    2.7e-7 at worst over these shapes and rows; with the weights' offset of 8 as a sum of its own it was 5.3e-7."""
    cfg = make(*shape)
    m = build(cfg)
    gen = torch.Generator(device="cuda").manual_seed(6)
    for rep in range(4):
        z = torch.randn(1, cfg.hidden, generator=gen, device="cuda")
        t = torch.exp(1.5 * torch.randn(1, cfg.hidden, generator=gen, device="cuda"))
        for x in (z * t, t, z.abs(), 1 + 0.1 * z):
            torch.cuda.synchronize()
            _, ids, w, _ = m.router_topk(0, z)
            got = torch.zeros_like(x)
            torch.cuda.synchronize()
            m.moe_ffn(0, x, ids, w, got)
            m.synchronize()
            want = exact(cfg, x, ids, w)
            assert (got.double() - want).norm() <= 3.5e-7 * want.norm(), rep
    m.close()


def test_one_token_long_shares():
    """One CTA for all rows: 384 tiles, summed like fp32 sums. A sum that stays in the tensor cores is cut off at every tile, 2e-6 and more."""
    cfg = make(2048, 768, 8, 8)
    m = build(cfg)
    m.set_ffn_ctas(1)
    x = torch.randn(1, 2048, generator=torch.Generator(device="cuda").manual_seed(7), device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, x)
    got = torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    m.synchronize()
    want = exact(cfg, x, ids, w)
    assert (got.double() - want).norm() <= 5e-7 * want.norm()
    m.close()


@pytest.mark.parametrize("shape", [(512, 200, 12, 3, 0), (1280, 896, 16, 6, 2), (2048, 333, 16, 4, 0)])
def test_one_token_device_side_wait_gives_the_same_bits(shape):
    """The kernel waits for arrivals in one lane and asks for the bytes in another; a small cache, so that every layer waits."""
    cfg = make(*shape, layers=4).replace(slots=shape[3] + 1)
    h = torch.randn(6, 1, cfg.hidden, generator=torch.Generator(device="cuda").manual_seed(8), device="cuda")
    m = build(cfg)
    runs = []
    for on in (0, 1):
        m.cache_reset()
        m.set_device_wait(on)
        torch.cuda.synchronize()
        out = [m.decode_step(row) for row in h]
        m.synchronize()
        runs.append((torch.stack(out), m.events()))
    assert torch.equal(runs[0][0], runs[1][0]) and runs[0][1] == runs[1][1]
    assert m.stats()["misses"] > 0
    m.close()


def moe(m, x, ids, w):
    got = torch.zeros_like(x)
    torch.cuda.synchronize()
    m.moe_ffn(0, x, ids, w, got)
    m.synchronize()
    return got


# every split of the columns over warps that the mma.sync kernel has (hidden 512 to 2048), tokens an expert from one to 64 on both kernels
BOTH = {f"hidden_{h}": (h, 256, 6, 2, 24) for h in range(512, 2049, 256)}
BOTH |= {"wide_rows_many_tokens": (2048, 768, 24, 8, 64), "few_experts": (2048, 1024, 12, 8, 64), "deep": (1024, 1152, 12, 3, 17), "one_token_an_expert": (768, 384, 128, 3, 7)}


@pytest.mark.parametrize("name", list(BOTH))
def test_both_batched_kernels(name):
    """The same call through each of the two kernels, and both against the roundings restated in 64 bits (see test_batched_kernels_round_alike)."""
    hidden, inter, n, k, nb = BOTH[name]
    cfg = make(hidden, inter, n, k, batch=nb)
    m = build(cfg)
    gen = torch.Generator(device="cuda").manual_seed(9)
    x = torch.randn(nb, hidden, generator=gen, device="cuda")
    torch.cuda.synchronize()
    _, ids, w, _ = m.router_topk(0, torch.randn(nb, hidden, generator=gen, device="cuda"))
    want = rounded(cfg, x, ids, w)
    for choice in (1, 2):
        m.test_grouped_q4(choice)
        got = moe(m, x, ids, w)
        assert m.test_grouped_q4() == [1, choice - 1]
        assert (got.double() - want).norm() <= 3e-4 * want.norm(), choice
    m.close()


def test_every_number_of_tokens_an_expert_on_both_kernels():
    """Experts with 64, 47, 33, 17, 16, 14 and 1 tokens in one launch, in narrow rows and in the widest."""
    counts = [64, 47, 33, 17, 16, 14, 1, 0]
    for hidden in (512, 2048):
        cfg = make(hidden, 256, 8, 3, batch=64)
        m = build(cfg)
        gen = torch.Generator(device="cuda").manual_seed(10)
        x = torch.randn(64, hidden, generator=gen, device="cuda")
        w = torch.rand(64, 3, generator=gen, device="cuda") + 0.1
        left, ids = list(counts), np.zeros((64, 3), np.int32)
        for t in range(64):                # the experts with the most tokens left, no expert twice a token
            for k, e in enumerate(sorted(range(8), key=lambda e: -left[e])[:3]):
                ids[t, k] = e
                left[e] -= 1
        assert sorted(np.bincount(ids.reshape(-1), minlength=8).tolist()) == sorted(counts)
        want = rounded(cfg, x, ids, w)
        for choice in (1, 2):
            m.test_grouped_q4(choice)
            got = moe(m, x, ids, w)
            assert ((got.double() - want).norm(dim=1) <= 2e-3 * want.norm(dim=1)).all(), (hidden, choice)
        assert m.test_grouped_q4() == [1, 1]
        m.close()


# (choice, hidden, inter, experts, top-k, slots): the last with 148 tasks and more in a wave, some of which fall to two CTAs
@pytest.mark.parametrize("choice,hidden,inter,n,k,few", [(1, 768, 384, 12, 4, 5), (2, 768, 384, 12, 4, 5), (2, 512, 1024, 40, 8, 30)])
def test_waves_and_host_free_steps_on_both_kernels(choice, hidden, inter, n, k, few):
    """A small cache (waves, copies, device-side waits) and a context that holds every expert give the same bits, launched and replayed."""
    cfg = make(hidden, inter, n, k, batch=9, layers=3)
    h = torch.randn(3, 9, cfg.hidden, generator=torch.Generator(device="cuda").manual_seed(11), device="cuda")
    outs = []
    for slots, wait in ((few, 0), (few, 1), (n, 0)):
        m = build(cfg.replace(slots=slots))
        m.test_grouped_q4(choice)
        m.set_device_wait(wait)
        torch.cuda.synchronize()
        o = [m.decode_step(row) for row in h] + [m.decode_step(h[0]) for _ in range(20)]       # (captured per trace slot: the last ones are replays)
        m.synchronize()
        outs.append(torch.stack(o))
        ran = m.test_grouped_q4()
        assert ran[2 - choice] == 0 and ran[choice - 1] >= 23 * cfg.n_layers
        m.close()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


GIVE_UP = {          # (shape, slots, batch, batched kernel)
    "one_token": ((1280, 896, 16, 6, 2), 8, 1, 0), "one_token_widest": ((2048, 333, 16, 4), 5, 1, 0),
    "batched_mma": ((2048, 256, 12, 8), 8, 16, 2), "batched_tcgen05": ((2048, 256, 12, 8), 8, 16, 1),
    "batched_mma_split": ((512, 1024, 40, 8), 30, 16, 2),       # (240 tasks in a full wave: CTAs that go on from what another has begun)
}


@pytest.mark.parametrize("name", list(GIVE_UP))
def test_wait_for_a_copy_runs_out(name):
    """An arrival that is never published (withheld on the host; the bytes land): the kernel gives up after its limit with nothing in flight, the
    host reads the time-out once, and after a cache reset the context gives the bits of before."""
    shape, slots, nb, choice = GIVE_UP[name]
    cfg = make(*shape, batch=nb, layers=2).replace(slots=slots)
    h = torch.randn(2, nb, cfg.hidden, generator=torch.Generator(device="cuda").manual_seed(12), device="cuda")
    m = build(cfg)
    m.set_policy("on_demand")
    m.test_grouped_q4(choice)
    torch.cuda.synchronize()
    want = [m.decode_step(row) for row in h]
    m.synchronize()
    assert m.test_grouped_q4()[2 - choice if choice else 0] == 0 and (nb == 1 or sum(m.test_grouped_q4()) > 0)
    m.set_device_wait(1)
    for withheld in (1, 2):
        m.set_device_wait_limit_us(3000)
        m.cache_reset()
        m.test_withhold_arrivals(withheld)
        t0 = time.perf_counter()
        with pytest.raises(SpmError) as e:
            m.decode_step(h[0])
            m.synchronize()
        assert e.value.code == -4 and time.perf_counter() - t0 < 1.9        # after the limit, not the 2 s default
        m.synchronize()                                                     # reported once
        m.set_device_wait_limit_us(0)
        m.cache_reset()
        got = [m.decode_step(row) for row in h]
        m.synchronize()
        for a, b in zip(got, want):
            assert torch.equal(a, b)
    m.close()
