"""4-bit experts through mma.sync operands: the one-token kernel at the edges of its tiles against 64-bit sums."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_edges import build

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
    for scale in (1.0, 1e-6, 3e4, 1e9):         # the last two: activations that take phase 2's scale down
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
