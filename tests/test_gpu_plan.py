"""Edges of the device-side plan of a batched host-free step and of the ranking made beside it."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_edges import build
from test_gpu_host_free import preload, rows, run

pytestmark = pytest.mark.gpu

PLANS = {
    # pairs: fewer than a warp, the most there can be; experts: a partly used mask word, one, all of them in every token
    "two_tokens": dict(n_experts=33, top_k=2, slots=33, batch=2),
    "most_pairs": dict(n_experts=129, top_k=16, slots=129, batch=64),
    "one_expert": dict(n_experts=1, top_k=1, slots=1, batch=63),
    "all_experts": dict(n_experts=16, top_k=16, slots=16, batch=64),
}


@pytest.mark.parametrize("name", list(PLANS))
def test_device_plan_and_ranking_equal_the_host_driven_step(name):
    cfg = synth.get_config("qwen3", n_layers=3, hidden=256, inter=128, budget=1, **PLANS[name])
    H = rows(cfg, 3)
    results = []
    for host_free in (1, 0):
        m = build(cfg)
        m.set_host_free(host_free)
        m.set_policy("adapter")
        preload(cfg, m)
        outs = run(m, H, sync_every=1)
        st = m.stats()
        assert st["host_free_steps"] == (3 if host_free else 0)
        results.append((np.stack(outs), m.events(), {k: st[k] for k in ("hits", "touches", "recall_sum", "recall_at")}))
        m.close()
    (a, ev_a, st_a), (b, ev_b, st_b) = results
    assert np.array_equal(a, b) and ev_a == ev_b and st_a == st_b


# (hidden, inter, experts, top-k, sequences): 2 to 16 d-tiles a unit, some that do not divide into parts evenly; fewer units than CTAs, about as many,
# and up to three times as many with whole units in front
@pytest.mark.parametrize("hidden,inter,n,k,nb", [(256, 384, 20, 2, 9), (768, 128, 40, 4, 30), (512, 256, 12, 3, 4), (1024, 1024, 24, 4, 16), (1280, 512, 48, 4, 40),
                                                 (1792, 640, 64, 6, 48), (2048, 768, 16, 8, 5), (2048, 128, 149, 4, 64)])
def test_units_cut_on_the_device_give_the_bits_of_the_host_plan(hidden, inter, n, k, nb):
    cfg = synth.get_config("qwen3", n_layers=2, hidden=hidden, inter=inter, n_experts=n, top_k=k, slots=n, batch=nb, budget=1, adapter_rank=4)
    H = rows(cfg, 2)
    outs = []
    for host_free in (1, 0):
        m = build(cfg, store_layers=1)
        m.set_host_free(host_free)
        preload(cfg, m)
        outs.append(run(m, H, sync_every=1))
        assert m.stats()["host_free_steps"] == (2 if host_free else 0)
        m.close()
    for a, b in zip(*outs):
        assert np.isfinite(a).all() and np.array_equal(a, b)


# sequences on either side of the lines between clusters of eight, one and two CTAs an SM, and clusters of four; experts on either side of what one warp ranks
@pytest.mark.parametrize("nb", [18, 19, 32, 33, 47, 64])
@pytest.mark.parametrize("hidden,n,k", [(256, 128, 16), (512, 131, 5), (2048, 37, 8)])
def test_routing_of_a_batch_equals_one_sequence_at_a_time(nb, hidden, n, k):
    cfg = synth.get_config("qwen3", n_layers=2, hidden=hidden, inter=128, n_experts=n, top_k=k, slots=n, batch=nb, budget=1, adapter_rank=5)
    m = build(cfg)
    h = torch.randn(nb, hidden, generator=torch.Generator(device="cuda").manual_seed(nb), device="cuda")
    h[nb // 2] = h[0]
    m._keep[1][0, 3] = m._keep[1][0, 9]         # two experts that always tie
    torch.cuda.synchronize()
    x, ids, w, logits = m.router_topk(0, h, want_logits=True)
    scores, order = m.adapter_predict(0, x)
    one = [m.router_topk(0, h[t:t + 1].contiguous(), want_logits=True) for t in range(nb)]
    each = [m.adapter_predict(0, x[t:t + 1].contiguous())[0] for t in range(nb)]
    m.synchronize()
    for t, (xt, it, wt, lt) in enumerate(one):
        assert torch.equal(x[t], xt[0]) and np.array_equal(ids[t], it[0]) and torch.equal(w[t], wt[0]) and torch.equal(logits[t], lt[0]), t
        ranked = sorted(range(n), key=lambda e: (-float(lt[0, e]), e))
        assert list(it[0]) == ranked[:k], t
    want = np.zeros(n, np.float32)
    for s in each:
        want += s                               # (fp32, in token order)
    assert np.array_equal(scores, want) and list(order) == sorted(range(n), key=lambda e: (-want[e], e))
    m.close()
