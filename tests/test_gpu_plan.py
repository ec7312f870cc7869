"""Edges of the device-side plan of a batched host-free step and of the ranking made beside it."""
import numpy as np
import pytest

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
