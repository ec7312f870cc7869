"""CPU-only checks of the C-ABI library: it builds for sm_100a, loads without a GPU, exports every
symbol include/spm.h declares, and its host-side slot table matches the policy oracle bit for bit."""
import os
import re

import numpy as np
import pytest

from oracle import ref_policy as P
from paper_2607_24787_b200 import binding as B
from paper_2607_24787_b200.build import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def lib():
    build()
    return B.load()


def test_header_symbols_exported(lib):
    hdr = open(os.path.join(ROOT, "include", "spm.h")).read()
    declared = sorted(set(re.findall(r"\b(spm_[a-z0-9_]+)\s*\(", hdr)))
    assert declared == B.EXPORTS, set(declared) ^ set(B.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_misaligned_buffers_are_refused_ahead_of_the_device():
    import torch
    if torch.cuda.is_available():
        pytest.skip("made-up addresses")
    for shared in (0, 1):
        cfg = B.make_cfg(2, 256, 16, 128, 2, shared, 8, B.DTYPE_FP32)
        # rms_gamma, router_w, adapter_a (checked where the adapter runs), adapter_b (read one element at a time), shared_experts
        for i, refused in enumerate((True, True, False, False, shared > 0)):
            at = [256] * 5
            at[i] += 8
            with pytest.raises(B.SpmError) as e:
                B.spm_init(cfg, 4, 2, B.Buffers(*at, 256, 256, 1 << 40, 1, 2, 0))
            assert e.value.code == (-1 if refused else -3)


def test_query_and_config_errors():
    cfg = B.make_cfg(48, 2048, 128, 768, 8, 0, 16, B.DTYPE_BF16)
    assert B.spm_expert_blob_bytes(cfg) == 9437184
    assert B.spm_query_arena(cfg, 16) > 48 * 16 * 9437184
    assert B.spm_expert_blob_bytes(B.make_cfg(12, 1280, 64, 896, 6, 2, 16, B.DTYPE_Q4)) == 1935360
    with pytest.raises(B.SpmError) as e:
        B.spm_query_arena(cfg, 4)                       # slots < top_k at batch 1
    assert e.value.code == -2
    with pytest.raises(B.SpmError):
        B.spm_query_arena(B.make_cfg(2, 1000, 16, 128, 2, 0, 8, B.DTYPE_BF16), 4)   # hidden not a multiple of 256
    with pytest.raises(B.SpmError):
        B.spm_query_arena(B.make_cfg(2, 256, 16, 128, 2, 15, 8, B.DTYPE_FP32), 4)   # top_k + shared too large


# Arena sizes from before the several-sequences kernel existed: device memory that callers have set aside.
# (layers, hidden, experts, inter, top_k, shared, rank, dtype, max_batch, slots): bytes, and whether the kernel is the default path
ARENAS = {
    (48, 2048, 128, 768, 8, 0, 16, B.DTYPE_BF16, 1, 16): (7250423296, False),
    (48, 2048, 128, 768, 8, 0, 16, B.DTYPE_BF16, 64, 32): (14530726656, False),
    (48, 2048, 128, 768, 8, 0, 16, B.DTYPE_Q4, 64, 32): (4112075520, False),
    (3, 2048, 1024, 128, 16, 0, 8, B.DTYPE_BF16, 64, 64): (320763904, False),
    (2, 256, 16, 128, 2, 0, 8, B.DTYPE_FP32, 64, 16): (13301248, False),
    (3, 512, 24, 250, 4, 1, 8, B.DTYPE_BF16, 4, 24): (56127232, False),
    (12, 1280, 64, 896, 6, 2, 16, B.DTYPE_BF16, 16, 64): (5286802944, True),
    (12, 1280, 64, 896, 6, 2, 16, B.DTYPE_Q4, 64, 8): (188558336, True),
    (2, 1024, 96, 640, 4, 1, 8, B.DTYPE_FP32, 64, 96): (1512209152, True),
}


@pytest.mark.parametrize("shape", list(ARENAS))
def test_arena_needs_no_more_than_it_did(shape):
    """Models that batch on the tensor cores or too little for the several-sequences kernel pay nothing for it; the others
    are told what it wants but are not refused without (checked on the host, ahead of the device)."""
    import torch
    L, d, n, i, k, s, r, dtype, nb, S = shape
    cfg = B.make_cfg(L, d, n, i, k, s, r, dtype, max_batch=nb)
    before, wants_more = ARENAS[shape]
    assert (B.spm_query_arena(cfg, S) > before) == wants_more
    if torch.cuda.is_available():
        return                                     # made-up addresses below: they must not reach a device
    for size, code in ((before, -3), (L * S * B.spm_expert_blob_bytes(cfg), -1)):
        with pytest.raises(B.SpmError) as e:
            B.spm_init(cfg, S, 2, B.Buffers(256, 256, 256, 256, 256, 256, 256, size, 1, 2, 0))
        assert e.value.code == code, str(e.value)


def test_init_fails_loudly_without_gpu():
    import torch
    if torch.cuda.is_available():
        pytest.skip("has a GPU")
    cfg = B.make_cfg(2, 256, 16, 128, 2, 0, 8, B.DTYPE_FP32)
    buf = B.Buffers(256, 256, 256, 256, None, 256, 256, 1 << 40, 1, 2, 0)
    with pytest.raises(B.SpmError) as e:
        B.spm_init(cfg, 4, 2, buf)
    assert e.value.code == -3


@pytest.mark.parametrize("n_units,n_dt,grid", [(192, 16, 148), (6, 2, 148), (755, 16, 148), (148, 16, 148), (48, 10, 148),
                                              (1, 4, 7), (300, 3, 16), (40, 1, 148)])
def test_grouped_kernel_chunk_plan(n_units, n_dt, grid):
    """Phase-2 chunk list of the batched tensor-core kernel: every (unit, d-tile) exactly once, in
    unit order (the units whose phase 1 ends first come first), chunk sizes shrinking towards the
    end of the list but never below the minimum while a unit has that many d-tiles left, so that
    the CTAs that take them in order run out of work together."""
    ch = B.spm_plan_grouped_chunks(n_units, n_dt, grid)
    seen = np.zeros((n_units, n_dt), int)
    for u, dt0, dt1 in ch:
        assert 0 <= dt0 < dt1 <= n_dt
        seen[u, dt0:dt1] += 1
    assert np.all(seen == 1)
    order = [(int(u), int(d0)) for u, d0, _ in ch]
    assert order == sorted(order)
    sizes = np.array([int(d1 - d0) for _, d0, d1 in ch])
    min_chunk = min(4, n_dt)
    assert sizes.min() >= min_chunk and sizes.max() <= n_dt
    total = n_units * n_dt
    # guided: no chunk is larger than its fair share of what was left when it was cut (or the minimum, or a unit's rest)
    left = total
    for (u, d0, d1), sz in zip(ch, sizes):
        fair = -(-left // (2 * grid))
        assert sz <= max(fair, min_chunk) + min_chunk - 1, (u, d0, d1, left)
        left -= sz
    # the tail is fine-grained: the last grid chunks are all near the minimum size (when there is that much work)
    if total >= 8 * grid * min_chunk and n_dt >= 2 * min_chunk:
        assert np.all(sizes[-grid:] <= 2 * min_chunk - 1)


def test_a_captured_step_is_replayed_only_where_everything_it_was_built_from_is_the_same(tmp_path):
    """Launch arguments that a caller can change are frozen in a captured host-free step: two steps that differ in any of
    them (the limit of the device-side waits among them) must not share a capture."""
    import shutil
    import subprocess
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    base = ["3", "8", "&h", "true", "37", "0", "0ull"]
    other = ["4", "7", "&k", "false", "36", "1", "5000ull"]
    keys = [base] + [base[:i] + [other[i]] + base[i + 1:] for i in range(len(base))]
    src = tmp_path / "key.cpp"
    src.write_text('#include "host_free_key.h"\nint main() {\n  float h = 0, k = 0;\n  const spm::HostFreeKey keys[] = {'
                   + ", ".join("{" + ", ".join(k) + "}" for k in keys)
                   + "};\n  int same = 0;\n  for (auto& a : keys) for (auto& b : keys) same += a == b;\n"
                   + f"  return same == {len(keys)} ? 0 : 1;\n}}\n")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2607_24787_b200", "csrc"), "-o", str(tmp_path / "key"), str(src)], check=True)
    assert subprocess.run([str(tmp_path / "key")]).returncode == 0


def test_rounds_of_tiles_never_wait_for_a_tile_that_nobody_asked_for(tmp_path):
    """Rings of one to eight stages, none to 400 tiles, as the one-token 4-bit kernels walk them: a round's tiles have been asked for when it waits for
    them, and a stage is filled again only behind the round that read it."""
    import shutil
    import subprocess
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    src = tmp_path / "rounds.cpp"
    src.write_text('''#include <cstdio>
#include "q4_rounds.h"
int main() {
  int bad = 0;
  for (int stages = 1; stages <= 8; ++stages)
    for (int tiles = 0; tiles <= 400; ++tiles) {
      spm::Q4Rounds r(tiles, stages);
      int asked = tiles < stages ? tiles : stages, k = 0, before = 0, rounds = 0;
      bool ok = true;
      for (; ok && r.left > 0; ++rounds) {
        const int nt = r.next(tiles - k);
        ok = nt >= (stages > 1) && nt <= spm::kQ4Super && k + nt <= asked;          // (waited for: k .. k + nt - 1)
        for (int u = k - before; u < k; ++u)                             // the stages of the round before
          if (u + stages < tiles) ok = ok && asked++ == u + stages;
        k += nt;
        before = nt;
      }
      ok = ok && k == tiles && asked == tiles && rounds <= 2 * ((tiles + stages - 1) / stages);
      if (!ok && bad++ < 20) std::printf("ring of %d, %d tiles: tile %d of round %d, %d asked for\\n", stages, tiles, k, rounds, asked);
    }
  return bad != 0;
}
''')
    subprocess.run(["g++", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2607_24787_b200", "csrc"), "-o", str(tmp_path / "rounds"), str(src)], check=True)
    walk = subprocess.run([str(tmp_path / "rounds")], capture_output=True, text=True)
    assert walk.returncode == 0, walk.stdout


def test_gpu_tests_of_odd_rings_have_rings_of_that_size(tmp_path):
    """The shapes with which the one-token 4-bit kernels are run on odd rings have the number of stages that the tests state (148 SMs), and more tiles."""
    import subprocess
    import test_gpu_q4_mma as Q
    import test_gpu_resident as R
    cases = []              # hidden, rows, stages, experts and adapter rank of a one-kernel step (else 0)
    cases += [(d, inter, st, 0, 0) for d, inter, st in Q.ODD_RINGS]
    cases += [(d, -(-(k + shared) * inter // (296 // nb)), st, 0, 0) for d, inter, n, k, shared, nb, st in Q.ODD_RINGS_BATCHED]
    for name, kw in R.CASES.items():
        if name.startswith("q4_ring_of"):
            st = {"three": 3, "five": 5, "seven": 7}[name.split("_")[3]]
            cases.append((kw["hidden"], -(-(kw["top_k"] + kw.get("n_shared", 0)) * kw["inter"] // 148), st, kw["n_experts"], kw["adapter_rank"]))
    src = tmp_path / "ring.cu"
    src.write_text('#include <cstdio>\n#include "resident_step.cuh"\nint main() {\n  const int cases[][5] = {'
                   + ", ".join("{%d, %d, %d, %d, %d}" % c for c in cases)
                   + """};
  int bad = 0;
  for (auto& c : cases) {
    int stages = 0;
    spm::ffn_gemv_q4_shape(c[0], c[1], c[3] ? spm::step_route_bytes(c[0], c[3], c[4], false) + 16 : 0, &stages);
    const int tiles = (c[1] + spm::kQ4Rows - 1) / spm::kQ4Rows;
    if (stages != c[2] || stages % 2 == 0 || tiles <= stages) { ++bad; std::printf("hidden %d, %d rows: %d stages, %d tiles\\n", c[0], c[1], stages, tiles); }
  }
  return bad != 0;
}
""")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "--expt-relaxed-constexpr", "-I",
                    os.path.join(ROOT, "paper_2607_24787_b200", "csrc"), "-o", str(tmp_path / "ring"), str(src)], check=True)
    got = subprocess.run([str(tmp_path / "ring")], capture_output=True, text=True)
    assert got.returncode == 0, got.stdout


def test_noalloc_argument_checks_run_before_any_gpu_work():
    """The allocation-free entry point refuses bad shapes, indices and misaligned pointers on the
    host, before it touches the device: so this runs without a GPU (addresses below are never
    dereferenced)."""
    cfg = B.make_cfg(1, 2048, 8, 64, 2, 0, 4, B.DTYPE_BF16)
    ok = 1 << 20                                            # a 16-byte aligned made-up address
    for args in ((ok + 8, ok, ok, ok), (ok, ok + 2, ok, ok), (ok, ok, ok + 4, ok), (ok, ok, ok, ok + 12)):
        blobs, w, x, h = args
        with pytest.raises(B.SpmError) as e:
            B.spm_ffn_noalloc(cfg, blobs, 8, [0, 1], w, x, h)
        assert e.value.code == -1 and "aligned" in str(e.value), args
    with pytest.raises(B.SpmError) as e:
        B.spm_ffn_noalloc(B.make_cfg(1, 4096, 8, 64, 2, 0, 4, B.DTYPE_BF16), ok, 8, [0, 1], ok, ok, ok)
    assert e.value.code == -2 and "scratch" in str(e.value)
    with pytest.raises(B.SpmError) as e:
        B.spm_ffn_noalloc(cfg, ok, 8, [0, 8], ok, ok, ok)   # blob index outside the 8 blobs
    assert e.value.code == -1
    with pytest.raises(B.SpmError) as e:
        B.spm_ffn_noalloc(cfg, ok, 8, list(range(17)), ok, ok, ok)   # more experts than SPM_MAX_TOPK
    assert e.value.code == -1


def drive(policy_obj, trace, ranks, L, budget, mode, drop=0):
    """Feed one recorded trace to either the oracle SlotPolicy or the library's Sim."""
    for t, per_layer in enumerate(trace):
        for l in range(L):
            policy_obj.demand(l, per_layer[l])
            if l <= L - 2 and mode != "on_demand":
                if mode == "hint":
                    sel, prot = policy_obj.plan(l + 1, per_layer[l + 1], budget, True)
                else:
                    sel, prot = policy_obj.plan(l + 1, ranks[t][l], budget, False)
                if mode == "pred0":
                    policy_obj.plan_only(l + 1, sel)
                elif isinstance(policy_obj, P.SlotPolicy):
                    dropped = {e for e in sel if drop and (policy_obj.step + e) % drop == 0}
                    policy_obj.prefetch(l + 1, sel, prot, dropped)
                else:
                    policy_obj.prefetch(l + 1, sel, prot, drop)
        if isinstance(policy_obj, P.SlotPolicy):
            policy_obj.step += 1
        else:
            policy_obj.end_step()
            policy_obj.check()                 # structural invariants of the library's table after every step


@pytest.mark.parametrize("mode,S,budget,nb,plain,drop", [
    ("adapter", 4, 2, 1, False, 0), ("adapter", 8, 3, 1, True, 0), ("hint", 6, 2, 1, False, 0),
    ("pred0", 4, 2, 1, False, 0), ("on_demand", 5, 0, 1, False, 0), ("adapter", 5, 2, 7, False, 0),
    ("adapter", 3, 4, 9, False, 3), ("hint", 16, 8, 4, False, 0), ("adapter", 16, 1, 1, False, 2),
])
def test_slot_table_matches_policy_oracle(mode, S, budget, nb, plain, drop):
    L, n, K, steps = 3, 24, 3, 80
    rng = np.random.default_rng(hash((mode, S, budget, nb)) % (1 << 31))
    trace, ranks = [], []
    for _ in range(steps):
        trace.append([sorted({int(e) for _ in range(nb) for e in rng.permutation(n)[:K]}) for _ in range(L)])
        ranks.append([[int(e) for e in rng.permutation(n)] for _ in range(L)])
    ref = P.SlotPolicy(L, n, S, plain)
    sim = B.Sim(L, n, S, plain)
    drive(ref, trace, ranks, L, budget, mode, drop)
    drive(sim, trace, ranks, L, budget, mode, drop)
    assert sim.events() == ref.events
    st = sim.stats()
    for k in ("hits", "hits_prefetched", "misses", "evictions", "wasted", "prefetch_issued", "touches",
              "waves", "planned"):
        assert st[k] == getattr(ref.stats, k), k
    for l in range(L):
        assert sim.slot_table(l) == ref.pools[l].slot_expert
    sim.close()


def test_sim_rejects_bad_arguments():
    sim = B.Sim(2, 8, 3)
    with pytest.raises(B.SpmError):
        sim.demand(5, [1])
    with pytest.raises(B.SpmError):
        sim.demand(0, [99])
    with pytest.raises(B.SpmError):
        sim.plan(1, [0, 1, 8], 2)
    sim.close()


def test_checkpoint_words_match_the_oracle_state_and_resume_identically():
    # export after a run = the oracle's table word for word; a fresh table that imports it and is
    # driven on gives the events an uninterrupted table gives
    L, n, K, S, budget, steps = 3, 24, 3, 6, 2, 60
    rng = np.random.default_rng(11)
    trace = [[sorted({int(e) for e in rng.permutation(n)[:K]}) for _ in range(L)] for _ in range(steps)]
    ranks = [[[int(e) for e in rng.permutation(n)] for _ in range(L)] for _ in range(steps)]
    ref = P.SlotPolicy(L, n, S, False)
    sim = B.Sim(L, n, S, False)
    half = steps // 2
    drive(ref, trace[:half], ranks[:half], L, budget, "adapter")
    drive(sim, trace[:half], ranks[:half], L, budget, "adapter")
    words = sim.export_state()
    assert words.size == 2 + 4 * L * S and words[0] == ref.tick and words[1] == ref.step == half
    for l in range(L):
        for s in range(S):
            w = words[2 + 4 * (l * S + s):6 + 4 * (l * S + s)]
            p = ref.pools[l]
            assert list(w) == [p.slot_expert[s], p.slot_tick[s], p.slot_origin[s], p.slot_used[s]], (l, s)
    resumed = B.Sim(L, n, S, False)
    resumed.import_state(words)
    n_before = len(sim.events())
    drive(sim, trace[half:], ranks[half:], L, budget, "adapter")
    drive(resumed, trace[half:], ranks[half:], L, budget, "adapter")
    assert resumed.events() == sim.events()[n_before:]
    assert [resumed.slot_table(l) for l in range(L)] == [sim.slot_table(l) for l in range(L)]
    # invalid states are refused and leave the table as it was
    keep = resumed.export_state()
    for bad in (words[:-1], np.concatenate((words, [0])), np.where(np.arange(words.size) == 2, n, words),
                np.where(np.arange(words.size) == 3, words[0] + 1, words)):
        with pytest.raises(B.SpmError):
            resumed.import_state(bad)
    dup = words.copy()
    dup[2 + 4] = dup[2]                    # the same expert in two slots of layer 0
    if dup[2] >= 0:
        with pytest.raises(B.SpmError):
            resumed.import_state(dup)
    assert np.array_equal(resumed.export_state(), keep)
    for x in (sim, resumed):
        x.close()


@pytest.mark.parametrize("array", [np.zeros(3, "datetime64[s]"), np.zeros((2, 0), np.int32), np.zeros(4, np.float16), np.zeros((), np.int64)])
def test_addresses_of_arrays_of_any_type(array):
    for writeable in (True, False):
        array.flags.writeable = writeable
        assert B._ptr(array) == array.ctypes.data
