"""GPU parity of the run-length, prefix-sharing simulator: every makespan must
equal the oracle's (and the simple device simulator's) for every tuning knob
setting, including forced hand-over of work items to the simple simulator."""
import math
import os

import numpy as np
import pytest

import oracle
from paper_1511_07983_gb300 import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def ko():
    import torch
    assert torch.cuda.is_available()
    from paper_1511_07983_gb300 import build, ko as kmod
    build.build()
    torch.cuda.init()
    return kmod


def _all(g, n):
    import torch
    out = torch.empty(math.factorial(n), dtype=torch.int64, device="cuda")
    g.eval_all(out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("lanes", [16, 32])
@pytest.mark.parametrize("levels", [0, 1, 3, 4, 6])
def test_single8_all_orders_every_config(ko, lanes, levels):
    s = synth.gen_set("single8")
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=40320)
    with ko.Gpu.from_set(s) as g:
        g.configure(lanes=lanes, levels=levels)
        assert np.array_equal(_all(g, 8), want)
        assert g.last_fallback_items() == 0


@pytest.mark.parametrize("seed", range(12))
def test_random_small_sets_exhaustive(ko, seed):
    # mixes of tiny and large N_SM, power-of-two and odd capacities, heavy smem
    n = 3 + seed % 6
    gpus = [(13, 65536, 49152, 64, 16), (148, 65536, 233472, 64, 32), (7, 32768, 49152, 48, 8),
            (40, 65536, 98304, 64, 32)]
    gpu = gpus[seed % len(gpus)]
    caps = (32768, 32768) if seed % 3 else (3000, 7001)
    s = synth.random_set(100 + seed, n, gpu=gpu, blk=(1, 5 * gpu[0]), c=(100, 30000),
                         c_cap=caps[0], m_cap=caps[1])
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=math.factorial(n))
    for lanes in (16, 32):
        with ko.Gpu.from_set(s) as g:
            g.configure(lanes=lanes)
            got = _all(g, n)
            assert np.array_equal(got, want), (lanes, int(np.argmax(got != want)))


@pytest.mark.parametrize("run_limit", [1, 2, 3])
def test_forced_handover_to_simple_simulator(ko, run_limit):
    s = synth.gen_set("sets10", 2, n=7)
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=5040)
    h = oracle.heuristic(s.gpu, s.kernels)
    st = oracle.exhaustive_stats(s.gpu, s.kernels, oracle.makespan(s.gpu, s.kernels, h),
                                 makespans=want)
    with ko.Gpu.from_set(s) as g:
        g.configure(run_limit=run_limit)
        assert np.array_equal(_all(g, 7), want)
        assert g.last_fallback_items() > 0
        r, hist = g.rank_order(h, nbins=4096)
    assert (r["min"], r["max"], r["n_better"], r["n_equal"], r["n_worse"]) == \
        (st["min"], st["max"], st["n_better"], st["n_equal"], st["n_worse"])
    assert np.array_equal(hist, st["hist"])


def test_every_item_handed_over_on_a_large_launch(ko):
    """More abandoned work items than any fixed list would hold: ten one-block
    kernels on a 2-SM GPU, one saved level (1,814,400 items of two orders) and
    one run per simulation allowed.  Every item's first kernel cuts the single
    run, so all items fail both run-length passes and reach the simple
    simulator; every makespan must still arrive, equal to the default
    configuration's (itself checked against the oracle on samples)."""
    import torch
    s = synth.random_set(41, 10, gpu=(2, 65536, 49152, 64, 4), blk=(1, 1))
    n_all = math.factorial(10)
    with ko.Gpu.from_set(s) as g:
        ref = torch.empty(n_all, dtype=torch.int64, device="cuda")
        g.eval_all(ref)
        torch.cuda.synchronize()
    ids = synth.random_indices(31, n_all, 500)
    assert np.array_equal(ref[torch.from_numpy(ids.astype(np.int64)).cuda()].cpu().numpy(),
                          oracle.makespans_idx(s.gpu, s.kernels, idx=ids))
    with ko.Gpu.from_set(s) as g:
        g.configure(run_limit=1, levels=1)
        out = torch.full((n_all,), -7, dtype=torch.int64, device="cuda")
        g.eval_all(out)
        torch.cuda.synchronize()
        assert g.last_fallback_items() == n_all // 2 > (1 << 20)
    assert torch.equal(out, ref)


@pytest.mark.parametrize("lanes", [16, 32])
def test_single12_index_sample(ko, lanes):
    s = synth.gen_set("single12")
    ids = synth.random_indices(77, math.factorial(12), 3000)
    with ko.Gpu.from_set(s) as g:
        g.configure(lanes=lanes)
        got = g.eval_orders(idx=ids)
    assert np.array_equal(got, oracle.makespans_idx(s.gpu, s.kernels, idx=ids))


def test_single12_full_space_as_benchmarked(ko, tmp_path):
    """The exhaustive N=12 launch in the configuration the benchmark times (the
    tuned lanes and depth, all 479,001,600 orders): seeded samples of the stored
    makespans, work-item boundaries and the first and last orders equal the
    oracle's one by one; the fused reductions agree with the stored makespans."""
    import shutil

    import torch
    s = synth.gen_set("single12")
    n_all = math.factorial(12)
    cache = tmp_path / "tune.json"
    shutil.copy(os.path.join(ROOT, "paper_1511_07983_gb300", "ko_tune_cache.json"), cache)
    with ko.Gpu.from_set(s) as g:
        choice = g.autotune(str(cache))
        per_item = math.factorial(choice["levels"] + 1)   # orders below one item's fixed prefix
        out = torch.empty(n_all, dtype=torch.int64, device="cuda")
        g.eval_all(out)
        r, hist = g.rank_order(None, nbins=4096)
        torch.cuda.synchronize()
        mh = oracle.makespan(s.gpu, s.kernels, g.heuristic_order().tolist())

    items = synth.random_indices(1213, n_all // per_item, 40).astype(np.int64)
    ids = np.concatenate([synth.random_indices(1212, n_all, 2000).astype(np.int64),
                          items * per_item, items * per_item + per_item - 1,
                          [0, 1, per_item - 1, per_item, n_all - per_item, n_all - 2, n_all - 1]])
    got = out[torch.from_numpy(ids).cuda()].cpu().numpy()
    assert np.array_equal(got, oracle.makespans_idx(s.gpu, s.kernels, idx=ids.astype(np.uint64)))

    lb, ub = oracle.bounds(s.gpu, s.kernels)
    mn, mx = int(out.min()), int(out.max())
    assert lb <= mn <= mx <= ub
    assert r["makespan"] == mh and r["n_total"] == n_all
    assert (r["min"], r["max"]) == (mn, mx)
    assert (r["n_better"], r["n_equal"], r["n_worse"]) == \
        (int((out < mh).sum()), int((out == mh).sum()), int((out > mh).sum()))
    bins = torch.div((out - mn) * 4096, mx - mn + 1, rounding_mode="floor")
    assert np.array_equal(hist.astype(np.int64), torch.bincount(bins, minlength=4096).cpu().numpy())


def test_simple_and_fast_agree_on_sets10(ko):
    s = synth.gen_set("sets10", 5)
    with ko.Gpu.from_set(s) as g:
        fast = _all(g, 10)
    with ko.Gpu.from_set(s) as g:
        g.configure(simple_only=True)
        simple = _all(g, 10)
    assert np.array_equal(fast, simple)
    ids = synth.random_indices(3, math.factorial(10), 3000).astype(np.int64)
    assert np.array_equal(fast[ids], oracle.makespans_idx(s.gpu, s.kernels, idx=ids.astype(np.uint64)))


@pytest.mark.parametrize("workload,count", [("batched", 40)])
def test_batched_sets_exhaustive_small(ko, workload, count):
    # every batched set with N <= 8 exhaustively against the oracle
    checked = 0
    for i in range(count):
        s = synth.gen_set(workload, i)
        if s.n > 8:
            continue
        want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=math.factorial(s.n))
        with ko.Gpu.from_set(s) as g:
            assert np.array_equal(_all(g, s.n), want), i
        checked += 1
    assert checked > 5


def test_autotune_choice_cache_and_exactness(ko, tmp_path):
    import json
    s = synth.gen_set("sets10", 7, n=8)
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=40320)
    cache = str(tmp_path / "tune.json")
    with ko.Gpu.from_set(s) as g:
        choice = g.autotune(cache)
        assert choice["lanes"] in (1, 16, 32) and 1 <= choice["levels"] <= 6
        assert choice["stack_global"] in (0, 1) and choice["lane_state"] in (0, 1, 2)
        assert np.array_equal(_all(g, 8), want)
    data = json.load(open(cache))
    assert data["S16_N8"]["lanes"] == choice["lanes"] and data["S16_N8"]["levels"] == choice["levels"]
    assert data["S16_N8"]["stack"] == choice["stack_global"] and data["S16_N8"]["shape"] == choice["lane_state"]
    with ko.Gpu.from_set(s) as g:   # second handle: served from the cache
        assert g.autotune(cache) == choice


@pytest.mark.parametrize("lanes", [16, 32])
@pytest.mark.parametrize("levels", [1, 3, 5])
def test_global_node_stack_is_exact(ko, lanes, levels):
    s = synth.gen_set("single8")
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=40320)
    with ko.Gpu.from_set(s) as g:
        g.configure(lanes=lanes, levels=levels, stack_global=True)
        assert np.array_equal(_all(g, 8), want)
        r, hist = g.rank_order(None, nbins=4096)
    h = oracle.heuristic(s.gpu, s.kernels)
    st = oracle.exhaustive_stats(s.gpu, s.kernels, oracle.makespan(s.gpu, s.kernels, h), makespans=want)
    assert (r["min"], r["max"], r["n_equal"]) == (st["min"], st["max"], st["n_equal"])
    assert np.array_equal(hist, st["hist"])


@pytest.mark.parametrize("case", ["sm1024", "one_block_per_sm", "no_smem", "huge_durations", "bk32_tiny_sm"])
def test_edge_gpus_match_oracle(ko, case):
    if case == "sm1024":        # many runs: hand-over to the wide pass and the simple simulator
        s = synth.random_set(41, 5, gpu=(1024, 65536, 233472, 64, 32), blk=(100, 3000), c=(1000, 50000))
    elif case == "one_block_per_sm":
        s = synth.random_set(42, 6, gpu=(7, 65536, 233472, 64, 1), blk=(1, 30))
    elif case == "no_smem":
        s = synth.random_set(43, 6, gpu=(13, 65536, 49152, 64, 16), blk=(5, 80))
        s.kernels[:, 1] = 0
    elif case == "huge_durations":  # durations reach 2^31: the run-length path does not apply
        s = synth.random_set(44, 5, gpu=(13, 65536, 49152, 64, 16), blk=(5, 60), c=(1 << 19, 1 << 20),
                             c_cap=1, m_cap=1)
    else:
        s = synth.random_set(45, 6, gpu=(2, 65536, 233472, 64, 32), blk=(1, 40))
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=math.factorial(s.n))
    with ko.Gpu.from_set(s) as g:
        got = _all(g, s.n)
        assert np.array_equal(got, want), case
        h = oracle.heuristic(s.gpu, s.kernels)
        r, hist = g.rank_order(h, nbins=128)
    st = oracle.exhaustive_stats(s.gpu, s.kernels, oracle.makespan(s.gpu, s.kernels, h), nbins=128,
                                 makespans=want)
    assert (r["min"], r["max"], r["n_better"], r["n_equal"], r["n_worse"]) == \
        (st["min"], st["max"], st["n_better"], st["n_equal"], st["n_worse"])
    assert np.array_equal(hist, st["hist"])


# ------------------------------------------------ choice by size (options left alone)

@pytest.mark.parametrize("gpu", [(13, 65536, 49152, 64, 16), (148, 65536, 233472, 64, 32),
                                 (16, 65536, 49152, 128, 16), (33, 1 << 19, 98304, 64, 32)])
@pytest.mark.parametrize("n", [1, 2, 6, 7, 8])
def test_default_space_equals_every_pinned_choice(ko, n, gpu):
    # N around the lines of the rule, 16 and more SMs, limits outside the packed usage word
    s = synth.random_set(700 + n, n, gpu=gpu, blk=(1, 5 * gpu[0]), c=(100, 30000))
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=math.factorial(n))
    with ko.Gpu.from_set(s) as g:
        assert np.array_equal(_all(g, n), want)
        assert ko.ko_get_option(g.h, ko.KO_OPT_LANES) == 16      # the handle's options stay
        assert ko.ko_get_option(g.h, ko.KO_OPT_LEVELS) == 4


@pytest.mark.parametrize("workload,n", [("single8", 8), ("single12", 9), ("single12", 13), ("single12", 14)])
@pytest.mark.parametrize("count", [16384, 16385, 28673, 53249])
def test_default_list_equals_a_pinned_choice(ko, workload, n, count):
    s = synth.gen_set(workload, 5, n=n)
    rows = synth.random_orders(count, n, count).astype(np.int8)
    rows[3, 0] = rows[3, 1]                                      # not a permutation
    with ko.Gpu.from_set(s) as g:
        got = g.eval_orders(orders=rows)
    with ko.Gpu.from_set(s) as g:
        g.configure(lanes=16)
        want = g.eval_orders(orders=rows)
    assert np.array_equal(got, want) and got[3] == -1
    pick = np.arange(0, count, 161)
    pick = pick[pick != 3]
    assert np.array_equal(got[pick], oracle.makespans_orders(s.gpu, s.kernels, rows[pick].astype(np.int32)))


def test_captured_list_after_a_space_only(ko):
    """A captured call takes no allocation: with the slabs of an earlier space
    (whose one-thread state is smaller) and a short list, a long list keeps the
    handle's options."""
    import torch
    s = synth.gen_set("single8", 3, n=9)
    rows = torch.from_numpy(synth.random_orders(8, 9, 20000).astype(np.int8)).cuda()
    with ko.Gpu.from_set(s) as g:
        _all(g, 9)
        g.eval_orders(orders=rows[:100], out=torch.zeros(100, dtype=torch.int64, device="cuda"))
        torch.cuda.synchronize()
        out = torch.zeros(20000, dtype=torch.int64, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            g.eval_orders(orders=rows, out=out)
        graph.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        want = g.eval_orders(orders=rows.cpu().numpy())
    assert np.array_equal(got, want)


@pytest.mark.parametrize("call,launches", [("list", 2), ("space7", 3), ("pinned16", 3), ("pinned1", 5)])
def test_route_by_launches(ko, call, launches):
    """The kernels a call enqueues tell its route: a warp per order is followed by
    the simple simulator only; a space's accumulators are reset first."""
    s = synth.gen_set("single8", 1, n=7)
    rows = synth.random_orders(4, 7, 16).astype(np.int8)
    with ko.Gpu.from_set(s) as g:
        if call.startswith("pinned"):
            g.configure(lanes=int(call[6:]))
        before = ko.ko_kernel_launches()
        if call == "space7":
            _all(g, 7)
        else:
            g.eval_orders(orders=rows)
        assert ko.ko_kernel_launches() - before == launches


# --------------------------------------- hand-over of spaces with pinned 16 or 32 lanes

@pytest.mark.parametrize("lanes", [16, 32])
@pytest.mark.parametrize("run_limit", [1, 2])
@pytest.mark.parametrize("n,levels", [(6, 1), (7, 1), (7, 2), (7, 3), (8, 2), (8, 4), (8, 6)])
def test_cut_hand_over_loses_no_order(ko, n, levels, run_limit, lanes):
    """(Nearly) every item fails the first pass and every part of it the wide one,
    which cuts a list of 42 to 20,160 items as far as it has segments: no more
    parts than the next list holds, so every order is written and counted."""
    import torch
    s = synth.gen_set("sets10", 2, n=n)
    n_all = math.factorial(n)
    want = oracle.makespans_idx(s.gpu, s.kernels, first=0, count=n_all)
    h = oracle.heuristic(s.gpu, s.kernels)
    st = oracle.exhaustive_stats(s.gpu, s.kernels, oracle.makespan(s.gpu, s.kernels, h), makespans=want)
    with ko.Gpu.from_set(s) as g:
        g.configure(lanes=lanes, levels=levels, run_limit=run_limit)
        out = torch.full((n_all,), -7, dtype=torch.int64, device="cuda")
        g.eval_all(out)
        assert g.last_fallback_items() > 0
        got = out.cpu().numpy()
        assert (got == -7).sum() == 0
        assert np.array_equal(got, want)
        r, hist = g.rank_order(h, nbins=4096)
    assert (r["min"], r["max"], r["n_better"], r["n_equal"], r["n_worse"]) == \
        (st["min"], st["max"], st["n_better"], st["n_equal"], st["n_worse"])
    assert np.array_equal(hist, st["hist"])


# ------------------------------------------------------- device memory of a space

def test_lists_of_a_large_space_stay_small(ko):
    """12 kernels, options left alone (20M items): the lists between the passes,
    node states and the simple simulator's scratch hold less than 1 GB."""
    import torch
    s = synth.gen_set("single12")
    out = torch.empty(math.factorial(12), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with ko.Gpu.from_set(s) as g:
        g.eval_all(out)
        torch.cuda.synchronize()
        held = free - torch.cuda.mem_get_info()[0]
    assert held < 1 << 30, held


def test_space_takes_the_handles_options_where_memory_is_short(ko):
    """400 MB left on the device: the choice by size (0.45 GB for this space) does
    not fit, the handle's own options (0.31 GB) do."""
    import torch
    s = synth.gen_set("sets10", 4, n=11)
    n_all = math.factorial(11)
    want = torch.empty(n_all, dtype=torch.int64, device="cuda")
    out = torch.full((n_all,), -7, dtype=torch.int64, device="cuda")
    for cfg in ({}, dict(lanes=16, levels=4)):      # both routes' kernels are loaded now
        with ko.Gpu.from_set(s) as g:
            g.configure(**cfg)
            g.eval_all(want)
            torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (400 << 20), dtype=torch.uint8, device="cuda")
    try:
        with ko.Gpu.from_set(s) as g:
            g.eval_all(out)
            torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(out, want)


# ----------------------------------- a warp per order: run pointers, capacities, limits

@pytest.mark.parametrize("n_sm", [1, 2, 31, 148, 1023, 1024])
@pytest.mark.parametrize("caps", [(32768, 32768), (3000, 7001), (32768, 5000)])
@pytest.mark.parametrize("n", [2, 11, 24])
def test_warp_per_order_edges(ko, n_sm, caps, n):
    """Up to 1,024 SMs (the pointer's field in a warp's keys), capacities that are
    no power of two, kernels alike enough that several runs end together."""
    s = synth.random_set(900 + n, n, gpu=(n_sm, 65536, 98304, 64, 16), blk=(1, 3 * n_sm + 5), c=(500, 520),
                         c_cap=caps[0], m_cap=caps[1])
    k = s.kernels.copy()
    k[::2, 4:6] = k[0, 4:6]
    s = synth.KernelSet(gpu=s.gpu, kernels=k)
    rows = synth.random_orders(n, n, 40)
    with ko.Gpu.from_set(s) as g:
        got = g.eval_orders(orders=rows.astype(np.int8))
    assert np.array_equal(got, oracle.makespans_orders(s.gpu, s.kernels, rows.astype(np.int32)))
