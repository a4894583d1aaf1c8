"""The routes a sampled cascade can take through the kernels, at the sizes where they change:
the warp spread kernel's queue and its hand-off, the non-tree target array of the block tier, and
the three launches of the allocation-free call. Counters and sums are integers: tolerance 0."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from paper_2302_13529_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _graph(n, src, dst, p, lt=False):
    """A graph from edge lists with one probability for all edges (LT: weights of 1 / in-degree)."""
    order = np.lexsort((dst, src))
    src, dst = np.asarray(src)[order], np.asarray(dst, np.int32)[order]
    row = np.zeros(n + 1, np.int32)
    row[1:] = np.cumsum(np.bincount(src, minlength=n))
    w = W.lt_wc_weights(dst, n) if lt else np.full(len(dst), int(p * 2**32) - 1, np.uint32)
    return W.Graph(n, row, dst, w)


def _star(leaves, p=1.0, chain=1):
    """Vertex 0 -> `leaves` vertices, then a chain after the last leaf (the queue fills in one level)."""
    n = 1 + leaves + chain
    src = [0] * leaves + list(range(leaves, leaves + chain))
    dst = list(range(1, leaves + 1)) + list(range(leaves + 1, leaves + chain + 1))
    return _graph(n, src, dst, p)


@pytest.mark.parametrize("leaves", [1, 31, 32, 33, 254, 255, 256, 257, 300, 1000])
@pytest.mark.parametrize("p", [1.0, 0.97])
def test_spread_around_the_queue_size(cuda_lib, leaves, p):
    g = _star(leaves, p)
    gh = cuda_lib.load_graph(g)
    for theta in (1, 7, 65):
        assert cuda_lib.estimate_spread(gh, [0], [], theta, 9, 2) == O.spread(g, [0], [], theta, 9, 2)
        st = cuda_lib.last_stats()
        assert st["samples"] == theta and st["reached"] == O.spread(g, [0], [], theta, 9, 2)
        if p == 1.0:  # every edge is live and examined once per sample, on either route
            assert st["examined_edges"] == theta * g.m and st["live_edges"] == theta * g.m


@pytest.mark.parametrize("model", ["ic", "lt"])
@pytest.mark.parametrize("k", [1, 3, 64])
def test_spread_sets_across_grabs_and_routes(cuda_lib, model, k):
    rng = np.random.default_rng(k)
    n, m = 900, 5000
    e = np.unique(rng.integers(0, n * n, m))
    e = e[e // n != e % n]
    g = _graph(n, e // n, e % n, 0.3, lt=model == "lt")
    seeds = [3, 5, 700]
    rest = np.setdiff1d(np.arange(n), seeds + [8])
    sets = [[int(x) for x in rng.choice(rest, k, replace=False)] for _ in range(5)]
    gh = cuda_lib.load_graph(g, model=model)
    for theta in (1, 33, 400):
        want = O.spread_sets(g, seeds, [8], sets, theta, 4, 1, model=model)
        assert np.array_equal(cuda_lib.estimate_spread_sets(gh, seeds, [8], sets, theta, 4, 1), want)


@pytest.mark.parametrize("deg", [1, 2, 3, 6])
def test_non_tree_targets_few_and_many(cuda_lib, deg):
    """Layered graphs whose samples have from a few hundred to several thousand non-tree edges:
    both ways to resolve their targets, on the regular and the allocation-free entry point (whose
    small slots hold neither the array nor the largest of these cascades)."""
    rng = np.random.default_rng(deg)
    layers, width = 12, 300
    n = layers * width
    src = np.concatenate([np.repeat(np.arange(i * width, (i + 1) * width), deg) for i in range(layers - 1)])
    dst = (src // width + 1) * width + rng.integers(0, width, len(src))
    keys = np.unique(src * n + dst)
    g = _graph(n, keys // n, keys % n, 0.9)
    gh = cuda_lib.load_graph(g)
    seeds, blocked = list(range(0, width, 2)), [width + 1, 2 * width + 7]
    want = O.decrease(g, seeds, blocked, 40, 6, 1)
    assert np.array_equal(cuda_lib.estimate_decrease(gh, seeds, blocked, 40, 6, 1), want)
    assert np.array_equal(cuda_lib.estimate_decrease_noalloc(gh, seeds, blocked, 40, 6, 1), want)


@pytest.mark.parametrize("deg", [3, 5, 31, 32, 33, 130])
def test_warp_tier_chunks(cuda_lib, deg):
    """Frontier chunks of one and of many 32-group windows, with empty rows between full ones."""
    rng = np.random.default_rng(deg)
    n, hubs = 400, 40
    src = np.repeat(np.arange(0, hubs), deg)
    dst = rng.integers(0, n, len(src))
    keys = np.unique((src * n + dst)[src != dst])
    g = _graph(n, keys // n, keys % n, 0.15)
    gh = cuda_lib.load_graph(g)
    seeds = [0, 7, 390, 399]
    for theta in (1, 500):
        assert np.array_equal(cuda_lib.estimate_decrease(gh, seeds, [], theta, 3, 0),
                              O.decrease(g, seeds, [], theta, 3, 0))


@pytest.mark.parametrize("deg,theta", [(1, 14_000), (6, 8_000)])
def test_noalloc_three_launches(cuda_lib, deg, theta):
    """More samples than 20 per whole-graph slot: the allocation-free call runs its warp tier, its
    small slots (which the cascades of the second graph outgrow) and the whole-graph slots."""
    rng = np.random.default_rng(deg)
    layers, width = 12, 300
    n = layers * width
    src = np.concatenate([np.repeat(np.arange(i * width, (i + 1) * width), deg) for i in range(layers - 1)])
    dst = (src // width + 1) * width + rng.integers(0, width, len(src))
    keys = np.unique(src * n + dst)
    g = _graph(n, keys // n, keys % n, 0.8 if deg == 1 else 0.45)
    gh = cuda_lib.load_graph(g)
    seeds, blocked = list(range(0, width, 3)), [width + 1, 2 * width + 7]
    want = O.decrease(g, seeds, blocked, theta, 6, 1)
    assert np.array_equal(cuda_lib.estimate_decrease_noalloc(gh, seeds, blocked, theta, 6, 1), want)


BIG = (1 << 18) + 40  # above 2^18 vertices: the visited bitmap is in the block's slot, whose ids are capped


def _big_star(leaves, seeds, p=1.0):
    """Seed 0 -> `leaves` vertices, the other seeds without edges, on a graph of BIG vertices."""
    dst = list(range(seeds, seeds + leaves))
    return _graph(BIG, [0] * leaves, dst, p)


@pytest.mark.parametrize("seeds", [1, 30, 300])
@pytest.mark.parametrize("room", [-300, -90, -2, -1, 0, 1])
def test_resumed_spread_cascade_against_the_slot_capacity(cuda_lib, monkeypatch, seeds, room):
    """257 leaves, one more than the warp kernel's queue: every cascade is handed over with the seeds
    and 256 leaves and needs 1 + |S| + 257 ids. A slot of fewer reports the capacity error, whether
    the hand-off itself fits it (room -1) or not; one of just as many gives the exact sum."""
    g = _big_star(257, seeds)
    gh = cuda_lib.load_graph(g)
    monkeypatch.setenv("IMIN_CTA_VERTEX_CAP", str(max(1 + seeds + 257 + room, 2)))
    s = list(range(seeds))
    if room < 0:
        for call in (lambda: cuda_lib.estimate_spread(gh, s, [], 40, 9, 2),
                     lambda: cuda_lib.estimate_spread_sets(gh, s, [], [[BIG - 1]], 40, 9, 2)):
            with pytest.raises(cuda_lib.IminError) as ei:
                call()
            assert ei.value.code == -4  # IMIN_ERR_CAPACITY
    else:
        assert cuda_lib.estimate_spread(gh, s, [], 40, 9, 2) == 40 * (seeds + 257)


@pytest.mark.parametrize("seeds,k", [(1, 3), (300, 1), (300, 64)])
def test_spread_sets_handed_over_on_a_large_graph(cuda_lib, seeds, k):
    """Blocker sets whose cascades outgrow the warp kernel on a graph with its bitmap in global memory,
    with few and with more than 256 seeds: the set's vertices stay blocked after the hand-off."""
    g = _big_star(400, seeds, 0.9)
    gh = cuda_lib.load_graph(g)
    s = list(range(seeds))
    rng = np.random.default_rng(k)
    sets = [[int(x) for x in seeds + rng.choice(400, k, replace=False)] for _ in range(3)]
    want = O.spread_sets(g, s, [seeds + 400], sets, 50, 4, 1)
    assert np.array_equal(cuda_lib.estimate_spread_sets(gh, s, [seeds + 400], sets, 50, 4, 1), want)


@pytest.mark.parametrize("cap", [2, 64, 101, 130, 1000])
@pytest.mark.parametrize("seeds,cutoff", [(100, "0"), (30, "0"), (30, "96"), (30, "192")])
def test_start_of_a_sample_against_the_slot_capacity(cuda_lib, monkeypatch, cap, seeds, cutoff):
    """A slot that cannot hold the seeds, or the vertices a warp found before it gave up, leaves the
    sample to the whole-graph tier: counters, blockers and the batched blockers stay the oracle's."""
    src = np.repeat(np.arange(400), 4)
    dst = np.random.default_rng(5).integers(0, 400, len(src))
    keys = np.unique((src * BIG + dst)[src != dst])
    g = _graph(BIG, keys // BIG, keys % BIG, 0.4)
    monkeypatch.setenv("IMIN_CTA_VERTEX_CAP", str(cap))
    monkeypatch.setenv("IMIN_TIER0_VERTICES", cutoff)
    gh = cuda_lib.load_graph(g)
    s = list(range(0, 2 * seeds, 2))
    got, st = cuda_lib.estimate_decrease(gh, s, [399], 60, 3, 1, stats=True)
    assert np.array_equal(got, O.decrease(g, s, [399], 60, 3, 1))
    assert sum(st["tier_samples"]) == 60
    if cap <= seeds:
        assert st["tier_samples"][3] == 0
    want = O.advanced_greedy(g, s, 2, 60, 3)
    assert np.array_equal(cuda_lib.advanced_greedy(gh, s, 2, 60, 3), want)
    assert np.array_equal(cuda_lib.batch_advanced_greedy([(gh, s, 2, 60, 3)])[0], want)


@pytest.mark.parametrize("edges", ["1", "3", "20"])
def test_non_tree_edges_of_a_hand_off_against_the_slot_capacity(cuda_lib, monkeypatch, edges):
    """Block-tier slots of fewer non-tree edges than the warp tier holds (48 at cutoff 192)."""
    src = np.repeat(np.arange(500), 6)
    dst = np.random.default_rng(6).integers(0, 500, len(src))
    keys = np.unique((src * 500 + dst)[src != dst])
    g = _graph(500, keys // 500, keys % 500, 0.25)
    monkeypatch.setenv("IMIN_CTA_EDGE_CAP", edges)
    monkeypatch.setenv("IMIN_TIER0_VERTICES", "192")
    gh = cuda_lib.load_graph(g)
    s = [0, 7, 14, 21]
    got, st = cuda_lib.estimate_decrease(gh, s, [], 3000, 3, 1, stats=True)
    assert np.array_equal(got, O.decrease(g, s, [], 3000, 3, 1))
    assert sum(st["tier_samples"]) == 3000 and st["tier_samples"][2] > 0
    want = O.advanced_greedy(g, s, 2, 500, 3)
    assert np.array_equal(cuda_lib.batch_advanced_greedy([(gh, s, 2, 500, 3)])[0], want)


def _pool_high():
    """Highest number of bytes in use in the device's default memory pool since the last call."""
    import ctypes

    cu = ctypes.CDLL("libcuda.so.1")
    pool, high, zero = ctypes.c_void_p(), ctypes.c_uint64(), ctypes.c_uint64(0)
    used_mem_high = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cu.cuMemPoolGetAttribute(pool, used_mem_high, ctypes.byref(high)) == 0
    assert cu.cuMemPoolSetAttribute(pool, used_mem_high, ctypes.byref(zero)) == 0  # down to what is in use
    return high.value


def test_spread_holds_only_what_it_uses(cuda_lib, monkeypatch):
    """The spread kernels have no whole-graph slots (1 GiB at this size), sample lists or counters: beside
    the block tier's slots, which an Alg. 2 call has too, a spread call holds its hand-offs, 1 KB a sample."""
    rp, col = W.chung_lu(20_000, 100_000, 2.1, 61)
    g = W.Graph(20_000, rp, col, W.wc_thresholds(col, 20_000))
    gh = cuda_lib.load_graph(g)
    monkeypatch.setenv("IMIN_TIER0_VERTICES", "0")
    _pool_high()
    cuda_lib.estimate_decrease(gh, [0, 1], [], 4000, 3, 0)
    alg2 = _pool_high()
    for call in (lambda: cuda_lib.estimate_spread(gh, [0, 1], [], 4000, 3, 0),
                 lambda: cuda_lib.estimate_spread_sets(gh, [0, 1], [], [[5]], 4000, 3, 0)):
        call()
        assert _pool_high() < alg2 - 900_000_000


@pytest.mark.parametrize("mib", [None, "1", "3"])
def test_spread_in_slices(cuda_lib, monkeypatch, mib):
    """More items than a slice holds (2^18, or what a lowered hand-off limit leaves: 992 and 2,978), with
    a last slice that is not full and cascades on both routes."""
    if mib is not None:
        monkeypatch.setenv("IMIN_SPREAD_HANDOFF_MIB", mib)
    g = _star(300, 0.87)  # 261 of 300 leaves on average, the queue holds 256
    gh = cuda_lib.load_graph(g)
    theta = 90_001 if mib is None else 2_001
    sets = [[5], [6], [301]]
    want = O.spread_sets(g, [0], [], sets, theta, 4, 1)
    assert np.array_equal(cuda_lib.estimate_spread_sets(gh, [0], [], sets, theta, 4, 1), want)
    assert cuda_lib.estimate_spread(gh, [0], [5], theta, 4, 1) == int(want[0])


@pytest.mark.parametrize("n,m,thetas", [
    (300, 1500, [4864, 4865]),        # a whole-graph slot for each of the 1,216 resident blocks
    (2047, 20_000, [1300, 1800]),     # 389 slots: the line is at 1,556, for slots with and without room
    (2048, 20_000, [1300, 1800]),     # for every vertex
    (2049, 20_000, [1300, 1800]),
    (8192, 65_536, [2000, 2001]),     # 227 slots
    (50_021, 400_009, [900, 1400]),   # 58 slots
])
def test_noalloc_route_by_samples(cuda_lib, n, m, thetas):
    """One launch up to the rule's number of samples, three beyond it, the same counters either way."""
    rp, col = W.chung_lu(n, m, 2.1, 71)
    g = W.Graph(n, rp, col, W.wc_thresholds(col, n))
    gh = cuda_lib.load_graph(g)
    s = W.uniform_seeds(n, 12, 72)
    launched = []
    for theta in thetas:
        c0 = cuda_lib.launch_count()
        got = cuda_lib.estimate_decrease_noalloc(gh, s, [], theta, 6, 1)
        launched.append(cuda_lib.launch_count() - c0)
        assert np.array_equal(got, O.decrease(g, s, [], theta, 6, 1))
    assert launched == [2, 4], launched  # the mask, then one or three tiers


@pytest.mark.parametrize("model", ["ic", "lt"])
@pytest.mark.parametrize("cutoff", ["64", "192"])
def test_few_and_many_samples_per_warp(cuda_lib, monkeypatch, model, cutoff):
    """Both register budgets of the warp tier on one graph: the line is at two samples per resident warp,
    12,160 with 5 blocks per SM and 7,296 with 3."""
    rp, col = W.chung_lu(1500, 7000, 2.1, 81)
    g = W.Graph(1500, rp, col, W.lt_wc_weights(col, 1500) if model == "lt" else W.wc_thresholds(col, 1500))
    monkeypatch.setenv("IMIN_TIER0_VERTICES", cutoff)
    gh = cuda_lib.load_graph(g, model=model)
    s = W.uniform_seeds(g.n, 100, 82)
    for theta in (7296, 7297, 9728, 9729, 12160, 12161):
        want = O.decrease(g, s, [], theta, 6, 1, model=model)
        assert np.array_equal(cuda_lib.estimate_decrease(gh, s, [], theta, 6, 1), want)
