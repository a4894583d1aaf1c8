"""When the warp/block cutoff is tuned: by the samples that the calls on a graph and seed-set size
class draw together, over all their rounds. Launch counts tell a call that tuned from one that ran
only its own kernels; results never depend on it."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from paper_2302_13529_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TIMED_CALLS = 15  # 5 candidates, 3 calls each, of at least 2 kernels


@pytest.fixture(autouse=True)
def _tuner_on(monkeypatch):
    monkeypatch.delenv("IMIN_TIER0_VERTICES", raising=False)
    monkeypatch.delenv("IMIN_AUTOTUNE", raising=False)


def _launches(lib, call):
    c0 = lib.launch_count()
    out = call()
    return lib.launch_count() - c0, out


def _chung_lu(n, m, seed):
    rp, col = W.chung_lu(n, m, 2.1, seed)
    return W.Graph(n, rp, col, W.wc_thresholds(col, n))


def test_all_rounds_of_a_greedy_call_count(cuda_lib):
    """160 rounds of 10^5 samples, each far shorter than the tuning, are more than 16 times the samples it
    times (15 calls of 65,536): the first call tunes."""
    g = _chung_lu(2000, 10000, 501)
    gh = cuda_lib.load_graph(g)
    s = W.uniform_seeds(g.n, 10, 502)
    first, b1 = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, 160, 100_000, 7))
    second, b2 = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, 160, 100_000, 7))
    third, b3 = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, 160, 100_000, 7))
    assert first >= second + 2 * TIMED_CALLS and second == third, (first, second, third)
    assert np.array_equal(b1, b2) and np.array_equal(b2, b3)


def test_short_calls_add_up_and_a_long_one_tunes(cuda_lib):
    """Calls of 1,000 samples: default cutoff, own kernels only. The 17th brings the sum past 16,384 and runs
    the warm-up, once. A batch query and a request count too, and the call that completes the sum tunes."""
    g = _chung_lu(2000, 10000, 511)
    gh = cuda_lib.load_graph(g)
    s = W.uniform_seeds(g.n, 10, 512)
    want = O.decrease(g, s, [], 1000, 3, 0)
    counts = []
    for _ in range(20):
        n, got = _launches(cuda_lib, lambda: cuda_lib.estimate_decrease(gh, s, [], 1000, 3, 0))
        assert np.array_equal(got, want)
        counts.append(n)
    assert counts[16] > counts[0] and set(counts[:16] + counts[17:]) == {counts[0]}, counts
    cuda_lib.batch_advanced_greedy([(gh, s, 75, 100_000, 7)])
    tuned, _ = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, 85, 100_000, 7))
    after, _ = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, 85, 100_000, 7))
    assert tuned >= after + 2 * TIMED_CALLS, (tuned, after)
    assert np.array_equal(cuda_lib.estimate_decrease(gh, s, [], 1000, 3, 0), want)


def test_huge_cascades_drop_the_warp_tier_below_1024_samples_a_round(cuda_lib, monkeypatch):
    """28 rounds of 600 samples on a graph whose cascades all outgrow the warp tier: the warm-up sees it,
    and the rounds run without that tier from then on, like calls with a forced cutoff of 0."""
    rp, col = W.chung_lu(8000, 48000, 2.1, 521)
    g = W.Graph(8000, rp, col, np.full(len(col), int(0.3 * 2**32), np.uint32))
    gh = cuda_lib.load_graph(g)
    hubs = np.argsort(-g.out_degree())[:20].astype(np.int32)
    cuda_lib.advanced_greedy(gh, hubs, 28, 600, 7)
    got, b = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, hubs, 3, 600, 7))
    monkeypatch.setenv("IMIN_TIER0_VERTICES", "0")
    forced, b0 = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, hubs, 3, 600, 7))
    monkeypatch.setenv("IMIN_TIER0_VERTICES", "96")
    with_warp, _ = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, hubs, 3, 600, 7))
    assert got == forced < with_warp, (got, forced, with_warp)
    assert np.array_equal(b, b0) and np.array_equal(b, O.advanced_greedy(g, hubs, 3, 600, 7))


def test_a_tuned_cutoff_is_shared_by_handles_of_one_graph(cuda_lib):
    """The first handle is tuned; a second one of the same graph takes its cutoff: the call that would
    otherwise run the warm-up launches only its own kernels and fills the same tiers."""
    g = W.graph_rmat_wc(12, 40000, seed=531)
    s = W.uniform_seeds(g.n, 20, seed=532)
    want = O.decrease(g, s, [], 2000, 43, 1)
    h1 = cuda_lib.load_graph(g)
    cuda_lib.autotune(h1, s, 43)
    n1, (d1, st1) = _launches(cuda_lib, lambda: cuda_lib.estimate_decrease(h1, s, [], 2000, 43, 1, stats=True))
    h2 = cuda_lib.load_graph(g)
    n2, (d2, st2) = _launches(cuda_lib, lambda: cuda_lib.estimate_decrease(h2, s, [], 2000, 43, 1, stats=True))
    assert n1 == n2 <= 4 and st1["tier_samples"] == st2["tier_samples"], (n1, n2, st1, st2)
    assert np.array_equal(d1, want) and np.array_equal(d2, want)


@pytest.mark.parametrize("theta,rounds,budget", [(100_000, 160, 5), (7_000, 1001, 4)])
def test_the_tuner_times_the_kernels_of_the_call(cuda_lib, theta, rounds, budget):
    """The warp tier has one instantiation for rounds of more than two samples per resident warp (5 blocks
    per SM) and one for fewer (4); the line lies at 7,296 samples where a cutoff leaves 3 blocks per SM,
    at 12,160 where it leaves 5. A call that tunes runs only its own, in the warm-up and the timed calls
    too, whatever their sample counts."""
    import re

    import torch
    from torch.profiler import ProfilerActivity, profile

    g = _chung_lu(2000, 10000, 541 + budget)
    gh = cuda_lib.load_graph(g)
    s = W.uniform_seeds(g.n, 10, 542)
    with profile(activities=[ProfilerActivity.CUDA]):  # the first use sets the profiler up
        torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        n, _ = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, rounds, theta, 7))
        torch.cuda.synchronize()
    own, _ = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, rounds, theta, 7))
    assert n >= own + 2 * TIMED_CALLS, (n, own)
    seen = [m.group(1) for e in prof.events() if (m := re.search(r"k_sample_tier<0, 0, (\d)u?>", e.name))]
    if not seen:
        pytest.skip("no kernel records from the profiler here")
    assert set(seen) == {str(budget)} and len(seen) > TIMED_CALLS, (set(seen), len(seen))


def test_equal_candidates_leave_the_default(cuda_lib):
    """Cascades of a few vertices: candidates from 64 on do the same work per sample, and what else a timed
    call of 0.05 ms costs (fewer blocks at larger cutoffs) may not decide between them."""
    rp, col = W.chung_lu(40_000, 200_000, 2.1, 551)
    g = W.Graph(40_000, rp, col, np.full(len(col), int(0.002 * 2**32), np.uint32))
    gh = cuda_lib.load_graph(g)
    s = W.uniform_seeds(g.n, 10, 552)
    assert [cuda_lib.autotune(gh, s, k) for k in range(12)] == [96] * 12


def test_a_costly_warm_up_runs_once_per_graph(cuda_lib):
    """A warm-up that shows huge cascades is repeated only in a process's first use of its kernels: later
    graphs of the kind pay for one (the mask and three tiers)."""
    counts = []
    for seed in (561, 562, 563):
        rp, col = W.chung_lu(8000, 48000, 2.1, seed)
        g = W.Graph(8000, rp, col, np.full(len(col), int(0.3 * 2**32), np.uint32))
        gh = cuda_lib.load_graph(g)
        hubs = np.argsort(-g.out_degree())[:20].astype(np.int32)
        n, _ = _launches(cuda_lib, lambda: cuda_lib.autotune(gh, hubs, 7))
        counts.append(n)
    assert counts[1] == counts[2] <= 4, counts


def test_a_first_short_call_runs_its_own_kernels_only(cuda_lib):
    """Short rounds, fewer than 16,384 samples over all of them, in one call of a driver or in the queries of
    a batch: no warm-up, whose 1,024 samples would be a good part of the call."""
    g = _chung_lu(3000, 15000, 571)
    s = W.uniform_seeds(g.n, 10, 572)
    gh = cuda_lib.load_graph(g)
    first, b1 = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, 16, 500, 7))
    second, b2 = _launches(cuda_lib, lambda: cuda_lib.advanced_greedy(gh, s, 16, 500, 7))
    assert first == second and np.array_equal(b1, b2), (first, second)
    graphs = [cuda_lib.load_graph(_chung_lu(3000, 15000, 573 + i)) for i in range(3)]
    items = [(h, s, 16, 500, 7) for h in graphs]
    first, r1 = _launches(cuda_lib, lambda: cuda_lib.batch_advanced_greedy(items))
    second, r2 = _launches(cuda_lib, lambda: cuda_lib.batch_advanced_greedy(items))
    assert first == second and all(np.array_equal(a, b) for a, b in zip(r1, r2)), (first, second)


def test_one_query_of_a_batch_does_not_set_the_capacity_for_all(cuda_lib):
    """Cascades of exactly 80 or 150 vertices besides the seeds: 96 and 192 are the smallest candidates that
    hold them. A batch of two of the first and one of the second runs its warp launch at 96 (the
    third query's samples go to the block tier), one of the second alone at 192."""
    def star(leaves, n):
        row = np.zeros(n + 1, np.int32)
        row[1:] = leaves
        return W.Graph(n, row, np.arange(20, 20 + leaves, dtype=np.int32), np.full(leaves, 2**32 - 1, np.uint32))

    s = list(range(20))
    graphs = [star(80, 900), star(80, 901), star(150, 902)]
    handles = [cuda_lib.load_graph(g) for g in graphs]
    cuts = [cuda_lib.autotune(h, s, 1) for h in handles]
    assert cuts == [96, 96, 192], cuts
    theta = 300
    items = [(h, s, 1, theta, 5) for h in handles]
    found = cuda_lib.batch_advanced_greedy(items)
    assert list(cuda_lib.last_stats()["tier_samples"]) == [2 * theta, 0, 0, theta]
    assert cuda_lib.batch_advanced_greedy(items[2:])[0].tolist() == found[2].tolist() == [20]
    assert list(cuda_lib.last_stats()["tier_samples"]) == [theta, 0, 0, 0]
