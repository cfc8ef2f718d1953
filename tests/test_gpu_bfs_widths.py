"""Every width of a BFS launch against the oracle: groups of 2 to 32 lanes with
and without parents, work dealt out in advance and by tickets, and a batch whose
words are split over two launches.  Graphs of many levels, and dense ones whose
degrees are alike, are not slowed by what large skewed graphs gain from."""
import os
import time
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2311_00869_gb300 as P

    return P


def _hub_graph(n, m, hub, seed):
    """Connected, with one vertex of `hub` further neighbours."""
    _, u, v, _ = synth.random_connected(n, m, 0.3, seed=seed)
    ends = np.arange(1, hub + 1)
    key = np.unique(np.concatenate([np.minimum(u, v).astype(np.int64) * n + np.maximum(u, v), ends]))
    s = np.where(np.arange(key.size) % 3 == 0, -1, 1).astype(np.int8)
    return n, (key // n).astype(np.int32), (key % n).astype(np.int32), s


def _counts_hashes(g, seed, t0, K):
    cores = os.cpu_count() or 1
    cut = np.linspace(0, K, min(K, 4 * cores) + 1).astype(int)
    with ThreadPoolExecutor(max_workers=cores) as ex:
        parts = list(ex.map(lambda i: O.sample(g, seed, t0 + int(cut[i]), int(cut[i + 1] - cut[i]), want_labels=False),
                            range(len(cut) - 1)))
    return (np.concatenate([p[k] for p in parts]) for k in ("counts", "hashes"))


# lanes asked for are used when they are one or two per half-word of the launch
@pytest.mark.parametrize("K,group", [(1, 2), (32, 4), (60, 2), (101, 4), (101, 8), (200, 8), (200, 16), (400, 16), (400, 32),
                                     (1000, 32)])
@pytest.mark.parametrize("parents", [False, True])
def test_group_of_every_width(P, K, group, parents):
    n, u, v, s = _hub_graph(900, 1500, 700, seed=61)
    g = O.clean_graph(n, u, v, s)
    sb = P.SignedBal(0)
    try:
        sb.load_graph(n, u, v, s)
        sb.set_tuning(bfs_group=group)
        par = sb.sample_trees(7, 40, K, want_parents=parents)
        counts, hashes = sb.frustration()
        ref = O.sample(g, 7, 40, K, want_labels=True, want_parents=True)
        assert np.array_equal(counts.cpu().numpy(), ref["counts"])
        assert np.array_equal(hashes.cpu().numpy().view(np.uint64), ref["hashes"])
        assert np.array_equal(P.unpack_labels(sb.label(), K), ref["labels"])
        if parents:
            assert np.array_equal(par.cpu().numpy(), ref["parents"])
    finally:
        sb.close()


# 120,001 vertices: 100 trees 4 lanes in 3 rounds and 400 trees 16 lanes in 14,
# 600 trees whole warps in 28; 20,000: whole warps in 4
@pytest.mark.parametrize("n,K", [(120001, 100), (120001, 400), (120001, 600), (20000, 600)])
def test_dealt_out_and_by_tickets(P, n, K):
    n, u, v, s = _hub_graph(n, 2 * n, 1500, seed=63)
    g = O.clean_graph(n, u, v, s)
    sb = P.SignedBal(0)
    try:
        sb.load_graph(n, u, v, s)
        sb.sample_trees(5, 11, K)
        counts, hashes = sb.frustration()
        want_c, want_h = _counts_hashes(g, 5, 11, K)
        assert np.array_equal(counts.cpu().numpy(), want_c)
        assert np.array_equal(hashes.cpu().numpy().view(np.uint64), want_h)
    finally:
        sb.close()


# 17, 18 and 23 words: two launches, one on a graph too small to fill a round
@pytest.mark.parametrize("n,K,launches", [(6000, 1030, 2), (6000, 1100, 2), (6000, 1472, 2), (1500, 1030, 1), (1500, 1472, 1)])
def test_words_split_over_two_launches(P, n, K, launches):
    n, u, v, s = _hub_graph(n, 2 * n, 700, seed=64)
    g = O.clean_graph(n, u, v, s)
    sb = P.SignedBal(0)
    try:
        sb.load_graph(n, u, v, s)
        par = sb.sample_trees(9, 3, K, want_parents=True)
        assert sb.stats()["bfs_launches"] == launches
        counts, hashes = sb.frustration()
        ref = O.sample(g, 9, 3, K, want_labels=True, want_parents=True)
        assert np.array_equal(counts.cpu().numpy(), ref["counts"])
        assert np.array_equal(hashes.cpu().numpy().view(np.uint64), ref["hashes"])
        assert np.array_equal(P.unpack_labels(sb.label(), K), ref["labels"])
        assert np.array_equal(par.cpu().numpy(), ref["parents"])
    finally:
        sb.close()


def test_split_words_with_slots_in_another_order(P):
    """262,144 vertices and more: 1100 trees of two launches, a spread of them
    against the oracle."""
    K, t0 = 1100, 4
    n, u, v, s = synth.random_connected(270001, 400000, 0.3, seed=62)
    g = O.clean_graph(n, u, v, s)
    sb = P.SignedBal(0)
    try:
        sb.load_graph(n, u, v, s)
        sb.sample_trees(3, t0, K)
        assert sb.stats()["bfs_launches"] == 2
        counts, hashes = (x.cpu().numpy() for x in sb.frustration())
        words = sb.label().cpu().numpy().view(np.uint64)
        picks = sorted({0, 1, 31, 32, 63, 64, 1023, 1024, 1055, 1056, 1087, 1088, 1099} | set(range(5, K, 97)))
        with ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as ex:
            refs = list(ex.map(lambda t: O.sample(g, 3, t0 + t, 1), picks))
        for t, ref in zip(picks, refs):
            assert counts[t] == ref["counts"][0] and hashes.view(np.uint64)[t] == ref["hashes"][0], t
            bits = (words[:, t // 64] >> np.uint64(t % 64)) & np.uint64(1)
            assert np.array_equal(bits.astype(np.uint8), ref["labels"][0]), t
    finally:
        sb.close()


def _ms(sb, K, reps=5):
    best = np.inf
    for _ in range(reps + 1):
        t = time.perf_counter()
        sb.sample_trees(1, 0, K)
        sb.sync()
        best = min(best, 1e3 * (time.perf_counter() - t))
    return best


def _grid(k):
    i = np.arange(k * k, dtype=np.int32).reshape(k, k)
    u, v = np.concatenate([i[:, :-1].ravel(), i[:-1].ravel()]), np.concatenate([i[:, 1:].ravel(), i[1:].ravel()])
    return k * k, u, v, np.where((u * 7 + v) % 5 == 0, -1, 1).astype(np.int8)


def test_levels_with_little_work_are_short(P):
    """A level of a 300 x 300 grid (two rounds of work) against one of a 100 x 100
    grid (less than one): 3.5 times as long is allowed (5.2 times when every warp
    drew tickets at each level)."""
    per_level = []
    sb = P.SignedBal(0)
    try:
        for k in (100, 300):
            sb.load_graph(*_grid(k))
            per_level.append(_ms(sb, 64) / sb.stats()["bfs_levels"])
    finally:
        sb.close()
    assert per_level[1] <= 3.5 * per_level[0], per_level


def test_dense_graphs_of_even_degrees_keep_narrow_groups(P):
    """100,000 vertices of about 60 neighbours, 64 trees: the rule's width takes at
    most 1.3 times what one lane per half-word does (4.3 times with whole warps)."""
    rng = np.random.Generator(np.random.PCG64(65))
    n = 100000
    key = np.unique(rng.integers(0, n, 6_000_000) * n + rng.integers(0, n, 6_000_000))
    u, v = key // n, key % n
    k = u < v
    sb = P.SignedBal(0)
    try:
        sb.load_graph(n, u[k].astype(np.int32), v[k].astype(np.int32), np.where(key[k] % 4 == 0, -1, 1).astype(np.int8))
        by_rule = _ms(sb, 64)
        sb.set_tuning(bfs_group=2)
        assert by_rule <= 1.3 * _ms(sb, 64)
    finally:
        sb.close()
