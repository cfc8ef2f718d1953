"""How the BFS spreads trees over lanes and work over warps never shows: any
group width gives the oracle's trees, and a graph large enough for slots in
another order than the trees gives them back in tree order everywhere."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2311_00869_gb300 as P

    return P


@pytest.mark.parametrize("group", [2, 8, 16, 32])
@pytest.mark.parametrize("K", [1, 33, 100, 520])
def test_group_widths_match_oracle(P, group, K):
    """Groups from one lane per half-word to 32 lanes per vertex, on a graph with
    a split row and leaves."""
    n, u, v, s = synth.random_connected(900, 1500, 0.3, seed=61)
    hub = np.arange(1, 700, dtype=np.int32)
    lo = np.concatenate([np.minimum(u, v), np.zeros_like(hub)]).astype(np.int64)
    hi = np.concatenate([np.maximum(u, v), hub]).astype(np.int64)
    _, first = np.unique(lo * n + hi, return_index=True)
    u, v = lo[first].astype(np.int32), hi[first].astype(np.int32)
    s = np.where(np.arange(first.size) % 3 == 0, -1, 1).astype(np.int8)
    g = O.clean_graph(n, u, v, s)
    sb = P.SignedBal(0)
    try:
        sb.load_graph(n, u, v, s)
        sb.set_tuning(bfs_group=group)
        for parents in (True, False):
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


@pytest.mark.parametrize("K", [64, 101])
def test_reordered_slots_give_trees_in_order(P, K):
    """262,144 vertices and more: counts, hashes, labels, parents and a cloud
    whose 3-bit keys send most trees through the exact comparison."""
    n, u, v, s = synth.random_connected(270001, 400000, 0.3, seed=62)
    g = O.clean_graph(n, u, v, s)
    ref = O.sample(g, 3, 9, K, want_labels=True, want_parents=True)
    sb = P.SignedBal(0)
    try:
        assert sb.load_graph(n, u, v, s)[:2] == (g.n, g.m)
        sb.cloud_reset(0, 3)
        par = sb.sample_trees(3, 9, K, want_parents=True)
        counts, hashes = sb.frustration()
        assert np.array_equal(counts.cpu().numpy(), ref["counts"])
        assert np.array_equal(hashes.cpu().numpy().view(np.uint64), ref["hashes"])
        assert np.array_equal(P.unpack_labels(sb.label(), K), ref["labels"])
        assert np.array_equal(par.cpu().numpy(), ref["parents"])
        cl, fr = sb.cloud()
        rc = O.cloud(ref["labels"], ref["counts"])
        assert np.array_equal(cl["first_tree"], rc["first_tree"] + 9) and np.array_equal(cl["S"], rc["S"])
        assert np.array_equal(cl["count"], rc["count"]) and fr == rc["S"].min()
        state = sb.cloud_state(0).cpu().numpy().view(np.uint64)
        bits = (state[:, None] >> np.arange(64, dtype=np.uint64)) & np.uint64(1)
        assert np.array_equal(bits.reshape(-1)[: g.n].astype(np.uint8), ref["labels"][0])
    finally:
        sb.close()
