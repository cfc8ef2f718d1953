"""Ingest of graphs in their natural vertex order (users before items, a star
from its centre, a path end to end): long stretches of ids that are never an
edge's smaller or larger end, and long chains of joins.  Edges and rows equal
the oracle's, and such an order does not make a load slow."""
import time

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def _signs(m):
    return np.where(np.arange(m) % 3 == 0, -1, 1).astype(np.int8)


def star(n, centre):
    v = np.delete(np.arange(n, dtype=np.int32), centre)
    return n, np.full(n - 1, centre, np.int32), v, _signs(n - 1)


def path(n):
    u = np.arange(n - 1, dtype=np.int32)
    return n, u, u + 1, _signs(n - 1)


def bipartite(users, items, m, seed=5):
    """Users 0 .. users - 1, then items; every vertex has an edge."""
    rng = np.random.Generator(np.random.PCG64(seed))
    u = np.concatenate([rng.integers(0, users, m), np.arange(items) % users, np.arange(users)])
    v = np.concatenate([(items * rng.random(m) ** 2).astype(np.int64), np.arange(items), rng.integers(0, items, users)])
    key = np.unique(u * items + v)
    rng.shuffle(key)
    return users + items, (key // items).astype(np.int32), (key % items + users).astype(np.int32), _signs(key.size)


def permuted(g, seed=6):
    p = np.random.Generator(np.random.PCG64(seed)).permutation(g[0]).astype(np.int32)
    return g[0], p[g[1]], p[g[2]], g[3]


@pytest.mark.parametrize("graph", [lambda n: star(n, 0), lambda n: star(n, n // 2), lambda n: star(n, n - 1), path,
                                   lambda n: bipartite(n // 5, n - n // 5, 2 * n),
                                   lambda n: bipartite(n - n // 5, n // 5, 2 * n)],
                         ids=["star_first", "star_middle", "star_last", "path", "users_items", "items_users"])
@pytest.mark.parametrize("n", [10, 1000, 70001])
def test_natural_orders_match_oracle(graph, n):
    import paper_2311_00869_gb300 as P

    g = graph(n)
    ref = O.clean_graph(*g)
    sb = P.SignedBal(0)
    try:
        assert sb.load_graph(*g)[:2] == (ref.n, ref.m)
        eu, ev, neg = (t.cpu().numpy() for t in sb.graph_edges())
        assert np.array_equal(eu, ref.eu) and np.array_equal(ev, ref.ev) and np.array_equal(neg, ref.eneg)
        rp, col, cneg = (t.cpu().numpy() for t in sb.graph_csr())
        assert np.array_equal(rp, ref.rowptr.astype(np.int32))
        assert np.array_equal(col, ref.col) and np.array_equal(cneg, ref.colneg)
    finally:
        sb.close()


def test_graphs_without_edges_between_others():
    """A run of single vertices in a batch: rows with nothing in them."""
    import paper_2311_00869_gb300 as P

    none = np.array([], np.int32)
    graphs = [path(50)] + [(1, none, none, none.astype(np.int8))] * 300 + [star(70, 3)]
    sb = P.SignedBal(0)
    try:
        nv, mv = sb.load_batch(graphs)
        assert list(nv) == [50] + [1] * 300 + [70] and list(mv) == [49] + [0] * 300 + [69]
        rp = sb.graph_csr()[0].cpu().numpy()
        deg = np.concatenate([[1], np.full(48, 2), [1], np.zeros(300, int), np.where(np.arange(70) == 3, 69, 1)])
        assert np.array_equal(rp, np.concatenate([[0], np.cumsum(deg)]))
    finally:
        sb.close()


def _load_ms(sb, g):
    import torch

    dev = (g[0],) + tuple(torch.from_numpy(a).cuda() for a in g[1:])
    best = np.inf
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        sb.load_graph(*dev)
        best = min(best, 1e3 * (time.perf_counter() - t))
    return best


def test_users_before_items_load_as_fast_as_any_order():
    """2 M users and 8 M items: half as long again as the same graph with its ids
    permuted is allowed (one thread filling each side's rows took 3.6 times)."""
    import paper_2311_00869_gb300 as P

    g = bipartite(2_000_000, 8_000_000, 22_000_000)
    sb = P.SignedBal(0)
    try:
        assert _load_ms(sb, g) <= 1.5 * _load_ms(sb, permuted(g))
    finally:
        sb.close()
