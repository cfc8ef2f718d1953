"""Ingest at sizes around the sort's 4096-key tiles and where components are
first joined on samples of the edges (2^16 edges and more): edges, CSR rows,
vertex map and the scorer's counts equal the oracle's."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 255, 4095, 4096, 4097, 8193, 65535, 65537, 200001])
@pytest.mark.parametrize("ids", [3, 8])  # edges per vertex id; many components at 1/3
def test_ingest_sizes_match_oracle(m, ids):
    import paper_2311_00869_gb300 as P

    n = max(2, m // ids if ids > 3 else m * 3 // 2)
    rng = np.random.Generator(np.random.PCG64(m + ids))
    # a heavy tail of degrees, with many equal ones
    a = (n * rng.random(m) ** 3).astype(np.int64)
    b = rng.integers(0, n, m)
    keep = a != b
    lo, hi = np.minimum(a, b)[keep], np.maximum(a, b)[keep]
    _, first = np.unique(lo * n + hi, return_index=True)
    order = rng.permutation(first.size)
    u, v = lo[first][order].astype(np.int32), hi[first][order].astype(np.int32)
    s = np.where(rng.random(u.size) < 0.3, -1, 1).astype(np.int8)
    again = rng.integers(0, max(u.size, 1), u.size // 9)
    u, v, s = np.concatenate([u, v[again]]), np.concatenate([v, u[again]]), np.concatenate([s, s[again]])
    g = O.clean_graph(n, u, v, s)
    sb = P.SignedBal(0)
    try:
        n1, m1, vmap = sb.load_graph(n, u, v, s, want_vmap=True)
        assert (n1, m1) == (g.n, g.m) and np.array_equal(vmap, g.vmap)
        if g.m == 0:
            return
        eu, ev, neg = (t.cpu().numpy() for t in sb.graph_edges())
        assert np.array_equal(eu, g.eu) and np.array_equal(ev, g.ev) and np.array_equal(neg, g.eneg)
        rp, col, cneg = (t.cpu().numpy() for t in sb.graph_csr())
        assert np.array_equal(rp, g.rowptr.astype(np.int32))
        assert np.array_equal(col, g.col) and np.array_equal(cneg, g.colneg)
        sb.sample_trees(5, 0, 3)
        ref = O.sample(g, 5, 0, 3, want_labels=False)
        assert np.array_equal(sb.frustration()[0].cpu().numpy(), ref["counts"])
    finally:
        sb.close()
