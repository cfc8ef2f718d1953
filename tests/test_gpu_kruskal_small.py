"""Kruskal trees of batches of small graphs (fewer vertices each than the edge
ends one would sample to find a largest component) against the oracle, with and
without rounds over light edges."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graphs", [
    lambda: [synth.random_connected(n, n + n // 3, 0.3, seed=n) for n in range(2, 41)],
    lambda: [synth.er_graph(16, 110, 0.3, seed=k) for k in range(1000)],
], ids=["sparse", "light_rounds"])
def test_small_graphs_match_oracle(graphs):
    import paper_2311_00869_gb300 as P

    graphs = graphs()
    K = 300
    sb = P.SignedBal(0)
    try:
        sb.load_batch(graphs)
        sb.sample_trees_kruskal(5, 2, K)
        counts, hashes = (x.cpu().numpy() for x in sb.batch_frustration())
        for g in range(0, len(graphs), max(1, len(graphs) // 60)):
            ref = O.mst_sample(O.clean_graph(*graphs[g]), 5, 2, K, want_labels=False)
            assert np.array_equal(counts[g], ref["counts"]), g
            assert np.array_equal(hashes[g].view(np.uint64), ref["hashes"]), g
    finally:
        sb.close()
