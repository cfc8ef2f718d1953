"""A captured batch step is replayed only while everything it was captured
with is as it was: buffers that a call with more trees has regrown, and a
barrier test in between, lead to a new capture."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


def _graphs():
    return [synth.chung_lu(n, 6.0, 2.5, 0.2, seed=70 + n) for n in (40, 333, 90, 1200, 7)]


def _check(sb, refs, seed, t0, K, steps):
    fr, ns = sb.batch_steps(seed, t0, K, steps, use_graph=True)
    sb.sync()
    counts, hashes = (t.cpu().numpy() for t in sb.batch_frustration())
    for g, r in enumerate(refs):
        ref = O.sample(r, seed, t0, K * steps)
        last = slice((steps - 1) * K, steps * K)
        assert fr[g] == ref["counts"].min(), g
        assert np.array_equal(counts[g], ref["counts"][last]), g
        assert np.array_equal(hashes[g].view(np.uint64), ref["hashes"][last]), g
        assert ns[g] == O.cloud(ref["labels"][last], ref["counts"][last])["S"].shape[0], g


@pytest.mark.parametrize("between", ["sample_trees", "batch_steps", "kruskal"])
def test_more_trees_between_two_captured_calls(between):
    import paper_2311_00869_gb300 as P

    graphs = _graphs()
    refs = [O.clean_graph(*g) for g in graphs]
    sb = P.SignedBal(0)
    try:
        sb.load_batch(graphs)
        _check(sb, refs, 3, 10, 64, 4)
        if between == "sample_trees":
            sb.sample_trees(3, 0, 1000)
        elif between == "kruskal":
            sb.sample_trees_kruskal(3, 0, 1000)
        else:
            sb.batch_steps(3, 0, 700, 1, use_graph=False)
        _check(sb, refs, 3, 500, 64, 4)
    finally:
        sb.close()


def test_capture_during_a_barrier_test_is_not_replayed():
    import paper_2311_00869_gb300 as P

    graphs = _graphs()
    refs = [O.clean_graph(*g) for g in graphs]
    sb = P.SignedBal(0)
    try:
        sb.load_batch(graphs)
        sb.set_tuning(wait_us=20000, stall_test=1)
        sb.batch_steps(3, 0, 64, 2, use_graph=True)
        with pytest.raises(P.SignedBalError) as e:
            sb.sync()
        assert e.value.code == -12
        _check(sb, refs, 3, 0, 64, 3)
    finally:
        sb.close()


@pytest.mark.parametrize("use_graph", [True, False])
def test_clouds_after_steps_are_the_last_steps(use_graph):
    """The batch that sb_batch_steps leaves is the last step's: the per-graph
    clouds taken from it name that step's trees."""
    import paper_2311_00869_gb300 as P

    graphs = _graphs()
    K, steps, t0 = 64, 3, 20
    sb = P.SignedBal(0)
    try:
        sb.load_batch(graphs)
        sb.batch_steps(5, t0, K, steps, use_graph=use_graph)
        sb.sync()
        cl = sb.batch_cloud()
        for g, r in enumerate(O.clean_graph(*x) for x in graphs):
            ref = O.sample(r, 5, t0 + (steps - 1) * K, K)
            rc = O.cloud(ref["labels"], ref["counts"], t0=t0 + (steps - 1) * K)
            assert cl["n_states"][g] == rc["S"].shape[0], g
            for k, o in (("first_tree", "first_tree"), ("count", "count"), ("S", "S"), ("hash", "H")):
                assert np.array_equal(cl["entries"][g][k], rc[o]), (g, k)
    finally:
        sb.close()
