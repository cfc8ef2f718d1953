"""A batch whose sampling gave up (a barrier that ran out of its bounded wait)
reaches no cloud: every route to one reports the failure and leaves the
states gathered before as they were."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu
TIMEOUT = -12


def _refused(P, call):
    with pytest.raises(P.SignedBalError) as e:
        call()
    assert e.value.code == TIMEOUT


def test_cloud_refuses_a_failed_batch_and_keeps_its_states():
    import paper_2311_00869_gb300 as P

    n, u, v, s = synth.random_connected(300, 900, 0.3, seed=43)
    g = O.clean_graph(n, u, v, s)
    sb = P.SignedBal(0)
    try:
        sb.load_graph(n, u, v, s)
        sb.cloud_reset()
        sb.sample_trees(3, 0, 64)
        before = sb.cloud()
        sb.set_tuning(wait_us=20000, stall_test=1)
        sb.sample_trees(3, 64, 64)
        _refused(P, sb.cloud)
        _refused(P, sb.cloud_insert)
        _refused(P, lambda: sb.cloud_state(0))
        sb.set_tuning(wait_us=0)
        sb.sample_trees(3, 64, 64)  # the same trees, this time grown to the end
        after = sb.cloud()
        ref = O.sample(g, 3, 0, 128)
        for k, (cl, fr) in ((64, before), (128, after)):
            rc = O.cloud(ref["labels"][:k], ref["counts"][:k])
            assert np.array_equal(cl["first_tree"], rc["first_tree"]) and np.array_equal(cl["S"], rc["S"])
            assert np.array_equal(cl["count"], rc["count"]) and fr == rc["S"].min()
    finally:
        sb.close()


@pytest.mark.parametrize("steps", [0, 2])
def test_batch_cloud_refuses_a_failed_batch(steps):
    import paper_2311_00869_gb300 as P

    graphs = [synth.chung_lu(n, 6.0, 2.5, 0.2, seed=n) for n in (50, 200)]
    sb = P.SignedBal(0)
    try:
        sb.load_batch(graphs)
        sb.set_tuning(wait_us=20000, stall_test=1)
        if steps:
            sb.batch_steps(1, 0, 64, steps, use_graph=False)
        else:
            sb.sample_trees(1, 0, 64)
        _refused(P, sb.batch_cloud)
    finally:
        sb.close()
