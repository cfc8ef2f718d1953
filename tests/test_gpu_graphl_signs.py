"""graphL's discrete losses from sign words: at widths around the kernels' 4, 32,
64 and 128 column steps, on a graph with split rows, the counts and flips equal
the oracle's on the same float32 state, with zeros of both signs in it."""
import numpy as np
import pytest
import torch

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def loaded():
    import paper_2311_00869_gb300 as P

    n, u, v, s = synth.random_connected(1201, 2500, 0.3, seed=41)
    hub = np.arange(1, 1100, dtype=np.int32)  # vertex 0 with over 1000 neighbours
    lo = np.concatenate([np.minimum(u, v), np.zeros_like(hub)]).astype(np.int64)
    hi = np.concatenate([np.maximum(u, v), hub]).astype(np.int64)
    _, first = np.unique(lo * n + hi, return_index=True)
    sign = np.where(np.arange(first.size) % 3 == 0, -1, 1).astype(np.int8)
    g = O.clean_graph(n, lo[first].astype(np.int32), hi[first].astype(np.int32), sign)
    sb = P.SignedBal(0)
    assert sb.load_graph(n, lo[first].astype(np.int32), hi[first].astype(np.int32), sign)[:2] == (g.n, g.m)
    yield sb, g
    sb.close()


def _gamma(n, R):
    gam = synth.gamma0(n, R, seed=R)
    gam[::7, :] = 0.0
    gam[3::7, R // 2] = -0.0
    return torch.from_numpy(gam).cuda()


@pytest.mark.parametrize("R", [1, 4, 31, 32, 36, 63, 64, 100, 129, 260])
def test_counts_and_flips_match_oracle(loaded, R):
    sb, g = loaded
    gam = _gamma(g.n, R)
    _, F_fwd = sb.graphL_fwd(gam)
    F, flip = sb.graphL_round(gam, want_flip=True)
    oF, oflip = O.graphl_round_f32(g, gam.cpu().numpy(), want_flip=True)
    assert np.array_equal(F.cpu().numpy(), oF) and np.array_equal(F_fwd.cpu().numpy(), oF)
    words = flip.cpu().numpy().view(np.uint64)
    bits = (words[:, :, None] >> np.arange(64, dtype=np.uint64)) & np.uint64(1)
    bits = bits.reshape(R, -1)
    assert np.array_equal(bits[:, : g.m].astype(np.uint8), oflip) and not bits[:, g.m:].any()


@pytest.mark.parametrize("R,lanes,steps", [(5, 0, 2), (36, 8, 3), (36, 16, 2), (100, 32, 3), (129, 0, 2), (64, 0, 1)])
def test_traced_losses_are_those_of_the_states(loaded, R, lanes, steps):
    """The trace holds the discrete loss of every step's input, whichever buffer
    the step reads; an in-place descent and one from an unaligned start give the
    same bits; no steps give the start point back."""
    sb, g = loaded
    sb.set_tuning(gl_lanes=lanes)
    gam = _gamma(g.n, R)
    out, exps, trace, F = sb.graphL_descent(gam, 0.05, steps, renorm_log2=4, trace=True)
    state = gam
    for s in range(steps):
        oF, _ = O.graphl_round_f32(g, state.cpu().numpy())
        assert np.array_equal(trace[s].cpu().numpy(), oF), s
        state = sb.graphL_descent(gam, 0.05, s + 1, renorm_log2=4)[0]
    assert torch.equal(state, out)
    oF, _ = O.graphl_round_f32(g, out.cpu().numpy())
    assert np.array_equal(F.cpu().numpy(), oF)
    again = gam.clone()
    assert torch.equal(sb.graphL_descent(again, 0.05, steps, renorm_log2=4, out=again)[0], out)
    odd = torch.empty(g.n * R + 1, device="cuda")[1:].view(g.n, R)
    odd.copy_(gam)
    assert torch.equal(sb.graphL_descent(odd, 0.05, steps, renorm_log2=4)[0], out)
    same, exps, _, F = sb.graphL_descent(gam, 0.05, 0)
    oF, _ = O.graphl_round_f32(g, gam.cpu().numpy())
    assert torch.equal(same, gam) and not exps.any() and np.array_equal(F.cpu().numpy(), oF)
    sb.set_tuning(gl_lanes=0)
