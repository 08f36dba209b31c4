"""The larger network's rollout in one launch against the layer-by-layer kernels: the same bits."""
import numpy as np
import pytest

import paper_1705_04862_b200.binding as pb

pytestmark = pytest.mark.gpu

LAYERED = 640          # environments of a learner whose layers are launched one by one, with the same eight slices of K


def _rollouts(n_e, t_max, A, times=2, **hp):
    g = pb.Paac("nature", n_e, t_max, A, seed=11, precision=pb.BF16, term_denom=3, **hp)
    out = []
    for _ in range(times):
        before = g.launch_count()
        g.rollout()
        launches = g.launch_count() - before
        got = {w: g.debug_read(w) for w in (pb.DBG_FRAMES, pb.DBG_NEXT_FRAMES, pb.DBG_ACTIONS, pb.DBG_SAMPLED, pb.DBG_REWARDS, pb.DBG_TERMINALS,
                                            pb.DBG_VALUES, pb.DBG_LOGITS, pb.DBG_UNIFORMS, pb.DBG_COUNTERS)}
        got.update({pb.DBG_ACT0 + l: g.debug_read(pb.DBG_ACT0 + l) for l in range(4)})
        out.append(got)
    assert g.error_word() == 0
    g.close()
    return launches, out


@pytest.mark.parametrize("A,hp", [(18, {}), (31, dict(environment=pb.ENV_PATTERN)), (2, dict(algorithm=pb.ALGO_NSTEP_Q, epsilon=0.2))])
def test_same_bits_as_layer_by_layer(A, hp):
    """One environment, a full set of clusters of four blocks, the first of two, one and two row chunks of the fully connected layer, all
    clusters of two; beyond, the layers are launched one by one."""
    T = 2
    launches, want = _rollouts(LAYERED, T, A, **hp)
    assert launches > 1
    for n in (1, 5, 16, 17, 33, 34, 64, 65, 74, 75):
        launches, got = _rollouts(n, T, A, **hp)
        assert (launches == 1) == (n <= 74), n
        for it in range(2):
            for w, x in got[it].items():
                y = want[it][w]
                slots = T + 1 if w == pb.DBG_VALUES else (1 if w == pb.DBG_NEXT_FRAMES else (3 if w == pb.DBG_COUNTERS else T))
                x, y = x.reshape(slots, n, -1), y.reshape(slots, LAYERED, -1)[:, :n]
                assert np.array_equal(x.view(np.uint8), np.ascontiguousarray(y).view(np.uint8)), (n, it, w, float(np.mean(x != y)))

