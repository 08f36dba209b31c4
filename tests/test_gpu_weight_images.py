"""The regrouped weights the optimiser's kernel writes beside the parameters against those made from the parameters by themselves."""
import numpy as np
import pytest

import paper_1705_04862_b200.binding as pb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("A", [2, 5, 18, 19, 31])
def test_images_of_an_update_are_those_of_the_parameters(A):
    """Setting the parameters to what they are makes every image anew: the next iteration's logits (first layer's image) and gradients
    (the other three) are the same bits, with each remainder of the parameter count modulo four (which the number of actions sets)."""
    a, b = (pb.Paac("nature", 6, 2, A, seed=9, precision=pb.BF16, lr=0.01, term_denom=3) for _ in range(2))
    for g in (a, b):
        g.rollout()
        g.update()
    assert np.array_equal(a.params(), b.params())
    b.set_params(b.params())
    for g in (a, b):
        g.rollout()
        g.update()
    for which in (pb.DBG_LOGITS, pb.DBG_GRAD, pb.DBG_RMS, pb.DBG_GACT0, pb.DBG_GACT0 + 1, pb.DBG_GACT0 + 2):
        assert np.array_equal(a.debug_read(which).view(np.uint32), b.debug_read(which).view(np.uint32)), which
    assert np.array_equal(a.params(), b.params())
    assert a.error_word() == 0 and b.error_word() == 0
    a.close(), b.close()
