"""Data and weight gradients of the float path on the tensor cores (two TF32 pieces to a value), every layer from the oracle's own
stored tensors: batches that fill less than a tile, k that ends inside a block of 32, and the sizes at which the library
takes them by itself."""
import pytest

import paper_1705_04862_b200.binding as pb
from parity_util import TOL, check_rollout, check_update, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arch,prec,n_e,t_max,n_actions,forced", [
    ("nips", "fp32", 1, 1, 2, True), ("nips", "fp32", 3, 2, 18, True), ("nips", "bf16", 5, 1, 6, True),
    ("nature", "fp32", 1, 1, 4, True), ("nature", "fp32", 5, 3, 32, True),
    ("nips", "fp32", 8, 5, 6, False), ("nips", "fp32", 33, 5, 6, False), ("nips", "bf16", 37, 4, 6, False), ("nips", "fp32", 65, 4, 5, False),
    ("nature", "fp32", 16, 5, 6, False), ("nature", "fp32", 43, 6, 18, False)])
def test_gradients_from_the_same_tensors(orc, arch, prec, n_e, t_max, n_actions, forced):
    cfg = dict(arch=arch, precision=prec, n_e=n_e, t_max=t_max, n_actions=n_actions, lr=0.0028, term_denom=50)
    o, g = make_pair(orc, cfg)
    if forced:
        g.set_option(pb.OPT_FP32_TENSOR_CORES, 1)
    for _ in range(2):
        check_rollout(orc, o, g, TOL[prec])
        check_update(orc, o, g, TOL[prec], inject=True)
    assert g.error_word() == 0
    g.close()
