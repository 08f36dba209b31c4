"""An update that is timed kernel by kernel keeps everything on one stream; one that is not runs the weight gradients beside the chain of
data gradients.  The same kernels add up the same numbers in the same groups."""
import numpy as np
import pytest

import paper_1705_04862_b200.binding as pb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arch,prec,n_e,t_max,n_actions,options", [
    ("nips", "fp32", 32, 5, 6, {}), ("nips", "bf16", 3, 2, 5, {}), ("nips", "fp32", 9, 3, 4, {pb.OPT_FP32_TENSOR_CORES: 1}),
    ("nature", "fp32", 16, 5, 18, {}), ("nature", "bf16", 37, 5, 6, {}), ("nature", "bf16", 8, 3, 4, {pb.OPT_UPDATE_CHUNKS: 3})])
def test_the_clipped_step_is_the_same_beside_the_chain_and_in_line(arch, prec, n_e, t_max, n_actions, options):
    """Every gradient is longer than clip_norm, so the parameters carry the last bits of its norm."""
    outs = []
    for timed in (True, False):
        g = pb.Paac(arch, n_e, t_max, n_actions, seed=5, precision=pb.BF16 if prec == "bf16" else pb.FP32, lr=0.0224, term_denom=50, clip_norm=1e-3)
        for option, value in options.items():
            g.set_option(option, value)
        g.profile(timed)
        out = []
        for _ in range(6):
            g.rollout()
            st = g.update()
            assert st["status"] == 0 and st["clip_scale"] < 1
            out.append((st["grad_norm"], g.params()))
        g.close()
        outs.append(out)
    for (norm, theta), (norm1, theta1) in zip(*outs):
        assert norm == norm1 and np.array_equal(theta, theta1)
