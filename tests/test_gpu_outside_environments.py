"""Steps of the external-environment mode fed from pinned memory, whole states and newest planes in turn, against the states they
should build and against the layers launched one by one."""
import numpy as np
import pytest

import paper_1705_04862_b200.binding as pb

pytestmark = pytest.mark.gpu

T, A = 4, 6


def _compare(arch, prec, n_e, layered_too, iterations=3):
    import torch
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()

    def learner(stream, n):
        with torch.cuda.stream(stream):
            return pb.Paac(arch, n, T, A, seed=6, precision=prec, lr=0.01, term_denom=5)

    # a learner whose neighbour is at work goes layer by layer; from 75 environments on both do
    g, layered, neighbour = learner(mine, n_e), learner(mine, n_e), learner(other, 1)
    if not layered_too:
        layered.set_option(pb.OPT_CUDA_GRAPHS, 0)
    gen = torch.Generator().manual_seed(n_e)
    state = torch.randint(0, 256, (n_e, 84, 84, 4), dtype=torch.uint8, generator=gen).pin_memory()
    planes = torch.empty(n_e, 84, 84, dtype=torch.uint8).pin_memory()
    acts, vals = np.zeros((2, n_e), np.int32), np.zeros((2, n_e), np.float32)
    for it in range(iterations):
        sent = []
        for t in range(T + 1):
            # whole states at even steps of even iterations and at odd ones of odd iterations, planes in between
            whole = t == 0 or (t + it) % 2 == 0
            ends = (torch.rand(n_e, generator=gen) < 0.3).to(torch.uint8)
            if t > 0:
                planes.copy_(torch.randint(0, 256, planes.shape, dtype=torch.uint8, generator=gen))
                pushed = torch.cat([state[..., 1:], planes[..., None]], dim=-1)
                pushed = torch.where(ends[:, None, None, None] != 0, planes[..., None].expand(-1, -1, -1, 4), pushed)
                state.copy_(torch.randint(0, 256, state.shape, dtype=torch.uint8, generator=gen) if whole else pushed)
            sent.append(state.numpy().copy())
            for i, l in enumerate((g, layered)):
                torch.cuda.synchronize()
                if i == 1 and layered_too:
                    with torch.cuda.stream(other):
                        torch.cuda._sleep(40_000_000)
                before = l.launch_count()
                if whole:
                    l.act_host(t, state, acts[i] if t < T else None, vals[i])
                else:
                    l.act_host_newest(t, planes, ends.numpy(), acts[i] if t < T else None, vals[i])
                assert (l.launch_count() - before == 1) == (i == 0 and layered_too)
                if t < T:
                    l.observe_host(t, (np.arange(n_e) % 3 - 1).astype(np.int8), ends.numpy())
            assert np.array_equal(vals[0].view(np.uint32), vals[1].view(np.uint32)), (it, t)
            assert t == T or np.array_equal(acts[0], acts[1]), (it, t)
        for l in (g, layered):
            assert np.array_equal(l.debug_read(pb.DBG_FRAMES), np.stack(sent[:T]).reshape(-1)), it
            assert np.array_equal(l.debug_read(pb.DBG_NEXT_FRAMES), sent[T].reshape(-1)), it
        for which in (pb.DBG_LOGITS, pb.DBG_UNIFORMS):
            assert np.array_equal(g.debug_read(which).view(np.uint32), layered.debug_read(which).view(np.uint32)), it
        assert g.update() == layered.update()
        assert np.array_equal(g.params(), layered.params())
    assert g.error_word() == 0 and layered.error_word() == 0
    for l in (g, layered, neighbour):
        l.close()


@pytest.mark.parametrize("arch,prec,n_e", [("nature", pb.BF16, 319), ("nature", pb.BF16, 321), ("nips", pb.FP32, 321)])
def test_recorded_and_launched_one_by_one(arch, prec, n_e):
    """Either side of where a step's launches follow the frame stack one by one, and the path on which they stay recorded."""
    _compare(arch, prec, n_e, layered_too=False, iterations=5)


@pytest.mark.parametrize("arch,prec,n_e", [("nature", pb.BF16, 1), ("nature", pb.BF16, 33), ("nature", pb.BF16, 34), ("nature", pb.BF16, 74),
                                           ("nips", pb.FP32, 9), ("nips", pb.BF16, 10), ("nips", pb.FP32, 18), ("nips", pb.FP32, 19),
                                           ("nips", pb.BF16, 37), ("nips", pb.FP32, 38), ("nips", pb.BF16, 74)])
def test_steps_in_one_launch_fetch_what_was_sent(arch, prec, n_e):
    """The smallest and the largest number of environments of every group of blocks, each block of which fetches a share of its own."""
    _compare(arch, prec, n_e, layered_too=True)
