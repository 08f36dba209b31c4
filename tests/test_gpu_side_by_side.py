"""Learners on streams of their own, side by side.  A rollout in one launch takes nearly every multiprocessor and its blocks wait for
one another, so it is launched only while no learner on another stream has work in flight; otherwise the layers are launched one by
one, with the same numbers."""
import numpy as np
import pytest

import paper_1705_04862_b200.binding as pb

pytestmark = pytest.mark.gpu

READ = (pb.DBG_FRAMES, pb.DBG_NEXT_FRAMES, pb.DBG_ACTIONS, pb.DBG_REWARDS, pb.DBG_VALUES, pb.DBG_LOGITS, pb.DBG_COUNTERS, pb.DBG_RMS)


def _learner(stream, arch, prec, n_e, seed=1, A=5, T=3):
    import torch
    with torch.cuda.stream(stream):
        return pb.Paac(arch, n_e, T, A, seed=seed, precision=prec, lr=0.01, term_denom=5)


def _launches(g, call):
    before = g.launch_count()
    call()
    return g.launch_count() - before


def _same(a, b):
    assert np.array_equal(a.params(), b.params())
    for which in READ:
        assert np.array_equal(a.debug_read(which).view(np.uint8), b.debug_read(which).view(np.uint8)), which


@pytest.mark.parametrize("arch,prec,n_e", [("nature", pb.BF16, 20), ("nature", pb.BF16, 64), ("nips", pb.FP32, 7), ("nips", pb.BF16, 60)])
def test_one_launch_only_while_nobody_else_is_at_work(arch, prec, n_e):
    """Whole rollouts and steps with environments outside: in one launch while the other learner's stream is idle or is the same
    one, layer by layer while it is busy; recorded or not, the numbers are those of a learner that is alone."""
    import torch
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    g, alone = _learner(mine, arch, prec, n_e), _learner(mine, arch, prec, n_e)
    beside = _learner(other, arch, prec, n_e)
    gen = torch.Generator().manual_seed(n_e)
    first = torch.randint(0, 256, (n_e, 84, 84, 4), dtype=torch.uint8, generator=gen).pin_memory()
    planes = torch.randint(0, 256, (3, n_e, 84, 84), dtype=torch.uint8, generator=gen).pin_memory()
    ends = (torch.rand(3, n_e, generator=gen) < 0.3).to(torch.uint8).numpy()
    for it in range(8):
        torch.cuda.synchronize()
        with torch.cuda.stream(mine if it % 4 == 3 else other):
            if it % 2:
                torch.cuda._sleep(200_000_000)                 # some 100 ms
        layered = it % 4 == 1
        assert (_launches(g, g.rollout) > 1) == layered, it
        torch.cuda.synchronize()
        alone.rollout()
        assert g.update() == alone.update()
        _same(g, alone)
    acts, vals = np.zeros((2, n_e), np.int32), np.zeros((2, n_e), np.float32)
    for t in range(4):
        for i, l in enumerate((g, alone)):
            torch.cuda.synchronize()
            if i == 0 and t != 2:
                with torch.cuda.stream(other):
                    torch.cuda._sleep(200_000_000)
            def step():
                if t == 0:
                    l.act_host(0, first, acts[i], vals[i])
                else:
                    l.act_host_newest(t, planes[t - 1], ends[t - 1], acts[i] if t < 3 else None, vals[i])
            assert (_launches(l, step) > 1) == (i == 0 and t != 2)
            if t < 3:
                l.observe_host(t, np.ones(n_e, np.int8), ends[t])
        assert np.array_equal(acts[0], acts[1]) and np.array_equal(vals[0], vals[1])
    assert g.update() == alone.update()
    _same(g, alone)
    assert g.error_word() == 0 and beside.error_word() == 0
    for l in (g, alone, beside):
        l.close()


def test_learners_side_by_side_are_learners_alone():
    """Several learners fed by one thread without waiting, enough for their rollouts to meet on the device."""
    import torch
    shapes = [("nature", pb.BF16, 64), ("nature", pb.BF16, 64), ("nature", pb.BF16, 8), ("nips", pb.FP32, 4), ("nips", pb.FP32, 74)]
    learners = [_learner(torch.cuda.Stream(), *s, seed=3 + i) for i, s in enumerate(shapes)]
    for _ in range(40):
        for g in learners:
            g.rollout()
        for g in learners:
            g.update(sync=False)
    torch.cuda.synchronize()
    for i, (s, g) in enumerate(zip(shapes, learners)):
        assert g.error_word() == 0
        alone = _learner(torch.cuda.current_stream(), *s, seed=3 + i)
        for _ in range(40):
            alone.rollout()
            alone.update(sync=False)
            torch.cuda.synchronize()
        _same(g, alone)
        alone.close()
    for g in learners:
        g.close()


@pytest.mark.parametrize("arch,prec", [("nature", pb.BF16), ("nips", pb.FP32)])
def test_a_rollout_recorded_by_the_caller_goes_layer_by_layer(arch, prec):
    """Replayed by the caller, it could meet any other learner's."""
    import torch
    stream = torch.cuda.Stream()
    a, b = (_learner(stream, arch, prec, 9) for _ in range(2))
    graph = torch.cuda.CUDAGraph()
    launched = []
    with torch.cuda.graph(graph, stream=stream):
        launched.append(_launches(a, a.rollout))
    assert launched[0] > 1
    with torch.cuda.stream(stream):
        graph.replay()
    assert _launches(b, b.rollout) == 1
    assert a.update() == b.update()
    _same(a, b)
    del graph
    a.close(), b.close()


def test_a_learner_on_the_per_thread_stream_counts_as_at_work():
    """Its stream is another one in every thread, so another thread cannot ask about it."""
    import torch
    g = _learner(torch.cuda.Stream(), "nips", pb.FP32, 4)
    assert _launches(g, g.rollout) == 1
    per_thread = _learner(torch.cuda.ExternalStream(2), "nips", pb.FP32, 4)
    assert per_thread.hp.stream == 2
    torch.cuda.synchronize()
    assert _launches(g, g.rollout) > 1
    torch.cuda.synchronize()
    assert _launches(per_thread, per_thread.rollout) == 1
    per_thread.close()
    torch.cuda.synchronize()
    assert _launches(g, g.rollout) == 1
    g.close()
