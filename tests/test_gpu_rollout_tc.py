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



@pytest.mark.parametrize("n_e,ring", [(1, True), (33, True), (64, False), (74, True)])
def test_outside_environments_same_bits_as_layer_by_layer(n_e, ring):
    """Steps of the external-environment mode in one launch (planes read from pinned memory, or copied first) against the states they
    should build and against the layer-by-layer kernels, restarts included; two iterations without sending step 0 again."""
    import torch
    T, A = 3, 6
    gen = torch.Generator().manual_seed(n_e)
    small, large = (pb.Paac("nature", n, T, A, seed=5, precision=pb.BF16, term_denom=3) for n in (n_e, LAYERED))
    first = torch.randint(0, 256, (LAYERED, 84, 84, 4), dtype=torch.uint8, generator=gen)
    state = first.clone()
    acts = [np.zeros(n, np.int32) for n in (n_e, LAYERED)]
    vals = [np.zeros(n, np.float32) for n in (n_e, LAYERED)]
    for it in range(2):
        for t in range(T + 1):
            if t == 0:
                for i, (g, n) in enumerate(((small, n_e), (large, LAYERED))):
                    g.act_host(0, first[:n].contiguous().pin_memory() if it == 0 else None, acts[i], vals[i])
            else:
                planes = torch.randint(0, 256, (LAYERED, 84, 84), dtype=torch.uint8, generator=gen)
                ends = (torch.rand(LAYERED, generator=gen) < 0.3).to(torch.uint8)
                pushed = torch.cat([state[..., 1:], planes[..., None]], dim=-1)
                state = torch.where(ends[:, None, None, None] != 0, planes[..., None].expand(-1, -1, -1, 4), pushed).contiguous()
                for i, (g, n) in enumerate(((small, n_e), (large, LAYERED))):
                    mine = planes[:n].contiguous()
                    g.act_host_newest(t, mine.pin_memory() if ring else mine.numpy(), ends[:n].numpy().copy(), acts[i] if t < T else None, vals[i])
            assert np.array_equal(vals[0].view(np.uint32), vals[1][:n_e].view(np.uint32)), (it, t)
            if t < T:
                assert np.array_equal(acts[0], acts[1][:n_e]), (it, t)
                for g, n in ((small, n_e), (large, LAYERED)):
                    g.observe_host(t, np.zeros(n, np.int8), np.zeros(n, np.uint8))
        assert np.array_equal(small.debug_read(pb.DBG_NEXT_FRAMES), state[:n_e].numpy().reshape(-1))
    assert small.error_word() == 0 and large.error_word() == 0
    small.close(), large.close()


def test_planes_of_more_environments_than_one_launch_takes():
    """The frame stack's restart flags are launch arguments, 2048 environments to a launch: states of either side of that line."""
    import torch
    n = 2051
    gen = torch.Generator().manual_seed(1)
    g = pb.Paac("nips", n, 1, 4, seed=2, precision=pb.FP32)
    first = torch.randint(0, 256, (n, 84, 84, 4), dtype=torch.uint8, generator=gen).pin_memory()
    planes = torch.randint(0, 256, (n, 84, 84), dtype=torch.uint8, generator=gen).pin_memory()
    ends = (torch.rand(n, generator=gen) < 0.5).to(torch.uint8)
    acts, vals = np.zeros(n, np.int32), np.zeros(n, np.float32)
    g.act_host(0, first, acts, vals)
    g.observe_host(0, np.zeros(n, np.int8), ends.numpy())
    g.act_host_newest(1, planes, ends.numpy(), None, vals)
    pushed = torch.cat([first[..., 1:], planes[..., None]], dim=-1)
    want = torch.where(ends[:, None, None, None] != 0, planes[..., None].expand(-1, -1, -1, 4), pushed)
    assert np.array_equal(g.debug_read(pb.DBG_NEXT_FRAMES), want.contiguous().numpy().reshape(-1))
    g.close()


@pytest.mark.parametrize("arch,prec,n_e", [("nature", pb.BF16, 1), ("nature", pb.BF16, 33), ("nature", pb.BF16, 74), ("nips", pb.FP32, 3),
                                           ("nips", pb.BF16, 18), ("nips", pb.FP32, 37), ("nips", pb.FP32, 74)])
def test_waits_between_blocks_give_up(arch, prec, n_e):
    """With one poll to a wait the first ones run out: the launch ends, the error word says so, the update is skipped.  Once the word is
    cleared the learner goes on, with whole rollouts and with steps of environments outside, as one to which nothing happened."""
    a, b = (pb.Paac(arch, n_e, 4, 6, seed=8, precision=prec, lr=0.01, term_denom=5) for _ in range(2))
    for g in (a, b):
        g.rollout()
        assert g.update()["status"] == 0
    theta, rms = a.params(), a.debug_read(pb.DBG_RMS).copy()
    with pytest.raises(pb.PaacError):
        a.set_option(pb.OPT_WAIT_POLLS, 0)
    rng = np.random.RandomState(n_e)
    first, planes = rng.randint(0, 256, (n_e, 84, 84, 4), dtype=np.uint8), rng.randint(0, 256, (4, n_e, 84, 84), dtype=np.uint8)
    acts, vals = np.zeros((2, n_e), np.int32), np.zeros((2, n_e), np.float32)

    def outside(i, g):
        seen = []
        for t in range(5):
            if t == 0:
                g.act_host(0, first, acts[i], vals[i])
            else:
                g.act_host_newest(t, planes[t - 1], None, acts[i] if t < 4 else None, vals[i])
            seen += [acts[i].copy(), vals[i].copy()]
            if t < 4:
                g.observe_host(t, np.ones(n_e, np.int8), np.zeros(n_e, np.uint8))
        return seen

    for limited in (lambda: a.rollout(), lambda: outside(0, a)):
        a.set_option(pb.OPT_WAIT_POLLS, 1)
        limited()
        assert a.error_word() == 1
        st = a.update()
        assert st["status"] == pb.ERR_TIMEOUT and st["clip_scale"] == 0.0
        a.set_option(pb.OPT_WAIT_POLLS, 2000000)
        a.clear_error_word()
        assert np.array_equal(a.params(), theta) and np.array_equal(a.debug_read(pb.DBG_RMS), rms)
        b.rollout()                                            # as many steps as the one that was cut short
        for which in (pb.DBG_NEXT_FRAMES, pb.DBG_COUNTERS):
            a.debug_write(which, b.debug_read(which))
        for again in range(2):
            for g in (a, b):
                g.rollout()
            for which in (pb.DBG_FRAMES, pb.DBG_NEXT_FRAMES, pb.DBG_ACTIONS, pb.DBG_REWARDS, pb.DBG_VALUES, pb.DBG_LOGITS, pb.DBG_UNIFORMS, pb.DBG_COUNTERS):
                assert np.array_equal(a.debug_read(which).view(np.uint8), b.debug_read(which).view(np.uint8)), which
        for x, y in zip(outside(0, a), outside(1, b)):
            assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
        for g in (a, b):
            assert g.update()["status"] == 0
        theta, rms = a.params(), a.debug_read(pb.DBG_RMS).copy()
        assert np.array_equal(theta, b.params())
    a.close(), b.close()
