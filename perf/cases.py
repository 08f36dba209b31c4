"""The work a user of this library has it do, as cases that can be timed and whose results can be compared.

A case is a dict of plain values.  Its "kind" says which entry points it goes through:

  train       one iteration of Algorithm 1 on the synthetic environments: rollout (network forward on every state,
              sampling, environment step, bootstrap) and update (returns, backward pass, clipping, RMSProp)
  host        the same iteration with the environments on the host, as in the paper's set-up: frames come in from
              pinned memory and actions go out, step by step
  preprocess  the paper's frame pre-processing of raw emulator frames on the device
  stack       the four-frame stack by itself on the device
  optimizer   clipping and RMSProp on arrays of the caller's

Sizes are those of paper_1705_04862_b200/configs.py and of the tests, and ragged ones between them.
"""
import functools
import math

import numpy as np
import torch

import paper_1705_04862_b200.binding as pb
from paper_1705_04862_b200.configs import COMMON, CONFIGS

FRAME = 84 * 84 * 4          # bytes of one state
RAW = 210 * 160 * 3          # bytes of one raw emulator frame
#: multiply-adds of the forward pass per state up to the heads, hidden units, parameters up to the heads, and the
#: first layer's multiply-adds (which the backward pass spends once, not twice)
NETS = {"nips": (20 * 20 * 16 * 256 + 9 * 9 * 32 * 256 + 2592 * 256, 256, 16 * 257 + 32 * 257 + 256 * 2593, 20 * 20 * 16 * 256),
        "nature": (20 * 20 * 32 * 256 + 9 * 9 * 64 * 512 + 7 * 7 * 64 * 576 + 3136 * 512, 512,
                   32 * 257 + 64 * 513 + 64 * 577 + 512 * 3137, 20 * 20 * 32 * 256)}


def _config(i, **more):
    """Configuration i of the repository as a training case, on a stream that the program made."""
    c = CONFIGS[i]
    return dict({k: c[k] for k in ("arch", "precision", "n_e", "t_max", "n_actions", "lr", "term_denom")}, kind="train",
                algorithm="a2c", environment="hashed", own_stream=True, stats=False, **more)


def listed():
    return [
        # the repository's five configurations: a few environments while a set-up is tried out, with the losses looked
        # at after every update, ...
        dict(_config(0), name="train_nips_fp32_4", stats=True),
        # ... the paper's own size, 32 environments, with the small network (here the way the binding is used at its
        # simplest, on torch's default stream) and with the large one, ...
        dict(_config(1), name="train_nips_fp32_32", own_stream=False),
        dict(_config(2), name="train_nature_bf16_32"),
        # ... the upper end of the paper's n_e study, and a device filled with environments
        dict(_config(3), name="train_nature_bf16_256"),
        dict(_config(4), name="train_nature_bf16_1024"),
        # a ragged batch with the value-based learner on the environment that can be learned, losses looked at
        dict(_config(2), name="train_q_nature_bf16_185", n_e=185, t_max=7, n_actions=5, term_denom=50, algorithm="q",
             environment="pattern", own_stream=False, stats=True),
        # the large network in float storage (reference runs that want float accuracy)
        dict(_config(1), name="train_nature_fp32_128", arch="nature", n_e=128),
        # emulators on the host: the paper's 32 workers with the newest frame of each sent, and many of them
        dict(_config(2), name="host_nature_bf16_32", kind="host", feed="newest", stats=True),
        dict(_config(4), name="host_nature_bf16_1024", kind="host", feed="newest", stats=True),
        # whole states sent (an emulator wrapper that keeps the stack itself), small network
        dict(_config(1), name="host_nips_fp32_32_whole", kind="host", feed="whole", stats=True),
        # raw frames of as many emulators as the largest configuration has environments
        dict(name="preprocess_1024", kind="preprocess", n=1024, reset=False),
        # the optimiser step by itself at the large network's parameter count, with the bf16 copy
        dict(name="optimizer_nature", kind="optimizer", n=_params("nature", 18), copy16=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train"] * 6 + ["host"] * 3 + ["preprocess", "stack", "optimizer"])
    if kind == "preprocess":
        return dict(kind=kind, n=_log(rng, 1, 1024), reset=rng.random() < 0.2)
    if kind == "stack":
        return dict(kind=kind, n=_log(rng, 1, 1024), restarts=rng.random() < 0.5)
    if kind == "optimizer":
        return dict(kind=kind, n=_log(rng, 1000, 4_000_000), copy16=rng.random() < 0.5)
    arch, precision, most = rng.choice([("nature", "bf16", 1024), ("nature", "bf16", 1024), ("nature", "bf16", 1024), ("nips", "fp32", 192),
                                        ("nips", "fp32", 192), ("nature", "fp32", 96), ("nips", "bf16", 192)])
    t_max = rng.choice([1, 3, 5, 5, 5, 5, 7, 10])
    n_e = max(1, _log(rng, 1, most) * 5 // max(5, t_max))
    case = dict(kind=kind, arch=arch, precision=precision, n_e=n_e, t_max=t_max, n_actions=rng.choice([2, 4, 5, 6, 9, 18]),
                lr=rng.choice([0.0028, 0.0224]), term_denom=rng.choice([20, 100, 200]), algorithm=rng.choice(["a2c", "a2c", "a2c", "q"]),
                environment="hashed", own_stream=rng.random() < 0.7, stats=rng.random() < 0.4)
    if kind == "host":
        case["feed"] = rng.choice(["newest", "newest", "whole"])
        if case["feed"] == "whole":          # four times the bytes over the host link
            case["n_e"] = max(1, n_e // 4)
    else:
        case["environment"] = rng.choice(["hashed", "hashed", "hashed", "pattern"])
    return case


def _params(arch, n_actions):
    _, hidden, below, _ = NETS[arch]
    return below + (n_actions + 1) * (hidden + 1)


def _view(g, address, count, dtype, shape):
    """`count` elements of the learner's workspace (a torch tensor the binding allocates) at a device address."""
    at = address - g._ws.data_ptr()
    return g._ws[at:at + count * torch.empty(0, dtype=dtype).element_size()].view(dtype).view(shape)


@functools.lru_cache(maxsize=None)
def _stream():
    return torch.cuda.Stream()


def _learner(case, seed):
    hp = {k: COMMON[k] for k in ("gamma", "rms_decay", "rms_eps", "clip_norm", "entropy_beta", "value_coef")}
    stream = _stream() if case["own_stream"] else torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        return pb.Paac(case["arch"], case["n_e"], case["t_max"], case["n_actions"], seed + 1,
                       precision=pb.BF16 if case["precision"] == "bf16" else pb.FP32, lr=case["lr"], term_denom=case["term_denom"],
                       algorithm=pb.ALGO_NSTEP_Q if case["algorithm"] == "q" else pb.ALGO_A2C,
                       environment=pb.ENV_PATTERN if case["environment"] == "pattern" else pb.ENV_HASHED, **hp)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def bytes_(*shape):
        return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=gen)

    s = {"case": case}
    if case["kind"] == "preprocess":
        n = case["n"]
        s.update(raw=[bytes_(n, 210, 160, 3) for _ in range(2)], before=None if case["reset"] else bytes_(n, 84, 84, 4),
                 out=torch.empty(n, 84, 84, 4, dtype=torch.uint8, device="cuda"))
    elif case["kind"] == "stack":
        n = case["n"]
        s.update(before=bytes_(n, 84, 84, 4), newest=bytes_(n, 84, 84), out=torch.empty(n, 84, 84, 4, dtype=torch.uint8, device="cuda"),
                 restart=(bytes_(n) < 3).to(torch.uint8) if case["restarts"] else None)
    elif case["kind"] == "optimizer":
        n = case["n"]
        # gradients of a training run: many small values, a few large ones, norms on both sides of the threshold
        s.update(theta=0.05 * torch.randn(n, device="cuda", generator=gen), rms=torch.zeros(n, device="cuda"),
                 grad=torch.randn(n, device="cuda", generator=gen) ** 3 * (60.0 * (0.5 + (seed % 7) / 7.0) / math.sqrt(15.0 * n)),
                 copy=torch.zeros(n, dtype=torch.bfloat16, device="cuda") if case["copy16"] else None,
                 norm=torch.zeros(2, device="cuda"))
    else:
        g = s["learner"] = _learner(case, seed)
        T, n_e, A = case["t_max"], case["n_e"], case["n_actions"]
        # the master parameters lead the learner's workspace; the gradient and the RMSProp state follow, each from
        # the next multiple of 256 bytes
        step = (4 * g.P + 255) // 256 * 256
        s["learned"] = {name: _view(g, g.hp.workspace + k * step, g.P, torch.float32, (g.P,))
                        for k, name in enumerate(("theta", "grad", "rms"))}
        if case["kind"] == "host":
            # what the emulators delivered: states or newest frames, clipped rewards (mostly 0) and ends of episodes
            whole = case["feed"] == "whole"
            u = torch.rand(T, n_e, device="cuda", generator=gen)
            s["rewards"] = ((u < 1 / 16).to(torch.int8) - (u > 15 / 16).to(torch.int8)).cpu().pin_memory()
            s["ends"] = (torch.rand(T, n_e, device="cuda", generator=gen) < 1 / case["term_denom"]).to(torch.uint8).cpu().pin_memory()
            s["first"] = bytes_(n_e, 84, 84, 4).cpu().pin_memory()
            s["frames"] = bytes_(*((T, n_e, 84, 84, 4) if whole else (T, n_e, 84, 84))).cpu().pin_memory()
            s["actions"] = torch.zeros(T, n_e, dtype=torch.int32).pin_memory()
            s["values"] = torch.zeros(T + 1, n_e, dtype=torch.float32).pin_memory()
            s["begun"] = False
    torch.cuda.synchronize()
    return s


def _losses(stats):
    """The losses and the gradient norm an update reports, where the program asked for them."""
    return None if stats is None else np.array([stats[k] for k in ("policy_loss", "value_loss", "entropy", "grad_norm", "clip_scale")], np.float32)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "preprocess":
        status = pb.preprocess(s["raw"][0], s["raw"][1], s["before"], s["out"], case["n"])
        return {"status": status, "state": s["out"]}
    if kind == "stack":
        status = pb.stack_push(s["before"], s["newest"], s["restart"], s["out"], case["n"])
        return {"status": status, "state": s["out"]}
    if kind == "optimizer":
        status = pb.clip_rmsprop_noalloc(s["theta"], s["rms"], s["grad"], case["n"], 0.0224, COMMON["rms_decay"], COMMON["rms_eps"],
                                         COMMON["clip_norm"], theta_bf16=s["copy"], norm_and_scale=s["norm"])
        return {"status": status, "theta": s["theta"], "rms": s["rms"], "theta16": s["copy"], "norm": s["norm"]}
    g, T, n_e, A = s["learner"], case["t_max"], case["n_e"], case["n_actions"]
    if kind == "train":
        v = g.rollout()
        stats = g.update(sync=case["stats"])
        return {"actions": _view(g, v.actions, T * n_e, torch.int32, (T, n_e)), "rewards": _view(g, v.rewards, T * n_e, torch.int8, (T, n_e)),
                "terminals": _view(g, v.terminals, T * n_e, torch.uint8, (T, n_e)),
                "values": _view(g, v.values, (T + 1) * n_e, torch.float32, (T + 1, n_e)),
                "logits": _view(g, v.logits, T * n_e * A, torch.float32, (T, n_e, A)),
                "uniforms": _view(g, v.uniforms, T * n_e, torch.float32, (T, n_e)),
                "frames": _view(g, v.frames, T * n_e * FRAME, torch.uint8, (T, n_e, 84, 84, 4)),
                "next_frames": _view(g, v.next_frames, n_e * FRAME, torch.uint8, (n_e, 84, 84, 4)),
                "learned": s["learned"], "losses": _losses(stats)}
    # host: step 0 of an iteration is the state the iteration before ended in, and is only sent the first time; an
    # environment whose episode ended starts its stack of frames afresh
    for t in range(T + 1):
        actions = s["actions"][t] if t < T else None
        if t == 0:
            g.act_host(0, None if s["begun"] else s["first"], actions, s["values"][0])
        elif case["feed"] == "whole":
            g.act_host(t, s["frames"][t - 1], actions, s["values"][t])
        else:
            g.act_host_newest(t, s["frames"][t - 1], s["ends"][t - 1], actions, s["values"][t])
        if t < T:
            g.observe_host(t, s["rewards"][t], s["ends"][t])
    s["begun"] = True
    stats = g.update(sync=case["stats"])
    return {"actions": s["actions"], "values": s["values"], "learned": s["learned"], "losses": _losses(stats)}


def work(case):
    """Bytes: frames and results written once, what comes in read once, parameters and optimiser state read and written
    once.  Operations: two per multiply-add of the forward passes, of the data gradients and of the weight gradients."""
    kind = case["kind"]
    if kind == "preprocess":
        return {"bytes": case["n"] * (2 * RAW + FRAME * (1 if case["reset"] else 2)), "flops": case["n"] * 84 * 84 * 24}
    if kind == "stack":
        return {"bytes": case["n"] * (2 * FRAME + FRAME // 4), "flops": 0}
    if kind == "optimizer":
        return {"bytes": case["n"] * (20 + 2 * case["copy16"]), "flops": case["n"] * 12}
    T, n_e, A = case["t_max"], case["n_e"], case["n_actions"]
    macs, hidden, _, first = NETS[case["arch"]]
    heads = (A + 1) * hidden
    forward, backward = 2.0 * (macs + heads), 2.0 * (2 * (macs + heads) - first)
    sent = FRAME // 4 if case.get("feed") == "newest" else FRAME
    per_step = sent + 4 * A + 16
    return {"bytes": T * n_e * per_step + n_e * FRAME + 16 * _params(case["arch"], A),
            "flops": (T + 1) * n_e * forward + T * n_e * backward}


def tolerance(case):
    if case["kind"] in ("preprocess", "stack"):
        return "exact"
    if case["kind"] == "optimizer":
        # float sums of up to millions of squares; the bf16 copy may round the other way
        return {"rel": 2e-5, "max": 1e-2}
    # float: sums in another order, and now and then a unit whose pre-activation is within rounding of zero is on in
    # one implementation and off in another, which moves whole terms of a few gradient elements.  bf16: every stored
    # activation is rounded to eight bits.  A uniform within rounding of a CDF boundary picks the neighbouring action.
    return {"rel": 2e-2 if case["precision"] == "bf16" else 1e-3, "max": 0.5, "differ": 0.005}
