"""Data and weight gradients of the float path on the tensor cores (two TF32 pieces to a value), every layer from the oracle's own
stored tensors: batches that fill less than a tile, k that ends inside a block of 32, and the sizes at which the library
takes them by itself."""
import numpy as np
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


DATA, WEIGHTS = "gact", "weights"


def contractions(arch, n):
    """The gradients' contractions of a float learner over n states, as (kind, layer, outputs, k)."""
    if arch == "nips":
        return [(WEIGHTS, 2, 2592 * 256, n), (DATA, 2, n * 2592, 256), (WEIGHTS, 1, 256 * 32, 81 * n), (DATA, 1, n * 100 * 64, 128),
                (WEIGHTS, 0, 256 * 16, 400 * n)]
    return [(WEIGHTS, 3, 3136 * 512, n), (DATA, 3, n * 3136, 512), (WEIGHTS, 2, 576 * 64, 49 * n), (DATA, 2, n * 81 * 64, 576),
            (WEIGHTS, 1, 512 * 64, 81 * n), (DATA, 1, n * 100 * 128, 256), (WEIGHTS, 0, 256 * 32, 400 * n)]


def on_tensor_cores(arch, kind, l, outputs, k):
    """The rule of the dispatch for contractions nobody chose a path for."""
    if kind == WEIGHTS:
        return k >= (512 if l == (2 if arch == "nips" else 3) else 2048) and outputs * k >= 64_000_000
    return outputs * k >= max(80_000_000, 11_000_000 * -(-k // 32))


def gradients(arch, prec, n_e, t_max, options, n_actions=6):
    """Gradients of one update, layer by layer, all from the same rollout whatever the options of the update."""
    g = pb.Paac(arch, n_e, t_max, n_actions, seed=9, precision=pb.BF16 if prec == "bf16" else pb.FP32, lr=0.0028, term_denom=50)
    g.rollout()
    for option, value in options.items():
        g.set_option(option, value)
    assert g.update()["status"] == 0 and g.error_word() == 0
    L = 2 if arch == "nips" else 3
    gact = [g.debug_read(pb.DBG_GACT0 + l).copy() for l in range(L + 1)]
    grad, at = g.debug_read(pb.DBG_GRAD), 0
    weights = []
    for J, co in ((256, 16), (256, 32), (2592, 256)) if arch == "nips" else ((256, 32), (512, 64), (576, 64), (3136, 512)):
        weights.append(grad[at:at + (J + 1) * co].copy())
        at += (J + 1) * co
    g.close()
    return {"gact": gact, "weights": weights}


AUTO, CORES_ONLY, TENSOR = {}, {pb.OPT_CUDA_CORES_ONLY: 1}, {pb.OPT_FP32_TENSOR_CORES: 1}


@pytest.mark.parametrize("arch,prec,n", [("nips", "bf16", n) for n in (39, 40, 96, 97, 98, 511, 512)]
                         + [("nips", "fp32", n) for n in (39, 40, 96, 97, 98, 132, 133, 511, 512)]
                         + [("nature", "fp32", n) for n in (19, 20, 25, 26, 27, 41, 42, 66, 67, 109, 110, 511, 512)])
def test_which_contractions_go_to_the_tensor_cores(arch, prec, n):
    """Just below and just above each line of the rule: what the library chooses by itself has the bits of the one contraction
    or of the other, and with CUDA_CORES_ONLY none has those of the tensor cores."""
    auto, cores, tensor = (gradients(arch, prec, n, 1, o) for o in (AUTO, CORES_ONLY, TENSOR))
    compared = 0
    for kind, l, outputs, k in contractions(arch, n):
        at = l - 1 if kind == DATA else l
        same_operand = np.array_equal(cores["gact"][l], tensor["gact"][l])
        # (a data gradient in bf16 storage is rounded to eight bits, where the two contractions nearly always meet)
        if same_operand and not (prec == "bf16" and kind == DATA):
            assert not np.array_equal(cores[kind][at], tensor[kind][at]), (kind, l)
        want = tensor if on_tensor_cores(arch, kind, l, outputs, k) else cores
        if np.array_equal(auto["gact"][l], want["gact"][l]):
            assert np.array_equal(auto[kind][at], want[kind][at]), (kind, l)
            compared += 1
    assert compared >= 2


@pytest.mark.parametrize("arch,hidden,width", [("nips", 256, 2592), ("nature", 512, 3136)])
def test_cuda_cores_only_keeps_float_chains(arch, hidden, width):
    """With CUDA_CORES_ONLY a data gradient of a float learner is one chain of fused multiply-adds over the hidden units, to the bit,
    at a size whose contraction goes to the tensor cores otherwise."""
    n = 160
    g = pb.Paac(arch, n, 1, 6, seed=9, precision=pb.FP32, lr=0.0028, term_denom=50)
    l = 2 if arch == "nips" else 3
    at = {"nips": 257 * 16 + 257 * 32, "nature": 257 * 32 + 513 * 64 + 577 * 64}[arch]
    w = g.params()[at:at + hidden * width].reshape(hidden, width).copy()
    g.rollout()
    g.set_option(pb.OPT_CUDA_CORES_ONLY, 1)
    assert g.update()["status"] == 0
    rows = slice(0, n, 23)
    got = g.debug_read(pb.DBG_GACT0 + l - 1).reshape(n, width)[rows]
    act = g.debug_read(pb.DBG_ACT0 + l - 1).reshape(n, width)[rows]
    out = g.debug_read(pb.DBG_GACT0 + l).reshape(n, hidden)[rows].astype(np.float64)
    g.close()
    chain = np.zeros(got.shape, np.float32)
    for k in range(hidden):       # the product is exact in 64 bits, and so nearly always is the sum
        chain = (chain + out[:, k, None] * w[k].astype(np.float64)).astype(np.float32)
    assert np.array_equal(got, np.where(act > 0, chain, np.float32(0)))


def poisoned(arch, n_e, t_max, options, poison):
    """The gradients of an update whose operands `poison` has changed: it gets the learner, the activations and the parameters."""
    g = pb.Paac(arch, n_e, t_max, 6, seed=9, precision=pb.FP32, lr=0.0028, term_denom=50)
    g.rollout()
    for option, value in options.items():
        g.set_option(option, value)
    L = 2 if arch == "nips" else 3
    act, theta = [g.debug_read(pb.DBG_ACT0 + l).copy() for l in range(L + 1)], g.params().copy()
    poison(act, theta)
    for l in range(L):
        g.debug_write_act(l, act[l])
    g.set_params(theta)
    g.update()
    out = {"gact": [g.debug_read(pb.DBG_GACT0 + l).copy() for l in range(L + 1)], "grad": g.debug_read(pb.DBG_GRAD).copy(), "act": act, "theta": theta}
    assert g.error_word() == 0
    g.close()
    return out


def assert_alike(got, want):
    """The same values are infinite, with the same sign, or not numbers; the others agree to float rounding."""
    finite = np.isfinite(want)
    assert np.array_equal(finite, np.isfinite(got))
    assert np.array_equal(got[~finite], want[~finite], equal_nan=True)
    assert np.linalg.norm(got[finite].astype(np.float64) - want[finite]) <= 1e-6 * np.linalg.norm(want[finite].astype(np.float64))


BIG = np.float32(3.4e38)          # rounds to infinity in fewer bits


@pytest.mark.parametrize("arch,n_e,t_max", [("nips", 64, 8), ("nature", 86, 6)])
def test_infinities_and_the_largest_values(arch, n_e, t_max):
    """Infinite, absent and very large activations and weights give on the tensor cores what they give in a chain of multiply-adds."""
    n, hidden, width = n_e * t_max, *((256, 2592) if arch == "nips" else (512, 3136))
    L = 2 if arch == "nips" else 3
    at = 257 * 16 + 257 * 32 if arch == "nips" else 257 * 32 + 513 * 64 + 577 * 64

    def activations(act, theta):
        for l, a in enumerate(act[:L]):
            a[[5, a.size // 2, a.size - 9]] = np.inf, BIG, np.nan

    def weights(act, theta):
        theta[at + 77], theta[at + 9 * width + 1000], theta[at + 200 * width + width - 1] = np.inf, BIG, -np.inf

    with np.errstate(invalid="ignore", over="ignore"):
        for poison in (activations, weights):
            got, want = poisoned(arch, n_e, t_max, AUTO, poison), poisoned(arch, n_e, t_max, CORES_ONLY, poison)
            assert_alike(got["gact"][L - 1], want["gact"][L - 1])
            # the fully connected layer once more from its own operands, in 64 bits
            g = got["gact"][L].reshape(n, hidden).astype(np.float64)
            x, w = got["act"][L - 1].reshape(n, width), got["theta"][at:at + hidden * width].reshape(hidden, width)
            assert_alike(got["gact"][L - 1].reshape(n, width), np.where(x > 0, g @ w.astype(np.float64), 0).astype(np.float32))
            weight_grad = got["grad"][at:at + hidden * width].reshape(hidden, width)
            assert_alike(weight_grad, (g.T @ x.astype(np.float64)).astype(np.float32))
            assert np.isfinite(weight_grad).all() == (poison is weights)
            if poison is activations:
                assert_alike(got["grad"], want["grad"])
                assert np.isposinf(got["grad"]).any() and np.isneginf(got["grad"]).any()
            else:
                for l in range(L - 1):
                    assert_alike(got["gact"][l], want["gact"][l])


def test_shape_sweep_cuda_cores_and_tensor_cores_agree():
    """Thirty ragged shapes, both networks, both algorithms and environments: the update's gradients from one rollout by chains of multiply-adds
    throughout and with every contraction on the tensor cores.  Each contraction is within 1e-6 of its own operands' sums in the 2-norm, and
    at most four follow one another.  Nothing has the same bits, so there were two implementations."""
    import random
    rnd = random.Random(11)
    combos = [(arch, n, t, a) for arch in ("nips", "nature") for n in (1, 2, 3, 5, 16, 37, 64, 100, 129, 255)
              for t in (1, 2, 5, 7) for a in (2, 3, 5, 18, 19, 32)]
    rnd.shuffle(combos)
    for i, (arch, n_e, T, A) in enumerate(combos[:30]):
        outs = []
        for option in (pb.OPT_CUDA_CORES_ONLY, pb.OPT_FP32_TENSOR_CORES):
            g = pb.Paac(arch, n_e, T, A, seed=5, precision=pb.FP32, lr=0.01, term_denom=50,
                        algorithm=pb.ALGO_NSTEP_Q if i % 3 == 0 else pb.ALGO_A2C, environment=pb.ENV_PATTERN if i % 4 == 0 else pb.ENV_HASHED)
            g.rollout()
            g.set_option(option, 1)
            assert g.update()["status"] == 0 and g.error_word() == 0, (arch, n_e, T, A)
            outs.append([g.debug_read(pb.DBG_GACT0 + l).copy() for l in range(2 if arch == "nips" else 3)] + [g.debug_read(pb.DBG_GRAD).copy()])
            g.close()
        for x, y in zip(*outs):
            d = np.linalg.norm(x.astype(np.float64) - y) / np.linalg.norm(x.astype(np.float64))
            assert 0 < d <= 8e-6, (arch, n_e, T, A, d)
