"""Gradients of the float path against sums in 64 bits, from the tensors the library itself stored: by itself it goes to the
tensor cores only where they are no further off than chains of float multiply-adds."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

import paper_1705_04862_b200.binding as pb
from test_gpu_float_contractions import DATA, WEIGHTS, contractions, on_tensor_cores

pytestmark = pytest.mark.gpu

CONV = {"nips": [(84, 4, 16, 8, 4), (20, 16, 32, 4, 2)], "nature": [(84, 4, 32, 8, 4), (20, 32, 64, 4, 2), (9, 64, 64, 3, 1)]}     # input side and channels, channels, kernel, stride
FC = {"nips": (2592, 256), "nature": (3136, 512)}


def errors(got, want, sizes, where=None):
    """2-norm of the error over that of the result, its largest value over that of the result, and its root mean square with every element's
    over the sum of its terms' sizes."""
    e, some = got - want, sizes > 0
    if where is not None:
        e, want, some = e * where, want * where, some & where
    return (e.norm() / want.norm()).item(), (e.abs().max() / want.abs().max()).item(), (e[some] / sizes[some]).pow(2).mean().sqrt().item()


def gradient_errors(arch, prec, n_e, t_max, option, updates):
    """{contraction: errors} of one update's gradients with `option` set for it."""
    def dev(x, *shape):
        return torch.from_numpy(np.ascontiguousarray(x)).cuda().to(torch.float64).reshape(shape)

    g = pb.Paac(arch, n_e, t_max, 6, seed=9, precision=pb.BF16 if prec == "bf16" else pb.FP32, lr=0.0028, term_denom=50)
    g.set_option(pb.OPT_CUDA_CORES_ONLY, 1)          # the same parameters and activations whatever the option
    for _ in range(updates):
        g.rollout()
        assert g.update()["status"] == 0
    g.rollout()
    theta = torch.from_numpy(g.params())
    theta = (theta.to(torch.bfloat16) if prec == "bf16" else theta).to(torch.float64).cuda()
    g.set_option(option, 1)
    assert g.update()["status"] == 0 and g.error_word() == 0
    n, L, (width, hidden) = n_e * t_max, len(CONV[arch]), FC[arch]
    grad, frames = dev(g.debug_read(pb.DBG_GRAD), -1), g.debug_read(pb.DBG_FRAMES)
    act = [dev(g.debug_read(pb.DBG_ACT0 + l), n, -1) for l in range(L)]
    gact = [dev(g.debug_read(pb.DBG_GACT0 + l), n, -1) for l in range(L + 1)]
    g.close()
    out, at = {}, 0
    for l, (H, C, CO, K, S) in enumerate(CONV[arch]):
        x = (dev(frames, n, H, H, C) if l == 0 else act[l - 1].view(n, H, H, C)).permute(0, 3, 1, 2)
        size = CO * K * K * C
        w, gw = (v[at:at + size].view(CO, K, K, C).permute(0, 3, 1, 2).reshape(CO, -1) for v in (theta, grad))
        at += size + CO
        scale = float(np.float32(1 / 255)) if l == 0 else 1.0
        sums, sizes, below, below_sizes = torch.zeros_like(gw), torch.zeros_like(gw), [], []
        for i in range(0, n, 64):
            windows, go = F.unfold(x[i:i + 64], K, stride=S).transpose(1, 2), gact[l][i:i + 64].view(-1, ((H - K) // S + 1) ** 2, CO)
            sums += torch.einsum("npc,npj->cj", go, windows)
            sizes += torch.einsum("npc,npj->cj", go.abs(), windows.abs())
            if l:
                below.append(F.fold((go @ w).transpose(1, 2), H, K, stride=S))
                below_sizes.append(F.fold((go.abs() @ w.abs()).transpose(1, 2), H, K, stride=S))
        out["weights", l] = errors(gw, sums * scale, sizes * scale)
        if l:
            out["data", l] = errors(gact[l - 1].view(n, H, H, C).permute(0, 3, 1, 2), torch.cat(below), torch.cat(below_sizes), x > 0)
    w, gw = (v[at:at + width * hidden].view(hidden, width) for v in (theta, grad))
    go, x = gact[L], act[L - 1]
    out["weights", L] = errors(gw, go.t() @ x, go.abs().t() @ x)
    out["data", L] = errors(gact[L - 1], go @ w, go.abs() @ w.abs(), x > 0)
    return out


@pytest.mark.parametrize("arch,prec,n_e,t_max,updates", [
    ("nips", "fp32", 1, 1, 0), ("nips", "fp32", 37, 3, 3), ("nips", "fp32", 133, 1, 0), ("nips", "fp32", 512, 1, 3), ("nips", "fp32", 96, 10, 3),
    ("nips", "bf16", 40, 1, 0), ("nips", "bf16", 271, 1, 30), ("nips", "bf16", 113, 7, 3),
    ("nature", "fp32", 1, 1, 0), ("nature", "fp32", 26, 1, 3), ("nature", "fp32", 42, 1, 0), ("nature", "fp32", 110, 1, 0), ("nature", "fp32", 128, 5, 3)])
def test_no_further_from_64_bits_than_the_cuda_cores(arch, prec, n_e, t_max, updates):
    """Every contraction on the tensor cores: 1e-6 in the 2-norm is sixteen roundings' worth, and two pieces of 11 bits leave at most 2^-21 of a
    product out, 2^-23 in the mean square; a pass that is lost leaves 2^-13.  And where the library takes them by itself, they are no further off than the
    multiply-adds' chain.  Bf16 storage rounds data gradients to eight bits after either."""
    cores, tensor = (gradient_errors(arch, prec, n_e, t_max, option, updates) for option in (pb.OPT_CUDA_CORES_ONLY, pb.OPT_FP32_TENSOR_CORES))
    rule = {(kind, l): on_tensor_cores(arch, kind, l, outputs, k) for kind, l, outputs, k in contractions(arch, n_e * t_max)}
    for key, (norm, largest, few) in tensor.items():
        if prec == "bf16" and key[0] == "data":
            assert norm <= 2.0 ** -9, (key, norm)
            continue
        assert norm <= 1e-6 and few <= 2.0 ** -23, (key, norm, few)
        if rule[DATA if key[0] == "data" else WEIGHTS, key[1]]:
            assert norm <= cores[key][0], (key, norm, cores[key])
