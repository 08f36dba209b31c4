"""Host-side checks that need no GPU: the C-ABI library loads, exports every symbol the header
declares, sizes workspaces, validates arguments, and refuses to run without a device."""
import ctypes as C
import itertools
import os
import re
import subprocess

import pytest

from paper_1705_04862_b200 import binding as pb
from paper_1705_04862_b200 import build as pbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_builds_and_exports_every_declared_symbol():
    pbuild.build()
    L = pb.lib()
    hdr = open(os.path.join(ROOT, "include", "paac.h")).read()
    hdr = re.sub(r"/\*.*?\*/", "", hdr, flags=re.S)
    declared = set(re.findall(r"\b(paac_[a-z_0-9]+)\s*\(", hdr))
    assert declared == set(pb.EXPORTS), declared ^ set(pb.EXPORTS)
    for name in declared:
        assert getattr(L, name) is not None


def test_struct_layouts_match_header():
    assert C.sizeof(pb.HParams) == 80 and pb.HParams.workspace.offset == 40 and pb.HParams.stream.offset == 56
    assert pb.HParams.algorithm.offset == 64 and pb.HParams.epsilon.offset == 68 and pb.HParams.environment.offset == 72
    assert C.sizeof(pb.UpdateStats) == 32 and pb.UpdateStats.timesteps.offset == 24
    assert C.sizeof(pb.RolloutView) == 64


def test_defaults_are_the_papers_hyperparameters():
    hp = pb.default_hparams()
    got = (hp.gamma, hp.lr, hp.rms_decay, hp.rms_eps, hp.clip_norm, hp.entropy_beta, hp.value_coef)
    want = (0.99, 0.0224, 0.99, 0.1, 40.0, 0.01, 1.0)
    assert all(abs(a - b) < 1e-7 for a, b in zip(got, want))
    assert hp.term_denom == 200 and hp.precision == pb.FP32
    assert hp.algorithm == pb.ALGO_A2C and abs(hp.epsilon - 0.1) < 1e-7


def test_workspace_sizing_and_argument_checks():
    hp = pb.default_hparams(precision=pb.BF16)
    big = pb.workspace_bytes(pb.ARCH_NATURE, 1024, 5, 18, hp)
    small = pb.workspace_bytes(pb.ARCH_NATURE, 32, 5, 18, hp)
    assert 0 < small < big < 4 << 30
    frames = 2 * 5 * 1024 * 84 * 84 * 4
    assert big > frames
    assert pb.workspace_bytes(2, 32, 5, 18, hp) == 0
    assert pb.workspace_bytes(pb.ARCH_NIPS, 0, 5, 4, hp) == 0
    assert pb.workspace_bytes(pb.ARCH_NIPS, 4, 0, 4, hp) == 0
    assert pb.workspace_bytes(pb.ARCH_NIPS, 4, 5, 33, hp) == 0
    assert pb.workspace_bytes(pb.ARCH_NIPS, 4, 5, 4, pb.default_hparams(term_denom=0)) == 0
    assert pb.workspace_bytes(pb.ARCH_NIPS, 4, 5, 4, pb.default_hparams(precision=5)) == 0


def test_null_handles_and_strerror():
    L = pb.lib()
    assert L.paac_rollout(None, None) == pb.ERR_ARG
    assert L.paac_update(None, None) == pb.ERR_ARG
    assert L.paac_destroy(None) == pb.ERR_ARG
    assert L.paac_param_count(None) == 0 and L.paac_debug_bytes(None, 0) == 0
    names = {L.paac_strerror(i) for i in range(9)}
    assert len(names) == 9 and L.paac_strerror(99) == b"unknown status"


def test_init_fails_loudly_without_a_gpu():
    import torch
    if torch.cuda.is_available():
        return
    L = pb.lib()
    h = C.c_void_p()
    hp = pb.default_hparams()
    assert L.paac_init(C.byref(h), pb.ARCH_NIPS, 4, 5, 4, C.byref(hp), 1) == pb.ERR_CUDA
    assert not h.value


def _compiled(tmp_path, source):
    """A library of plain C++ that includes one of the headers the host code shares with nothing on a device."""
    src, so = tmp_path / "host.cpp", tmp_path / "host.so"
    src.write_text(source)
    csrc = os.path.join(ROOT, "paper_1705_04862_b200", "csrc")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", csrc, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


HOST_VIEW = """
#include "host_view.h"
// ranges: start, size, device address of the start, pinned -- four numbers each
extern "C" uintptr_t view(uintptr_t p, size_t bytes, const uint64_t* ranges, int n) {
  return (uintptr_t)paac::host_view((const uint8_t*)p, bytes, [&](const uint8_t* at, paac::HostRange& r) {
    for (int i = 0; i < n; ++i, ranges += 4)
      if ((uintptr_t)at - ranges[0] < ranges[1]) {
        r = paac::HostRange{ranges[3] != 0, (uintptr_t)at - ranges[0] + ranges[2], ranges[2], (size_t)ranges[1]};
        return true;
      }
    return false;
  });
}
"""


@pytest.mark.parametrize("p,size,ranges,readable", [
    (0x1000, 0x1000, [(0x1000, 0x1000, 0x1000, 1)], True),                               # the whole allocation
    (0x1010, 0xFF0, [(0x1000, 0x1000, 0x1000, 1)], True),                                # up to its last byte
    (0x1010, 0xFF1, [(0x1000, 0x1000, 0x1000, 1)], False),                               # one byte further
    (0x1000, 0x3000, [(0x1000, 0x1000, 0x1000, 1)], False),                              # a registered piece of a larger array
    (0x1000, 0x3000, [(0x1000, 0x1000, 0x1000, 1), (0x3000, 0x1000, 0x3000, 1)], False),   # both ends, not the middle
    (0x1000, 0x2000, [(0x1000, 0x1000, 0x1000, 1), (0x2000, 0x1000, 0x2000, 1)], False),   # two allocations side by side
    (0x1000, 16, [], False),                                                            # nothing known
    (0x1000, 16, [(0x1000, 0x1000, 0x1000, 0)], False),                                  # known, not pinned
    (0x1000, 16, [(0x1000, 0x1000, 0x9000, 1)], False),                                  # seen elsewhere by the device
    (0x1000, 2 ** 64 - 1, [(0x1000, 0x1000, 0x1000, 1)], False),                         # a length that wraps around
])
def test_host_buffers_are_read_in_place_only_where_all_of_them_is_pinned(tmp_path, p, size, ranges, readable):
    view = _compiled(tmp_path, HOST_VIEW).view
    view.argtypes, view.restype = [C.c_uint64, C.c_size_t, C.POINTER(C.c_uint64), C.c_int], C.c_uint64
    flat = [x for r in ranges for x in r] or [0]
    assert view(p, size, (C.c_uint64 * len(flat))(*flat), len(ranges)) == (p if readable else 0)


PER_DEVICE = """
#include "per_device.h"
static paac::PerDevice<int> cache;
static int calls = 0;
extern "C" int get(int device, int works) {          // 100 * device + the call it was made in, or -1
  const int* v = cache.get(device, [&](int& out) { out = 100 * device + ++calls; return works != 0; });
  return v ? *v : -1;
}
"""


def test_what_belongs_to_a_device_is_made_once_on_each(tmp_path):
    """The pre-processing kernel's attribute and the built-in array's address: looked up on every device that is used,
    once, and again after a failure."""
    get = _compiled(tmp_path, PER_DEVICE).get
    assert [get(0, 1), get(0, 1), get(1, 1), get(0, 1), get(1, 0)] == [1, 1, 102, 1, 102]
    assert [get(63, 0), get(63, 1), get(63, 0)] == [-1, 6304, 6304]
    assert [get(-1, 1), get(64, 1)] == [-1, -1]


def _word_accesses():
    """(elements, bits of an element) of every load and store that step_words.cuh makes."""
    text = open(os.path.join(ROOT, "paper_1705_04862_b200", "csrc", "step_words.cuh")).read()
    found = re.findall(r'"(ld|st)\.[a-z.]*global\.(?:v(\d)\.)?[a-z](\d+) ', text)
    return {kind: sorted({(int(n or 1), int(bits)) for k, n, bits in found if k == kind}) for kind in ("ld", "st")}


def _torn_reads(store, load):
    """Whether a reader may find the new step beside the old value.  Elements of a vector access are accesses of their own, in any
    order; four-byte pieces, a value and then its step, eight bytes a word."""
    pieces = store[0] * store[1] // 32
    writes, reads = ([range(i * w // 32, (i + 1) * w // 32) for i in range(n)] for n, w in (store, load))
    for order in itertools.permutations([("w", e) for e in writes] + [("r", e) for e in reads]):
        memory, seen = [0] * pieces, [0] * pieces
        for what, element in order:
            for i in element:
                if what == "w":
                    memory[i] = 1
                else:
                    seen[i] = memory[i]
        if any(seen[i + 1] > seen[i] for i in range(0, pieces, 2)):
            return True
    return False


def test_a_word_that_carries_its_step_is_never_seen_in_part():
    assert _torn_reads((4, 32), (4, 32)) and _torn_reads((2, 32), (1, 64)) and not _torn_reads((1, 64), (1, 64))
    accesses = _word_accesses()
    assert [n * bits for n, bits in accesses["ld"]] == [n * bits for n, bits in accesses["st"]] == [64, 128]
    for load, store in zip(accesses["ld"], accesses["st"]):
        assert not _torn_reads(store, load), (store, load)


# preprocess.cu as it is, but for launches that are recorded instead of made
LAUNCHES = """
#include <cuda_runtime.h>
static int attributes = -1;
static cudaError_t outcome = cudaSuccess, last = cudaSuccess;
template <class K, class... Args> static cudaError_t recorded(const cudaLaunchConfig_t* cfg, K, Args&&...) {
  attributes = (int)cfg->numAttrs;
  if (outcome != cudaSuccess) last = outcome;
  return outcome;
}
static cudaError_t take_last() { const cudaError_t e = last; last = cudaSuccess; return e; }
#define cudaLaunchKernelEx recorded
#define cudaGetLastError take_last
#define cudaGetDevice(device) (*(device) = 0, cudaSuccess)
#define cudaFuncSetAttribute(...) cudaSuccess
#include "preprocess.cu"
extern "C" int push_with(int dependent_launch) {
  paac::pdl_enabled() = dependent_launch != 0;
  attributes = -1;
  const uint8_t* p = (const uint8_t*)4096;
  return paac_stack_push(p, p, nullptr, (uint8_t*)p, 1, nullptr) == PAAC_OK ? attributes : -2;
}
extern "C" int status_and_error_left(int call, int outcome_of_launch, int error_before) {      // 100 * status + what the caller finds
  const uint8_t* p = (const uint8_t*)4096;
  outcome = (cudaError_t)outcome_of_launch;
  last = (cudaError_t)error_before;
  const int status = call == 0 ? paac_stack_push(p, p, nullptr, (uint8_t*)p, 1, nullptr) : paac_preprocess(p, p, nullptr, (uint8_t*)p, 1, nullptr);
  outcome = cudaSuccess;
  return 100 * status + (int)take_last();
}
"""


def _compiled_cuda(tmp_path, source):
    src, so = tmp_path / "host.cu", tmp_path / "host.so"
    src.write_text(source)
    subprocess.run([pbuild.NVCC] + pbuild.FLAGS + ["-shared", "-I", pbuild.CSRC, str(src), "-o", str(so)], check=True)
    return so


def test_entry_points_without_a_context_follow_the_launch_option(tmp_path):
    push = C.CDLL(str(_compiled_cuda(tmp_path, LAUNCHES))).push_with
    assert [push(1), push(0), push(1)] == [1, 0, 1]


@pytest.mark.parametrize("call", [0, 1])
def test_a_failed_launch_leaves_no_error_behind(tmp_path, call):
    of = C.CDLL(str(_compiled_cuda(tmp_path, LAUNCHES))).status_and_error_left
    assert of(call, 0, 0) == 0
    assert of(call, 9, 0) == 100 * pb.ERR_CUDA          # the launch fails
    assert of(call, 0, 1) == 100 * pb.ERR_CUDA          # an error that the caller had not looked at
