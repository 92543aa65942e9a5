"""The sort of the screen's lists (csrc/list_sort.cuh) on its own, against numpy's sort of the same 64-bit keys.

In a whole call the fix-up recomputes what lies close together, so that the lists do not show in what order the screen had left it.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ONE = np.float32(1.0).view(np.uint32)          # its low byte is 0: scores that differ in that byte alone share a sort word


@pytest.fixture(scope="module")
def sort_lists(tmp_path_factory):
    lib_path = str(tmp_path_factory.mktemp("list_sort") / "list_sort.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-I", os.path.join(ROOT, "paper_2607_25291_b200", "csrc"), "-o", lib_path,
                           os.path.join(ROOT, "tests", "list_sort_kernel.cu")])
    lib = ctypes.CDLL(lib_path)
    lib.sort_lists.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]

    def run(scores):
        """scores [lists, J] float32 -> (sorted keys [lists, J] uint64, cycles [lists])"""
        lists, J = scores.shape
        dev = torch.from_numpy(np.ascontiguousarray(scores)).cuda()
        out = torch.zeros(lists, 256, dtype=torch.int64, device="cuda")
        cycles = torch.zeros(lists, dtype=torch.int64, device="cuda")
        per = 2 if J <= 64 else (4 if J <= 128 else 8)
        assert lib.sort_lists(dev.data_ptr(), lists, J, per, out.data_ptr(), cycles.data_ptr()) == 0
        return out.cpu().numpy().view(np.uint64)[:, :J], cycles.cpu().numpy()

    return run


def scores_of(kind, lists, J, rng):
    ids = np.arange(J, dtype=np.uint32)
    if kind == "spread":
        x = rng.gamma(2.0, size=(lists, J)).astype(np.float32)
        return np.where(rng.random((lists, J)) < 0.1, -x, x)              # (some flagged)
    if kind == "equal":
        return np.full((lists, J), 0.75, dtype=np.float32)
    if kind == "zero":
        return np.zeros((lists, J), dtype=np.float32)
    if kind == "rising":                                                  # one sort word, in the reverse of its order
        return np.tile((ONE + ids).view(np.float32), (lists, 1))
    if kind == "falling":
        return np.tile((ONE + ids[::-1]).view(np.float32), (lists, 1))
    if kind == "one word":
        return (ONE + rng.integers(0, 256, (lists, J)).astype(np.uint32)).view(np.float32)
    if kind == "rising runs":                                             # as many runs as lists, all lengths among them
        run = 1 + np.arange(lists, dtype=np.uint32)[:, None] % J
        return (ONE - 256 * (ids // run) + ids % run % 256).astype(np.uint32).view(np.float32)
    if kind == "limits":                                                  # infinities, NaN, the smallest and largest values, flagged ones too
        pool = np.array([np.inf, -np.inf, np.nan, 0.0, 1e-45, -1e-45, 1.1754944e-38, 3.4028235e38, -3.4028235e38, 1.0], dtype=np.float32)
        return pool[rng.integers(0, len(pool), (lists, J))]
    raise ValueError(kind)


def sorted_keys(scores):
    J = scores.shape[1]
    high = np.where(np.isnan(scores), np.uint32(0x7fffffff), np.abs(scores).view(np.uint32))             # (what fabsf makes of a NaN)
    high = high | np.where(scores < 0, np.uint32(0x80000000), np.uint32(0))
    keys = (high.astype(np.uint64) << np.uint64(32)) | (np.uint64(0xffffffff) - np.arange(J, dtype=np.uint64))
    return np.sort(keys, axis=1)[:, ::-1]


@pytest.mark.parametrize("kind", ["spread", "equal", "zero", "rising", "falling", "one word", "rising runs", "limits"])
@pytest.mark.parametrize("J", [1, 17, 33, 63, 64, 65, 128, 129, 200, 255, 256])
def test_lists_are_sorted_whatever_their_scores(sort_lists, J, kind):
    scores = scores_of(kind, 67, J, np.random.default_rng(J))
    got, _ = sort_lists(scores)
    assert np.array_equal(got, sorted_keys(scores))


@pytest.mark.parametrize("kind", ["equal", "rising", "one word"])
def test_lists_of_scores_close_together_take_a_bounded_time(sort_lists, kind):
    """256 candidates, their scores in one sort word: at most six times the time of scores far apart.  (By instructions, words sorted and
    settled in two turns come to some 1,050, with six turns and a second sort of words to 2,300, 128 turns to 10,500.)"""
    rng = np.random.default_rng(1)
    far, close = (np.median([sort_lists(scores_of(k, 64, 256, rng))[1] for _ in range(3)]) for k in ("spread", kind))
    assert close <= 6 * far, (close, far)
