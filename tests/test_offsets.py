"""Utterance offsets are the caller's data: which row a closing kernel fetches ahead of the streaming
kernel's end, for offsets of every kind, from the very functions the kernels call."""
import ctypes as C
import itertools
import os
import subprocess

import pytest
import torch

import helpers as H
from conftest import ROOT
from paper_2603_11243_b200 import binding as ssd

INT64_MAX, INT64_MIN = (1 << 63) - 1, -(1 << 63)
SOURCE = """
#include "ssd_ranges.cuh"
extern "C" long long row(long long i0, long long i1, long long M, int k) {
    return ssd::ranges::row_of_utterance(i0, i1, M, k);
}
extern "C" int sound(long long i0, long long i1, long long M) { return ssd::ranges::rows_sound(i0, i1, M); }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("ranges")
    (d / "r.cpp").write_text(SOURCE)
    # -ftrapv: signed arithmetic that overflows on the way ends the process
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-ftrapv", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2603_11243_b200", "csrc"), str(d / "r.cpp"), "-o", str(d / "r.so")],
                   check=True)
    lib = C.CDLL(str(d / "r.so"))
    lib.row.restype = C.c_longlong
    lib.row.argtypes = [C.c_longlong, C.c_longlong, C.c_longlong, C.c_int]
    lib.sound.argtypes = [C.c_longlong] * 3
    return lib


def test_rows_fetched_ahead_lie_inside_the_matrix(host):
    ends = [INT64_MIN, INT64_MIN + 500, -1, 0, 1, 3, 7, 30, 31, 1 << 31, INT64_MAX - 1024, INT64_MAX - 5, INT64_MAX]
    for M, i0, i1 in itertools.product((0, 1, 7, 30), ends, ends):
        inside = 0 <= i0 <= i1 <= M
        assert bool(host.sound(i0, i1, M)) == inside
        for k in (0, 1, 6, 29, 30, 511, 1023):
            want = i0 + k if inside and k < i1 - i0 else -1
            assert host.row(i0, i1, M, k) == want, (M, i0, i1, k)


@pytest.mark.gpu
@pytest.mark.parametrize("kernel", [0, 1, 2])
def test_offsets_at_the_ends_of_int64(cuda_device, kernel):
    """Flagged and treated as empty, the sound utterances beside them unharmed."""
    M, V, dev = 30, 900, cuda_device
    g = torch.Generator().manual_seed(9)
    x = torch.randn((M, V), generator=g).bfloat16().to(dev)
    ids = x.float().argmax(1).to(torch.int32)
    off = torch.tensor([0, 10, INT64_MAX - 100, 20, 30, INT64_MIN + 100, 5, INT64_MAX, INT64_MAX - 1000, 12, 30],
                       dtype=torch.int64, device=dev)
    bad = [0, 1, 1, 0, 1, 1, 1, 1, 1, 0]
    lens = [10, 0, 0, 10, 0, 0, 0, 0, 0, 18]
    o = H.opts(kernel=kernel)
    v = ssd.ssd_verify(x, off, ids, 0.0, opts=o)
    e = ssd.ssd_verify_early_exit(x, off, ids, 0.0, opts=o)
    stats = ssd.ssd_verify_shard(x, 0, off, ids, opts=o)
    c = ssd.ssd_verify_combine(stats[None], V, off, ids, 0.0)
    torch.cuda.synchronize()
    for out in (v, e, c):
        assert H.status_u32(out["utt_status"]).tolist() == [ssd.UTT_BAD_OFFSETS * b for b in bad]
        assert out["accepted_len"].tolist() == lens
        assert out["all_accepted"].tolist() == [1 - b for b in bad]
