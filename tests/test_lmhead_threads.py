"""space_lmhead_verify from several threads, each with its own context, on the host side alone (csrc/lmhead.cu against
a stand-in for the CUDA runtime, no GPU): the kernels are the process's, so what one call raises of their limits another
must not lower before the first has launched."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2402_11809_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def B():
    build.build()
    from paper_2402_11809_b200 import binding
    return binding


@pytest.fixture(scope="module")
def lib(B, tmp_path_factory):
    so = tmp_path_factory.mktemp("fake") / "lmhead_fake.so"
    cmd = [build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
           "-Xlinker", "-Bsymbolic", "-cudart", "none", os.path.join(build.CSRC, "lmhead.cu"),
           os.path.join(HERE, "lmhead_calls_fake.cu"), os.path.join(HERE, "fake_launch_limits.cpp"), "-o", str(so)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    lib = C.CDLL(str(so))
    lib.fake_lmhead_two.argtypes = [C.POINTER(B.LmHeadArgs)] * 2 + [C.c_int, C.POINTER(C.c_int), C.POINTER(C.c_size_t)]
    lib.fake_lmhead_launches.argtypes = [C.POINTER(B.LmHeadArgs)]
    return lib


def _args(B, batch, k, V, D, sample):
    a = B.LmHeadArgs()
    a.batch, a.k, a.vocab, a.hidden_dim = batch, k, V, D
    a.hidden_row_stride = a.weight_row_stride = D
    a.mode, a.temperature, a.eos_id = B.MODE_SAMPLE if sample else B.MODE_GREEDY, 1.0, -1
    # (nothing is read: the first launch stands for all of the call)
    a.hidden = a.weight = a.cand = a.cand_prob = a.n_accept = a.out_tokens = a.n_out = a.next_cand = a.next_cand_prob = a.finished = 4096
    return a


# A call whose launch needs more shared memory than the other thread's, for each build of the kernel: tokens on M, rows
# on M, sampling; and by phase, before each of its launches.
@pytest.mark.parametrize("big,small", [((1, 5, 32000, 4096), (1, 1, 30011, 256)), ((5, 5, 32000, 4096), (1, 1, 40, 64)),
                                       ((16, 5, 32000, 4096), (1, 1, 40, 64))])
@pytest.mark.parametrize("sample", [False, True])
@pytest.mark.parametrize("at", [1, 2, 3])
def test_another_threads_call_before_a_launch(B, lib, big, small, sample, at):
    a, b = _args(B, *big, sample), _args(B, *small, sample)
    rc, smem = (C.c_int * 2)(), C.c_size_t()
    for x, y in ((a, b), (b, a)):
        lib.fake_lmhead_two(C.byref(x), C.byref(y), at, rc, C.byref(smem))
        assert list(rc) == [B.OK, B.OK]
        assert smem.value <= 227 * 1024


# Beyond 256 block rows a group of sequences takes three launches (targets, gather, masks), each group two passes over the
# embedding.  As many sequences as an accumulator of 128 rows holds, up to D = 16384; beyond it the gathered rows' buffer
# (128 * 16384 elements) decides, never on fewer than 128 * 8192 // (k D), greedy or sampling.
@pytest.mark.parametrize("sample", [False, True])
@pytest.mark.parametrize("batch,k,D,groups", [(12, 5, 16384, 1), (17, 5, 12288, 1), (21, 5, 16384, 1), (22, 5, 16384, 2),
                                              (9, 7, 16384, 1), (128, 1, 16384, 2), (42, 2, 8192, 1), (65, 1, 24008, 2)])
def test_groups_of_wide_hidden_rows(B, lib, batch, k, D, groups, sample):
    assert lib.fake_lmhead_launches(C.byref(_args(B, batch, k, 32000, D, sample))) == 3 * groups
