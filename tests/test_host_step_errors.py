"""space_step_host when something goes wrong, on the host side alone (csrc/space_api.cu against a stand-in for the
CUDA runtime, no GPU): a bad argument is found before anything is launched, and a failing call returns only when
nothing that it launched can still touch the caller's buffers, with no status bits left for the next call."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2402_11809_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))
BATCH, K, VOCAB, HEADS, DIM, CAP = 2, 2, 64, 2, 64, 64


@pytest.fixture(scope="module")
def B():
    build.build()
    from paper_2402_11809_b200 import binding
    return binding


@pytest.fixture(scope="module")
def lib(B, tmp_path_factory):
    so = tmp_path_factory.mktemp("fake") / "libspace_fake.so"
    cmd = [build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
           "-Xlinker", "-Bsymbolic", "-cudart", "none", os.path.join(build.CSRC, "space_api.cu"),
           os.path.join(HERE, "host_step_fake.cu"), os.path.join(HERE, "fake_cuda_runtime.cpp"), "-o", str(so)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    lib = C.CDLL(str(so))
    lib.space_create.argtypes = [C.POINTER(C.c_void_p), C.POINTER(B.Config)]
    lib.space_step_host.argtypes = [C.c_void_p, C.POINTER(B.HostStepArgs), C.c_void_p]
    lib.fake_reset.argtypes, lib.fake_calls.restype = [C.c_long, C.c_int], C.c_long
    lib.fake_vstatus.argtypes = [C.c_void_p, C.c_int]
    return lib


def _step(B, lib, **over):
    """A context and a valid call on it, changed by `over`; the arrays are kept alive by the caller."""
    ctx = C.c_void_p()
    cfg = B.Config(device=0, max_batch=BATCH, n_q_heads=HEADS, n_kv_heads=HEADS, head_dim=DIM, k_max=K, vocab=VOCAB, host_staging=1, s_cap=CAP)
    lib.fake_reset(0, 0)
    assert lib.space_create(C.byref(ctx), C.byref(cfg)) == B.OK
    n_q = (K + 1) ** 2
    z = lambda n, t: np.zeros(n + 16, t)  # noqa: E731
    h = dict(q=z(BATCH * n_q * HEADS * DIM, np.uint16), k_cache=z(BATCH * HEADS * CAP * DIM, np.uint16), v_cache=z(BATCH * HEADS * CAP * DIM, np.uint16),
             logits=z(BATCH * n_q * VOCAB, np.uint16), cand=z(BATCH * K, np.int32), cand_prob=z(BATCH * K, np.float32), kv_len=z(BATCH, np.int32),
             out=z(BATCH * n_q * HEADS * DIM, np.float32), n_accept=z(BATCH, np.int32), out_tokens=z(BATCH * (K + 1), np.int32), n_out=z(BATCH, np.int32),
             next_cand=z(BATCH * K, np.int32), next_cand_prob=z(BATCH * K, np.float32), finished=z(BATCH, np.uint8), status=z(BATCH, np.int32))
    ptr = {n: (a.ctypes.data + 15) // 16 * 16 for n, a in h.items()}
    args = dict(batch=BATCH, k=K, vocab=VOCAB, logits_dtype=B.DTYPE_BF16, mode=B.MODE_GREEDY, eos_id=-1, scale=0.125, temperature=1.0, **ptr)
    args.update(over)
    return ctx, B.HostStepArgs(**args), h


@pytest.mark.parametrize("resident,pageable", [(1, 0), (1, 1), (0, 0), (0, 1)])
@pytest.mark.parametrize("bad", [dict(scale=0.0), dict(scale=float("nan")), dict(mask_variant=7), dict(mode=5), dict(logits_dtype=9)])
def test_bad_argument_launches_nothing(B, lib, bad, resident, pageable):
    ctx, args, keep = _step(B, lib, cache_resident=resident, **bad)
    lib.fake_reset(0, pageable)
    assert lib.space_step_host(ctx, C.byref(args), None) == B.E_INVALID_ARG
    assert lib.fake_calls() == 0 and not lib.fake_in_flight()


@pytest.mark.parametrize("resident,pageable", [(1, 0), (1, 1), (0, 0), (0, 1)])
def test_failing_call_leaves_nothing_behind(B, lib, resident, pageable):
    ctx, args, keep = _step(B, lib, cache_resident=resident)
    lib.fake_reset(0, pageable)
    assert lib.space_step_host(ctx, C.byref(args), None) == B.OK
    n = lib.fake_calls()
    assert n >= 8 and not lib.fake_in_flight()
    for fail in range(1, n + 1):
        lib.fake_reset(fail, pageable)
        assert lib.space_step_host(ctx, C.byref(args), None) == B.E_CUDA, fail
        assert not lib.fake_in_flight(), fail
        assert [lib.fake_vstatus(ctx, b) for b in range(BATCH)] == [0] * BATCH, fail
