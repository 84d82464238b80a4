"""Cuts of the attention kernels' flat list, on the host: every piece of a (sequence, kv head) names the same cut, from the
lengths alone.  The pieces are counted by that number on a counter that outlives the call, so a piece that took it for
another one (as one whose wait had run out once did: 1) would leave the counter off for every later call."""
import ctypes as C
import itertools
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2402_11809_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module", params=["tc", "rows"])
def lib(request, tmp_path_factory):
    so = tmp_path_factory.mktemp("cut") / "attn_cut.so"
    cmd = [build._nvcc(), "-gencode", "arch=compute_100a,code=compute_100a", "-O0", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
           "-cudart", "static", "-Xlinker", "--unresolved-symbols=ignore-all", os.path.join(HERE, "attn_cut_host.cu"), "-o", str(so)]
    if request.param == "rows":
        cmd.insert(1, "-DKERNEL_ROWS")
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    return C.CDLL(str(so), os.RTLD_LAZY), request.param


@pytest.mark.parametrize("lens,H_kv,n_q,groups", [
    ((9000,), 1, 49, 36), ((16000, 800, 127, 640, 0), 4, 36, 148), ((9001,), 2, 49, 37), ((16000, 300), 1, 64, 64),
    ((-1, 5000, -1, 1), 3, 16, 120), ((128, 127, 129), 8, 4, 148), ((4000,) * 7, 5, 25, 148), ((100,), 1, 4, 148)])
def test_every_piece_names_the_same_cut(lib, lens, H_kv, n_q, groups):
    lib, kernel = lib
    seq = np.array(lens, np.int32)
    prefix, out = np.zeros(len(lens) + 1, np.int32), np.zeros(7 * (groups + len(lens) * H_kv + 8), np.int32)
    p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    n = lib.host_list_pieces(p(seq), p(prefix), len(lens), H_kv, n_q, groups, p(out))
    pieces = out[:7 * n].reshape(n, 7)
    seen = 0
    for (b, h), it in itertools.groupby(pieces, key=lambda v: (v[1], v[2])):
        it = list(it)
        first, tiles = it[0][0], -(-(lens[b] + n_q) // 128)
        assert sum(v[3] for v in it) == tiles == it[0][4]
        assert [v[0] for v in it] == list(range(first, first + len(it)))         # consecutive groups
        slot = first if kernel == "rows" else b * H_kv + h + first
        assert all((v[5], v[6]) == (slot, len(it)) for v in it)
        # counted in any order, with any piece the last one: exactly one finds all others there, and the counter is back
        for last in range(len(it)):
            count = found = 0
            for v in it[last + 1:] + it[:last + 1]:
                if count == v[6] - 1:
                    count, found = 0, found + 1
                else:
                    count += 1
            assert (count, found) == (0, 1)
        seen += 1
    assert seen == H_kv * sum(L >= 0 for L in lens)


@pytest.mark.parametrize("src", ["attn_tc.cu", "attn_rows.cu"])
def test_no_wait_decides_how_a_piece_is_counted(src):
    text = open(os.path.join(build.CSRC, src)).read()
    for call in ("cut_d = share_cut(", "note_if_last("):
        at = text.index(call)
        condition = text[text.rindex("if (", 0, at):at]
        assert not re.search(r"\bok\b", condition), condition
