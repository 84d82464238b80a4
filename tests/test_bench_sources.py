"""bench.py reports a kernel's DRAM traffic only while the sources that the capture was taken of are unchanged: the
hash it compares follows every header that a kernel includes."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join("paper_2402_11809_b200", "csrc")
TABLES = {**bench.ATTN_TRAFFIC, **bench.LMHEAD_TRAFFIC}


@pytest.mark.parametrize("fname,headers", [("attn_tc.cu", ("common.cuh", "tc_common.cuh", "attn_common.cuh")),
                                           ("attn_rows.cu", ("common.cuh", "tc_common.cuh", "attn_common.cuh")),
                                           ("lmhead.cu", ("common.cuh", "tc_common.cuh"))])
def test_hash_follows_every_included_header(tmp_path, fname, headers):
    for d in (CSRC, "include"):
        shutil.copytree(os.path.join(bench.ROOT, d), tmp_path / d)
    before = bench.source_hash(fname, str(tmp_path))
    assert before == bench.source_hash(fname)
    for path in [os.path.join(CSRC, n) for n in (fname,) + headers] + [os.path.join("include", "space.h")]:
        text = (tmp_path / path).read_text()
        (tmp_path / path).write_text(text + "\n")
        assert bench.source_hash(fname, str(tmp_path)) != before, path
        (tmp_path / path).write_text(text)
    assert bench.source_hash(fname, str(tmp_path)) == before
    unrelated = tmp_path / CSRC / "commit.cu"
    unrelated.write_text(unrelated.read_text() + "\n")
    assert bench.source_hash(fname, str(tmp_path)) == before


def test_unchanged_sources_report_their_capture():
    for name, (nbytes, fname, digest) in TABLES.items():
        expect = nbytes if digest == bench.source_hash(fname) else None
        assert bench.measured_traffic(TABLES, name) == expect
