"""Kernels whose launch bounds leave few registers spill none of them (ptxas' own report)."""
import os
import re
import subprocess

import pytest

from paper_2402_11809_b200 import build


def spills(src, obj):
    cmd = [build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-Xptxas", "-v",
           "-c", os.path.join(build.CSRC, src), "-o", str(obj)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    return {m[1]: int(m[2]) for m in re.finditer(r"Compiling entry function '(\w+)'.*?\n.*?\n.*?(\d+) bytes spill stores", res.stderr)}


@pytest.mark.parametrize("src,kernel,most", [("verify.cu", "verify", 0)])
def test_no_spills(tmp_path, src, kernel, most):
    found = {n: b for n, b in spills(src, tmp_path / (src + ".o")).items() if kernel in n}
    assert len(found) > 8 and max(found.values()) <= most, found
