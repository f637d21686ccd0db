"""No caller drops the error of a launch: the launch functions are [[nodiscard]] and their callers compile cleanly."""
import os
import re
import subprocess

import pytest

from paper_2512_01055_gb300 import build

CSRC = build.CSRC


def test_every_launch_function_is_nodiscard():
    decl = open(os.path.join(CSRC, "tc_internal.cuh")).read()
    names = re.findall(r"^(\[\[nodiscard\]\] )?cudaError_t (\w+)\(", decl, re.M)
    assert len(names) >= 13
    assert [n for mark, n in names if not mark] == []


@pytest.mark.parametrize("src", ["tc_serve.cu", "tc_api.cu", "tc_noalloc.cu"])
def test_callers_use_every_result(src, tmp_path):
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-c", os.path.join(CSRC, src), "-o",
                        str(tmp_path / "out.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert "nodiscard" not in r.stderr and "unused-result" not in r.stderr, r.stderr
