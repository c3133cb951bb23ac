"""The least-squares workspace after a failed allocation, on the CPU: the function that
reserves it, compiled for the host with stand-ins for the CUDA calls."""
import os
import re
import shutil
import subprocess

import pytest

from paper_1612_09001_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1612_09001_gb300", "csrc")


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host C++ compiler")
def test_failed_growth_leaves_no_stale_capacity(tmp_path):
    src = open(os.path.join(CSRC, "gram_api.cu")).read()
    part = re.search(r"^// Floats between the forward tables.*?^dpd_status reserve\(.*?^}\n", src, re.S | re.M)
    (tmp_path / "reserve_part.h").write_text(part.group(0))
    exe = str(tmp_path / "t")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    r = subprocess.run(["g++", "-std=c++17", "-g", "-I", str(tmp_path), "-I", os.path.join(HERE, "..", "include"), "-I", CSRC,
                        "-I", cuda, os.path.join(HERE, "hoststub", "reserve_main.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
