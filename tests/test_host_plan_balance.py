"""Balance of the batched plan's work lists, on the CPU: the plan's host code with the CUDA
calls replaced by host-memory stand-ins and the launch by one that keeps the list."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = os.path.join(ROOT, "paper_1612_09001_gb300", "csrc", "batched_api.cu")


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host C++ compiler")
def test_short_streams_spread_over_the_ctas(tmp_path):
    """Many streams shorter than a sub-block, beside a long one and alone: no CTA takes
    more than 1.5 times the mean (a list by valid samples alone gave one CTA up to 39 times)."""
    src = open(SRC).read()
    src = src.replace('#include <cuda_runtime.h>', '#include "stub_cuda.h"')
    src = src.replace('#include "dpd_batched.cuh"', '#include "stub_batched.h"')
    src = src.replace('#include "../../include/dpd.h"', '#include "dpd.h"')
    src = re.sub(r"^namespace dpd \{\n.*?^\}  // namespace dpd\n", "", src, count=1, flags=re.S | re.M)
    (tmp_path / "api_host.cpp").write_text(src)
    stub = open(os.path.join(HERE, "hoststub", "stub_batched.h")).read()
    stub, k = re.subn(r"(inline cudaError_t launch_batched_\d+\(const BatchArgs &a,[^{]*)\{ return 0; \}",
                      r"\1{ return record(a); }", stub)
    assert k == 2
    stub = stub.replace("inline cudaError_t launch_wl_table", "int record(const BatchArgs &a);\ninline cudaError_t launch_wl_table")
    (tmp_path / "stub_batched.h").write_text(stub)
    shutil.copy(os.path.join(HERE, "hoststub", "plan_balance_main.cpp"), tmp_path / "main.cpp")
    exe = str(tmp_path / "t")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(tmp_path), "-I", os.path.join(HERE, "hoststub"),
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.dirname(SRC),
                        str(tmp_path / "api_host.cpp"), str(tmp_path / "main.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, (r.returncode, r.stdout + r.stderr)
    print(r.stdout)
    # shape 8 has 8 samples per thread: its items are dealt out in order
    dealt = re.findall(r"in order: (\d)\nmix .* shape (\d)", r.stdout)
    assert len(dealt) == 12 and all((d == "1") == (v == "8") for d, v in dealt), r.stdout
    worst = [float(v) for v in re.findall(r"largest ([0-9.]+) of the mean", r.stdout)]
    assert len(worst) == 12 and max(worst) <= 1.5, r.stdout
