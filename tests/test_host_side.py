"""The library's host side on the CPU: csrc/capi.cpp and csrc/mechanism.cpp linked
against a CUDA runtime in host memory (tests/native/fakecuda.h) whose default stream
finishes its work as late as it may, and kernels that only leave traces."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2501_00011_gb300", "csrc")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    out = str(tmp_path_factory.mktemp("hostside") / "hostside")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "native", "hostside.cpp"),
                    os.path.join(CSRC, "capi.cpp"), os.path.join(CSRC, "mechanism.cpp"), "-ldl", "-o", out], check=True)
    return out


@pytest.mark.parametrize("scenario", ["create_is_complete", "pipeline_is_ordered", "pipeline_memory",
                                      "pipeline_shape", "graph_order", "shape_rule", "register_choice"])
def test_host_side(exe, scenario):
    r = subprocess.run([exe, scenario], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
