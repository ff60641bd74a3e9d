"""A plan's tables have reached device memory when fr_plan_create returns
(csrc/api.cu over tests/c/fake_cuda.h, in which a copy from pageable memory is
done only when something waits for it, as CUDA allows).  No GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build_host_test(name, tmp_path):
    """tests/c/<name>.cc, which includes api.cu over the fake runtime, compiled by the host compiler."""
    from paper_2509_03047_gb300 import build

    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    exe = str(tmp_path / name)
    cmd = ["g++", "-std=c++17", "-O1", "-isystem", cuda, "-I", os.path.join(ROOT, "tests", "c"), "-I",
           os.path.join(ROOT, "paper_2509_03047_gb300", "csrc"), os.path.join(ROOT, "tests", "c", name + ".cc"), "-o",
           exe, "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not available")
def test_plan_tables_are_on_the_device_when_creation_returns(tmp_path):
    r = subprocess.run([build_host_test("plan_upload_test", tmp_path)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "plan_upload ok" in r.stdout
