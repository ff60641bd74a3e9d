"""A plan's tables have reached device memory when fr_plan_create returns
(csrc/api.cu over tests/c/fake_cuda.h, in which a copy from pageable memory is
done only when something waits for it, as CUDA allows), and a status that
fr_sync_status returns has been cleared there.  No GPU."""
import shutil
import subprocess

import pytest

from host_tests import build_host_test


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not available")
def test_plan_tables_are_on_the_device_when_creation_returns(tmp_path):
    r = subprocess.run([build_host_test("plan_upload_test", tmp_path)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "plan_upload ok" in r.stdout


@pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not available")
def test_status_is_cleared_when_it_is_returned(tmp_path):
    r = subprocess.run([build_host_test("sync_status_test", tmp_path)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "sync_status ok" in r.stdout
