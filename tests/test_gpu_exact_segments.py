"""GPU tests of the sum segments that are redone exactly: by the whole warp for
up to 2 of its lanes, lane by lane beyond that.

A lane owns bytes 16l..16l+15 of every 512-byte block.  NaN and infinities put
into 1 to 5 and 32 lanes of one segment take both ways, with elements whose
squares under- or overflow fp32 among them (added in fp64) and in a segment cut
short; counts must equal the oracle's and sums agree to 1e-9."""
import os
import subprocess

import pytest
import torch

from gpu_helpers import compare_full

pytestmark = pytest.mark.gpu

fr = pytest.importorskip("paper_2509_03047_gb300.flashrec")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("shift", [0, 4])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("lanes", [1, 2, 3, 4, 5, 32])
def test_segments_redone_exactly(dtype, lanes, shift):
    gen = torch.Generator(device="cuda").manual_seed(lanes)
    per_lane = 16 // dtype.itemsize
    tensors = []
    for blocks in (1, 31, 32, 33, 70):
        n = blocks * 512 // dtype.itemsize
        base = torch.randn(n + 16, generator=gen, device="cuda").to(dtype)
        x = base[shift // dtype.itemsize:][:n]
        rows = x.view(blocks, 32, per_lane)
        where = torch.randperm(32, generator=gen, device="cuda")[:lanes]
        rows[blocks // 2, where, 1] = float("nan")
        rows[0, where[:1], 0] = float("-inf")
        if blocks > 31:  # odd elements in the same lanes
            rows[3, where, 2] = 1e-25
            rows[5, where, 3] = 1e25
            rows[7, where, 0] = 3e-39
        tensors.append(x)
    compare_full(tensors, 64 * 1024)


@pytest.mark.parametrize("seg_blocks", [32, 64])
def test_the_two_ways_return_the_same_bits(seg_blocks, tmp_path):
    """tests/c/exact_span_test.cu, for segments of the library's size and of twice that."""
    from paper_2509_03047_gb300 import build

    exe = str(tmp_path / "exact_span_test")
    cmd = [build.nvcc()] + build.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                                         "-DFR_SEG_BLOCKS=%d" % seg_blocks,
                                         os.path.join(ROOT, "tests", "c", "exact_span_test.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "exact_span ok" in r.stdout
