"""GPU tests of the sum segments that are redone exactly: by the whole warp for
up to 2 of its lanes (1 where squares are tiny), lane by lane beyond that.

A lane owns bytes 16l..16l+15 of every 512-byte block.  NaN and infinities put
into 1 to 5 and 32 lanes of one segment take both ways, among ordinary values,
in whole segments and short ones; so do lanes whose squares all underflow fp32
and lanes with one that overflows it, each in a state of its own, so that every
such square counts in the sum (added in fp64).  Counts must equal the oracle's
and sums agree to 1e-9; and a lane's share must be the same bit for bit either
way."""
import os
import subprocess

import pytest
import torch

from gpu_helpers import compare_full, table_np

pytestmark = pytest.mark.gpu

fr = pytest.importorskip("paper_2509_03047_gb300.flashrec")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _rows(blocks, dtype, shift, base):
    """A view of `base` off the 16-byte boundary by `shift` bytes, and the same as (block, lane, element of it)."""
    n = blocks * 512 // dtype.itemsize
    x = base[shift // dtype.itemsize:][:n]
    return x, x.view(blocks, 32, 16 // dtype.itemsize)


@pytest.mark.parametrize("shift", [0, 4])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("lanes", [1, 2, 3, 4, 5, 32])
@pytest.mark.parametrize("kind", ["nan", "tiny", "huge"])
def test_segments_redone_exactly(dtype, lanes, shift, kind):
    gen = torch.Generator(device="cuda").manual_seed(lanes)
    tensors = []
    for blocks in (1, 31, 32, 33, 70):
        base = torch.randn(blocks * 512 // dtype.itemsize + 16, generator=gen, device="cuda").to(dtype)
        where = torch.randperm(32, generator=gen, device="cuda")[:lanes]
        if kind == "tiny":  # the sum is that of squares below fp32's range, in these lanes; exact zeros elsewhere
            values = (base.float() * 1e-25).to(dtype)
            x, rows = _rows(blocks, dtype, shift, values)
            keep = torch.zeros(32, dtype=torch.bool, device="cuda")
            keep[where] = True
            rows[:, ~keep] = 0
            rows[blocks // 2, where, 3] = 3e-39  # (subnormal)
        else:
            x, rows = _rows(blocks, dtype, shift, base)
            if kind == "huge":
                rows[blocks // 3, where, 3] = 1e25
            else:
                rows[blocks // 2, where, 1] = float("nan")
                rows[0, where[:1], 0] = float("-inf")
        tensors.append(x)
    compare_full(tensors, 64 * 1024)


@pytest.mark.parametrize("shift", [0, 4])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("center", [1e-12, 1e-11, 1e-10])
def test_second_moments_around_the_line(dtype, center, shift):
    """Values spread as Adam's second moments are: from none to all lanes of a segment have sums too small for the fast
    path, with elements among them whose squares are added in fp64."""
    gen = torch.Generator(device="cuda").manual_seed(3)
    n = 60 * 16384 // dtype.itemsize
    values = torch.randn(n + 16, generator=gen, device="cuda").mul_(2.0).exp_().mul_(center).to(dtype)
    compare_full([values[shift // dtype.itemsize:][:n]], 64 * 1024)


@pytest.mark.parametrize("shift", [0, 4])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_one_lane_adds_the_same_bits_with_others_redone_beside_it(dtype, shift):
    """Lane 9 alone, and the same with lanes that hold NaN only, which add nothing but make the lanes go side by side."""
    gen = torch.Generator(device="cuda").manual_seed(5)
    values = torch.randn(32, 16 // dtype.itemsize, generator=gen, device="cuda").to(dtype)
    values[7, 1], values[8, 0], values[9, 2] = float("nan"), 1e-25, 1e-41
    tensors = []
    for others in (0, 1, 2, 4, 31):
        x, rows = _rows(32, dtype, shift, torch.zeros(16384 // dtype.itemsize + 16, dtype=dtype, device="cuda"))
        rows[:, 9] = values
        for lane in [l for l in range(32) if l != 9][:others]:
            rows[:, lane] = float("nan")
        tensors.append(x)
    table = table_np(fr.Plan(tensors, 16 * 1024).fingerprint())
    per_lane = values.numel()
    assert table["nonfinite"].tolist() == [1 + n * per_lane for n in (0, 1, 2, 4, 31)]
    assert len(set(table["sumsq"].view("int64").tolist())) == 1
    want = float(values.double().masked_fill(values.isnan(), 0.0).square().sum())
    assert abs(table["sumsq"][0] - want) <= 1e-9 * want


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
