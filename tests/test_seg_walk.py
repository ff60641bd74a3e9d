"""The planner's segment walk (csrc/seg_walk.h), compiled with the host C++
compiler and checked by tests/c/seg_walk_test.cc against the plain rule: the
same run boundaries as split_ranges over all segments' costs, pieces that cover
every segment once and in order, and each chunk's records in one run.  And the
host tables of gf2.cuh: powers of x against square-and-multiply, the per-chunk
CRC term against the CRC of the oracle.  No GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_03047_gb300", "csrc")
FLAGS = ["-std=c++17", "-O1", "-Wall", "-D__host__=", "-D__device__=", "-I", CSRC]

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="g++ not available")


def _run(tmp_path, src):
    exe = str(tmp_path / "t")
    r = subprocess.run(["g++"] + FLAGS + [src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def test_seg_walk(tmp_path):
    assert "seg_walk ok" in _run(tmp_path, os.path.join(ROOT, "tests", "c", "seg_walk_test.cc"))


def test_block_powers(tmp_path):
    blocks = [0, 1, 31, 32, 4095, 4096, 4097, 65536 + 5, (1 << 24) - 1, 1 << 24, (1 << 24) + 33, 10485760]
    src = tmp_path / "t.cc"
    src.write_text('#include <cstdio>\n#include "gf2.cuh"\nint main() {\n' + "".join(
        '  std::printf("%%d\\n", frk::host_xpow8_blocks(%dull) == frk::gf_xpow(%dull));\n' % (b, 8 * 512 * b)
        for b in blocks) + "}\n")
    assert _run(tmp_path, str(src)).split() == ["1"] * len(blocks)


def test_crc_xor_term(tmp_path, orc):
    """The term of n bytes is the CRC of n zero bytes (whose raw CRC is 0)."""
    import numpy as np

    sizes = [0, 1, 3, 4, 511, 4095, 4096, 4097, 65536, 262143, (1 << 24) - 1, 1 << 24, (1 << 24) + 4099, 50331648]
    src = tmp_path / "t.cc"
    src.write_text('#include <cstdio>\n#include "gf2.cuh"\nint main() {\n' + "".join(
        '  std::printf("%%08x\\n", frk::host_crc_xor_term(%dull));\n' % n for n in sizes) + "}\n")
    got = [int(v, 16) for v in _run(tmp_path, str(src)).split()]
    assert got == [orc.crc32c(np.zeros(n, dtype=np.uint8)) for n in sizes]


def test_power_tables_are_constants_of_the_program(tmp_path):
    """No call fills a table: a process's first plan takes what a later one takes."""
    src = tmp_path / "t.cc"
    src.write_text('#include <cstdio>\n#include "gf2.cuh"\nusing namespace frk;\nint main() {\n' + "".join(
        "  { constexpr const DigitTables& T = Digits<%s, %d>::T;\n"
        "    static_assert(T.low[4095] == gf_mulmod(%s, gf_xpow(8ull * %d * 4095)), \"low\");\n"
        "    static_assert(T.high[4095] == gf_xpow(8ull * %d * 4096 * 4095), \"high\"); }\n" % (s, u, s, u, u)
        for s, u in (("0xFFFFFFFFu", 1), ("kOne", 512))) + '  std::puts("ok");\n}\n')
    assert _run(tmp_path, str(src)) == "ok\n"
