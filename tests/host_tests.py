"""Programs of tests/c that include csrc/api.cu over tests/c/fake_cuda.h, built with the host compiler."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build_host_test(name, out_dir):
    from paper_2509_03047_gb300 import build

    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    exe = os.path.join(str(out_dir), name)
    cmd = ["g++", "-std=c++17", "-O1", "-isystem", cuda, "-I", os.path.join(ROOT, "tests", "c"), "-I", build.CSRC,
           os.path.join(ROOT, "tests", "c", name + ".cc"), "-o", exe, "-ldl"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


def plan_units(out_dir, tensors, codes, chunk_bytes, n_batches, n_sm):
    """Claimable units of a pack or unpack launch, as {batch: {sweep class: units}}; batch None is the whole-state
    launch.  `codes`: the tensors' element types (fr_dtype)."""
    lines = ["%d %d %d %d" % (n_sm, chunk_bytes, n_batches, len(tensors))]
    lines += ["%d %d %d" % (t.data_ptr(), t.numel() * t.element_size(), c) for t, c in zip(tensors, codes)]
    r = subprocess.run([build_host_test("plan_units", out_dir)], input="\n".join(lines) + "\n", capture_output=True,
                       text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    out = {}
    for line in r.stdout.splitlines():
        batch, cls, units = (int(v) for v in line.split())
        out.setdefault(None if batch < 0 else batch, {})[cls] = units
    return out
