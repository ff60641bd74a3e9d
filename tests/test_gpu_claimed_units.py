"""GPU tests of the work units that pack and unpack warps claim at run time.

A pack or unpack launch leaves the last few percent of each class's segments
out of the warps' own runs, where the class has at least four segments per warp,
and cuts them into units that warps claim through one counter per batch.  The
counter wraps to zero on a launch's last claim, so the next launch on the plan
finds it so.  The state here has all six classes (bf16, fp32 and bytes, on and
off the 16-byte boundary), each with units, which the tests assert for this
GPU's SMs from the planner itself (tests/c/plan_units.cc).  Outputs must equal
the oracle's, and those of many launches queued back to back with no host
synchronization, the state changing in between, must be right each time (a
counter left non-zero would make a later launch skip units: stale payload bytes,
records and sums), for the whole-state calls and for the batched restore, whose
batches each have a counter."""
import numpy as np
import pytest
import torch

from gpu_helpers import compare_full
from host_tests import plan_units

pytestmark = pytest.mark.gpu

fr = pytest.importorskip("paper_2509_03047_gb300.flashrec")

MiB = 1024 * 1024
CLASSES = {0, 1, 2, 3, 4, 5}  # element type * 2 + (on the 16-byte boundary)


@pytest.fixture(autouse=True)
def _free_memory():
    yield
    torch.cuda.synchronize()
    torch.cuda.empty_cache()


def _values(count, dtype, gen):
    if dtype == torch.uint8:
        return torch.randint(0, 256, (count,), generator=gen, device="cuda", dtype=dtype)
    return torch.randn(count, generator=gen, device="cuda").to(dtype)


def _state(rounds=1):
    """60 MiB per class and a small tensor; `rounds`: that in so many parts, class by class in turn."""
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    out = []
    for _ in range(rounds):
        for dtype, shift in ((torch.bfloat16, 0), (torch.bfloat16, 3), (torch.float32, 0), (torch.float32, 1),
                             (torch.uint8, 0), (torch.uint8, 5)):
            n = 60 * MiB // rounds // dtype.itemsize + 77
            out.append(_values(n + 16, dtype, g)[shift:shift + n])
    return out + [torch.randn(12345, generator=g, device="cuda")]


def _like(state):
    """Empty tensors that lie on and off the 16-byte boundary as those of `state` do."""
    out = []
    for t in state:
        shift = t.storage_offset()
        out.append(torch.empty(t.numel() + shift, dtype=t.dtype, device="cuda")[shift:])
    return out


def _assert_units(tmp_path, state, n_batches=1):
    """Every class of the whole-state launch, and of every batch, has claimable units."""
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    codes = [fr.fr_dtype_of(t) for t in state]
    units = plan_units(tmp_path, state, codes, 1 * MiB, n_batches, n_sm)
    assert set(units) == ({None} if n_batches == 1 else {None, *range(n_batches)})
    for launch, per_class in units.items():
        assert set(per_class) == CLASSES and min(per_class.values()) > 0, (launch, per_class)


def _same(a, b):
    return all(torch.equal(x.view(torch.uint8), y.view(torch.uint8)) for x, y in zip(a, b))


def test_claimed_units_match_the_oracle(tmp_path):
    state = _state()
    _assert_units(tmp_path, state)
    compare_full(state, 1 * MiB, flips=np.array([8 * 4096 + 3, 8 * (9 << 20) + 1, 8 * (300 << 20)], dtype=np.int64))


def test_many_launches_back_to_back(tmp_path):
    st = _state()
    plan = fr.Plan(st, 1 * MiB)
    out = _like(st)
    plan_r = fr.Plan(out, 1 * MiB)
    _assert_units(tmp_path, st)
    _assert_units(tmp_path, out)
    n = 12
    packed = [plan.new_packed() for _ in range(n)]
    counts = torch.empty((2, n), dtype=torch.int64, device="cuda")
    tabs, tabs_r = ([plan.new_table() for _ in range(n)] for _ in range(2))
    want, fused, plain = [], [], []
    for i in range(n):  # no synchronization between the launches
        for t in st:
            t.add_(1)
        want.append([t.clone() for t in st])
        fr.fr_pack_fp(plan.handle, packed[i], tabs[i])
        fr.fr_unpack_verify_fp(plan_r.handle, packed[i], None, counts[0, i:i + 1], tabs_r[i])
        fused.append([t.clone() for t in out])
    for i in range(n):
        fr.fr_unpack_verify(plan_r.handle, packed[i], None, counts[1, i:i + 1])
        plain.append([t.clone() for t in out])
    torch.cuda.synchronize()
    assert counts.tolist() == [[0] * n] * 2
    for i in range(n):
        ref = fr.Plan(want[i], 1 * MiB)
        table = ref.fingerprint()
        assert torch.equal(tabs[i], table) and torch.equal(tabs_r[i], table), "launch %d: tables" % i
        assert _same(fused[i], want[i]), "launch %d: restored tensors" % i
        assert _same(plain[i], want[i]), "launch %d: tensors of the plain unpack" % i
        ref.close()
    plan_r.close()
    plan.close()


def test_batched_restore_repeated(tmp_path):
    batches = 3
    st = _state(rounds=2 * batches)
    out = _like(st)
    _assert_units(tmp_path, st, batches)
    _assert_units(tmp_path, out, batches)
    src, dst = fr.Plan(st, 1 * MiB, n_batches=batches), fr.Plan(out, 1 * MiB, n_batches=batches)
    staging = src.new_packed()
    fa, fb = src.new_table(), dst.new_table()
    cnt = torch.empty(1, dtype=torch.int64, device="cuda")
    for k in range(4):
        for t in st:
            t.add_(1)
        for t in out:
            t.view(torch.uint8).fill_(0xA5)
        fr.fr_restore_fp(src.handle, dst.handle, staging, 1, None, cnt, fa, fb)
        torch.cuda.synchronize()
        assert int(cnt.item()) == 0, "round %d" % k
        ref_tab = fr.Plan(st, 1 * MiB).fingerprint()
        assert torch.equal(fa, ref_tab) and torch.equal(fb, ref_tab), "round %d: tables" % k
        assert _same(out, st), "round %d: restored tensors" % k
    src.close()
    dst.close()
