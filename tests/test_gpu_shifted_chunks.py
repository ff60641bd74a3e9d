"""GPU tests of chunks that do not start on a 16-byte boundary: every shift
that an element type allows, at piece lengths around the sweep's register
stages (4 and 8 blocks) and sum segments (32 blocks).

The outputs of a chunk depend on its bytes alone, so a state of shifted views
must give the table and the packed buffer of the same bytes at aligned
addresses, bit for bit; that aligned state is compared with the oracle.  The
destinations lie back to back with a few filled bytes between them, so a
granule shared with a neighbour shows a byte written too many."""
import pytest
import torch

from gpu_helpers import compare_full

pytestmark = pytest.mark.gpu

fr = pytest.importorskip("paper_2509_03047_gb300.flashrec")

BLOCKS = [1, 2, 3, 4, 5, 7, 8, 9, 11, 12, 15, 16, 17, 31, 32, 33, 35, 36, 37, 39, 40, 41, 47, 48, 49, 63, 64, 65, 72, 73]


def _values(dtype, nbytes, gen, kind):
    if dtype == torch.uint8:
        return torch.randint(0, 256, (nbytes,), generator=gen, device="cuda", dtype=torch.uint8)
    n = nbytes // dtype.itemsize
    x = torch.randn(n, generator=gen, device="cuda")
    if kind == 1:
        x[n // 3] = float("nan")
        x[n // 2] = float("-inf")
    elif kind == 2:
        x = x * 1e-25  # squares underflow fp32: the exact path
    elif kind == 3:
        x = torch.zeros_like(x)
    return x.to(dtype)


def _carve(sizes, dtype, shift, gap, fill):
    """Views of the given byte sizes at addresses = shift (mod 16), at least `gap` filled bytes apart (a gap under 16: only the first one is at `shift`)."""
    at, offs = 256 + shift, []
    for n in sizes:
        offs.append(at)
        at += n + gap
        at += (shift - at) % 16 if gap >= 16 else 0
    whole = torch.full((at + 256,), fill, dtype=torch.uint8, device="cuda")
    views = []
    for n, o in zip(sizes, offs):
        v = whole[o:o + n]
        views.append(v if dtype == torch.uint8 else v.view(dtype))
    return whole, offs, views


CASES = ([(torch.uint8, s) for s in range(1, 16)] + [(torch.bfloat16, s) for s in range(2, 16, 2)]
         + [(torch.float32, s) for s in (4, 8, 12)])


@pytest.mark.parametrize("dtype,shift", CASES)
def test_shifted_equals_aligned(dtype, shift):
    gen = torch.Generator(device="cuda").manual_seed(100 + shift)
    eb = dtype.itemsize
    sizes = [512 * b + eb * (i % 5) for i, b in enumerate(BLOCKS)]
    aligned = [_values(dtype, n, gen, i % 7) for i, n in enumerate(sizes)]
    _, _, src = _carve(sizes, dtype, shift, 16, 0)
    for a, s in zip(aligned, src):
        s.copy_(a)
        assert s.data_ptr() % 16 == shift
    chunk = 40 * 512  # one more than a segment: whole and split tensors
    compare_full(aligned, chunk)
    pa, ps = fr.Plan(aligned, chunk), fr.Plan(src, chunk)
    table, packed = pa.fingerprint(), pa.pack()
    assert torch.equal(ps.fingerprint(), table)
    got, got_table = ps.pack_fp()
    assert torch.equal(got, packed) and torch.equal(got_table, table)
    # destinations at the same shift, the next one starting `eb` bytes later
    for fused in (False, True):
        whole, offs, dst = _carve(sizes, dtype, shift, eb, 0xA5)
        pd = fr.Plan(dst, chunk)
        if fused:
            _, n, t = pd.unpack_verify_fp(packed)
            assert torch.equal(t, table)
        else:
            _, n = pd.unpack_verify(packed)
        assert n == 0
        want = torch.full_like(whole, 0xA5)
        for a, o, nb in zip(aligned, offs, sizes):
            want[o:o + nb] = a.view(torch.uint8)
        assert torch.equal(whole, want)


def test_chunk_size_that_is_not_a_multiple_of_16():
    """An aligned tensor whose chunks start at every 4-byte boundary."""
    gen = torch.Generator(device="cuda").manual_seed(7)
    ts = [_values(torch.float32, 300004, gen, 0), _values(torch.bfloat16, 200002, gen, 1),
          _values(torch.uint8, 100001, gen, 0)]
    for chunk in (1028, 17 * 512 + 4, 33 * 512 + 8, 65 * 512 + 12):
        compare_full(ts, chunk)


def test_resend_of_shifted_chunks():
    gen = torch.Generator(device="cuda").manual_seed(9)
    sizes = [512 * b + 4 for b in BLOCKS]
    _, _, src = _carve(sizes, torch.float32, 4, 16, 0)
    for i, s in enumerate(src):
        s.copy_(_values(torch.float32, sizes[i], gen, i % 4))
    whole, offs, dst = _carve(sizes, torch.float32, 12, 16, 0xA5)
    chunk = 40 * 512
    ps, pd = fr.Plan(src, chunk), fr.Plan(dst, chunk)
    packed, table = ps.pack_fp()
    start = fr.fr_plan_chunk(ps.handle, 0)[3]
    packed[start::4096] ^= 1  # nearly every chunk fails
    _, n, table_r = pd.unpack_verify_fp(packed)
    assert n > len(sizes) // 2
    fr.fr_resend_fp(ps.handle, pd.handle, packed, table, table_r)
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    fr.fr_unpack_collect(pd.handle, None, count)
    torch.cuda.synchronize()
    assert int(count.item()) == 0 and torch.equal(table, table_r) and torch.equal(table, ps.fingerprint())
    want = torch.full_like(whole, 0xA5)
    for s, o, nb in zip(src, offs, sizes):
        want[o:o + nb] = s.view(torch.uint8)
    assert torch.equal(whole, want)
