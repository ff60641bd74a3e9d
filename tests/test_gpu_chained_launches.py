"""A call's kernels start while the kernel before them ends.  Nothing may be read
too early or written too late, whatever runs before and after on the stream:
results of calls enqueued back to back, with other kernels rewriting their
inputs in between, equal those of the same calls with a wait after each; and a
pipeline over two streams replays from a graph.  Source and destination lie on
and off the 16-byte boundary: the sweeps of shifted chunks keep what they read
in L1."""
import pytest
import torch

pytestmark = pytest.mark.gpu

fr = pytest.importorskip("paper_2509_03047_gb300.flashrec")


# (element type, bytes off the 16-byte boundary of the source, of the destination)
PLACES = [(torch.float32, 0, 0), (torch.float32, 4, 0), (torch.float32, 0, 4), (torch.bfloat16, 2, 6)]


def _views(sizes, dtype, shift):
    """Zeros, each tensor `shift` bytes off the boundary."""
    k = shift // dtype.itemsize
    return [torch.zeros(n + k, dtype=dtype, device="cuda")[k:] for n in sizes]


def _state(sizes, dtype, shift, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = _views(sizes, dtype, shift)
    for t in out:
        t.copy_(torch.randn(t.numel(), device="cuda", generator=g))
    return out


def _sizes(total):
    """Tensors of odd sizes: one large, some with a tail, some of less than a block."""
    return [total, 1, 127, 128, 4099, 65536 + 3, 33, 262144 + 77]


# chunk counts below and above one tile of the compaction, and a state of many waves of finalize
@pytest.mark.parametrize("place", PLACES)
@pytest.mark.parametrize("total,chunk", [(1000, 4096), (1 << 20, 16384), (40 << 20, 4096), (40 << 20, 1 << 20)])
def test_back_to_back_calls_equal_calls_with_waits(total, chunk, place):
    dtype, shift, shift_out = place

    def run(wait):
        src = _state(_sizes(total), dtype, shift)
        dst = _views(_sizes(total), dtype, shift_out)
        a, b = fr.Plan(src, chunk), fr.Plan(dst, chunk)
        packed, out = a.new_packed(), []
        mism = torch.empty(a.n_chunks, dtype=torch.int32, device="cuda")
        div = torch.empty(a.n_chunks, dtype=torch.int32, device="cuda")

        def sync():
            if wait:
                torch.cuda.synchronize()

        for k in range(4):
            ta, tb, tc = a.new_table(), a.new_table(), b.new_table()
            nmis, ndiv = (torch.empty(1, dtype=torch.int64, device="cuda") for _ in range(2))
            for t in src:
                t.mul_(1.25)
            sync()
            fr.fr_fingerprint(a.handle, ta)
            sync()
            for t in src:
                t.add_(k + 1)
            sync()
            fr.fr_pack_fp(a.handle, packed, tb)
            sync()
            packed[packed.numel() // 2 :: 100003] ^= 1
            sync()
            fr.fr_unpack_verify_fp(b.handle, packed, mism, nmis, tc)
            sync()
            fr.fr_diff(tb, tc, a.n_chunks, div, ndiv)
            sync()
            out += [ta.clone(), tb.clone(), tc.clone(), nmis.clone(), ndiv.clone(), packed.clone()]
            out += [t.clone() for t in dst]
            packed.fill_(0)
            fr.fr_pack(a.handle, packed)
            sync()
            fr.fr_unpack_verify(b.handle, packed, mism, nmis)
            sync()
            out += [nmis.clone()] + [t.clone() for t in dst]
        torch.cuda.synchronize()
        return [t.reshape(-1).view(torch.uint8) for t in out]

    got, want = run(False), run(True)
    assert all(torch.equal(x, y) for x, y in zip(got, want))


@pytest.mark.parametrize("place", PLACES)
def test_batches_on_two_streams_replay_from_a_graph(place):
    dtype, shift, shift_out = place
    src = _state(_sizes(8 << 20), dtype, shift, 1)
    dst = _views(_sizes(8 << 20), dtype, shift_out)
    batches = 6
    a = fr.fr_plan_create_batched(src, 65536, batches)
    b = fr.fr_plan_create_batched(dst, 65536, batches)
    whole = fr.Plan(src, 65536)
    packed, want = whole.new_packed(), whole.new_packed()
    count = torch.empty(1, dtype=torch.int64, device="cuda")
    s, r = torch.cuda.Stream(), torch.cuda.Stream()

    def pipeline():
        r.wait_stream(s)
        for i in range(batches):
            fr.fr_pack_batch(a, i, packed, s)
            r.wait_stream(s)
            fr.fr_unpack_verify_batch(b, i, packed, r)
        fr.fr_unpack_collect(b, None, count, r)
        s.wait_stream(r)

    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        pipeline()
    for k in range(3):
        for t in src:
            t.add_(1)
        fr.fr_pack(whole.handle, want)
        for t in dst:
            t.fill_(k)
        packed.fill_(k)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(packed, want) and int(count.item()) == 0
        assert all(torch.equal(x, y) for x, y in zip(src, dst))
    fr.fr_plan_destroy(a)
    fr.fr_plan_destroy(b)
