"""What is timed: calls that a program restoring training state makes, from the smallest state to a model shard.

A training job keeps, per parameter, a bf16 weight and three fp32 buffers (master weight and the two Adam moments).  To recover
a failed rank without a checkpoint it fingerprints that state, packs it into a transfer buffer, and unpacks and verifies it on
the restarted rank.  Cases differ in the call (`op`), in how the state lies in memory (`layout`) and in its size:

  op           fingerprint   the table that two replicas compare (read-only sweep)
               static        the same for a process that may not allocate device memory; plans on every call
               pack          state -> transfer buffer
               unpack        transfer buffer with a few bits flipped in transit -> state, and the list of failing chunks
               step          one whole recovery through a device buffer: pack and unpack with both tables, then their diff
               restore       the pipelined recovery in batches on two streams, through a device or a pinned host buffer
               reshard       a ZeRO shard rebuilt from replicas that are sharded another way (plans, restore, check)
  layout       model         one allocation per buffer (512-byte aligned, as PyTorch's allocator places them), in tensor order;
                             transformer shapes: embedding, attention, MLP and norm tensors
               fragments     thousands of fp32 tensors of sizes spread from `lo` to `hi` bytes, each its own allocation
               flat          ZeRO / FSDP flat groups: every parameter is a view into one bf16 and three fp32 buffers, back to
                             back, so that parameters of odd sizes start at any element; a few opaque byte buffers of odd
                             sizes (random-number and data-loader state) ride along

All values a call writes come back whole: tables as their integer and their sum-of-squares columns, and the transfer buffer and
the restored state as integers.  Each is a function of the state's bytes alone (sums are taken in an order fixed by
position in the chunk, as replicas compare them bit for bit), so they are compared exactly.
"""
import math

import numpy as np
import torch

from paper_2509_03047_gb300 import flashrec as fr
from paper_2509_03047_gb300 import shards

KiB, MiB = 1 << 10, 1 << 20
F32, BF16, U8 = torch.float32, torch.bfloat16, torch.uint8


def listed():
    return [
        # A unit test's or a smoke run's model, three NaNs in it: latency and launches.
        dict(name="tiny_fingerprint", op="fingerprint", layout="model", hidden=128, ffn=512, layers=4, vocab=2048,
             chunk=64 * KiB, nonfinite=3),
        dict(name="tiny_step", op="step", layout="model", hidden=128, ffn=512, layers=4, vocab=2048, chunk=64 * KiB,
             nonfinite=3),
        # A small language model on an agent inside the training process, where no device memory is free.
        dict(name="small_static", op="static", layout="model", hidden=512, ffn=2048, layers=8, vocab=32000, chunk=1 * MiB,
             nonfinite=0),
        # The 124M-parameter GPT-2 shapes of the benchmark: each direction by itself.
        dict(name="gpt2s_fingerprint", op="fingerprint", layout="model", hidden=768, ffn=3072, layers=12, vocab=50257,
             chunk=1 * MiB, nonfinite=0),
        dict(name="gpt2s_pack", op="pack", layout="model", hidden=768, ffn=3072, layers=12, vocab=50257, chunk=1 * MiB,
             nonfinite=0),
        dict(name="gpt2s_unpack", op="unpack", layout="model", hidden=768, ffn=3072, layers=12, vocab=50257,
             chunk=1 * MiB, nonfinite=0, flips=10),
        # The same state through pinned host memory, one re-send round allowed: the two-way host link bounds it.
        dict(name="gpt2s_restore_pinned", op="restore", layout="model", hidden=768, ffn=3072, layers=12, vocab=50257,
             chunk=1 * MiB, nonfinite=0, batches=16, pinned=True),
        # A fragmented optimizer partition: 50,000 tensors from 1 KiB to 512 KiB, a few Inf and NaN.
        dict(name="fragments_fingerprint", op="fingerprint", layout="fragments", tensors=50000, lo=1 * KiB, hi=512 * KiB,
             sizes_seed=0, chunk=256 * KiB, nonfinite=106),
        dict(name="fragments_step", op="step", layout="fragments", tensors=50000, lo=1 * KiB, hi=512 * KiB, sizes_seed=0,
             chunk=256 * KiB, nonfinite=106),
        # Flat groups whose parameters have odd sizes: 2- and 4-byte aligned views, all three sweeps.
        dict(name="flat_step", op="step", layout="flat", tensors=400, lo=1001, hi=4000003, sizes_seed=1, chunk=1 * MiB,
             nonfinite=0),
        # One rank of four rebuilt from three replicas' shards of 100 million parameters (350 MB), through the public helper.
        dict(name="reshard_4_from_3", op="reshard", elems=100000007, n_dst=4, rank=1, n_src=3, chunk=1 * MiB, batches=8),
        # A tensor-parallel rank of an 8B-parameter Llama (14 GB): the largest.
        dict(name="llama8b_tp8_step", op="step", layout="model", hidden=4096, ffn=14336, layers=32, vocab=128256, tp=8,
             chunk=4 * MiB, nonfinite=0),
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    """Another call on another state: 2 MB to 6 GB, chunks of 16 KiB to 16 MiB, at most 50,000 tensors and 150,000 chunks."""
    op = rng.choice(["fingerprint", "pack", "unpack", "step", "step", "restore", "static", "reshard"])
    chunk = rng.choice([16, 32, 64, 128, 256, 512, 1024, 2048, 4096, 16384]) * KiB
    if rng.random() < 0.15:  # a chunk size of the caller's own, a multiple of 4 only
        chunk = chunk // 2 + 4 * rng.randrange(1, chunk // 8)
    # the static call's limits: 16,384 chunks, 2 GiB in 16 KiB segments
    total = _log(rng, 2 << 20, min(1500 << 20 if op == "static" else 6 << 30, chunk * (8000 if op == "static" else 100000)))
    if op == "reshard":
        n_dst, n_src = rng.randrange(2, 17), rng.randrange(1, 17)
        return dict(op=op, elems=min(total // 14 * n_dst, 400000000) + rng.randrange(16), n_dst=n_dst,
                    rank=rng.randrange(n_dst), n_src=n_src, chunk=chunk, batches=rng.choice([1, 2, 5, 8, 16]))
    case = dict(op=op, chunk=chunk, nonfinite=rng.choice([0, 0, 3, 50]))
    if op == "unpack":
        case.update(flips=rng.choice([0, 1, 10, 100]))
    if op == "restore":
        case.update(batches=rng.choice([2, 4, 8, 16]), pinned=rng.random() < 0.5)
    layout = rng.choice(["model", "fragments", "flat"])
    case.update(layout=layout)
    if layout == "model":
        hidden = 8 * _log(rng, 8, 256)
        layers = max(1, min(48, total // (14 * 14 * hidden * hidden)))
        vocab = max(64, min(128256, (total // 14 - 12 * layers * hidden * hidden) // hidden))
        return dict(case, hidden=hidden, ffn=4 * hidden, layers=layers, vocab=vocab)
    hi = min(_log(rng, 4 * KiB, 16 * MiB), max(4 * KiB, total // 8))
    lo = rng.choice([4, 512, 1 * KiB])
    mean = (hi - lo) / math.log(hi / lo)
    unit = mean if layout == "fragments" else 14 * mean / 4  # flat: lo and hi count fp32 bytes of one buffer
    tensors = int(max(3, min(total / unit, 50000 if layout == "fragments" else 10000)))
    if op == "static":
        tensors = min(tensors, 1800)
    if layout == "flat":
        lo, hi = max(1, lo // 4), hi // 4
    return dict(case, tensors=tensors, lo=lo, hi=hi, sizes_seed=rng.randrange(1 << 30))


# ---------------------------------------------------------------- the state's layout, from the case alone


def _model_params(case):
    """Elements of every parameter of a decoder: an embedding, per layer a fused QKV (or a tensor-parallel rank's q, k, v), the
    output projection, the MLP and two norms, and a final norm."""
    h, f, layers, vocab, tp = case["hidden"], case["ffn"], case["layers"], case["vocab"], case.get("tp", 1)
    if tp > 1:  # gated MLP, grouped queries with one key-value head of 128 per rank, untied head
        layer = [h, h // tp * h, 128 * h, 128 * h, h * (h // tp), h, f // tp * h, f // tp * h, h * (f // tp)]
        return [vocab // tp * h] + layer * layers + [h, vocab // tp * h]
    layer = [h, h, 3 * h * h, 3 * h, h * h, h, h, h, h * f, f, f * h, h]
    return [vocab * h] + layer * layers + [h, h]


def _spread_sizes(case):
    r = np.random.default_rng(case["sizes_seed"])
    a, b = math.log(case["lo"]), math.log(case["hi"])
    return np.exp(a + r.random(case["tensors"]) * (b - a)).astype(np.int64)


def _spans(case):
    """([(dtype, byte offset, bytes)] in plan order, bytes of the one buffer that holds them all)."""
    spans, at = [], 0
    if case["layout"] == "model":
        for n in _model_params(case):
            for dtype, eb in ((BF16, 2), (F32, 4), (F32, 4), (F32, 4)):
                spans.append((dtype, at, eb * n))
                at += -(-eb * n // 512) * 512
        return spans, at
    if case["layout"] == "fragments":
        for n in np.maximum(4, _spread_sizes(case) // 4 * 4).tolist():
            spans.append((F32, at, n))
            at += -(-n // 512) * 512
        return spans, at
    sizes = np.maximum(1, _spread_sizes(case)).tolist()
    starts = np.concatenate([[0], np.cumsum(sizes)]).tolist()
    base = []
    for eb in (2, 4, 4, 4):
        base.append(at)
        at += -(-eb * starts[-1] // 512) * 512
    for i, n in enumerate(sizes):
        for b, (dtype, eb) in zip(base, ((BF16, 2), (F32, 4), (F32, 4), (F32, 4))):
            spans.append((dtype, b + eb * starts[i], eb * n))
    for n in (5000, 33, 2500001):  # random-number, counter and data-loader state
        spans.append((U8, at, n))
        at += n
    return spans, -(-at // 512) * 512


def _shard(case):
    q = -(-case["elems"] // case["n_dst"])
    return max(0, min(case["elems"], (case["rank"] + 1) * q) - case["rank"] * q)


# ---------------------------------------------------------------- inputs


def _views(flat, spans):
    typed = {t: flat.view(t) for t in (F32, BF16, U8)}
    return [typed[t][at // t.itemsize:(at + n) // t.itemsize] for t, at, n in spans]


def _adam_values(n, gen):
    """Weight, master, first and second moment of n parameters, as early training has them."""
    master = torch.randn(n, generator=gen, device="cuda") * 0.02
    weight = master.to(BF16)
    m = torch.randn(n, generator=gen, device="cuda") * 1e-3
    v = (torch.randn(n, generator=gen, device="cuda") * 1e-3).square_()
    return weight, weight.float(), m, v


def _fill(case, flat, spans, views, gen):
    if case["layout"] == "model":
        for i in range(0, len(views), 4):
            for view, values in zip(views[i:i + 4], _adam_values(views[i].numel(), gen)):
                view.copy_(values)
    elif case["layout"] == "fragments":
        flat.view(F32).normal_(generator=gen)
    else:
        groups = len(views) - 3
        n = sum(v.numel() for v in views[0:groups:4])
        for k, values in enumerate(_adam_values(n, gen)):
            t, at = spans[k][0], spans[k][1]
            flat.view(t)[at // t.itemsize:at // t.itemsize + n] = values
        for v in views[groups:]:
            v.random_(0, 256, generator=gen)
    if case["nonfinite"]:
        f32 = [v for v in views if v.dtype == F32]
        where = torch.randint(0, 1 << 62, (2, case["nonfinite"]), generator=gen, device="cuda").tolist()
        for k, (i, j) in enumerate(zip(*where)):
            v = f32[i % len(f32)]
            v[j % v.numel()] = (math.nan, math.inf, -math.inf)[k % 3]


class _State:
    """What a program has in hand before the call: buffers, plans and, where it keeps them, streams."""


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = _State()
    s.case, s.op = case, case["op"]
    if s.op == "reshard":
        n, n_dst, rank, n_src = case["elems"], case["n_dst"], case["rank"], case["n_src"]
        full = _adam_values(n, gen)
        s.sources = [shards.make_shards(full, n_src, j) for j in range(n_src)]
        del full
        k = _shard(case)
        s.dst = [torch.zeros(k, dtype=t, device="cuda") for t in (BF16, F32, F32, F32)]
        return s
    spans, nbytes = _spans(case)
    s.flat = torch.zeros(nbytes, dtype=U8, device="cuda")
    s.views = _views(s.flat, spans)
    _fill(case, s.flat, spans, s.views, gen)
    batches = case.get("batches", 1)
    if s.op == "static":
        chunks = sum(-(-n // case["chunk"]) for _, _, n in spans)
        s.table = torch.zeros(16 * chunks, dtype=U8, device="cuda")
        return s
    s.plan = fr.Plan(s.views, case["chunk"], n_batches=batches)
    s.table = s.plan.new_table()
    if s.op != "fingerprint":
        s.packed = s.plan.new_packed(pinned=case.get("pinned", False))
    if s.op in ("unpack", "step", "restore"):
        s.out = torch.zeros(nbytes, dtype=U8, device="cuda")
        s.out_plan = fr.Plan(_views(s.out, spans), case["chunk"], n_batches=batches)
        s.out_table = s.out_plan.new_table()
        s.failing = torch.zeros(s.plan.n_chunks, dtype=torch.int32, device="cuda")
        s.n_failing = torch.zeros(1, dtype=torch.int64, device="cuda")
        s.diverged, s.n_diverged = torch.zeros_like(s.failing), torch.zeros_like(s.n_failing)
    if s.op == "unpack":
        s.plan.pack(s.packed)
        at = torch.randint(0, s.packed.numel(), (case["flips"],), generator=gen, device="cuda").unique()
        s.packed[at] = s.packed[at] ^ 4
    if s.op == "restore":
        s.streams = torch.cuda.Stream(), torch.cuda.Stream()
    return s


# ---------------------------------------------------------------- the call


def _columns(table):
    """A fingerprint table's two integer columns and its sums of squares."""
    return table.view(torch.int32).view(-1, 4)[:, :2], table.view(torch.float64).view(-1, 2)[:, 1]


def run(s):
    if s.op == "fingerprint":
        fr.fr_fingerprint(s.plan.handle, s.table)
        return {"table": _columns(s.table)}
    if s.op == "static":
        fr.fr_fingerprint_static(s.views, s.case["chunk"], s.table)
        return {"table": _columns(s.table)}
    if s.op == "pack":
        fr.fr_pack(s.plan.handle, s.packed)
        return {"packed": s.packed.view(torch.int64)}
    if s.op == "unpack":
        fr.fr_unpack_verify(s.out_plan.handle, s.packed, s.failing, s.n_failing)
        return {"state": s.out.view(torch.int64), "failing": s.failing, "n_failing": s.n_failing}
    if s.op == "reshard":
        c = s.case
        left, diverged, _ = shards.restore_shard([c["elems"]] * 4, s.dst, c["n_dst"], c["rank"], s.sources, c["n_src"],
                                                 c["chunk"], n_batches=c["batches"])
        bits = [t.view(torch.int16 if t.dtype == BF16 else torch.int32) for t in s.dst]
        return {"state": bits, "n_failing": left, "n_diverged": diverged.numel()}
    if s.op == "step":
        fr.fr_pack_fp(s.plan.handle, s.packed, s.table)
        fr.fr_unpack_verify_fp(s.out_plan.handle, s.packed, s.failing, s.n_failing, s.out_table)
        fr.fr_diff(s.table, s.out_table, s.plan.n_chunks, s.diverged, s.n_diverged)
    else:
        sender, receiver = s.streams
        current = torch.cuda.current_stream()
        sender.wait_stream(current)
        receiver.wait_stream(current)
        fr.fr_restore_fp(s.plan.handle, s.out_plan.handle, s.packed, 1, s.failing, s.n_failing, s.table, s.out_table,
                         sender, receiver)
        fr.fr_diff(s.table, s.out_table, s.plan.n_chunks, s.diverged, s.n_diverged, receiver)
        current.wait_stream(receiver)
    return {"table": _columns(s.table), "restored_table": _columns(s.out_table), "packed": s.packed.view(torch.int64),
            "state": s.out.view(torch.int64), "failing": s.failing, "n_failing": s.n_failing, "diverged": s.diverged,
            "n_diverged": s.n_diverged}


# ---------------------------------------------------------------- what it cannot do without


def work(case):
    if case["op"] == "reshard":  # into the transfer buffer and out of it again
        k, pieces = _shard(case), 4 * min(case["n_src"], 1 + -(-case["n_src"] // case["n_dst"]))
        chunks = pieces + 14 * k // case["chunk"]
        return {"bytes": 4 * 14 * k + 128 * chunks, "flops": 4 * 4 * k}
    spans, _ = _spans(case)
    state = sum(n for _, _, n in spans)
    chunks = sum(-(-n // case["chunk"]) for _, _, n in spans)
    elems = sum(n // t.itemsize for t, _, n in spans if t != U8)
    if case["op"] in ("fingerprint", "static"):
        return {"bytes": state + 16 * chunks, "flops": 2 * elems}
    if case["op"] == "pack":
        return {"bytes": 2 * state + 64 * chunks, "flops": 2 * elems}
    if case["op"] == "unpack":
        return {"bytes": 2 * state + 64 * chunks, "flops": 0}
    return {"bytes": 4 * state + (128 + 64) * chunks, "flops": 4 * elems}


def tolerance(case):
    return "exact"


def exact(case, seed):
    """The tables' sums of squares in 64 bits; the other outputs are bytes, counts and checksums."""
    if case["op"] in ("pack", "unpack", "reshard"):
        return None
    gen = torch.Generator(device="cuda").manual_seed(seed)
    spans, nbytes = _spans(case)
    flat = torch.zeros(nbytes, dtype=U8, device="cuda")
    views = _views(flat, spans)
    _fill(case, flat, spans, views, gen)
    sums = []
    for v in views:
        if v.dtype == U8:
            sums.append(torch.zeros(-(-v.numel() // case["chunk"]), dtype=torch.float64, device="cuda"))
            continue
        per = case["chunk"] // v.itemsize
        for a in range(0, v.numel(), 64 * per):  # 64 chunks at a time
            x = v[a:a + 64 * per].double()
            x = x.masked_fill_(~x.isfinite(), 0.0).square_()
            whole = x.numel() // per
            if whole:
                sums.append(x[:whole * per].view(whole, per).sum(1))
            if x.numel() % per:
                sums.append(x[whole * per:].sum().view(1))
    table = None, torch.cat(sums)
    if case["op"] in ("fingerprint", "static"):
        return {"table": table}
    return {"table": table, "restored_table": table, "packed": None, "state": None, "failing": None, "n_failing": None,
            "diverged": None, "n_diverged": None}
