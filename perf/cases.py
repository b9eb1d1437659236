"""The work that a user of the chunk-dedup library has it do, as cases that can be timed.

A case is an upload: payloads (the host-to-device copies of a program that loads
weights) that a cache has seen none, some or all of before.  prepare() makes
the bytes, the cache in the state that the upload meets, and the outputs;
run() makes the upload through the public entry points once.  An upload that
changes the cache starts from a snapshot of it, so that every pass meets the
same cache; outputs are compared bit for bit.

Fields of a case:
  how      "calls"  one gleam_dedup_copy_async per payload
           "slots"  one gleam_dedup_copy_batch per payload, for the slots of its chunks (what
                    gleam_block_check takes when the block is freed)
           "batch"  one gleam_dedup_copy_batch
           "host"   one gleam_dedup_copy_host_batch, payloads left in page-locked memory
  seen     "new"     no chunk is cached (a first load; the cache holds other chunks
                     unless `prefill` is 0)
           "again"   every chunk is cached, behind a few others (the same model loaded again)
           "variant" the model is cached, and `share` of its chunks carry one flipped
                     bit (a fine-tuned variant of it)
           "half"    half of the full chunks are cached
           "repeats" a quarter zero chunks, a quarter copies of 16 patterns, half new
           "swap"    three variants take turns in a GLEAM_EVICT_LRU cache that holds
                     two, so that each upload evicts the oldest one's own chunks
  chunk    chunk size of the cache
  sizes    "layers": `count` Llama-3-8B decoder layers, 9 bf16 tensors each;
           "gpt2": GPT-2 small, 148 fp32 tensors; "log": `count` payloads, log-uniform
           in [lo, hi] bytes; "one": one payload of `lo` bytes
  align    payload k starts at a multiple of this (256: an allocation each; 8: tensors
           back to back in one checkpoint blob, behind its 8-byte length word)
  overlap  GLEAM_OVERLAP_CALLS
"""
import math

import torch

from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300 import workloads as W
from paper_2607_23115_gb300.cache import Cache, DedupOutputs

KiB, MiB = 1024, 1 << 20
DEV = "cuda"
SWAPPED = 3  # variants that take turns


def _case(how, seen, chunk, sizes, **more):
    c = dict(how=how, seen=seen, chunk=chunk, sizes=sizes, count=1, lo=0, hi=0, align=256,
             overlap=False, prefill=0, share=0.0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest thing an interposer sees: a bias vector copied again; a launch and a
        # few round trips
        _case("slots", "again", 4 * KiB, "one", lo=6000, name="call_6kb_again"),
        # an application's own mix of small copies, none seen before
        _case("calls", "new", 4 * KiB, "log", count=48, lo=4 * KiB, hi=MiB,
              prefill=16 * MiB, name="stream_4kb_1mb_new"),
        # a fine-tuned decoder layer, intercepted one tensor at a time
        _case("calls", "variant", 64 * KiB, "layers", share=0.10, name="layer_calls_variant"),
        # the same from a server that lets consecutive calls overlap
        _case("calls", "variant", 64 * KiB, "layers", share=0.10, overlap=True, name="layer_calls_overlap"),
        # four layers of the fine-tuned model handed over at once; the largest
        _case("batch", "variant", 64 * KiB, "layers", count=4, share=0.10, name="layers4_batch_variant"),
        # the first load of a small model into an empty cache, then a later load of it
        _case("batch", "new", 4 * KiB, "gpt2", name="gpt2_batch_new"),
        _case("batch", "again", 4 * KiB, "gpt2", name="gpt2_batch_again"),
        # one mid-sized fp16 buffer, half of it known
        _case("calls", "half", 4 * KiB, "one", lo=64 * MiB, name="one_64mb_half"),
        # zero-padded and tied tensors: many equal chunks inside one payload, fine chunks
        _case("calls", "repeats", KiB, "one", lo=256 * MiB, name="one_256mb_repeats"),
        # tensors back to back in a checkpoint blob on the device: 8-byte alignment, ragged ends
        _case("batch", "variant", 16 * KiB, "log", count=40, lo=64 * KiB,
              hi=32 * MiB, align=8, share=0.10, name="blob_batch_variant"),
        # models taking turns in a cache too small for all of them
        _case("batch", "swap", 64 * KiB, "layers", share=0.10, name="layer_batch_swap"),
        # the sender's order: decide what to send while the tensors are still in host memory
        _case("host", "variant", 64 * KiB, "log", count=12, lo=256 * KiB,
              hi=32 * MiB, share=0.10, name="host_batch_variant"),
    ]


def draw(rng):
    how = rng.choice(["calls", "calls", "batch", "batch", "host"])
    seen = rng.choice(["new", "again", "variant", "half", "repeats", "swap"])
    if seen == "swap" and how == "host":
        seen = "variant"
    if seen == "again" and how == "calls":
        how = "slots"
    chunk = rng.choice([1, 4, 16, 64]) * KiB
    top = {"calls": 384 * MiB, "slots": 384 * MiB, "batch": 512 * MiB, "host": 96 * MiB}[how]
    if seen == "swap":
        top //= 2
    total = int(math.exp(rng.uniform(math.log(64 * KiB), math.log(top))))
    if seen == "repeats":
        n = max(1, total // chunk) * chunk
        return _case(how, seen, chunk, "one", lo=n)
    count = int(math.exp(rng.uniform(0, math.log(56))))
    if count == 1:
        shape = dict(sizes="one", lo=total)
    else:  # log-uniform in [hi / 64, hi] has a mean of about hi / 4.2
        hi = max(8 * KiB, int(min(total, 4.2 * total / count)))
        shape = dict(sizes="log", count=count, lo=max(KiB, hi // 64), hi=hi)
    return _case(how, seen, chunk, align=rng.choice([256, 256, 8]),
                 overlap=how in ("calls", "slots") and seen != "swap" and rng.random() < 0.5,
                 prefill=16 * MiB if seen == "new" and rng.random() < 0.5 else 0,
                 share=rng.choice([0.02, 0.10, 0.3]) if seen in ("variant", "swap") else 0.0, **shape)


# ---------------------------------------------------------------------------
# the payloads: sizes (the same for every seed), places in one blob, chunks
# ---------------------------------------------------------------------------

def _sizes(case):
    chunk = case["chunk"]
    if case["sizes"] == "layers":
        return [2 * math.prod(s) for _, s in W.llama3_8b_shapes()[1:1 + 9 * case["count"]]]
    if case["sizes"] == "gpt2":
        return [4 * math.prod(s) for _, s in W.gpt2_small_shapes()]
    if case["sizes"] == "one":
        sizes = [case["lo"]]
    else:
        sizes = W.loguniform_sizes(case["count"], case["lo"], case["hi"])
    # a last chunk of a few bytes could equal another by chance: at least 64 bytes
    return [s if s % chunk == 0 or s % chunk >= 64 else s + 64 for s in sizes]


def _layout(case):
    """(sizes, offsets, bytes of the blob, per payload (first chunk, chunks))."""
    sizes = _sizes(case)
    offs, pos = [], 0 if case["align"] >= 16 else 8
    for s in sizes:
        offs.append(pos)
        pos += -(-s // case["align"]) * case["align"]
    spans, n = [], 0
    for s in sizes:
        spans.append((n, -(-s // case["chunk"])))
        n += spans[-1][1]
    return sizes, offs, pos + 64, spans


def _full(case):
    """Per payload, the chunks that a miss or hit may be drawn from: whole ones, unless it has none."""
    sizes, _, _, spans = _layout(case)
    return [z // case["chunk"] or m for z, (_, m) in zip(sizes, spans)]


def _changed(case):
    """Per payload, how many chunks a variant changes: `share` of all, spread evenly; at least one."""
    got, at, done = [], 0.0, 0
    for f in _full(case):
        at += case["share"] * f
        got.append(min(f, int(at) - done))
        done += got[-1]
    if not done:
        got[0] = 1
    return got


def _misses(case):
    """(chunks of the upload, how many of them miss); the same for every seed."""
    _, _, _, spans = _layout(case)
    n = spans[-1][0] + spans[-1][1]
    if case["seen"] == "new":
        return n, n
    if case["seen"] == "again":
        return n, 0
    if case["seen"] in ("variant", "swap"):
        return n, sum(_changed(case))
    if case["seen"] == "half":
        return n, n - sum(f // 2 for f in _full(case))
    q = n // 4
    return n, n - 2 * q + min(1, q) + min(16, q)  # the first zero chunk, of each pattern, and the rest


def work(case):
    """Every payload byte read, the cached copy of every hit on the cache read (each hit is
    confirmed byte for byte), every missed byte written to the packed output and to the arena."""
    total = sum(_layout(case)[0])
    n, miss = _misses(case)
    missed = miss / n
    hit = 0.0 if case["seen"] == "repeats" else 1 - missed  # there, hits repeat the payload's own bytes
    return {"bytes": total * (1 + hit + 2 * missed), "flops": 0}


def tolerance(case):
    return "exact"  # masks, indices, counts, slots and bytes


# ---------------------------------------------------------------------------
# state
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _weights(nbytes, g):
    """Weight-like bytes: bf16 values ~N(0, 0.02)."""
    out = torch.empty(-(-nbytes // 2), dtype=torch.bfloat16, device=DEV)
    step = 1 << 27
    for k in range(0, out.numel(), step):
        m = min(step, out.numel() - k)
        out[k:k + m] = torch.randn(m, generator=g, device=DEV).mul_(0.02)
    return out.view(torch.uint8)[:nbytes]


def _flip(blob, starts, lens, g):
    """One bit of each of these chunks."""
    r = torch.rand(starts.numel(), generator=g, device=DEV, dtype=torch.float64)
    bit = (r * (lens * 8)).long().clamp_(max=lens * 8 - 1)
    at = starts + bit // 8
    blob[at] = blob[at] ^ (torch.ones_like(bit) << (bit % 8)).to(torch.uint8)


class _State:
    pass


def prepare(case, seed):
    C, g = case["chunk"], _gen(seed)
    sizes, offs, blob_bytes, spans = _layout(case)
    n = spans[-1][0] + spans[-1][1]
    starts = torch.cat([torch.arange(k, dtype=torch.int64, device=DEV) * C + o for o, (_, k) in zip(offs, spans)])
    ends = torch.cat([torch.full((k,), o + s, dtype=torch.int64, device=DEV) for o, s, (_, k) in zip(offs, sizes, spans)])
    lens = torch.minimum(ends - starts, torch.tensor(C, device=DEV))
    s = _State()
    s.case, s.turn = case, 0
    blob = _weights(blob_bytes, g)
    miss = torch.zeros(n, dtype=torch.bool, device=DEV)
    flags, fill, slots = 0, [], n + 64

    def pick(counts):  # so many chunks of each payload, at random
        return torch.cat([first + torch.randperm(f, generator=g, device=DEV)[:k]
                          for (first, _), f, k in zip(spans, _full(case), counts)])

    if case["overlap"]:
        flags |= B.GLEAM_OVERLAP_CALLS
    blobs = [blob]
    if case["seen"] == "new":
        miss[:] = True
        if case["prefill"]:
            fill = [_weights(case["prefill"], g)]
            slots += case["prefill"] // C
    elif case["seen"] == "again":
        others = 1 + int(torch.randint(0, 32, (1,), generator=g, device=DEV))
        fill = [_weights(others * C, g), blob]
    elif case["seen"] in ("variant", "swap"):
        picked = pick(_changed(case))
        k = picked.numel()
        miss[picked] = True
        if case["seen"] == "variant":
            fill = [blob.clone()]
            _flip(blob, starts[picked], lens[picked], g)
            slots += k
        else:
            flags |= B.GLEAM_EVICT_LRU
            blobs = [blob] + [blob.clone() for _ in range(SWAPPED - 1)]
            for at, b in enumerate(blobs):  # a byte of each chunk's own, so that no two are equal
                pos = starts[picked] + (lens[picked] * (2 * at + 1)) // (2 * SWAPPED)
                b[pos] = b[pos] ^ 0x55
            fill = blobs[1:]
            slots = n + k
    elif case["seen"] == "half":
        picked = pick([f // 2 for f in _full(case)])  # whole chunks: a payload of one has none
        miss[:] = True
        miss[picked] = False
        if picked.numel():  # gathered 16 MiB at a time
            at = torch.arange(C, device=DEV)
            fill = [torch.cat([blob[starts[p].unsqueeze(1) + at].flatten()
                               for p in picked.split(max(1, (16 * MiB) // C))])]
    else:  # repeats: one payload of whole chunks
        q = n // 4
        rows = blob[offs[0]:offs[0] + n * C].view(n, C)
        order = torch.randperm(n, generator=g, device=DEV)
        zero, tied = order[:q], order[q:2 * q]
        which = torch.randint(0, 16, (q,), generator=g, device=DEV)
        which[:min(16, q)] = torch.arange(min(16, q), device=DEV)
        rows[zero] = 0
        rows[tied] = _weights(16 * C, g).view(16, C)[which]
        miss[order[2 * q:]] = True
        if q:
            miss[zero.min()] = True
            for k in range(min(16, q)):
                miss[tied[which == k].min()] = True
    # the cache as the upload meets it
    s.cache = Cache(slots * C, C, flags)
    s.cache.reserve(n)

    def payloads(b):
        return [b[o:o + z] for o, z in zip(offs, sizes)]

    for f in fill:
        if f.numel() == blob_bytes:
            ps = payloads(f)
            outs = [DedupOutputs.alloc(p.numel(), C, DEV) for p in ps]
            s.cache.dedup_batch(ps, outs)
        else:
            s.cache.dedup(f)
    torch.cuda.synchronize()
    # outputs, each kind in one buffer; bytes past a payload's last miss are unspecified, so
    # the packed bytes are returned per payload up to there (or whole where all miss)
    words = [(k + 31) // 32 for _, k in spans]
    s.mask = torch.zeros(sum(words), dtype=torch.int32, device=DEV)
    s.idx = torch.zeros(n, dtype=torch.int32, device=DEV)
    s.slots = torch.zeros(n, dtype=torch.int32, device=DEV)
    s.results = torch.zeros((len(sizes), B.RESULT_WORDS), dtype=torch.int64, device=DEV)
    poffs, ppos = W.layout(sizes)
    packed = torch.zeros(ppos, dtype=torch.uint8, device=DEV)
    s.outs, s.res, slot_views, w = [], [], [], 0
    for k, (z, (first, m)) in enumerate(zip(sizes, spans)):
        s.outs.append(DedupOutputs(s.mask[w:w + words[k]], s.idx[first:first + m], packed[poffs[k]:poffs[k] + z]))
        s.res.append(s.results[k])
        slot_views.append(s.slots[first:first + m])
        w += words[k]
    missed = torch.where(miss, lens, torch.zeros_like(lens)).cumsum(0).cpu()
    ends_at = [int(missed[f + m - 1]) for f, m in spans]
    got = [e - b for e, b in zip(ends_at, [0] + ends_at[:-1])]
    if got == sizes:
        s.packed = [packed]
    else:
        s.packed = [o.miss_bytes[:b] for o, b in zip(s.outs, got) if b]
    # the arguments that a program keeps for its calls
    if case["how"] == "host":
        blobs = [b.cpu().pin_memory() for b in blobs]
    s.bufs = [payloads(b) for b in blobs]
    s.items = None
    if case["how"] == "slots":
        s.items = [[Cache.batch_items([p], [o], [r], [v]) for p, o, r, v in zip(b, s.outs, s.res, slot_views)]
                   for b in s.bufs]
    elif case["how"] != "calls":
        s.items = [Cache.batch_items(b, s.outs, s.res, slot_views) for b in s.bufs]
    s.total = torch.zeros(B.RESULT_WORDS, dtype=torch.int64, device=DEV)
    s.snap = s.cache.snapshot() if case["seen"] in ("new", "variant", "half", "repeats") else None
    return s


def run(s):
    turn, s.turn = s.turn, (s.turn + 1) % len(s.bufs)
    if s.snap is not None:
        s.cache.restore(s.snap)
    how = s.case["how"]
    if how == "calls":
        for buf, out, res in zip(s.bufs[turn], s.outs, s.res):
            s.cache.dedup_async(buf, out, res)
        return {"mask": s.mask, "idx": s.idx, "results": s.results, "packed": s.packed}
    if how == "slots":
        for item in s.items[turn]:
            s.cache.dedup_batch(None, items=item)
    elif how == "batch":
        s.cache.dedup_batch(None, total=s.total, items=s.items[turn])
    else:
        s.cache.dedup_host_batch(total=s.total, items=s.items[turn])
    return {"mask": s.mask, "idx": s.idx, "slots": s.slots, "results": s.results, "total": s.total,
            "packed": s.packed}
