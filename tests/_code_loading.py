"""Run by itself (python -m tests._code_loading), so that no kernel has run before:
makes caches, then the calls of many routes, each beside a kernel that runs on
another stream, and prints the calls that ended only after that kernel, which is
what a call does that loads device code."""
import torch

from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300 import workloads as W
from paper_2607_23115_gb300.cache import Cache, DedupOutputs, fingerprint
from tests import _native

DEV = torch.device("cuda:0")
KiB = 1024
HOLD_NS = 60_000_000


class Route:
    def __init__(self, name, how, C, nch, flags=0, offset=0, spec=0, small=None):
        self.name, self.how, self.C, self.n = name, how, C, nch * C
        host = W.random_bytes(self.n + offset, seed=nch + C)
        self.buf = (host.pin_memory() if how == "host" else host.to(DEV))[offset:]
        self.gc = Cache(2 * self.n + 64 * C, C, flags)
        self.gc.debug_set(B.GLEAM_DEBUG_SPECULATE, spec)
        if small is not None:
            self.gc.debug_set(B.GLEAM_DEBUG_SMALL_CALLS, small)
        self.gc.reserve(nch)
        self.out = DedupOutputs.alloc(self.n, C, DEV)
        self.res = torch.zeros(B.RESULT_WORDS, dtype=torch.int64, device=DEV)
        self.words = torch.zeros(nch, dtype=torch.int64, device=DEV)
        self.slots = torch.zeros(nch, dtype=torch.int32, device=DEV)
        self.offs = torch.arange(nch, dtype=torch.int64, device=DEV) * C
        self.count = torch.zeros(1, dtype=torch.int64, device=DEV)

    def call(self, stream):
        if self.how == "async":
            self.gc.dedup_async(self.buf, self.out, self.res, stream)
        elif self.how == "host":
            self.gc.dedup_host(self.buf, self.out, self.res, stream)
        elif self.how == "noalloc":
            rc = B.gleam_dedup_copy_noalloc(self.gc.handle, self.buf, self.n, self.out.hit_mask,
                                            self.out.miss_idx, self.out.miss_bytes, self.res, stream)
            assert rc == 0, rc
        elif self.how == "fingerprint":
            fingerprint(self.buf, self.C, self.words, stream)
        else:
            self.gc.block_check(self.buf, self.offs, self.slots, count=self.count, stream=stream)


def main():
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    routes = [
        Route("few large chunks", "async", 64 * KiB, 100),
        Route("few large chunks, 5 to a block", "async", 16 * KiB, 1500),
        Route("few large chunks, 8 to a block", "async", 4 * KiB, 2400),
        Route("one-launch resolve", "async", 4 * KiB, 4000),
        Route("the same, no write-through", "async", 4 * KiB, 4000, spec=2),
        Route("unaligned", "async", 4 * KiB, 4000, offset=8),
        Route("unaligned, large chunks", "async", 32 * KiB, 2500, offset=8),
        Route("big stages", "async", 32 * KiB, 2500),
        Route("big stages, no write-through", "async", 32 * KiB, 2500, spec=2),
        Route("k_dedup and k_pack", "async", KiB, 20000),
        Route("small call", "async", KiB, 20),
        Route("small call, no write-through", "async", KiB, 20, spec=2),
        Route("small call, unaligned", "async", KiB, 20, offset=8),
        Route("small call, large chunks", "async", 32 * KiB, 4, small=64),
        Route("small call, large chunks, unaligned", "async", 32 * KiB, 4, small=64, offset=8),
        Route("LRU", "async", 4 * KiB, 300, B.GLEAM_EVICT_LRU),
        Route("KEY16", "async", 4 * KiB, 300, B.GLEAM_KEY16),
        Route("paper identifiers", "async", 4 * KiB, 300, B.GLEAM_PAPER_IDS),
        Route("paper identifiers, unaligned", "async", 4 * KiB, 300, B.GLEAM_PAPER_IDS, offset=8),
        Route("checked", "async", KiB, 300, B.GLEAM_DEBUG_CHECKS),
        Route("overlapping", "async", 64 * KiB, 100, B.GLEAM_OVERLAP_CALLS),
        Route("host payload", "host", 4 * KiB, 300),
        Route("allocation-free", "noalloc", 4 * KiB, 5000),
        Route("allocation-free, unaligned", "noalloc", KiB, 5000, offset=4),
        Route("fingerprint", "fingerprint", KiB, 5000),
        Route("fingerprint, unaligned", "fingerprint", KiB, 5000, offset=4),
        Route("fingerprint, large chunks", "fingerprint", 64 * KiB, 100),
        Route("fingerprint, 1,500 chunks", "fingerprint", 16 * KiB, 1500),
        Route("fingerprint, 2,400 chunks", "fingerprint", 4 * KiB, 2400),
        Route("block check", "check", 4 * KiB, 300),
    ]
    for _ in range(2):  # the helper's own kernel
        _native.hold(KiB, 1000, other)
        torch.cuda.synchronize()
    late = []
    for r in routes:
        for k in range(2):  # all new, all cached
            torch.cuda.synchronize()
            _native.hold(KiB, HOLD_NS, other)
            held = other.record_event()
            r.call(mine)
            mine.synchronize()
            if held.query():
                late.append("%s, call %d" % (r.name, k))
    torch.cuda.synchronize()
    print("routes %d, late: %s" % (len(routes), "; ".join(late) or "none"))


if __name__ == "__main__":
    main()
