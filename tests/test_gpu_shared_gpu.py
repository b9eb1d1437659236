"""Calls whose kernels do not get the GPU to themselves: another kernel holds
shared memory on every SM, or a second cache's calls run on a second stream.
Payloads of more than about 10 MB with repeated chunks then have blocks of the
one-launch resolve kernel that start after the others are through."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300 import workloads as W
from paper_2607_23115_gb300.cache import Cache, DedupOutputs, result_dict
from tests import _native
from tests._parity import DEV, compare_cache

pytestmark = pytest.mark.gpu
KiB, MiB = 1024, 1 << 20


def _repeating(nch, C, seed, repeats):
    """nch chunks and a ragged tail; `repeats` of the chunks equal earlier ones."""
    host = W.random_bytes(nch * C + 100, seed=seed)
    rows = host[:nch * C].view(nch, C)
    rng = np.random.default_rng(seed)
    to = rng.choice(np.arange(1, nch), repeats, replace=False)
    for k in to:
        rows[int(k)] = rows[int(rng.integers(0, k))]
    return host


class _Side:
    """A cache, its oracle and its calls, enqueued first and checked later."""

    def __init__(self, C, nslots, flags=0):
        self.gc, self.oc = Cache(nslots * C, C, flags), oracle.OracleCache(nslots * C, C)
        self.C, self.calls = C, []

    def add(self, host):
        out = DedupOutputs.alloc(host.numel(), self.C, DEV)
        res = torch.zeros(B.RESULT_WORDS, dtype=torch.int64, device=DEV)
        self.calls.append((host, host.to(DEV), out, res))

    def enqueue(self, k, stream):
        _, buf, out, res = self.calls[k]
        self.gc.dedup_async(buf, out, res, stream)

    def check(self):
        for host, _, out, res in self.calls:
            rc, mask, idx, packed = self.oc.dedup(host.numpy())
            r = result_dict(res)
            assert r["status"] == 0 and r["n_miss"] == rc and r["miss_bytes"] == len(packed)
            assert np.array_equal(out.hit_mask.cpu().numpy().view(np.uint32)[:len(mask)], mask)
            assert np.array_equal(out.miss_idx.cpu().numpy().view(np.uint32)[:rc], idx)
            assert np.array_equal(out.miss_bytes.cpu().numpy()[:len(packed)], packed)
        compare_cache(self.gc, self.oc)


@pytest.mark.parametrize("flags", [0, B.GLEAM_OVERLAP_CALLS])
@pytest.mark.parametrize("nch", [2800, 4096, 9000])
def test_beside_a_kernel_that_leaves_room_for_one_block_per_sm(nch, flags):
    C = 4 * KiB
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    for beside in (False, True):  # first alone: loading device code waits for running kernels
        side = _Side(C, 4 * nch, flags)
        for k, repeats in enumerate((1, nch // 4, 0)):
            side.add(_repeating(nch, C, 10 * nch + k, repeats))
        side.add(side.calls[0][0])
        side.gc.reserve(2 * nch)
        with side.gc:
            torch.cuda.synchronize()
            for k in range(len(side.calls)):
                if beside:
                    _native.hold(130 * KiB, 150_000_000, other)
                    held = other.record_event()
                side.enqueue(k, mine)
                mine.synchronize()
                assert not beside or not held.query(), "did not run beside the other kernel"
                torch.cuda.synchronize()
            side.check()


@pytest.mark.parametrize("flags", [0, B.GLEAM_OVERLAP_CALLS])
def test_two_caches_on_two_streams(flags):
    C = 4 * KiB
    sides = [_Side(C, 40000, flags) for _ in range(2)]
    for k in range(6):
        for s, side in enumerate(sides):
            side.add(_repeating(3000 + 2500 * ((k + s) % 3), C, 100 * s + k, 200 + 100 * k))
    for side in sides:
        side.add(side.calls[0][0])
        side.gc.reserve(10000)
    streams = [torch.cuda.Stream() for _ in sides]
    torch.cuda.synchronize()
    for k in range(7):
        for side, stream in zip(sides, streams):
            side.enqueue(k, stream)
    torch.cuda.synchronize()
    for side in sides:
        side.check()
        side.gc.close()
