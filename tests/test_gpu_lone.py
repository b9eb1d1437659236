"""Calls whose chunks each have a warp of their own (few chunks of at least 4
KiB): chunk counts around a block's and a wave's limits, lengths around the
stages and the rings, one flipped bit at the edges of stages, payloads of any
alignment; outputs and cache against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300 import workloads as W
from paper_2607_23115_gb300.cache import Cache, DedupOutputs, fingerprint
from tests._parity import DEV, compare_cache, dedup_both, to_device

pytestmark = pytest.mark.gpu
KiB = 1024


@pytest.mark.parametrize("offset", [0, 8, 3])
@pytest.mark.parametrize("n", [4096, 4096 + 31, 8 * KiB - 32, 9 * KiB + 16, 64 * KiB + 1, 300001])
def test_whole_buffer_fingerprint(n, offset):
    host = W.random_bytes(n, seed=n)
    d = to_device(host, offset)
    for C in (0, 4096, 4096 + 32, 5 * KiB + 512, 9001):
        got = fingerprint(d, C).cpu().numpy().view(np.uint64)
        assert np.array_equal(got, oracle.fingerprint(host.numpy(), C)), C


@pytest.mark.parametrize("flags", [0, B.GLEAM_KEY16, B.GLEAM_OVERLAP_CALLS])
@pytest.mark.parametrize("offset", [0, 8, 5])
@pytest.mark.parametrize("C", [4 * KiB, 7 * KiB + 32, 33 * KiB])
def test_stage_edges(C, offset, flags):
    """70 chunks and tails around the stages; then sent again with one bit
    flipped in each chunk, at places around the stages' and rings' edges."""
    for tail in (0, 500, 512, 1023, 1024 + 40, 4 * KiB - 1):
        gc, oc = Cache(300 * C, C, flags), oracle.OracleCache(300 * C, C, flags & B.GLEAM_KEY16)
        host = W.random_bytes(70 * C + tail, seed=tail)
        with gc:
            dedup_both(gc, oc, host, offset=offset)
            dedup_both(gc, oc, host, offset=(offset * 3) % 16)
            edges = [0, 511, 512, 1023, 1024, 2047, 3 * KiB, 4095, 4 * KiB, 5 * KiB - 1, 5 * KiB,
                     8 * KiB, 9 * KiB - 1, C - 1]
            host = host.clone()
            for i in range(0, 70, 2):
                host[i * C + min(C - 1, edges[(i // 2) % len(edges)])] ^= 1 << (i % 8)
            dedup_both(gc, oc, host, offset=offset)
            compare_cache(gc, oc, check_bytes=150)


@pytest.mark.parametrize("mode", [1, 2])  # the write-through of likely misses always on, off
@pytest.mark.parametrize("n", [65, 304, 305, 609, 1217, 1825, 2432, 2433])
def test_chunk_counts(n, mode):
    """Chunks per block 1, 2, 3, 5, 7, 8 with a last block part-filled, and one
    chunk too many for the wave; a first load, then half of it changed."""
    C = 4 * KiB
    gc, oc = Cache(2 * n * C, C), oracle.OracleCache(2 * n * C, C)
    host = W.random_bytes(n * C - 100, seed=n)
    with gc:
        gc.debug_set(B.GLEAM_DEBUG_SPECULATE, mode)
        dedup_both(gc, oc, host)
        host = host.clone()
        host.view(-1)[::2 * C] ^= 2
        host[7 * C:9 * C] = host[20 * C:22 * C]  # in-call duplicates
        dedup_both(gc, oc, host)
        compare_cache(gc, oc)


def test_batch_of_mixed_payloads():
    """Several payloads to a block, at mixed alignments, equal chunks among them."""
    C = 4 * KiB
    gc, oc = Cache(2000 * C, C), oracle.OracleCache(2000 * C, C)
    sizes = [3 * C + 700, 40, 90 * C, C, 130 * C + 2049, 5 * C - 1]
    parts = [W.random_bytes(s, seed=40 + k) for k, s in enumerate(sizes)]
    parts[4][10 * C:60 * C] = parts[2][:50 * C]
    with gc:
        for rep in range(2):
            bufs = [to_device(p, (5 * k) % 16) for k, p in enumerate(parts)]
            outs = [DedupOutputs.alloc(s, C, DEV) for s in sizes]
            res = torch.zeros(len(sizes), B.RESULT_WORDS, dtype=torch.int64, device=DEV)
            gc.dedup_batch(bufs, outs, [res[k] for k in range(len(sizes))])
            torch.cuda.synchronize()
            for k, s in enumerate(sizes):
                rc, mask, idx, packed = oc.dedup(parts[k].numpy())
                assert res[k, 0].item() == 0 and res[k, 1].item() == rc
                assert np.array_equal(outs[k].hit_mask.cpu().numpy().view(np.uint32)[:len(mask)], mask)
                assert np.array_equal(outs[k].miss_idx.cpu().numpy().view(np.uint32)[:rc], idx)
                assert np.array_equal(outs[k].miss_bytes.cpu().numpy()[:len(packed)], packed)
            parts[2] = parts[2].clone()
            parts[2][::3 * C] ^= 1
        compare_cache(gc, oc, check_bytes=200)


def test_small_calls_either_way():
    """Calls of at most 64 chunks as the library runs them, and with the
    single-block kernel asked for: equal to the oracle both times."""
    C = 4 * KiB
    for limit in (None, 64):
        gc, oc = Cache(600 * C, C), oracle.OracleCache(600 * C, C)
        with gc:
            if limit is not None:
                gc.debug_set(B.GLEAM_DEBUG_SMALL_CALLS, limit)
            for n in (1, 100, 511, 512, C - 1, C, C + 1, 9 * C + 700, 63 * C, 64 * C - 5):
                host = W.random_bytes(n, seed=n)
                for offset in (0, 8, 0):
                    dedup_both(gc, oc, host, offset=offset)
                host = host.clone()
                host[n // 2] ^= 16
                dedup_both(gc, oc, host)
            compare_cache(gc, oc, check_bytes=300)
