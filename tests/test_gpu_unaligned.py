"""Payloads at any byte alignment: hashed, compared and copied from the 16-byte
pieces they lie in.  Every alignment of a 16-byte piece, lengths around the
stage, piece and chunk edges, payloads that end inside a piece; outputs and cache
against the oracle, and the bytes around an unaligned output left alone."""
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


@pytest.mark.parametrize("offset", range(1, 16))
def test_fingerprints(offset):
    host = W.random_bytes(9000 + offset, seed=offset)
    d = to_device(host, offset)
    for C in (5, 31, 32, 48, 100, 512, 1000, 4096, 0):
        for n in (host.numel(), 33, 511 if C != 5 else 17):
            got = fingerprint(d[:n], C).cpu().numpy().view(np.uint64)
            assert np.array_equal(got, oracle.fingerprint(host.numpy()[:n], C)), (C, n)


@pytest.mark.usefixtures("call_path")
@pytest.mark.parametrize("offset,packed_offset", [(1, 0), (2, 3), (4, 0), (7, 7), (8, 0), (8, 8),
                                                  (12, 5), (15, 0), (0, 1)])
@pytest.mark.parametrize("C", [32, 1 * KiB, 4 * KiB, 32 * KiB])
def test_calls_match_oracle(C, offset, packed_offset):
    """First sight, again, then with flipped bits, at few chunks and at many."""
    cap = 400 * C
    gc, oc = Cache(cap, C), oracle.OracleCache(cap, C)
    with gc:
        for n in (1, 15, 31, 33, C - 1, C, C + 1, 5 * C + 511, 5 * C + 513, 70 * C + C // 2 + 1):
            host = W.random_bytes(n, seed=n)
            dedup_both(gc, oc, host, offset=offset, packed_offset=packed_offset)
            dedup_both(gc, oc, host, offset=(offset + 8) % 16, packed_offset=packed_offset)
            host = host.clone()
            host[n // 3] ^= 4
            host[-1] ^= 1
            dedup_both(gc, oc, host, offset=offset, packed_offset=packed_offset)
        compare_cache(gc, oc, check_bytes=200)


@pytest.mark.parametrize("key16", [False, True])
def test_batch_of_mixed_alignments(key16):
    """Payloads back to back at odd places of one blob, equal chunks among them
    at other alignments, in one call."""
    C, flags = 1 * KiB, B.GLEAM_KEY16 if key16 else 0
    gc, oc = Cache(4000 * C, C, flags), oracle.OracleCache(4000 * C, C, flags)
    sizes = [40 * C + 9, 3 * C, 700, 90 * C + 1, 1, 64 * C + 1023, 40 * C + 9]
    parts = [W.random_bytes(s, seed=k) for k, s in enumerate(sizes)]
    parts[3][5 * C:25 * C] = parts[0][10 * C:30 * C]   # in-call duplicates, shifted
    parts[6][:] = parts[0]
    blob = torch.cat([W.random_bytes(3, seed=99)] + parts)
    with gc:
        for rep in range(2):
            big = torch.empty(blob.numel(), dtype=torch.uint8, device=DEV)
            big.copy_(blob)
            pos, bufs, outs, guards = 3, [], [], []
            for k, s in enumerate(sizes):
                bufs.append(big[pos:pos + s])
                pos += s
                o = DedupOutputs.alloc(s, C, DEV)
                room = torch.full((s + 64,), 0xA5, dtype=torch.uint8, device=DEV)
                o.miss_bytes = room[k + 16:k + 16 + s]
                guards.append(room)
                outs.append(o)
            res = torch.zeros(len(sizes), B.RESULT_WORDS, dtype=torch.int64, device=DEV)
            gc.dedup_batch(bufs, outs, [res[k] for k in range(len(sizes))])
            torch.cuda.synchronize()
            for k, s in enumerate(sizes):
                rc, mask, idx, packed = oc.dedup(parts[k].numpy())
                assert res[k, 0].item() == 0 and res[k, 1].item() == rc
                assert np.array_equal(outs[k].hit_mask.cpu().numpy().view(np.uint32)[:len(mask)], mask)
                assert np.array_equal(outs[k].miss_idx.cpu().numpy().view(np.uint32)[:rc], idx)
                assert np.array_equal(outs[k].miss_bytes.cpu().numpy()[:len(packed)], packed)
                room = guards[k].cpu().numpy()
                assert (room[:k + 16] == 0xA5).all() and (room[k + 16 + s:] == 0xA5).all()
            parts = [p.clone() for p in parts]
            parts[5][::3000] ^= 1
            blob = torch.cat([W.random_bytes(3, seed=99)] + parts)
        compare_cache(gc, oc, check_bytes=300)


@pytest.mark.parametrize("shift", [1, 8, 13])
def test_block_check_at_odd_offsets(shift):
    C = 4 * KiB
    host = W.random_bytes(20 * C + 77, seed=5)
    with Cache(64 * C, C) as gc:
        n = (host.numel() + C - 1) // C
        d = host.to(DEV)
        out, slots = DedupOutputs.alloc(host.numel(), C, DEV), torch.zeros(n, dtype=torch.int32, device=DEV)
        gc.dedup_batch(None, items=Cache.batch_items([d], [out], None, [slots]))
        block = to_device(host, shift)
        offs = torch.arange(n, dtype=torch.int64, device=DEV) * C
        assert gc.block_check(block, offs, slots).item() == 0
        for at in (0, 15, 16, C - 1, 7 * C + 500, host.numel() - 1):
            block[at] ^= 8
            bad = torch.zeros(n, dtype=torch.uint8, device=DEV)
            assert gc.block_check(block, offs, slots, mismatch=bad).item() == 1
            assert bad[at // C].item() == 1
            block[at] ^= 8
