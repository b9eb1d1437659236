"""Waits for the misses' bulk copies that run out: the limit is so short that a
one-payload call (whose blocks pass no grid barrier) may give up on a copy.  The
call then reports GLEAM_ERR_TIMEOUT, with its copies landed and the cache as it
was."""
import pytest
import torch

import oracle
from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300 import workloads as W
from paper_2607_23115_gb300.cache import Cache, DedupOutputs, result_dict
from tests._parity import DEV, compare_cache, dedup_both

pytestmark = pytest.mark.gpu
KiB = 1024


@pytest.mark.parametrize("C,nch", [(4 * KiB, 16000), (4 * KiB, 3000), (64 * KiB, 2000)])
def test_another_caches_call_behind_it_is_right(C, nch):
    gc = Cache(3 * nch * C, C)
    other, oc = Cache(400 * C, C), oracle.OracleCache(400 * C, C)
    gc.debug_set(B.GLEAM_DEBUG_SPECULATE, 2)  # every miss is copied
    gc.debug_set(B.GLEAM_DEBUG_WAIT_LIMIT_NS, 1)
    buf = W.random_bytes(nch * C - 40, seed=nch).to(DEV)
    out = DedupOutputs.alloc(buf.numel(), C, DEV)
    res = torch.zeros(B.RESULT_WORDS, dtype=torch.int64, device=DEV)
    with gc, other:
        gc.dedup_async(buf, out, res)
        for seed in (1, 2, 1):
            dedup_both(other, oc, W.random_bytes(120 * C + 50, seed=seed))
        assert result_dict(res)["status"] in (0, B.GLEAM_ERR_TIMEOUT)
        compare_cache(other, oc)


@pytest.mark.parametrize("flags", [0, B.GLEAM_OVERLAP_CALLS, B.GLEAM_PAPER_IDS])
@pytest.mark.parametrize("C,nch", [(4 * KiB, 16000), (64 * KiB, 2000), (4 * KiB, 3000)])
def test_the_cache_stays_as_it_was(C, nch, flags):
    gc = Cache(3 * nch * C, C, flags)
    oc = oracle.OracleCache(3 * nch * C, C, oracle.PAPER_IDS if flags == B.GLEAM_PAPER_IDS else 0)
    gc.debug_set(B.GLEAM_DEBUG_SPECULATE, 2)
    host = W.random_bytes(nch * C - 40, seed=nch)
    buf, out = host.to(DEV), DedupOutputs.alloc(host.numel(), C, DEV)
    res = torch.zeros(B.RESULT_WORDS, dtype=torch.int64, device=DEV)
    with gc:
        dedup_both(gc, oc, W.random_bytes(50 * C, seed=1))
        before = gc.stats()
        gc.debug_set(B.GLEAM_DEBUG_WAIT_LIMIT_NS, 1)
        failed = 0
        for _ in range(3):
            gc.dedup_async(buf, out, res)
            torch.cuda.synchronize()
            if result_dict(res)["status"] == 0:  # no wait ran out
                oc.dedup(host.numpy())
                break
            assert result_dict(res)["status"] == B.GLEAM_ERR_TIMEOUT
            assert gc.stats() == before
            compare_cache(gc, oc)
            failed += 1
        gc.debug_set(B.GLEAM_DEBUG_WAIT_LIMIT_NS, 4_000_000_000)
        dedup_both(gc, oc, host)
        dedup_both(gc, oc, torch.cat([host[5 * C:], host[:5 * C]]))
        compare_cache(gc, oc)
    if not failed:
        pytest.skip("no wait ran out at this size")
