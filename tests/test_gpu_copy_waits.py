"""Waits for the misses' bulk copies that run out: the limit is so short that a
one-payload call (whose blocks pass no grid barrier) may give up on a copy.  The
call then reports GLEAM_ERR_TIMEOUT, with its copies landed."""
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
