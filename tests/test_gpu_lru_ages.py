"""GLEAM_EVICT_LRU: which slots a call evicts when their ages (calls since the
last use) lie around the edges of the age histogram: one bin per age below
4,096, one for all greater ages, from which the order of the last uses decides.
The clock is moved forward between calls; the oracle, whose clock counts its
calls, keeps the same order."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300.cache import Cache
from tests._parity import compare_cache, dedup_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 99, 100, 101, 350, 600])
@pytest.mark.parametrize("gaps", [(1, 1, 1, 1, 1, 1), (1, 1, 1, 1, 1, 4095), (1, 1, 1, 1, 1, 4096),
                                  (1, 1, 4000, 95, 1, 1), (5, 70000, 3, 65536, 4097, 2),
                                  (1 << 20, 1, 1, 1, 1 << 20, 5000), (1, 1, 1, 1, 1, 1 << 31)])
def test_ages(gaps, k):
    C, per = 64, 100
    n = per * len(gaps)
    rng = np.random.default_rng(k)
    new = lambda m: torch.from_numpy(rng.integers(0, 256, m * C, dtype=np.uint8))
    gc, oc = Cache(n * C, C, B.GLEAM_EVICT_LRU), oracle.OracleCache(n * C, C, oracle.EVICT_LRU)
    clock = 0
    with gc:
        for gap in gaps:  # the cache filled by one call per clock value
            gc.debug_set(B.GLEAM_DEBUG_CLOCK, clock)
            clock += 1
            assert dedup_both(gc, oc, new(per)) == per
            clock += gap - 1
        for step in range(3):
            gc.debug_set(B.GLEAM_DEBUG_CLOCK, clock)
            clock += 1
            assert dedup_both(gc, oc, new(k)) == k
            compare_cache(gc, oc, check_bytes=n)
            assert gc.stats()["evictions"] == oc.stats()["evictions"] == (step + 1) * k
