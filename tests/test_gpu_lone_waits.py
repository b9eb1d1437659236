"""k_hash_lone with a limit on the waits between its warps so short that they may
run out: a dedup call's chunks then have their right fingerprints, or the call
has recorded GLEAM_ERR_TIMEOUT; gleam_fingerprint, which has no status, gives the
right ones in any case."""
import numpy as np
import pytest

import oracle
from paper_2607_23115_gb300 import binding as B
from paper_2607_23115_gb300 import workloads as W
from tests import _native
from tests._parity import to_device

pytestmark = pytest.mark.gpu
KiB = 1024
LIMITS = [0, 300, 3_000, 30_000, 4_000_000_000]


@pytest.mark.parametrize("nch,C", [(5, 64 * KiB), (300, 64 * KiB), (2400, 16 * KiB), (700, 5 * KiB)])
@pytest.mark.parametrize("offset", [0, 8])
def test_a_dedup_call_reports_it(nch, C, offset):
    host = W.random_bytes(nch * C - 100, seed=nch)
    want = oracle.fingerprint(host.numpy(), C)
    buf = to_device(host, offset)
    for limit in LIMITS:
        for _ in range(4):
            fp, err = _native.hash_alone(buf, C, True, limit)
            assert err in (0, B.GLEAM_ERR_TIMEOUT)
            assert err or np.array_equal(fp, want), limit
    assert err == 0


@pytest.mark.parametrize("nch,C", [(5, 64 * KiB), (2400, 16 * KiB), (700, 5 * KiB), (650, 4096 + 9)])
@pytest.mark.parametrize("offset", [0, 8, 3])
def test_fingerprints_are_right_all_the_same(nch, C, offset):
    host = W.random_bytes(nch * C - 100, seed=nch)
    want = oracle.fingerprint(host.numpy(), C)
    buf = to_device(host, offset)
    for limit in LIMITS:
        for _ in range(4):
            fp, err = _native.hash_alone(buf, C, False, limit)
            assert err == 0 and np.array_equal(fp, want), limit
