"""The end of a call whose every chunk is a cache hit, which the resolve kernel
publishes itself: run on its own arrays, so that an error or a barrier that only
some blocks pass can be put there beforehand."""
import pytest
import torch

from paper_2607_23115_gb300 import binding as B
from tests import _native

pytestmark = pytest.mark.gpu


def _published(o, nch):
    assert (o.status, o.hits, o.calls) == (0, nch, 1)
    assert o.mask0 == (1 << min(32, nch)) - 1 and o.slots_ok == nch
    assert o.uses_new == nch and o.ctl_left == 0


@pytest.mark.parametrize("grid,nch", [(1, 1), (1, 31), (1, 300), (2, 300), (7, 2000)])
def test_published(grid, nch):
    torch.cuda.synchronize()
    _published(_native.all_hits(grid, nch), nch)


@pytest.mark.parametrize("grid,nch", [(1, 1), (1, 300), (2, 300), (7, 2000)])
def test_an_error_of_the_hash_kernel(grid, nch):
    """Reported, the hit slots' last uses given back, and no mask written."""
    torch.cuda.synchronize()
    o = _native.all_hits(grid, nch, err=B.GLEAM_ERR_INTERNAL)
    assert (o.status, o.hits, o.calls) == (B.GLEAM_ERR_INTERNAL, 0, 0)
    assert o.uses_old == nch and o.mask0 == 0 and o.ctl_left == 0


@pytest.mark.parametrize("grid,arrived", [(2, 1), (7, 1), (7, 3), (7, 6), (32, 1), (32, 16)])
def test_a_wait_that_only_some_blocks_see_run_out(grid, arrived):
    """Blocks counted at the barrier beforehand: the first of the grid's blocks pass
    it, the others wait until their limit.  The call fails as a whole."""
    torch.cuda.synchronize()
    for _ in range(20):  # which blocks pass differs
        o = _native.all_hits(grid, 2000, bar_count=arrived, wait_ns=1_000_000)
        assert (o.status, o.hits, o.calls) == (B.GLEAM_ERR_TIMEOUT, 0, 0)
        assert o.uses_old == 2000 and o.ctl_left == 0
