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
