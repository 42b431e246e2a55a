"""Device memory when the library's pool runs out: a block whose free is still pending on
another stream has to serve (the allocation's stream waits for it), as it does in the
device's default pool."""
import ctypes

import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu
MB = 1 << 20


# the pool holds one block, or both
@pytest.mark.parametrize("blocks", [1, 2])
def test_allocation_waits_for_a_pending_free(blocks):
    require_gpu()
    from tests import native
    lib = native.library("mem_pool")
    fn = lib.alloc_behind_free
    fn.argtypes = [ctypes.c_size_t, ctypes.c_size_t, ctypes.c_longlong]
    assert fn(192 * MB, blocks * 192 * MB + 32 * MB, 10 ** 8) == 0
