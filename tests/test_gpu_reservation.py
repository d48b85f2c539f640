"""A reservation made with a queue's word as read earlier is refused only when the queue is full,
not because another command has taken the slot that the old word names."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import PAGE, Ctx, build_user_kernel  # noqa: E402


@pytest.mark.parametrize("depth", [64, 256])
def test_an_old_word_is_read_again(depth):
    L = build_user_kernel("reserve_demo")
    L.reserve_demo.restype = C.c_int
    L.reserve_demo.argtypes = [C.c_void_p, C.c_uint32, C.c_void_p, C.c_void_p]
    n = 300  # more rounds than slots
    got = torch.full((n,), -1, dtype=torch.int32, device="cuda:0")
    with Ctx(64 * PAGE, cache_bytes=64 * PAGE, ways=8, num_queues=1, queue_depth=depth) as c:
        assert L.reserve_demo(c.h, n, got.data_ptr(), c.stream) == 0
        torch.cuda.synchronize()
        c.check()
        assert (got == 1).all(), int((got != 1).sum())
        st = c.stats()
        assert st["commands"] == 2 * n and st["sq_full"] == 0
