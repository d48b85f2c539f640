"""A user kernel's CTA has agile::kWarps warps: shared memory sized by it holds every warp's share."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import PAGE, Ctx, build_user_kernel  # noqa: E402


@pytest.mark.parametrize("app_warps", [1, 7, 153, 1000])
def test_shared_memory_sized_by_kwarps(app_warps):
    L = build_user_kernel("shape_demo")
    L.shape_demo.restype = C.c_int
    L.shape_demo.argtypes = [C.c_void_p] * 4 + [C.c_uint32, C.c_void_p]
    outside, lost = (torch.zeros(1, dtype=torch.int32, device="cuda:0") for _ in range(2))
    seen = torch.zeros(app_warps, dtype=torch.int32, device="cuda:0")
    with Ctx(64 * PAGE, cache_bytes=64 * PAGE, ways=8, num_queues=8, queue_depth=64) as c:
        assert L.shape_demo(c.h, outside.data_ptr(), lost.data_ptr(), seen.data_ptr(), app_warps, c.stream) == 0
        torch.cuda.synchronize()
        c.check()
    assert outside.item() == 0 and lost.item() == 0
    assert (seen == 1).all()
