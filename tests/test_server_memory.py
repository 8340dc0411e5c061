"""The server's memory estimate against what a plan takes: every byte that plan creation asks
its allocator for, and the batch buffers, are counted against the budget.
"""
import ctypes

import pytest

from paper_2506_04489_gb300 import serve

CODE = {"fp64": 0, "fp32": 1, "mixed": 2, "df32": 3}


@pytest.mark.parametrize("precision", list(CODE))
def test_sizes_that_no_plan_takes_have_an_estimate(precision):
    from paper_2506_04489_gb300 import build
    build.build()
    from paper_2506_04489_gb300 import _native as N
    cfg = N.ServerConfig(-1.0, 1.0, 1e9, 2, 4, 2, 2, 2 * 128 ** 3, 256 ** 3)
    for n in (1, 1025, 1100, 2000):
        assert N.lib.sp_server_entry_bytes(cfg, n, CODE[precision]) == serve.entry_bytes(n, precision, 2) > 0


# tuned lengths (128), longer transforms (200, 100), Bluestein tables (101), the 2n multiplier
# kept beside the longer one's (126 double-float, 158 FP32), grids left on 2n (50 FP64)
@pytest.mark.gpu
@pytest.mark.parametrize("max_batch", [1, 4])
@pytest.mark.parametrize("n", [16, 50, 100, 101, 126, 128, 158, 200, 300])
@pytest.mark.parametrize("precision", list(CODE))
def test_estimate_covers_the_plan(n, precision, max_batch):
    import torch
    from paper_2506_04489_gb300 import _native as N
    asked = []

    def alloc(nbytes, device, ctx):
        asked.append(nbytes)
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), device=int(device)))

    def release(ptr, nbytes, device, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    a = N.Allocator(N.ALLOC_FN(alloc), N.RELEASE_FN(release), None)
    h = ctypes.c_void_p()
    torch.cuda.init()
    rc = N.lib.sp_plan_create_ex(ctypes.byref(h), (ctypes.c_int * 3)(n, n, n), (ctypes.c_double * 3)(-1, -1, -1),
                                 (ctypes.c_double * 3)(1, 1, 1), 2, None, None, 0, 1e-4, CODE[precision], max_batch,
                                 ctypes.byref(a))
    assert rc == 0, N.lib.sp_last_error()
    N.check(N.lib.sp_plan_destroy(h), "destroy")
    held = sum(asked) + 2 * max_batch * n ** 3 * (4 if precision == "fp32" else 8)
    cfg = N.ServerConfig(-1.0, 1.0, 1e12, max_batch, 4, 2, 2, 2 * 128 ** 3, 256 ** 3)
    need = N.lib.sp_server_entry_bytes(cfg, n, CODE[precision])
    assert held <= need <= held + (1 << 20)
    assert need == serve.entry_bytes(n, precision, max_batch)
