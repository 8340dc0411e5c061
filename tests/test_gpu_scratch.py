"""The precompute with little device memory left for its scratch: a grid whose scratch fitted
before its passes ran on longer transforms still fits, and the multiplier and the solve are
the same bit for bit.
"""
import contextlib
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_04489_gb300 import Plan  # noqa: E402

MB = 1 << 20


class _PoolProps(ctypes.Structure):  # cudaMemPoolProps
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("locationType", ctypes.c_int),
                ("locationId", ctypes.c_int), ("security", ctypes.c_void_p), ("maxSize", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@contextlib.contextmanager
def _pool_of(nbytes):
    """Stream-ordered allocations of this process come from a pool of at most nbytes."""
    torch.cuda.init()
    rt = ctypes.CDLL("libcudart.so.13")
    old, pool = ctypes.c_void_p(), ctypes.c_void_p()
    props = _PoolProps(allocType=1, handleTypes=0, locationType=1, locationId=0, maxSize=nbytes)
    assert rt.cudaDeviceGetMemPool(ctypes.byref(old), 0) == 0
    assert rt.cudaMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert rt.cudaDeviceSetMemPool(0, pool) == 0
    try:
        yield
    finally:
        torch.cuda.synchronize()
        assert rt.cudaDeviceSetMemPool(0, old) == 0
        assert rt.cudaMemPoolDestroy(pool) == 0


# (grid, precision, pool): 500 x 500 x 20 took 140 MB of quadrature tables when its passes ran
# on 2n, 150^3 68 MB of one operand; 32 MB and less is what a plan of longer transforms may
# leave of them (the workspaces hold 131, 65, 34, 143 and 10 MB)
CASES = [((500, 500, 20), "fp32", 150 * MB), ((150, 150, 150), "fp32", 80 * MB), ((150, 150, 150), "fp32", 32 * MB),
         ((101, 97, 83), "df32", 8 * MB), ((256, 128, 128), "df32", 2 * MB), ((48, 80, 66), "fp64", 4 * MB)]


@pytest.mark.parametrize("n,precision,room", CASES)
def test_precompute_fits_in_little_memory(n, precision, room):
    rho = torch.from_numpy(np.random.default_rng(sum(n)).standard_normal(n)).cuda()
    plans, M, u = [], [], []
    for limit in (None, room):
        plan = Plan(n, -1.0, 1.0, precision=precision, allocator="torch", precompute=False)
        with contextlib.nullcontext() if limit is None else _pool_of(limit):
            plan.precompute()
            plan.sync()
        u.append(plan.solve(rho.to(plan.dtype)))
        M.append(plan.tables()["M"])
        plans.append(plan)
    assert torch.equal(u[0], u[1])
    assert np.array_equal(M[0], M[1])
    for p in plans:
        p.close()
