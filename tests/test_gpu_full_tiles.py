"""Every transform length on every axis at the tiles of real grids: batches large enough that
no tile is made smaller to fill the chip, and lines that leave the last tile partly filled.
Tiles change which lines share a CTA, never a line's arithmetic, so each right-hand side equals
its solve alone (smaller tiles) bit for bit; one is checked against numpy's transforms.
"""
import ctypes
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_04489_gb300 import Plan, serve, _native as N  # noqa: E402

TOL = {"fp64": 1e-12, "df32": 1e-12, "fp32": 1e-5}


def _cases():
    """(grid, batch): one axis on each length F, an odd size below F/2 where there is one.  Line
    passes see 33 columns (5 tiles of 8, 9 of 4) of at least 7 x 16 outer indices and right-hand
    sides; z passes 105 lines, 53 pairs, of 304 tiles and more at up to 32 pairs a tile."""
    prev = 0
    for F in serve.F_LENGTHS:
        n = F // 2 - 1 if F - 2 > prev else F // 2
        prev = F
        yield (n, 8, 31), 16
        yield (7, n, 31), 16
        yield (7, 15, n), 192 if F <= 96 else 96


@pytest.mark.parametrize("precision", list(TOL))
@pytest.mark.parametrize("n,nb", list(_cases()))
def test_full_and_partial_tiles(n, nb, precision):
    plan = Plan(n, -1.0, 1.0, precision=precision, max_batch=nb)
    radices = (ctypes.c_int * 24)()
    N.check(N.lib.sp_plan_launch_config(plan.handle, None, None, None, radices, None), "sp_plan_launch_config")
    assert math.prod(r for r in radices if r) == math.prod(serve.transform_length(m, "fp32") for m in n)
    gen = torch.Generator(device="cuda").manual_seed(sum(n))
    rho = torch.rand((nb, *n), dtype=plan.dtype, device="cuda", generator=gen)
    u = plan.solve_batched(rho)
    for b in (0, nb // 2, nb - 1):
        assert torch.equal(u[b], plan.solve(rho[b].contiguous()))
    plan.sync()
    M = plan.tables()["M"]
    plan.close()
    k = [np.minimum(np.arange(2 * m), 2 * m - np.arange(2 * m)) for m in n]
    spec = np.fft.rfftn(rho[1].double().cpu().numpy(), s=[2 * m for m in n], axes=(0, 1, 2))
    spec *= M[np.ix_(k[0], k[1], k[2][: n[2] + 1])]
    ref = np.fft.irfftn(spec, s=[2 * m for m in n], axes=(0, 1, 2))[: n[0], : n[1], : n[2]] * 8 * np.prod(n)
    assert np.abs(u[1].double().cpu().numpy() - ref).max() <= TOL[precision] * np.abs(ref).max()
