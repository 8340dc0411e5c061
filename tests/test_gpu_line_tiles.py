"""FP32 line passes whose multiplier rows are staged in shared memory: every column tile of the
32-value plans (a tile of one or two columns copies single values, four and more whole 16-byte
chunks; the last tile of 33 columns is partial) against the convolution in FP64."""
import numpy as np
import pytest

BOX = (-1.0, 1.0)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp32", "mixed"])
@pytest.mark.parametrize("n0,tile", [(256, 1), (256, 2), (256, 4), (256, 8), (256, 16), (512, 1), (512, 2), (512, 4), (512, 8)])
def test_staged_multiplier_rows(n0, tile, precision):
    import torch
    from paper_2506_04489_gb300 import Plan
    n = (n0, 32, 32)
    plan = Plan(n, *BOX, precision=precision)
    plan.set_launch_config(line=(tile, 0, 0))
    rho = torch.from_numpy(np.random.default_rng(n0 + tile).random(n) + 0.1).to("cuda", dtype=plan.dtype)
    u = plan.solve(rho).double().cpu().numpy()
    plan.sync()
    M = plan.tables()["M"]
    plan.close()
    k = [np.minimum(np.arange(2 * m), 2 * m - np.arange(2 * m)) for m in n]
    full = M[np.ix_(k[0], k[1], k[2][: n[2] + 1])]
    spec = np.fft.rfftn(rho.double().cpu().numpy(), s=[2 * m for m in n], axes=(0, 1, 2)) * full
    ref = np.fft.irfftn(spec, s=[2 * m for m in n], axes=(0, 1, 2))[: n[0], : n[1], : n[2]] * 8 * np.prod(n)
    assert np.abs(u - ref).max() <= 1e-5 * np.abs(ref).max()  # the FP32 parity bar
