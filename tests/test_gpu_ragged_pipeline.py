"""FP32 y passes of ragged lengths on the pipelined kernel: calls with enough tiles to take it
(sixteen right-hand sides of 32 x n x 31), an odd n below F / 2 and the whole F / 2, against the
convolution in FP64."""
import numpy as np
import pytest

BOX = (-1.0, 1.0)


@pytest.mark.gpu
@pytest.mark.parametrize("F", [256, 288, 320, 384, 400, 432, 512, 576, 640, 768, 864])
@pytest.mark.parametrize("full", [False, True])
def test_ragged_y_passes(F, full):
    import torch
    from paper_2506_04489_gb300 import Plan
    # full: 2n = F; n2 = 31 makes the grid take the lengths F whatever 2n has
    n, batch = (32, F // 2 if full else F // 2 - 3, 31), 16
    plan = Plan(n, *BOX, precision="fp32", max_batch=batch)
    rho = torch.from_numpy(np.random.default_rng(F + full).random((batch, *n)) + 0.1).to("cuda", dtype=torch.float32)
    u = plan.solve_batched(rho).double().cpu().numpy()
    plan.sync()
    M = plan.tables()["M"]
    plan.close()
    k = [np.minimum(np.arange(2 * m), 2 * m - np.arange(2 * m)) for m in n]
    kernel = M[np.ix_(k[0], k[1], k[2][: n[2] + 1])]
    for b in (0, batch - 1):
        spec = np.fft.rfftn(rho[b].double().cpu().numpy(), s=[2 * m for m in n], axes=(0, 1, 2)) * kernel
        ref = np.fft.irfftn(spec, s=[2 * m for m in n], axes=(0, 1, 2))[: n[0], : n[1], : n[2]] * 8 * np.prod(n)
        assert np.abs(u[b] - ref).max() <= 1e-5 * np.abs(ref).max()  # the FP32 parity bar
