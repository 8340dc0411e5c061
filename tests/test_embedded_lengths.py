"""Solve passes on transform lengths F >= 2n (grids whose padded length has no tuned plan):
the change of period of the multiplier is exact, every length F solves to the parity
tolerance on every axis, and the host's and the library's length rules agree.
"""
import numpy as np
import pytest

from paper_2506_04489_gb300 import serve

TOL = {"fp64": 1e-12, "df32": 1e-12, "fp32": 1e-5, "mixed": 1e-5}
BOX = ((-1.0, -1.0, -1.0), (1.0, 1.0, 1.0))


@pytest.mark.parametrize("n,F", [(2, 4), (5, 16), (7, 16), (13, 32), (37, 80), (50, 100), (61, 128)])
def test_change_of_period_is_exact(n, F):
    # K_j from the multiplier of period 2n, cut to |j| <= n - 1, as a multiplier of period F:
    # both give the same aperiodic convolution (1D; the axes are independent)
    rng = np.random.default_rng(n)
    k = np.arange(2 * n)
    M = rng.standard_normal(n + 1)[np.minimum(k, 2 * n - k)]
    rho = rng.standard_normal(n)
    ref = np.fft.ifft(M * np.fft.fft(rho, 2 * n)).real[:n] * 2 * n
    q, kk = np.arange(F)[:, None], np.arange(n + 1)[None, :]

    def dirichlet(b):  # sum over |j| <= n - 1 of cos(j b)
        return sum(np.cos(j * b) for j in range(-(n - 1), n))

    b0, b1 = 2 * np.pi * (q / F - kk / (2 * n)), 2 * np.pi * (q / F + kk / (2 * n))
    T = np.where((kk == 0) | (kk == n), 0.5, 1.0) * (dirichlet(b0) + dirichlet(b1)) / F
    MF = T @ M[: n + 1]
    got = np.fft.ifft(MF * np.fft.fft(rho, F)).real[:n] * F
    # rounding: sums of 2n terms of size 1 with 2n x F evaluations of cos, far below 1e-11
    assert np.abs(got - ref).max() <= 1e-11 * np.abs(ref).max()


def test_length_rule_matches_the_library():
    from paper_2506_04489_gb300 import build
    build.build()
    from paper_2506_04489_gb300 import _native as N
    cfg = N.ServerConfig(-1.0, 1.0, 1e9, 2, 4, 2, 2, 2 * 128 ** 3, 256 ** 3)
    for n in range(2, 1025):
        for prec, code in (("fp64", 0), ("fp32", 1), ("mixed", 2), ("df32", 3)):
            assert N.lib.sp_server_entry_bytes(cfg, n, code) == serve.entry_bytes(n, prec, 2), (n, prec)


def _grids():
    """(n0, n1, n2) with one axis on each length F (an odd grid size below F/2 where the
    neighbouring length leaves one, else F/2), the others short."""
    prev = 0
    for F in serve.F_LENGTHS:
        n = F // 2 - 1 if F - 2 > prev else F // 2
        prev = F
        for ax in range(3):
            g = [8, 16, 8]
            g[ax] = n
            yield tuple(g)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "df32", "fp32", "mixed"])
@pytest.mark.parametrize("n", list(_grids()))
def test_every_length_on_every_axis(n, precision):
    import torch
    from paper_2506_04489_gb300 import Plan
    plan = Plan(n, *BOX, precision=precision)
    rho = np.random.default_rng(sum(n)).random(n) + 0.1
    t = torch.from_numpy(rho).to("cuda", dtype=plan.dtype)
    u = plan.solve(t).double().cpu().numpy()
    plan.sync()
    M = plan.tables()["M"]  # the FP64 multiplier on the 2n octant (checked elsewhere)
    plan.close()
    k = [np.minimum(np.arange(2 * m), 2 * m - np.arange(2 * m)) for m in n]
    full = M[np.ix_(k[0], k[1], k[2][: n[2] + 1])]
    spec = np.fft.rfftn(t.double().cpu().numpy(), s=[2 * m for m in n], axes=(0, 1, 2)) * full
    ref = np.fft.irfftn(spec, s=[2 * m for m in n], axes=(0, 1, 2))[: n[0], : n[1], : n[2]] * 8 * np.prod(n)
    assert np.abs(u - ref).max() <= TOL[precision] * np.abs(ref).max()


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_noalloc_at_the_scratch_limit(precision):
    # 2n passes fit the static scratch where the longer transforms' workspace does not
    import ctypes
    import torch
    from paper_2506_04489_gb300 import Plan, _native
    n = {"fp64": (125, 125, 125), "fp32": (158, 158, 158)}[precision]
    plan = Plan(n, *BOX, precision=precision)
    rho = torch.rand(n, dtype=plan.dtype, device="cuda")
    ref = plan.solve(rho)
    u = torch.full_like(rho, float("nan"))
    rc = _native.lib.sp_solve_noalloc(plan.handle, ctypes.c_void_p(rho.data_ptr()), ctypes.c_void_p(u.data_ptr()),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, _native.lib.sp_last_error()
    torch.cuda.synchronize()
    plan.close()
    assert float((u - ref).abs().max() / ref.abs().max()) <= TOL[precision]
