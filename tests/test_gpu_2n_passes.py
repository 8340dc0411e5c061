"""The 2n solve passes (runtime-radix stages and Bluestein's algorithm), through every entry
point of the solve: plans whose longer transforms' workspace was refused by the allocator, as
on a full device, and flat grids whose short axes would round up too far.  Which passes a plan
runs is read from its workspace and its radices.
"""
import ctypes
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2506_04489_gb300.plan as plan_module  # noqa: E402
from paper_2506_04489_gb300 import Plan, serve, _native as N  # noqa: E402

TOL = {"fp64": 1e-12, "df32": 1e-12, "fp32": 1e-5, "mixed": 1e-5}
LO, HI = (-1.0, -1.0, -1.0), (1.0, 1.0, 1.0)


def _work(n, F, precision, max_batch):
    c = 16 if precision in ("fp64", "df32") else 8
    return c * max_batch * n[0] * F[1] * ((F[2] // 2 + 1 + 7) // 8 * 8)


def _longer(n):
    return [2 * m if 2 * m in serve.TUNED_LENGTHS else next(f for f in serve.F_LENGTHS if f >= 2 * m) for m in n]


def _runs_2n(plan):
    r = (ctypes.c_int * 24)()
    N.check(N.lib.sp_plan_launch_config(plan.handle, None, None, None, r, None), "sp_plan_launch_config")
    for ax in range(3):
        f = [x for x in r[8 * ax:8 * ax + 8] if x]  # none: Bluestein's algorithm
        if f and (math.prod(f) != 2 * plan.n[ax] or max(f) > 8):
            return False
    return plan.workspace_bytes == _work(plan.n, [2 * m for m in plan.n], plan.precision, plan.max_batch)


def _refused_plan(monkeypatch, n, precision, max_batch=1):
    """A plan whose allocator refuses the longer transforms' workspace (once)."""
    size = _work(n, _longer(n), precision, max_batch)
    refused = []

    def alloc(nbytes, device, ctx):
        if nbytes == size and not refused:
            refused.append(nbytes)
            return None
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), device=int(device)))

    def release(ptr, nbytes, device, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    a = N.Allocator(N.ALLOC_FN(alloc), N.RELEASE_FN(release), None)
    monkeypatch.setattr(plan_module, "torch_allocator", lambda: a)
    torch.cuda.init()
    plan = Plan(n, LO, HI, precision=precision, max_batch=max_batch, allocator="torch")
    assert refused == [size] and _runs_2n(plan)
    return plan


def _check_entry_points(plan, oracle):
    n, nb = plan.n, plan.max_batch
    rng = np.random.default_rng(sum(n))
    host = [torch.from_numpy(rng.standard_normal(n)).to(plan.dtype) for _ in range(nb)]
    rho = torch.stack(host).cuda()
    alone = torch.stack([plan.solve(rho[b].contiguous()) for b in range(nb)])
    assert torch.equal(plan.solve_batched(rho), alone)
    out = torch.full_like(rho, float("nan"))
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        graph = plan.capture(rho, out, stream)
        graph.launch(stream)
    stream.synchronize()
    graph.close()
    assert torch.equal(out, alone)
    outs = [torch.empty(n, dtype=plan.dtype).pin_memory() for _ in range(nb)]
    plan.solve_host_stream([h.pin_memory() for h in host], outs)
    plan.sync()
    _, _, M = oracle.plan_tables(n, LO, HI)
    for b in range(nb):
        assert torch.equal(outs[b], alone[b].cpu())
        ref = oracle.solve(M, host[b].double().numpy())
        assert np.abs(alone[b].double().cpu().numpy() - ref).max() <= TOL[plan.precision] * np.abs(ref).max()
    plan.close()


# radix 3, 5 and 7 stages (20, 28, 40; 70, 50, 80; 98, 100, 24), Bluestein's algorithm on every
# axis (22, 26, 34), on some (44, 32, 122), at 254
@pytest.mark.parametrize("n", [(10, 14, 20), (35, 25, 40), (49, 50, 12), (11, 13, 17), (22, 16, 61), (8, 127, 8)])
@pytest.mark.parametrize("precision", list(TOL))
def test_refused_workspace_runs_2n(oracle, monkeypatch, n, precision):
    _check_entry_points(_refused_plan(monkeypatch, n, precision, max_batch=2), oracle)


# F would be 128 x 128 x 16 (6.6 times the points) and 128 x 16 x 128 (4.5 times)
@pytest.mark.parametrize("n", [(50, 50, 2), (50, 3, 49)])
@pytest.mark.parametrize("precision", list(TOL))
def test_flat_grids_run_2n(oracle, n, precision):
    plan = Plan(n, LO, HI, precision=precision, max_batch=2)
    assert _runs_2n(plan)
    _check_entry_points(plan, oracle)


# FP64 pays for padding in full once a batch fills the chip, and where the one Bluestein axis
# holds little of the work; measured on F against 2n: 1.8, 1.7, 1.5, 1.2, 1.2, 1.1 and 1.8 times
# the time; then 0.69, 0.90 and 0.67, a growth of 2.1, and a growth of 1
@pytest.mark.parametrize("n,nb,longer", [((100, 2, 11), 45, False), ((20, 4, 10), 125, False), ((98, 9, 9), 12, False),
                                         ((12, 12, 12), 128, False), ((14, 14, 14), 128, False), ((21, 18, 9), 29, False),
                                         ((784, 2, 436), 1, False), ((18, 18, 18), 1, True), ((25, 25, 25), 27, True),
                                         ((18, 50, 24), 200, True), ((50, 50, 50), 1, False), ((16, 48, 80), 4, True)])
def test_fp64_runs_the_faster_length(n, nb, longer):
    plan = Plan(n, LO, HI, precision="fp64", max_batch=nb, precompute=False)
    assert _runs_2n(plan) != longer
    plan.close()


@pytest.mark.parametrize("n,nb", [((20, 4, 10), 125), ((98, 9, 9), 12), ((12, 12, 12), 128)])
def test_fp64_batches_on_2n(oracle, n, nb):
    plan = Plan(n, LO, HI, precision="fp64", max_batch=nb)
    assert _runs_2n(plan)
    _check_entry_points(plan, oracle)


# the longest lengths (2048 by radix stages, 2042 by Bluestein's algorithm with M = 4096): a
# density shifted by one cell has the potential shifted by one cell; two solves are compared,
# each held to the parity tolerance
@pytest.mark.parametrize("n,axis", [((1024, 8, 9), 0), ((8, 1024, 9), 1), ((8, 9, 1024), 2),
                                    ((1021, 8, 9), 0), ((8, 1021, 9), 1), ((8, 9, 1021), 2)])
@pytest.mark.parametrize("precision", list(TOL))
def test_longest_lengths_on_2n(monkeypatch, n, axis, precision):
    rho = np.random.default_rng(sum(n) + axis).random(n)
    last = [slice(None)] * 3
    last[axis] = -1
    rho[tuple(last)] = 0.0
    plan = _refused_plan(monkeypatch, n, precision)
    u, us = (plan.solve(torch.from_numpy(np.ascontiguousarray(r)).to("cuda", dtype=plan.dtype)).double().cpu().numpy()
             for r in (rho, np.roll(rho, 1, axis=axis)))
    plan.close()
    head, tail = [slice(None)] * 3, [slice(None)] * 3
    head[axis], tail[axis] = slice(1, None), slice(None, -1)
    assert np.abs(us[tuple(head)] - u[tuple(tail)]).max() <= 2 * TOL[precision] * np.abs(u).max()
