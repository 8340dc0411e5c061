"""A server whose budget holds a size's plan on 2n but not on the longer transforms that its
passes run with room: the requests are served, within the budget.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2506_04489_gb300 import Plan, serve, workloads as W  # noqa: E402

# two solves are compared, each held to the parity tolerance
TOL = {"fp32": 2e-5, "df32": 2e-12}


@pytest.mark.parametrize("prepare", [False, True])
@pytest.mark.parametrize("n,precision", [(49, "fp32"), (50, "df32"), (83, "df32"), (97, "fp32")])
def test_budget_that_holds_2n_only(n, precision, prepare):
    mb, c = 4, 16 if precision == "df32" else 8
    f, ldz = serve.transform_length(n, precision), (n + 1 + 7) // 8 * 8
    longer = mb * c * n * (f * ((f // 2 + 1 + 7) // 8 * 8) - 2 * n * ldz)  # of workspace
    budget = serve.entry_bytes(n, precision, mb) - longer // 2
    assert longer > 0
    dt = torch.float32 if precision == "fp32" else torch.float64
    rhos = [torch.from_numpy(W.gaussian_mixture(n, -1.0, 1.0, i)).to(dt).pin_memory() for i in range(6)]
    srv = serve.Server(budget_bytes=budget, max_batch=mb, slots=2).start()
    if prepare:
        srv.prepare([(n, precision)])
        assert srv._stats()[2] > 0  # resident before any request
    futs = [srv.submit(r, 1e-6 if precision == "fp32" else 1e-12) for r in rhos]
    got = [fut.result(timeout=120) for fut in futs]
    srv.stop()
    assert 0 < srv.peak_bytes <= budget
    plan = Plan(n, -1.0, 1.0, precision=precision)
    for r, u in zip(rhos, got):
        ref = plan.solve(r.cuda()).cpu().double()
        assert float((u.double() - ref).abs().max() / ref.abs().max()) <= TOL[precision]
    plan.close()
