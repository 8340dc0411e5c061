"""Performance cases of the free-space Poisson solver: what a program that uses it has it do.

A case is one call of the public Python face (``Plan.solve``, ``solve_batched``, a captured
graph, ``solve_host_stream``, or ``precompute`` followed by a solve) on a grid of
n0 x n1 x n2 points.  The listed cases span the sizes and types the package's own
configurations, tests and benchmark use, with grid sizes a user picks freely (100, 150, a
prime) beside the powers of two; ``draw`` takes any size of the same ranges.

Calls
  solve    one density in device memory -> its potential (a new output tensor)
  batched  ``batch`` densities in one call
  graph    ``batch`` densities replayed as a captured graph on fixed buffers, autotuned
  host     ``batch`` densities in page-locked host memory through solve_host_stream
  new_box  the multiplier of the plan is precomputed again (its box or table is new to the
           program, as for the first request of a size or after a remesh), then one solve

The mixed precision (float64 arrays, FP32 passes) has no case of its own: it runs the FP32
cases' passes between float64 buffers.
"""
import math

import numpy as np
import torch

from paper_2506_04489_gb300 import Plan

BOX = (-1.0, 1.0)
PRECISIONS = ("fp32", "df32", "fp64")


def _case(name, call, n, precision, density, batch=1):
    n = (n, n, n) if isinstance(n, int) else n
    c = {"call": call, "n0": n[0], "n1": n[1], "n2": n[2], "precision": precision, "density": density, "batch": batch}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest documented grid, FP64: a handful of launches on little data
        _case("solve_32_fp64", "solve", 32, "fp64", "gaussian"),
        # a small request of the served mix
        _case("solve_64_fp32", "solve", 64, "fp32", "mixture"),
        # a small anisotropic grid whose sizes are no powers of two, native FP64
        _case("solve_48x40x36_fp64", "solve", (48, 40, 36), "fp64", "mixture"),
        # a decimal grid size at FP64 accuracy
        _case("solve_100_df32", "solve", 100, "df32", "mixture"),
        # a prime grid size (a cell-centred code with an odd number of points)
        _case("solve_101_df32", "solve", 101, "df32", "bump"),
        # a flat rectangular box, noisy density (binned particles), FP32
        _case("solve_240x180x75_fp32", "solve", (240, 180, 75), "fp32", "noisy"),
        # the headline grid in both accuracies
        _case("solve_256_df32", "solve", 256, "df32", "bump"),
        _case("solve_256_fp32", "solve", 256, "fp32", "bump"),
        # the single large solve, FP32 passes
        _case("solve_512_fp32", "solve", 512, "fp32", "bump"),
        # many right-hand sides on one grid: tuned, captured and replayed
        _case("graph_64x128_df32", "graph", 128, "df32", "mixture", 64),
        # time from host memory to host memory, copies overlapped with the solves
        _case("host_4x150_df32", "host", 150, "df32", "mixture", 4),
        # a new box: the precompute and its first solve
        _case("new_box_128_df32", "new_box", 128, "df32", "oscillating"),
    ]


def draw(rng):
    """A case of the listed ranges: 16 to 300 points an axis (FP64: 16 to 128), at most 2.7e7
    points a call, any of the calls, cubes and rectangular boxes, odd sizes among them."""
    precision = rng.choice(("fp32", "fp32", "df32", "df32", "fp64"))
    call = rng.choice(("solve", "solve", "solve", "batched", "graph", "host", "new_box"))
    top = 128 if precision == "fp64" else 300

    def size():
        return int(round(math.exp(rng.uniform(math.log(16), math.log(top)))))

    n = size()
    shape = (n, n, n)
    if rng.random() < 0.5:
        shape = (n, size(), size())
    batch = 1
    if call in ("batched", "graph", "host"):
        most = max(2, min(32, int(2.7e7 / (shape[0] * shape[1] * shape[2]))))
        batch = int(round(math.exp(rng.uniform(math.log(2), math.log(most)))))
    return _case(None, call, shape, precision, rng.choice(("mixture", "bump", "oscillating", "noisy")), batch)


# ----------------------------------------------------------------------------- inputs
def _axes(n, dev):
    return [torch.linspace(BOX[0], BOX[1], m, dtype=torch.float64, device=dev) for m in n]


def _r2(n, dev, c=(0.0, 0.0, 0.0)):
    x, y, z = (t - s for t, s in zip(_axes(n, dev), c))
    return x[:, None, None] ** 2 + y[None, :, None] ** 2 + z[None, None, :] ** 2


def _gauss(n, dev, c, s):
    e = [torch.exp(-((t - q) ** 2) / (2 * s * s)) for t, q in zip(_axes(n, dev), c)]
    return torch.einsum("i,j,k->ijk", *e) / ((2 * math.pi) ** 1.5 * s ** 3)


def _density(kind, n, seed, dev="cuda"):
    """One density (float64): the package's workloads with seeded parameters."""
    g = np.random.Generator(np.random.PCG64(seed))
    c = g.uniform(-0.1, 0.1, size=3)
    if kind == "gaussian":  # normalised Gaussian near the origin
        return _gauss(n, dev, c, float(g.uniform(0.08, 0.12)))
    if kind == "bump":  # compactly supported exp(-1/(1 - r^2/R^2))
        q = 1.0 - _r2(n, dev, c) / float(g.uniform(0.75, 0.85)) ** 2
        return torch.where(q > 0, torch.exp(-1.0 / q.clamp_min(1e-3)), torch.zeros_like(q))
    if kind == "oscillating":  # Gaussian times a product of cosines
        x, y, z = (torch.cos(float(g.uniform(6, 9)) * math.pi * t) for t in _axes(n, dev))
        return torch.exp(-_r2(n, dev, c) / (2 * 0.25 ** 2)) * torch.einsum("i,j,k->ijk", x, y, z)
    out = torch.zeros(n, dtype=torch.float64, device=dev)
    for _ in range(int(g.integers(1, 9))):  # mixture of 1..8 Gaussians
        centre, s, w = g.uniform(-0.5, 0.5, size=3), float(g.uniform(0.05, 0.2)), float(g.uniform(-1, 1))
        out += w * _gauss(n, dev, centre, s)
    if kind == "noisy":  # with the sampling noise of binned particles
        gen = torch.Generator(device=dev).manual_seed(int(seed))
        out += 0.05 * out.abs().max() * torch.randn(n, dtype=torch.float64, device=dev, generator=gen)
    return out


def _densities(case, seed):
    n = (case["n0"], case["n1"], case["n2"])
    dt = torch.float32 if case["precision"] == "fp32" else torch.float64
    return torch.stack([_density(case["density"], n, seed * 1000 + b).to(dt) for b in range(case["batch"])])


# ----------------------------------------------------------------------------- the cases
def prepare(case, seed):
    n, batch, call = (case["n0"], case["n1"], case["n2"]), case["batch"], case["call"]
    rho = _densities(case, seed)
    plan = Plan(n, *BOX, precision=case["precision"], max_batch=batch if call in ("batched", "graph") else 1)
    s = {"call": call, "plan": plan}
    if call == "graph":
        s["rho"], s["out"] = rho, torch.empty_like(rho)
        plan.autotune(batch)
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        s["graph"] = plan.capture(s["rho"], s["out"], st)
        torch.cuda.current_stream().wait_stream(st)
    elif call == "host":
        s["rho"] = [r.cpu().pin_memory() for r in rho]
        s["out"] = [torch.empty_like(r).pin_memory() for r in s["rho"]]
    else:
        s["rho"] = rho if call == "batched" else rho[0]
    return s


def run(s):
    plan, call = s["plan"], s["call"]
    if call == "solve":
        return plan.solve(s["rho"])
    if call == "batched":
        return plan.solve_batched(s["rho"])
    if call == "graph":
        s["graph"].launch()
        return s["out"]
    if call == "host":
        return plan.solve_host_stream(s["rho"], s["out"])
    plan.precompute()
    return plan.solve(s["rho"])


def work(case):
    """Bytes: densities in and potentials out, and the multiplier octant (the plan's table:
    read by a solve, written by a precompute).  Flops: the pruned padded transforms of a
    solve at 5 N log2 N a complex line of length N = 2n, the multiply, and for a new box the
    contraction of about 530 separable terms that makes the multiplier."""
    n0, n1, n2 = case["n0"], case["n1"], case["n2"]
    N0, N1, N2 = 2 * n0, 2 * n1, 2 * n2
    io = 4 if case["precision"] == "fp32" else 8
    octant = (n0 + 1) * (n1 + 1) * (n2 + 1)
    z = n0 * n1 * 2.5 * N2 * math.log2(N2)
    y = n0 * (n2 + 1) * 5 * N1 * math.log2(N1)
    x = N1 * (n2 + 1) * 5 * N0 * math.log2(N0)
    flops = case["batch"] * (2 * (x + y + z) + 2 * N0 * N1 * (n2 + 1))
    nbytes = case["batch"] * 2 * io * n0 * n1 * n2 + io * octant
    if case["call"] == "new_box":
        flops += 2 * 2 * 530 * octant
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------------------- in 64 bits
def _gs_table(delta, eps=1e-4, step=0.1, eta=1e-17):
    """Trapezoidal rule for 1/(8 pi r) = sum_s w_s exp(-a_s r^2) on (eps, delta]."""
    lo = math.log(eta * math.sqrt(math.pi) / (2 * delta))
    hi = math.log(math.sqrt(math.log(1 / eta)) / eps) + 0.5
    tau = lo + step * np.arange(int(math.ceil((hi - lo) / step)) + 1)
    return np.exp(tau) * step / (4 * math.pi ** 1.5), np.exp(2 * tau)


def _axis_tables(a, n, L, dev):
    """2 int_0^L {1, y^2} exp(-a y^2) cos(pi k y / L) dy, k = 0..n: closed forms where the
    window cuts nothing (a L^2 >= 40), else 16-point Gauss panels, after two integrations by
    parts where the wavenumber is high (kappa^2 >= 4 a)."""
    a = torch.tensor(a, dtype=torch.float64, device=dev)[:, None]
    k = torch.arange(n + 1, dtype=torch.float64, device=dev)[None, :]
    kap = math.pi * k / L
    q = kap * kap / (4 * a)
    G = torch.sqrt(math.pi / a) * torch.exp(-q)
    H = math.sqrt(math.pi) / (2 * a * torch.sqrt(a)) * (1 - 2 * q) * torch.exp(-q)
    m = int((a[:, 0] * L * L < 40).sum())
    if m:
        P = max(n, 8)
        gx, gw = np.polynomial.legendre.leggauss(16)
        t = torch.tensor(0.5 * (1 + gx), dtype=torch.float64, device=dev)
        panel = torch.arange(P, dtype=torch.float64, device=dev)[:, None]
        y = (L * (panel + t) / P).reshape(-1)
        wq = torch.tensor(0.5 * (L / P) * gw, dtype=torch.float64, device=dev).repeat(P)
        ph = torch.remainder(k[0, :, None, None] * panel, 2.0 * P) + k[0, :, None, None] * t  # whole part exact
        C = torch.cos(math.pi * torch.remainder(ph.reshape(n + 1, -1) / P, 2.0))
        b, yy = a[:m], (y * y)[None, :]
        e = wq * torch.exp(-b * yy)
        eL = torch.exp(-b * L * L)
        sgn = 1 - 2 * torch.remainder(k, 2.0)
        k2 = kap * kap
        high = (k2 >= 4 * b) & (k > 0)
        k2 = torch.where(k > 0, k2, torch.ones_like(k2))
        forms = (
            (e, (16 * b ** 4 * yy ** 2 - 48 * b ** 3 * yy + 12 * b ** 2) * e, -2 * b * L * eL,
             (-8 * b ** 3 * L ** 3 + 12 * b ** 2 * L) * eL),
            (e * yy, (16 * b ** 4 * yy ** 3 - 112 * b ** 3 * yy ** 2 + 156 * b ** 2 * yy - 24 * b) * e,
             (2 * L - 2 * b * L ** 3) * eL, (-24 * b * L + 36 * b ** 2 * L ** 3 - 8 * b ** 3 * L ** 5) * eL))
        for out, (p0, p4, d1, d3) in zip((G, H), forms):
            parts = sgn * (d1 / k2 - d3 / k2 ** 2) + (p4 @ C.T) / k2 ** 2
            out[:m] = 2 * torch.where(high, parts, p0 @ C.T)
    return G, H


def _multiplier(n, dev="cuda"):
    """-|kappa|^2 Vhat / (8 n0 n1 n2) on the octant [k0][k1][k2], k_p = 0..n_p."""
    h = [(BOX[1] - BOX[0]) / (m - 1) for m in n]
    L = [m * s for m, s in zip(n, h)]
    w, a = _gs_table(math.sqrt(sum(v * v for v in L)))
    (G0, H0), (G1, H1), (G2, H2) = (_axis_tables(a, m, s, dev) for m, s in zip(n, L))
    w = torch.tensor(w, dtype=torch.float64, device=dev)[:, None]
    kk = [(math.pi / s * torch.arange(m + 1, dtype=torch.float64, device=dev)) ** 2 for m, s in zip(n, L)]
    out = torch.empty([m + 1 for m in n], dtype=torch.float64, device=dev)
    B = torch.cat([G2, H2])
    for k0 in range(n[0] + 1):
        g, v = w * G0[:, k0:k0 + 1], w * H0[:, k0:k0 + 1]
        A = torch.cat([v * G1 + g * H1, g * G1])
        out[k0] = -(kk[0][k0] + kk[1][:, None] + kk[2][None, :]) * (A.T @ B)
    return out / (8.0 * n[0] * n[1] * n[2])


def exact(case, seed):
    """The padded convolution itself in 64 bits, on the densities as the call gets them."""
    n = (case["n0"], case["n1"], case["n2"])
    M = _multiplier(n)
    fold = [torch.minimum(torch.arange(2 * m), 2 * m - torch.arange(2 * m)).to(M.device) for m in n[:2]]
    N = [2 * m for m in n]
    res = []
    for rho in _densities(case, seed):
        F = torch.fft.rfftn(rho.double(), s=N)
        for i in range(N[0]):
            F[i] *= M[fold[0][i]][fold[1]]
        u = torch.fft.irfftn(F, s=N)[:n[0], :n[1], :n[2]] * float(N[0] * N[1] * N[2])
        del F
        res.append(u.contiguous())
    if case["call"] == "host":
        return [u.cpu() for u in res]
    return torch.stack(res) if case["call"] in ("batched", "graph") else res[0]
