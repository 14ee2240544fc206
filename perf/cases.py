"""What is timed: the calls that a user of this solver makes, over the range of sizes it is used at.

A case is one of five kinds of call:

* "step"      coefficients for a new sample set, right-hand side and solve (Hierarchy.set_samples, rhs, solve): the
              unit of work of every outer loop over fields, targets or regularisations;
* "cycle"     one multigrid cycle on single-precision vectors (Hierarchy.cycle), as a preconditioner applies it;
* "batch"     independent instances of uneven size solved together (Batch.solve);
* "boundary"  the solve of the Neumann boundary control problem (BoundaryHierarchy.solve);
* "infer" / "train"  the warm-start network: prediction for a batch, and a gradient pass.

Sizes are those of inputs.CONFIGS, of the tests, of the benchmark and of the paper's tables (N = 8, 27, 64, 125).  Launch
shapes stay at the library's defaults (no autotuning), so a case is the same work wherever it runs.
"""
import math
import types

import numpy as np
import torch

import paper_2302_13680_gb300 as P
from paper_2302_13680_gb300 import learned

DEVICE = "cuda"


def listed():
    return [
        # the smallest workload of the benchmark in plain double precision: launches, host decisions and latency
        dict(name="step_n31_N8_fp64", kind="step", n=31, N=8, K=4, nu=1e-4, amp=0.5, fp32=False, fgmres=False,
             coarse="averaged", region=False, tol=1e-10, cycles=10),
        # a control on a subregion, the sample count of a tensor quadrature (27), a small grid
        dict(name="step_n63_N27_region", kind="step", n=63, N=27, K=8, nu=1e-4, amp=1.0, fp32=True, fgmres=False,
             coarse="averaged", region=True, tol=1e-10, cycles=18),
        # the sample count of the paper's main table (125, odd) on a middle grid
        dict(name="step_n127_N125", kind="step", n=127, N=125, K=8, nu=1e-4, amp=1.0, fp32=True, fgmres=False,
             coarse="averaged", region=False, tol=1e-10, cycles=14),
        # the benchmark's second workload: mixed precision, time to 1e-10
        dict(name="step_n255_N64", kind="step", n=255, N=64, K=16, nu=1e-6, amp=1.0, fp32=True, fgmres=False,
             coarse="averaged", region=False, tol=1e-10, cycles=18),
        # the benchmark's headline workload, 537 million unknowns
        dict(name="step_n1023_N256", kind="step", n=1023, N=256, K=32, nu=1e-5, amp=1.0, fp32=True, fgmres=False,
             coarse="averaged", region=False, tol=2e-9, cycles=13),
        # the paper's own outer method: GMRES preconditioned by the V-cycle, double precision throughout
        dict(name="step_n255_N64_fgmres", kind="step", n=255, N=64, K=16, nu=1e-6, amp=1.0, fp32=False, fgmres=True,
             coarse="averaged", region=False, tol=1e-10, cycles=13),
        # the paper's Galerkin coarse operators, single-precision cycles in double-precision refinement
        dict(name="step_n255_N64_galerkin", kind="step", n=255, N=64, K=16, nu=1e-6, amp=1.0, fp32=True, fgmres=False,
             coarse="galerkin", region=False, tol=1e-10, cycles=18),
        # one W(1,1) cycle as a preconditioner in a user's own single-precision Krylov loop
        dict(name="cycle_n127_N100_w11", kind="cycle", n=127, N=100, K=16, nu=1e-4, amp=1.0, gamma=2, sweeps=1),
        # uneven independent instances (other grids, sample counts, regularisations) in one call
        dict(name="batch_20", kind="batch", count=20, shapes=4, tol=1e-10, cycles=14),
        # Neumann boundary control at the paper's N_h = 4032 and N = 125, damped Jacobi cycles in double precision
        dict(name="boundary_n63_N125", kind="boundary", n=63, N=125, K=8, nu=1e-4, amp=1.0, tol=1e-10, cycles=22),
        # the warm start's prediction of a batch of controls
        dict(name="infer_S256_B8", kind="infer", S=256, B=8),
        # the warm start's training: forward, loss and the gradients of every layer
        dict(name="train_S256_B8", kind="train", S=256, B=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "cycle", "batch", "boundary", "infer", "train"])
    if kind in ("step", "cycle"):
        n = rng.choice([31, 63, 127, 255, 511])
        N = _log_int(rng, 6, 256 if n < 511 else 128)
        if rng.random() < 0.3:
            N = max(8, N // 8 * 8)   # a round sample count, as often chosen
        nu, K = 10.0 ** rng.uniform(-6.0, -3.0), rng.choice([4, 8, 16])
        if kind == "cycle":
            return dict(kind="cycle", n=min(n, 255), N=N, K=K, nu=nu, amp=1.0, gamma=rng.choice([1, 2]),
                        sweeps=rng.choice([1, 2]))
        form = rng.choice(["fp32", "fp32", "fp32", "region", "fp64", "fgmres", "galerkin"])
        if form in ("fgmres", "galerkin"):
            n, N = min(n, 255), min(N, 128)
        return dict(kind="step", n=n, N=N, K=K, nu=nu, amp=1.0, fp32=form in ("fp32", "region", "galerkin"),
                    fgmres=form == "fgmres", coarse="galerkin" if form == "galerkin" else "averaged",
                    region=form == "region", tol=2e-9 if n > 255 else 1e-10, cycles=16)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 20), shapes=rng.randint(100, 10000), tol=1e-10, cycles=14)
    if kind == "boundary":
        return dict(kind="boundary", n=rng.choice([15, 31, 63]), N=_log_int(rng, 5, 160), K=8,
                    nu=10.0 ** rng.uniform(-6.0, -2.0), amp=1.0, tol=1e-10, cycles=22)
    return dict(kind=kind, S=32 * rng.randint(1, 8), B=rng.randint(1, 8 if kind == "train" else 16))


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _target(n, rng, rows=None):
    """A sum of eight random sine modes at the interior nodes (rows = n), or on the rows y = 0, h, ... (rows = n + 1)."""
    h = 1.0 / (n + 1)
    x = (np.arange(n) + 1.0) * h
    y = x if rows is None else np.arange(rows) * h
    out = np.zeros((y.size, n))
    for _ in range(8):
        a, b, c = rng.integers(1, 5), rng.integers(1, 5), rng.standard_normal()
        f = np.sin(b * np.pi * y) if rows is None else np.cos((b - 0.5) * np.pi * y)
        out += c * f[:, None] * np.sin(a * np.pi * x)[None, :]
    return out


def _problem(case, seed):
    rng = np.random.default_rng(seed)
    xi = rng.standard_normal((case["N"], case["K"]))
    rows = case["n"] + 1 if case["kind"] == "boundary" else None
    return xi, _target(case["n"], rng, rows)


REGION = (0.25, 0.75, 0.25, 0.75)


def _instances(case, seed):
    """The batch's instances: grids, sample counts and regularisations from case["shapes"], fields and targets from the seed."""
    shape = np.random.default_rng(case["shapes"])
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        n, N, nu = int(shape.choice([63, 127, 255])), int(shape.integers(16, 129)), float(10.0 ** shape.uniform(-6.0, -3.0))
        out.append(types.SimpleNamespace(n=n, N=N, nu=nu, amp=1.0, xi=rng.standard_normal((N, 16)), yd=_target(n, rng)))
    return out


def _net_weights(seed):
    """Weights and biases of a network in training: He-normal convolutions, a head that all layers' gradients reach."""
    rng = np.random.default_rng(seed)
    w = {}
    for name, ci, co, _ in learned.CONVS:
        w[name] = ((rng.standard_normal((co, 9 * ci)) * math.sqrt(2.0 / (9 * ci))).astype(np.float32),
                   (0.05 * rng.standard_normal(co)).astype(np.float32))
    w["head"] = ((0.2 * rng.standard_normal((1, 32))).astype(np.float32), np.zeros(1, np.float32))
    return w


def _net_data(case, seed):
    """Targets y_d, mean log-coefficients and controls of a batch, each of unit size."""
    rng = np.random.default_rng(seed + 7)
    n = case["S"] - 1
    unit = lambda a: a / (np.abs(a).max() + 1e-30)  # noqa: E731
    return [np.stack([unit(_target(n, rng)).reshape(-1) for _ in range(case["B"])]) for _ in range(3)]


def prepare(case, seed):
    dev = torch.device(DEVICE)
    kind = case["kind"]
    if kind in ("infer", "train"):
        net = learned.WarmStartNet(S=case["S"], batch=case["B"], seed=seed)
        for name, (w, b) in _net_weights(seed).items():
            net.set(name, "w", w)
            net.set(name, "b", b)
        yd, mlk, u = (torch.tensor(a, device=dev) for a in _net_data(case, seed))
        n = case["S"] - 1
        return dict(kind=kind, net=net, yd=yd, mlk=mlk, n=n, X=net.pack_inputs(yd, mlk, n), T=net.pack_targets(u, n))
    if kind == "batch":
        probs = _instances(case, seed)
        B = P.Batch(probs)
        fs = []
        for pr in probs:
            h = 1.0 / (pr.n + 1)
            yd = torch.tensor(pr.yd.reshape(-1, 1), device=dev)
            fy = (h * h / pr.N * yd).expand(-1, pr.N).contiguous()
            fs.append((fy, torch.zeros(pr.n ** 2, dtype=torch.float64, device=dev), torch.zeros_like(fy)))
        return dict(kind=kind, B=B, fs=fs, xs=B.zeros(), tol=case["tol"], opts=P.CycleOptions(precision=P.FP32))
    xi, yd = _problem(case, seed)
    if kind == "boundary":
        H = P.BoundaryHierarchy(case["n"], case["N"], xi, case["nu"], case["amp"])
        f = H.rhs(torch.tensor(yd.reshape(-1), device=dev))
        return dict(kind=kind, H=H, f=f, x=H.zeros(0), tol=case["tol"])
    H = P.Hierarchy(case["n"], case["N"], xi, case["nu"], case["amp"], coarse=case.get("coarse", "averaged"),
                    control_box=REGION if case.get("region") else None)
    if kind == "cycle":
        f = tuple(t.float() for t in _cycle_rhs(case, seed, dev))
        return dict(kind=kind, H=H, f=f, x=H.zeros(0, torch.float32),
                    opts=P.CycleOptions(precision=P.FP32, gamma=case["gamma"], n1=case["sweeps"], n2=case["sweeps"]))
    return dict(kind=kind, H=H, x=H.zeros(0), xi=torch.tensor(xi, device=dev),
                yd=torch.tensor(yd.reshape(-1), device=dev), tol=case["tol"],
                opts=P.CycleOptions(precision=P.FP32 if case["fp32"] else P.FP64),
                method=P.METHOD_FGMRES if case["fgmres"] else P.METHOD_CYCLE)


def _cycle_rhs(case, seed, dev):
    """A residual as a Krylov loop meets it: unit-size smooth and rough parts in every block (single-precision values)."""
    n, N = case["n"], case["N"]
    g = torch.Generator(device=dev).manual_seed(int(seed))
    rnd = lambda *s: torch.randn(*s, generator=g, device=dev, dtype=torch.float32).double()  # noqa: E731
    yd = torch.tensor(_problem(case, seed)[1].reshape(-1, 1), device=dev).float().double()
    return yd + 0.5 * rnd(n * n, N), rnd(n * n), 0.5 * rnd(n * n, N) + yd


def run(s):
    kind = s["kind"]
    if kind == "step":
        H = s["H"]
        H.set_samples(s["xi"])
        f = H.rhs(s["yd"])
        for t in s["x"]:
            t.zero_()
        H.solve(s["opts"], f, s["x"], method=s["method"], tol=s["tol"], maxit=200)
        return s["x"]
    if kind == "cycle":
        for t in s["x"]:
            t.zero_()
        s["H"].cycle(s["opts"], s["x"], s["f"])
        return s["x"]
    if kind == "batch":
        for x in s["xs"]:
            for t in x:
                t.zero_()
        s["B"].solve(s["opts"], s["fs"], s["xs"], tol=s["tol"], maxit=200)
        return s["xs"]
    if kind == "boundary":
        for t in s["x"]:
            t.zero_()
        s["H"].solve(s["f"], s["x"], tol=s["tol"], maxit=200)
        return s["x"]
    net = s["net"]
    if kind == "infer":
        return net.forward(net.pack_inputs(s["yd"], s["mlk"], s["n"]))
    pred = net.forward(s["X"])
    loss = net.loss(s["T"], s["n"])
    net.backward()
    return dict(pred=pred, loss=loss, gw=[net.get(k, "gw") for k in learned.LAYERS],
                gb=[net.get(k, "gb") for k in learned.LAYERS])


def work(case):
    """Bytes and operations of the method itself.  A solve: the two face arrays written once, then per V(2,2) cycle the
    least traffic of red-black sweeps, residual, transfers and correction (203 bytes per fine node-sample and cycle with
    4-byte numbers, twice that with 8-byte ones; coarse grids add a third) and about 130 operations; a single cycle: its
    sweeps' share.  The network: activations between layers written and read once, two operations per weight and pixel."""
    kind = case["kind"]
    if kind in ("infer", "train"):
        px = case["B"] * case["S"] ** 2
        acts, flops = 0.0, 0.0
        for _, ci, co, lv in learned.CONVS:
            acts += (ci + co) * 2.0 * px / 4 ** lv
            flops += 18.0 * ci * co * px / 4 ** lv
        k = 1 if kind == "infer" else 3
        return dict(bytes=k * acts + 4.0 * px, flops=k * flops)
    if kind == "batch":
        ns = sum(pr.n ** 2 * pr.N for pr in _instances(case, 0))
        return dict(bytes=ns * (16.0 + 203.0 * case["cycles"]), flops=ns * 130.0 * 4 / 3 * case["cycles"])
    ns = float(case["n"] ** 2 * case["N"])
    if kind == "cycle":
        return dict(bytes=ns * 24.0 * (1.0 + 2.0 * case["sweeps"]), flops=ns * 60.0 * case["sweeps"])
    wide = 1.0 if case.get("fp32") else 2.0
    return dict(bytes=ns * (16.0 + 203.0 * wide * case["cycles"]), flops=ns * 130.0 * 4 / 3 * case["cycles"])


# ---- the same results in plain torch, 64 bits -----------------------------------------------------------------------

def _hm(a, b):
    return 2.0 * a * b / (a + b)


def _faces(n, xi, amp, dev):
    t = torch.arange(n + 2, dtype=torch.float64, device=dev) / (n + 1)
    k = torch.arange(1, xi.shape[1] + 1, dtype=torch.float64, device=dev)
    phi = (torch.sin(math.pi * t[:, None] * k) / k) @ torch.tensor(xi, device=dev).T
    kap = torch.exp(amp * torch.sin(math.pi * t)[:, None, None] * phi[None])
    return kap


class _Grid:
    """One grid of the rediscretised hierarchy, arrays [n, n, N]."""

    def __init__(self, n, N, nu, kx, ky, region, dtype):
        h2 = 1.0 / (n + 1) ** 2
        self.n, self.N, self.kx, self.ky = n, N, kx.to(dtype), ky.to(dtype)
        self.c, self.G, self.d = h2 / N, nu * h2, -h2
        self.a = self.kx[:, :-1] + self.kx[:, 1:] + self.ky[:-1] + self.ky[1:]
        i = torch.arange(n, device=kx.device)
        self.red = ((i[:, None] + i[None, :]) % 2 == 0)
        self.chi = None
        if region:
            s = (i + 1.0) / (n + 1)
            inside = (s >= REGION[0] - 1e-9) & (s <= REGION[1] + 1e-9)
            self.chi = (inside[:, None] & inside[None, :]).to(torch.float64)
        self.isig = 1.0 / (self.G + self.c * self.d * self.d * (1.0 / self.a.double() ** 2).sum(-1))

    def off(self, v):
        o = torch.zeros_like(v)
        o[:, 1:] += self.kx[:, 1:-1] * v[:, :-1]
        o[:, :-1] += self.kx[:, 1:-1] * v[:, 1:]
        o[1:] += self.ky[1:-1] * v[:-1]
        o[:-1] += self.ky[1:-1] * v[1:]
        return o

    def residual(self, x, f):
        y, u, p = x
        cu = u if self.chi is None else self.chi * u
        ry = f[0] - self.c * y - (self.a * p - self.off(p))
        rp = f[2] - (self.a * y - self.off(y)) - (self.d * cu).to(y.dtype)[..., None]
        ru = f[1] - self.G * cu - self.d * p.sum(-1, dtype=torch.float64)
        return ry, (ru if self.chi is None else self.chi * ru), rp

    def sweep(self, x, f):
        y, u, p = x
        for mask in (self.red, ~self.red):
            bp, by = f[0] + self.off(p), f[2] + self.off(y)
            t = (self.c * by / self.a - bp) / self.a
            un = (f[1] + self.d * t.sum(-1, dtype=torch.float64)) * self.isig
            un = un if self.chi is None else self.chi * un
            yn = (by - (self.d * un).to(y.dtype)[..., None]) / self.a
            pn = (bp - self.c * yn) / self.a
            y = torch.where(mask[..., None], yn, y)
            p = torch.where(mask[..., None], pn, p)
            u = torch.where(mask, un, u)
        return y, u, p


def _coarser(kx, ky):
    """Face coefficients of the next grid: series along a face, full weighting across it."""
    nc = (kx.shape[0] - 1) // 2
    hx, hy = _hm(kx[:, 0:2 * nc + 1:2], kx[:, 1:2 * nc + 2:2]), _hm(ky[0:2 * nc + 1:2], ky[1:2 * nc + 2:2])
    kx2 = 0.25 * hx[0:2 * nc:2] + 0.5 * hx[1:2 * nc:2] + 0.25 * hx[2:2 * nc + 1:2]
    ky2 = 0.25 * hy[:, 0:2 * nc:2] + 0.5 * hy[:, 1:2 * nc:2] + 0.25 * hy[:, 2:2 * nc + 1:2]
    return kx2, ky2


def _restrict(v):
    for d in (0, 1):
        v = v.transpose(0, d)
        v = (0.5 * (v[0:-1:2] + v[2::2]) + v[1::2]).transpose(0, d)
    return v


def _prolong(v):
    for d in (0, 1):
        v = v.transpose(0, d)
        o = torch.zeros((2 * v.shape[0] + 1,) + tuple(v.shape[1:]), dtype=v.dtype, device=v.device)
        o[1::2] = v
        o[0:-1:2] += 0.5 * v
        o[2::2] += 0.5 * v
        v = o.transpose(0, d)
    return v


class _Exact:
    def __init__(self, n, xi, nu, amp, region=False, dtype=torch.float64, coarsest=3):
        N, dev = xi.shape[0], torch.device(DEVICE)
        kap = _faces(n, xi, amp, dev)
        kx, ky = _hm(kap[1:-1, :-1], kap[1:-1, 1:]), _hm(kap[:-1, 1:-1], kap[1:, 1:-1])
        del kap
        self.top = _Grid(n, N, nu, kx, ky, region, torch.float64)
        self.grids = [self.top if dtype == torch.float64 else _Grid(n, N, nu, kx, ky, region, dtype)]
        while n > coarsest:
            kx, ky = _coarser(kx, ky)
            n = (n - 1) // 2
            self.grids.append(_Grid(n, N, nu, kx, ky, region, dtype))
        g, m = self.grids[-1], n * n
        eye = torch.eye(m, dtype=torch.float64, device=dev).reshape(m, n, n, 1).expand(m, n, n, N)
        A = torch.stack([g.a.double() * e - g.off(e.to(g.a.dtype)).double() for e in eye])   # [col, n, n, N]
        self.inv = torch.linalg.inv(A.reshape(m, m, N).permute(2, 1, 0))
        M = g.G * torch.eye(m, dtype=torch.float64, device=dev) + g.c * g.d * g.d * (self.inv @ self.inv).sum(0)
        if region:
            c = g.chi.reshape(-1)
            M = M * c[:, None] * c[None, :] + torch.diag(1.0 - c)
        self.Minv = torch.linalg.inv(M)

    def bottom(self, f):
        g, n = self.grids[-1], self.grids[-1].n
        ap = lambda v: torch.einsum("jab,bj->aj", self.inv, v)  # noqa: E731
        fy, fp = (t.double().reshape(n * n, -1) for t in (f[0], f[2]))
        b = f[1].reshape(-1) - g.d * (ap(fy) - g.c * ap(ap(fp))).sum(-1)
        u = self.Minv @ (b if g.chi is None else b * g.chi.reshape(-1))
        y = ap(fp - g.d * u[:, None])
        p = ap(fy - g.c * y)
        return y.reshape(n, n, -1).to(f[0].dtype), u.reshape(n, n), p.reshape(n, n, -1).to(f[0].dtype)

    def cycle(self, x, f, sweeps=2, gamma=1, l=0):
        if l == len(self.grids) - 1:
            return self.bottom(f)
        g = self.grids[l]
        for _ in range(sweeps):
            x = g.sweep(x, f)
        fc = tuple(_restrict(t) for t in g.residual(x, f))
        xc = tuple(torch.zeros_like(t) for t in fc)
        for _ in range(gamma):
            xc = self.cycle(xc, fc, sweeps, gamma, l + 1)
        du = _prolong(xc[1])
        x = (x[0] + _prolong(xc[0]), x[1] + (du if g.chi is None else g.chi * du), x[2] + _prolong(xc[2]))
        for _ in range(sweeps):
            x = g.sweep(x, f)
        return x

    def solve(self, f, cycles):
        """The solution of S x = f: cycles in the hierarchy's precision on double-precision residuals."""
        x = tuple(torch.zeros_like(t) for t in f)
        t = self.grids[0].a.dtype
        for _ in range(cycles):
            r = self.top.residual(x, f)
            sc = max(float(b.abs().max()) for b in r)
            if sc == 0.0:
                break
            r = (r[0].div_(sc).to(t), r[1] / sc, r[2].div_(sc).to(t))
            e = self.cycle(tuple(torch.zeros_like(b) for b in r), r)
            for a, b in zip(x, e):
                a.add_(b, alpha=sc)
        return x


def _solution(n, xi, yd, nu, amp, region, cycles):
    ex = _Exact(n, xi, nu, amp, region, torch.float32)
    N, dev = xi.shape[0], ex.top.a.device
    fy = (torch.tensor(yd, device=dev) * ex.top.c)[..., None].expand(n, n, N).contiguous()
    x = ex.solve((fy, torch.zeros(n, n, dtype=torch.float64, device=dev), torch.zeros_like(fy)), cycles)
    return x[0].reshape(n * n, N), x[1].reshape(-1), x[2].reshape(n * n, N)


def _boundary_solution(case, seed):
    """Elimination of y and p row by row (block tridiagonal matrices), then of the control on the edge."""
    n, N, nu = case["n"], case["N"], case["nu"]
    dev = torch.device(DEVICE)
    xi, yd = _problem(case, seed)
    kap, h = _faces(n, xi, case["amp"], dev), 1.0 / (n + 1)
    kx, ky = _hm(kap[:-1, :-1], kap[:-1, 1:]), _hm(kap[:-1, 1:-1], kap[1:, 1:-1])
    kx[0] *= 0.5
    kx, ky = kx.permute(2, 0, 1), ky.permute(2, 0, 1)          # [N, rows, .]
    mass = torch.full((n + 1, n), h * h, dtype=torch.float64, device=dev)
    mass[0] *= 0.5
    inv = []
    for r in range(n + 1):
        south = ky[:, r - 1] if r else torch.zeros_like(ky[:, 0])
        T = torch.diag_embed(kx[:, r, :-1] + kx[:, r, 1:] + ky[:, r] + south)
        T -= torch.diag_embed(kx[:, r, 1:-1], 1) + torch.diag_embed(kx[:, r, 1:-1], -1)
        if r:
            T = T - south[:, :, None] * inv[-1] * south[:, None, :]
        inv.append(torch.linalg.inv(T))

    def solve(b):                                              # [N, rows, n, m]
        b = b.clone()
        for r in range(1, n + 1):
            b[:, r] += ky[:, r - 1, :, None] * (inv[r - 1] @ b[:, r - 1])
        b[:, n] = inv[n] @ b[:, n]
        for r in range(n - 1, -1, -1):
            b[:, r] = inv[r] @ (b[:, r] + ky[:, r, :, None] * b[:, r + 1])
        return b

    B = torch.zeros(N, n + 1, n, n, dtype=torch.float64, device=dev)
    B[:, 0] = h * torch.eye(n, dtype=torch.float64, device=dev)
    Z = solve(B).reshape(N, -1, n)
    w, t = mass.reshape(-1) / N, torch.tensor(yd, device=dev).reshape(-1)
    M = nu * h * torch.eye(n, dtype=torch.float64, device=dev) + (Z.transpose(1, 2) @ (w[:, None] * Z)).sum(0)
    u = torch.linalg.solve(M, (Z.transpose(1, 2) @ (w * t)[None, :, None]).sum(0))
    y = Z @ u
    p = solve((w[:, None] * (t[:, None] - y)).reshape(N, n + 1, n, 1))
    return y[..., 0].T.contiguous(), u[:, 0], p.reshape(N, -1).T.contiguous()


def _net_exact(case, seed):
    F, dev, S, n = torch.nn.functional, torch.device(DEVICE), case["S"], case["S"] - 1
    par = {k: (torch.tensor(w, device=dev).bfloat16().double(), torch.tensor(b, device=dev).double())
           for k, (w, b) in _net_weights(seed).items()}
    yd, mlk, u = (torch.tensor(a, device=dev).reshape(-1, n, n) for a in _net_data(case, seed))
    x = torch.zeros(case["B"], 8, S, S, dtype=torch.float64, device=dev)
    x[:, 0, :n, :n], x[:, 1, :n, :n] = yd.float().bfloat16().double(), mlk.float().bfloat16().double()
    for w, b in par.values():
        w.requires_grad_(case["kind"] == "train")
        b.requires_grad_(case["kind"] == "train")

    def conv(k, t):
        w, b = par[k]
        co, ci = b.numel(), t.shape[1]
        q, tp = 0.0, F.pad(t, (1, 1, 1, 1))
        for tap in range(9):
            part = tp[:, :, tap // 3:tap // 3 + t.shape[2], tap % 3:tap % 3 + t.shape[3]]
            q = q + torch.einsum("oc,bchw->bohw", w.reshape(co, 9, ci)[:, tap], part)
        return F.relu(q + b[None, :, None, None])

    up = lambda t, s: F.interpolate(t, scale_factor=2, mode="nearest") + s  # noqa: E731
    s0 = conv("c0b", conv("c0a", x))
    s1 = conv("c1b", conv("c1a", F.avg_pool2d(s0, 2)))
    s2 = conv("c2b", conv("c2a", F.avg_pool2d(s1, 2)))
    b3 = conv("c3b", conv("c3a", F.avg_pool2d(s2, 2)))
    e0 = conv("d0", up(conv("d1", up(conv("d2", up(b3, s2)), s1)), s0))
    w, b = par["head"]
    pred = torch.einsum("c,bchw->bhw", w.reshape(-1), e0) + b
    if case["kind"] == "infer":
        return pred
    loss = ((pred[:, :n, :n] - u.float().double()) ** 2).sum() / (case["B"] * n * n)
    loss.backward()
    return dict(pred=pred.detach(), loss=loss.detach().reshape(1), gw=[par[k][0].grad for k in learned.LAYERS],
                gb=[par[k][1].grad for k in learned.LAYERS])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("infer", "train"):
        return _net_exact(case, seed)
    if kind == "boundary":
        return _boundary_solution(case, seed)
    if kind == "batch":
        return [_solution(pr.n, pr.xi, pr.yd, pr.nu, pr.amp, False, 26) for pr in _instances(case, seed)]
    xi, yd = _problem(case, seed)
    if kind == "step":
        return _solution(case["n"], xi, yd, case["nu"], case["amp"], case["region"], 45 if case["region"] else 26)
    ex = _Exact(case["n"], xi, case["nu"], case["amp"])
    n = case["n"]
    f = tuple(t.float().double().reshape(n, n, *t.shape[1:]) for t in _cycle_rhs(case, seed, ex.top.a.device))
    x = ex.cycle(tuple(torch.zeros_like(t) for t in f), f, case["sweeps"], case["gamma"])
    return x[0].reshape(n * n, -1), x[1].reshape(-1), x[2].reshape(n * n, -1)
