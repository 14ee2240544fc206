"""Edges of the launch rules: boundary-control nodes over one to eight warps
(and the general kernels above 256 samples) with odd numbers of sweeps, the
cluster coarsest solve with fewer samples than CTAs, half-sweeps and
restrictions on grids beyond the L2 cache (walked backwards), norms of blocks
that do not fill a CTA, face coefficients over more than the FP32 range, and
coarsest solves right behind a new sample set.

Tolerances, relative to each block's largest entry: FP64 single operators and
sweeps 1e-11 (the oracle's parity bar is 1e-12; sums over up to 257 samples
add one digit), direct coarsest solves 1e-10, FP32 sweeps 2e-5 (100 roundings
of 2^-24 and the FP32 faces), norms 1e-13 (pairwise FP64 sums)."""
import numpy as np
import pytest
import torch

import inputs
import oracle.boundary as Bd
import oracle.cmg_oracle as O
import scipy.sparse.linalg as spla

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2302_13680_gb300 import build

    build.build()
    import paper_2302_13680_gb300 as P

    return P


def dev(blocks, N, dtype=torch.float64):
    y, u, p = (np.ascontiguousarray(b) for b in blocks)
    return tuple(torch.tensor(b, dtype=dtype, device="cuda") for b in (y.reshape(-1, N), u.reshape(-1), p.reshape(-1, N)))


def check(got, ref, tol, what):
    for name, g, r in zip("yup", got, ref):
        r = torch.tensor(np.ascontiguousarray(r)).reshape(g.shape)
        e = float((g.double().cpu() - r).abs().max() / r.abs().max().clamp_min(1e-300))
        assert e <= tol, f"{what} block {name}: {e:.3e} > {tol:.1e}"


@pytest.mark.parametrize("N", [1, 7, 32, 33, 64, 65, 125, 256, 257])
def test_boundary_samples_over_warps(P, N):
    n, K, nu, amp = 7, 3, 1e-3, 0.8
    xi = inputs.draw_xi(N, N, K)
    H = P.BoundaryHierarchy(n, N, xi, nu, amp, coarsest_n=3)
    ns, S = Bd.hierarchy(n, N, nu, O.sine_mode_field(xi, amp), coarsest_n=3)
    rng = np.random.default_rng(N)

    def blocks(z, nl):
        m = (nl + 1) * nl
        return z[: m * N], z[m * N: m * N + nl], z[m * N + nl:]

    z, f = rng.standard_normal(S[0].shape[0]), rng.standard_normal(S[0].shape[0])
    fd, r = dev(blocks(f, n), N), H.zeros(0)
    H.residual(0, dev(blocks(z, n), N), fd, r)
    check(r, blocks(f - S[0] @ z, n), 1e-11, "residual")
    for sweeps in (1, 2, 3):
        x, ref = dev(blocks(z, n), N), z
        H.smooth(0, 0.5, sweeps, x, fd)
        for _ in range(sweeps):
            ref = Bd.jacobi_sweep(S[0], n, N, ref, f, 0.5)
        check(x, blocks(ref, n), 1e-11, f"{sweeps} sweeps")
    fc = rng.standard_normal(S[1].shape[0])
    xc = H.zeros(1)
    H.coarse_solve(dev(blocks(fc, ns[1]), N), xc)
    check(xc, blocks(spla.spsolve(S[1].tocsc(), fc), ns[1]), 1e-10, "coarsest solve")
    H.close()


def test_sweep_and_restriction_beyond_l2(P):
    """127^2 nodes, 180 samples: the arrays of a FP64 half-sweep exceed the L2."""
    n, N = 127, 180
    xi = inputs.draw_xi(5, N, 3)
    H = P.Hierarchy(n, N, xi, 1e-4, 0.5)
    lev = O.make_level(n, N, 1e-4, O.sine_mode_field(xi, 0.5))
    rng = np.random.default_rng(1)
    shapes = ((n, n, N), (n, n), (n, n, N))
    x, f = (tuple(rng.standard_normal(s) for s in shapes) for _ in range(2))
    xd = dev(x, N)
    H.smooth(0, P.CycleOptions(), 1, xd, dev(f, N))
    check(xd, O.rbgs_sweep(lev, x, f), 1e-11, "sweep")
    c = H.zeros(1)
    H.restrict(0, dev(f, N), c)
    check(c, O.restrict(n, f), 1e-11, "restriction")
    H.close()


def test_fp32_sweep_beyond_l2(P):
    """255^2 nodes, 90 samples (rows padded to 92) in FP32, against FP64."""
    n, N = 255, 90
    H = P.Hierarchy(n, N, inputs.draw_xi(6, N, 3), 1e-4, 0.5)
    g = torch.Generator(device="cuda").manual_seed(1)
    x = tuple(torch.randn(t.shape, generator=g, device="cuda").double() for t in H.zeros(0))
    f = tuple(torch.randn(t.shape, generator=g, device="cuda").double() for t in x)
    x32, f32 = tuple(t.float() for t in x), tuple(t.float() for t in f)
    H.smooth(0, P.CycleOptions(precision=P.FP32), 1, x32, f32)
    H.smooth(0, P.CycleOptions(), 1, x, f)
    check(x32, tuple(t.cpu().numpy() for t in x), 2e-5, "sweep")
    H.close()


@pytest.mark.parametrize("n,N", [(3, 1), (7, 3), (31, 33), (127, 50)])
def test_norm_of_ragged_blocks(P, n, N):
    H = P.Hierarchy(n, N, inputs.draw_xi(N, N, 3), 1e-3, 0.5)
    v = tuple(torch.randn(t.shape, device="cuda", dtype=torch.float64) for t in H.zeros(0))
    ref = np.sqrt(sum(float((t.cpu() ** 2).sum()) for t in v))
    assert abs(H.norm(0, v) - ref) <= 1e-13 * ref
    H.close()


@pytest.mark.parametrize("amp", [0.0, 5.0, 25.0, 60.0])
def test_faces_over_a_wide_range(P, amp):
    """kappa up to e^(+-150) at amp = 60, far beyond the FP32 range.  Per entry against
    the sum of the terms' magnitudes; the exponential's argument of up to 150,
    rounded to 2^-53 a few times on both sides, moves a face by 150 * 8 *
    2^-53 = 1.4e-13 of itself."""
    n, N, K = 15, 5, 3
    xi = inputs.draw_xi(3, N, K)
    H = P.Hierarchy(n, N, xi, 1e-3, amp)
    lev = O.make_level(n, N, 1e-3, O.sine_mode_field(xi, amp))
    y = np.random.default_rng(2).standard_normal((n, n, N))
    zero = np.zeros((n, n))
    r = H.zeros(0)
    H.residual(0, dev((y, zero, np.zeros_like(y)), N), None, r)
    ref = O.apply_A(lev, y).reshape(-1, N)
    size = (lev.a * np.abs(y) + O.offdiag_sum(lev, np.abs(y))).reshape(-1, N)
    assert np.all(np.abs(r[2].cpu().numpy() - ref) <= 1e-11 * size)
    H.close()


@pytest.mark.parametrize("fp32", [False, True])
def test_coarsest_solve_behind_new_samples(P, fp32):
    """A single grid, whose cycle is the coarsest solve: directly behind the
    set-up on the stream the result is the one after a synchronisation."""
    n, N, K = 3, 100, 3
    H = P.Hierarchy(n, N, inputs.draw_xi(1, N, K), 1e-3, 0.5)
    opts = P.CycleOptions(precision=P.FP32 if fp32 else P.FP64)
    dt = torch.float32 if fp32 else torch.float64
    f = tuple(torch.randn(t.shape, device="cuda", dtype=dt) for t in H.zeros(0))
    for seed in range(2, 8):
        xi = torch.tensor(inputs.draw_xi(seed, N, K), device="cuda")
        a, b = (tuple(torch.zeros_like(t) for t in f) for _ in range(2))
        H.set_samples(xi)
        H.cycle(opts, a, f)
        H.sync()
        H.cycle(opts, b, f)
        assert all(torch.equal(s, t) for s, t in zip(a, b))
    H.close()


def test_fgmres_with_many_basis_vectors(P):
    """A weak preconditioner: the basis passes the group sizes of the dots
    (8) and the updates (16).  The solution at relative residual 1e-11 is the
    cycle iteration's within 1e-7 (as for the Galerkin solutions: the control
    block's sensitivity)."""
    n, N = 31, 5
    pr = inputs.make_problem(n=n, N=N, K=3, nu=1e-3, amp=0.5, seed=4, target="modes")
    H = P.Hierarchy(n, N, pr.xi, pr.nu, pr.amp)
    f = H.rhs(torch.tensor(pr.yd.reshape(-1), device="cuda"))
    x, z = H.zeros(0), H.zeros(0)
    weak = P.CycleOptions(smoother=P.SMOOTH_JACOBI, theta=0.2, n1=1, n2=0)
    st, _ = H.solve(weak, f, x, method=P.METHOD_FGMRES, tol=1e-11, maxit=200, restart=40)
    assert st.iters > 17
    H.solve(P.CycleOptions(), f, z, tol=1e-12, maxit=60)
    check(x, tuple(t.cpu().numpy() for t in z), 1e-7, "solution")
    H.close()


@pytest.mark.parametrize("n,N", [(255, 324), (255, 328), (127, 264), (127, 268)])
def test_zero_guess_sweep_with_or_after_the_restriction(P, n, N):
    """Coarse grids on both sides of the lines between one launch and two (n = 255
    in FP32, n = 127 in FP64): FP32 against FP64 cycles from zero, 1e-4 (the
    bound the padded rows' cycles are held to)."""
    H = P.Hierarchy(n, N, inputs.draw_xi(N, N, 3), 1e-4, 0.5)
    g = torch.Generator(device="cuda").manual_seed(2)
    f = tuple(torch.randn(t.shape, generator=g, device="cuda").double() for t in H.zeros(0))
    x, a = H.zeros(0), H.zeros(0, torch.float32)
    H.cycle(P.CycleOptions(), x, f)
    H.cycle(P.CycleOptions(precision=P.FP32), a, tuple(t.float() for t in f))
    check(a, tuple(t.cpu().numpy() for t in x), 1e-4, "cycle")
    H.close()
