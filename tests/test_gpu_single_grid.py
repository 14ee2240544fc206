"""A Galerkin handle of a single grid (n = coarsest_n) has no coarse operators:
its operator, cycle and solves are the 5-point problem's, bit for bit those of
the other coarse rules, and what Galerkin handles refuse stays refused."""
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2302_13680_gb300 import build

    build.build()
    import paper_2302_13680_gb300 as P

    return P


@pytest.mark.parametrize("n,N", [(3, 5), (3, 64), (7, 9), (7, 130)])
@pytest.mark.parametrize("fp32", [False, True])
def test_single_galerkin_grid(P, n, N, fp32):
    pr = inputs.make_problem(n=n, N=N, K=3, nu=1e-3, amp=0.5, seed=N, target="modes")
    prec, dt = (P.FP32, torch.float32) if fp32 else (P.FP64, torch.float64)
    out = []
    for coarse in ("averaged", "galerkin"):
        H = P.Hierarchy(n, N, pr.xi, pr.nu, pr.amp, coarsest_n=n, coarse=coarse)
        g = torch.Generator(device="cuda").manual_seed(n)
        f = tuple(torch.randn(t.shape, generator=g, device="cuda").to(dt) for t in H.zeros(0))
        x, r, y, z = H.zeros(0, dt), H.zeros(0, dt), H.zeros(0, dt), H.zeros(0)
        H.cycle(P.CycleOptions(precision=prec), x, f)
        H.residual(0, x, f, r)
        H.coarse_solve(f, y)
        b = H.rhs(torch.tensor(pr.yd.reshape(-1), device="cuda"))
        st, _ = H.solve(P.CycleOptions(precision=prec), b, z, tol=1e-11)
        assert st.relres <= 1e-11
        if coarse == "galerkin":
            with pytest.raises(P.CMGError):
                H.ssn_solve(P.CycleOptions(precision=prec), torch.zeros(n * n, dtype=torch.float64, device="cuda"),
                            z[1].clone(), 1e-2, -1.0, 1.0)
        out.append([*x, *r, *y, *z])
        H.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
