"""Direct coarsest solves with the solution written over the right side: the
same bits as into a separate vector.

The cluster kernel (grids of up to 12 nodes) spreads the samples over eight
CTAs that all need the control block of the right side, which one of them
overwrites, as does the two-kernel form of the square's problem (49 nodes, or more
samples than one CTA's shared memory holds); repeated, since a late reader
would see it only now and then.  Sample counts below, at and above one per
CTA, and the single-CTA kernels."""
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


@pytest.mark.parametrize("coarsest_n,N", [(1, 1), (1, 40), (3, 3), (3, 8), (3, 125), (3, 1024), (7, 12)])
def test_boundary_coarsest_solve_in_place(P, coarsest_n, N):
    n = 2 * coarsest_n + 1
    H = P.BoundaryHierarchy(n, N, inputs.draw_xi(N, N, 3), 1e-3, 0.8, coarsest_n=coarsest_n)
    single = P.BoundaryHierarchy(coarsest_n, N, inputs.draw_xi(N, N, 3), 1e-3, 0.8, coarsest_n=coarsest_n)
    for _ in range(20):
        f = tuple(torch.randn_like(t) for t in H.zeros(1))
        x = H.zeros(1)
        H.coarse_solve(f, x)
        over = tuple(t.clone() for t in f)
        H.coarse_solve(over, over)
        assert all(torch.equal(a, b) for a, b in zip(over, x))
        # on a single grid the cycle is that solve
        y, over = single.zeros(0), tuple(t.clone() for t in f)
        single.cycle(y, f)
        single.cycle(over, over)
        assert all(torch.equal(a, b) for a, b in zip(over, y))
    H.close()
    single.close()


@pytest.mark.parametrize("coarsest_n,N", [(1, 5), (3, 9), (3, 216), (3, 256), (3, 500), (7, 5), (7, 130), (7, 500)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["fp64", "fp32"])
def test_coarsest_solve_in_place(P, coarsest_n, N, dtype):
    n = 2 * coarsest_n + 1
    H = P.Hierarchy(n, N, inputs.draw_xi(N, N, 3), 1e-3, 0.8, coarsest_n=coarsest_n)
    single = P.Hierarchy(coarsest_n, N, inputs.draw_xi(N, N, 3), 1e-3, 0.8, coarsest_n=coarsest_n) if coarsest_n > 1 else None
    opts = P.CycleOptions(precision=P.FP32 if dtype == torch.float32 else P.FP64)
    for _ in range(20):
        f = tuple(torch.randn_like(t) for t in H.zeros(1, dtype))
        x, over = H.zeros(1, dtype), tuple(t.clone() for t in f)
        H.coarse_solve(f, x)
        H.coarse_solve(over, over)
        assert all(torch.equal(a, b) for a, b in zip(over, x))
        if single is None:
            continue
        y, over = single.zeros(0, dtype), tuple(t.clone() for t in f)
        single.cycle(opts, y, f)
        single.cycle(opts, over, over)
        assert all(torch.equal(a, b) for a, b in zip(over, y))
    H.close()
