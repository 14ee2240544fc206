"""Sample counts that are not a multiple of four: the handle's FP32 arrays have
padded rows (up to three samples with stiff faces and zero data per node).
FP32 cycles against FP64 cycles on the same inputs, and refined solutions
against FP64 ones, over every remainder, both smoothers, V and W, the cluster
tail, local control, FP32-preconditioned FGMRES, nodal coarse grids (not
padded) and a handle reused after a failed (NaN) cycle.

Tolerances: FP32 cycles 1e-4 of each block's largest entry (the bound the
FP32 Galerkin cycles are held to); solutions at relative residual 1e-11
within 1e-8 (the FP64 solve's own bound in the full-size test is 1e-9)."""
import numpy as np
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu
NS = [8, 9, 10, 11, 13, 27, 125, 130]


@pytest.fixture(scope="module")
def P():
    from paper_2302_13680_gb300 import build

    build.build()
    import paper_2302_13680_gb300 as P

    return P


def rel(a, b):
    return max(float((x.double() - y.double()).abs().max() / y.double().abs().max()) for x, y in zip(a, b))


@pytest.mark.parametrize("N", NS)
@pytest.mark.parametrize("kw", [dict(), dict(gamma=2, n1=1, n2=1), dict(smoother=1), dict(tail_n=15)],
                         ids=["V22", "W11", "jacobi", "tail"])
def test_fp32_cycle_equals_fp64_cycle(P, N, kw):
    n = 31
    for box in (None, (0.25, 0.75, 0.25, 0.75)):
        H = P.Hierarchy(n, N, inputs.draw_xi(N, N, 4), 1e-4, 0.5, control_box=box)
        g = torch.Generator(device="cuda").manual_seed(N)
        f = tuple(torch.randn(t.shape, generator=g, device="cuda").double() for t in H.zeros(0))
        x64 = tuple(torch.randn(t.shape, generator=g, device="cuda").double() for t in f)
        x32, f32 = tuple(t.float() for t in x64), tuple(t.float() for t in f)
        nan = tuple(torch.full_like(t, float("nan")) for t in f32)
        H.cycle(P.CycleOptions(precision=P.FP32, **kw), nan, f32)   # leaves NaN in the handle's work vectors
        H.cycle(P.CycleOptions(precision=P.FP32, **kw), x32, f32)
        H.cycle(P.CycleOptions(**kw), x64, f)
        assert rel(x32, x64) <= 1e-4
        H.close()


@pytest.mark.parametrize("N", NS)
@pytest.mark.parametrize("coarse", ["averaged", "nodal"])
def test_refined_solution_equals_fp64(P, N, coarse):
    n = 31
    pr = inputs.make_problem(n=n, N=N, K=4, nu=1e-4, amp=0.5, seed=N, target="modes")
    H = P.Hierarchy(n, N, pr.xi, pr.nu, pr.amp, coarse=coarse)
    f = H.rhs(torch.tensor(pr.yd.reshape(-1), device="cuda"))
    ref = H.zeros(0)
    H.solve(P.CycleOptions(), f, ref, tol=1e-11)
    for opts, method in ((P.CycleOptions(precision=P.FP32), P.METHOD_CYCLE),
                         (P.CycleOptions(precision=P.FP32, tail_n=15), P.METHOD_CYCLE),
                         (P.CycleOptions(precision=P.FP32, ctl32=1), P.METHOD_CYCLE),
                         (P.CycleOptions(precision=P.FP32), P.METHOD_FGMRES)):
        for _ in range(2):   # the second solve reuses the captured loop and the work vectors
            x = H.zeros(0)
            st, _ = H.solve(opts, f, x, method=method, tol=1e-11)
            assert rel(x, ref) <= 1e-8, (opts, method)
    H.close()
