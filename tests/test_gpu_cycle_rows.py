"""FP32 cycles on a caller's vectors where the handle pads its rows (N >= 9, not
a multiple of four): on small grids on rows of N throughout, without copies;
above by copies into padded rows.  Same results, no more launches than the
cycle has steps, and a later padded solve does not see what such a cycle left
in the handle's vectors.

Tolerance 1e-4 of each block's largest entry, as FP32 against FP64 cycles in
the padding tests; every block must be finite."""
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu
CYCLES = [dict(), dict(gamma=2, n1=1, n2=1), dict(smoother=1), dict(tail_n=15), dict(freeze_u=1)]
IDS = ["V22", "W11", "jacobi", "tail", "frozen"]


@pytest.fixture(scope="module")
def P():
    from paper_2302_13680_gb300 import build

    build.build()
    import paper_2302_13680_gb300 as P

    return P


def vectors(H, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return tuple(torch.randn(t.shape, generator=g, device="cuda") for t in H.zeros(0))


def close(got, ref, tol):
    for name, a, b in zip("yup", got, ref):
        e = float((a.double() - b).abs().max() / b.abs().max())
        assert e <= tol, (name, e)   # false for a NaN


@pytest.mark.parametrize("n,N", [(7, 9), (15, 27), (15, 66), (15, 67), (31, 41), (63, 62), (63, 63)])
@pytest.mark.parametrize("kw", CYCLES, ids=IDS)
@pytest.mark.parametrize("box", [None, (0.25, 0.75, 0.25, 0.75)], ids=["all", "local"])
def test_cycle_equals_fp64_cycle(P, n, N, kw, box):
    H = P.Hierarchy(n, N, inputs.draw_xi(N, N, 4), 1e-4, 0.5, control_box=box)
    x, f = vectors(H, n), vectors(H, N)
    x64, f64 = tuple(t.double() for t in x), tuple(t.double() for t in f)
    for _ in range(2):
        H.cycle(P.CycleOptions(precision=P.FP32, **kw), x, f)
        H.cycle(P.CycleOptions(**kw), x64, f64)
    close(x, x64, 1e-4)
    H.close()


@pytest.mark.parametrize("n,N", [(7, 9), (15, 65), (63, 27)])
def test_small_cycle_makes_no_copies(P, n, N):
    from paper_2302_13680_gb300.cmg import kernel_launches

    count = []
    for samples in (N, 4 * ((N + 3) // 4)):
        H = P.Hierarchy(n, samples, inputs.draw_xi(1, samples, 4), 1e-4, 0.5)
        x, f = vectors(H, 1), vectors(H, 2)
        H.cycle(P.CycleOptions(precision=P.FP32), x, f)
        before = kernel_launches()
        H.cycle(P.CycleOptions(precision=P.FP32), x, f)
        count.append(kernel_launches() - before)
        H.close()
    assert count[0] <= count[1]


@pytest.mark.parametrize("coarsest_n", [1, 3, 7])
@pytest.mark.parametrize("tail_n", [0, 15])
def test_padded_solve_after_a_cycle_on_rows_of_n(P, coarsest_n, tail_n):
    """Coarsest grids of 1, 9 and 49 nodes (the last by two kernels): the solve's
    iterates are the same bits before and after cycles that leave NaN or large
    values in the handle's vectors."""
    n, N = 31, 27
    pr = inputs.make_problem(n=n, N=N, K=4, nu=1e-4, amp=0.5, seed=N, target="modes")
    H = P.Hierarchy(n, N, pr.xi, pr.nu, pr.amp, coarsest_n=coarsest_n)
    f = H.rhs(torch.tensor(pr.yd.reshape(-1), device="cuda"))
    opts = P.CycleOptions(precision=P.FP32, tail_n=tail_n)
    sols = []
    for fill in (None, float("nan"), 1e20):
        if fill is not None:
            v = tuple(torch.full_like(t, fill, dtype=torch.float32) for t in f)
            for kw in CYCLES:
                H.cycle(P.CycleOptions(precision=P.FP32, **kw), tuple(t.clone() for t in v), v)
        x = H.zeros(0)
        H.solve(opts, f, x, tol=1e-15, maxit=3, raise_on_fail=False)
        sols.append(x)
    for x in sols[1:]:
        assert all(torch.equal(a, b) for a, b in zip(x, sols[0]))
    H.close()


@pytest.mark.parametrize("N", [9, 27, 125, 130])
@pytest.mark.parametrize("method", ["cycle", "fgmres"])
def test_refined_solution_block_by_block(P, N, method):
    """FP32 cycles on padded rows inside FP64 refinement or FGMRES, to 1e-11:
    every block within 1e-8 of the FP64 solution."""
    pr = inputs.make_problem(n=31, N=N, K=4, nu=1e-4, amp=0.5, seed=N, target="modes")
    H = P.Hierarchy(31, N, pr.xi, pr.nu, pr.amp)
    f = H.rhs(torch.tensor(pr.yd.reshape(-1), device="cuda"))
    x, ref = H.zeros(0), H.zeros(0)
    H.solve(P.CycleOptions(), f, ref, tol=1e-11)
    H.solve(P.CycleOptions(precision=P.FP32), f, x, method=P.METHOD_FGMRES if method == "fgmres" else P.METHOD_CYCLE,
            tol=1e-11)
    close(x, ref, 1e-8)
    H.close()
