"""Launch-shape targets take effect where cmg.h says they do."""
import numpy as np
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


def lane_sum(p, lanes, width, chunks):
    """sum_j p[:, j] in the node kernels' order: a lane adds its chunks' samples
    one after another, then the lanes pairwise at half the distance each time."""
    nodes, N = p.shape
    v = np.zeros((nodes, lanes))
    for s in range(chunks):
        for k in range(width):
            for lane in range(lanes):
                j = (lane + s * lanes) * width + k
                if j < N:
                    v[:, lane] += p[:, j]
    while v.shape[1] > 1:
        h = v.shape[1] // 2
        v = v[:, :h] + v[:, h:]
    return v[:, 0]


@pytest.mark.parametrize("N", [64, 45])
@pytest.mark.parametrize("target", [1, 2, 4])
def test_fp64_residual_takes_the_grid_s_target(P, N, target):
    """The control row of S (0, 0, p) is -h^2 sum_j p_j, bit for bit in the
    order of the map that the target asks for."""
    from paper_2302_13680_gb300.cmg import sample_map

    n = 31
    H = P.Hierarchy(n, N, inputs.draw_xi(1, N, 3), 1e-3, 0.5)
    H.set_tuning(P.FP64, [target] * (H.levels - 1) + [0])
    x, r = H.zeros(0), H.zeros(0)
    x[2].normal_(generator=torch.Generator(device="cuda").manual_seed(N))
    H.residual(0, x, None, r)
    ref = lane_sum(x[2].cpu().numpy(), *sample_map(N, 8, n * n, target))
    assert np.array_equal(r[1].cpu().numpy(), -ref / (n + 1) ** 2)
    H.close()


@pytest.mark.parametrize("n,N,fp32,margin", [(511, 256, True, 1.03), (255, 64, True, 1.1), (255, 64, False, 1.06),
                                             (127, 54, True, 1.1)])
def test_autotuned_cycle_is_not_slower_than_the_default(P, n, N, fp32, margin):
    """The size rule is one of the tuner's candidates and all are judged on the
    cycle's launches, so a tuned V(2,2) cycle takes at most the default's time:
    medians of nine alternating measurements and a margin for their spread (below
    1 % where the kernels' time dominates the launches')."""
    H = P.Hierarchy(n, N, inputs.draw_xi(1, N, 8), 1e-5, 1.0)
    prec, dt = (P.FP32, torch.float32) if fp32 else (P.FP64, torch.float64)
    chosen = H.autotune(prec)
    opts, x = P.CycleOptions(precision=prec), H.zeros(0, dt)
    f = tuple(torch.randn_like(t) for t in x)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    times = {True: [], False: []}
    for i in range(20):
        H.set_tuning(prec, chosen if i % 2 else None)
        H.cycle(opts, x, f)
        ev[0].record()
        for _ in range(5):
            H.cycle(opts, x, f)
        ev[1].record()
        ev[1].synchronize()
        if i > 1:
            times[bool(i % 2)].append(ev[0].elapsed_time(ev[1]))
        for t in x:
            t.zero_()
    H.close()
    assert chosen[-1] == 0 and all((t & ~64) in (0, 1, 2, 4, 17, 18, 33) for t in chosen)
    assert np.median(times[True]) <= margin * np.median(times[False]), (chosen, times)
