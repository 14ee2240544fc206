"""Bounded waits of the patch convolution, the weight gradient and the head
(cmg_nn_conv.cu), through the C ABI.

With one poll per wait every launch gives up, drains what it has in flight,
frees its tensor memory and sets its status word; with the default limit the
same context then computes the right results.  The polls are for the launch's
own copies: time spent behind a preceding kernel of the stream does not count
(measured, first layer's shape: 8 polls suffice alone, and behind a kernel of
200 us 32 did not while the MMA thread polled through it; held to 16)."""
import ctypes

import pytest
import torch

from test_gpu_nn_conv import data, lib, ptr  # noqa: F401  (module fixture)

pytestmark = pytest.mark.gpu


@pytest.fixture
def limit(lib):  # noqa: F811
    fn = lib.cmg_nn_set_wait_limit
    fn.restype, fn.argtypes = ctypes.c_int, [ctypes.c_longlong]

    def put(polls):
        assert fn(polls) == 0

    yield put
    put(0)


class Conv:
    def __init__(self, lib, B, H, W, C, Cout):  # noqa: F811
        self.lib, self.dim = lib, (B, H, W, C, Cout)
        X, Wt, bias = data(B, H, W, C, Cout, seed=C)
        self.X, self.Wt, self.bias = X.cuda(), Wt.cuda(), bias.cuda()
        self.Y = torch.zeros(B * H * W, Cout, dtype=torch.bfloat16, device="cuda")
        self.status = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def run(self):
        B, H, W, C, Cout = self.dim
        assert self.lib.cmg_nn_conv3x3_bf16(ptr(self.X), B, H, W, C, ptr(self.Wt), Cout, ptr(self.bias), 1, ptr(self.Y),
                                            ptr(self.status), self.s) == 0

    def expected(self):
        B, H, W, C, Cout = self.dim
        col = torch.empty(B * H * W, 9 * C, dtype=torch.bfloat16, device="cuda")
        Y = torch.empty_like(self.Y)
        st = torch.zeros_like(self.status)
        assert self.lib.cmg_nn_im2col(ptr(self.X), ptr(col), B, H, W, C, 0, self.s) == 0
        assert self.lib.cmg_nn_gemm_bf16(ptr(col), 9 * C, ptr(self.Wt), 9 * C, B * H * W, Cout, 9 * C, ptr(self.bias), 1,
                                         None, ptr(Y), Cout, ptr(st), self.s) == 0
        return Y


@pytest.mark.parametrize("C,Cout", [(8, 32), (32, 64), (64, 64)])
def test_exhausted_convolution_sets_status_and_context_survives(lib, limit, C, Cout):  # noqa: F811
    k = Conv(lib, 2, 128, 128, C, Cout)
    torch.cuda.synchronize()
    limit(1)
    k.run()
    torch.cuda.synchronize()
    limit(0)
    assert int(k.status.item()) == 1
    k.status.zero_()
    k.run()
    ref = k.expected()
    torch.cuda.synchronize()
    assert int(k.status.item()) == 0
    assert torch.equal(k.Y, ref)


@pytest.mark.parametrize("where", ["forward", "backward"])
def test_exhausted_network_reports_and_a_new_handle_works(lib, limit, where):  # noqa: F811
    from paper_2302_13680_gb300 import learned
    from paper_2302_13680_gb300.cmg import CMGError

    g = torch.Generator().manual_seed(1)
    X = torch.randn(4, 64, 64, 8, generator=g).bfloat16().cuda()
    d = torch.randn(4, 64, 64, generator=g).bfloat16().cuda()

    def step(polls_forward=0, polls_backward=0):
        net = learned.WarmStartNet(S=64, batch=4, seed=5)
        net.set("head", "w", torch.linspace(-0.3, 0.3, 32).reshape(1, 32).numpy())
        try:
            limit(polls_forward)
            pred = net.forward(X)
            limit(polls_backward)
            net.backward(d)
            torch.cuda.synchronize()
            limit(0)
            net.check_status()
            return [pred] + [torch.tensor(net.get(k, w)) for k in learned.LAYERS for w in ("gw", "gb")]
        finally:
            net.close()

    before = step()
    with pytest.raises(CMGError):
        step(**{"polls_" + where: 1})
    assert all(torch.equal(a, b) for a, b in zip(before, step()))


def test_polls_are_not_spent_behind_the_preceding_kernel(lib, limit):  # noqa: F811
    long, short = Conv(lib, 64, 256, 256, 8, 32), Conv(lib, 1, 16, 16, 8, 32)
    torch.cuda.synchronize()
    for _ in range(10):
        limit(0)
        long.run()
        limit(16)
        short.run()
        torch.cuda.synchronize()
    limit(0)
    assert int(long.status.item()) == 0
    assert int(short.status.item()) == 0
    assert torch.equal(short.Y, short.expected())
