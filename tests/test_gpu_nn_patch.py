"""The patch convolution (cmg_nn_conv.cu) where its 8 x 16 pixel tiles, its
channel padding and its stores can go wrong: images smaller than a tile,
ragged in both directions, exactly one tile, single rows and columns, output
counts that leave 16-byte chunks, sectors or the MMA width unfilled, no bias.
The same products are summed in the same order as by im2col + GEMM, so the
results are the same bits; rows past the output stay untouched."""
import ctypes

import pytest
import torch

from test_gpu_nn_conv import data, lib, ptr  # noqa: F401  (module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [8, 32, 64])
@pytest.mark.parametrize("B,H,W,Cout", [(1, 1, 1, 5), (3, 16, 8, 32), (2, 17, 9, 64), (1, 15, 23, 24), (2, 33, 7, 40),
                                        (1, 2, 50, 1), (1, 129, 65, 48), (40, 48, 24, 33)])
def test_patch_conv_edges(lib, B, H, W, C, Cout):  # noqa: F811
    X, Wt, bias = data(B, H, W, C, Cout, seed=H * 100 + W + C + Cout)
    P = B * H * W
    Xd, Wd, bd = X.cuda(), Wt.cuda(), (bias.cuda() if Cout % 3 else None)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    Y = torch.full((P + 4, Cout), 7.0, dtype=torch.bfloat16, device="cuda")
    assert lib.cmg_nn_conv3x3_bf16(ptr(Xd), B, H, W, C, ptr(Wd), Cout, ptr(bd), 1, ptr(Y), ptr(status), s) == 0
    col = torch.empty(P, 9 * C, dtype=torch.bfloat16, device="cuda")
    Y2 = torch.empty(P, Cout, dtype=torch.bfloat16, device="cuda")
    assert lib.cmg_nn_im2col(ptr(Xd), ptr(col), B, H, W, C, 0, s) == 0
    assert lib.cmg_nn_gemm_bf16(ptr(col), 9 * C, ptr(Wd), 9 * C, P, Cout, 9 * C, ptr(bd), 1, None, ptr(Y2), Cout,
                                ptr(status), s) == 0
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert torch.equal(Y[:P], Y2)
    assert bool((Y[P:] == 7.0).all())


@pytest.mark.parametrize("S,B", [(96, 1), (160, 2)])
def test_gradients_on_ragged_tiles(S, B):
    """Prediction, loss and every gradient on resolutions whose lower levels
    (12, 24, 20, 40) leave the tiles' rows or columns unfilled, against
    automatic differentiation of the float64 oracle: norm-wise within the
    bounds that BF16 storage gives at any size (3 % forward, 6 % gradients)."""
    import oracle.unet_oracle as U
    from paper_2302_13680_gb300 import learned

    g = torch.Generator().manual_seed(S)
    X = torch.zeros(B, S, S, 8)
    X[..., :2] = torch.randn(B, S, S, 2, generator=g)
    X, tgt, m = X.to(torch.bfloat16), torch.randn(B, S, S, generator=g), S - 1
    net = learned.WarmStartNet(S=S, batch=B + 1, seed=3)
    try:
        net.set("head", "w", (torch.randn(1, 32, generator=g) * 0.2).numpy())
        for k in learned.LAYERS[:-1]:
            rows, _ = net.shape(k)
            net.set(k, "b", (torch.randn(rows, generator=g) * 0.05).numpy())
        pred = net.forward(X.cuda())
        loss = float(net.loss(tgt.cuda(), m))
        net.backward()
        net.check_status()
        params = {k: (torch.tensor(net.get(k, "w16"), dtype=torch.float64).requires_grad_(True),
                      torch.tensor(net.get(k, "b"), dtype=torch.float64).requires_grad_(True)) for k in learned.LAYERS}
        ref = U.forward(params, X.double())
        ref_loss = U.masked_mse(ref, tgt.double(), m)
        ref_loss.backward()
        rel = lambda a, b: float(torch.linalg.norm(a - b) / torch.linalg.norm(b))  # noqa: E731
        assert rel(pred.double().cpu(), ref.detach()) <= 3e-2
        assert abs(loss - float(ref_loss.detach())) <= 3e-2 * float(ref_loss.detach())
        for k in learned.LAYERS:
            assert rel(torch.tensor(net.get(k, "gw"), dtype=torch.float64), params[k][0].grad) <= 6e-2, k
            assert rel(torch.tensor(net.get(k, "gb"), dtype=torch.float64), params[k][1].grad) <= 6e-2, k
    finally:
        net.close()
