"""Every gradient of the warm-start network against the same chain built from
the exported layer kernels (im2col, GEMM, flip3x3, relu_bwd, upsample_bwd,
avgpool backward, add, outer), which store the same BF16 tensors between
layers: the forward activations and each layer's dZ are the same bits, so a
weight gradient is compared with the 64-bit sum of the same BF16 products.

Tolerances, per entry, against the sum of the products' magnitudes: a weight
gradient adds 4096 products (256 MMAs of 16) into one FP32 accumulator before
the slices are added, each step off by at most one truncation, 2^-23:
256 * 2^-23 = 3.1e-5, and up to 32 additions of slices and thread sums,
32 * 2^-24; a bias gradient at most 250 FP32 additions one after another,
1.5e-5.  A tile, a tap or a halo pixel left out moves an entry by its share of
the pixels, at these sizes 1e-4 and more.

Images: lower levels below one 8 x 16 tile (4 x 4), ragged in both
directions, slices of one tile, of several, and of the most (32)."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 256 * 2.0 ** -23 + 32 * 2.0 ** -24
V, I, Q = ctypes.c_void_p, ctypes.c_int, ctypes.c_longlong


@pytest.fixture(scope="module")
def mod():
    from paper_2302_13680_gb300 import build

    build.build()
    from paper_2302_13680_gb300 import learned

    return learned


class Layers:
    """The exported layer kernels on CUDA tensors, NHWC BF16."""

    ARGS = dict(im2col=[V, V, I, I, I, I, I, V], relu_bwd=[V, V, V, Q, V], avgpool=[V, V, I, I, I, I, I, V],
                upsample_add=[V, V, V, I, I, I, I, V], upsample_bwd=[V, V, I, I, I, I, V], add=[V, V, V, Q, V],
                outer=[V, V, V, Q, I, V], flip3x3=[V, V, I, I, V],
                gemm_bf16=[V, Q, V, Q, I, I, I, V, I, V, V, I, V, V])

    def __init__(self, lib):
        self.lib = lib
        self.stream = V(torch.cuda.current_stream().cuda_stream)
        self.status = torch.zeros(1, dtype=torch.int32, device="cuda")

    def call(self, name, *args):
        fn = getattr(self.lib, "cmg_nn_" + name)
        fn.restype, fn.argtypes = I, self.ARGS[name]
        assert fn(*[V(a.data_ptr()) if isinstance(a, torch.Tensor) else a for a in args], self.stream) == 0, name

    def new(self, *shape, dtype=torch.bfloat16):
        return torch.empty(*shape, dtype=dtype, device="cuda")

    def cols(self, X):
        B, H, W, C = X.shape
        col = self.new(B * H * W, 9 * C)
        self.call("im2col", X, col, B, H, W, C, 0)
        return col

    def gemm(self, A, W, bias, relu, dtype=torch.bfloat16):
        out = self.new(A.shape[0], W.shape[0], dtype=dtype)
        o32, o16 = (out, None) if dtype == torch.float32 else (None, out)
        self.call("gemm_bf16", A, A.shape[1], W, W.shape[1], A.shape[0], W.shape[0], A.shape[1], bias, relu, o32, o16,
                  W.shape[0], self.status)
        return out

    def conv(self, X, W, bias, relu):
        return self.gemm(self.cols(X), W, bias, relu).reshape(*X.shape[:3], -1)

    def data_grad(self, dZ, W):
        C = W.shape[1] // 9
        Wf = self.new(C, 9 * W.shape[0])
        self.call("flip3x3", W, Wf, W.shape[0], C)
        return self.conv(dZ, Wf, None, 0)

    def relu_bwd(self, y, dy):
        dz = torch.empty_like(y)
        self.call("relu_bwd", y, dy, dz, y.numel())
        return dz

    def pool(self, X):
        B, H, W, C = X.shape
        Y = self.new(B, H // 2, W // 2, C)
        self.call("avgpool", X, Y, B, H, W, C, 0)
        return Y

    def pool_bwd(self, dY, skip):
        B, H, W, C = skip.shape
        dX, out = torch.empty_like(skip), torch.empty_like(skip)
        self.call("avgpool", dY, dX, B, H, W, C, 1)
        self.call("add", dX, skip, out, skip.numel())
        return out

    def up_add(self, X, skip):
        Y = torch.empty_like(skip)
        self.call("upsample_add", X, skip, Y, *skip.shape)
        return Y

    def up_bwd(self, dY):
        B, H, W, C = dY.shape
        dX = self.new(B, H // 2, W // 2, C)
        self.call("upsample_bwd", dY, dX, B, H // 2, W // 2, C)
        return dX


def chain(k, par, X, dpred):
    """Prediction and, per layer, (input, gradient before its ReLU)."""
    a, inp = {}, {}

    def conv(name, x):
        inp[name] = x
        a[name] = k.conv(x, par[name][0], par[name][1], 1)
        return a[name]

    s0 = conv("c0b", conv("c0a", X))
    s1 = conv("c1b", conv("c1a", k.pool(s0)))
    s2 = conv("c2b", conv("c2a", k.pool(s1)))
    b3 = conv("c3b", conv("c3a", k.pool(s2)))
    e2 = conv("d2", k.up_add(b3, s2))
    e1 = conv("d1", k.up_add(e2, s1))
    e0 = conv("d0", k.up_add(e1, s0))
    w16, b, w32 = par["head"]
    pred = k.gemm(e0.reshape(-1, 32), w16, b, 0, torch.float32)
    dz = {}

    def back(name, dy, data=True):
        dz[name] = k.relu_bwd(a[name], dy)
        return k.data_grad(dz[name], par[name][0]) if data else None

    g = torch.empty_like(e0)
    k.call("outer", dpred, w32, g, dpred.numel(), 32)
    g0 = back("d0", g)
    g1 = back("d1", k.up_bwd(g0))
    g2 = back("d2", k.up_bwd(g1))
    p3 = back("c3a", back("c3b", k.up_bwd(g2)))
    p2 = back("c2a", back("c2b", k.pool_bwd(p3, g2)))
    p1 = back("c1a", back("c1b", k.pool_bwd(p2, g1)))
    back("c0a", back("c0b", k.pool_bwd(p1, g0)), data=False)
    return pred.reshape(dpred.shape), {n: (inp[n], dz[n]) for n in dz}, e0


def check(got, ref, size, what):
    assert bool(torch.isfinite(ref).all()) and float(size.max()) > 0.0, what
    worst = float(((got.double() - ref).abs() / size.clamp_min(1e-300)).max())
    assert worst <= TOL, (what, worst)


@pytest.mark.parametrize("S,B", [(32, 1), (32, 3), (96, 2), (160, 1), (64, 8), (256, 10)])
def test_gradients_equal_the_sums_of_their_products(mod, S, B):
    net = mod.WarmStartNet(S=S, batch=B, seed=S)
    k = Layers(net.lib)
    g = torch.Generator().manual_seed(S + B)
    net.set("head", "w", (torch.randn(1, 32, generator=g) * 0.2).numpy())
    par = {}
    for name in mod.LAYERS:
        net.set(name, "b", (torch.randn(net.shape(name)[0], generator=g) * 0.05).numpy())
        par[name] = [torch.tensor(net.get(name, "w16")).bfloat16().cuda(), torch.tensor(net.get(name, "b")).cuda(),
                     torch.tensor(net.get(name, "w")).cuda()]
    X = torch.randn(B, S, S, 8, generator=g).bfloat16().cuda()
    dpred = torch.randn(B, S, S, generator=g).bfloat16().cuda()
    pred, layers, e0 = chain(k, par, X, dpred)
    got = net.forward(X)
    net.backward(dpred)
    torch.cuda.synchronize()
    net.check_status()
    assert int(k.status.item()) == 0
    assert torch.equal(got, pred)
    for name, (x, dz) in layers.items():
        gw = size = gb = sb = 0.0
        for b in range(B):   # an image at a time: the 64-bit patch matrices are large
            col, z = k.cols(x[b:b + 1]).double(), dz[b].reshape(-1, dz.shape[-1]).double()
            gw, size = gw + z.T @ col, size + z.abs().T @ col.abs()
            gb, sb = gb + z.sum(0), sb + z.abs().sum(0)
        check(torch.tensor(net.get(name, "gw")).cuda(), gw, size, name + " weights")
        check(torch.tensor(net.get(name, "gb")).cuda(), gb, sb, name + " bias")
    d, y = dpred.reshape(-1, 1).double(), e0.reshape(-1, 32).double()
    check(torch.tensor(net.get("head", "gw")).cuda(), d.T @ y, d.abs().T @ y.abs(), "head weights")
    check(torch.tensor(net.get("head", "gb")).cuda(), d.sum(0), d.abs().sum(0), "head bias")
    net.close()
