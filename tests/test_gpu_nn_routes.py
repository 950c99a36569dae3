"""The routes of the network's layers at the sizes where they change, against
the FP64 oracle: images whose levels run on the tensor-core convolution, on
the warp-level one and on both, the weight copies that each reads after an
update, output channels that are no whole groups of 16, and the bias gradient
over one to ten groups.

Tolerances as in the tests of single layers (FP32 accumulation of BF16-exact
inputs, 1e-5; a BF16 output 8e-3) and of the whole network (BF16 activations
and gradients of 23 layers: forward 3e-2, gradient 8e-2 in L2)."""
import ctypes

import numpy as np
import pytest

import lbib_inputs as li

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1503_06726_gb300 import build, lbib
    build.build()
    lbib.load()
    return lbib


def bf16(shape, seed, scale=1.0):
    import torch
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(*shape, generator=g) * scale).to(torch.bfloat16)


def f64(t):
    return t.float().numpy().astype(np.float64)


def rel_inf(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# rows of 128 .. 4 pixels: tensor cores at the first level, one output channel written;
# 160 .. 5: the warp-level kernel first (its 16 output channels) and last;
# 64 .. 2 with more rows than columns
@pytest.mark.parametrize("H,W", [(32, 128), (64, 160), (96, 64)])
def test_network_after_an_update_matches_oracle(lb, H, W):
    import torch
    from oracle import nn as onn
    n = 2
    rng = np.random.default_rng(8)
    net = lb.NeuralOperator(n, H, W)
    p = li.nop_init_params(21, onn.nop_shapes())
    net.set_params((p + 0.01 * rng.normal(size=p.size)).astype(np.float32))
    mask = (rng.uniform(size=(n, H, W)) < 0.5).astype(np.uint8)
    src = (mask * (rng.uniform(size=(n, H, W)) < 0.3)).astype(np.uint8)
    D, k, s = rng.uniform(0.05, 0.2, n), rng.uniform(1e-4, 1e-2, n), np.full(n, 1e-3)
    phi = rng.uniform(0, 1, (n, H, W)) * (s / k)[:, None, None]
    dm, ds = torch.from_numpy(mask).cuda(), torch.from_numpy(src).cuda()
    dphi = torch.from_numpy(phi.astype(np.float32)).cuda()
    net.train_step(dm, ds, D, k, s, dphi, lr=1e-3)  # the copies are made anew
    rnd = lambda a: torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16) \
        .double().numpy()
    x = onn.features(mask, src, D, k)
    x[..., 2:] = rnd(x[..., 2:])
    y, cache = onn.forward(rnd(net.get_params()), x)
    out = net.forward(dm, ds, D, k, s).cpu().numpy()
    assert rel_l2(out, y[..., 0] * (s / k)[:, None, None]) < 3e-2
    loss = net.train_step(dm, ds, D, k, s, dphi, update=False)
    rloss, dy = onn.loss(y, (phi * (k / s)[:, None, None])[..., None])
    assert loss == pytest.approx(rloss, rel=5e-2)
    assert rel_l2(net.get_grads().astype(np.float64), onn.backward(dy, cache)) < 8e-2
    net.close()


@pytest.mark.parametrize("H,W,Ci,Co", [(8, 128, 32, 1), (6, 32, 16, 24), (5, 8, 32, 40),
                                       (4, 256, 16, 7), (8, 16, 32, 48)])
def test_output_channel_remainders(lb, orc, H, W, Ci, Co):
    import torch
    L, N = lb.load(), 2
    x, w = bf16((N, H, W, Ci), 1), bf16((3, 3, Ci, Co), 2, 0.1)
    bias = torch.randn(Co, generator=torch.Generator().manual_seed(3))
    st = torch.cuda.current_stream().cuda_stream
    wf = w.permute(0, 1, 3, 2).reshape(9, Co, Ci).contiguous().cuda()
    nb = ctypes.c_uint64(0)
    assert L.lbib_nn_tile_weights_tc(Ci, Co, None, None, ctypes.byref(nb), st) == 0
    wt = torch.empty(int(nb.value), dtype=torch.bfloat16, device="cuda")
    assert L.lbib_nn_tile_weights_tc(Ci, Co, wf.data_ptr(), wt.data_ptr(), None, st) == 0
    dx, dbias = x.cuda(), bias.cuda()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = orc.conv3x3(f64(x), f64(w), bias.double().numpy())
    for dtype, f32, tol in ((torch.float32, 1, 1e-5), (torch.bfloat16, 0, 8e-3)):
        buf = torch.full((N * H * W * Co + 16,), 7.0, dtype=dtype, device="cuda")
        n = N * H * W * Co
        call = lambda out: L.lbib_nn_conv3x3_tc(N, H, W, Ci, 0, Co, dx.data_ptr(), None,
                                                wt.data_ptr(), dbias.data_ptr(), out, 0, f32,
                                                err.data_ptr(), st)
        assert call(buf.data_ptr() + buf.element_size()) == -1  # off the 16-byte boundary
        assert call(buf.data_ptr()) == 0
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        assert rel_inf(f64(buf[:n].float().cpu()).reshape(N, H, W, Co), ref) < tol
        assert (buf[n:] == 7).all()


@pytest.mark.parametrize("H,W,Co", [(5, 128, 16), (8, 32, 80), (6, 16, 112), (4, 256, 160)])
def test_bias_gradient_groups(lb, orc, H, W, Co):
    import torch
    L, N, Ci = lb.load(), 2, 48
    x, g = bf16((N, H, W, Ci), 4), bf16((N, H, W, Co), 5)
    dx, dg = x.cuda(), g.cuda()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    dw = torch.zeros((9, Ci, Co), device="cuda")
    db = torch.zeros(Co, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    assert L.lbib_nn_conv3x3_wgrad_tc(N, H, W, Ci, 0, Co, dx.data_ptr(), None, dg.data_ptr(),
                                      dw.data_ptr(), db.data_ptr(), err.data_ptr(), st) == 0
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    rw, rb = orc.conv3x3_wgrad(f64(x), f64(g))
    assert rel_inf(dw.cpu().numpy().reshape(3, 3, Ci, Co), rw) < 1e-5
    assert rel_inf(db.cpu().numpy(), rb) < 1e-5
