"""Channel counts outside the network's layers (csrc/nn_conv.cu): every multiple of 16
that the convolution primitive accepts, against 27 shifted FP64 matrix products.

The weight gradient sums B D^3 <= 1536 products in FP32 per element: relative error
(2-norm) of the order of 2^-24 times the square root of their number, 2e-6; 1e-5 as for
the network's own layers.  A guard behind dW and db shows a store beyond their ends."""
import ctypes as C

import pytest
import torch

from paper_1305_2418_gb300 import build, mgfr

pytestmark = pytest.mark.gpu

TAPS = [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)]


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU test run without a GPU"
    build.build()
    return torch.device("cuda:0")


def rel(a, b):
    return float((a.double() - b).norm() / b.norm())


def grads(X, G, ci, co):
    gf = G.double().reshape(-1, co)
    gw = torch.stack([torch.roll(X.double(), tuple(-q for q in d), (1, 2, 3)).reshape(-1, ci).T
                      @ gf for d in TAPS])
    return gw, gf.sum(0)


@pytest.mark.parametrize("B,D", [(1, 4), (3, 8)])
@pytest.mark.parametrize("ci,co", [(16, 48), (48, 48), (16, 80), (32, 96), (80, 112), (256, 112),
                                   (16, 128), (80, 64), (48, 32), (32, 16)])
def test_weight_gradient_of_any_channel_count(dev, B, D, ci, co):
    r = torch.Generator(device=dev).manual_seed(100 * ci + co + D)
    x = torch.randn((B, D, D, D, ci), generator=r, device=dev).to(torch.bfloat16)
    g = torch.randn((B, D, D, D, co), generator=r, device=dev).to(torch.bfloat16)
    nw = 27 * ci * co
    gw, db = torch.full((nw + 4096,), 7.0, device=dev), torch.full((co + 4096,), 7.0, device=dev)
    st = mgfr.lib().mgfr_nn_conv3d(
        2, B, D, ci, co, C.c_void_p(x.data_ptr()), None, None, 0, C.c_void_p(g.data_ptr()),
        C.c_void_p(gw.data_ptr()), C.c_void_p(db.data_ptr()),
        C.c_void_p(torch.cuda.current_stream(dev).cuda_stream))
    assert st == mgfr.MGFR_OK
    want_gw, want_db = grads(x, g, ci, co)
    got = gw[:nw].reshape(27, ci, co)
    assert rel(got, want_gw) <= 1e-5
    for c in range(0, co, 16):  # every group of output channels by itself
        assert rel(got[:, :, c:c + 16], want_gw[:, :, c:c + 16]) <= 1e-5, c
    assert rel(db[:co], want_db) <= 1e-5
    assert bool((gw[nw:] == 7.0).all()) and bool((db[co:] == 7.0).all())
