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


def at_offset(t, values):
    """The same values `values` elements off a fresh buffer's start (256-byte aligned)."""
    flat = torch.empty(t.numel() + values, dtype=t.dtype, device=t.device)
    v = flat[values:].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("off", [1, 2, 3, 7, 8])
@pytest.mark.parametrize("ci,co", [(80, 32), (16, 48), (48, 64)])
def test_gradients_of_views_at_any_element(dev, off, ci, co):
    """Op 2 outside the network's pairs reads x and g value by value: views at any element
    are accepted, and give what the aligned tensors give, bit by bit."""
    r = torch.Generator(device=dev).manual_seed(off + co)
    x = torch.randn((2, 8, 8, 8, ci), generator=r, device=dev).to(torch.bfloat16)
    g = torch.randn((2, 8, 8, 8, co), generator=r, device=dev).to(torch.bfloat16)
    w = torch.zeros((27, ci, co), dtype=torch.bfloat16, device=dev)
    want_db, db = torch.empty(co, device=dev), torch.empty(co, device=dev)
    want = mgfr.conv3d(2, x, w, g=g, db=want_db)
    got = mgfr.conv3d(2, at_offset(x, off), w, g=at_offset(g, off), db=db)
    assert torch.equal(got, want) and torch.equal(db, want_db)
    assert rel(db, g.double().reshape(-1, co).sum(0)) <= 1e-5


@pytest.mark.parametrize("ci,co,need", [(16, 16, 8), (96, 32, 8), (80, 32, 2)])
def test_misaligned_tensors_are_refused(dev, ci, co, need):
    """`need`: the elements of BF16 that the kernels load at a time."""
    x = torch.zeros((1, 16, 16, 16, ci), dtype=torch.bfloat16, device=dev)
    g = torch.zeros((1, 16, 16, 16, co), dtype=torch.bfloat16, device=dev)
    w = torch.zeros((27, ci, co), dtype=torch.bfloat16, device=dev)
    for off in (1, need // 2, need - 1):
        for call in (lambda: mgfr.conv3d(0, at_offset(x, off), w),
                     lambda: mgfr.conv3d(1, x, w, g=at_offset(g, off))):
            with pytest.raises(mgfr.MGFRError):
                call()
        if need == 8:
            for a, b in ((at_offset(x, off), g), (x, at_offset(g, off))):
                with pytest.raises(mgfr.MGFRError):
                    mgfr.conv3d(2, a, w, g=b)
    assert float(mgfr.conv3d(0, at_offset(x, need), w).abs().max()) == 0.0
