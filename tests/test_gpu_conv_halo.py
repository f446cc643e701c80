"""Convolution kernels on resident blocks (csrc/nn_tc.cu) against 27 shifted FP64
matrix products, at the smallest grid of the blocks (16^3: one block per axis or
two, so every halo wraps), at 32^3, and for several samples.

Forward and input gradient accumulate 27 Cin (27 Cout) products in FP32, the
weight gradient B D^3: relative error (2-norm) below 2^-24 times the square root
of the number of terms, 1e-5 at 32768 x 3; the forward output is BF16 (2^-9)."""
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


@pytest.mark.parametrize("B,D", [(1, 16), (3, 16), (2, 32)])
@pytest.mark.parametrize("ci,co", [(16, 16), (48, 16), (16, 32), (32, 32), (96, 32), (32, 64),
                                   (192, 64), (128, 128)])
def test_layer_on_resident_blocks(dev, B, D, ci, co):
    g = torch.Generator(device=dev)
    g.manual_seed(1000 * ci + 10 * co + B)

    def rn(*shape):
        return torch.randn(shape, generator=g, device=dev).to(torch.bfloat16)

    x, w, gy = rn(B, D, D, D, ci), rn(27, ci, co), rn(B, D, D, D, co)
    bias = torch.randn(co, generator=g, device=dev)
    y = mgfr.conv3d(0, x, w, bias=bias, relu=False)
    gx = mgfr.conv3d(1, x, w, g=gy)
    db = torch.empty(co, device=dev)
    gw = mgfr.conv3d(2, x, w, g=gy, db=db)
    X, W, G = x.double(), w.double(), gy.double()
    want_y = bias.double() + sum(torch.roll(X, tuple(-q for q in d), (1, 2, 3)) @ W[t]
                                 for t, d in enumerate(TAPS))
    want_gx = sum(torch.roll(G, d, (1, 2, 3)) @ W[t].T for t, d in enumerate(TAPS))
    gf = G.reshape(-1, co)
    want_gw = torch.stack([torch.roll(X, tuple(-q for q in d), (1, 2, 3)).reshape(-1, ci).T @ gf
                           for d in TAPS])
    assert rel(y, want_y) <= 2.0 ** -9
    assert rel(gx, want_gx) <= 1e-5
    assert rel(gw, want_gw) <= 1e-5
    for t in range(27):  # every tap by itself: a misplaced one would hide in the norm
        assert rel(gw[t], want_gw[t]) <= 1e-5, t
    assert rel(db, gf.sum(0)) <= 1e-5
    assert torch.equal(gw, mgfr.conv3d(2, x, w, g=gy))  # fixed summation order
