"""The scratch that the convolution primitive keeps between calls (csrc/unet.cu)."""
import pytest
import torch

from paper_1305_2418_gb300 import build, mgfr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU test run without a GPU"
    build.build()
    return torch.device("cuda:0")


@pytest.fixture
def empty_scratch(dev):
    """No kept blocks: destroying a context gives those of its device back."""
    mgfr.Solver(0).close()


def layer(dev, ci, co, D=16, seed=0):
    r = torch.Generator(device=dev).manual_seed(seed + 1000 * ci + co)

    def rn(*shape):
        return torch.randn(shape, generator=r, device=dev).to(torch.bfloat16)

    return rn(1, D, D, D, ci), rn(27, ci, co), rn(1, D, D, D, co)


def test_error_word_is_in_the_callers_stream_order(dev, empty_scratch):
    """Calls on a stream that is not in order with the default stream, while that is busy:
    on fresh blocks (each layer larger than the last) and on kept ones.  The kernels'
    error word is cleared on the call's own stream, so no call reads another value."""
    layers = [layer(dev, ci, co) for ci, co in ((16, 16), (32, 32), (96, 32), (80, 32))]
    want = [(mgfr.conv3d(0, x, w), mgfr.conv3d(1, x, w, g=g), mgfr.conv3d(2, x, w, g=g))
            for x, w, g in layers]
    mgfr.Solver(0).close()
    side = torch.cuda.Stream(dev)
    torch.cuda.synchronize()
    got = []
    for rep in range(2):
        torch.cuda._sleep(400_000_000)  # the default stream: busy for about 0.2 s
        with torch.cuda.stream(side):
            got = [(mgfr.conv3d(0, x, w), mgfr.conv3d(1, x, w, g=g), mgfr.conv3d(2, x, w, g=g))
                   for x, w, g in layers]  # raises where a call reports a wait that gave up
    torch.cuda.synchronize()
    for a, b in zip(want, got):
        assert all(torch.equal(p, q) for p, q in zip(a, b))


def test_largest_blocks_are_kept(dev, empty_scratch):
    """Calls in ascending size: the block that stays is the one that serves them all, so a
    repeated call of the largest allocates nothing.  192 -> 64 sums its weight gradient
    over 43 partials of 27 x 192 x 64 (57 MB), beside four smaller blocks."""
    small = [(16, 16), (16, 32), (32, 32), (32, 64)]
    for ci, co in small:
        x, w, _ = layer(dev, ci, co)
        mgfr.conv3d(0, x, w)
    x, w, g = layer(dev, 192, 64)
    mgfr.conv3d(2, x, w, g=g)
    torch.cuda.synchronize()
    big = 43 * 27 * 192 * 64 * 4
    free0 = torch.cuda.mem_get_info(dev)[0]
    mgfr.Solver(0).close()  # what it gives back was kept
    kept = torch.cuda.mem_get_info(dev)[0] - free0
    assert kept >= big
    # and the limits hold over many sizes, two of them above half of the limit
    for ci, co in small + [(192, 64), (128, 128), (64, 128), (192, 64), (96, 32), (48, 16)]:
        x, w, g = layer(dev, ci, co)
        mgfr.conv3d(2, x, w, g=g)
    torch.cuda.synchronize()
    free1 = torch.cuda.mem_get_info(dev)[0]
    mgfr.Solver(0).close()
    kept = torch.cuda.mem_get_info(dev)[0] - free1
    assert big <= kept <= (128 << 20) + 8 * (2 << 20)  # 2 MB: an allocation's granularity
