"""The network's set-up on a context of its own stream while the default stream is busy: the
parameters, the optimiser's moments and the kernels' error word are written in the order
of the context's stream (csrc/unet.cu, unet_set)."""
import numpy as np
import pytest
import torch

from paper_1305_2418_gb300 import build, mgfr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU test run without a GPU"
    build.build()
    return torch.device("cuda:0")


def steps(dev, busy):
    side = torch.cuda.Stream(dev)
    d = torch.from_numpy(np.stack([synth.lognormal_delta(32, 50.0, 1.0, 60 + i)
                                   for i in range(2)])).to(dev)
    t = -0.1 * d
    torch.cuda.synchronize()
    out = []
    with torch.cuda.stream(side):
        s = mgfr.Solver(0, stream=side)
        for rep in range(2):
            if busy:
                with torch.cuda.stream(torch.cuda.default_stream(dev)):
                    torch.cuda._sleep(100_000_000)
            s.unet_init(7)
            for _ in range(2):
                out.append(s.unet_train_step(d, [1e-5, 1e-6], t))
            p = s.unet_params()
            s.unet_set_params(p)
            out.append(s.unet_predict(d[0].contiguous(), 1e-5).clone())
            out.append(torch.from_numpy(p))
        torch.cuda.synchronize()
        s.close()
    return out


def test_set_up_while_the_default_stream_is_busy(dev):
    idle, busy = steps(dev, False), steps(dev, True)
    half = len(idle) // 2
    for a, b, c in zip(idle, idle[half:], busy + busy[half:]):
        assert a == b if isinstance(a, float) else torch.equal(a, b)
        assert a == c if isinstance(a, float) else torch.equal(a, c)
