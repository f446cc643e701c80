"""Calls that find too little device memory: they return MGFR_E_OOM, later calls of the same
context work, and what the library holds in reserve never makes a call fail.

The device is filled by one torch allocation (nothing is written to it) up to some
memory left."""
import contextlib
import gc

import numpy as np
import pytest
import torch

from paper_1305_2418_gb300 import build, mgfr, synth

pytestmark = pytest.mark.gpu
GB = 1 << 30


@pytest.fixture(scope="module")
def dev():
    assert torch.cuda.is_available(), "GPU test run without a GPU"
    build.build()
    return torch.device("cuda:0")


def free_bytes(dev):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info(dev)[0]


@contextlib.contextmanager
def only(dev, leave):
    """At most about `leave` bytes free inside."""
    gc.collect()
    torch.cuda.empty_cache()
    hold = torch.empty(max(0, free_bytes(dev) - int(leave)), dtype=torch.uint8, device=dev)
    try:
        yield
    finally:
        del hold
        torch.cuda.empty_cache()


def fails_for_memory(call):
    with pytest.raises(mgfr.MGFRError) as e:
        call()
    assert e.value.status == mgfr.MGFR_E_OOM


def field(dev, N, seed):
    r = torch.Generator(device=dev).manual_seed(seed)
    d = torch.exp(0.5 * torch.randn((N, N, N), generator=r, device=dev, dtype=torch.float64))
    return d / d.mean() - 1.0


@pytest.mark.parametrize("prec", [mgfr.PREC_FP64, mgfr.PREC_MIXED])
def test_a_dense_solve_after_one_without_memory(dev, prec):
    """256^3 takes 0.7 GB and more beside its 0.13 GB result: with 0.65 GB it fails twice, a
    small solve after that works, and 256^3 works once there is room."""
    box = 100.0
    big, small = field(dev, 256, 1), field(dev, 32, 2)
    with mgfr_solver(precision=prec) as s:
        want_small = s.solve_density(small, box)["fr"].clone()
        want_big = s.solve_density(big, box)["fr"].clone()
    torch.cuda.empty_cache()
    with mgfr_solver(precision=prec) as s:
        with only(dev, 0.65 * GB):
            fails_for_memory(lambda: s.solve_density(big, box, want_acc=False))
            fails_for_memory(lambda: s.solve_density(big, box, want_acc=False))
            assert torch.equal(s.solve_density(small, box)["fr"], want_small)
        assert torch.equal(s.solve_density(big, box)["fr"], want_big)
        assert torch.equal(s.solve_density(small, box)["fr"], want_small)


def test_a_prediction_after_one_without_memory(dev):
    """The network's arrays for 128^3 take 1.8 GB."""
    big, small = field(dev, 128, 3), field(dev, 32, 4)
    rng = np.random.default_rng(5)
    with mgfr_solver() as s:
        s.unet_init(1)
        p = s.unet_params()
        p[-17:] = 0.3 * rng.standard_normal(17)
        s.unet_set_params(p)
        want_small = s.unet_predict(small, 1e-5).clone()
        want_big = s.unet_predict(big, 1e-5).clone()
        s.unet_predict(small, 1e-5)  # the arrays of 128^3 are given back
        with only(dev, 1.0 * GB):
            fails_for_memory(lambda: s.unet_predict(big, 1e-5))
            fails_for_memory(lambda: s.unet_predict(big, 1e-5))
            assert torch.equal(s.unet_predict(small, 1e-5), want_small)
        assert torch.equal(s.unet_predict(big, 1e-5), want_big)


@contextlib.contextmanager
def mgfr_solver(**kw):
    s = mgfr.Solver(0, **kw)
    try:
        yield s
    finally:
        s.close()
