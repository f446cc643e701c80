"""Settings of the batched solve from call to call on one context (csrc/batch.cu)."""
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


@pytest.mark.parametrize("N,count", [(8, 400), (16, 180), (32, 1)])
def test_settings_of_a_call_are_its_own(dev, N, count):
    """A tolerance, and a limit on the cycles, set between two calls on the same sizes,
    however many, hold for the next: each solve meets the tolerance asked for, by the
    residual of the u it returns (formed here in FP64)."""
    box, fr0 = 100.0, 1e-5
    ds = [torch.from_numpy(synth.lognormal_delta(N, box, 1.0, 700 + i)).to(dev)
          for i in range(count)]
    s = mgfr.Solver(0, precision=mgfr.PREC_MIXED)
    for tol in (1e-4, 1e-12, 1e-6, 1e-9):
        s.set_config(tol_rel=tol)
        outs, st = s.batch_solve(ds, [box] * count, [fr0] * count, want_u=True)
        assert st == mgfr.MGFR_OK
        for o in outs:
            t = o["stats"]
            assert t["res_l2_final"] <= tol * t["f_l2"]
        for d, o in list(zip(ds, outs))[::37]:
            r, f = residual(o["u"], d, box, fr0)
            assert r <= 1.01 * tol * f + 1e-13 * f * (N / 6.28) ** 2
    # other smoothing: not the cycle counts of before
    s.set_config(tol_rel=1e-9, n_pre=1, n_post=1)
    less, st = s.batch_solve(ds, [box] * count, [fr0] * count)
    assert st == mgfr.MGFR_OK
    assert sum(o["stats"]["vcycles"] + o["stats"]["outer_iters"] for o in less) \
        > sum(o["stats"]["vcycles"] + o["stats"]["outer_iters"] for o in outs)
    s.set_config(tol_rel=1e-12, max_vcycles=2)
    outs, st = s.batch_solve(ds, [box] * count, [fr0] * count, allow_noconverge=True)
    assert st == mgfr.MGFR_E_NOCONVERGE
    assert all(o["stats"]["vcycles"] + o["stats"]["outer_iters"] <= 2 for o in outs)
    s.close()


def residual(u, delta, box, fr0, om=0.3):
    """(||f - L(u)||, ||f||) of the discrete equation for n = 1, a = 1 in FP64."""
    N = u.shape[0]
    h2 = (box / N) ** 2
    rt = om + 4.0 * (1.0 - om)
    alpha = 1.0 / 2997.92458 ** 2 / -fr0
    E = torch.exp(u)
    lap = 0.0
    for ax in range(3):
        for sh in (1, -1):
            lap = lap + 0.5 * (torch.roll(E, sh, ax) + E) * (torch.roll(u, sh, ax) - u)
    L = lap / h2 + alpha * rt * (1.0 - torch.exp(-0.5 * u))
    f = -alpha * om * delta
    return float((f - L).norm()), float(f.norm())
