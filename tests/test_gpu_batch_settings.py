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


@pytest.mark.parametrize("tol", [1e-9, 1e-12])  # pairs of floats, FP64
@pytest.mark.parametrize("most", [1, 2, 3, 5, 6])
def test_a_solve_at_its_limit_returns_its_last_iterate(dev, tol, most):
    """max_vcycles reached in the FP32 cycles (the first five or so) or after them: u, f_R and
    the residual belong to each other, the residual falls with the cycles, and the verdict
    is the residual's."""
    box, fr0, N = 100.0, [1e-4, 1e-5, 1e-6], 32
    ds = [torch.from_numpy(synth.lognormal_delta(N, box, 1.5, 900 + i)).to(dev) for i in range(3)]
    s = mgfr.Solver(0, precision=mgfr.PREC_MIXED, tol_rel=tol, max_vcycles=most)
    outs, st = s.batch_solve(ds, [box] * 3, fr0, want_u=True, allow_noconverge=True)
    s.close()
    met = []
    for d, q, o in zip(ds, fr0, outs):
        t = o["stats"]
        r, f = residual(o["u"], d, box, q)
        assert t["vcycles"] + t["outer_iters"] <= most
        assert t["f_l2"] == pytest.approx(f, rel=1e-12)
        # the stored residual is FP32's rounding of an FP64 (48-bit) one
        assert t["res_l2_final"] == pytest.approx(r, rel=1e-5, abs=1e-13 * f * (N / 6.28) ** 2)
        assert float((o["fr"] / (-q * torch.exp(o["u"])) - 1.0).abs().max()) <= 1e-12
        assert float(o["u"].abs().max()) > 0.0 and t["res_l2_final"] < 0.3 ** most * t["res_l2_init"]
        met.append(t["res_l2_final"] <= tol * t["f_l2"])
    assert st == (mgfr.MGFR_OK if all(met) else mgfr.MGFR_E_NOCONVERGE)


def test_a_loose_tolerance_met_in_the_last_cycle_allowed(dev):
    """Met by the FP32 cycles alone, at the limit."""
    box, N = 100.0, 32
    d = torch.from_numpy(synth.lognormal_delta(N, box, 1.5, 900)).to(dev)
    s = mgfr.Solver(0, precision=mgfr.PREC_MIXED, tol_rel=0.1)
    for most in (1, 2, 3):
        s.set_config(max_vcycles=most)
        outs, st = s.batch_solve([d], [box], [1e-5], want_u=True, allow_noconverge=True)
        r, f = residual(outs[0]["u"], d, box, 1e-5)
        assert (st == mgfr.MGFR_OK) == (r <= 0.1 * f)
    assert st == mgfr.MGFR_OK  # three cycles leave less than a tenth
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
