"""GPU checks of the FP64 form on grids whose V-cycles share their FP64 residual in pairs
(csrc/solver.cu, kPairMin .. kPairMax).

The pairs are the single cycles up to FP32 roundings of the first correction, and the last
cycle always starts from an FP64 residual: the same number of cycles, at any tolerance and
at a limit on the cycles, and the same solution within what is left of those roundings
(2^-24 of the correction before last, reduced by the last cycle: 1e-8 of u and below).
The other side is the same solve in calls of one cycle each, from the last call's u: a call
with one cycle left forms its FP64 residual after it."""
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


@pytest.mark.parametrize("tol", [3e-6, 1e-8, 1e-12])
@pytest.mark.parametrize("sig,fr0,kw", [(1.5, 1e-5, {}), (2.5, 1e-6, {}),
                                        (1.0, 1e-4, dict(n=2, n_pre=1, n_post=1))])
def test_same_cycles_as_single_ones(dev, tol, sig, fr0, kw):
    N, box = 128, 200.0
    d = torch.from_numpy(synth.lognormal_delta(N, box, sig, 311)).to(dev)
    one = mgfr.Solver(0, fr0_abs=fr0, tol_rel=tol, max_vcycles=1, **kw)
    u, cycles = None, 0
    while True:
        ref = one.solve_density(d, box, u_init=u, want_u=True, allow_noconverge=True)
        cycles, u = cycles + 1, ref["u"]
        assert cycles < 100
        if ref["status"] == mgfr.MGFR_OK:
            break
    one.close()
    # the limit exactly at the cycles needed, one with room, and one too few
    for most in (cycles, 200, cycles - 1):
        s = mgfr.Solver(0, fr0_abs=fr0, tol_rel=tol, max_vcycles=most, **kw)
        out = s.solve_density(d, box, allow_noconverge=True)
        assert out["stats"]["vcycles"] == min(cycles, most)
        if most >= cycles:
            assert out["status"] == mgfr.MGFR_OK
            assert float((out["fr"] / ref["fr"] - 1.0).abs().max()) <= 1e-8
        else:
            assert out["status"] == mgfr.MGFR_E_NOCONVERGE
        s.close()


@pytest.mark.parametrize("tol", [1e-6, 1e-8, 1e-10])
def test_poisson_pairs(dev, tol):
    """The particle-mesh potential on 128^3 (csrc/pm.cu): the cycles needed are the
    smallest limit that suffices, and the forces are those of a solve to 1e-12 within the
    tolerance (||r|| <= tol ||rhs||; 10 for the force of smooth modes over their source)."""
    N0, box = 64, 100.0
    pos = synth.poisson_particles(synth.lognormal_delta(32, box, 1.5, 411), box, 8.0, 412)
    p = torch.from_numpy(np.ascontiguousarray(pos)).to(dev)

    def accel(tol, most, fails=False):
        s = mgfr.Solver(0, fr0_abs=1e-5, max_level=1, tol_rel=1e-3, max_vcycles=50)
        s.solve_particles(p, N0, box)
        s.set_config(tol_rel=tol, max_vcycles=most)
        try:
            if fails:
                with pytest.raises(mgfr.MGFRError):
                    s.pm_accel(p, 1)
                return None, None
            return s.pm_accel(p, 1)
        finally:
            s.close()

    exact, _ = accel(1e-12, 100)
    acc, st = accel(tol, 100)
    again, st2 = accel(tol, st["vcycles"])
    assert st2["vcycles"] == st["vcycles"]
    accel(tol, st["vcycles"] - 1, fails=True)
    scale = float(exact.abs().max())
    assert float((acc - exact).abs().max()) <= 10 * tol * scale
    assert float((again - acc).abs().max()) <= 10 * tol * scale
