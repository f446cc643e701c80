"""GPU checks of the FP32 V-cycles on dense levels (csrc/mg32.cu).

The FP64 form forms its V-cycle's correction in FP32, in the deviation from the
FP64 iterate.  FP32 resolves a correction to about 1e-6 of itself, so the
iterates are those of the V-cycle in FP64 throughout up to 1e-6 of each cycle's
correction, and the next cycle's FP64 residual holds what is left: the same
number of cycles, and the same solution to 1e-6 of the last correction (below
1e-8 of u where the solve stops at 1e-8).  mgfr_solve_density_noalloc runs the
V-cycle in FP64 throughout and is the other side here.
"""
import ctypes as C

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


def noalloc(delta, box, a, cfg):
    fr, st = torch.empty_like(delta), mgfr.Stats()
    rc = mgfr.lib().mgfr_solve_density_noalloc(C.byref(cfg), mgfr._ptr(delta), delta.shape[0], box,
                                               a, mgfr._ptr(fr), None, None, C.byref(st))
    torch.cuda.synchronize()
    assert rc == mgfr.MGFR_OK
    return fr.cpu().numpy(), st


# each size is another split of the levels over the cluster kernel (8^3 and
# 4^3 in one block, 16^3 and 32^3 as slabs, 64^3 above it)
@pytest.mark.parametrize("N", [8, 16, 32, 64])
@pytest.mark.parametrize("sig,fr0,a,kw", [
    (1.5, 1e-5, 1.0, {}),
    (2.0, 1e-6, 1.0, dict(n=2)),
    (1.0, 1e-4, 0.6, dict(prolong_linear=0, n_pre=1, n_post=3)),
    (1.5, 1e-5, 1.0, dict(n_pre=0, n_post=2)),
])
def test_fp32_corrections_follow_the_fp64_cycles(dev, N, sig, fr0, a, kw):
    box = 3.0 * N
    d = torch.from_numpy(synth.lognormal_delta(N, box, sig, 40 + N)).to(dev)
    ref, rst = noalloc(d, box, a, mgfr.default_config(fr0_abs=fr0, max_vcycles=400, **kw))
    for prec in (mgfr.PREC_FP64, mgfr.PREC_MIXED):
        s = mgfr.Solver(0, fr0_abs=fr0, max_vcycles=400, precision=prec, **kw)
        out = s.solve_density(d, box, a)
        if prec == mgfr.PREC_FP64:
            assert out["stats"]["vcycles"] == rst.vcycles
        # both stop at 1e-8: the FP64 form along the same iterates, the mixed
        # form at another point within the tolerance
        rel = np.abs(out["fr"].cpu().numpy() / ref - 1.0).max()
        assert rel <= (1e-8 if prec == mgfr.PREC_FP64 else 1e-5), rel
        s.close()


def test_fp64_form_still_reaches_fp64_tolerances(dev):
    """The residual and the iterate are FP64: a tolerance far below FP32's
    rounding is reached as before."""
    N, box = 32, 100.0
    d = torch.from_numpy(synth.lognormal_delta(N, box, 1.5, 77)).to(dev)
    ref, rst = noalloc(d, box, 1.0, mgfr.default_config(tol_rel=1e-13))
    s = mgfr.Solver(0, tol_rel=1e-13)
    out = s.solve_density(d, box)
    assert out["stats"]["res_l2_final"] <= 1e-13 * out["stats"]["f_l2"]
    # two iterates at 1e-13 of ||f||; the operator's smallest eigenvalue is its
    # mass term, f / mass ~ u: 1e-11 leaves a factor of 100
    assert np.abs(out["fr"].cpu().numpy() / ref - 1.0).max() <= 1e-11
    s.close()


@pytest.mark.parametrize("u0", [-20.0, -50.0, -90.0, -300.0])
def test_far_starts_converge_in_fp64(dev, u0):
    """Starts whose residual FP32 cannot resolve against f (and e^u below its
    range): the first cycles run in FP64."""
    N, box = 16, 100.0
    d = torch.from_numpy(synth.lognormal_delta(N, box, 1.0, 78)).to(dev)
    s = mgfr.Solver(0)
    want = s.solve_density(d, box)["fr"]
    out = s.solve_density(d, box, u_init=torch.full_like(d, u0))
    assert out["stats"]["vcycles"] <= 20
    # both within 1e-8 ||f|| of the solution
    assert float((out["fr"] / want - 1.0).abs().max()) <= 1e-6
    s.close()


@pytest.mark.parametrize("tol", [1e-8, 1e-12])
def test_batch_in_both_precisions(dev, tol):
    """The batched kernel holds its iterate in double-float pairs, or in FP64 for
    tolerances below 1e-10; sizes from one vector per row up, several solves."""
    sizes, fr0s, ns = [8, 32, 16, 8, 64], [1e-5, 1e-6, 1e-4, 1e-6, 1e-5], [1, 2, 1, 1, 3]
    ds = [torch.from_numpy(synth.lognormal_delta(N, 3.0 * N, 1.5, 600 + q)).to(dev)
          for q, N in enumerate(sizes)]
    boxes = [3.0 * N for N in sizes]
    s = mgfr.Solver(0, precision=mgfr.PREC_MIXED, tol_rel=tol, max_vcycles=300)
    outs, st = s.batch_solve(ds, boxes, fr0s, ns=ns, want_acc=True, want_u=True)
    assert st == mgfr.MGFR_OK
    for q, o in enumerate(outs):
        assert o["stats"]["res_l2_final"] <= tol * o["stats"]["f_l2"]
        one = mgfr.Solver(0, fr0_abs=fr0s[q], n=ns[q], tol_rel=1e-12, max_vcycles=300)
        ref = one.solve_density(ds[q], boxes[q], want_u=True)
        one.close()
        # both within tol ||f|| of the solution; 1e3 for the operator's inverse
        assert float((o["fr"] / ref["fr"] - 1.0).abs().max()) <= 1e3 * tol
        assert float((o["u"] - ref["u"]).abs().max()) <= 1e3 * tol
        scale = float(ref["acc"].abs().max())
        assert float((o["acc"] - ref["acc"]).abs().max()) <= 1e3 * tol * scale
    s.close()


@pytest.mark.parametrize("sig,fr0,levels,kw", [
    (1.5, 1e-5, 2, {}),
    (2.0, 1e-6, 3, dict(n_pre=1, n_post=2)),
    (1.0, 1e-4, 1, dict(n=2, prolong_linear=0)),
])
def test_refined_levels_in_fp64_with_fp32_corrections(dev, sig, fr0, levels, kw):
    """The FP64 form of the refined levels: a tolerance far below FP32's rounding
    is reached on every level, and f_R there agrees with the oracle's sweeps."""
    import oracle
    N0, box = 16, 50.0
    pos = synth.poisson_particles(synth.lognormal_delta(N0, box, sig, 90), box, 2.0, 91)
    s = mgfr.Solver(0, fr0_abs=fr0, max_level=levels, tol_rel=1e-12, max_vcycles=300, **kw)
    out = s.solve_particles(torch.from_numpy(pos).to(dev), N0, box)
    st = out["stats"]
    nlev = st["n_levels"]
    assert nlev >= 2 and max(st["level_res"][1:nlev]) <= 1e-12
    A = oracle.AMR(pos, N0, box, levels, 8)
    A.deposit()
    A.set_model(fr0, n=kw.get("n", 1))
    rc, _ = A.solve(tol=1e-12, max_vcycles=400, prolong_linear=bool(kw.get("prolong_linear", 1)))
    assert rc == 0
    for l in range(nlev):
        fr = s.level_field(l, mgfr.FIELD_FR)
        ref, _ = A.level_force(l, bool(kw.get("prolong_linear", 1)))
        if l > 0:
            perm = np.argsort(s.level_keys(l), kind="stable")
            fr = fr[(8 * perm[:, None] + np.arange(8)[None, :]).ravel()]
        # both at 1e-12 of ||f||; 1e3 for the operator's inverse
        assert np.abs(fr / ref - 1.0).max() <= 1e-9, l
    s.close()
