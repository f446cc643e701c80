"""Calls that find too little device memory: they return MGFR_E_OOM, later calls of the same
context work, and what the library holds in reserve never makes a call fail.

The device is filled by one torch allocation (nothing is written to it) up to some
memory left.  What the driver itself frees when memory runs out is of the order of 0.1 GB:
the sizes leave or lack several times that."""
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
    """512^3 takes 3.7 GB and more beside its 1 GB result: with 2.5 GB it fails twice, a
    small solve after that works, and 512^3 works once there is room."""
    box = 100.0
    big, small = field(dev, 512, 1), field(dev, 32, 2)
    with mgfr_solver(precision=prec) as s:
        want_small = s.solve_density(small, box)["fr"].clone()
        want_big = s.solve_density(big, box)["fr"].clone()
    torch.cuda.empty_cache()
    with mgfr_solver(precision=prec) as s:
        with only(dev, 2.5 * GB):
            fails_for_memory(lambda: s.solve_density(big, box, want_acc=False))
            fails_for_memory(lambda: s.solve_density(big, box, want_acc=False))
            assert torch.equal(s.solve_density(small, box)["fr"], want_small)
        assert torch.equal(s.solve_density(big, box)["fr"], want_big)
        assert torch.equal(s.solve_density(small, box)["fr"], want_small)


def test_an_fp64_solve_without_the_fp32_arrays(dev):
    """512^3 in the FP64 form: its FP64 arrays take 3.6 GB, the FP32 ones of the correction
    cycles 1.8 GB more.  Without room for those the cycles run in FP64: the same field
    within the tolerance (1e-8 of the source, 1e2 for the operator's inverse); with room
    again they are back."""
    box, big = 100.0, field(dev, 512, 1)
    with mgfr_solver() as s:
        out = s.solve_density(big, box)
        want, launches = out["fr"].cpu(), out["stats"]["gpu_launches"]
        del out
    with mgfr_solver() as s:
        with only(dev, (1.0 + 3.6 + 0.7) * GB):
            for _ in range(2):
                out = s.solve_density(big, box, want_acc=False)
                assert out["status"] == mgfr.MGFR_OK
                got = out["fr"].cpu()
                # a launch per half-sweep of every grid: more than the cycles in FP32
                assert out["stats"]["gpu_launches"] > 1.5 * launches
                del out
                assert float((got / want - 1.0).abs().max()) <= 1e-6
        out = s.solve_density(big, box)
        assert torch.equal(out["fr"].cpu(), want) and out["stats"]["gpu_launches"] == launches


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


# ---- the refined levels' reserve ------------------------------------------------
N0, BOX = 64, 100.0


def particles(dev, n, part, seed):
    """n particles, uniform in the first `part` of the box along x: at 100 and more per base
    cell two levels are refined wherever there are particles."""
    r = torch.Generator(device=dev).manual_seed(seed)
    p = torch.rand((n, 3), generator=r, device=dev, dtype=torch.float64) * BOX
    p[:, 0] *= part
    return p


def held(dev, call):
    """Device memory that stays taken after the call, beside torch's."""
    gc.collect()
    torch.cuda.empty_cache()
    before = free_bytes(dev)
    call()
    torch.cuda.empty_cache()
    return before - free_bytes(dev)


def rel(a, b):
    return float((a - b).norm() / b.norm())


def test_a_kept_level_does_not_take_a_later_solves_memory(dev):
    """All of the box refined, then 0.6 of it with more particles: the second solve gets the
    memory that it takes by itself, which is less than what it needs beside the first
    one's level arrays (1 GB more).  The same hierarchy and forces as by itself; the
    masses are summed by atomics, whose order may flip FP32 roundings (6e-8 each)."""
    first, second = particles(dev, 33_000_000, 1.0, 1), particles(dev, 55_000_000, 0.6, 2)
    cfg = dict(precision=mgfr.PREC_MIXED, max_level=2, tol_rel=1e-5)
    own = second.numel() * 8 + (8 << 20)  # the force array and f_R, torch's
    with mgfr_solver(**cfg) as s:
        need = held(dev, lambda: s.solve_particles(second, N0, BOX))
        want = s.solve_particles(second, N0, BOX)["acc"].cpu()
        levels = [s.level_info(l) for l in range(3)]
        pm_need = held(dev, lambda: s.pm_accel(second, 2))
        want_pm = s.pm_accel(second, 2)[0].cpu()
    with mgfr_solver(**cfg) as s:
        has = held(dev, lambda: s.solve_particles(first, N0, BOX))
        assert s.level_info(2)[1] > 1.5 * levels[2][1]
        with only(dev, need - has + own + (256 << 20)):
            got = s.solve_particles(second, N0, BOX)["acc"].cpu()
            assert [s.level_info(l) for l in range(3)] == levels
        assert rel(got, want) <= 1e-6
        # and again with room, on the arrays that it now has
        assert rel(s.solve_particles(second, N0, BOX)["acc"].cpu(), want) <= 1e-6
    # a particle-mesh force after it, the levels still holding more than they need
    with mgfr_solver(**cfg) as s:
        s.solve_particles(first, N0, BOX)
        s.solve_particles(second, N0, BOX, want_acc=False)
        d0 = s.effective_density(2)
        with only(dev, pm_need + own - (256 << 20)):
            got = s.pm_accel(second, 2)[0].cpu()
        assert rel(got, want_pm) <= 1e-6
        # the hierarchy is still there, its fields as they were
        assert torch.equal(s.effective_density(2), d0)
        assert [s.level_info(l) for l in range(3)] == levels
        fr = s.level_field(2, mgfr.FIELD_FR)
        assert np.isfinite(fr).all() and (fr < 0.0).all()


def test_an_fp64_particle_solve_without_the_fp32_arrays(dev):
    """512^3 base, one level of some 60 M cells: room for exact level arrays, but for half of
    the dense grids' FP32 arrays (1.8 GB) only.  Two solutions to 1e-9 of the source,
    the force at the particles within 1e-5 (1e2 for the operator's inverse, 1e2 for its
    gradient)."""
    pos = particles(dev, 80_000_000, 0.05, 7)
    cfg = dict(max_level=1, tol_rel=1e-9)
    with mgfr_solver(**cfg) as s:
        need = held(dev, lambda: s.solve_particles(pos, 512, BOX))
        out = s.solve_particles(pos, 512, BOX)
        want, n = out["acc"].cpu(), s.level_info(1)[0]
        launches = out["stats"]["gpu_launches"]
        del out
    reserve = n // 16 * 8 * 139
    own = pos.numel() * 8 + 512 ** 3 * 8
    with mgfr_solver(**cfg) as s:
        with only(dev, need - reserve - (900 << 20) + own):
            out = s.solve_particles(pos, 512, BOX)
            assert out["status"] == mgfr.MGFR_OK
            got = out["acc"].cpu()
            assert out["stats"]["gpu_launches"] > 1.2 * launches
            del out
        assert rel(got, want) <= 1e-5
        assert rel(s.solve_particles(pos, 512, BOX)["acc"].cpu(), want) <= 1e-9


def test_a_force_in_the_room_of_the_solve(dev):
    """The particle-mesh force's arrays (32 bytes per cell of 512^3: 4.3 GB) in what phi and
    the solve's 21 bytes per cell leave: the solve's arrays make room, and come back."""
    pos = particles(dev, 300_000, 1.0, 9)
    with mgfr_solver(precision=mgfr.PREC_MIXED, tol_rel=1e-5) as s:
        s.solve_particles(pos, 64, BOX)
        want = s.pm_accel(pos, 3)[0].clone()
    with mgfr_solver(precision=mgfr.PREC_MIXED, tol_rel=1e-5) as s:
        s.solve_particles(pos, 64, BOX)
        with only(dev, (8 + 32 + 4) * 512 ** 3):
            assert rel(s.pm_accel(pos, 3)[0], want) <= 1e-9
            assert rel(s.pm_accel(pos, 3)[0], want) <= 1e-9
        assert rel(s.pm_accel(pos, 3)[0], want) <= 1e-9
        phi = s.pm_potential(64, 3)[0]
        assert bool(torch.isfinite(phi).all())
