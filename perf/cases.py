"""The work a user of the field solver has it do, as measurable cases.

Every case goes through the public binding (`paper_1305_2418_gb300.mgfr`): the
periodic density solve in both precisions, the particle solve on a refined
hierarchy, the batched solve, the particle-mesh force, and the network that
predicts an initial guess (a convolution layer forward and backward, a
prediction, a training step).  Sizes are those of the repository's workloads,
tests and benchmark.  Inputs are lognormal fields and Poisson-sampled
particles (the recipe of `synth.py`), drawn on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_1305_2418_gb300 import mgfr

DEV = "cuda:0"
OMEGA_M = 0.3
U_SCALE = 0.01
# the network's convolutions: (input channels, output channels, resolution level)
CONVS = [(16, 16, 0), (16, 16, 0), (16, 32, 1), (32, 32, 1), (32, 64, 2), (64, 64, 2),
         (64, 128, 3), (128, 128, 3), (192, 64, 2), (64, 64, 2), (96, 32, 1), (32, 32, 1),
         (48, 16, 0), (16, 16, 0)]
LAYERS = sorted({(ci, co) for ci, co, _ in CONVS})


# ---- the cases ----------------------------------------------------------------
def listed():
    return [
        # the smallest call: one low-resolution field in the default precision
        # (the repository's 32^3 workload), a matter of latency
        dict(name="density32_fp64", kind="density", N=32, box=100.0, a=1.0, fr0=1e-5, n=1,
             sigma=1.0, mixed=False),
        # an ordinary field in the default precision
        dict(name="density128_fp64", kind="density", N=128, box=100.0, a=1.0, fr0=1e-5, n=1,
             sigma=1.5, mixed=False),
        # the evaluation fields of the learned start: 256^3, mixed precision
        dict(name="density256_mixed", kind="density", N=256, box=100.0, a=1.0, fr0=1e-5, n=1,
             sigma=1.5, mixed=True),
        # a small refined hierarchy in the default precision
        dict(name="particles64_fp64", kind="particles", N=64, grid=64, box=100.0, a=1.0, fr0=1e-5,
             n=1, sigma=1.5, nbar=1.0, levels=2, mixed=False, host=False),
        # many particles on a coarse base: 256^3 particles, 64^3 base, 3 levels
        # (the adaptive-against-fixed-grid comparison)
        dict(name="particles64_deep_mixed", kind="particles", N=64, grid=256, box=100.0, a=1.0,
             fr0=1e-6, n=1, sigma=1.5, nbar=1.0, levels=3, mixed=True, host=False),
        # the ordinary simulation step: 256^3 particles, 256^3 base, 2 levels
        dict(name="particles256_mixed", kind="particles", N=256, grid=256, box=100.0, a=1.0,
             fr0=1e-5, n=1, sigma=1.5, nbar=1.0, levels=2, mixed=True, host=False),
        # the largest: 512^3 particles, 512^3 base, 3 levels (the headline workload)
        dict(name="particles512_mixed", kind="particles", N=512, grid=512, box=100.0, a=1.0,
             fr0=1e-6, n=1, sigma=2.0, nbar=1.0, levels=3, mixed=True, host=False),
        # a parameter scan / training-set generation: 96 fields of mixed sizes in one call
        dict(name="batch96", kind="batch", count=96, lgmin=5, lgmax=7, box=100.0, pick=4242),
        # the particle-mesh force of the total mass in a time step
        dict(name="pm_accel256", kind="pm", N=256, grid=256, box=100.0, a=1.0, fr0=1e-5, n=1,
             sigma=1.5, nbar=1.0, levels=2, lpm=0, what=mgfr.PM_TOTAL),
        # one decoder layer of the network, forward and both gradients
        dict(name="conv_96_32_4x32", kind="conv", B=4, D=32, cin=96, cout=32),
        # the network's prediction for a 256^3 field (inference)
        dict(name="predict256", kind="predict", D=256, box=100.0, fr0=1e-5, sigma=1.5),
        # one step of the network's training (mini-batch of four 64^3 fields)
        dict(name="train_4x64", kind="train", B=4, D=64, box=25.0, sigma=1.25),
    ]


def draw(rng):
    kind = rng.choice(["density", "density", "particles", "particles", "batch", "pm", "conv",
                       "conv", "predict", "train"])
    fr0 = 10.0 ** rng.uniform(-6.0, -4.0)
    sigma = rng.uniform(0.5, 2.0)
    a = rng.choice([1.0, rng.uniform(0.5, 1.0)])
    box = rng.uniform(50.0, 200.0)
    if kind == "density":
        mixed = rng.random() < 0.5
        return dict(kind=kind, N=1 << rng.randint(3, 8 if mixed else 7), box=box, a=a, fr0=fr0,
                    n=rng.choice([1, 1, 2]), sigma=sigma, mixed=mixed)
    if kind == "particles":
        mixed = rng.random() < 0.67
        N = 1 << rng.randint(4, 8 if mixed else 6)
        # particles per base cell 0.5 .. 2, sampled on the base grid
        return dict(kind=kind, N=N, grid=N, box=box, a=a, fr0=fr0, n=1, sigma=min(sigma, 1.75),
                    nbar=rng.uniform(0.5, 2.0), levels=rng.randint(1, 3), mixed=mixed,
                    host=mixed and rng.random() < 0.3)
    if kind == "batch":
        lgmin = rng.randint(3, 5)
        return dict(kind=kind, count=int(round(2.0 ** rng.uniform(0.0, 6.5))), lgmin=lgmin,
                    lgmax=rng.randint(lgmin, 7), box=box, pick=rng.randint(0, 1 << 20))
    if kind == "pm":
        N = 1 << rng.randint(4, 8)
        return dict(kind=kind, N=N, grid=N, box=box, a=a, fr0=fr0, n=1, sigma=min(sigma, 1.75),
                    nbar=rng.uniform(0.5, 2.0), levels=rng.randint(1, 2),
                    lpm=rng.randint(0, 1), what=rng.choice([mgfr.PM_MATTER, mgfr.PM_TOTAL]))
    if kind == "conv":
        # the network's layers and a few channel counts beside them
        cin, cout = rng.choice(LAYERS + [(80, 32), (48, 64)])
        lg = rng.randint(3, 7 if cin * cout <= 2048 else 5)
        return dict(kind=kind, B=rng.randint(1, 3), D=1 << lg, cin=cin, cout=cout)
    if kind == "predict":
        return dict(kind=kind, D=1 << rng.randint(5, 8), box=box, fr0=fr0, sigma=sigma)
    return dict(kind=kind, B=rng.randint(1, 5), D=1 << rng.randint(5, 6),
                box=rng.uniform(12.5, 50.0), sigma=sigma)


# ---- inputs ---------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _lognormal(N, sigma, g):
    """Lognormal density contrast with P(k) ~ k^-1.5 and mean 0 (FP64, on the GPU)."""
    fk = torch.fft.rfftn(torch.randn((N, N, N), generator=g, device=DEV, dtype=torch.float64))
    n1 = torch.fft.fftfreq(N, d=1.0 / N, device=DEV, dtype=torch.float64)
    nz = torch.fft.rfftfreq(N, d=1.0 / N, device=DEV, dtype=torch.float64)
    k2 = n1[:, None, None] ** 2 + n1[None, :, None] ** 2 + nz[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    fk *= k2.pow_(-0.375)
    fk[0, 0, 0] = 0.0
    f = torch.fft.irfftn(fk, s=(N, N, N))
    del fk, k2
    f *= sigma / f.std()
    f = torch.exp(f)
    f /= f.mean()
    return f.sub_(1.0)


def _particles(case, seed):
    """Particles Poisson-sampled from a lognormal field (a given number of them),
    ordered by the cells of the sampling grid."""
    G, box = case["grid"], case["box"]
    count = int(round(case["nbar"] * float(G) ** 3))
    g = _gen(seed)
    lam = _lognormal(G, case["sigma"], g).add_(1.0).reshape(-1).cumsum(0)
    at = torch.rand(count, generator=g, device=DEV, dtype=torch.float64).sort()[0].mul_(lam[-1])
    cells = torch.searchsorted(lam, at, right=True).clamp_(max=G ** 3 - 1).to(torch.int32)
    del lam, at
    pos = torch.rand((cells.numel(), 3), generator=g, device=DEV, dtype=torch.float64)
    for ax, div in enumerate((G * G, G, 1)):
        pos[:, ax] += torch.remainder(torch.div(cells, div, rounding_mode="floor"), G)
    del cells
    pos *= box / G
    pos.clamp_(0.0, float(np.nextafter(box, 0.0)))
    return pos


# A simulation keeps one Solver and calls it with the particles of each step, so
# the states of one particle case (other seeds: other particles) share theirs.
_kept = {}


def _particle_solver(case):
    cfg = dict(precision=mgfr.PREC_MIXED if case["mixed"] else mgfr.PREC_FP64,
               fr0_abs=case["fr0"], n=case["n"], max_level=case["levels"])
    key = (case["N"], case["box"], tuple(sorted(cfg.items())))
    if key not in _kept:
        _kept.clear()
        _kept[key] = mgfr.Solver(0, **cfg)
    return _kept[key]


def _batch_items(case):
    rng = np.random.default_rng(case["pick"])
    sizes = [int(v) for v in 1 << rng.integers(case["lgmin"], case["lgmax"] + 1, case["count"])]
    sizes[0] = 1 << case["lgmax"]
    sig = rng.uniform(0.5, 2.0, case["count"])
    fr0 = 10.0 ** rng.uniform(-6.0, -4.0, case["count"])
    return sizes, [float(s) for s in sig], [float(v) for v in fr0]


def _weights(seed):
    """He-normal convolutions, small biases and a head that is not zero."""
    rng = np.random.default_rng(seed)
    p = []
    for ci, co, _ in CONVS:
        p.append(rng.standard_normal(27 * ci * co, dtype=np.float32) * math.sqrt(2.0 / (27 * ci)))
        p.append(0.02 * rng.standard_normal(co, dtype=np.float32))
    p.append(0.3 * rng.standard_normal(17, dtype=np.float32))
    return np.concatenate(p).astype(np.float32)


def _network(seed):
    """A Solver with a network of these weights."""
    s = mgfr.Solver(0)
    s.unet_init(0)
    s.unet_set_params(_weights(seed))
    return s


def _target(delta, box):
    """A field like the solution: the local screening value of the density
    smoothed over about a Compton length."""
    N = delta.shape[-1]
    n1 = torch.fft.fftfreq(N, d=1.0 / N, device=DEV, dtype=torch.float64)
    nz = torch.fft.rfftfreq(N, d=1.0 / N, device=DEV, dtype=torch.float64)
    k2 = (n1[:, None, None] ** 2 + n1[None, :, None] ** 2 + nz[None, None, :] ** 2) \
        * (2.0 * math.pi / box) ** 2
    sm = torch.fft.irfftn(torch.fft.rfftn(delta) / (1.0 + 4.0 * k2), s=(N, N, N))
    return -2.0 * torch.log(torch.clamp(1.0 + OMEGA_M / 3.1 * sm, min=0.3)) * 0.3


def _conv_inputs(case, seed):
    g = _gen(seed)
    B, D, ci, co = case["B"], case["D"], case["cin"], case["cout"]

    def rn(*shape):
        return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)

    x = torch.relu(rn(B, D, D, D, ci)).to(torch.bfloat16)
    w = (rn(27, ci, co) * math.sqrt(2.0 / (27 * ci))).to(torch.bfloat16)
    b = 0.1 * rn(co)
    gy = (rn(B, D, D, D, co) * (rn(B, D, D, D, co) > 0)).to(torch.bfloat16)
    return x, w, b, gy


def _train_inputs(case, seed):
    B, D = case["B"], case["D"]
    g = _gen(seed)
    d = torch.stack([_lognormal(D, case["sigma"], g) for _ in range(B)])
    t = torch.stack([_target(d[i], case["box"]) for i in range(B)])
    fr0 = 10.0 ** np.random.default_rng(seed).uniform(-6.0, -4.0, B)
    return d, fr0, t


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "density":
        s["delta"] = _lognormal(case["N"], case["sigma"], _gen(seed))
        s["solver"] = mgfr.Solver(0, fr0_abs=case["fr0"], n=case["n"],
                                  precision=mgfr.PREC_MIXED if case["mixed"] else mgfr.PREC_FP64)
    elif kind == "particles":
        s["solver"] = _particle_solver(case)
        s["pos"] = _particles(case, seed)
        if case["host"]:
            s["pos"] = s["pos"].cpu().pin_memory()
            s["acc"] = torch.empty_like(s["pos"], pin_memory=True)
    elif kind == "batch":
        sizes, sig, s["fr0s"] = _batch_items(case)
        g = _gen(seed)
        s["deltas"] = [_lognormal(N, q, g) for N, q in zip(sizes, sig)]
        s["boxes"] = [case["box"]] * len(sizes)
        s["solver"] = mgfr.Solver(0, precision=mgfr.PREC_MIXED)
    elif kind == "pm":
        s["solver"] = mgfr.Solver(0, precision=mgfr.PREC_MIXED, fr0_abs=case["fr0"], n=case["n"],
                                  max_level=case["levels"])
        s["pos"] = _particles(case, seed)
        s["solver"].solve_particles(s["pos"], case["N"], case["box"], case["a"], want_acc=False)
    elif kind == "conv":
        s["x"], s["w"], s["b"], s["g"] = _conv_inputs(case, seed)
        s["db"] = torch.empty(case["cout"], device=DEV, dtype=torch.float32)
    elif kind == "predict":
        s["delta"] = _lognormal(case["D"], case["sigma"], _gen(seed))
        s["solver"] = _network(seed)
    else:
        s["delta"], s["fr0s"], s["target"] = _train_inputs(case, seed)
        s["solver"] = _network(seed)
    torch.cuda.empty_cache()  # the library allocates outside torch's pool
    return s


# ---- one pass ---------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "density":
        o = s["solver"].solve_density(s["delta"], s["box"], s["a"])
        return {"fr": o["fr"], "acc": o["acc"]}
    if kind == "particles":
        if s["host"]:
            o = s["solver"].solve_particles_host(s["pos"], s["N"], s["box"], s["a"],
                                                 acc_out=s["acc"], want_fr=True)
        else:
            o = s["solver"].solve_particles(s["pos"], s["N"], s["box"], s["a"])
        return {"fr": o["fr"], "acc": o["acc"]}
    if kind == "batch":
        outs, _ = s["solver"].batch_solve(s["deltas"], s["boxes"], s["fr0s"], want_u=True)
        # f_R and u of every field, each set as one array
        return {k: torch.cat([o[k].reshape(-1) for o in outs]) for k in ("fr", "u")}
    if kind == "pm":
        acc, _ = s["solver"].pm_accel(s["pos"], s["lpm"], s["what"])
        return {"acc": acc}
    if kind == "conv":
        return {"y": mgfr.conv3d(0, s["x"], s["w"], bias=s["b"], relu=True),
                "gx": mgfr.conv3d(1, s["x"], s["w"], g=s["g"]),
                "gw": mgfr.conv3d(2, s["x"], s["w"], g=s["g"], db=s["db"]),
                "gb": s["db"]}
    if kind == "predict":
        return {"u": s["solver"].unet_predict(s["delta"], s["fr0"])}
    loss = s["solver"].unet_train_step(s["delta"], s["fr0s"], s["target"])
    return {"loss": loss, "grads": s["solver"].unet_grads()}


# ---- what a pass cannot do without -------------------------------------------------
def _unet_flops(voxels):
    return sum(2.0 * 27 * ci * co * voxels / 8 ** lv for ci, co, lv in CONVS)


def work(case):
    kind = case["kind"]
    if kind == "density":
        n = float(case["N"]) ** 3  # delta in; f_R and the force out; one residual and one update
        return {"bytes": 8 * 5 * n, "flops": 120 * n}
    if kind == "particles":
        n, p = float(case["N"]) ** 3, case["nbar"] * float(case["grid"]) ** 3
        return {"bytes": 8 * n + 48 * p, "flops": 120 * n + 100 * p}
    if kind == "batch":
        n = float(sum(N ** 3 for N in _batch_items(case)[0]))
        return {"bytes": 8 * 3 * n, "flops": 120 * n}
    if kind == "pm":
        n, p = float(case["N"] << case["lpm"]) ** 3, case["nbar"] * float(case["grid"]) ** 3
        return {"bytes": 8 * n + 48 * p, "flops": 20 * n + 60 * p}
    if kind == "conv":
        m, ci, co = float(case["B"]) * case["D"] ** 3, case["cin"], case["cout"]
        return {"bytes": m * (2 * ci + 4 * co + 4 * ci) + 27 * ci * co * 6,
                "flops": 3 * 2 * 27.0 * ci * co * m}
    if kind == "predict":
        m = float(case["D"]) ** 3
        return {"bytes": 16 * m, "flops": _unet_flops(m)}
    m = float(case["B"]) * case["D"] ** 3
    return {"bytes": 16 * m + 4 * 1466065 * 7, "flops": 3 * _unet_flops(m)}


# ---- the same in plain torch, 64 bits --------------------------------------------
def _model(fr0, a, n):
    ol = 1.0 - OMEGA_M
    rt, rt1 = OMEGA_M / a ** 3 + 4.0 * ol, OMEGA_M + 4.0 * ol
    fbar = -fr0 * (rt1 / rt) ** (n + 1)
    alpha = a * a / 2997.92458 ** 2 / fbar
    return fbar, alpha * rt, -alpha * OMEGA_M / a ** 3


def _shifts(x):
    return [torch.roll(x, q, d) for d in (1, 2, 3) for q in (1, -1)]


def _op(u, art, np1, ih2):
    E = torch.exp(u)
    s = 0.0
    for un in _shifts(u):
        s = s + 0.5 * (torch.exp(un) + E) * (un - u)
    return s * ih2 + art * (1.0 - torch.exp(-u / np1))


def _relax(u, f, art, np1, ih2, sweeps):
    N = u.shape[-1]
    i = torch.arange(N, device=DEV)
    par = (i[:, None, None] + i[None, :, None] + i[None, None, :]) & 1
    for _ in range(sweeps):
        for c in (0, 1):
            E = torch.exp(u)
            flux = sd = sb = 0.0
            for un in _shifts(u):
                b, d = 0.5 * (torch.exp(un) + E), un - u
                flux, sd, sb = flux + b * d, sd + d, sb + b
            s = torch.exp(-u / np1)
            L = flux * ih2 + art * (1.0 - s)
            dL = (0.5 * E * sd - sb) * ih2 + art / np1 * s
            u = torch.where(par == c, u - ((L - f) / dL).clamp_(-2.0, 2.0), u)
    return u


def _coarsen(x):
    B, N = x.shape[0], x.shape[-1]
    return x.reshape(B, N // 2, 2, N // 2, 2, N // 2, 2).mean(dim=(2, 4, 6))


def _refine(c):
    N = 2 * c.shape[-1]
    up = [x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)
          for x in (c, *(0.125 * (torch.roll(c, -1, d) - torch.roll(c, 1, d)) for d in (1, 2, 3)))]
    sign = 2.0 * (torch.arange(N, device=DEV, dtype=torch.float64) % 2) - 1.0
    return up[0] + sign[:, None, None] * up[1] + sign[None, :, None] * up[2] + sign * up[3]


def _cycle(u, f, art, np1, ih2):
    if u.shape[-1] <= 4:
        return _relax(u, f, art, np1, ih2, 60)
    u = _relax(u, f, art, np1, ih2, 2)
    c0, rc = _coarsen(u), _coarsen(f - _op(u, art, np1, ih2))
    ihc = 0.25 * ih2
    c1 = _cycle(c0, rc + _op(c0, art, np1, ihc), art, np1, ihc)
    return _relax(u + _refine(c1 - c0), f, art, np1, ih2, 2)


def _field(delta, box, a, fr0, n):
    """u of a batch of fields [B, N, N, N] (fr0: one per field), to rounding."""
    N = delta.shape[-1]
    m = [_model(q, a, n) for q in fr0]
    fbar, art, src = (torch.tensor([x[k] for x in m], device=DEV, dtype=torch.float64)
                      .reshape(-1, 1, 1, 1) for k in range(3))
    f, ih2 = src * delta, (N / box) ** 2
    u, last = torch.zeros_like(f), math.inf
    for _ in range(60):
        u = _cycle(u, f, art, n + 1.0, ih2)
        r = f - _op(u, art, n + 1.0, ih2)
        r = float((r.flatten(1).norm(dim=1) / f.flatten(1).norm(dim=1)).max())
        if r < 1e-13 or (r < 1e-10 and r > 0.5 * last):
            break
        last = r
    return u, fbar


def _central(x, h):
    return torch.stack([(torch.roll(x, -1, d) - torch.roll(x, 1, d)) / (2.0 * h)
                        for d in range(3)])


def _base_mass(pos, case):
    """Mass per base cell (in particles): every particle is a cube with the side of
    its leaf cell; a cell with more than 8 particles is refined, with its 26
    neighbours that exist."""
    N = case["N"]
    t = pos * (N / case["box"])
    lam = torch.zeros(t.shape[0], device=DEV, dtype=torch.int64)
    exists = torch.ones((N,) * 3, device=DEV, dtype=torch.bool)
    for l in range(case["levels"]):
        n = N << l
        c = torch.floor(t * 2.0 ** l).long()
        idx = (c[:, 0] * n + c[:, 1]) * n + c[:, 2]
        del c
        hot = (torch.bincount(idx, minlength=n ** 3) > 8).reshape(n, n, n) & exists
        for d in range(3):
            hot = hot | torch.roll(hot, 1, d) | torch.roll(hot, -1, d)
        hot &= exists
        lam += hot.reshape(-1)[idx].long()
        exists = hot.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)
    half = 0.5 * 2.0 ** (-lam.double())
    i0, w = [], []
    for d in range(3):
        lo = t[:, d] - half
        i = torch.floor(lo)
        w0 = torch.minimum(i + 1.0 - lo, 2.0 * half) / (2.0 * half)
        i0.append(i.long())
        w.append((w0, 1.0 - w0))
    mass = torch.zeros(N ** 3, device=DEV, dtype=torch.float64)
    for q in range(8):
        b = (q >> 2, (q >> 1) & 1, q & 1)
        c = [torch.remainder(i0[d] + b[d], N) for d in range(3)]
        mass.index_add_(0, (c[0] * N + c[1]) * N + c[2], w[0][b[0]] * w[1][b[1]] * w[2][b[2]])
    return mass.reshape(N, N, N)


def _pm_matter(case, pos):
    """-grad phi of the matter at the particles on the base grid, by FFT."""
    N, h = case["N"], case["box"] / case["N"]
    d = _base_mass(pos, case) * (float(N) ** 3 / pos.shape[0]) - 1.0
    c = 2.0 * torch.cos(2.0 * math.pi * torch.arange(N, device=DEV, dtype=torch.float64) / N) - 2.0
    lap = (c[:, None, None] + c[None, :, None] + c[None, None, : N // 2 + 1]) / (h * h)
    lap[0, 0, 0] = 1.0
    fk = torch.fft.rfftn(d) * (1.5e4 * OMEGA_M / case["a"]) / lap
    fk[0, 0, 0] = 0.0
    g = -_central(torch.fft.irfftn(fk, s=(N, N, N)), h).reshape(3, -1)
    t = pos / h - 0.5
    i0 = torch.floor(t)
    w = t - i0
    acc = torch.zeros_like(pos)
    for q in range(8):
        b = (q >> 2, (q >> 1) & 1, q & 1)
        idx, wt = 0, 1.0
        for d in range(3):
            idx = idx * N + torch.remainder(i0[:, d].long() + b[d], N)
            wt = wt * (w[:, d] if b[d] else 1.0 - w[:, d])
        acc += wt[:, None] * g[:, idx].T
    return acc


TAPS = [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)]


def _conv64(x, w, b=None):
    y = 0.0
    for t, d in enumerate(TAPS):
        y = y + torch.roll(x, tuple(-q for q in d), (1, 2, 3)) @ w[t]
    return y if b is None else y + b


def _unet64(delta, fr0, p):
    """v = asinh(u / 0.01) of the network with parameters p [flat], FP64."""
    ws, off = [], 0
    for ci, co, _ in CONVS:
        w = p[off:off + 27 * ci * co].reshape(27, ci, co)
        off += 27 * ci * co
        ws.append((w, p[off:off + co]))
        off += co
    rt = OMEGA_M + 4.0 * (1.0 - OMEGA_M)
    ul = (-2.0 * torch.log(torch.clamp(1.0 + OMEGA_M / rt * delta, min=1e-6))).clamp(-20.0, 5.0)
    f = torch.as_tensor(np.log10(fr0) + 5.0, device=DEV, dtype=torch.float64)
    x = torch.zeros(delta.shape + (16,), device=DEV, dtype=torch.float64)
    x[..., 0] = torch.log(torch.clamp(1.0 + delta, min=1e-3))
    x[..., 1] = f.reshape(-1, 1, 1, 1)
    x[..., 2] = 1.0
    x[..., 3] = torch.asinh(ul / U_SCALE) / 5.0

    def block(x, i):
        for w, b in ws[i:i + 2]:
            x = torch.relu(_conv64(x, w, b))
        return x

    def pool(x):
        B, D, C = x.shape[0], x.shape[1] // 2, x.shape[-1]
        return x.reshape(B, D, 2, D, 2, D, 2, C).mean(dim=(2, 4, 6))

    def up(x):
        return x.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    e0 = block(x, 0)
    e1 = block(pool(e0), 2)
    e2 = block(pool(e1), 4)
    d = block(pool(e2), 6)
    for e, i in ((e2, 8), (e1, 10), (e0, 12)):
        d = block(torch.cat([up(d), e], -1), i)
    return d @ p[off:off + 16] + p[off + 16]


def exact(case, seed):
    kind = case["kind"]
    if kind == "density":
        u, fbar = _field(_lognormal(case["N"], case["sigma"], _gen(seed))[None], case["box"],
                         case["a"], [case["fr0"]], case["n"])
        fr = (fbar * torch.exp(u))[0]
        return {"fr": fr, "acc": _central(fr, case["box"] / case["N"]) / (2.0 * case["a"])}
    if kind == "particles":
        # f_R on the base; the force needs the whole hierarchy.  Counts of the
        # finest flagged level are kept as a full grid, too large beyond 1024^3
        if case["N"] << (case["levels"] - 1) > 1024:
            return None
        pos = _particles(case, seed)
        d = _base_mass(pos, case) * (float(case["N"]) ** 3 / pos.shape[0]) - 1.0
        u, fbar = _field(d[None], case["box"], case["a"], [case["fr0"]], case["n"])
        return {"fr": (fbar * torch.exp(u))[0], "acc": None}
    if kind == "batch":
        sizes, sig, fr0 = _batch_items(case)
        g = _gen(seed)
        deltas = [_lognormal(N, q, g) for N, q in zip(sizes, sig)]
        us = [None] * len(sizes)
        for N in sorted(set(sizes)):
            at = [i for i, q in enumerate(sizes) if q == N]
            u, fb = _field(torch.stack([deltas[i] for i in at]), case["box"], 1.0,
                           [fr0[i] for i in at], 1)
            for k, i in enumerate(at):
                us[i] = (float(fb.reshape(-1)[k]), u[k].reshape(-1))
        return {"fr": torch.cat([fb * torch.exp(u) for fb, u in us]),
                "u": torch.cat([u for _, u in us])}
    if kind == "pm":
        if case["what"] != mgfr.PM_MATTER or case["lpm"] != 0:
            return None  # needs the solution (or the leaves) of the refined levels
        return {"acc": _pm_matter(case, _particles(case, seed))}
    if kind == "conv":
        x, w, b, g = (q.double() for q in _conv_inputs(case, seed))
        gx = sum(torch.roll(g, d, (1, 2, 3)) @ w[t].T for t, d in enumerate(TAPS))
        gf = g.reshape(-1, case["cout"])
        gw = torch.stack([torch.roll(x, tuple(-q for q in d), (1, 2, 3))
                          .reshape(-1, case["cin"]).T @ gf for d in TAPS])
        return {"y": torch.relu(_conv64(x, w, b)), "gx": gx, "gw": gw, "gb": gf.sum(0)}
    if kind == "predict":
        p = _weights(seed)
        d = _lognormal(case["D"], case["sigma"], _gen(seed))[None]
        with torch.no_grad():
            v = _unet64(d, np.array([case["fr0"]]), torch.as_tensor(p, device=DEV).double())
        return {"u": U_SCALE * torch.sinh(v[0])}
    p = _weights(seed)
    d, fr0, t = _train_inputs(case, seed)
    q = torch.as_tensor(p, device=DEV).double().requires_grad_()
    loss = (_unet64(d, fr0, q) - torch.asinh(t / U_SCALE)).square().mean()
    loss.backward()
    return {"loss": float(loss), "grads": q.grad.cpu().numpy()}
