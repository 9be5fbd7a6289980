"""Performance cases of the PW advection library, through its public entry points.

Each case names the entry point that it stands for in ``kind``:

``advect``     pw.advect into kept output fields: the call that a model makes once per time step.
``split``      one step of the mean + perturbation path from FP64 winds: pw.split_field of u, v, w, the
               host table from the three level means, pw.advect in mode "split".
``batch``      pw.Batch.run over many domains of uneven sizes (an ensemble or a nest), one launch.
``adjoint``    pw.advect_adjoint: the gradient of variational data assimilation.
``rollout``    forward-Euler steps under autograd with periodic halos and checkpoints, and their backward.
``energy``     pw.energy_budget: the FP64 conservation diagnostic of a step's winds and source terms.

Winds are sums of travelling sinusoids with 1 % noise and a 5 m/s mean of u (w = 0 on the ground and at the
lid), or i.i.d. uniform in [-10, 10] m/s; both periodic in x and y. Grids are uniform (20 m) or stretched
(10 m growing by 3 % a level), with or without an exponential density.
"""
import math
import random

import numpy as np
import torch

from paper_2107_13500_gb300 import autograd, pw

ES = {"f64": 8, "paired": 8, "f32": 4, "split": 4}
TORCH = {"f64": torch.float64, "paired": torch.float64, "f32": torch.float32, "split": torch.float32}


def listed():
    return [
        # A small domain (the 64-cubed correctness configuration) in FP64: latency, launches and host work count.
        dict(name="f64_64", kind="advect", mode="f64", nx=64, ny=64, nz=64, winds="iid", stretch=False, density=False, dx=50.0, dy=50.0, aligned=True),
        # The headline workload: 16.8M points, native FP64, smooth winds, stretched grid without density.
        dict(name="f64_512x512x64", kind="advect", mode="f64", nx=512, ny=512, nz=64, winds="modes", stretch=True, density=False, dx=50.0, dy=50.0, aligned=True),
        # Ragged sizes, density, dx != dy and fields that start on a 16-byte boundary (the scalar path), FP64.
        dict(name="f64_ragged_density", kind="advect", mode="f64", nx=1000, ny=250, nz=37, winds="modes", stretch=True, density=True, dx=40.0, dy=60.0, aligned=False),
        # The largest: 134M points in the default arithmetic (paired), i.i.d. winds.
        dict(name="paired_1024x1024x128", kind="advect", mode="paired", nx=1024, ny=1024, nz=128, winds="iid", stretch=False, density=False, dx=50.0, dy=50.0, aligned=True),
        # Float fields kept as such: the FP32 step of the same workload as the headline.
        dict(name="f32_512x512x64", kind="advect", mode="f32", nx=512, ny=512, nz=64, winds="modes", stretch=True, density=False, dx=50.0, dy=50.0, aligned=True),
        # FP64 winds evaluated through the mean + perturbation path, splitting included, with density.
        dict(name="split_step_512x512x64", kind="split", mode="split", nx=512, ny=512, nz=64, winds="modes", stretch=True, density=True, dx=50.0, dy=50.0, aligned=True),
        # Ensembles of uneven domains (x, y in 32..384, z in 32..128) in one launch: FP64-accurate and FP32.
        dict(name="batch_paired_20", kind="batch", mode="paired", domains=20, lo=32, hi=384, zlo=32, zhi=128, winds="iid", stretch=True, density=False, dx=50.0, dy=50.0, aligned=True),
        dict(name="batch_f32_20", kind="batch", mode="f32", domains=20, lo=32, hi=384, zlo=32, zhi=128, winds="iid", stretch=True, density=False, dx=50.0, dy=50.0, aligned=True),
        # The gradient of one evaluation: FP64 at the assimilation size, FP32 on the large workload.
        dict(name="adjoint_f64_256x256x64", kind="adjoint", mode="f64", nx=256, ny=256, nz=64, winds="iid", stretch=False, density=False, dx=50.0, dy=50.0, aligned=True),
        dict(name="adjoint_f32_512x512x64", kind="adjoint", mode="f32", nx=512, ny=512, nz=64, winds="modes", stretch=True, density=False, dx=50.0, dy=50.0, aligned=True),
        # A differentiable time integration and its backward (forward kernel, halo fill and fold, adjoint).
        dict(name="rollout_paired_4x256x256x64", kind="rollout", mode="paired", nx=256, ny=256, nz=64, steps=4, every=2, winds="modes", stretch=True, density=False, dx=50.0, dy=50.0, aligned=True),
        # The conservation diagnostic of the headline workload.
        dict(name="energy_512x512x64", kind="energy", mode="f64", nx=512, ny=512, nz=64, winds="modes", stretch=True, density=True, dx=50.0, dy=50.0, aligned=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("advect", "advect", "advect", "split", "batch", "adjoint", "adjoint", "rollout", "energy"))
    mode = {"advect": ("f64", "paired", "f32"), "split": ("split",), "batch": ("f64", "paired", "f32"), "adjoint": ("f64", "paired", "f32"),
            "rollout": ("f64", "paired"), "energy": ("f64", "f32")}[kind]
    case = dict(kind=kind, mode=rng.choice(mode), winds=rng.choice(("modes", "iid")), stretch=rng.random() < 0.6, density=rng.random() < 0.4,
                dx=rng.choice((50.0, 50.0, 40.0)), dy=50.0, aligned=rng.random() < 0.75)
    if kind == "batch":
        case.update(domains=rng.randint(4, 20), lo=32, hi=rng.randint(64, 384), zlo=32, zhi=rng.randint(33, 128))
        return case
    # the largest point count of each kind keeps a drawn case cheaper than the largest listed one
    most = {"advect": 40e6, "split": 20e6, "adjoint": 17e6, "rollout": 2e6, "energy": 20e6}[kind]
    while True:
        nx, ny, nz = _log_int(rng, 48, 1024), _log_int(rng, 48, 1024), _log_int(rng, 16, 128)
        if nx * ny * nz <= most:
            break
    case.update(nx=nx, ny=ny, nz=nz)
    if kind == "rollout":
        case.update(steps=rng.randint(2, 4), every=rng.choice((0, 2)))
    return case


# ---------------------------------------------------------------- inputs

def _dz(case, nz):
    return 10.0 * 1.03 ** np.maximum(np.arange(nz) - 1, 0) if case["stretch"] else np.full(nz, 20.0)


def _grid(case, nz):
    """dz, rho (w levels) and rhon (u levels); densities None without stratification."""
    dz = _dz(case, nz)
    if not case["density"]:
        return dz, None, None
    zw = np.concatenate([[0.0], np.cumsum(dz[1:])])
    zn = np.concatenate([[0.0], 0.5 * (zw[:-1] + zw[1:])])
    if nz > 1:
        zn[0] = -zn[1]
    return dz, 1.2 * np.exp(-zw / 8000.0), 1.2 * np.exp(-zn / 8000.0)


def _halo(t, nx, ny):
    t[:, :, 0] = t[:, :, nx]
    t[:, :, nx + 1] = t[:, :, 1]
    t[:, 0, :] = t[:, ny, :]
    t[:, ny + 1, :] = t[:, 1, :]
    return t


def _field(case, nx, ny, nz, gen, mean=0.0, rigid=False, dtype=torch.float64):
    f = pw.empty_field(nx, ny, nz, dtype, aligned=case["aligned"])
    if case["winds"] == "iid":
        val = torch.rand((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64).mul_(20.0).sub_(10.0)
    else:
        val = torch.rand((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64).mul_(0.1).add_(mean - 0.05)
        p = torch.rand((4, 2), generator=gen, device="cuda", dtype=torch.float64).cpu().numpy()
        q = torch.randint(1, 4, (4, 3), generator=gen, device="cuda").cpu().numpy()
        x, y, z = (torch.arange(n, device="cuda", dtype=torch.float64) / n for n in (nx, ny, nz))
        for m in range(4):
            ang = 2 * math.pi * (int(q[m, 0]) * x[None, :] + int(q[m, 1]) * y[:, None])
            ph = math.pi * int(q[m, 2]) * z + 2 * math.pi * float(p[m, 1])
            val.add_(torch.cos(ph)[:, None, None] * torch.sin(ang)[None], alpha=0.5 + 1.5 * float(p[m, 0]))
            val.add_(torch.sin(ph)[:, None, None] * torch.cos(ang)[None], alpha=0.5 + 1.5 * float(p[m, 0]))
        if rigid:
            val[0] = 0.0
            val[nz - 1] = 0.0
    f[:, 1:ny + 1, 1:nx + 1] = val
    return _halo(f, nx, ny)


def _winds(case, nx, ny, nz, gen, dtype):
    return [_field(case, nx, ny, nz, gen, 5.0, dtype=dtype), _field(case, nx, ny, nz, gen, dtype=dtype),
            _field(case, nx, ny, nz, gen, rigid=True, dtype=dtype)]


def _cotangents(case, nx, ny, nz, gen, dtype):
    out = []
    for _ in range(3):
        f = pw.empty_field(nx, ny, nz, dtype, aligned=case["aligned"])
        f[:, 1:ny + 1, 1:nx + 1] = torch.rand((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64).mul_(2.0).sub_(1.0)
        out.append(f)
    return out


def _sizes(case, seed):
    """Domain sizes of a batch: they belong to the case, not to the seed, so that every pass does the same work."""
    r = random.Random(4)
    return [(r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"]), r.randint(case["zlo"], case["zhi"])) for _ in range(case["domains"])]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    mode, kind = case["mode"], case["kind"]
    dt = TORCH[mode]
    if kind == "batch":
        doms = []
        for nx, ny, nz in _sizes(case, seed):
            dz, rho, rhon = _grid(case, nz)
            c = pw.make_coeffs(nz, case["dx"], case["dy"], dz, rho, rhon).to_device()
            u, v, w = _winds(case, nx, ny, nz, gen, dt)
            doms.append(dict(u=u, v=v, w=w, nx=nx, ny=ny, coeffs=c))
        return dict(case=case, batch=pw.Batch(doms, mode, 0))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dz, rho, rhon = _grid(case, nz)
    s = dict(case=case, coeffs=pw.make_coeffs(nz, case["dx"], case["dy"], dz, rho, rhon).to_device())
    if kind == "split":
        s["winds"] = _winds(case, nx, ny, nz, gen, torch.float64)
        s["pert"] = [pw.empty_field(nx, ny, nz, torch.float32, aligned=case["aligned"]) for _ in range(3)]
        s["out"] = tuple(pw.field_like(s["pert"][0]) for _ in range(3))
        return s
    s["winds"] = _winds(case, nx, ny, nz, gen, dt)
    if kind == "advect":
        s["out"] = tuple(pw.field_like(s["winds"][0]) for _ in range(3))
    elif kind == "adjoint":
        s["cot"] = _cotangents(case, nx, ny, nz, gen, dt)
        s["out"] = tuple(pw.field_like(s["winds"][0]) for _ in range(3))
    elif kind == "rollout":
        s["cot"] = _cotangents(case, nx, ny, nz, gen, dt)
    elif kind == "energy":
        s["tend"] = pw.advect(*s["winds"], s["coeffs"], nx, ny, mode=mode)
        s["weights"] = [torch.from_numpy(a).cuda() for a in pw.make_energy_weights(nz, dz, rho, rhon)]
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    case = s["case"]
    kind, mode = case["kind"], case["mode"]
    if kind == "batch":
        s["batch"].run()
        return [list(o) for o in s["batch"].outputs()]
    nx, ny, c = case["nx"], case["ny"], s["coeffs"]
    if kind == "advect":
        return list(pw.advect(*s["winds"], c, nx, ny, mode=mode, out=s["out"]))
    if kind == "split":
        means = [pw.split_field(f, nx, ny, out=p)[1] for f, p in zip(s["winds"], s["pert"])]
        table = torch.from_numpy(pw.make_split_table(c, *(m.cpu().numpy() for m in means))).cuda()
        out = pw.advect(*s["pert"], c, nx, ny, mode="split", split_table=table, out=s["out"])
        return dict(out=list(out), pert=s["pert"], means=means)
    if kind == "adjoint":
        return list(pw.advect_adjoint(*s["winds"], c, nx, ny, *s["cot"], mode=mode, out=s["out"]))
    if kind == "energy":
        return list(pw.energy_budget(*s["winds"], *s["tend"], nx, ny, *s["weights"]))
    x = [t.detach().requires_grad_() for t in s["winds"]]
    y = autograd.rollout(*x, c, nx, ny, 0.5, case["steps"], mode=mode, checkpoint_every=case["every"])
    g = torch.autograd.grad(y, x, s["cot"])
    return dict(state=[t.detach() for t in y], grad=list(g))


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    es = ES[case["mode"]]
    if case["kind"] == "batch":
        sizes = _sizes(case, 0)
    else:
        sizes = [(case["nx"], case["ny"], case["nz"])]
    cells = sum((nx + 2) * (ny + 2) * nz for nx, ny, nz in sizes)
    pts = sum(nx * ny * nz for nx, ny, nz in sizes)
    kind = case["kind"]
    if kind in ("advect", "batch"):
        return dict(bytes=3 * es * (cells + pts), flops=63 * pts)
    if kind == "split":
        # FP64 winds read, perturbations written and read again, source terms written
        return dict(bytes=3 * (8 + 4 + 4) * cells + 3 * 4 * pts, flops=(63 + 6) * pts)
    if kind == "adjoint":
        return dict(bytes=3 * es * (2 * cells + pts), flops=150 * pts)
    if kind == "energy":
        return dict(bytes=6 * es * pts, flops=9 * pts)
    # per step: forward (u, v, w in, the new state out) twice where it is recomputed, and the adjoint
    fwd = 3 * es * 2 * cells * (2 if case["every"] else 1)
    return dict(bytes=case["steps"] * (fwd + 3 * es * 3 * cells), flops=case["steps"] * 280 * pts)


# ---------------------------------------------------------------- the same in 64 bits

def _coeffs64(case, nz):
    """tcx, tcy and tzc1, tzc2, tzd1, tzd2 (numpy float64, level k at index k-1)."""
    dz, rho, rhon = _grid(case, nz)
    rw = np.ones(nz) if rho is None else rho
    rn = np.ones(nz) if rhon is None else rhon
    zw = np.concatenate([[0.0], np.cumsum(dz[1:])])
    zu = np.concatenate([[0.0], 0.5 * (zw[:-1] + zw[1:])])
    if nz > 1:
        zu[0] = -zu[1]
    c = np.zeros((4, nz))
    k = np.arange(1, nz)
    c[0, 1:] = 0.25 * rw[k - 1] / (rn[k] * dz[k])
    c[1, 1:] = 0.25 * rw[k] / (rn[k] * dz[k])
    k = np.arange(1, nz - 1)
    c[2, 1:nz - 1] = 0.25 * rn[k] / (rw[k] * (zu[k + 1] - zu[k]))
    c[3, 1:nz - 1] = 0.25 * rn[k + 1] / (rw[k] * (zu[k + 1] - zu[k]))
    return 0.25 / case["dx"], 0.25 / case["dy"], c


def _advect64(u, v, w, case, nx, ny):
    """su, sv, sw (nz, ny, nx) of double fields with halo, term by term."""
    nz = u.shape[0]
    tcx, tcy, c = _coeffs64(case, nz)
    c = [torch.from_numpy(a).to(u.device)[:, None, None] for a in c]

    def at(f, dj=0, di=0, k0=0, k1=None):
        return f[k0:k1, 1 + dj:1 + dj + ny, 1 + di:1 + di + nx]

    K = dict(k0=1)              # levels 2..nz
    D = dict(k0=0, k1=nz - 1)   # the level below each
    M = dict(k0=1, k1=nz - 1)   # levels 2..nz-1
    U = dict(k0=2, k1=nz)       # the level above each of those
    B = dict(k0=0, k1=nz - 2)   # the level below each of those
    zero = torch.zeros((nz, ny, nx), dtype=torch.float64, device=u.device)
    if nz < 2:
        return [zero, zero.clone(), zero.clone()]

    def horizontal(q, au, bu, av, bv, lv):
        """tcx[q(i-1) Fx(i-1/2) - q(i+1) Fx(i+1/2)] + tcy[...]: au + bu (av + bv) with (dj, di, level range)."""
        fx = lambda s: at(*au(s)) + at(*bu(s))
        fy = lambda s: at(*av(s)) + at(*bv(s))
        r = tcx * (at(q, 0, -1, *lv) * fx(-1) - at(q, 0, 1, *lv) * fx(0))
        return r + tcy * (at(q, -1, 0, *lv) * fy(-1) - at(q, 1, 0, *lv) * fy(0))

    k = (1, None)
    su = horizontal(u, lambda s: (u, 0, s, *k), lambda s: (u, 0, s + 1, *k), lambda s: (v, s, 0, *k), lambda s: (v, s, 1, *k), k)
    su = su + c[0][1:] * at(u, **D) * (at(w, **D) + at(w, 0, 1, **D))
    sv = horizontal(v, lambda s: (u, 0, s, *k), lambda s: (u, 1, s, *k), lambda s: (v, s, 0, *k), lambda s: (v, s + 1, 0, *k), k)
    sv = sv + c[0][1:] * at(v, **D) * (at(w, **D) + at(w, 1, 0, **D))
    sw = None
    if nz > 2:
        up = torch.zeros_like(su)
        up[:nz - 2] = c[1][1:nz - 1] * at(u, **U) * (at(w, **M) + at(w, 0, 1, **M))
        su = su - up
        up = torch.zeros_like(sv)
        up[:nz - 2] = c[1][1:nz - 1] * at(v, **U) * (at(w, **M) + at(w, 1, 0, **M))
        sv = sv - up
        m, n = (1, nz - 1), (2, nz)
        sw = horizontal(w, lambda s: (u, 0, s, *m), lambda s: (u, 0, s, *n), lambda s: (v, s, 0, *m), lambda s: (v, s, 0, *n), m)
        wc = at(w, **M)
        sw = sw + c[2][1:nz - 1] * at(w, **B) * (wc + at(w, **B)) - c[3][1:nz - 1] * at(w, **U) * (wc + at(w, **U))
    pad = lambda t, a, b: torch.cat([zero[:a], t, zero[:b]])
    return [pad(su, 1, 0), pad(sv, 1, 0), zero if sw is None else pad(sw, 1, 1)]


def _in_layout(vals, like, nx, ny):
    """Interior values in the layout of a zeroed output field."""
    out = []
    for t in vals:
        f = torch.zeros(like.shape, dtype=torch.float64, device=t.device)
        f[:, 1:ny + 1, 1:nx + 1] = t
        out.append(f)
    return out


def _wrap(i):
    """The interior i with a periodic halo, out of place and differentiable."""
    i = torch.cat([i[:, :, -1:], i, i[:, :, :1]], dim=2)
    return torch.cat([i[:, -1:], i, i[:, :1]], dim=1)


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "batch":
        return [_in_layout(_advect64(d["u"].double(), d["v"].double(), d["w"].double(), case, d["nx"], d["ny"]), d["u"], d["nx"], d["ny"])
                for d in s["batch"].domains]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x = [t.double() for t in s["winds"]]
    if kind == "advect":
        return _in_layout(_advect64(*x, case, nx, ny), s["winds"][0], nx, ny)
    if kind == "split":
        means = [f[:, 1:ny + 1, 1:nx + 1].mean(dim=(1, 2)) for f in x]
        pert = []
        for f, m, p in zip(x, means, s["pert"]):
            g = torch.zeros(p.shape, dtype=torch.float64, device=f.device)
            g[:, :, :nx + 2] = f[:, :, :nx + 2] - m[:, None, None]
            pert.append(g)
        return dict(out=_in_layout(_advect64(*x, case, nx, ny), s["pert"][0], nx, ny), pert=pert, means=means)
    if kind == "energy":
        level = torch.zeros((nz, 6), dtype=torch.float64, device="cuda")
        for f, (q, t) in enumerate(zip(x, s["tend"])):
            p = q[:, 1:ny + 1, 1:nx + 1] * t.double()[:, 1:ny + 1, 1:nx + 1]
            level[:, f], level[:, f + 3] = p.sum(dim=(1, 2)), p.abs().sum(dim=(1, 2))
        wt = torch.stack([s["weights"][i] for i in (0, 0, 1, 0, 0, 1)], dim=1)
        return [(wt * level).sum(dim=0), level]
    g = [t.double() for t in s["cot"]]
    x = [t[:, :, :nx + 2].clone().requires_grad_() for t in x]
    if kind == "adjoint":
        gr = torch.autograd.grad(_advect64(*x, case, nx, ny), x, [t[:, 1:ny + 1, 1:nx + 1] for t in g])
    else:
        y = x
        for _ in range(case["steps"]):
            t = _advect64(*y, case, nx, ny)
            y = [_wrap(f[:, 1:ny + 1, 1:nx + 1] + 0.5 * a) for f, a in zip(y, t)]
        gr = torch.autograd.grad(y, x, [t[:, :, :nx + 2] for t in g])

    def wide(ts):
        out = [torch.zeros(like.shape, dtype=torch.float64, device="cuda") for like in s["winds"]]
        for f, t in zip(out, ts):
            f[:, :, :nx + 2] = t.detach()
        return out

    return wide(gr) if kind == "adjoint" else dict(state=wide(y), grad=wide(gr))
