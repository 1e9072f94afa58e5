"""What a user of this library has it do, as cases that can be timed and checked.

Every case is one call sequence through the public binding (:mod:`paper_2605_01774_gb300.elbm`):
start a lattice from a concentration field, advance it, read the state back and, where a program
monitors its run, take the conservation diagnostics.  The families are the library's own
workloads: a decaying Fourier mode, an advected anisotropic plume, a two-phase porous medium
between Dirichlet faces, a stirred box (per-node velocity), a driven source benchmark, a sweep of
many small boxes, a gradient for per-node tensor parameters, and the two-dimensional channel.

``exact`` repeats a pass in FP64 with plain torch tensor operations.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2605_01774_gb300 import elbm as E

ELEM = {"f64": 8, "f32": 4, "f16dev": 2, "bf16dev": 2}


# ---------------------------------------------------------------------------- the cases
def listed():
    return [
        # A small test-sized plume: forty steps of a box that fits in a fraction of the chip; launches
        # and latency are all of it.
        dict(name="plume_24_f32", kind="plume", nx=24, ny=24, nz=24, prec="f32", steps=40, diagnostics=False),
        # Rotated Fourier mode at rest in FP64, 200 steps: the validation run of the tensor map.
        dict(name="decay_32_f64", kind="decay", nx=32, ny=32, nz=32, prec="f64", steps=200),
        # The anisotropic plume in FP64, the reference arithmetic of every error figure; uneven box.
        dict(name="plume_96_f64", kind="plume", nx=96, ny=80, nz=72, prec="f64", steps=20, diagnostics=True),
        # A porous sample of odd size (a cut of a scan) in FP32: tensor field, source, Dirichlet faces.
        dict(name="porous_121_f32", kind="porous", nx=121, ny=75, nz=50, prec="f32", steps=50),
        # The headline run: 256^3 plume in FP32, then the concentration and the diagnostics a
        # monitoring program reads.
        dict(name="plume_256_f32", kind="plume", nx=256, ny=256, nz=256, prec="f32", steps=12, diagnostics=True),
        # The same box with a wider plume in the 16-bit deviation storage.
        dict(name="plume_256_f16dev", kind="plume", nx=256, ny=256, nz=256, prec="f16dev", steps=16, width=16.0,
             diagnostics=False),
        # The large porous workload in the storage it is meant for.
        dict(name="porous_384_f16dev", kind="porous", nx=384, ny=384, nz=384, prec="f16dev", steps=20),
        # A box stirred by a velocity that differs in every node (FP32, uneven sides).
        dict(name="stirred_160_f32", kind="stirred", nx=160, ny=144, nz=128, prec="f32", steps=16),
        # The source-driven benchmark with a time-dependent source, in FP64 as it is published.
        dict(name="driven_128_f64", kind="driven", nx=128, ny=128, nz=128, prec="f64", steps=12),
        # An orientation sweep: 512 boxes of uneven size stepped together.
        dict(name="sweep_512", kind="sweep", boxes=512, nmin=16, nmax=96, steps=10),
        # One gradient of an inverse problem: forward sweep, checkpoints, reverse sweep.
        dict(name="inverse_64_f32", kind="inverse", nx=64, ny=64, nz=64, prec="f32", steps=32, every=8),
        # The two-dimensional channel with velocity and tensor fields, with its diagnostics.
        dict(name="channel_4096_f32", kind="channel", nx=4096, ny=4096, prec="f32", steps=40, fields=True,
             diagnostics=True),
    ]


def _side(rng, lo, hi):
    """A box side: log-uniform, odd and even alike."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi, most):
    while True:
        nx, ny, nz = (_side(rng, lo, hi) for _ in range(3))
        if rng.random() < 0.4:
            nx = max(8, nx // 8 * 8)                 # rows of whole 16-byte groups are common
        if nx * ny * nz <= most:
            return dict(nx=nx, ny=ny, nz=nz)


def draw(rng):
    kind = rng.choice(["plume", "plume", "plume", "decay", "porous", "porous", "stirred", "driven", "sweep",
                       "inverse", "channel", "channel"])
    if kind == "plume":
        prec = rng.choice(["f32", "f32", "f16dev", "f64"])
        most = 1.2e6 if prec == "f64" else 1.7e7
        box = _box(rng, 20, 110 if prec == "f64" else 400, most)
        steps = rng.randint(5, 20) if prec == "f64" else rng.randint(4, 12)
        return dict(kind=kind, **box, prec=prec, steps=steps, diagnostics=rng.random() < 0.5)
    if kind == "decay":
        prec = rng.choice(["f64", "f32"])
        return dict(kind=kind, **_box(rng, 16, 80, 3e5), prec=prec, steps=rng.randint(20, 200))
    if kind == "porous":
        prec = rng.choice(["f32", "f16dev", "bf16dev", "f64"])
        most = 1e6 if prec == "f64" else 2e7
        return dict(kind=kind, **_box(rng, 24, 100 if prec == "f64" else 400, most), prec=prec,
                    steps=rng.randint(5, 40))
    if kind == "stirred":
        return dict(kind=kind, **_box(rng, 24, 200, 4e6), prec="f32", steps=rng.randint(5, 16))
    if kind == "driven":
        n = _side(rng, 32, 120)
        prec = rng.choice(["f64", "f32"])
        return dict(kind=kind, nx=n, ny=n, nz=n, prec=prec, steps=rng.randint(4, 12))
    if kind == "sweep":
        nmin = rng.randint(8, 32)
        return dict(kind=kind, boxes=_side(rng, 16, 256), nmin=nmin, nmax=rng.randint(nmin + 8, 96),
                    steps=rng.randint(4, 20))
    if kind == "inverse":
        prec = rng.choice(["f32", "f64"])
        most = 3e4 if prec == "f64" else 2.7e5
        return dict(kind=kind, **_box(rng, 16, 80, most), prec=prec,
                    steps=rng.randint(30, 100) if prec == "f64" else rng.randint(12, 32), every=rng.randint(6, 40))
    prec = rng.choice(["f32", "f32", "f64"])
    hi = 700 if prec == "f64" else 4096
    return dict(kind=kind, nx=_side(rng, 64, hi), ny=_side(rng, 64, hi), prec=prec, steps=rng.randint(10, 40),
                fields=rng.random() < 0.6, diagnostics=rng.random() < 0.5)


# --------------------------------------------------------------------------- the inputs
def _rotation(angles):
    """Rz(a) Ry(b) Rz(c) as a 3x3 list; angles are floats or equally shaped tensors."""
    a, b, c = angles
    trig = (lambda t: (torch.cos(t), torch.sin(t))) if torch.is_tensor(a) else (lambda t: (math.cos(t), math.sin(t)))
    (ca, sa), (cb, sb), (cc, sc) = trig(a), trig(b), trig(c)
    return [[ca * cb * cc - sa * sc, -ca * cb * sc - sa * cc, ca * sb],
            [sa * cb * cc + ca * sc, -sa * cb * sc + ca * cc, sa * sb],
            [-sb * cc, sb * sc, cb]]


_UPPER = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


def _tensor6(eig, rot):
    """(xx, xy, xz, yy, yz, zz) of R diag(eig) R^T."""
    return [sum(rot[r][k] * eig[k] * rot[s][k] for k in range(3)) for r, s in _UPPER]


def _haar(g):
    return (g.uniform(0, 2 * math.pi), math.acos(g.uniform(-1, 1)), g.uniform(0, 2 * math.pi))


def _axes(case, dev="cuda"):
    """Node coordinates, FP64, each shaped to broadcast over [Nz, Ny, Nx]."""
    ax = [torch.arange(case[k], dtype=torch.float64, device=dev) for k in ("nx", "ny", "nz")]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _bump(case, centre, width):
    """Gaussian bump over the nodes, FP64 [Nz, Ny, Nx]."""
    x, y, z = _axes(case)
    r2 = (x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2
    return torch.exp(-0.5 * r2 / width ** 2)


def _smooth_noise(case, seed, sigma):
    """Zero-mean noise of unit variance, low-passed over about `sigma` nodes, FP32 [Nz, Ny, Nx]."""
    shape = (case["nz"], case["ny"], case["nx"])
    sigma = min(sigma, min(shape) / 6.0)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, device="cuda"))
    k = [torch.fft.fftfreq(n, device="cuda") for n in shape[:2]] + [torch.fft.rfftfreq(shape[2], device="cuda")]
    for axis, kk in enumerate(k):
        f *= torch.exp(-2.0 * (math.pi * sigma * kk) ** 2).reshape([-1 if a == axis else 1 for a in range(3)])
    n = torch.fft.irfftn(f, s=shape)
    n -= n.mean()
    return n / n.std().clamp_min(1e-12)


def _inputs(case, seed):
    """Everything a pass is given, from the case and the seed alone.  Fields are GPU tensors of the
    element type that the library takes; uniform tensors and velocities are lists of floats."""
    g = np.random.Generator(np.random.PCG64(seed))
    real = torch.float64 if case.get("prec") == "f64" else torch.float32
    kind, p = case["kind"], {}
    dims = [case[k] for k in ("nx", "ny", "nz") if k in case]
    mid = [(n - 1) / 2.0 for n in dims]
    if kind == "decay":
        x, y, z = _axes(case)
        wave = 2 * math.pi * (x / case["nx"] + y / case["ny"] + 0 * z)
        p["D"] = _tensor6((0.05, 0.005, 0.0005), _rotation(_haar(g)))
        p["phi0"] = (1.0 + 0.1 * torch.sin(wave + g.uniform(0, 2 * math.pi))).to(real)
        p["u"] = [0.0, 0.0, 0.0]
    elif kind == "plume":
        p["D"] = _tensor6((0.1, 1e-3, 1e-5), _rotation(_haar(g)))
        p["u"] = [0.05 * g.uniform(0.8, 1.2), 0.03 * g.uniform(0.8, 1.2), 0.02 * g.uniform(0.8, 1.2)]
        # the plume is 8 nodes wide, narrower where the box is small
        width = case.get("width", min(8.0, min(dims) / 6.0))
        p["phi0"] = _bump(case, [m + g.uniform(-1, 1) for m in mid], width).to(real)
    elif kind == "porous":
        pore = _smooth_noise(case, seed, 3.0)
        some = pore.reshape(-1)[:: max(1, pore.numel() // 1000000)]
        pore = pore <= torch.quantile(some, 0.6)
        x, y, z = (t.to(torch.float32) for t in _axes(case))
        angles = []
        for _ in range(3):
            kx, ky, kz = (int(v) for v in g.integers(1, 3, size=3))
            ph = 2 * math.pi * (kx * x / dims[0] + ky * y / dims[1] + kz * z / dims[2]) + g.uniform(0, 2 * math.pi)
            angles.append(g.uniform(0, 2 * math.pi) + 0.5 * torch.sin(ph))
        eig = [torch.where(pore, a, b) for a, b in zip((3e-2, 3e-3, 1e-6), (1e-2, 1e-4, 1e-6))]
        rot = _rotation(angles)
        # formed in FP64 plane by plane, so that the rounded tensor stays positive definite
        p["D_field"] = torch.stack([sum(rot[r][k].double() * eig[k].double() * rot[s][k].double()
                                        for k in range(3)).to(torch.float32) for r, s in _UPPER])
        p["source"] = (1e-4 * _bump(case, mid, min(16.0, min(dims) / 6.0))).to(torch.float32)
        p["phi0"] = (2.0 - (x + 0.5) / dims[0] + torch.zeros_like(pore, dtype=torch.float32)).to(real)
        p["walls"] = (2.0, 1.0)
        p["u"] = [0.0, 0.0, 0.0]
    elif kind == "stirred":
        x, y, z = (2 * math.pi * t / n for t, n in zip(_axes(case), dims))
        a, b, c = (g.uniform(0, 2 * math.pi) for _ in range(3))
        one = torch.ones(dims[::-1], dtype=torch.float64, device="cuda")
        # a divergence-free stirring flow
        p["u_field"] = torch.stack([0.04 * (torch.sin(y + a) + torch.cos(z + b)) * one,
                                    0.04 * (torch.sin(z + c) + torch.cos(x + a)) * one,
                                    0.04 * (torch.sin(x + b) + torch.cos(y + c)) * one]).to(torch.float32)
        p["D"] = _tensor6((0.05, 0.01, 0.002), _rotation(_haar(g)))
        p["phi0"] = (0.1 + _bump(case, mid, min(8.0, min(dims) / 6.0))).to(real)
    elif kind == "driven":
        n = case["nx"]
        x, y, z = (2 * math.pi * t / n for t in _axes(case))
        shift, d = 2.0, (1e-2, 1e-2, 1e-6)
        shape = torch.sin(x) * torch.sin(y) * torch.sin(z)
        field = torch.zeros((6,) + tuple(shape.shape), dtype=torch.float64, device="cuda")
        field[0], field[3], field[5] = d[0] * (2.0 - shape), d[1], d[2]
        p["D_field"] = field.to(torch.float32)
        p["u"] = [v / n for v in (1.0, g.uniform(0.8, 1.2), g.uniform(0.8, 1.2))]
        p["phi0"] = (shift + shape).to(real)
        rate = 1.0 - 4 * math.pi ** 2 * (2 * d[0] + d[1] + d[2])
        p["source"] = (shape * (1.0 + 4 * math.pi ** 2 * d[0] * torch.sin(y) * torch.sin(z))
                       + 2 * math.pi * (torch.cos(x) * torch.sin(y) * torch.sin(z))).to(torch.float32)
        dt = 1.0 / n ** 2
        p["amplitudes"] = dt * np.exp(rate * (np.arange(case["steps"]) + 0.5) * dt)
    elif kind == "sweep":
        # the sizes of the boxes belong to the case: every seed has the same ones
        sizes = np.random.Generator(np.random.PCG64(case["boxes"]))
        p["edges"] = sizes.integers(case["nmin"], case["nmax"] + 1, size=case["boxes"]).astype(np.int32)
        tensors, start = [], []
        for n in p["edges"]:
            r = 10.0 ** g.uniform(0.0, 4.0)
            tensors.append(_tensor6((0.05, 0.05 / math.sqrt(r), 0.05 / r), _rotation(_haar(g))))
            t = 2 * math.pi * torch.arange(int(n), device="cuda", dtype=torch.float64) / int(n)
            wave = 1.0 + 0.1 * torch.sin(t[None, :] + t[:, None] + g.uniform(0, 2 * math.pi))
            start.append(wave.to(torch.float32).reshape(-1).repeat(int(n)))
        p["D"], p["phi0"] = np.array(tensors), torch.cat(start)
    elif kind == "inverse":
        p["u"] = [0.02, 0.0, 0.0]
        th = [math.log(d) + 0.3 * _smooth_noise(case, seed + 101 + k, 6.0).double()
              for k, d in enumerate((1e-2, 1e-3, 1e-4))]
        th += [g.uniform(0, 2 * math.pi) + 0.5 * _smooth_noise(case, seed + 104 + k, 6.0).double() for k in range(3)]
        width = min(6.0, min(dims) / 6.0)
        p["theta"] = torch.stack(th).to(real)
        p["phi0"] = (0.1 + _bump(case, mid, width)).to(real)
        p["obs"] = [max(1, case["steps"] // 2), case["steps"]]
        # snapshots of a plume that went elsewhere: the first gradients of an inversion
        p["targets"] = torch.stack([0.1 + 0.6 * _bump(case, [mid[0] + 0.05 * t, mid[1], mid[2] + 0.03 * t],
                                                      1.2 * width) for t in p["obs"]]).to(real)
        p["guard"] = 1e-8 if case["prec"] == "f64" else 3e-4
    else:  # channel
        nx, ny = dims
        x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
        y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
        s = torch.sin(2 * math.pi * (y + 0.5) / ny + g.uniform(0, 1))
        weak = 10.0 ** g.uniform(-4, -2)
        if case["fields"]:
            one = torch.ones((ny, nx), dtype=torch.float64, device="cuda")
            p["u_field"] = torch.stack([0.04 * (0.5 + 0.5 * s) * one,
                                        -0.01 * torch.cos(2 * math.pi * y / ny) * one]).to(torch.float32)
            ang = 0.6 + 0.8 * s + 0.1 * torch.sin(2 * math.pi * x / nx)
            a, b = 0.03 * (1 + 0.3 * s) * one, weak * (1 + 0.2 * torch.cos(2 * math.pi * y / ny)) * one
            c, sn = torch.cos(ang), torch.sin(ang)
            p["D_field"] = torch.stack([c * c * a + sn * sn * b, c * sn * (a - b), sn * sn * a + c * c * b]
                                       ).to(torch.float32)
        else:
            p["u"] = [0.04, 0.01 * g.uniform(0.5, 1.5)]
            c, sn = math.cos(0.6), math.sin(0.6)
            p["D"] = [c * c * 0.03 + sn * sn * weak, c * sn * (0.03 - weak), sn * sn * 0.03 + c * c * weak]
        p["phi0"] = (1.0 + 0.5 * torch.exp(-((x - nx / 2) ** 2 / (2 * (nx / 6) ** 2)
                                             + (y - ny / 2) ** 2 / (2 * (ny / 5) ** 2)))).to(real)
    return p


# ------------------------------------------------------------------------------ a pass
class _Handle:
    """A handle that is given back with the state that holds it."""

    def __init__(self, h, destroy):
        self.h, self._destroy = h, destroy

    def __del__(self):
        self._destroy(self.h)


def _reads_phi_only(case):
    """Programs that keep 16-bit deviations of a plume read its concentration; all others read the
    whole state."""
    return case["kind"] == "plume" and case["prec"] in ("f16dev", "bf16dev")


def prepare(case, seed):
    p = _inputs(case, seed)
    kind = case["kind"]
    real = torch.float64 if case.get("prec") == "f64" else torch.float32
    s = dict(case=case, p=p)
    if kind == "sweep":
        h = E.elbm_batch_create(p["edges"], p["D"])
        s["handle"] = _Handle(h, E.elbm_batch_destroy)
        s["phi"] = torch.empty_like(p["phi0"])
        s["pops"] = torch.empty((27,) + (int(p["edges"][0]),) * 3, dtype=torch.float32, device="cuda")
        return s
    if kind == "inverse":
        h = E.elbm_adjoint_create((case["nx"], case["ny"], case["nz"]), case["prec"])
        s["handle"] = _Handle(h, E.elbm_adjoint_destroy)
        E.elbm_adjoint_configure(h, p["u"], p["guard"], case["every"])
        s["grad"] = torch.empty_like(p["theta"])
        return s
    if kind == "channel":
        lat = E.Lattice2D((case["nx"], case["ny"]), case["prec"])
        if case["fields"]:
            E.elbm2d_set_tensor_field(lat.h, p["D_field"])
            E.elbm2d_set_velocity_field(lat.h, p["u_field"])
        else:
            E.elbm2d_set_tensor_uniform(lat.h, p["D"])
            E.elbm2d_set_velocity_uniform(lat.h, p["u"])
        s["handle"] = lat
        s["phi"] = torch.empty((case["ny"], case["nx"]), dtype=real, device="cuda")
        s["pops"] = torch.empty((9, case["ny"], case["nx"]), dtype=real, device="cuda")
        return s
    dims = (case["nx"], case["ny"], case["nz"])
    lat = E.Lattice(dims, case["prec"], bc=p.get("walls"))
    if "D_field" in p:
        E.elbm_set_tensor_field(lat.h, p["D_field"])
    else:
        E.elbm_set_tensor_uniform(lat.h, p["D"])
    if "u_field" in p:
        E.elbm_set_velocity_field(lat.h, p["u_field"])
    else:
        E.elbm_set_velocity_uniform(lat.h, p["u"])
    if "source" in p:
        E.elbm_set_source(lat.h, p["source"])
    s["handle"] = lat
    s["phi"] = torch.empty(dims[::-1], dtype=real, device="cuda")
    if case["prec"] == "f64":
        s["flux"] = torch.empty((3,) + dims[::-1], dtype=real, device="cuda")
    if not _reads_phi_only(case):
        s["pops"] = torch.empty((27,) + dims[::-1], dtype=real, device="cuda")
    return s


def run(s):
    case, p, h = s["case"], s["p"], s["handle"].h
    kind = case["kind"]
    if kind == "sweep":
        E.elbm_batch_init_equilibrium(h, p["phi0"])
        E.elbm_batch_step(h, case["steps"], 0)
        E.elbm_batch_read_phi(h, s["phi"])
        E.elbm_batch_read_populations(h, 0, s["pops"])
        return {"phi": s["phi"], "populations": s["pops"]}
    if kind == "inverse":
        J, _ = E.elbm_adjoint_misfit(h, p["theta"], p["phi0"], case["steps"], p["obs"], p["targets"], s["grad"])
        return {"J": J, "grad": s["grad"]}
    if kind == "channel":
        E.elbm2d_init_equilibrium(h, p["phi0"])
        E.elbm2d_step(h, case["steps"])
        E.elbm2d_read_moments(h, s["phi"])
        E.elbm2d_read_populations(h, s["pops"])
        out = {"phi": s["phi"], "populations": s["pops"]}
        if case["diagnostics"]:
            d = E.elbm2d_reduce(h)
            out.update(mass=d["mass"], entropy=d["entropy"], gmin=d["gmin"])
        return out
    E.elbm_init_equilibrium(h, p["phi0"])
    if "amplitudes" in p:
        E.elbm_step_source_schedule(h, p["amplitudes"])
    else:
        E.elbm_step(h, case["steps"])
    E.elbm_read_moments(h, s["phi"], s.get("flux"))
    out = {"phi": s["phi"]}
    if "flux" in s:
        out["flux"] = s["flux"]
    if "pops" in s:
        E.elbm_read_populations(h, s["pops"])
        out["populations"] = s["pops"]
    if case.get("diagnostics"):
        d = E.elbm_reduce(h)
        # the plume's far tails round to about zero, so its smallest population says nothing
        out.update(mass=d["mass"], entropy=d["entropy"])
    return out


# ------------------------------------------------------------------ what a pass must do
def work(case):
    """Bytes and operations of one pass: the start read and the state written once, every step
    reads and writes the whole state and reads the per-node fields, and each read-out reads the
    state and writes its result."""
    kind, steps = case["kind"], case["steps"]
    if kind == "sweep":
        n = case["boxes"] * sum(e ** 3 for e in range(case["nmin"], case["nmax"] + 1)) / (case["nmax"] + 1 - case["nmin"])
        return {"bytes": n * (216 * steps + 112 + 112), "flops": n * 330 * steps}
    if kind == "inverse":
        n, e = case["nx"] * case["ny"] * case["nz"], ELEM[case["prec"]]
        # forward once, and one reverse step per step: state, adjoint state in and out, tensor
        return {"bytes": n * steps * e * ((54 + 6) + (81 + 6 + 12)), "flops": n * steps * (700 + 1500)}
    e = ELEM[case["prec"]]
    real = 8 if case["prec"] == "f64" else 4
    if kind == "channel":
        n = case["nx"] * case["ny"]
        state = 9 * e
        per = 2 * state + ((3 * e + 8) if case["fields"] else 0)
        reads = (state + real) + 2 * state + (state if case["diagnostics"] else 0)
        return {"bytes": n * (real + state + per * steps + reads), "flops": n * steps * (330 if case["fields"] else 220)}
    n = case["nx"] * case["ny"] * case["nz"]
    state = 27 * e + (4 if e == 2 else 0)
    fields = (6 * real if kind in ("porous", "driven") else 0) + (4 if kind in ("porous", "driven") else 0)
    fields += 12 if kind == "stirred" else 0
    reads = state + real * (4 if case["prec"] == "f64" else 1)
    reads += 0 if _reads_phi_only(case) else state + 27 * real
    reads += state if case.get("diagnostics") else 0
    still = kind in ("decay", "porous")
    return {"bytes": n * (real + state + (2 * state + fields) * steps + reads),
            "flops": n * steps * (330 if still else 1000 if kind == "stirred" else 700)}


# -------------------------------------------------------------------- the same in FP64
def _velocities(d):
    """Velocities [Q][d] in the library's order and weights [Q] of the tensor-product set."""
    one = (-1, 0, 1)
    cs = [(a, b) for a in one for b in one] if d == 2 else [(a, b, c) for a in one for b in one for c in one]
    w = [math.prod(2 / 3 if v == 0 else 1 / 6 for v in c) for c in cs]
    return cs, torch.tensor(cs, dtype=torch.float64, device="cuda"), torch.tensor(w, dtype=torch.float64, device="cuda")


def _complement(D):
    """T = 2I - (I/2 + 3D)^-1 = 12 D (I + 6D)^-1 for D [..., d, d]."""
    eye = torch.eye(D.shape[-1], dtype=torch.float64, device=D.device)
    return 12.0 * torch.linalg.solve(eye + 6.0 * D, D)


def _full(d6):
    """Full matrices [..., d, d] of packed symmetric components ([6, ...] or [3, ...])."""
    if len(d6) == 3:
        rows = [[d6[0], d6[1]], [d6[1], d6[2]]]
    else:
        rows = [[d6[0], d6[1], d6[2]], [d6[1], d6[3], d6[4]], [d6[2], d6[4], d6[5]]]
    return torch.stack([torch.stack(r, -1) for r in rows], -2)


class _Exact:
    """One lattice in FP64 (d = 2 or 3), state [Q, Nd..N1]."""

    def __init__(self, d, u, T, theta, walls=None, source=None, fallback=True):
        self.cs, self.c, self.w = _velocities(d)
        self.u, self.T, self.theta, self.walls, self.source, self.fallback = u, T, theta, walls, source, fallback
        self.moving = bool((u != 0).any())
        node = (1,) * d
        self.wb = self.w.reshape((-1,) + node)
        ub = u if u.dim() > 1 else u.reshape((-1,) + node)
        cu = torch.tensordot(self.c, ub, dims=1)
        uu = (ub * ub).sum(0)
        self.ub, self.P = ub, 1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu
        self.K = 1 / self.P - 1
        self.L = torch.log(self.P) - 3 * cu + 1.5 * uu
        self.still = (ub == 0).all(0)

    def start(self, phi0):
        return phi0 * (self.wb * self.P)

    def collide(self, g):
        w, c = self.wb, self.c
        phi = g.sum(0)
        j = torch.tensordot(c.T.contiguous(), g, dims=1) - phi * self.ub
        if self.T.dim() == 2:
            Tj = torch.tensordot(self.T, j, dims=1)
        else:
            Tj = torch.einsum("...ab,b...->a...", self.T, j)
        a = Tj - j
        out = phi * (w * self.P) + 3 * w * torch.tensordot(c, a, dims=1)
        if self.moving:
            dh = g - phi * (w * self.P) - 3 * w * torch.tensordot(c, j, dims=1)
            safe = torch.where(phi > 0, phi, torch.ones_like(phi))
            den = (dh * dh / (w * self.P)).sum(0) / safe
            num = (dh * (3 * self.K * torch.tensordot(c, a, dims=1) / safe + self.L)).sum(0)
            on = (phi > 1e-300) & (den > self.theta ** 2 * phi) & ~self.still
            out = out - torch.where(on, num / torch.where(on, den, torch.ones_like(den)), torch.zeros_like(den)) * dh
            del dh
        if self.fallback:
            need = (out < 0).any(0)
            if bool(need.any()):
                om = out - g
                ratio = torch.where(om < 0, g / torch.where(om < 0, -om, torch.ones_like(om)),
                                    torch.full_like(om, math.inf)).amin(0).clamp(0, 1)
                out = g + torch.where(need, ratio, torch.ones_like(ratio)) * om
        return out

    def stream(self, post):
        d = post.dim() - 1
        planes = []
        for i, cv in enumerate(self.cs):
            r = torch.roll(post[i], shifts=tuple(cv), dims=tuple(range(d - 1, -1, -1)))
            if self.walls is not None and cv[0] != 0:
                face = 0 if cv[0] > 0 else -1
                wall = self.walls[0] if cv[0] > 0 else self.walls[1]
                r[..., face] = 2 * self.w[i] * wall - post[len(self.cs) - 1 - i][..., face]
            planes.append(r)
        return torch.stack(planes)

    def step(self, g, amplitude=1.0):
        if self.source is None:
            return self.stream(self.collide(g))
        half = 0.5 * amplitude * self.source * (self.wb * self.P)
        return self.stream(self.collide(g + half)) + half


def _diagnostics(g, w):
    pos = g > 0
    mass, h = 0.0, 0.0
    for i in range(len(w)):
        mass += float(g[i].sum())
        v = g[i][pos[i]]
        h += float((v * torch.log(v / w[i])).sum())
    return mass, h


def exact(case, seed):
    p = _inputs(case, seed)
    kind = case["kind"]
    f64 = lambda v: torch.as_tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
    if kind == "sweep":
        phi, first, at = [], None, 0
        for n, d6 in zip(p["edges"], p["D"]):
            n = int(n)
            lat = _Exact(3, f64([0.0, 0.0, 0.0]), _complement(_full(f64(d6))), 1e-8)
            g = lat.start(p["phi0"][at:at + n ** 3].double().reshape(n, n, n))
            for _ in range(case["steps"]):
                g = lat.step(g)
            phi.append(g.sum(0).reshape(-1))
            first = g if first is None else first
            at += n ** 3
        return {"phi": torch.cat(phi), "populations": first}
    if kind == "inverse":
        return _exact_inverse(case, p)
    if kind == "channel":
        d, key = 2, "f64"
    else:
        d, key = 3, "f64"
    D = p["D_field"].double() if "D_field" in p else f64(p["D"])
    u = p["u_field"].double() if "u_field" in p else f64(p["u"])
    T = _complement(_full(D))
    del D
    lat = _Exact(d, u, T, 1e-8 if case["prec"] == key else 3e-4, p.get("walls"),
                 p["source"].double() if "source" in p else None)
    g = lat.start(p["phi0"].double())
    amp = p.get("amplitudes", [1.0] * case["steps"])
    for a in amp:
        g = lat.step(g, float(a))
    out = {"phi": g.sum(0)}
    if d == 3 and case["prec"] == "f64":
        j = torch.tensordot(lat.c.T.contiguous(), g, dims=1) - out["phi"] * lat.ub
        out["flux"] = 0.5 * (torch.tensordot(T, j, dims=1) if T.dim() == 2 else torch.einsum("...ab,b...->a...", T, j))
    if d == 2 or not _reads_phi_only(case):
        out["populations"] = g
    if case.get("diagnostics"):
        out["mass"], out["entropy"] = _diagnostics(g, lat.w)
        if d == 2:
            out["gmin"] = float(g.min())
    return out


def _exact_inverse(case, p):
    """Misfit and gradient by reverse-mode differentiation through the FP64 steps."""
    theta = p["theta"].double().requires_grad_(True)
    u = torch.as_tensor(p["u"], dtype=torch.float64, device="cuda")
    target = p["targets"].double()

    def tensor(th):
        R = _rotation((th[3], th[4], th[5]))
        t = [12 * torch.exp(th[k]) / (1 + 6 * torch.exp(th[k])) for k in range(3)]
        return _full(torch.stack(_tensor6(t, R)))

    def some(g, th, n):
        lat = _Exact(3, u, tensor(th), p["guard"], fallback=False)
        for _ in range(n):
            g = lat.step(g)
        return g

    g = _Exact(3, u, torch.zeros(3, 3, dtype=torch.float64, device="cuda"), p["guard"]).start(p["phi0"].double())
    J, at = 0.0, 0
    for o, t in enumerate(p["obs"]):
        while at < t:
            n = min(5, t - at)
            g = torch.utils.checkpoint.checkpoint(some, g, theta, n, use_reentrant=False)
            at += n
        J = J + 0.5 * ((g.sum(0) - target[o]) ** 2).sum()
    J.backward()
    return {"J": float(J.detach()), "grad": theta.grad}
