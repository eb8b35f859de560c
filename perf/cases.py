"""What the framework's users have it do, as timed cases.

A case is one pass through the public entry points: a solver (or a batch of
boxes) is advanced by a number of Tau1 steps and its state is read out. The
boxes, media, faces and storage formats are those of the benchmark, the
profiles, the tests and the paper's own set-ups: a channel, overlapping-sphere
porous media, the 2D channel driven by constant-density faces, the porosity
layouts, and a mix of boxes as the serving loop steps it.

Outputs are the state in the precision that the solver holds it in: FP64 boxes
return float64 fields, FP32 boxes float32, FP16S float16, BF16S bfloat16 (the
export of FP32 and BF16S storage is exact, so nothing is lost by that).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_14742_gb300 import Batch, Tau1
from paper_2312_14742_gb300 import lbm

STATE = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f16s": 2, "bf16s": 2}
G = (1e-5, 2e-6, -3e-6)


def _box(name, q, nx, ny, nz, storage, steps, phi=0.9, radius=8.0, layout="dense", walls="", faces=False, check=False):
    """walls: the axes that are not periodic, their first and last planes solid
    (unless they carry the constant-density faces, which lie on x)."""
    return {"name": name, "q": q, "nx": nx, "ny": ny, "nz": nz, "storage": storage, "steps": steps, "phi": phi,
            "radius": radius, "layout": layout, "walls": walls, "faces": faces, "check": check}


def listed():
    return [
        # the validation channel, stepped between convergence checks: launches and latency
        _box("channel_32_f32", 19, 32, 32, 32, "f32", 100, phi=1.0, walls="z", check=True),
        # the paper's 2D pressure-driven validation channel, in FP64
        _box("channel2d_1000x100_f64", 9, 1000, 100, 1, "f64", 100, phi=1.0, walls="xy", faces=True),
        # the benchmark's box: overlapping spheres at porosity 0.9
        _box("porous_256_q19_f32", 19, 256, 256, 256, "f32", 40),
        # the same medium on the larger lattice
        _box("porous_256_q27_f32", 27, 256, 256, 256, "f32", 30),
        # the largest box: the paper's dense 512 x 256 x 256, in the capacity-saving format
        _box("porous_512x256x256_q19_bf16s", 19, 512, 256, 256, "bf16s", 20),
        # a user's own box: sizes that fit no tile, walls on two axes
        _box("duct_250x130x90_q19_f32", 19, 250, 130, 90, "f32", 60, phi=0.85, radius=6.0, walls="yz"),
        # odd sizes in scaled FP16
        _box("porous_161x127x101_q19_f16s", 19, 161, 127, 101, "f16s", 70, phi=0.8, radius=6.0),
        # an FP64 run, as for a reference permeability
        _box("porous_128_q19_f64", 19, 128, 128, 128, "f64", 12, phi=0.8, radius=6.0),
        # few fluid nodes: the compact and the sparse layout
        _box("compact_320_phi03_f32", 19, 320, 320, 320, "f32", 16, phi=0.3, radius=12.0, layout="compact"),
        _box("sparse_192_phi025_f32", 19, 192, 192, 192, "f32", 40, phi=0.25, radius=8.0, layout="sparse"),
        # the paper's 2D performance size
        _box("channel2d_4000_f32", 9, 4000, 4000, 1, "f32", 40, phi=1.0, walls="xy", faces=True),
        # a mix of boxes stepped together between two convergence checks, as the serving loop does
        {"name": "serving_mix_f32", "batch": True, "q": 19, "storage": "f32", "steps": 100, "boxes": 12,
         "min_edge": 32, "max_edge": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("dense", "dense", "dense", "plane", "compact", "sparse", "batch"))
    if kind == "batch":
        c = {"batch": True, "q": rng.choice((19, 27)), "storage": rng.choice(("f32", "f16s", "bf16s")),
             "steps": rng.choice((100, 130)), "boxes": rng.randint(3, 14), "min_edge": 32,
             "max_edge": rng.choice((64, 96, 128))}
        return c
    if kind == "plane":
        nx, ny = _log(rng, 60, 4000), _log(rng, 40, 3000)
        c = _box("", 9, nx, ny, 1, rng.choice(("f64", "f32", "f16s", "bf16s")) if nx * ny < 1 << 21 else
                 rng.choice(("f32", "f16s", "bf16s")), rng.choice((40, 64)), phi=1.0, walls="xy",
                 faces=rng.random() < 0.7)
    elif kind == "dense":
        storage = rng.choice(("f32", "f32", "f64", "f16s", "bf16s"))
        top = 120 if storage == "f64" else 260
        if rng.random() < 0.5:  # sizes that a user rounds to
            s = [16 * max(1, _log(rng, 24, top) // 16) for _ in range(3)]
        else:
            s = [_log(rng, 24, top) for _ in range(3)]
        c = _box("", rng.choice((19, 19, 27)), *s, storage, 10 if storage == "f64" else rng.choice((20, 40)),
                 phi=round(rng.uniform(0.5, 1.0), 2), radius=round(rng.uniform(3.0, 10.0), 1),
                 walls=rng.choice(("", "", "z", "yz", "x")), check=rng.random() < 0.2)
    else:
        s = [32 * rng.randint(1, 9) if rng.random() < 0.7 else _log(rng, 32, 288) for _ in range(3)]
        c = _box("", rng.choice((19, 19, 27)), *s, rng.choice(("f32", "f32", "bf16s")), rng.choice((10, 20)),
                 phi=round(rng.uniform(0.15, 0.6), 2), radius=round(rng.uniform(5.0, 12.0), 1), layout=kind,
                 walls=rng.choice(("", "z")))
    c.pop("name")
    return c


# ---- inputs ------------------------------------------------------------------------------

def _spheres(shape, radius, phi, seed):
    """Overlapping spheres at uniform random centres, periodic, with as many
    spheres as a porosity phi takes in the mean; a uint8 mask on the GPU."""
    nz, ny, nx = shape
    solid = torch.zeros(nz * ny * nx, dtype=torch.uint8, device="cuda")
    if phi >= 1.0:
        return solid.view(shape)
    count = max(1, int(round(-math.log(phi) * nx * ny * nz / (4.0 / 3.0 * math.pi * radius ** 3))))
    rnd = np.random.RandomState(seed % (1 << 31))
    centres = torch.from_numpy(rnd.random_sample((count, 3)) * np.array([nx, ny, nz])).cuda()
    r = int(math.ceil(radius)) + 1
    o = torch.arange(-r, r + 1, device="cuda")
    for part in centres.split(max(1, (1 << 26) // (2 * r + 1) ** 3)):
        base = part.floor().long()
        ax = [base[:, a, None] + o for a in range(3)]
        d = [(ax[a] - part[:, a, None]).square() for a in range(3)]
        near = d[2][:, :, None, None] + d[1][:, None, :, None] + d[0][:, None, None, :] <= radius * radius
        at = ((ax[2] % nz)[:, :, None, None] * ny + (ax[1] % ny)[:, None, :, None]) * nx + (ax[0] % nx)[:, None, None, :]
        solid[at[near]] = 1
    return solid.view(shape)


def _geometry(case, seed):
    shape = (case["nz"], case["ny"], case["nx"])
    solid = _spheres(shape, case["radius"], case["phi"], seed)
    if "z" in case["walls"]:
        solid[0], solid[-1] = 1, 1
    if "y" in case["walls"]:
        solid[:, 0], solid[:, -1] = 1, 1
    if "x" in case["walls"] and not case["faces"]:
        solid[:, :, 0], solid[:, :, -1] = 1, 1
    return solid


def _fields(solid, seed, plane):
    """A flow under way: a few long waves of density and velocity and some
    noise, zero on the solid nodes (float64, as set_fields takes them)."""
    rnd = np.random.RandomState((seed + 77) % (1 << 31))
    nz, ny, nx = solid.shape
    x, y, z = (torch.arange(n, device="cuda", dtype=torch.float64) * (2.0 * math.pi / n) for n in (nx, ny, nz))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    fluid = (solid == 0).double()
    out = []
    for amp in (0.01, 0.03, 0.03, 0.03):
        k, ph = rnd.randint(1, 4, 3), rnd.uniform(0, 2 * math.pi, 3)
        w = torch.sin(k[0] * x + ph[0])[None, None, :] + torch.sin(k[1] * y + ph[1])[None, :, None]
        w = w + (torch.sin(k[2] * z + ph[2])[:, None, None] if nz > 1 else 0.0)
        noise = torch.rand(solid.shape, generator=gen, device="cuda", dtype=torch.float64) - 0.5
        out.append(((w / 3.0 + 0.2 * noise) * amp * fluid).contiguous())
    if plane:
        out[3].zero_()
    return out


def _periodic(case):
    return tuple(0 if a in case["walls"] else 1 for a in "xyz")


def _pressure(case):
    return (0, 1.01, 0.99) if case["faces"] else None


def _force(case):
    return (0.0, 0.0, 0.0) if case["faces"] else (G if case["q"] != 9 else (G[0], G[1], 0.0))


def _mix(case, seed):
    """(mask, g) of the boxes of a batch: cubes, edges in multiples of 16."""
    rnd = np.random.RandomState((seed + 5) % (1 << 31))
    edges = list(range(case["min_edge"], case["max_edge"] + 1, 16))
    for b in range(case["boxes"]):
        e = edges[(b * 5 + 3) % len(edges)]
        phi, r = rnd.uniform(0.3, 0.95), rnd.uniform(3.0, 8.0)
        yield _spheres((e, e, e), r, phi, seed * 64 + b), (1e-5, 0.0, 0.0)


def prepare(case, seed):
    dt = STATE[case["storage"]]
    if case.get("batch"):
        b = Batch(case["q"], case["storage"], capacity=16, graph_steps=50)
        slots, outs = [], []
        for mask, g in _mix(case, seed):
            slots.append(b.admit(mask, (1, 1, 1), g))
            outs.append(torch.empty((4,) + tuple(mask.shape), dtype=torch.float64, device="cuda"))
        b.synchronize()
        return {"case": case, "batch": b, "slots": slots, "outs": outs, "dt": dt}
    solid = _geometry(case, seed)
    t = Tau1(case["q"], (case["nx"], case["ny"], case["nz"]), storage=case["storage"], periodic=_periodic(case),
             g=_force(case), layout=case["layout"])
    t.set_geometry(solid)
    t.set_fields(*_fields(solid, seed, case["q"] == 9))
    if case["faces"]:
        t.set_pressure(*_pressure(case))
    t.synchronize()
    outs = [torch.empty(tuple(solid.shape), dtype=torch.float64, device="cuda") for _ in range(4)]
    return {"case": case, "solver": t, "outs": outs, "dt": dt}


# ---- one pass ------------------------------------------------------------------------------

def run(state):
    case, dt = state["case"], state["dt"]
    if case.get("batch"):
        b = state["batch"]
        b.step(case["steps"])
        stats = b.stats(state["slots"])
        res = []
        for slot, out in zip(state["slots"], state["outs"]):
            p = [f.data_ptr() for f in out]
            b._check(lbm.lbm_tau1_batch_get_fields(b.b, slot, *p, 1))
            res.append(out.to(dt))
        return {"fields": res, "fluid": np.array([s["n_fluid"] for s in stats]),
                "permeability": np.array([s["permeability"] for s in stats], dtype=np.float32)}
    t = state["solver"]
    t.step(case["steps"])
    res = {}
    if case["check"]:
        s = t.reduce()
        res["fluid"] = s["n_fluid"]
        res["mean_u"] = np.array(s["mean_u_fluid"], dtype=np.float64 if case["storage"] == "f64" else np.float32)
    names = ("drho", "ux", "uy", "uz")[: 3 if case["q"] == 9 else 4]
    for name, f in zip(names, t.get_fields(state["outs"])):
        res[name] = f.to(dt)
    return res


# ---- what a pass cannot do without -----------------------------------------------------------

def _node_work(q, dims, storage):
    """Bytes and operations of one node's update: (rho, u) read and written
    once, and q equilibria formed and summed."""
    return 2 * (dims + 1) * BYTES[storage], 10 * q


def work(case):
    """Each step reads and writes the fluid nodes' state once; the fields are
    written once per pass. The share of fluid nodes is the medium's porosity."""
    if case.get("batch"):
        edges = list(range(case["min_edge"], case["max_edge"] + 1, 16))
        n = sum(edges[(b * 5 + 3) % len(edges)] ** 3 for b in range(case["boxes"]))
        fluid = 0.6 * n
        dims = 3
    else:
        n = case["nx"] * case["ny"] * case["nz"]
        fluid = case["phi"] * n
        dims = 2 if case["q"] == 9 else 3
    b, f = _node_work(case["q"], dims, case["storage"])
    return {"bytes": case["steps"] * fluid * b + n * (dims + 1) * BYTES[case["storage"]],
            "flops": case["steps"] * fluid * f}


# ---- the same pass in 64 bits, from the method's definition --------------------------------------

def _lattice(q):
    w = {0: 4.0 / 9.0, 1: 1.0 / 9.0, 2: 1.0 / 36.0}, {0: 1.0 / 3.0, 1: 1.0 / 18.0, 2: 1.0 / 36.0}, \
        {0: 8.0 / 27.0, 1: 2.0 / 27.0, 2: 1.0 / 54.0, 3: 1.0 / 216.0}
    w = w[{9: 0, 19: 1, 27: 2}[q]]
    r = (-1, 0, 1)
    return [((x, y, z), w[x * x + y * y + z * z]) for z in ((0,) if q == 9 else r) for y in r for x in r
            if x * x + y * y + z * z in w]


def _tau1(q, solid, fields, periodic, g, steps, pressure=None):
    """Tau1 from its definition: every node sums the equilibria of its
    neighbours; a wall link takes the node's own equilibrium in the opposite
    direction; constant-density faces after Zou and He."""
    lat = _lattice(q)
    shape = solid.shape
    # a wall: a solid node, or one beyond a non-periodic face
    pad = torch.ones([n + 2 for n in shape], dtype=torch.bool, device="cuda")
    pad[1:-1, 1:-1, 1:-1] = solid != 0

    def wrap(p):
        for dim, per in zip((2, 1, 0), periodic):
            if per:
                n = shape[dim]
                p.narrow(dim, 0, 1).copy_(p.narrow(dim, n, 1))
                p.narrow(dim, n + 1, 1).copy_(p.narrow(dim, 1, 1))
        return p

    def source(p, c):
        return p[1 - c[2]:1 - c[2] + shape[0], 1 - c[1]:1 - c[1] + shape[1], 1 - c[0]:1 - c[0] + shape[2]]

    wrap(pad)
    fluid = (solid == 0)
    wall = {c: source(pad, c) for c, _ in lat}
    padded = [torch.zeros([n + 2 for n in shape], dtype=torch.float64, device="cuda") for _ in range(4)]

    def feq(w, c, d, v, vv):
        cv = sum(ci * vi for ci, vi in zip(c, v) if ci) if any(c) else torch.zeros_like(d)
        return w * (d + (1.0 + d) * (3.0 * cv + 4.5 * cv * cv - 1.5 * vv))

    for _ in range(steps):
        d, v = fields[0], [f + gi for f, gi in zip(fields[1:], g)]
        own_vv = v[0] * v[0] + v[1] * v[1] + v[2] * v[2]
        for p, f in zip(padded, [d] + v):
            p[1:-1, 1:-1, 1:-1] = f
            wrap(p)
        tot = torch.zeros_like(d)
        mom = [torch.zeros_like(d) for _ in range(3)]
        if pressure:
            zh = [torch.zeros_like(d[:, :, 0]), torch.zeros_like(d[:, :, 0])]
        for c, w in lat:
            s = [source(p, c) for p in padded]
            f = feq(w, c, s[0], s[1:], s[1] * s[1] + s[2] * s[2] + s[3] * s[3])
            if any(c):
                f = torch.where(wall[c], feq(w, tuple(-i for i in c), d, v, own_vv), f)
            tot += f
            for a in range(3):
                if c[a]:
                    mom[a] += c[a] * f
            if pressure:
                for side, (sgn, at) in enumerate(((1, 0), (-1, -1))):
                    if c[0] != sgn:
                        zh[side] += (1.0 if c[0] == 0 else 2.0) * f[:, :, at]
        new = [tot] + [m / (1.0 + tot) for m in mom]
        if pressure:
            for side, (sgn, at, rho) in enumerate(((1, 0, pressure[1]), (-1, -1, pressure[2]))):
                new[0][:, :, at] = rho - 1.0
                new[1][:, :, at] = sgn * (rho - 1.0 - zh[side]) / rho
                new[2][:, :, at] = 0.0
                new[3][:, :, at] = 0.0
        fields = [torch.where(fluid, f, torch.zeros_like(f)) for f in new]
    return fields


def exact(case, seed):
    if case.get("batch"):
        res, count, perm = [], [], []
        for mask, g in _mix(case, seed):
            zero = [torch.zeros(mask.shape, dtype=torch.float64, device="cuda") for _ in range(4)]
            f = _tau1(case["q"], mask, zero, (1, 1, 1), g, case["steps"])
            res.append(torch.stack(f))
            nf = int((mask == 0).sum())
            count.append(nf)
            perm.append(float((f[1].sum() + 0.5 * g[0] * nf) / mask.numel() / 6.0 / g[0]))
        return {"fields": res, "fluid": np.array(count), "permeability": np.array(perm)}
    solid = _geometry(case, seed)
    g = _force(case)
    f = _tau1(case["q"], solid, _fields(solid, seed, case["q"] == 9), _periodic(case), g, case["steps"], _pressure(case))
    res = {}
    if case["check"]:
        nf = int((solid == 0).sum())
        res["fluid"] = nf
        res["mean_u"] = np.array([float(u.sum()) / nf + 0.5 * gi for u, gi in zip(f[1:], g)])
    names = ("drho", "ux", "uy", "uz")[: 3 if case["q"] == 9 else 4]
    res.update(zip(names, f))
    return res
