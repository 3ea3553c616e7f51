"""Measured workloads of the Gaussian-surface mesher: what a program that
meshes molecules asks of the public entry points, from a single ligand to a
million-atom assembly.

A case is a dict of plain values; `prepare` makes the inputs a caller has in
hand (seeded synthetic molecules and, where a caller keeps them, output
buffers), `run` is one call through the public API with its whole result.
"""
import math

import numpy as np
import torch

import paper_1611_03474_gb300 as gs
from paper_1611_03474_gb300.autograd import gaussian_surface, volume_area

ISO, MIN_EDGE, MAX_DEPTH, CUTOFF = 1.0, 0.25, 3, 1e-8
RADII = (1.2, 1.7, 1.55, 1.52, 1.8)
RADII_WEIGHTS = (0.5, 0.3, 0.08, 0.1, 0.02)
MODES = {"fp64": gs.GS_PREC_FP64, "mixed": gs.GS_PREC_MIXED}


def listed():
    return [
        # one small molecule (an open 100-atom chain) with the call's defaults:
        # arrays on the host in and out, FP64.  Launches and host waits count.
        dict(name="chain 100 host fp64", kind="host", shape="chain", atoms=100, units=1, D=0.5, precision=1e-3,
             mode="fp64"),
        # a peptide-sized fold in the mixed form into device buffers that a
        # loop over conformations keeps
        dict(name="peptide 523 mixed", kind="into", shape="fold", atoms=523, units=1, D=0.9, precision=1e-3,
             mode="mixed", buffers="device"),
        # a protein in the reference form (every sum in FP64)
        dict(name="protein 20000 fp64", kind="into", shape="fold", atoms=20000, units=1, D=0.5, precision=1e-3,
             mode="fp64", buffers="device"),
        # the same size in the mixed form, the everyday call
        dict(name="protein 20000 mixed", kind="into", shape="fold", atoms=20000, units=1, D=0.5, precision=1e-3,
             mode="mixed", buffers="device"),
        # a complex of several chains whose mesh goes to a host program:
        # page-locked inputs and output buffers kept across calls
        dict(name="complex 23317 pinned mixed", kind="into", shape="fold", atoms=3331, units=7, D=0.9, precision=1e-3,
             mode="mixed", buffers="pinned"),
        # a virus-shell assembly of a million atoms, the largest call
        dict(name="assembly 1000020 mixed", kind="into", shape="fold", atoms=16667, units=60, D=0.5, precision=1e-3,
             mode="mixed", buffers="device"),
        # a coarse precision: cubes accepted on several levels, joined through
        # constrained vertex values (the adaptive meshes of the method)
        dict(name="adaptive 50004 mixed", kind="into", shape="fold", atoms=4167, units=12, D=0.5, precision=5e-2,
             mode="mixed", buffers="device"),
        dict(name="adaptive 2500 fp64", kind="into", shape="fold", atoms=2500, units=1, D=0.9, precision=5e-2,
             mode="fp64", buffers="device"),
        # many molecules of uneven size in one call (a screening set), host
        # arrays in and out
        dict(name="batch 16 mixed", kind="batch", molecules=16, smallest=60, largest=4000, precision=1e-3,
             mode="mixed"),
        # shape optimisation: mesh, enclosed volume and area, and their
        # gradient with respect to centres, radii and D, on device tensors
        dict(name="gradient 10000 mixed", kind="gradient", shape="fold", atoms=10000, units=1, D=0.5, precision=1e-3,
             mode="mixed"),
        # the field and its gradient at scattered points (a projection or a
        # visualisation step), FP64
        dict(name="field 20000 x 400001 fp64", kind="field", shape="fold", atoms=20000, units=1, D=0.5,
             points=400001, mode="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    mode, D = rng.choice(("fp64", "mixed", "mixed")), rng.choice((0.5, 0.9))
    kind = rng.choice(("host", "into", "into", "into", "into", "batch", "gradient", "field"))
    precision = rng.choice((1e-3, 1e-3, 5e-2))
    if kind == "host":
        shape = rng.choice(("chain", "fold"))
        return dict(kind=kind, shape=shape, atoms=_log(rng, 20, 200 if shape == "chain" else 1500), units=1, D=D,
                    precision=precision, mode=mode)
    if kind == "batch":
        return dict(kind=kind, molecules=rng.randrange(2, 17), smallest=_log(rng, 30, 120),
                    largest=_log(rng, 300, 5000), precision=1e-3, mode=mode)
    if kind == "gradient":
        return dict(kind=kind, shape="fold", atoms=_log(rng, 100, 12000), units=1, D=D, precision=precision,
                    mode=mode)
    if kind == "field":
        return dict(kind=kind, shape="fold", atoms=_log(rng, 200, 20000), units=1, D=D,
                    points=_log(rng, 1000, 500000), mode="fp64")
    units = rng.choice((1, 1, rng.randrange(2, 61)))
    top = 20000 if mode == "mixed" else 12000 // units
    return dict(kind=kind, shape="fold", atoms=_log(rng, 60, max(200, min(top, 500000 // units))), units=units, D=D,
                precision=precision, mode=mode, buffers=rng.choice(("device", "device", "pinned")))


# ---------------------------------------------------------------- molecules

def _packing(n, gen, radius, min_sep):
    """n centres in a ball: every one 1.5 A from the one it is bonded to and
    at least min_sep from all others, grown at random places (a few starts
    spread over the ball, then bonds from centres already placed)."""
    dev = gen.device
    cell, slots = min_sep, 6
    m = int(math.ceil(2 * radius / cell)) + 3
    grid = torch.full((m * m * m, slots), -1, dtype=torch.int64, device=dev)
    fill = torch.zeros(m * m * m, dtype=torch.int64, device=dev)
    pts = torch.zeros((n, 3), dtype=torch.float64, device=dev)
    a = torch.arange(-1, 2, device=dev)
    near = (a[:, None, None] + m * (a[None, :, None] + m * a[None, None, :])).reshape(-1)
    have, starts = 0, max(1, n // 40)

    def cell_of(p):
        q = torch.floor((p + radius) / cell).to(torch.int64) + 1
        return q[:, 0] + m * (q[:, 1] + m * q[:, 2])

    while have < n:
        k = min(2 * starts, 2048) if have < starts else 4096
        step = torch.randn((k, 3), dtype=torch.float64, device=dev, generator=gen)
        step = step / step.norm(dim=1, keepdim=True)
        if have < starts:
            u = torch.rand((k, 1), dtype=torch.float64, device=dev, generator=gen)
            parent = torch.full((k,), -2, dtype=torch.int64, device=dev)
            p = step * radius * u ** (1.0 / 3.0)
        else:
            parent = torch.randint(0, have, (k,), device=dev, generator=gen)
            p = pts[parent] + 1.5 * step
        ok = (p * p).sum(1) <= radius * radius
        p, parent = p[ok], parent[ok]
        c = cell_of(p)
        other = grid[(c[:, None] + near[None, :])].reshape(len(p), -1)
        d2 = ((pts[other.clamp(min=0)] - p[:, None, :]) ** 2).sum(2)
        bad = (other >= 0) & (other != parent[:, None]) & (d2 < min_sep * min_sep)
        ok = ~bad.any(1)
        p, c = p[ok], c[ok]
        # among this round's centres the first of two that are too close stays
        d2 = ((p[:, None, :] - p[None, :, :]) ** 2).sum(2)
        first = torch.ones(d2.shape, dtype=torch.bool, device=dev).tril(-1)
        ok = ~((d2 < min_sep * min_sep) & first).any(1)
        p, c = p[ok], c[ok]
        rank = ((c[:, None] == c[None, :]) & first[:len(c), :len(c)]).sum(1)
        ok = fill[c] + rank < slots
        p, c, rank = p[ok], c[ok], rank[ok]
        p, c, rank = p[:n - have], c[:n - have], rank[:n - have]
        grid[c, fill[c] + rank] = torch.arange(have, have + len(p), device=dev)
        fill.index_add_(0, c, torch.ones_like(c))
        pts[have:have + len(p)] = p
        have += len(p)
    return pts


def _chain(n, rng):
    """An open chain: 1.5 A bonds, at least 2.5 A between atoms not bonded."""
    pts = np.zeros((n, 3))
    i = 1
    while i < n:
        v = rng.standard_normal(3)
        p = pts[i - 1] + 1.5 * v / np.linalg.norm(v)
        if i < 2 or ((pts[:i - 1] - p) ** 2).sum(1).min() >= 6.25:
            pts[i] = p
            i += 1
        elif rng.random() < 0.02:
            i = max(1, i - 8)   # a trapped end: step back
    return pts


def _rotations(n, rng):
    q, r = np.linalg.qr(rng.standard_normal((n, 3, 3)))
    q = q * np.sign(np.diagonal(r, axis1=1, axis2=2))[:, None, :]
    q[:, :, 0] *= np.linalg.det(q)[:, None]
    return q


def _molecule(shape, atoms, units, seed):
    """(centres [n, 3], radii [n]) as float64 numpy arrays: a chain, a ball
    of 0.1 atoms per cubic angstrom, or rotated copies of such a ball spread
    over a spherical shell (250 A for 60 copies of 16,667 atoms)."""
    rng = np.random.default_rng(seed)
    if shape == "chain":
        xyz = _chain(atoms, rng)
    else:
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        gen = torch.Generator(device=dev)
        gen.manual_seed(int(rng.integers(1 << 40)))
        radius = (3.0 * atoms / (4.0 * math.pi * 0.1)) ** (1.0 / 3.0)
        xyz = _packing(atoms, gen, radius, 1.8).cpu().numpy()
        xyz = xyz + rng.uniform(-20, 20, 3)
    r = rng.choice(RADII, size=len(xyz), p=RADII_WEIGHTS)
    if units > 1:
        xyz = xyz - xyz.mean(axis=0)
        rad = np.sqrt((xyz ** 2).sum(1).max())
        k = np.arange(units) + 0.5
        th, ph = np.arccos(1 - 2 * k / units), math.pi * (1 + math.sqrt(5.0)) * k
        at = np.stack([np.cos(ph) * np.sin(th), np.sin(ph) * np.sin(th), np.cos(th)], axis=1)
        gap = min(np.sqrt(((at[:, None] - at[None]) ** 2).sum(2) + 9 * np.eye(units)).min(), 2.0)
        shell = max(250.0 * rad / 34.1 * math.sqrt(units / 60.0), (2 * rad + 5.0) / gap)
        xyz = np.concatenate([xyz @ R.T + shell * t for R, t in zip(_rotations(units, rng), at)])
        r = np.tile(r, units)
    return np.ascontiguousarray(xyz), np.ascontiguousarray(r)


def _batch_sizes(case):
    rng = np.random.default_rng(case["molecules"] + case["largest"])
    n = np.exp(rng.uniform(math.log(case["smallest"]), math.log(case["largest"]), case["molecules"])).astype(int)
    n[0], n[-1] = case["smallest"], case["largest"]
    return n, rng.choice([0.5, 0.9], size=len(n))


# ---------------------------------------------------------------- one pass

def _room(atoms, units=1, shape="fold"):
    """vertices (and cubes) that any mesh of so many atoms fits into; it has
    about twice as many triangles"""
    if shape == "chain":
        return 4096 + 700 * atoms
    return 4096 + units * (40 * atoms + int(1200 * atoms ** (2.0 / 3.0)))


def _buffers(nv, **kw):
    return (torch.zeros((nv, 3), dtype=torch.float64, **kw), torch.zeros((2 * nv, 3), dtype=torch.int32, **kw),
            torch.zeros(nv, dtype=torch.int64, **kw), torch.zeros(nv, dtype=torch.int64, **kw))


def prepare(case, seed):
    kind, s = case["kind"], dict(case)
    if kind == "batch":
        ns, Ds = _batch_sizes(case)
        s["molecules"] = [_molecule("fold", int(n), 1, seed + 101 * i) + (float(D),)
                          for i, (n, D) in enumerate(zip(ns, Ds))]
        # the scene the caller collects the meshes in
        s["scene"] = [x.numpy() for x in _buffers(sum(_room(int(n)) for n in ns))]
        return s
    xyz, r = _molecule(case["shape"], case["atoms"], case["units"], seed)
    if kind == "host":
        s.update(xyz=xyz, r=r, scene=[x.numpy() for x in _buffers(_room(case["atoms"], 1, case["shape"]))])
        return s
    s.update(xyz=torch.from_numpy(xyz).cuda(), r=torch.from_numpy(r).cuda())
    if kind == "into":
        kw = dict(device="cuda") if case["buffers"] == "device" else dict(pin_memory=True)
        if case["buffers"] == "pinned":
            s.update(xyz=torch.from_numpy(xyz).pin_memory(), r=torch.from_numpy(r).pin_memory())
        s["out"] = _buffers(_room(case["atoms"], case["units"]), **kw)
    elif kind == "gradient":
        s["scene"] = _buffers(_room(case["atoms"]), device="cuda")[:2]
    elif kind == "field":
        rng = np.random.default_rng(seed + 5)
        at = xyz[rng.integers(0, len(r), case["points"])] + rng.normal(0, 2.5, (case["points"], 3))
        s.update(p=torch.from_numpy(at).cuda(), phi=torch.empty(case["points"], dtype=torch.float64, device="cuda"),
                 g=torch.empty((case["points"], 3), dtype=torch.float64, device="cuda"))
    return s


def _collect(scene, meshes):
    """The meshes one after the other in the caller's own arrays."""
    at, sizes = [0, 0, 0, 0], []
    for m in meshes:
        parts = (m.vertices, m.triangles, m.vertex_keys.view(np.int64), m.cube_keys.view(np.int64))
        for i, (whole, part) in enumerate(zip(scene, parts)):
            whole[at[i]:at[i] + len(part)] = part
            at[i] += len(part)
        sizes.append([len(part) for part in parts])
    return scene, np.array(sizes)


def run(s):
    mode = MODES[s["mode"]]
    if s["kind"] == "host":
        m = gs.mesh_gaussian_surface(s["xyz"], s["r"], s["D"], ISO, s["precision"], MAX_DEPTH, min_edge=MIN_EDGE,
                                     precision_mode=mode)
        return _collect(s["scene"], [m])
    if s["kind"] == "into":
        sizes = gs.mesh_gaussian_surface_into(s["xyz"], s["r"], s["D"], ISO, s["precision"], MAX_DEPTH, *s["out"],
                                              min_edge=MIN_EDGE, precision_mode=mode,
                                              stream=torch.cuda.current_stream())
        return s["out"], sizes
    if s["kind"] == "batch":
        ms = gs.mesh_gaussian_surface_batch(s["molecules"], ISO, s["precision"], MAX_DEPTH, min_edge=MIN_EDGE,
                                            precision_mode=mode)
        return _collect(s["scene"], ms)
    if s["kind"] == "gradient":
        x, r = s["xyz"].requires_grad_(), s["r"].requires_grad_()
        D = torch.tensor(s["D"], dtype=torch.float64, device=x.device, requires_grad=True)
        v, t = gaussian_surface(x, r, D, c=ISO, precision=s["precision"], max_depth=MAX_DEPTH, min_edge=MIN_EDGE,
                                precision_mode=mode)
        vol, area = volume_area(v, t)
        gx, gr, gD = torch.autograd.grad(vol + area, (x, r, D))
        s["scene"][0][:len(v)] = v.detach()
        s["scene"][1][:len(t)] = t
        return s["scene"], (len(v), len(t)), vol.detach(), area.detach(), gx, gr, gD
    gs.gs_eval_field(s["xyz"], s["r"], s["D"], ISO, s["p"], grad=True, precision_mode=mode,
                     stream=torch.cuda.current_stream(), out=(s["phi"], s["g"]))
    return s["phi"], s["g"]


def _mean_radius_cubed(D):
    return sum(w * (r * r - math.log(CUTOFF * ISO) / D) ** 1.5 for r, w in zip(RADII, RADII_WEIGHTS))


def work(case):
    """Bytes: centres and radii read, the results written.  Operations: per
    (cube, atom) term a rank-one update of 64 coefficients and its factors
    (144), per (point, atom) term a distance, an exponential and a sum (12,
    with the gradient 18).  Terms and mesh sizes per atom are those of
    molecules of 0.1 atoms per cubic angstrom: in a mesh about 43 vertices, 86
    triangles and 43 cubes per atom, 205 examined cubes with 42 terms each
    and 43 lattice vertices with 95 terms each at D = 0.5, the terms scaling
    with the cutoff spheres' volume (a tenth of the cubes at a coarse
    precision in FP64 terms stay: the same levels are examined)."""
    if case["kind"] == "field":
        terms = case["points"] * 0.1 * 4.19 * _mean_radius_cubed(case["D"])
        return {"bytes": 32.0 * case["atoms"] + 56.0 * case["points"], "flops": 18.0 * terms}
    if case["kind"] == "batch":
        lo, hi = case["smallest"], case["largest"]
        n, D = case["molecules"] * (hi - lo) / math.log(hi / lo), 0.7
    else:
        n, D = float(case["atoms"] * case["units"]), case["D"]
    rel = _mean_radius_cubed(D) / _mean_radius_cubed(0.5)
    flops = n * rel * (144.0 * 205 * 42 + 12.0 * 43 * 95)
    nbytes = n * (32 + 43 * 32 + 86 * 12 + 43 * 8.0)
    if case["kind"] == "gradient":
        nbytes = n * (32 + 43 * 24 + 86 * 24 + 43 * 24 + 32.0)
        flops += n * rel * 43 * 95 * 20.0
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """The field and its gradient summed in 64 bits over all atoms within
    their cutoff radii.  The meshes have no value apart from the method's own
    construction (which cubes are split, how pieces are cut and ordered), so
    their cases give none."""
    if case["kind"] != "field":
        return None
    s = prepare(case, seed)
    x, r, p, D = s["xyz"], s["r"], s["p"], case["D"]
    R2 = r * r - math.log(CUTOFF * ISO) / D
    phi, g = torch.empty_like(s["phi"]), torch.empty_like(s["g"])
    step = max(1, 30_000_000 // len(r))
    for i in range(0, len(p), step):
        d = p[i:i + step, None, :] - x[None, :, :]
        d2 = (d * d).sum(2)
        t = torch.where(d2 <= R2, torch.exp(-D * (d2 - r * r)), torch.zeros((), dtype=torch.float64, device=p.device))
        phi[i:i + step] = t.sum(1)
        g[i:i + step] = -2.0 * D * torch.einsum("ij,ijk->ik", t, d)
    return phi, g
