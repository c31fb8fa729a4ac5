"""Performance cases of the coupling path: what a solver has this library do, through the public
entry points of ``paper_2605_20565_gb300``, from a 1,000-marker verification run to the
many-bubble step with 50 million particles.

A case is a dict of plain values; ``listed()`` gives the standing ones and ``draw(rng)`` more of
the same ranges.  ``prepare`` makes what a program holds before the call (octree, tables, batch,
workspaces, points, forces, fields; drawn from the seed), ``run`` makes one pass, ``work``
states the bytes and operations a pass cannot do without, and ``exact`` restates the pass in
64 bits with plain torch (its own octree, search, stencils and sums).

Kinds of pass:
  step    one coupling step on a batch: every marker (Peskin-4) and particle (trilinear) located
          and interpolated by the batch's graph, the force field cleared and the marker forces
          spread (sorted).
  track   one tracking step in a periodic box: batch, AB2 advection with drag, spreading, removal
          of the mean force.
  query   single calls without tables: locate, then trilinear interpolation at the hosts found.
  ibm     single calls on the markers of one or more bodies: delta-kernel interpolation, direct
          forcing, spreading with marker volumes.
  mdf     multi-direct forcing rounds on a velocity field.
  learned host search with the trained index.
  readapt the work of a re-adaptation: Morton order of the particles, octree build, tables,
          field on the new leaves.
  body    per-body sums: internal-fluid momenta at the internal markers, force and torque at the
          surface markers.
"""
import math

import numpy as np
import torch

import paper_2605_20565_gb300 as ot

# Launch shape of the batches of a long run: what the autotuner picks for the workloads of
# bench.py with the tables built (128 threads, one 32-point row per marker item, eight per
# particle item, 32 resident warps per SM).  A program keeps such a shape from run to run.
TUNED = {"block": 128, "tile": 1, "tri_tile": 8, "tri_blocks_per_sm": 8}

# Meshes (levels, bubbles, diameters, shell width in diameters), the shapes of bench.py's
# workloads: a verification sphere, one bubble with a two-diameter shell, 64 bubbles of disparate
# size, and 256 bubbles with thin shells.
VERIFY = dict(lmin=3, lmax=5, bubbles=1, dmin=0.4, dmax=0.4, shell=0.25)
SINGLE = dict(lmin=5, lmax=9, bubbles=1, dmin=0.1, dmax=0.1, shell=2.0)
MANY = dict(lmin=4, lmax=10, bubbles=64, dmin=0.02, dmax=0.1, shell=0.25)
SWARM = dict(lmin=4, lmax=10, bubbles=256, dmin=0.01, dmax=0.08, shell=0.06)


def listed():
    return [
        # the verification mesh stepped as bench.py does: 11,000 points, where launches count
        dict(name="step_verify", kind="step", **VERIFY, markers=1_000, particles=10_000, clustered=False, tuned=False),
        # one rising bubble, half of the particles around it
        dict(name="step_single", kind="step", **SINGLE, markers=50_000, particles=10_000_000, clustered=True,
             tuned=True),
        # the headline workload: 64 bubbles and 50 million uniform particles
        dict(name="step_many", kind="step", **MANY, markers=2_000_000, particles=50_000_000, clustered=False,
             tuned=True),
        # a step of a tracking run in a periodic box, particles kept in Morton order, Re-dependent drag
        dict(name="track_periodic", kind="track", **SWARM, markers=1_000_000, particles=20_000_000, drag=20.0),
        # probes sampled from a solution once, FP32, no tables (an odd count)
        dict(name="query_single", kind="query", **SINGLE, points=5_000_011, fp64=False),
        # a verification in FP64 on the many-bubble mesh
        dict(name="query_many_fp64", kind="query", **MANY, points=300_007, fp64=True),
        # one body of a few thousand markers, forced by single calls (latency of a small solver)
        dict(name="ibm_small", kind="ibm", **VERIFY, markers=2_503, kernel="peskin4", fp64=False),
        # markers in the order their surface was meshed, the paper's 3-point kernel, FP64
        dict(name="ibm_roma_fp64", kind="ibm", **SINGLE, markers=90_001, kernel="roma3", fp64=True),
        # three rounds of multi-direct forcing on the markers of 64 bubbles
        dict(name="mdf_many", kind="mdf", **MANY, markers=1_000_000, rounds=3),
        # host search with the learned index, 30 % of the points at bubble surfaces
        dict(name="learned_many", kind="learned", **MANY, points=10_000_000),
        # a tracking run's re-adaptation
        dict(name="readapt_swarm", kind="readapt", **SWARM, particles=20_000_000),
        # internal momenta and surface forces of 64 bubbles
        dict(name="body_many", kind="body", **MANY, markers=2_000_000),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def markers(lo, hi):  # at most 12 to a finest cell's face of the bubbles' surfaces
        most = 12.0 * math.pi * 4.0 ** mesh["lmax"] * float(np.sum(_diameters(mesh) ** 2))
        return size(min(lo, 0.2 * most), min(hi, most))

    kind = rng.choice(["step", "track", "query", "ibm", "mdf", "learned", "readapt", "body"])
    mesh = dict(rng.choice([VERIFY, SINGLE, MANY, SWARM] if kind in ("step", "query", "ibm") else
                           [SINGLE, MANY, SWARM]))
    if mesh["bubbles"] > 1:
        mesh["bubbles"] = size(8, mesh["bubbles"])
        mesh["lmax"] = rng.choice([9, 10])
    mesh["shell"] = round(mesh["shell"] * rng.uniform(0.8, 1.0), 4)
    c = dict(kind=kind, **mesh)
    if kind == "step":
        c.update(markers=markers(500, 2_000_000), particles=size(5_000, 50_000_000), clustered=rng.random() < 0.3,
                 tuned=rng.random() < 0.6)
    elif kind == "track":
        c.update(markers=markers(20_000, 1_000_000), particles=size(100_000, 20_000_000), drag=rng.choice([0.0, 20.0]))
    elif kind == "query":
        c.update(points=size(1_000, 5_000_000), fp64=rng.random() < 0.3)
    elif kind == "ibm":
        c.update(markers=markers(300, 1_000_000), kernel=rng.choice(["peskin4", "peskin4", "roma3"]),
                 fp64=rng.random() < 0.3)
    elif kind == "mdf":
        c.update(markers=markers(5_000, 1_000_000), rounds=rng.choice([1, 2, 3, 5]))
    elif kind == "learned":
        c.update(points=size(100_000, 10_000_000))
    elif kind == "readapt":
        c.update(particles=size(100_000, 20_000_000))
    else:
        c.update(markers=markers(20_000, 2_000_000))
    return c


# --- inputs -------------------------------------------------------------------------------------

def _gen(seed, what):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 64 + what)


def _uniform(seed, what, n):
    return torch.rand((3, n), generator=_gen(seed, what), dtype=torch.float64, device="cuda")


def _normal(seed, what, n, dtype=torch.float64):
    return torch.randn((3, n), generator=_gen(seed, what), dtype=dtype, device="cuda")


def _diameters(case):
    return np.exp(np.linspace(math.log(case["dmax"]), math.log(case["dmin"]), case["bubbles"]))


def bubbles(case):
    """The case's geometry (the mesh is part of the case; the seed draws what lives on it): centres
    (B, 3), diameters (B,) and the octree's spheres (B, 5).  Non-overlapping bubbles, diameters
    spread evenly over [dmin, dmax] in the logarithm, their shells inside the cube and centres a
    diameter or more from the walls; shells at least four finest cells wide."""
    rng = np.random.default_rng(case["bubbles"])
    h = 2.0 ** -case["lmax"]
    d = _diameters(case)
    c = np.empty((0, 3))
    for k in range(d.size):
        m = min(max(d[k], (0.5 + case["shell"]) * d[k]) + 4.0 * h, 0.45)
        while True:
            p = m + (1.0 - 2.0 * m) * rng.random(3)
            if np.all(np.linalg.norm(c - p, axis=1) >= 0.5 * (d[:k] + d[k])):
                break
        c = np.vstack([c, p])
    return c, d, np.column_stack([c, 0.5 * d, np.maximum(case["shell"] * d, 4.0 * h)])


def _split(total, d):
    q = total * d ** 2 / np.sum(d ** 2)
    n = np.floor(q).astype(np.int64)
    n[np.argsort(n - q, kind="stable")[:total - int(n.sum())]] += 1
    return n


def _markers(case, seed, c, d, ordered):
    """Markers (3, n) on the bubbles, counts in proportion to d^2, outward normals (3, n), body
    offsets (B + 1,): a randomly turned Fibonacci lattice on each, in the lattice's order or, with
    ordered, in Morton order of the finest cells (a long run stores its markers so)."""
    n = _split(case["markers"], d)
    rng = np.random.default_rng([int(seed), 2])
    pos, nrm = [], []
    for b in range(d.size):
        i = torch.arange(int(n[b]), dtype=torch.float64, device="cuda")
        z = 1.0 - (2.0 * i + 1.0) / max(int(n[b]), 1)
        rho = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
        lon = i * (math.pi * (3.0 - math.sqrt(5.0)))
        turn = torch.as_tensor(np.linalg.qr(rng.normal(size=(3, 3)))[0], device="cuda")
        v = turn @ torch.stack([rho * torch.cos(lon), rho * torch.sin(lon), z])
        p = torch.as_tensor(c[b], device="cuda")[:, None] + 0.5 * d[b] * v
        if ordered:
            o = torch.argsort(_morton(_cells(p, case["lmax"])), stable=True)
            p, v = p[:, o], v[:, o]
        pos.append(p)
        nrm.append(v)
    start = np.concatenate([[0], np.cumsum(n)])
    return torch.cat(pos, 1).contiguous(), torch.cat(nrm, 1).contiguous(), start


def _particles(case, seed, n, c, d):
    """Uniform points; clustered: half of them around the first bubble; near: 30 % at surfaces."""
    p = _uniform(seed, 3, n)
    if case.get("clustered"):
        m = n // 2
        g = torch.as_tensor(c[0], device="cuda")[:, None] + 0.5 * d[0] * _normal(seed, 4, m)
        inside = ((g >= 0.0) & (g < 1.0)).all(0)
        p[:, n - m:] = torch.where(inside, g, p[:, n - m:])
    if case["kind"] == "learned":
        m = int(0.3 * n)
        rng = np.random.default_rng([int(seed), 3])
        pick = torch.as_tensor(rng.choice(d.size, m, p=d ** 2 / np.sum(d ** 2)), device="cuda")
        g = _normal(seed, 4, m)
        r = 0.5 * torch.as_tensor(d, device="cuda")[pick] * (1.0 + 0.1 * _normal(seed, 5, m)[0])
        g = torch.as_tensor(c, device="cuda")[pick].T + g / torch.linalg.norm(g, dim=0) * r
        p[:, n - m:] = torch.clamp(g, 0.0, 1.0 - 2.0 ** -53)
    return p


def _internal(c, d, h):
    """Points inside each body on a cubic lattice of spacing h: positions (3, n), offsets (B + 1,)."""
    pts, start = [], [0]
    for b in range(d.size):
        m = int(0.5 * d[b] / h)
        g = torch.arange(-m, m + 1, dtype=torch.float64, device="cuda") * h
        off = torch.stack(torch.meshgrid(g, g, g, indexing="ij")).reshape(3, -1)
        off = off[:, (off ** 2).sum(0) < (0.5 * d[b] - 0.5 * h) ** 2]
        pts.append(torch.as_tensor(c[b], device="cuda")[:, None] + off)
        start.append(start[-1] + off.shape[1])
    return torch.cat(pts, 1).contiguous(), start


def _modes(seed, count):
    """Solenoidal Fourier modes: integer wave vectors up to 8, amplitudes |n|^(-5/3), phases."""
    rng = np.random.default_rng([int(seed), 4])
    n = rng.integers(-8, 9, size=(count, 3))
    n[(n == 0).all(1)] = 1
    r = np.linalg.norm(n, axis=1, keepdims=True)
    a = rng.normal(size=(count, 3))
    a -= (a * n).sum(1, keepdims=True) / r ** 2 * n
    return n, a / np.linalg.norm(a, axis=1, keepdims=True) * r ** (-5.0 / 3.0), 2.0 * math.pi * rng.random(count)


def _field(keys, levels, seed, fp64=False):
    """(N, 4) velocity at the leaf centres: eight Fourier modes."""
    n, a, ph = _modes(seed, 8)
    out = torch.zeros((keys.numel(), 4), dtype=torch.float64 if fp64 else torch.float32, device="cuda")
    for s in range(0, keys.numel(), 1 << 24):
        at = slice(s, s + (1 << 24))
        x = _demorton(keys[at]).double() + 0.5 * torch.pow(2.0, 21.0 - levels[at].double())
        for k in range(n.shape[0]):
            turns = (n[k, 0] * x[0] + n[k, 1] * x[1] + n[k, 2] * x[2]) * 2.0 ** -21  # exact
            turns = (turns - torch.floor(turns)).to(out.dtype)
            w = torch.cos(turns * (2.0 * math.pi) + ph[k])
            for j in range(3):
                out[at, j] += a[k, j] * w
    return out


def _inputs(case, seed):
    """Everything drawn from the seed, the same for the library's pass and the restatement."""
    c, d, spheres = bubbles(case)
    g = dict(spheres=spheres)
    kind, h = case["kind"], 2.0 ** -case["lmax"]
    if "markers" in case:
        g["m"], g["normal"], g["start"] = _markers(case, seed, c, d, kind not in ("ibm", "body"))
        nm = case["markers"]
        g["F"] = (g["normal"] + 0.2 * _normal(seed, 6, nm)).to(torch.float32)
        if kind in ("ibm", "mdf", "body"):
            area = torch.as_tensor(np.repeat(math.pi * d ** 2 / np.maximum(_split(nm, d), 1), _split(nm, d)),
                                   device="cuda")
            g["dV"] = area * h
            g["U"] = (0.1 * _normal(seed, 7, nm)).to(torch.float32)
    if "particles" in case or "points" in case:
        n = case.get("particles", case.get("points"))
        g["p"] = _particles(case, seed, n, c, d)
        if kind == "track":
            o = torch.argsort(_morton(_cells(g["p"], 8)), stable=True)
            g["p"] = g["p"][:, o].contiguous()
            g["v"], g["ap"], g["vp"] = (s * _normal(seed, 8 + k, n, torch.float32)
                                        for k, s in enumerate((0.3, 0.3, 0.3)))
    if kind == "body":
        g["q"], g["qstart"] = _internal(c, d, h)
        g["xb"] = torch.as_tensor(c, device="cuda")
        g["uq"] = 0.5 * _normal(seed, 9, g["q"].shape[1], torch.float32)
    return g


DT, TAU, RHO = 5e-4, 5e-3, 1.0  # a step of half a finest cell at unit speed; particle response time


def _kernel(case):
    return ot.OT_ROMA3 if case.get("kernel") == "roma3" else ot.OT_PESKIN4


def prepare(case, seed):
    g = _inputs(case, seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "body":  # the sums need no octree
        for k in ("m", "F", "q", "uq", "xb"):
            s[k] = g[k]
        s["dV"] = g["dV"].to(torch.float32)
        s["start"], s["qstart"] = (torch.as_tensor(g[k], dtype=torch.int64, device="cuda") for k in ("start", "qstart"))
        return s
    tree = s["tree"] = ot.ot_octree_build(g["spheres"], case["lmin"], case["lmax"])
    n_leaves = ot.ot_octree_info(tree)[0]
    if kind == "readapt":  # the buffer that the run's tables live in, sized on the first octree
        s["spheres"], s["p"], s["modes"] = g["spheres"], g["p"], _modes(seed, 32)
        need = ot.ot_octree_mates_bytes(tree)
        s["buffer"] = torch.empty(need + need // 10, dtype=torch.uint8, device="cuda")
        return s
    if kind == "learned":
        s["p"] = g["p"]
        ot.ot_index_train(tree, root=ot.OT_ROOT_MLP, n_leaf_models=1 << 18, n_mid_models=4096, epochs=1, steps=64)
        s["host"] = torch.empty(g["p"].shape[1], dtype=torch.int32, device="cuda")
        return s
    fp64 = bool(case.get("fp64"))
    if kind == "track":
        ot.ot_octree_set_periodic(tree, True)
    field = s["field"] = _field(*ot.ot_octree_copy_leaves(tree), seed, fp64)
    dtype = field.dtype
    if kind == "query":
        n = case["points"]
        s["p"] = g["p"]
        s["host"] = torch.empty(n, dtype=torch.int32, device="cuda")
        s["u"] = torch.empty((3, n), dtype=dtype, device="cuda")
        s["ws"] = torch.empty(ot.ot_interpolate_workspace_size(tree, ot.OT_TRILINEAR, fp64), dtype=torch.uint8,
                              device="cuda")
        return s
    m, nm = g["m"], case["markers"]
    s["m"] = m
    s["um"] = torch.empty((3, nm), dtype=dtype, device="cuda")
    if kind in ("ibm", "mdf"):
        s["U"], s["dV"] = g["U"], g["dV"].to(dtype)
        if kind == "mdf":
            s["u"] = torch.empty_like(field)
            return s
    s["F"] = g["F"].to(dtype)
    s["f"] = torch.zeros_like(field)
    s["ws"] = torch.empty(ot.ot_spread_workspace_size(tree, _kernel(case), nm), dtype=torch.uint8, device="cuda")
    if kind == "ibm":
        return s
    ot.ot_octree_build_mates(tree)
    p, n = g["p"], case["particles"]
    s["p"] = p
    s["up"] = torch.empty((3, n), dtype=torch.float32, device="cuda")
    groups = [dict(kernel=ot.OT_PESKIN4, x=m[0], y=m[1], z=m[2], u=s["um"]),
              dict(kernel=ot.OT_TRILINEAR, x=p[0], y=p[1], z=p[2], u=s["up"])]
    if kind == "step":
        s["hm"], s["hp"] = (torch.empty(k, dtype=torch.int32, device="cuda") for k in (nm, n))
        groups[0]["host"], groups[1]["host"] = s["hm"], s["hp"]
    else:
        s["v"], s["ap"], s["vp"] = g["v"], g["ap"], g["vp"]
        s["mean"] = torch.empty(3, dtype=torch.float64, device="cuda")
        s["ws_mean"] = torch.empty(ot.ot_field_mean_workspace_size(tree), dtype=torch.uint8, device="cuda")
    s["batch"] = ot.ot_batch_create(tree, groups, field, launch=TUNED if case.get("tuned", True) else None)
    return s


def run(s):
    case = s["case"]
    kind, tree = case["kind"], s.get("tree")
    if kind == "body":
        p, ang_p = ot.ot_body_sums(s["q"][0], s["q"][1], s["q"][2], s["uq"], s["qstart"], s["xb"], RHO,
                                   w=2.0 ** (-3 * case["lmax"]))
        f, ang_f = ot.ot_body_sums(s["m"][0], s["m"][1], s["m"][2], s["F"], s["start"], s["xb"], -1.0, dV=s["dV"])
        return p, ang_p, f, ang_f
    if kind == "readapt":
        perm = ot.ot_points_morton_order(s["p"][0], s["p"][1], s["p"][2])
        s["tree"] = tree = ot.ot_octree_build(s["spheres"], case["lmin"], case["lmax"])
        ot.ot_octree_build_mates_in(tree, s["buffer"])
        field = ot.ot_field_fourier(tree, *s["modes"])
        keys, levels = ot.ot_octree_copy_leaves(tree)
        return perm, keys, levels, field
    if kind == "learned":
        return ot.ot_locate(tree, s["p"][0], s["p"][1], s["p"][2], search=ot.OT_LEARNED, host=s["host"])
    if kind == "query":
        x, y, z = s["p"][0], s["p"][1], s["p"][2]
        ot.ot_locate(tree, x, y, z, host=s["host"])
        interpolate = ot.ot_interpolate_f64 if case["fp64"] else ot.ot_interpolate
        interpolate(tree, ot.OT_TRILINEAR, x, y, z, s["field"], host_in=s["host"], u=s["u"], workspace=s["ws"])
        return s["host"], s["u"]
    x, y, z = s["m"][0], s["m"][1], s["m"][2]
    if kind == "mdf":
        s["u"].copy_(s["field"])  # the solver's new velocity
        f, slip = ot.ot_ibm_mdf(tree, ot.OT_PESKIN4, x, y, z, s["U"], s["u"], RHO, DT, case["rounds"], dV=s["dV"],
                                slip=True)
        return s["u"], f, slip
    if kind == "ibm":
        k = _kernel(case)
        if case["fp64"]:
            ot.ot_interpolate_f64(tree, k, x, y, z, s["field"], u=s["um"])
        else:
            ot.ot_interpolate(tree, k, x, y, z, s["field"], u=s["um"])
            ot.ot_marker_force(s["um"], DT, F=s["F"], U=s["U"])
        s["f"].zero_()
        spread = ot.ot_spread_f64 if case["fp64"] else ot.ot_spread
        spread(tree, k, ot.OT_SORTED, x, y, z, s["F"], s["f"], dV=s["dV"], workspace=s["ws"])
        return s["um"], s["F"], s["f"]
    ot.ot_batch_run(s["batch"])
    if kind == "track":
        ot.ot_advect_ab2(s["p"], s["v"], s["ap"], s["vp"], s["up"], TAU, case["drag"], DT, first=False, periodic=True)
    s["f"].zero_()
    ot.ot_spread(tree, ot.OT_PESKIN4, ot.OT_SORTED, x, y, z, s["F"], s["f"], workspace=s["ws"])
    if kind == "step":
        return s["um"], s["hm"], s["up"], s["hp"], s["f"]
    ot.ot_field_subtract_mean(tree, s["f"], mean=s["mean"], workspace=s["ws_mean"])
    return s["um"], s["up"], s["p"], s["v"], s["ap"], s["vp"], s["f"]


# --- the least work -----------------------------------------------------------------------------

def _leaf_count(case):
    """About the octree's leaves: the finest cells of the shells and the coarser ones around them."""
    h = 2.0 ** -case["lmax"]
    n = 8.0 ** case["lmin"]
    for d in _diameters(case):
        r, w = 0.5 * float(d), max(case["shell"] * float(d), 4.0 * h) + h
        n += min(1.0, 4.0 / 3.0 * math.pi * ((r + w) ** 3 - max(r - w, 0.0) ** 3)) / h ** 3
    return min(n, 8.0 ** case["lmax"])


def work(case):
    """Each input read once, each output written once: positions, forces, volumes, velocities and
    hosts of the points; the field values of the leaves that the points reach; the force field."""
    kind, n = case["kind"], _leaf_count(case)
    e = 8 if case.get("fp64") else 4
    m, p = case.get("markers", 0), case.get("particles", case.get("points", 0))
    cells = min(n, 64.0 * m)                     # leaves that the stencils reach, at most
    reach = min(n, 8.0 * p + 64.0 * m)            # leaves whose values are read, at most
    spread, tri = 64 * 8, 8 * 7 + 12              # operations of a marker's stencil, of a particle
    if kind == "step":
        return dict(bytes=m * (24 + 12 + 12 + 4) + p * (24 + 12 + 4) + 16 * reach + 16 * n,
                    flops=2 * m * spread + p * tri)
    if kind == "track":
        return dict(bytes=m * (24 + 12 + 12) + p * (24 + 12 + 72 + 60) + 16 * reach + 16 * n,
                    flops=2 * m * spread + p * (tri + 60))
    if kind == "query":
        return dict(bytes=p * (24 + 4 + 3 * e) + 4 * e * reach, flops=p * tri)
    if kind == "ibm":
        return dict(bytes=m * (24 + 3 * e + 3 * e + e) + 4 * e * cells + 4 * e * n, flops=2 * m * spread)
    if kind == "mdf":
        return dict(bytes=m * (24 + 12 + 4) + 16 * n * 3, flops=(2 * case["rounds"] + 1) * m * spread)
    if kind == "learned":
        return dict(bytes=p * 28 + 8 * min(n, p), flops=p * 64)
    if kind == "readapt":  # the points, the leaves, their level-mate rows and the field
        return dict(bytes=p * 28 + n * (9 + 9 + 256 + 16 + 16), flops=n * 32 * 10)
    inside = math.pi / 6 * float(np.sum(_diameters(case) ** 3)) * 8.0 ** case["lmax"]  # internal markers
    return dict(bytes=inside * 36 + m * 40, flops=(inside + m) * 15)


# --- the same pass in 64 bits ---------------------------------------------------------------------

def _part(v):
    for shift, mask in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                        (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        v = (v | (v << shift)) & mask
    return v


def _compact(v):
    v = v & 0x1249249249249249
    for shift, mask in ((2, 0x10C30C30C30C30C3), (4, 0x100F00F00F00F00F), (8, 0x1F0000FF0000FF),
                        (16, 0x1F00000000FFFF), (32, 0x1FFFFF)):
        v = (v ^ (v >> shift)) & mask
    return v


def _morton(c):
    return _part(c[0]) | (_part(c[1]) << 1) | (_part(c[2]) << 2)


def _demorton(k):
    return torch.stack([_compact(k), _compact(k >> 1), _compact(k >> 2)])


def _cells(x, level):
    return torch.floor(x * 2.0 ** level).to(torch.int64)


def _children(cells):
    return (cells[:, None] * 8 + torch.arange(8, device="cuda")).reshape(-1)


def _near(cells, l, spheres):
    """Cells of level l whose box lies within a shell of its sphere's surface."""
    h = 2.0 ** -l
    hit = torch.zeros(cells.numel(), dtype=torch.bool, device="cuda")
    for s in range(0, cells.numel(), 1 << 23):
        lo = _demorton(cells[s:s + (1 << 23)]).double() * h
        for c0, c1, c2, r, w in spheres.tolist():
            near = torch.zeros_like(lo[0])
            far = torch.zeros_like(lo[0])
            for d, c in enumerate((c0, c1, c2)):
                hi = lo[d] + h
                e = torch.clamp(torch.maximum(lo[d] - c, c - hi), min=0.0)
                near = near + e * e
                e = torch.maximum(torch.abs(c - lo[d]), torch.abs(c - hi))
                far = far + e * e
            hit[s:s + (1 << 23)] |= torch.maximum(torch.sqrt(near) - r, r - torch.sqrt(far)) <= w
    return hit


class _Tree:
    """The octree, its searches and its cell means in plain torch."""

    def __init__(self, case, spheres, periodic=False):
        lmin, lmax = case["lmin"], case["lmax"]
        self.lmin, self.lmax, self.periodic = lmin, lmax, periodic
        self.refined = {}
        cells = torch.arange(8 ** lmin, device="cuda")
        for l in range(lmin, lmax):
            self.refined[l] = cells[_near(cells, l, spheres)]
            cells = _children(self.refined[l])
        for l in range(lmax - 1, lmin, -1):  # the parents of a refined cell's neighbours are refined
            c = _demorton(self.refined[l])
            side = [[torch.clamp(c[d] + o, 0, 2 ** l - 1) >> 1 for o in (-1, 1)] for d in range(3)]
            need = [self.refined[l - 1]] + [torch.unique(_morton((side[0][i], side[1][j], side[2][k])))
                                            for i in (0, 1) for j in (0, 1) for k in (0, 1)]
            self.refined[l - 1] = torch.unique(torch.cat(need))
        keys, levels = [], []
        for l in range(lmin, lmax + 1):
            cells = torch.arange(8 ** lmin, device="cuda") if l == lmin else _children(self.refined[l - 1])
            if l < lmax:
                cells = cells[~self._in(self.refined[l], cells)]
            keys.append(cells << (3 * (21 - l)))
            levels.append(torch.full_like(cells, l, dtype=torch.uint8))
        keys, levels = torch.cat(keys), torch.cat(levels)
        order = torch.argsort(keys)
        self.keys, self.levels = keys[order], levels[order]

    @staticmethod
    def _in(sorted_cells, cells):
        if sorted_cells.numel() == 0:
            return torch.zeros_like(cells, dtype=torch.bool)
        at = torch.searchsorted(sorted_cells, cells).clamp(max=sorted_cells.numel() - 1)
        return sorted_cells[at] == cells

    def locate(self, keys):
        return torch.searchsorted(self.keys, keys, right=True) - 1

    def means(self, field):
        """Mean of the field over every refined cell, level by level."""
        out = {}
        for l in range(self.lmax - 1, self.lmin - 1, -1):
            if self.refined[l].numel() == 0:
                continue
            ch = _children(self.refined[l])
            v = field[self.locate(ch << (3 * (20 - l)))]
            if l + 1 in out:
                deep = self._in(self.refined[l + 1], ch)
                v[deep] = out[l + 1][torch.searchsorted(self.refined[l + 1], ch[deep])]
            out[l] = v.reshape(-1, 8, 3).mean(1)
        return out

    def trilinear(self, x, field):
        """Host leaves (n,) and velocities (3, n)."""
        host, u = torch.empty(x.shape[1], dtype=torch.int64, device="cuda"), torch.empty_like(x)
        means = self.means(field)
        for s in range(0, x.shape[1], 1 << 22):
            at = torch.arange(s, min(s + (1 << 22), x.shape[1]), device="cuda")
            host[at] = self.locate(_morton(_cells(x[:, at], 21)))
            lev = self.levels[host[at]]
            for l in range(self.lmin, self.lmax + 1):
                i = at[lev == l]
                if i.numel() == 0:
                    continue
                c = _cells(x[:, i], l)
                t = x[:, i] * 2.0 ** l - c - 0.5
                nb = c + torch.where(t >= 0, 1, -1)
                if self.periodic:
                    nb = nb & (2 ** l - 1)
                else:
                    nb = torch.where((nb < 0) | (nb >= 2 ** l), c, nb)
                t = torch.abs(t)
                acc = torch.zeros((3, i.numel()), dtype=torch.float64, device="cuda")
                for k in range(8):
                    b = [(k >> d) & 1 for d in range(3)]
                    w = torch.ones_like(t[0])
                    for d in range(3):
                        w = w * (t[d] if b[d] else 1.0 - t[d])
                    cell = _morton([nb[d] if b[d] else c[d] for d in range(3)])
                    leaf = self.locate(cell << (3 * (21 - l)))
                    v = field[leaf]
                    deep = self.levels[leaf] > l
                    if bool(deep.any()):
                        v[deep] = means[l][torch.searchsorted(self.refined[l], cell[deep])]
                    acc += w * v.T
                u[:, i] = acc
        return host, u

    def stencils(self, x, kernel):
        """Chunks (marker slice, leaves, weights): the delta kernel's stencil cells."""
        width = 4 if kernel == ot.OT_PESKIN4 else 3
        for s in range(0, x.shape[1], 1 << 18):
            at = slice(s, min(s + (1 << 18), x.shape[1]))
            c = _cells(x[:, at], self.lmax)
            t = x[:, at] * 2.0 ** self.lmax - c - 0.5
            first = c - 2 + (t >= 0).to(torch.int64) if width == 4 else c - 1
            w = []
            for a in range(width):
                r = torch.abs(t + (c - first - a))
                if width == 4:
                    near = (3 - 2 * r + torch.sqrt(torch.clamp(1 + 4 * r - 4 * r * r, min=0.0))) / 8
                    far = (5 - 2 * r - torch.sqrt(torch.clamp(-7 + 12 * r - 4 * r * r, min=0.0))) / 8
                    w.append(torch.where(r <= 1, near, torch.where(r <= 2, far, torch.zeros_like(r))))
                else:
                    near = (1 + torch.sqrt(torch.clamp(1 - 3 * r * r, min=0.0))) / 3
                    far = (5 - 3 * r - torch.sqrt(torch.clamp(1 - 3 * (1 - r) ** 2, min=0.0))) / 6
                    w.append(torch.where(r <= 0.5, near, torch.where(r <= 1.5, far, torch.zeros_like(r))))
            leaves, weights = [], []
            for k in range(width ** 3):
                a = (k % width, k // width % width, k // width ** 2)
                cell = torch.stack([first[d] + a[d] for d in range(3)])
                if self.periodic:
                    cell = cell & (2 ** self.lmax - 1)
                inside = ((cell >= 0) & (cell < 2 ** self.lmax)).all(0)
                key = _morton(cell.clamp(min=0, max=2 ** self.lmax - 1)) << (3 * (21 - self.lmax))
                leaf = self.locate(key)
                ok = inside & (self.keys[leaf] == key) & (self.levels[leaf] == self.lmax)
                leaves.append(leaf)
                weights.append(torch.where(ok, w[a[0]][0] * w[a[1]][1] * w[a[2]][2], torch.zeros_like(w[0][0])))
            yield at, torch.stack(leaves), torch.stack(weights)

    def interpolate(self, x, field, kernel):
        u = torch.empty_like(x)
        for at, leaf, w in self.stencils(x, kernel):
            for d in range(3):
                u[d, at] = (w * field[:, d][leaf]).sum(0)
        return u

    def spread(self, x, F, kernel, dV=None):
        f = torch.zeros((self.keys.numel(), 4), dtype=torch.float64, device="cuda")
        for at, leaf, w in self.stencils(x, kernel):
            if dV is not None:
                w = w * dV[at] * 8.0 ** self.lmax
            for d in range(3):
                f[:, d].index_add_(0, leaf.reshape(-1), (w * F[d, at]).reshape(-1))
        return f


def exact(case, seed):
    g = _inputs(case, seed)
    kind = case["kind"]
    if kind == "learned":
        return None  # host indices only
    if kind == "body":
        def sums(x, v, w, start, scale):
            body = torch.repeat_interleave(torch.arange(len(start) - 1, device="cuda"),
                                           torch.as_tensor(np.diff(start), device="cuda"))
            v, r = v.double() * w, x - g["xb"][body].T
            out = []
            for a in (v, torch.linalg.cross(r, v, dim=0)):
                out.append(scale * torch.zeros((len(start) - 1, 3), dtype=torch.float64,
                                               device="cuda").index_add_(0, body, a.T))
            return out
        return (*sums(g["q"], g["uq"], 2.0 ** (-3 * case["lmax"]), g["qstart"], RHO),
                *sums(g["m"], g["F"], g["dV"].float().double(), g["start"], -1.0))
    tree = _Tree(case, g["spheres"], kind == "track")
    if kind == "readapt":
        n, a, ph = _modes(seed, 32)
        out = torch.zeros((tree.keys.numel(), 4), dtype=torch.float64, device="cuda")
        x = (_demorton(tree.keys).double() + 0.5 * torch.pow(2.0, 21.0 - tree.levels.double())) * 2.0 ** -21
        for k in range(32):
            turns = n[k, 0] * x[0] + n[k, 1] * x[1] + n[k, 2] * x[2]
            w = torch.cos((turns - torch.floor(turns)) * (2.0 * math.pi) + ph[k])
            for j in range(3):
                out[:, j] += a[k, j] * w
        return None, None, None, out
    field = _field(tree.keys, tree.levels, seed, bool(case.get("fp64"))).double()[:, :3].contiguous()
    if kind == "query":
        return None, tree.trilinear(g["p"], field)[1]
    kernel = _kernel(case)
    if kind == "mdf":
        u, f = field, torch.zeros_like(field)
        U, dV, slip = g["U"].double(), g["dV"].float().double(), []
        for it in range(case["rounds"] + 1):
            e = U - tree.interpolate(g["m"], u, kernel)
            slip.append(torch.sqrt((e ** 2).sum()))
            if it < case["rounds"]:
                F = tree.spread(g["m"], e / DT, kernel, dV)[:, :3]
                u, f = u + DT / RHO * F, f + F
        pad = torch.zeros((field.shape[0], 1), dtype=torch.float64, device="cuda")
        return torch.cat([u, pad], 1), torch.cat([f, pad], 1), torch.stack(slip)
    um = tree.interpolate(g["m"], field, kernel)
    if kind == "ibm":
        F, dV = g["F"].double(), g["dV"]
        if not case["fp64"]:
            F, dV = (g["U"].double() - um) / DT, dV.float().double()
        return um, F, tree.spread(g["m"], F, kernel, dV)
    f = tree.spread(g["m"], g["F"].double(), kernel)
    up = tree.trilinear(g["p"], field)[1]
    if kind == "step":
        return um, None, up, None, f
    v, ap, vp = g["v"].double(), g["ap"].double(), g["vp"].double()
    rel = up - v
    drag = 1.0 + 0.15 * (case["drag"] * torch.sqrt((rel ** 2).sum(0))) ** 0.687 if case["drag"] > 0 else 1.0
    a = drag * rel / TAU
    x = g["p"] + DT * (1.5 * v - 0.5 * vp)
    f[:, :3] -= (f[:, :3] * torch.pow(8.0, -tree.levels.double())[:, None]).sum(0)
    return um, up, x - torch.floor(x), v + DT * (1.5 * a - 0.5 * ap), a, v, f
