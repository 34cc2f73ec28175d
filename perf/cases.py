"""The work this library is measured on, through its public entry points.

Each case is one call sequence of a user's program on synthetic inputs of the
repository's own recipes (``dec_inputs``): jittered-lattice Delaunay meshes of
the unit cube (or the Kuhn lattice), lognormal conductivity per tet, penny
discs, Dirichlet values.  A case's ``kind`` says which part of the path a pass
covers:

  path      mesh_upload, hodge_assemble, laplacian_build, solve, k_eff
  mesh      mesh_upload, with the edge list and the structure of L read back
  hodge     hodge_assemble on an uploaded mesh, *1 and crack states read back
  system    laplacian_build, solve, k_eff on an assembled mesh
  solve     solve and k_eff on a built system
  study     hodge_assemble (new material), laplacian_build, solve, k_eff
  growth    hodge_assemble, laplacian_build, crack_evolve (largest flux)
  paths     hodge_assemble, laplacian_build, crack_paths (random orders)
  tet       tet_solve, the tet-centred form

Meshes: the Delaunay mesh of a jittered lattice with ``cells`` cells per axis, in
one of the cube's 48 orientations (the seed picks it: other coordinates, tets and
edges, the same counts), mirrored ``copies`` times per axis (boundary nodes move
tangentially only, so a mesh and its mirror image share their face).  That gives
(cells * copies + 1)^3 nodes within a fraction of a second.  Nodes and tets are
numbered as ``dec_inputs`` numbers them.
"""
import ctypes
import math

import numpy as np
import torch

from dec_inputs import (canonical_tets, crack_scales, delaunay_lattice, jittered_lattice,
                        kuhn_lattice, penny_discs)
from paper_2104_05999_gb300 import abi

# Solves stop at a relative residual of 1e-12, the tolerance of the kuhn9
# workload and of the parity tests: T then carries errors near 1e-11 and two
# right solvers can be told from a wrong one.  The tet-centred form stops at
# 1e-11 as its tests do (its FP64 residual levels off near 1e-12).
RTOL = 1e-12
RTOL_TET = 1e-11
MAX_ITER = 100000

_DEFAULT = dict(kind="path", mesh="delaunay", cells=9, copies=7, sigma=0.0, fields=1, discs=0,
                rmin=0.0, rmax=0.0, states=1, sets=1, random_t0=False, precond="fsai",
                mode="fp64", steps=0, paths=0)


def _case(name=None, **kw):
    c = dict(_DEFAULT, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the kuhn9 workload: the smallest problem a user checks the library
        # with, every call a few microseconds of work
        _case("kuhn9-path", kind="path", mesh="kuhn", cells=8, copies=1, random_t0=True,
              precond="jacobi", mode="fp64"),
        # the lognormal64 workload, a whole call in mixed precision: a new
        # mesh with one material
        _case("lognormal64-path", kind="path", cells=9, copies=7, sigma=1.0, mode="mixed"),
        # a new mesh of two million nodes: the integer work of every program
        _case("mesh127", kind="mesh", cells=18, copies=7),
        # a heterogeneous, cracked material on it (hetero192's recipe)
        _case("hodge127", kind="hodge", cells=18, copies=7, sigma=1.5, discs=1500,
              rmin=0.03, rmax=0.09),
        # the cracked128 workload in FP64: set-up and solve of one system
        _case("cracked127-fp64", kind="system", cells=18, copies=7, discs=2000, rmin=0.02,
              rmax=0.06, mode="fp64"),
        # the cracked128 workload's solve in its own mode
        _case("cracked127-mixed", kind="solve", cells=21, copies=6, discs=2000, rmin=0.02,
              rmax=0.06, mode="mixed"),
        # the hetero192 workload, the largest: 8 Dirichlet sets of one
        # heterogeneous cracked cube, set-up and batched solve
        _case("hetero172-sets", kind="system", cells=19, copies=9, sigma=1.5, discs=5000,
              rmin=0.02, rmax=0.06, sets=8, precond="shared", mode="batched"),
        # the growth96 workload: 64 states of a growing disc population
        _case("growth96-states", kind="solve", cells=19, copies=5, discs=1500, rmin=0.02,
              rmax=0.05, states=64, precond="shared", mode="batched"),
        # 16 materials on one 64^3 mesh, new ones at every pass
        _case("fields64", kind="study", cells=9, copies=7, sigma=1.0, fields=16,
              precond="shared", mode="batched"),
        # deterministic crack growth on the paper's crack-study mesh size
        _case("growth15-flux", kind="growth", cells=14, copies=1, steps=24, mode="fp64"),
        # stochastic cracking: 64 Monte-Carlo paths on the same mesh
        _case("growth15-paths", kind="paths", cells=14, copies=1, steps=8, paths=64),
        # the paper's own tet-centred system on the 64^3 cube
        _case("tet64", kind="tet", cells=9, copies=7, random_t0=True),
    ]


def _lattice(rng, lo, hi):
    """(cells, copies) of a lattice of lo..hi nodes per axis, log-uniform."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if n <= 22:
        return max(lo - 1, int(n) - 1), 1
    copies = max(2, round((n - 1) / rng.randint(9, 20)))
    return min(21, max(8, int((n - 1) / copies))), copies


def draw(rng):
    """A case of the listed ones' ranges.  Radii scale with the lattice so that
    about the same share of dual faces is cut, as make_workload does."""
    what = rng.choice(["path", "mesh", "hodge", "fp64", "mixed", "sets", "states", "fields",
                       "flux", "paths", "tet"])

    def cracks(cells, copies, base, count, r0, r1):
        n = cells * copies + 1
        f = base / n
        return dict(discs=max(1, round(count / f ** 3 * rng.uniform(0.5, 1.3))), rmin=r0 * f,
                    rmax=r1 * f)

    if what == "path":
        if rng.random() < 0.3:
            return _case(kind="path", mesh="kuhn", cells=rng.randint(4, 15), copies=1,
                         random_t0=True, precond="jacobi", mode="fp64")
        cells, copies = _lattice(rng, 9, 100)
        return _case(kind="path", cells=cells, copies=copies, sigma=rng.uniform(0.3, 1.5),
                     mode=rng.choice(["fp64", "mixed"]))
    if what == "mesh":
        cells, copies = _lattice(rng, 9, 150)
        return _case(kind="mesh", cells=cells, copies=copies)
    if what == "hodge":
        cells, copies = _lattice(rng, 12, 140)
        c = _case(kind="hodge", cells=cells, copies=copies, sigma=rng.choice([0.0, 1.0, 1.5]),
                  fields=1)
        c.update(cracks(cells, copies, 128, 2000, 0.02, 0.06))
        if c["sigma"] == 0.0:
            c["states"] = rng.choice([1, 1, 5, 33])
        return c
    if what in ("fp64", "mixed"):
        cells, copies = _lattice(rng, 14, 130)
        c = _case(kind=rng.choice(["system", "solve"]), cells=cells, copies=copies,
                  sigma=rng.choice([0.0, 1.0]), mode=what, random_t0=True,
                  sets=rng.choice([1, 1, 2]))
        c.update(cracks(cells, copies, 128, 2000, 0.02, 0.06))
        return c
    if what == "sets":
        cells, copies = _lattice(rng, 20, 125)
        c = _case(kind=rng.choice(["system", "solve"]), cells=cells, copies=copies, sigma=1.5,
                  sets=rng.choice([2, 5, 8, 8, 13, 16]), precond="shared", mode="batched",
                  random_t0=True)
        c.update(cracks(cells, copies, 192, 5000, 0.02, 0.06))
        return c
    if what == "states":
        cells, copies = _lattice(rng, 16, 85)
        c = _case(kind=rng.choice(["study", "solve"]), cells=cells, copies=copies,
                  states=rng.randint(3, 64), precond="shared", mode="batched")
        c.update(cracks(cells, copies, 96, 1500, 0.02, 0.05))
        return c
    if what == "fields":
        cells, copies = _lattice(rng, 14, 75)
        return _case(kind=rng.choice(["study", "solve"]), cells=cells, copies=copies,
                     sigma=rng.uniform(0.5, 1.5), fields=rng.randint(2, 40), precond="shared",
                     mode="batched")
    if what == "flux":
        return _case(kind="growth", cells=rng.randint(8, 17), copies=1,
                     steps=rng.randint(5, 40), mode="fp64",
                     precond=rng.choice(["fsai", "fsai", "jacobi"]))
    if what == "paths":
        return _case(kind="paths", cells=rng.randint(8, 16), copies=1,
                     steps=rng.randint(3, 10), paths=rng.randint(5, 64))
    cells, copies = _lattice(rng, 12, 70)
    return _case(kind="tet", cells=cells, copies=copies, random_t0=True)


# ------------------------------------------------------------------ inputs

def _sort_tets(t, n):
    """Rows in lexicographic order (every row's own order kept)."""
    t = t.long()
    order = torch.argsort(t[:, 2] * n + t[:, 3], stable=True)
    t = t[order]
    order = torch.argsort(t[:, 0] * n + t[:, 1], stable=True)
    return t[order].int().contiguous()


_tiles = {}       # Delaunay meshes by cells per axis: Qhull takes most of a preparation


def _tile(e, seed):
    """The mesh of (e + 1)^3 nodes in orientation seed % 48 (numpy arrays)."""
    if e not in _tiles:
        xyz = jittered_lattice(e + 1, np.random.default_rng(1000 + e))
        _tiles[e] = xyz, delaunay_lattice(xyz, e + 1, block=e + 1, workers=1)
    xyz, tets = _tiles[e]
    axes = ((0, 1, 2), (1, 2, 0), (2, 0, 1), (0, 2, 1), (2, 1, 0), (1, 0, 2))[seed % 48 // 8]
    g = np.arange((e + 1) ** 3)
    idx = [g % (e + 1), g // (e + 1) % (e + 1), g // (e + 1) ** 2]
    idx = [idx[a] for a in axes]
    xyz = xyz[:, axes].copy()
    for a in range(3):
        if seed >> a & 1:
            idx[a] = e - idx[a]
            xyz[:, a] = 1.0 - xyz[:, a]
    new = idx[0] + (e + 1) * (idx[1] + (e + 1) * idx[2])      # old node -> new node
    out = np.empty_like(xyz)
    out[new] = xyz
    return out, canonical_tets(new[tets], out)


def _mesh(case, seed):
    """xyz f64[n, 3], tets i32[m, 4] (CUDA tensors) of the case's cube."""
    e, r = case["cells"], case["copies"]
    dev = torch.device("cuda")
    if case["mesh"] == "kuhn":
        xyz, tets = kuhn_lattice(e * r + 1)
        return torch.from_numpy(xyz).to(dev), torch.from_numpy(tets).to(dev)
    tile, tets = (torch.from_numpy(a).to(dev) for a in _tile(e, seed))
    tets = tets.long()
    if r == 1:
        return tile, tets.int().contiguous()
    N = e * r + 1
    # node I of an axis belongs to copy c, at tile position i (mirrored in odd copies)
    g = torch.arange(N, device=dev)
    c = torch.clamp(g // e, max=r - 1)
    i = torch.where(c % 2 == 0, g - c * e, e - (g - c * e))
    iz, iy, ix = i[:, None, None], i[None, :, None], i[None, None, :]
    src = (ix + (e + 1) * (iy + (e + 1) * iz)).reshape(-1)
    shape = (N, N, N)
    copy_of = [c[None, None, :].expand(shape).reshape(-1), c[None, :, None].expand(shape).reshape(-1),
               c[:, None, None].expand(shape).reshape(-1)]
    cols = []
    for ax in range(3):
        t = tile[src, ax]
        k = copy_of[ax]
        cols.append((k + torch.where(k % 2 == 0, t, 1.0 - t)) / r)
    xyz = torch.stack(cols, dim=1).contiguous()
    del src, copy_of, cols
    # tets of every copy: local lattice indices mapped to global ones
    li = [tets % (e + 1), (tets // (e + 1)) % (e + 1), tets // (e + 1) ** 2]
    parts = []
    for cz in range(r):
        for cy in range(r):
            for cx in range(r):
                gl = [cc * e + (v if cc % 2 == 0 else e - v) for cc, v in zip((cx, cy, cz), li)]
                parts.append((gl[0] + N * (gl[1] + N * gl[2])).int())
    t = torch.sort(torch.cat(parts), dim=1).values
    del parts
    p = [xyz[t[:, k].long()] for k in range(4)]
    vol = ((p[1] - p[0]) * torch.cross(p[2] - p[0], p[3] - p[0], dim=1)).sum(1)
    flip = vol < 0
    t = torch.stack([t[:, 0], t[:, 1], torch.where(flip, t[:, 3], t[:, 2]),
                     torch.where(flip, t[:, 2], t[:, 3])], dim=1)
    return xyz, _sort_tets(t, N ** 3)


def _inputs(case, seed):
    """Mesh, tags, Dirichlet values, conductivity, discs and scales as a
    user's program holds them: on the GPU (discs and scales on the host)."""
    rngs = [np.random.default_rng(s) for s in np.random.SeedSequence(seed).spawn(3)]
    xyz, tets = _mesh(case, seed)
    dev = xyz.device
    m, n = len(tets), len(xyz)
    face = (xyz == 0.0) | (xyz == 1.0)
    tags = torch.where(face.any(1), 2, 0).to(torch.uint8)
    dirichlet = face[:, 0]
    tags[dirichlet] = 1
    gen = torch.Generator(device=dev).manual_seed(int(rngs[0].integers(1 << 62)))
    T0 = torch.zeros((case["sets"], n), dtype=torch.float64, device=dev)
    T0[:, dirichlet] = torch.rand((case["sets"], int(dirichlet.sum())), generator=gen,
                                  dtype=torch.float64, device=dev)
    # set 0: 1 on x = 0 and 0 on x = 1, or uneven temperatures around them
    T0[0] *= 0.5 if case["random_t0"] else 0.0
    T0[0] += (xyz[:, 0] == 0.0).double()
    k = None
    if case["sigma"] > 0.0:
        z = torch.randn((case["fields"], m), generator=gen, dtype=torch.float64, device=dev)
        k = torch.exp(case["sigma"] * z)
        k = k[0] if case["fields"] == 1 else k
    discs = penny_discs(case["discs"], case["rmin"], case["rmax"], rngs[1]) if case["discs"] else None
    scales = crack_scales(case["states"]) if case["states"] > 1 else None
    return dict(xyz=xyz, tets=tets, tags=tags, T0=T0, k=k, discs=discs, scales=scales,
                rng=rngs[2])


_PRECOND = {"jacobi": abi.DEC_PRECOND_JACOBI, "fsai": abi.DEC_PRECOND_FSAI,
            "shared": abi.DEC_PRECOND_FSAI_SHARED}
_MODE = {"fp64": abi.DEC_MODE_FP64, "mixed": abi.DEC_MODE_MIXED,
         "batched": abi.DEC_MODE_MIXED_BATCHED}


def _instances(case):
    return max(case["states"], case["fields"], case["sets"])


def _hodge(s):
    c = s["case"]
    if c["fields"] > 1:
        s["ctx"].dec_hodge_assemble_fields(s["k"], s["discs"])
    else:
        s["ctx"].dec_hodge_assemble(s["k"], s["discs"], s["scales"])


def _system(s):
    s["ctx"].dec_laplacian_build(s["T0"], _PRECOND[s["case"]["precond"]])


def _solve(s):
    ctx = s["ctx"]
    ctx.dec_solve(RTOL, MAX_ITER, _MODE[s["case"]["mode"]], s["T"])
    q_in, q_out, energy = ctx.dec_k_eff()
    return {"T": s["T"], "q_in": q_in, "q_out": q_out, "energy": energy}


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    ctx = s["ctx"] = abi.Context(device=0)
    n, dev = len(s["xyz"]), s["xyz"].device
    if kind in ("path", "system", "solve", "study"):
        s["T"] = torch.zeros((_instances(case), n), dtype=torch.float64, device=dev)
    torch.cuda.synchronize()
    if kind == "path":
        return s
    # the mesh, and what of the path comes before the measured part
    ctx.dec_mesh_upload(s["xyz"], s["tets"], s["tags"])
    _, m, ne, nnz, _ = ctx.sizes()
    i32 = dict(dtype=torch.int32, device=dev)
    if kind == "mesh":
        s["out"] = {"E": torch.zeros((ne, 2), **i32), "t2e": torch.zeros((m, 6), **i32),
                    "rowptr": torch.zeros(n + 1, **i32), "col": torch.zeros(nnz, **i32)}
    if kind == "hodge":
        s["out"] = {"w": torch.zeros(ne, dtype=torch.float64, device=dev),
                    "first_cut": torch.zeros(ne, dtype=torch.uint8, device=dev)}
    if kind in ("system", "solve", "paths"):
        _hodge(s)
    if kind == "solve":
        _system(s)
    if kind == "paths":
        # every path its own random order of conducting edges
        w, _ = ctx.dec_get_hodge()
        live = np.flatnonzero(w > 1e-3 * w.max())
        s["orders"] = np.stack([s["rng"].choice(live, case["steps"], replace=False)
                                for _ in range(case["paths"])]).astype(np.int32)
    torch.cuda.synchronize()
    return s


def _address(t):
    return ctypes.c_void_p(t.data_ptr())


def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"]
    if kind == "path":
        ctx.dec_mesh_upload(s["xyz"], s["tets"], s["tags"])
        _hodge(s)
        _system(s)
        return _solve(s)
    if kind == "mesh":
        ctx.dec_mesh_upload(s["xyz"], s["tets"], s["tags"])
        o = s["out"]                     # the C entry points, into the user's device buffers
        ctx._check(ctx.lib.dec_get_edges(ctx.h, _address(o["E"]), _address(o["t2e"])))
        ctx._check(ctx.lib.dec_get_csr(ctx.h, 0, _address(o["rowptr"]), _address(o["col"]),
                                       None, None))
        return o
    if kind == "hodge":
        _hodge(s)
        o = s["out"]
        ctx._check(ctx.lib.dec_get_hodge(ctx.h, _address(o["w"]), _address(o["first_cut"])))
        return o
    if kind == "system":
        _system(s)
        return _solve(s)
    if kind == "solve":
        return _solve(s)
    if kind == "study":
        _hodge(s)
        _system(s)
        return _solve(s)
    if kind == "growth":
        _hodge(s)
        _system(s)
        _, cracked, k_eff = ctx.dec_crack_evolve(abi.DEC_CRACK_MAX_FLUX, s["case"]["steps"],
                                                 rtol=RTOL, mode=_MODE[s["case"]["mode"]])
        return {"cracked": cracked, "k_eff": k_eff}
    if kind == "paths":
        _hodge(s)
        _system(s)
        _, k_eff, steps = ctx.dec_crack_paths(s["orders"], rtol=RTOL)
        return {"k_eff": np.concatenate(k_eff), "steps": steps}
    r = ctx.dec_tet_solve(s["T0"][0], rtol=RTOL_TET)
    return {"alpha": r["alpha"], "q_in": r["q_in"], "q_out": r["q_out"]}


# -------------------------------------------------------------------- work

def _sizes(case):
    """Nodes, tets, edges and lattice size, by the usual counts of these meshes."""
    N = case["cells"] * case["copies"] + 1
    n = N ** 3
    per = 5.0 if case["mesh"] == "kuhn" else 5.95
    m = per * (N - 1) ** 3 + 2.0 * (N - 1) ** 2
    return n, m, n + m + 3.0 * (N - 1) ** 2, N


def work(case):
    """Inputs read once, outputs written once, and for a solve the operator
    and preconditioner once per iteration (3.7 iterations per lattice node
    with a sparse approximate inverse, twice that with Jacobi) unless they fit
    the 129 MB L2, with the FP64 vectors of CG's definition left out."""
    n, m, ne, N = _sizes(case)
    B = _instances(case)
    kind = case["kind"]
    nnz = 2 * ne + n
    mesh = 24 * n + 16 * m + n
    edges = 8 * ne + 24 * m
    hodge = mesh + (8 * m * case["fields"] if case["sigma"] else 0) + 9 * ne
    fp64 = case["mode"] == "fp64"
    its = 3.7 * N if case["precond"] != "jacobi" else 7.4 * N
    per_entry = 12 if fp64 else 8
    half = 12 if fp64 else 6
    own = B if case["mode"] == "batched" and case["sets"] == 1 else 1    # factors
    once = per_entry * nnz + (0 if case["precond"] == "jacobi" else
                              2 * (half + 2 * (own - 1)) * (nnz + n) / 2)
    calls = 1 if case["mode"] == "batched" else B
    flops_it = B * (2 * nnz + 2 * (nnz + n) + 12 * n)
    solve = 16 * n * B + calls * once * (its if once > 129e6 else 1)
    if kind == "mesh":
        return {"bytes": mesh + edges + 4 * (n + nnz), "flops": 30 * m}
    if kind == "hodge":
        return {"bytes": hodge, "flops": 400 * m}
    if kind == "tet":
        it = 13.0 * N
        return {"bytes": 8 * (n + m) + 100 * m * (it if 100 * m > 129e6 else 1),
                "flops": it * m * 45}
    if kind in ("growth", "paths"):
        it = 4.5 * N * (case["steps"] + 1)
        P = max(1, case["paths"])
        return {"bytes": hodge + once * P + 8 * P * case["steps"],
                "flops": it * P * (4 * nnz + 14 * n)}
    total = solve + {"path": mesh + hodge, "system": 8 * n, "study": hodge, "solve": 0}[kind]
    return {"bytes": total, "flops": its * flops_it + (400 * m if kind in ("path", "study") else 0)}


# ------------------------------------------------------------------- exact
# The same quantities in plain torch FP64, written from the definitions.

_EDGES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


def _cross(a, b):
    return torch.cross(a, b, dim=-1)


def _dot(a, b):
    return (a * b).sum(-1)


def _tri_centre(p, q, r):
    a, b = q - p, r - p
    ab = _cross(a, b)
    num = _cross(_dot(a, a)[..., None] * b - _dot(b, b)[..., None] * a, ab)
    return p + num / (2.0 * _dot(ab, ab))[..., None]


def _tet_centre(P):
    a, b, c = P[1] - P[0], P[2] - P[0], P[3] - P[0]
    num = (_dot(a, a)[..., None] * _cross(b, c) + _dot(b, b)[..., None] * _cross(c, a) +
           _dot(c, c)[..., None] * _cross(a, b))
    return P[0] + num / (2.0 * _dot(a, _cross(b, c)))[..., None]


def _exact_edges(tets, n):
    t = tets.long()
    lo = torch.stack([torch.minimum(t[:, a], t[:, b]) for a, b in _EDGES], 1)
    hi = torch.stack([torch.maximum(t[:, a], t[:, b]) for a, b in _EDGES], 1)
    key, t2e = torch.unique(lo * n + hi, return_inverse=True)
    return torch.stack([key // n, key % n], 1), t2e


def _exact_hodge(s, t2e, ne):
    """*1 per field [F, ne]: signed dual areas over edge lengths times the
    dual face's mean conductivity (weights: unsigned part areas)."""
    t = s["tets"].long()
    P = [s["xyz"][t[:, v]] for v in range(4)]
    cT = _tet_centre(P)
    geo = torch.zeros(ne, dtype=torch.float64, device=t.device)
    area = torch.zeros_like(geo)
    k = None if s["k"] is None else s["k"].reshape(-1, len(t))
    ku = None if k is None else torch.zeros((len(k), ne), dtype=torch.float64, device=t.device)
    for j, (a, b) in enumerate(_EDGES):
        mid, length = 0.5 * (P[a] + P[b]), torch.linalg.norm(P[b] - P[a], dim=1)
        u = torch.zeros(len(t), dtype=torch.float64, device=t.device)
        for c in range(4):
            if c in (a, b):
                continue
            d = 6 - a - b - c
            cF = _tri_centre(P[a], P[b], P[c])
            e = (P[b] - P[a]) / length[:, None]
            inward = P[c] - P[a]
            inward = inward - _dot(inward, e)[:, None] * e
            h1 = _dot(cF - mid, inward) / torch.linalg.norm(inward, dim=1)
            nrm = _cross(P[b] - P[a], P[c] - P[a])
            nrm = nrm * torch.sign(_dot(P[d] - P[a], nrm))[:, None]
            h2 = _dot(cT - P[a], nrm) / torch.linalg.norm(nrm, dim=1)
            piece = 0.5 * h1 * h2 / length
            geo.index_add_(0, t2e[:, j], piece)
            u = u + piece.abs()
        area.index_add_(0, t2e[:, j], u)
        if k is not None:
            for f in range(len(k)):
                ku[f].index_add_(0, t2e[:, j], u * k[f])
    if k is None:
        return geo[None]
    return torch.where(area > 0, geo * ku / area, torch.zeros_like(ku))


def _exact_cuts(s, t2e, ne):
    """First crack state that cuts each edge's dual face (states: never)."""
    scales = np.array([1.0]) if s["scales"] is None else s["scales"]
    dev = s["xyz"].device
    first = torch.full((ne,), len(scales), dtype=torch.int64, device=dev)
    if s["discs"] is None:
        return first
    t = s["tets"].long()
    P = [s["xyz"][t[:, v]] for v in range(4)]
    cT = _tet_centre(P)
    ball = torch.linalg.norm(cT - P[0], dim=1) * (1 + 1e-9)
    cTx, cTy, cTz = (v.contiguous() for v in cT.unbind(1))
    pairs = []
    for q, (cx, cy, cz, nx, ny, nz, r) in enumerate(s["discs"].tolist()):
        vx, vy, vz = cTx - cx, cTy - cy, cTz - cz
        reach = ball + r * float(scales[-1])
        near = (vx * nx + vy * ny + vz * nz).abs_() <= ball
        near &= vx.square_().add_(vy.square_()).add_(vz.square_()) <= reach.square_()
        at = near.nonzero()[:, 0]
        pairs.append(torch.stack([at, torch.full_like(at, q)], 1))
    at, q = torch.cat(pairs).unbind(1)
    discs = torch.from_numpy(s["discs"]).to(dev)
    sc = torch.from_numpy(np.asarray(scales)).to(dev)
    for part in torch.split(torch.arange(len(at), device=dev), 1 << 21):
        i, D = at[part], discs[q[part]]
        V = [p[i] for p in P]
        cen, nrm, rad = D[:, :3], D[:, 3:6], D[:, 6]
        for j, (a, b) in enumerate(_EDGES):
            rho = torch.full((len(i),), math.inf, dtype=torch.float64, device=dev)
            for c in range(4):
                if c in (a, b):
                    continue
                T = [0.5 * (V[a] + V[b]), _tri_centre(V[a], V[b], V[c]), cT[i]]
                d = [_dot(x - cen, nrm) for x in T]
                # end points of the segment where the plane meets the triangle
                lo = torch.full((len(i), 3), math.nan, dtype=torch.float64, device=dev)
                hi = lo.clone()
                for x, y in ((0, 1), (1, 2), (0, 2)):
                    hit = d[x] * d[y] < 0
                    X = T[x] + (d[x] / (d[x] - d[y]))[:, None] * (T[y] - T[x])
                    new = hit & lo[:, 0].isnan()
                    hi = torch.where((hit & ~new)[:, None], X, hi)
                    lo = torch.where(new[:, None], X, lo)
                for x in range(3):
                    hit = d[x] == 0
                    new = hit & lo[:, 0].isnan()
                    hi = torch.where((hit & ~new)[:, None], T[x], hi)
                    lo = torch.where(new[:, None], T[x], lo)
                flat = (d[0] == 0) & (d[1] == 0) & (d[2] == 0)
                hi = torch.where(hi.isnan(), lo, hi)
                w = hi - lo
                ww = _dot(w, w)
                at01 = torch.where(ww > 0, (_dot(cen - lo, w) / ww).clamp(0, 1), torch.zeros_like(ww))
                dist = torch.linalg.norm(cen - lo - at01[:, None] * w, dim=1)
                dist = torch.where(flat | dist.isnan(), torch.full_like(dist, math.inf), dist)
                rho = torch.minimum(rho, dist)
            cut = torch.searchsorted(sc, rho / rad)      # first state with scale >= rho / r
            first.scatter_reduce_(0, t2e[i, j], cut, "amin")
    return first


def _block_pcg(E, W, dirichlet, T0, tol=1e-15, most=20000):
    """T [B, n] of sum_j w_ij (T_i - T_j) = 0 at free nodes, by Jacobi PCG
    restarted from the true residual; W [1 or B, ne], T0 [1 or B, n]."""
    i, j = E[:, 0], E[:, 1]
    B, n = max(len(W), len(T0)), T0.shape[1]
    free = ~dirichlet
    diag = torch.zeros((len(W), n), dtype=torch.float64, device=W.device)
    diag.index_add_(1, i, W).index_add_(1, j, W)
    inv = torch.where(free & (diag > 0), 1.0 / diag, torch.zeros_like(diag))

    def apply(x):
        f = W * (x[:, i] - x[:, j])
        y = torch.zeros((B, n), dtype=torch.float64, device=W.device)
        y.index_add_(1, i, f).index_add_(1, j, -f)
        return y * free

    T = torch.where(dirichlet, T0, torch.zeros_like(T0)).expand(B, n).clone()
    b = (-apply(T)).square().sum(1)
    best, held = math.inf, 0
    for _ in range(12):                       # restarts
        r = -apply(T)
        rr = (r.square().sum(1) / b).max().item()
        if rr <= tol ** 2 or held >= 2:
            break
        held = held + 1 if rr > 0.25 * best else 0
        best = min(best, rr)
        z = inv * r
        p = z.clone()
        rz = (r * z).sum(1)
        stop = r.square().sum(1) * 1e-16
        for it in range(most):
            q = apply(p)
            alpha = torch.where(rz > 0, rz / (p * q).sum(1), torch.zeros_like(rz))
            T += alpha[:, None] * p
            r -= alpha[:, None] * q
            z = inv * r
            new = (r * z).sum(1)
            p = z + torch.where(rz > 0, new / rz, torch.zeros_like(rz))[:, None] * p
            rz = new
            if it % 32 == 31 and bool((r.square().sum(1) <= stop).all()):
                break
    return T


def _exact_k_eff(E, W, T, x, dirichlet):
    i, j = E[:, 0], E[:, 1]
    d = T[:, i] - T[:, j]
    f = W * d
    net = torch.zeros_like(T)
    net.index_add_(1, i, f).index_add_(1, j, -f)
    return ((net * (dirichlet & (x == 0.0))).sum(1), -(net * (dirichlet & (x == 1.0))).sum(1),
            (f * d).sum(1))


def _exact_tet(s):
    t = s["tets"].long()
    n, m = len(s["xyz"]), len(t)
    P = [s["xyz"][t[:, v]] for v in range(4)]
    cT = _tet_centre(P)
    tri, height, area = [], [], []
    for v in range(4):
        o = [w for w in range(4) if w != v]
        A, B, C = (P[w] for w in o)
        nrm = _cross(B - A, C - A)
        size = torch.linalg.norm(nrm, dim=1)
        height.append(_dot(cT - A, nrm) / size * torch.sign(_dot(P[v] - A, nrm)))
        area.append(0.5 * size)
        tri.append(torch.sort(t[:, o], dim=1).values)
    tri, height, area = torch.cat(tri), torch.cat(height), torch.cat(area)
    owner = torch.arange(m, device=t.device).repeat(4)
    order = torch.argsort(tri[:, 2], stable=True)
    order = order[torch.argsort(tri[order, 0] * n + tri[order, 1], stable=True)]
    tri, height, area, owner = tri[order], height[order], area[order], owner[order]
    same = (tri[1:] == tri[:-1]).all(1)
    pair = same.nonzero()[:, 0]
    single = torch.ones(4 * m, dtype=torch.bool, device=t.device)
    single[pair] = False
    single[pair + 1] = False
    w_in = 1.0 / torch.clamp((height[pair] + height[pair + 1]) / area[pair], min=1e-8)
    a, b = owner[pair], owner[pair + 1]
    wall = single & (s["tags"][tri] == 1).all(1)
    w_out = 1.0 / torch.clamp(height[wall] / area[wall], min=1e-8)
    c, tw = owner[wall], tri[wall]
    value = s["T0"][0][tw].mean(1)
    # the wall faces as edges to Dirichlet nodes appended after the tets
    nw = len(c)
    E = torch.cat([torch.stack([a, b], 1),
                   torch.stack([c, m + torch.arange(nw, device=t.device)], 1)])
    W = torch.cat([w_in, w_out])[None]
    T0 = torch.cat([torch.zeros(m, dtype=torch.float64, device=t.device), value])[None]
    dirichlet = torch.arange(m + nw, device=t.device) >= m
    T = _block_pcg(E, W, dirichlet, T0)[0]
    flow = w_out * (value - T[c])
    x = s["xyz"][:, 0][tw]
    return {"alpha": T[:m], "q_in": flow[(x == 0.0).all(1)].sum(),
            "q_out": -flow[(x == 1.0).all(1)].sum()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "mesh":
        return None                               # whole numbers only
    n, m, ne, N = _sizes(case)
    solves = {"growth": case["steps"] + 1, "paths": (case["steps"]) * case["paths"]}.get(
        kind, _instances(case))
    if kind not in ("hodge", "tet") and N * solves * ne > 6e9 and kind not in ("growth", "paths"):
        return None                               # over about 20 seconds
    s = _inputs(case, seed)
    if kind == "tet":
        return _exact_tet(s)
    n = len(s["xyz"])
    E, t2e = _exact_edges(s["tets"], n)
    W = _exact_hodge(s, t2e, len(E))
    if kind == "hodge":
        return {"w": W[0], "first_cut": None}
    cut = _exact_cuts(s, t2e, len(E))
    if case["states"] > 1:
        W = W * (cut[None] > torch.arange(case["states"], device=cut.device)[:, None])
    else:
        W = W * (cut > 0)
    dirichlet = s["tags"] == 1
    x = s["xyz"][:, 0]
    if kind == "growth":
        k_eff = []
        for _ in range(case["steps"]):
            T = _block_pcg(E, W, dirichlet, s["T0"])
            flux = torch.where(W[0] > 0, (W[0] * (T[0, E[:, 0]] - T[0, E[:, 1]])).abs(),
                               torch.full_like(W[0], -1.0))
            W[0, int(flux.argmax())] = 0.0
            T = _block_pcg(E, W, dirichlet, s["T0"])
            k_eff.append(_exact_k_eff(E, W, T, x, dirichlet)[0][0])
        return {"cracked": None, "k_eff": torch.stack(k_eff)}
    if kind == "paths":
        # the conducting edges, as prepare() picks them
        w = W[0].cpu().numpy()
        live = np.flatnonzero(w > 1e-3 * w.max())
        orders = np.stack([s["rng"].choice(live, case["steps"], replace=False)
                           for _ in range(case["paths"])])
        W = W.repeat(case["paths"], 1)
        rows = torch.arange(case["paths"], device=W.device)
        k_eff = []
        for step in range(case["steps"]):
            W[rows, torch.from_numpy(orders[:, step]).to(W.device)] = 0.0
            T = _block_pcg(E, W, dirichlet, s["T0"])
            k_eff.append(_exact_k_eff(E, W, T, x, dirichlet)[0])
        return {"k_eff": torch.stack(k_eff, 1).reshape(-1), "steps": None}
    T = _block_pcg(E, W, dirichlet, s["T0"])
    q_in, q_out, energy = _exact_k_eff(E, W, T, x, dirichlet)
    return {"T": T, "q_in": q_in, "q_out": q_out, "energy": energy}
