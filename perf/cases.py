"""Performance cases: the calls that users of the library spend their time in,
over the range of sizes, meshes, precisions and solvers that it is used with.

A case is one of five calls (``"call"``):

* ``simulate``  assemble, solve for the pressure, take explicit transport
  steps, release the system: one whole run on one mesh;
* ``resample``  new permeabilities on an assembled mesh and a solve: the inner
  loop of an uncertainty study;
* ``transport`` explicit steps on fluxes that are already known: the long run
  of a tracer through one pressure field;
* ``batch``     ``simulate`` for many independent realisations at once;
* ``product``   one product with the eliminated matrix: the inner step of a
  caller's own Krylov method.

Meshes are jittered lattices of hexahedra (the fast path of the interface), of
tetrahedra or of triangular prisms (the general polyhedral descriptor), with a
network of axis-aligned rectangular fractures and a lognormal anisotropic
matrix permeability, p = 1 - x on the sides x = 0 and x = 1; the prism meshes
instead carry one injector and two producers and no Dirichlet node.  The mesh
and the network belong to the case; node positions and permeabilities come
from the seed.  Solves run to the interface's default tolerance.
"""
import math
import random

import numpy as np
import torch

import paper_1602_03641_gb300 as vag

DEV = "cuda"
RTOL = 1e-12   # the default of System.solve

PRECISION = {"fp64": vag.VAG_FP64, "mixed": vag.VAG_MIXED, "fp64_pc32": vag.VAG_FP64_PC32}
PRECOND = {"jacobi": vag.VAG_PC_JACOBI, "chebyshev": vag.VAG_PC_CHEBYSHEV, "aggregation": vag.VAG_PC_AMG,
           "classical": vag.VAG_PC_AMG_RS}
KRYLOV = {"cg": vag.VAG_KRYLOV_CG, "bicgstab": vag.VAG_KRYLOV_BICGSTAB, "gmres": vag.VAG_KRYLOV_GMRES}


def _case(name, call, cells, dims, fractures, ratio, precision, precond, krylov="cg", steps=0, mem="device", count=1):
    nx, ny, nz = dims
    return {"name": name, "call": call, "cells": cells, "nx": nx, "ny": ny, "nz": nz, "fractures": fractures,
            "ratio": ratio, "precision": precision, "precond": precond, "krylov": krylov, "steps": steps, "mem": mem,
            "count": count}


def listed():
    return [
        # the smallest run: every launch and every wait counts, with the interface's default solver
        _case("run_hex8", "simulate", "hex", (8, 8, 8), 1, 1e4, "fp64", "jacobi", steps=10),
        # a small ragged mesh handed over as numpy arrays, results back in numpy arrays
        _case("run_hex_ragged_host", "simulate", "hex", (29, 23, 19), 5, 1e3, "fp64", "aggregation", steps=100,
              mem="host"),
        # the 64^3 benchmark: FP64 aggregation-AMG CG and 200 steps
        _case("run_hex64", "simulate", "hex", (64, 64, 64), 4, 1e4, "fp64", "aggregation", steps=200),
        # the headline: 128^3 with 50 fractures, FP32 classical-AMG CG inside FP64 refinement, 1000 steps
        _case("run_hex128", "simulate", "hex", (128, 128, 128), 50, 1e4, "mixed", "classical", steps=1000),
        # tetrahedra through the general descriptor, permeability ratio 20
        _case("run_tet36", "simulate", "tet", (36, 36, 36), 8, 20.0, "mixed", "classical", steps=200),
        # prisms with vertical fractures and wells, no Dirichlet node
        _case("run_prism_wells", "simulate", "prism", (72, 48, 12), 12, 1e4, "mixed", "classical", steps=200),
        # an uncertainty study on a fixed mesh: FP32 aggregation-AMG CG inside refinement
        _case("resample_hex48", "resample", "hex", (48, 48, 48), 10, 1e5, "mixed", "aggregation"),
        # the same on a large mesh: FP64 CG with the FP32 classical V-cycle
        _case("resample_hex96", "resample", "hex", (96, 96, 96), 30, 1e4, "fp64_pc32", "classical"),
        # restarted GMRES with the classical V-cycle in FP64, the solver pair of the paper's tables
        _case("resample_gmres_hex56", "resample", "hex", (56, 56, 56), 12, 1e2, "fp64", "classical", "gmres"),
        # a tracer run on known fluxes, a box of another shape
        _case("transport_hex_box", "transport", "hex", (140, 90, 61), 20, 1e4, "mixed", "classical", steps=500),
        # independent realisations of 16 to 40 cells a side in one batch
        _case("batch32", "batch", "hex", (40, 40, 40), 8, 1e4, "mixed", "classical", steps=100, count=32),
        # one product with the FP64 matrix on the caller's vectors
        _case("product_hex80", "product", "hex", (80, 80, 80), 16, 1e4, "fp64", "jacobi"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choice(["simulate", "simulate", "simulate", "resample", "resample", "transport", "batch", "product"])
    cells = rng.choice(["hex", "hex", "tet", "prism"]) if call in ("simulate", "resample") else "hex"
    solvers = [("fp64", "aggregation", "cg"), ("fp64", "classical", "cg"), ("mixed", "aggregation", "cg"),
               ("mixed", "classical", "cg"), ("fp64_pc32", "classical", "cg"), ("fp64", "classical", "gmres"),
               ("fp64", "aggregation", "bicgstab")]
    n = _log(rng, 7, {"hex": 110, "tet": 56, "prism": 80}[cells])
    if call == "simulate" and n < 24 or call == "resample" and rng.random() < 0.2:   # one-level solvers: small meshes
        n = min(n, 40.0)
        solvers += [("fp64", "jacobi", "cg"), ("fp64", "chebyshev", "cg")]
    dims = [max(5, round(n * rng.uniform(0.75, 1.3))) for _ in range(3)]
    if cells == "prism":
        dims = [max(10, dims[0]), max(10, dims[1]), max(4, dims[2] // 4)]
    precision, precond, krylov = rng.choice(solvers)
    if call in ("batch", "transport"):
        precision, precond, krylov = rng.choice([("mixed", "classical", "cg"), ("fp64", "aggregation", "cg")])
    count = 1
    if call == "batch":
        count = rng.randint(2, 32)
        dims = [rng.randint(16, 44)] * 3
    steps = 0 if call in ("resample", "product") else round(_log(rng, 1, 600))
    mem = "host" if call == "simulate" and n < 40 and rng.random() < 0.3 else "device"
    case = _case("", call, cells, dims, rng.randint(1, 20), round(10 ** rng.uniform(1.0, 5.0), 1), precision, precond,
                 krylov, steps, mem, count)
    del case["name"]
    return case


# ----------------------------------------------------------------------------
# meshes
# ----------------------------------------------------------------------------

_CUBE = [(l & 1, (l >> 1) & 1, (l >> 2) & 1) for l in range(8)]
# the cells that each lattice cube is cut into, by its corners
_CUT = {"hex": [(0, 1, 2, 3, 4, 5, 6, 7)],
        "tet": [(0, 1, 3, 7), (0, 3, 2, 7), (0, 2, 6, 7), (0, 6, 4, 7), (0, 4, 5, 7), (0, 5, 1, 7)],
        "prism": [(0, 1, 3, 4, 5, 7), (0, 3, 2, 4, 7, 6)]}
_FACES = {"hex": [(0, 2, 6, 4), (1, 3, 7, 5), (0, 1, 5, 4), (2, 3, 7, 6), (0, 1, 3, 2), (4, 5, 7, 6)],
          "tet": [(1, 2, 3), (0, 3, 2), (0, 1, 3), (0, 2, 1)],
          "prism": [(0, 1, 2), (3, 4, 5), (0, 1, 4, 3), (1, 2, 5, 4), (2, 0, 3, 5)]}


def _sizes(case):
    """Lattice sizes of each realisation of the case."""
    dims = (case["nx"], case["ny"], case["nz"])
    if case["call"] != "batch":
        return [dims]
    rng = random.Random("%d realisations up to %d" % (case["count"], dims[0]))
    return [dims] + [(n, n, n) for n in (rng.randint(min(16, dims[0]), dims[0]) for _ in range(case["count"] - 1))]


def _rectangles(kind, dims, n_frac, rng):
    """(axis, plane, low and high corner in lattice indices) of each fracture; vertical ones in a prism mesh."""
    out = []
    for _ in range(n_frac):
        axis = rng.randrange(2 if kind == "prism" else 3)
        lo, hi = [0, 0, 0], list(dims)
        plane = rng.randint(1, dims[axis] - 1)
        lo[axis] = hi[axis] = plane
        for a in range(3):
            if a != axis and not (kind == "prism" and a == 2):
                length = max(2, round(rng.uniform(0.1, 0.6) * dims[a]))
                lo[a] = rng.randint(0, dims[a] - length)
                hi[a] = lo[a] + length
        out.append((axis, lo, hi))
    return out


def _mesh(kind, dims, n_frac):
    """The lattice of one realisation: node indices and ids, cells, faces and fractures (no coordinates yet)."""
    nx, ny, nz = dims
    grid = torch.meshgrid(torch.arange(nz + 1, device=DEV), torch.arange(ny + 1, device=DEV),
                          torch.arange(nx + 1, device=DEV), indexing="ij")
    ijk = torch.stack([g.reshape(-1) for g in grid[::-1]], 1)
    corner = torch.tensor([i + (nx + 1) * (j + (ny + 1) * k) for i, j, k in _CUBE], device=DEV)
    inner = (ijk < torch.tensor(dims, device=DEV)).all(1)
    base = torch.arange(ijk.shape[0], device=DEV)[inner]
    cut = torch.tensor(_CUT[kind], device=DEV)
    cells = (base[:, None, None] + corner[cut]).reshape(-1, cut.shape[1])
    # every face of the mesh once, keyed by its three smallest nodes
    local = torch.tensor([f + (-1,) * (4 - len(f)) for f in _FACES[kind]], device=DEV)
    every = torch.where(local >= 0, cells[:, local.clamp(min=0)], -1).reshape(-1, 4)
    low = torch.where(every < 0, 1 << 40, every).sort(1).values
    key = (low[:, 0] << 40) + ((low[:, 1] - low[:, 0]) << 20) + (low[:, 2] - low[:, 0])
    uniq, face_of = torch.unique(key, return_inverse=True)
    first = torch.full((uniq.numel(),), key.numel(), device=DEV)
    first.scatter_reduce_(0, face_of, torch.arange(key.numel(), device=DEV), "amin")
    faces = every[first]
    at = ijk[torch.where(faces < 0, faces[:, :1], faces)]
    fmin, fmax = at.amin(1), at.amax(1)

    def inside(axis, lo, hi):
        return ((fmin >= torch.tensor(lo, device=DEV)) & (fmax <= torch.tensor(hi, device=DEV))).all(1)

    rng = random.Random("%s %s %d" % (kind, tuple(dims), n_frac))
    rects = _rectangles(kind, dims, n_frac, rng)
    on = torch.zeros(faces.shape[0], dtype=torch.bool, device=DEV)
    frozen = torch.zeros_like(ijk, dtype=torch.bool)   # coordinates that keep a fracture planar
    for axis, lo, hi in rects:
        hit = inside(axis, lo, hi)
        on |= hit
        frozen[faces[hit].clamp(min=0).reshape(-1).unique(), axis] = True
    sides = (ijk == 0) | (ijk == torch.tensor(dims, device=DEV))
    frozen |= (sides[:, :2] if kind == "prism" else sides).any(1, keepdim=True)
    ff = on.nonzero().reshape(-1)
    wells = []
    if kind == "prism":   # each well perforates the central layers of one column of fracture faces
        for axis, lo, hi in rects[:1] + rects[-1:]:
            other = 1 - axis
            for m in (lo[other], hi[other] - 1):
                l, h = list(lo), list(hi)
                l[other], h[other], l[2], h[2] = m, m + 1, dims[2] // 4, dims[2] - dims[2] // 4
                wells.append(inside(axis, l, h)[ff].nonzero().reshape(-1))
    return {"kind": kind, "dims": dims, "ijk": ijk, "cells": cells, "faces": faces, "frozen": frozen, "ff": ff,
            "cell_faces": face_of.reshape(cells.shape[0], -1), "wells": wells}


def _fields(mesh, ratio, gen):
    """Coordinates and physical data on a mesh, drawn from gen, as the interface takes them."""
    dims = torch.tensor(mesh["dims"], device=DEV, dtype=torch.float64)
    prism = mesh["kind"] == "prism"
    size = torch.tensor([600.0, 400.0, 60.0] if prism else [1.0, 1.0, 1.0], device=DEV, dtype=torch.float64)
    ijk = mesh["ijk"].double()
    d = torch.rand(ijk.shape, generator=gen, device=DEV, dtype=torch.float64) * 0.4 - 0.2
    d[mesh["frozen"]] = 0.0
    if prism:
        d[:, 2] = 0.0   # plane layers
        plan = (mesh["dims"][0] + 1) * (mesh["dims"][1] + 1)
        d[:, :2] = d[:plan, :2].repeat(mesh["dims"][2] + 1, 1)   # vertical edges
        d[mesh["frozen"]] = 0.0
    xyz = (ijk + d) / dims * size
    n_cells, n_ff = mesh["cells"].shape[0], mesh["ff"].numel()
    k = 10.0 ** (torch.randn(n_cells, generator=gen, device=DEV, dtype=torch.float64) * (0.3 if prism else 1.0))
    a = torch.randn(3, generator=gen, device=DEV, dtype=torch.float64)
    a = a / a.norm()
    t = 0.0 if prism else 9.0
    unit = 1e-15 if prism else 1.0
    i, j = torch.tensor([0, 1, 2, 0, 0, 1], device=DEV), torch.tensor([0, 1, 2, 1, 2, 2], device=DEV)
    lam = unit * k[:, None] * ((i == j).double() + t * a[i] * a[j])
    dn = torch.nonzero((mesh["ijk"][:, 0] == 0) | (mesh["ijk"][:, 0] == mesh["dims"][0])).reshape(-1)
    if prism:
        dn = dn[:0]
    f = {"xyz": xyz, "lambda_m": lam.contiguous(), "mu": 1e-3 if prism else 1.0,
         "lambda_f": torch.full((n_ff,), ratio * unit, device=DEV, dtype=torch.float64),
         "d_f": torch.full((n_ff,), 1.0 if prism else 1e-2, device=DEV, dtype=torch.float64),
         "dir_nodes": dn.int(), "dir_values": 1.0 - xyz[dn, 0], "cbar": (mesh["ijk"][dn, 0] == 0).double(),
         "phi_m": torch.full((n_cells,), 0.1 if prism else 0.2, device=DEV, dtype=torch.float64),
         "phi_f": torch.full((n_ff,), 0.1 if prism else 0.4, device=DEV, dtype=torch.float64)}
    if prism:   # the first well injects at a given rate, the others produce at pressure 0
        perf = torch.cat(mesh["wells"])
        which = torch.cat([torch.full_like(w, q) for q, w in enumerate(mesh["wells"])])
        perf, keep = np.unique(perf.cpu().numpy(), return_index=True)
        injects = (which.cpu().numpy()[keep] == 0)
        q = mesh["dims"]
        wi = vag.peaceman_wi(np.full(perf.size, 600.0 / q[0]), 60.0 / q[2], 1.0, ratio * unit, 0.1, f["mu"])
        f["wells"] = {"ff": perf.astype(np.int32), "wi": np.where(injects, 0.0, wi), "pw": np.zeros(perf.size),
                      "q": np.where(injects, 1e-4 / max(1, injects.sum()), 0.0), "cin": injects.astype(np.float64)}
    return f


def _problem(case, seed, which=0, fresh=0):
    """Mesh and fields of realisation `which`; fresh > 0: other permeabilities on the same mesh."""
    kind = case["cells"]
    mesh = _mesh(kind, _sizes(case)[which], case["fractures"])
    gen = torch.Generator(device=DEV)
    fields = _fields(mesh, case["ratio"], gen.manual_seed(1000003 * int(seed) + 131 * which))
    if fresh:
        other = _fields(mesh, case["ratio"], gen.manual_seed(1000003 * int(seed) + 131 * which + fresh))
        fields["lambda_m"], fields["lambda_f"] = other["lambda_m"], 2.0 * other["lambda_f"]
    return mesh, fields


def _arguments(mesh, f, mem):
    """The arrays of Context.assemble or Context.assemble_general, on the host or on the device."""
    q = {k: f[k] for k in ("lambda_m", "lambda_f", "d_f", "dir_nodes", "dir_values")}
    q["xyz"], q["lambda_m"] = f["xyz"].reshape(-1), f["lambda_m"].reshape(-1)
    if mesh["kind"] == "hex":
        q["cell_nodes"] = mesh["cells"].int().reshape(-1)
        q["ff_nodes"] = mesh["faces"][mesh["ff"]].int().reshape(-1)
    else:
        used = mesh["faces"] >= 0
        q["face_node_ptr"] = torch.nn.functional.pad(used.sum(1).cumsum(0), (1, 0)).int()
        q["face_node_idx"] = mesh["faces"][used].int()
        n, per = mesh["cell_faces"].shape
        q["cell_face_ptr"] = (torch.arange(n + 1, device=DEV) * per).int()
        q["cell_face_idx"] = mesh["cell_faces"].int().reshape(-1)
        q["ff_face_ids"] = mesh["ff"].int()
    if "wells" in f:
        q["wells"] = {k: torch.from_numpy(v).to(DEV) for k, v in f["wells"].items()}
    q = {k: v.contiguous() if torch.is_tensor(v) else v for k, v in q.items()}
    if mem == "host":
        q = {k: ({a: b.cpu().numpy() for a, b in v.items()} if isinstance(v, dict) else v.cpu().numpy())
             for k, v in q.items()}
    q["mu"] = f["mu"]
    return q


# ----------------------------------------------------------------------------
# what a user's program holds, and one pass
# ----------------------------------------------------------------------------

class _State:
    """A context on the caller's stream, the inputs of a call, and what the call keeps between passes."""

    def __init__(self, case, seed):
        self.case = case
        self.stream = torch.cuda.Stream()
        self.ctx = vag.Context(0)
        self.ctx.set_stream(self.stream.cuda_stream)
        parts = [_problem(case, seed, w) for w in range(len(_sizes(case)))]
        self.problems = [_arguments(m, f, case["mem"]) for m, f in parts]
        union = {k: torch.cat([f[k] for _, f in parts]) for k in ("phi_m", "phi_f", "cbar")}
        # initial concentration: cbar on the Dirichlet nodes, 0 elsewhere
        starts = np.cumsum([0] + [f["xyz"].shape[0] for _, f in parts])
        dn = torch.cat([f["dir_nodes"].long() + int(s) for s, (_, f) in zip(starts, parts)])
        self.n_cv = int(starts[-1]) + union["phi_m"].numel() + union["phi_f"].numel()
        union["c0"] = torch.zeros(self.n_cv, device=DEV, dtype=torch.float64)
        union["c0"][dn] = union["cbar"]
        self.union = {k: v.cpu().numpy() for k, v in union.items()} if case["mem"] == "host" else union
        self.how = {"precision": PRECISION[case["precision"]], "precond": PRECOND[case["precond"]],
                    "krylov": KRYLOV[case["krylov"]], "rtol": RTOL}
        self.system = None
        torch.cuda.synchronize()   # the inputs are ready before the context's stream reads them
        if case["call"] == "resample":
            self.system = self.assemble()
            f = _problem(case, seed, fresh=1)[1]
            self.new = {"lambda_m": f["lambda_m"].reshape(-1).contiguous(), "lambda_f": f["lambda_f"],
                        "d_f": f["d_f"], "mu": f["mu"], "wells": self.problems[0].get("wells")}
        elif case["call"] == "transport":
            self.system = self.assemble()
            self.system.solve(out=torch.empty(self.n_cv, device=DEV, dtype=torch.float64), **self.how)
        elif case["call"] == "product":
            self.system = self.assemble()
            gen = torch.Generator(device=DEV).manual_seed(int(seed))
            self.x = torch.randn(self.system.info().n_rows, generator=gen, device=DEV, dtype=torch.float64)
        torch.cuda.synchronize()

    def assemble(self):
        if self.case["call"] == "batch":
            return self.ctx.assemble_batch(self.problems)
        p = self.problems[0]
        return (self.ctx.assemble if self.case["cells"] == "hex" else self.ctx.assemble_general)(**p)

    def vector(self):
        return (np.empty(self.n_cv) if self.case["mem"] == "host"
                else torch.empty(self.n_cv, device=DEV, dtype=torch.float64))

    def concentration(self):
        c0 = self.union["c0"]
        return c0.copy() if self.case["mem"] == "host" else c0.clone()

    def move(self, system):
        c = self.concentration()
        system.transport(c, self.union["phi_m"], self.union["phi_f"], self.union["cbar"], self.case["steps"], cfl=0.9)
        return c


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    call = state.case["call"]
    with torch.cuda.stream(state.stream):
        if call in ("simulate", "batch"):
            system = state.assemble()
            u, _ = system.solve(out=state.vector(), **state.how)
            c = state.move(system)
            system.close()
            return {"u": u, "c": c}
        if call == "resample":
            state.system.update_props(**state.new)
            u, _ = state.system.solve(out=state.vector(), **state.how)
            return {"u": u}
        if call == "transport":
            return {"c": state.move(state.system)}
        return {"y": state.system.spmv(state.x, torch.empty_like(state.x))}


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------

def _counts(case):
    """Nodes, cells, fracture faces (about) and cell-node pairs of all realisations."""
    nv = nc = nf = pairs = 0
    for nx, ny, nz in _sizes(case):
        cut = _CUT[case["cells"]]
        nv += (nx + 1) * (ny + 1) * (nz + 1)
        nc += len(cut) * nx * ny * nz
        pairs += len(cut) * len(cut[0]) * nx * ny * nz
        for axis, lo, hi in _rectangles(case["cells"], (nx, ny, nz), case["fractures"],
                                        random.Random("%s %s %d" % (case["cells"], (nx, ny, nz), case["fractures"]))):
            area = math.prod(hi[a] - lo[a] for a in range(3) if a != axis)
            nf += area * (2 if case["cells"] == "tet" else 1)
    return nv, nc, nf, pairs


def work(case):
    """Every input read once and every output written once; the flops of the local matrices, of one product with the
    eliminated matrix (how many a solver takes is its own affair) and of the transport steps."""
    nv, nc, nf, pairs = _counts(case)
    n_cv = nv + nc + nf
    rows = nv + nf
    nnz = 27 * nv * (1 if case["cells"] == "hex" else 0.6) + 20 * nf
    tets = {"hex": 24, "tet": 12, "prism": 18}[case["cells"]]
    fields = 48 * nc + 16 * nf
    mesh = 24 * nv + 4 * pairs + 16 * nf
    local = nc * tets * 100
    steps = case["steps"]
    if case["call"] == "product":
        return {"bytes": 12 * nnz + 16 * rows, "flops": 2 * nnz}
    if case["call"] == "resample":
        return {"bytes": fields + mesh + 8 * n_cv, "flops": local + 2 * nnz}
    moved = 8 * (nc + nf) + 16 * n_cv
    flow = steps * (2 * (pairs + 6 * nf) + n_cv)
    if case["call"] == "transport":
        return {"bytes": moved + 8 * (pairs + 6 * nf), "flops": flow}
    return {"bytes": fields + mesh + 8 * n_cv + moved, "flops": local + 2 * nnz + flow}


# ----------------------------------------------------------------------------
# the same results from the definitions, in plain torch
# ----------------------------------------------------------------------------

def _cell_matrices(mesh, f):
    """[n_cells, m, m] over (centre, nodes, faces), P1 on the tetrahedra (centre, face centre, edge of the face), and
    the cell volumes; faces that carry no fracture are interpolated from their nodes."""
    nodes = mesh["cells"]
    nc, nn = nodes.shape
    table = _FACES[mesh["kind"]]
    m = 1 + nn + len(table)
    x = f["xyz"][nodes]
    centre = x.mean(1)
    lam = f["lambda_m"].reshape(nc, 6)[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].reshape(nc, 3, 3) / f["mu"]
    M = torch.zeros(nc, m, m, device=DEV, dtype=torch.float64)
    vol = torch.zeros(nc, device=DEV, dtype=torch.float64)
    for lf, face in enumerate(table):
        xs = x[:, list(face)].mean(1)
        for a, b in zip(face, face[1:] + face[:1]):
            e = [xs - centre, x[:, a] - centre, x[:, b] - centre]
            n = [torch.linalg.cross(e[1], e[2]), torch.linalg.cross(e[2], e[0]), torch.linalg.cross(e[0], e[1])]
            det = (e[0] * n[0]).sum(1)
            G = torch.stack([-(n[0] + n[1] + n[2])] + n, 1) / det[:, None, None]
            S = G @ lam @ G.transpose(1, 2) * (det.abs() / 6)[:, None, None]
            at = torch.tensor([0, 1 + nn + lf, 1 + a, 1 + b], device=DEV)
            M[:, at[:, None], at[None, :]] += S
            vol += det.abs() / 6
    fracture = torch.full((mesh["faces"].shape[0],), -1, device=DEV)
    fracture[mesh["ff"]] = torch.arange(mesh["ff"].numel(), device=DEV)
    ff = fracture[mesh["cell_faces"]]
    for lf, face in enumerate(table):
        s, q = 1 + nn + lf, [1 + a for a in face]
        plain = (ff[:, lf] < 0).double()
        w = (plain / len(face))[:, None]
        for a in q:
            M[:, a] += w * M[:, s]
        for a in q:
            M[:, :, a] += w * M[:, :, s]
        M[:, s] *= 1 - plain[:, None]
        M[:, :, s] *= 1 - plain[:, None]
    return M, vol, ff


def _fracture_matrices(mesh, f):
    """[n_ff, 5, 5] over (face, nodes), tangential P1 on the triangles (face centre, edge), the areas and the nodes."""
    nodes = mesh["faces"][mesh["ff"]]
    size = (nodes >= 0).sum(1)
    x = f["xyz"][nodes.clamp(min=0)] * (nodes >= 0)[..., None]
    xs = x.sum(1) / size[:, None]
    M = torch.zeros(nodes.shape[0], 5, 5, device=DEV, dtype=torch.float64)
    area = torch.zeros(nodes.shape[0], device=DEV, dtype=torch.float64)
    for q in (3, 4):
        pick = (size == q).nonzero().reshape(-1)
        for t in range(q):
            u = (t + 1) % q
            a, b, s = x[pick, t], x[pick, u], xs[pick]
            A = torch.linalg.cross(a - s, b - s).norm(dim=1) / 2
            E = torch.stack([b - a, s - b, a - s], 1)
            S = E @ E.transpose(1, 2) * (f["d_f"][pick] * f["lambda_f"][pick] / f["mu"] / (4 * A))[:, None, None]
            at = [0, 1 + t, 1 + u]
            for i in range(3):
                for j in range(3):
                    M[pick, at[i], at[j]] += S[:, i, j]
            area[pick] += A
    return M, area, nodes


def _coo(parts, n):
    """Sum of (rows, columns, values) triples as an n x n CSR matrix."""
    i = torch.cat([p[0].reshape(-1) for p in parts])
    j = torch.cat([p[1].reshape(-1) for p in parts])
    v = torch.cat([p[2].reshape(-1) for p in parts])
    keep = (i >= 0) & (j >= 0)
    return torch.sparse_coo_tensor(torch.stack([i[keep], j[keep]]), v[keep], (n, n)).coalesce().to_sparse_csr()


def _cg(A, diag, b, rounds=4, most=20000):
    """Jacobi-CG, restarted from the true residual, until it no longer falls."""
    x = torch.zeros_like(b)
    best, res = x, math.inf
    for _ in range(rounds):
        r = b - A @ x
        if float(r.norm()) >= 0.5 * res:
            break
        best, res = x.clone(), float(r.norm())
        z = r / diag
        p, rz = z, r @ z
        for k in range(most):
            q = A @ p
            alpha = rz / (p @ q)
            x = x + alpha * p
            r = r - alpha * q
            z = r / diag
            new = r @ z
            p, rz = z + (new / rz) * p, new
            if k % 50 == 49 and float(r.norm()) <= 1e-15 * float(b.norm()):
                break
    r = b - A @ x
    return x if float(r.norm()) < res else best


def _exact_one(case, mesh, f):
    """(pressure blocks, concentration blocks), each (nodes, fracture faces, cells), and the eliminated matrix with its
    row order."""
    nodes = mesh["cells"]
    nc, nn = nodes.shape
    nv, nf = f["xyz"].shape[0], mesh["ff"].numel()
    M, vol, ff = _cell_matrices(mesh, f)
    Mf, area, fn = _fracture_matrices(mesh, f)
    dof = torch.cat([nodes, torch.where(ff >= 0, nv + ff, -1)], 1)
    fdof = torch.cat([nv + torch.arange(nf, device=DEV)[:, None], fn], 1)
    # eliminate the cell centres
    B, b0, kk = M[:, 1:, 1:], M[:, 1:, 0], M[:, 0, 0]
    S = B - b0[:, :, None] * b0[:, None, :] / kk[:, None, None]
    dn = f["dir_nodes"].long()
    free = torch.ones(nv + nf, dtype=torch.bool, device=DEV)
    free[dn] = False
    parts = [(dof[:, :, None].expand_as(S), dof[:, None, :].expand_as(S), S),
             (fdof[:, :, None].expand_as(Mf), fdof[:, None, :].expand_as(Mf), Mf)]
    u = torch.zeros(nv + nf, device=DEV, dtype=torch.float64)
    u[dn] = f["dir_values"]
    rhs = torch.zeros_like(u)
    wells = f.get("wells")
    if wells is not None:
        w = {k: torch.from_numpy(v).to(DEV) for k, v in wells.items()}
        wf = w["ff"].long()
        parts.append((nv + wf, nv + wf, w["wi"]))
        rhs[nv + wf] = w["wi"] * w["pw"] + w["q"]
    row = torch.where(free, free.long().cumsum(0) - 1, -1)
    n = int(free.sum())
    A = _coo([(torch.where(i >= 0, row[i], -1), torch.where(j >= 0, row[j], -1), v) for i, j, v in parts], n)
    for i, j, v in parts[:2]:   # the Dirichlet columns
        known = (i >= 0) & (j >= 0) & ~free[j.clamp(min=0)]
        rhs.index_add_(0, i[known], -v[known] * u[j[known]])
    if case["call"] == "product":
        return None, None, A
    idx = torch.arange(n, device=DEV)
    ones = torch.zeros(n, device=DEV, dtype=torch.float64)
    crow, col, val = A.crow_indices(), A.col_indices(), A.values()
    own = torch.repeat_interleave(idx, crow[1:] - crow[:-1]) == col
    ones[col[own]] = val[own]
    u[free] = _cg(A, ones, rhs[free])
    del A, crow, col, val, own
    at = torch.where(dof >= 0, u[dof.clamp(min=0)], 0.0)
    uK = -(b0 * at).sum(1) / kk
    pressure = (u[:nv], u[nv:], uK)
    if not case["steps"]:
        return pressure, None, None
    # fluxes from cells and from fracture faces, and the wells' rates
    F = (B @ torch.where(dof >= 0, uK[:, None] - at, 0.0)[:, :, None])[:, :, 0]
    uf = torch.where(fn >= 0, u[nv:, None] - u[fn.clamp(min=0)], 0.0)
    Ff = (Mf[:, 1:, 1:] @ uf[:, :, None])[:, :, 0]
    src = torch.cat([(nv + nf + torch.arange(nc, device=DEV))[:, None].expand_as(dof)[dof >= 0],
                     (nv + torch.arange(nf, device=DEV))[:, None].expand_as(fn)[fn >= 0]])
    dst = torch.cat([dof[dof >= 0], fn[fn >= 0]])
    flux = torch.cat([F[dof >= 0], Ff[fn >= 0]])
    n_cv = nv + nf + nc
    omega = 0.5
    isdir = torch.zeros(nv, dtype=torch.bool, device=DEV)
    isdir[dn] = True
    onfrac = torch.zeros(nv, dtype=torch.bool, device=DEV)
    onfrac[fn[fn >= 0]] = True
    phi = torch.zeros(n_cv, device=DEV, dtype=torch.float64)
    pore, fpore = vol * f["phi_m"], area * f["d_f"] * f["phi_f"]
    give = (~isdir & ~onfrac)[nodes].double() * (omega / nn * pore)[:, None]
    phi.index_add_(0, nodes.reshape(-1), give.reshape(-1))
    phi[nv + nf:] = pore - give.sum(1)
    fsize = (fn >= 0).sum(1)
    fgive = ((fn >= 0) & ~isdir[fn.clamp(min=0)]).double() * (omega / fsize * fpore)[:, None]
    phi.index_add_(0, fn.clamp(min=0).reshape(-1), fgive.reshape(-1))
    phi[nv:nv + nf] = fpore - fgive.sum(1)
    out = torch.zeros(n_cv, device=DEV, dtype=torch.float64)
    forth, back = flux > 0, flux < 0
    out.index_add_(0, src[forth], flux[forth])
    out.index_add_(0, dst[back], -flux[back])
    given = torch.zeros(n_cv, device=DEV, dtype=torch.float64)   # injected concentration x rate
    if wells is not None:
        rate = w["wi"] * (u[nv + wf] - w["pw"]) - w["q"]
        out.index_add_(0, nv + wf, rate.clamp(min=0))
        given.index_add_(0, nv + wf, (-rate).clamp(min=0) * w["cin"])
    moves = torch.cat([~isdir, torch.ones(nf + nc, dtype=torch.bool, device=DEV)])
    bound = torch.where(moves & (out > 0), phi / out.clamp(min=1e-300), math.inf)
    h = 0.9 * bound.min() / torch.where(moves, phi, 1.0) * moves
    diag = torch.arange(n_cv, device=DEV)
    W = _coo([(diag, diag, 1 - h * out), (dst[forth], src[forth], h[dst[forth]] * flux[forth]),
              (src[back], dst[back], -h[src[back]] * flux[back])], n_cv)
    c = torch.zeros(n_cv, device=DEV, dtype=torch.float64)
    c[dn] = f["cbar"]
    given = given * h
    for _ in range(case["steps"]):
        c = W @ c + given
    return pressure, (c[:nv], c[nv:nv + nf], c[nv + nf:]), None


def exact(case, seed):
    sizes = _sizes(case)
    fresh = 1 if case["call"] == "resample" else 0
    got = [_exact_one(case, *_problem(case, seed, w, fresh)) for w in range(len(sizes))]
    if case["call"] == "product":
        A = got[0][2]
        x = torch.randn(A.shape[0], generator=torch.Generator(device=DEV).manual_seed(int(seed)), device=DEV,
                        dtype=torch.float64)
        return {"y": A @ x}
    u, c = (None if got[0][k] is None else torch.cat([torch.cat([g[k][b] for g in got]) for b in range(3)])
            for k in (0, 1))
    if case["call"] == "transport":
        return {"c": c}
    if case["call"] == "resample":
        return {"u": u}
    return {"u": u, "c": c}
