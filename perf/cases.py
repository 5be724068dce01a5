"""The work that a user of the assembly engine has it do, as measurable cases.

A case is a dict of plain values; ``prepare`` makes what a program holds before
the call (mesh handle, pattern, buffers, operator), ``run`` is one pass through
the public entry points of ``paper_1805_03949_gb300.fea``, ``work`` the bytes
and operations the pass cannot do without, and ``exact`` its result in 64-bit
torch arithmetic that shares no code with the engine.

Meshes are jittered boxes built on the GPU: hexahedra, Kuhn tetrahedra, and
cells of the four element types in zones (the shapes of the engine's own
synthetic workloads).  Everything random comes from the seed.
"""
import math

import torch

from paper_1805_03949_gb300 import fea

TET, PYR, PRISM, HEX = 0, 1, 2, 3
NN = (4, 5, 6, 8)
DEV = "cuda"
F64 = torch.float64

# material of the elastoplastic and hyperelastic solids (the engine's defaults)
YOUNG, POISSON = 1.0, 0.3
SIGMA0, SIGMA_INF, DELTA, HARDENING = 1e-3, 3e-3, 300.0, 1e-2
# nodal displacement amplitudes: about 30 % of the Gauss points yield / strains of a few percent
J2_AMPLITUDE, NH_AMPLITUDE = 2.2722e-5, 4e-4


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a small scalar problem (24,576 elements), where latency and launches count
        _assembly("poisson_tet_16_fp64", "tet", 16, "diffusion", tet_rule=0),
        # the operator's defaults (FP64, atomic scatter) on a tetrahedral mechanics mesh
        _assembly("elasticity_tet_30_fp64", "tet", 30, "elasticity"),
        # the same on hexahedra: the plain method that every variant is compared with
        _assembly("elasticity_hex_63_fp64", "hex", 63, "elasticity"),
        # the large mechanics mesh in the mixed-precision block-task variant (2.1 M elements, 4.1 GB of A)
        _assembly("elasticity_hex_128_fp32_block", "hex", 128, "elasticity", precision="fp32", scatter="block"),
        # four element types in one work-stealing launch, mixed precision, k = 1 + x^2
        _assembly("diffusion_mixed_70_fp32_steal", "mixed", 70, "diffusion", precision="fp32", schedule="steal", k2=1.0),
        # the same kind of mesh, one FP64 launch per element type
        _assembly("diffusion_mixed_45_fp64", "mixed", 45, "diffusion", k2=1.0),
        # a Newton step of the elastoplastic solid: tangent, internal force and new state
        _assembly("j2_hex_72_fp32", "hex", 72, "j2", precision="fp32"),
        # its element loop alone: state and stress at every Gauss point, no scatter
        {"name": "j2_points_hex_80", "path": "points", "mesh": "hex", "n": 80},
        # a Newton step of the finite-strain solid with its inertia term
        _assembly("neohooke_hex_41_fp64", "hex", 41, "neohooke", mass=0.5),
        # many small and medium systems at once (serving): one captured launch
        {"name": "batch_64_fp32", "path": "batch", "count": 64, "lo": 1000, "hi": 60000, "precision": "fp32"},
        # a new mesh: upload, CSR pattern and element-to-nonzero map
        {"name": "pattern_mixed_45", "path": "pattern", "mesh": "mixed", "n": 45, "ndof": 3},
        # the product with the assembled matrix that follows in a Krylov solver
        {"name": "spmv_hex_96", "path": "spmv", "mesh": "hex", "n": 96, "ndof": 3},
    ]


def _assembly(name, mesh, n, op, precision="fp64", scatter="atomic", schedule="per_type", tet_rule=1, k2=0.0, mass=0.0):
    return {"name": name, "path": "assembly", "mesh": mesh, "n": n, "op": op, "precision": precision,
            "scatter": scatter, "schedule": schedule, "tet_rule": tet_rule, "k2": k2, "mass": mass}


# cells per axis: smallest and largest drawn, by mesh; the larger end is for the light operators
_RANGE = {"hex": (6, 96), "tet": (5, 40), "mixed": (5, 60)}


def _draw_n(rng, mesh, top=None):
    lo, hi = _RANGE[mesh]
    hi = min(hi, top or hi)
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["assembly"] * 8 + ["points", "batch", "pattern", "spmv"])
    if path == "points":
        mesh = rng.choice(["hex", "hex", "tet", "mixed"])
        return {"path": path, "mesh": mesh, "n": _draw_n(rng, mesh, 80)}
    if path == "batch":
        return {"path": path, "count": rng.randint(8, 64), "lo": rng.randint(500, 3000),
                "hi": int(round(math.exp(rng.uniform(math.log(6e3), math.log(6e4))))),
                "precision": rng.choice(["fp32", "fp32", "fp64"])}
    if path == "pattern":
        mesh = rng.choice(["hex", "tet", "mixed"])
        return {"path": path, "mesh": mesh, "n": _draw_n(rng, mesh, 64), "ndof": rng.choice([1, 3])}
    if path == "spmv":
        mesh = rng.choice(["hex", "tet", "mixed"])
        return {"path": path, "mesh": mesh, "n": _draw_n(rng, mesh), "ndof": rng.choice([1, 3])}
    op = rng.choice(["diffusion", "diffusion", "elasticity", "elasticity", "elasticity", "j2", "neohooke"])
    mesh = rng.choice(["hex", "hex", "tet", "mixed"])
    precision = rng.choice(["fp64", "fp32"])
    scatter, schedule = "atomic", "per_type"
    if op in ("diffusion", "elasticity"):
        scatter = rng.choice(["atomic", "atomic", "block", "rows"])
    if scatter == "atomic" and op != "neohooke":
        schedule = rng.choice(["per_type", "per_type", "steal"])
    top = 60 if precision == "fp64" or op in ("j2", "neohooke") else None
    if op in ("j2", "neohooke") and precision == "fp64":
        top = 44
    c = _assembly(None, mesh, _draw_n(rng, mesh, top), op, precision, scatter, schedule,
                  tet_rule=rng.choice([0, 1]), k2=rng.choice([0.0, 1.0]) if op == "diffusion" else 0.0,
                  mass=rng.choice([0.0, 0.5]) if op == "neohooke" else 0.0)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# meshes, on the GPU
# ---------------------------------------------------------------------------
class Mesh:
    """coords [N, 3], types [E], conn_offsets [E + 1], conn: CUDA tensors, and the connectivity per type."""

    def __init__(self, coords, groups, n_elems):
        # groups: {type: (element ids, connectivity [n, nn])}
        self.coords, self.groups = coords, groups
        self.types = torch.empty(n_elems, dtype=torch.uint8, device=DEV)
        nn = torch.empty(n_elems, dtype=torch.int64, device=DEV)
        for t, (ids, _) in groups.items():
            self.types[ids] = t
            nn[ids] = NN[t]
        self.conn_offsets = torch.zeros(n_elems + 1, dtype=torch.int64, device=DEV)
        torch.cumsum(nn, 0, out=self.conn_offsets[1:])
        self.conn = torch.empty(sum(c.numel() for _, c in groups.values()), dtype=torch.int32, device=DEV)
        for t, (ids, c) in groups.items():
            at = self.conn_offsets[ids][:, None] + torch.arange(NN[t], device=DEV)
            self.conn[at.reshape(-1)] = c.reshape(-1).to(torch.int32)

    @property
    def n_nodes(self):
        return self.coords.shape[0]

    @property
    def n_elems(self):
        return self.types.shape[0]


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _kuhn():
    """The 6 tetrahedra of a cell that share its main diagonal, positively oriented."""
    out = []
    for a, b, odd in ((0, 1, 0), (0, 2, 1), (1, 0, 1), (1, 2, 0), (2, 0, 0), (2, 1, 1)):
        p = [[0, 0, 0], [0, 0, 0], [0, 0, 0], [1, 1, 1]]
        p[1][a] = p[2][a] = p[2][b] = 1
        out.append([p[0], p[1], p[3], p[2]] if odd else p)
    return out


_CORNERS = [(0, 0, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1), (1, 1, 1), (0, 1, 1)]


def _templates():
    """Elements of one cell in half-cell units, by type: 6 tets, 6 pyramids with the centre as apex, 2 prisms, 8 hexes."""
    tets = [[[2 * v for v in p] for p in t] for t in _kuhn()]
    faces = [[0, 1, 2, 3], [4, 7, 6, 5], [0, 3, 7, 4], [1, 5, 6, 2], [0, 4, 5, 1], [3, 2, 6, 7]]
    pyrs = [[[2 * v for v in _CORNERS[k]] for k in f] + [[1, 1, 1]] for f in faces]
    tris = [[(0, 0), (2, 0), (2, 2)], [(0, 0), (2, 2), (0, 2)]]
    prisms = [[[x, y, z] for z in (0, 2) for x, y in t] for t in tris]
    hexes = [[[o[0] + c[0], o[1] + c[1], o[2] + c[2]] for c in _CORNERS] for o in _CORNERS]
    return {TET: tets, PYR: pyrs, PRISM: prisms, HEX: hexes}


def _jittered(ijk, dims, g, amount):
    """Lattice positions in the unit cube, interior points moved by up to `amount` spacings per axis."""
    d = torch.tensor(dims, dtype=F64, device=DEV)
    move = (2.0 * torch.rand(ijk.shape, generator=g, dtype=F64, device=DEV) - 1.0) * amount
    inside = ((ijk > 0) & (ijk < d)).all(1, keepdim=True)
    return (ijk + torch.where(inside, move, torch.zeros_like(move))) / d


def _box(etype, nx, ny, nz, g):
    """A box of nx ny nz cells, one hexahedron or six tetrahedra each."""
    k, j, i = torch.meshgrid(*(torch.arange(n + 1, device=DEV) for n in (nz, ny, nx)), indexing="ij")
    ijk = torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)], 1).to(F64)
    coords = _jittered(ijk, (nx, ny, nz), g, 0.2 if etype == HEX else 0.1)
    k, j, i = torch.meshgrid(*(torch.arange(n, device=DEV) for n in (nz, ny, nx)), indexing="ij")
    off = torch.tensor([_CORNERS] if etype == HEX else _kuhn(), device=DEV)
    stride = torch.tensor([1, nx + 1, (nx + 1) * (ny + 1)], device=DEV)
    first = (i.reshape(-1) + stride[1] * j.reshape(-1) + stride[2] * k.reshape(-1))[:, None, None]
    conn = (first + (off * stride).sum(2)).reshape(-1, NN[etype])
    return Mesh(coords, {etype: (torch.arange(len(conn), device=DEV), conn)}, len(conn))


def _mixed(n, g):
    """n^3 cells in zones of one element type each (40 / 10 / 20 / 30 % of the elements), cell by cell.

    The zones depend on n alone, so that every seed has the same pattern and work."""
    cells = n ** 3
    z = _generator(n)
    per = torch.tensor([6, 6, 2, 8], device=DEV)
    share = torch.tensor([0.4, 0.1, 0.2, 0.3], dtype=F64, device=DEV) / per
    bound = torch.round(torch.cumsum(share / share.sum(), 0) * cells).to(torch.int64)
    k, j, i = torch.meshgrid(*(torch.arange(n, device=DEV) for _ in range(3)), indexing="ij")
    c = torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)], 1)
    wave = torch.randint(1, 4, (6, 3), generator=z, device=DEV).to(F64)
    phase = 2 * math.pi * torch.rand(6, generator=z, dtype=F64, device=DEV)
    field = torch.sin(2 * math.pi * ((c + 0.5).to(F64) / n) @ wave.T + phase).sum(1)
    zone = torch.empty(cells, dtype=torch.int64, device=DEV)
    zone[torch.argsort(field, stable=True)] = torch.searchsorted(bound, torch.arange(cells, device=DEV), right=True).clamp(max=3)
    count = per[zone]
    first = torch.cumsum(count, 0) - count
    m = 2 * n + 1
    ids, fine = {}, {}
    for t, tmpl in _templates().items():
        cell = torch.nonzero(zone == t).reshape(-1)
        off = torch.tensor(tmpl, device=DEV)
        p = 2 * c[cell][:, None, None, :] + off
        fine[t] = (p[..., 0] + m * (p[..., 1] + m * p[..., 2])).reshape(-1, NN[t])
        ids[t] = (first[cell][:, None] + torch.arange(len(tmpl), device=DEV)).reshape(-1)
    used, inverse = torch.unique(torch.cat([fine[t].reshape(-1) for t in fine]), return_inverse=True)
    ijk = torch.stack([used % m, (used // m) % m, used // (m * m)], 1).to(F64)
    coords = _jittered(ijk, (2 * n, 2 * n, 2 * n), g, 0.1)
    groups, at = {}, 0
    for t in fine:
        if len(ids[t]):
            groups[t] = (ids[t], inverse[at:at + fine[t].numel()].reshape(-1, NN[t]))
        at += fine[t].numel()
    return Mesh(coords, groups, int(count.sum()))


def _make_mesh(case, g):
    n = case["n"]
    if case["mesh"] == "mixed":
        return _mixed(n, g)
    # ragged boxes: the number of elements is no multiple of a tile
    return _box(HEX if case["mesh"] == "hex" else TET, n, n, max(1, n - n % 3), g)


def _renumbered(mesh, g):
    """The mesh with its nodes numbered anew inside windows of 64, as meshers leave them: near in space, in no order."""
    at = torch.arange(mesh.n_nodes, device=DEV)
    order = torch.argsort(torch.div(at, 64, rounding_mode="floor") + torch.rand(len(at), generator=g, dtype=F64, device=DEV))
    new = torch.empty_like(order)
    new[order] = at
    return Mesh(mesh.coords[order], {t: (ids, new[c]) for t, (ids, c) in mesh.groups.items()}, mesh.n_elems)


def _displacement(coords, g, amplitude):
    """A smooth field: 8 sine modes with unit amplitude vectors."""
    k = torch.randint(1, 5, (8, 3), generator=g, device=DEV).to(F64)
    a = torch.randn((8, 3), generator=g, dtype=F64, device=DEV)
    a = a / a.norm(dim=1, keepdim=True)
    phase = 2 * math.pi * torch.rand(8, generator=g, dtype=F64, device=DEV)
    return amplitude * torch.sin(2 * math.pi * coords @ k.T + phase) @ a


def _inputs(case, seed):
    """Mesh, displacements and committed plastic state: the same tensors for the engine and for exact()."""
    g = _generator(seed)
    mesh = _make_mesh(case, g)
    kind = case.get("op", "j2" if case["path"] == "points" else None)
    u = state = None
    if kind in ("j2", "neohooke"):
        u = _displacement(mesh.coords, g, J2_AMPLITUDE if kind == "j2" else NH_AMPLITUDE)
    if kind == "j2":
        # committed by an earlier step at 70 % of the load, which a part of the points yielded in
        state = _points(mesh, 0.7 * u, torch.zeros((mesh.n_elems, 8, 7), dtype=F64, device=DEV))[0]
    return mesh, u, state


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
class State:
    """What a program holds; closes its handles when it goes."""

    def __init__(self, case):
        self.case, self.systems, self.batch = case, [], None

    def __del__(self):
        if self.batch is not None:
            self.batch.close()
        for s in self.systems:
            s.close()


_KIND = {"diffusion": fea.FEA_OP_DIFFUSION, "elasticity": fea.FEA_OP_ELASTICITY, "j2": fea.FEA_OP_J2,
         "neohooke": fea.FEA_OP_NEOHOOKE}
_PRECISION = {"fp64": fea.FEA_FP64, "fp32": fea.FEA_FP32_INTEGRATE}
_SCATTER = {"atomic": fea.FEA_SCATTER_ATOMIC, "block": fea.FEA_SCATTER_BLOCK, "rows": fea.FEA_SCATTER_ROWS}
_SCHEDULE = {"per_type": fea.FEA_SCHED_PER_TYPE, "steal": fea.FEA_SCHED_STEAL}


def prepare(case, seed):
    st = State(case)
    if case["path"] == "batch":
        return _prepare_batch(st, case, seed)
    mesh, u, state = _inputs(case, seed)
    if case["path"] == "pattern":
        st.mesh = _renumbered(mesh, _generator(seed + 1))
        return st
    st.u, st.state_in = u, state
    if case["path"] == "points":
        st.handle = fea.System(fea.fea_mesh_upload(mesh.coords, mesh.types, mesh.conn_offsets, mesh.conn), 3,
                               mesh.n_nodes, mesh.n_elems, None, None, None, None, None)
        st.systems.append(st.handle)
        st.state_out = torch.zeros_like(state)
        st.stress = torch.zeros((mesh.n_elems, 8, 6), dtype=F64, device=DEV)
        st.op = fea.make_operator(kind=fea.FEA_OP_J2, young=YOUNG, poisson=POISSON, u=u, state_in=state,
                                  state_out=st.state_out)
        return st
    ndof = case["ndof"] if case["path"] == "spmv" else 1 if case["op"] == "diffusion" else 3
    st.system = fea.System.from_mesh(mesh, ndof, with_cols=False)
    st.systems.append(st.system)
    if case["path"] == "spmv":
        op = fea.make_operator(kind=fea.FEA_OP_DIFFUSION if ndof == 1 else fea.FEA_OP_ELASTICITY, poisson=POISSON)
        st.system.assemble(op)
        st.x = torch.randn(st.system.b.shape, generator=_generator(seed + 1), dtype=F64, device=DEV)
        st.y = torch.empty_like(st.x)
        return st
    st.state_out = torch.zeros_like(state) if state is not None else None
    st.op = fea.make_operator(kind=_KIND[case["op"]], precision=_PRECISION[case["precision"]],
                              scatter=_SCATTER[case["scatter"]], schedule=_SCHEDULE[case["schedule"]],
                              tet_rule=case["tet_rule"], k0=1.0, k2=case["k2"], young=YOUNG, poisson=POISSON, u=u,
                              state_in=state, state_out=st.state_out, mass=case["mass"])
    return st


def _batch_boxes(case, seed):
    """(element type, nx, ny, nz) of every mesh: tets or hexes, sizes log-uniform in [lo, hi] elements."""
    g = torch.Generator()
    g.manual_seed(int(seed))
    # the sizes come from the case, the coordinates from the seed: every pass has the same work
    sizes = torch.Generator()
    sizes.manual_seed(case["count"] * 100003 + case["hi"])
    out = []
    for _ in range(case["count"]):
        r, k = torch.rand(2, generator=sizes, dtype=F64).tolist()
        want = math.exp(math.log(case["lo"]) + r * (math.log(case["hi"]) - math.log(case["lo"])))
        etype = TET if k < 0.5 else HEX
        cells = want / (6 if etype == TET else 1)
        n = max(1, round(cells ** (1 / 3)))
        out.append((etype, n, n, max(1, round(cells / (n * n)))))
    return out


def _batch_meshes(case, seed):
    return [_box(*box, _generator(seed * 1000 + i)) for i, box in enumerate(_batch_boxes(case, seed))]


def _prepare_batch(st, case, seed):
    meshes = _batch_meshes(case, seed)
    st.systems = [fea.System.from_mesh(m, 3, with_cols=False) for m in meshes]
    # one pool for all systems, each system's values on a 16-byte boundary
    at = [0]
    for s in st.systems:
        at += [at[-1] + s.A.numel() + (s.A.numel() & 1)]
    st.A = torch.zeros(at[-1], dtype=F64, device=DEV)
    bt = [0]
    for s in st.systems:
        bt += [bt[-1] + s.b.numel() + (s.b.numel() & 1)]
    st.b = torch.zeros(bt[-1], dtype=F64, device=DEV)
    for k, s in enumerate(st.systems):
        s.A = st.A[at[k]:at[k] + s.A.numel()]
        s.b = st.b[bt[k]:bt[k] + s.b.numel()]
    op = fea.make_operator(kind=fea.FEA_OP_ELASTICITY, precision=_PRECISION[case["precision"]], young=YOUNG,
                           poisson=POISSON, chunk=64)
    st.batch = fea.Batch(op, st.systems)
    st.batch.capture()
    return st


def run(st):
    path = st.case["path"]
    if path == "assembly":
        st.system.assemble(st.op)
        out = {"A": st.system.A, "b": st.system.b}
        if st.state_out is not None:
            out["state"] = st.state_out
        return out
    if path == "points":
        fea.fea_element_loop(st.op, st.handle.handle, st.stress)
        return {"state": st.state_out, "stress": st.stress}
    if path == "batch":
        st.batch.assemble()
        return {"A": st.A, "b": st.b}
    if path == "spmv":
        fea.fea_spmv(st.system.handle, st.case["ndof"], st.system.row_ptr, st.system.A, st.x, st.y)
        return {"y": st.y}
    s = fea.System.from_mesh(st.mesh, st.case["ndof"])
    out = {"row_ptr": s.row_ptr, "col_idx": s.col_idx, "node_map": s.node_map}
    s.close()
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _counts(case):
    """Elements by type, nodes and node-graph entries (closed forms; near ones for the mixed mesh)."""
    n = case["n"]
    m = max(1, n - n % 3)
    if case["mesh"] == "hex":
        return {HEX: n * n * m}, (n + 1) ** 2 * (m + 1), (3 * n + 1) ** 2 * (3 * m + 1)
    if case["mesh"] == "tet":
        return _tet_box(n, n, m)
    share = n ** 3 / (0.4 / 6 + 0.1 / 6 + 0.2 / 2 + 0.3 / 8)
    elems = {TET: round(0.4 * share), PYR: round(0.1 * share), PRISM: round(0.2 * share), HEX: round(0.3 * share)}
    cells = {TET: elems[TET] / 6, PYR: elems[PYR] / 6, PRISM: elems[PRISM] / 2, HEX: elems[HEX] / 8}
    nodes = cells[TET] + 2 * cells[PYR] + cells[PRISM] + 8 * cells[HEX]
    graph = 15 * cells[TET] + (23 + 9) * cells[PYR] + 21 * cells[PRISM] + 27 * 8 * cells[HEX]
    return elems, nodes, graph


def _tet_box(nx, ny, nz):
    px, py, pz = nx + 1, ny + 1, nz + 1
    edges = nx * py * pz + px * ny * pz + px * py * nz + nx * ny * pz + nx * py * nz + px * ny * nz + nx * ny * nz
    return {TET: 6 * nx * ny * nz}, px * py * pz, px * py * pz + 2 * edges


# operations per element: geometry and gradients per point, then the upper
# triangle of the element matrix (a linear tet needs one point's worth of both)
def _element_flops(t, op, tet_rule):
    nn, nq = NN[t], (1 if t == TET and op in ("diffusion", "elasticity") else 4 if t == TET else 6 if t == PRISM else 8)
    pairs = nn * (nn + 1) // 2
    geometry = 150 + 18 * (nn - 1)
    point = {"diffusion": 0, "elasticity": 0, "j2": 250, "neohooke": 150}[op]
    pair = {"diffusion": 7, "elasticity": 18, "j2": 42, "neohooke": 42}[op]
    return nq * (geometry + point + pairs * pair)


def work(case):
    path = case["path"]
    if path == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for etype, nx, ny, nz in _batch_boxes(case, 0):
            if etype == TET:
                c = _tet_box(nx, ny, nz)
            else:
                c = ({HEX: nx * ny * nz}, (nx + 1) * (ny + 1) * (nz + 1), (3 * nx + 1) * (3 * ny + 1) * (3 * nz + 1))
            w = _assembly_work(*c, "elasticity", 1)
            total = {k: total[k] + w[k] for k in total}
        return total
    elems, nodes, graph = _counts(case)
    conn = sum(4 * NN[t] * k for t, k in elems.items())
    n_elems = sum(elems.values())
    if path == "assembly":
        return _assembly_work(elems, nodes, graph, case["op"], case["tet_rule"])
    if path == "points":
        nq = {TET: 4, PYR: 8, PRISM: 6, HEX: 8}
        points = sum(nq[t] * k for t, k in elems.items())
        return {"bytes": conn + 48 * nodes + points * (2 * 56 + 48), "flops": points * 430.0}
    if path == "spmv":
        d = case["ndof"]
        return {"bytes": 8 * d * d * graph + 4 * graph + 8 * nodes * (3 * d + 1), "flops": 2.0 * d * d * graph}
    d = case["ndof"]
    # mesh in; row pointers, scalar columns and the map out
    return {"bytes": conn + 9 * n_elems + 24 * nodes + 8 * d * nodes + 4 * d * d * graph
            + sum(4 * NN[t] ** 2 * k for t, k in elems.items()), "flops": 0.0}


def _assembly_work(elems, nodes, graph, op, tet_rule):
    d = 1 if op == "diffusion" else 3
    by = 8 * d * d * graph + 16 * d * nodes + 24 * nodes
    by += sum((4 * NN[t] + 4 * NN[t] ** 2) * k for t, k in elems.items())
    if op in ("j2", "neohooke"):
        by += 24 * nodes
    if op == "j2":
        by += sum(2 * 8 * 7 * 8 * k for k in elems.values())
    return {"bytes": float(by), "flops": float(sum(_element_flops(t, op, tet_rule) * k for t, k in elems.items()))}


# ---------------------------------------------------------------------------
# exact: plain torch in 64 bits
# ---------------------------------------------------------------------------
def _rule(t, tet_rule=1):
    """Points [q, 3] and weights [q] of the reference element."""
    g = 1.0 / math.sqrt(3.0)
    gp = (-g, g)
    if t == TET:
        if not tet_rule:
            return [[0.25] * 3], [1.0 / 6.0]
        a, b = (5 + 3 * math.sqrt(5.0)) / 20, (5 - math.sqrt(5.0)) / 20
        return [[a if q == j + 1 else b for j in range(3)] for q in range(4)], [1.0 / 24.0] * 4
    if t == PRISM:
        tri = [(1 / 6, 1 / 6), (2 / 3, 1 / 6), (1 / 6, 2 / 3)]
        return [[x, y, z] for z in gp for x, y in tri], [1.0 / 6.0] * 6
    if t == HEX:
        return [[gp[q & 1], gp[(q >> 1) & 1], gp[q >> 2]] for q in range(8)], [1.0] * 8
    # pyramid: 2 x 2 Gauss times 2-point Gauss-Jacobi (weight (1 - t)^2) on the collapsed cube
    r = math.sqrt(10.0) / 15.0
    s = (1 / 3 - r, 1 / 3 + r)
    w1 = (1 / 12 - s[0] / 3) / (s[1] - s[0])
    return ([[gp[q & 1] * (1 - s[q >> 2]), gp[(q >> 1) & 1] * (1 - s[q >> 2]), s[q >> 2]] for q in range(8)],
            [1 / 3 - w1] * 4 + [w1] * 4)


def _shape(t, p):
    """N [a] and dN [a][3] at one reference point."""
    x, y, z = p
    if t == TET:
        return [1 - x - y - z, x, y, z], [[-1.0, -1.0, -1.0], [1.0, 0, 0], [0, 1.0, 0], [0, 0, 1.0]]
    if t == PRISM:
        L, Lx, Ly = (1 - x - y, x, y), (-1.0, 1.0, 0.0), (-1.0, 0.0, 1.0)
        N, D = [], []
        for h, hz in (((1 - z) / 2, -0.5), ((1 + z) / 2, 0.5)):
            N += [v * h for v in L]
            D += [[Lx[i] * h, Ly[i] * h, L[i] * hz] for i in range(3)]
        return N, D
    if t == HEX:
        N, D = [], []
        for c in _CORNERS:
            s = [2 * v - 1 for v in c]
            f = [(1 + s[0] * x) / 2, (1 + s[1] * y) / 2, (1 + s[2] * z) / 2]
            N.append(f[0] * f[1] * f[2])
            D.append([s[0] / 2 * f[1] * f[2], s[1] / 2 * f[0] * f[2], s[2] / 2 * f[0] * f[1]])
        return N, D
    w = 1 - z
    N, D = [], []
    for sx, sy in ((-1, -1), (1, -1), (1, 1), (-1, 1)):
        a, b = w + sx * x, w + sy * y
        N.append(a * b / (4 * w))
        D.append([sx * b / (4 * w), sy * a / (4 * w), (a * b - w * (a + b)) / (4 * w * w)])
    return N + [z], D + [[0.0, 0.0, 1.0]]


def _reference(t, tet_rule):
    P, w = _rule(t, tet_rule)
    NS = [_shape(t, p) for p in P]
    to = lambda v: torch.tensor(v, dtype=F64, device=DEV)  # noqa: E731
    return to([n for n, _ in NS]), to([d for _, d in NS]), to(w)


def _geometry(x, dN, w):
    """Gradients [e, q, a, 3] and w det J [e, q] of elements with nodes x [e, a, 3]."""
    d = x[:, 1:] - x[:, :1]  # the Jacobian from differences: no loss to the position of the element
    J = torch.einsum("eai,qaj->eqij", d, dN[:, 1:])
    det = (J[..., 0, :] * torch.linalg.cross(J[..., 1, :], J[..., 2, :])).sum(-1)
    cof = torch.stack([torch.linalg.cross(J[..., 1, :], J[..., 2, :]), torch.linalg.cross(J[..., 2, :], J[..., 0, :]),
                       torch.linalg.cross(J[..., 0, :], J[..., 1, :])], -2)
    return torch.einsum("eqij,qaj->eqai", cof, dN) / det[..., None, None], w * det


def _return_map(eps, state):
    """Radial return of strains [.., 3, 3] from states [.., 7]: stress, new state, normal, theta, theta bar."""
    mu = YOUNG / (2 * (1 + POISSON))
    kappa = YOUNG / (3 * (1 - 2 * POISSON))
    r23 = math.sqrt(2.0 / 3.0)
    p = state[..., [0, 3, 5, 3, 1, 4, 5, 4, 2]].reshape(*state.shape[:-1], 3, 3)
    an = state[..., 6]
    e = eps - p
    tr = e.diagonal(dim1=-2, dim2=-1).sum(-1)
    eye = torch.eye(3, dtype=F64, device=DEV)
    s = 2 * mu * (e - tr[..., None, None] / 3 * eye)
    norm = s.square().sum((-2, -1)).sqrt()
    sy = lambda a: SIGMA0 + HARDENING * a + (SIGMA_INF - SIGMA0) * -torch.expm1(-DELTA * a)  # noqa: E731
    plastic = norm > r23 * sy(an)
    dg = torch.zeros_like(norm)
    for _ in range(10):  # well past convergence
        a = an + r23 * dg
        slope = HARDENING + (SIGMA_INF - SIGMA0) * DELTA * torch.exp(-DELTA * a)
        dg = dg + (norm - 2 * mu * dg - r23 * sy(a)) / (2 * mu + 2.0 / 3.0 * slope)
    dg = torch.where(plastic, dg, torch.zeros_like(dg))
    a = an + r23 * dg
    n = torch.where(plastic[..., None, None], s / norm.clamp(min=1e-300)[..., None, None], torch.zeros_like(s))
    theta = torch.where(plastic, 1 - 2 * mu * dg / norm.clamp(min=1e-300), torch.ones_like(norm))
    slope = HARDENING + (SIGMA_INF - SIGMA0) * DELTA * torch.exp(-DELTA * a)
    bar = torch.where(plastic, 1 / (1 + slope / (3 * mu)) - (1 - theta), torch.zeros_like(norm))
    sig = s - 2 * mu * dg[..., None, None] * n + kappa * tr[..., None, None] * eye
    p = p + dg[..., None, None] * n
    new = torch.stack([p[..., 0, 0], p[..., 1, 1], p[..., 2, 2], p[..., 0, 1], p[..., 1, 2], p[..., 0, 2], a], -1)
    return sig, new, n, theta, bar


def _voigt(sig):
    return torch.stack([sig[..., 0, 0], sig[..., 1, 1], sig[..., 2, 2], sig[..., 0, 1], sig[..., 1, 2], sig[..., 0, 2]], -1)


_CHUNK = 65536


def _points(mesh, u, state):
    """New state and stress of every Gauss point (unused point slots stay 0)."""
    new = torch.zeros_like(state)
    stress = torch.zeros((mesh.n_elems, 8, 6), dtype=F64, device=DEV)
    for t, (ids, conn) in mesh.groups.items():
        _, dN, w = _reference(t, 1)
        for k in range(0, len(ids), 4 * _CHUNK):
            e, c = ids[k:k + 4 * _CHUNK], conn[k:k + 4 * _CHUNK]
            G, _ = _geometry(mesh.coords[c], dN, w)
            H = torch.einsum("eai,eqaj->eqij", u[c], G)
            sig, st, _, _, _ = _return_map((H + H.transpose(-1, -2)) / 2, state[e, :len(w)])
            new[e, :len(w)] = st
            stress[e, :len(w)] = _voigt(sig)
    return new, stress


def _element_matrices(case, x, u, state, N, dN, w):
    """A^e [e, a, c, b, d] and b^e [e, a, c]; the new state where the operator has one."""
    G, W = _geometry(x, dN, w)
    op = case.get("op", "elasticity")
    lam = YOUNG * POISSON / ((1 + POISSON) * (1 - 2 * POISSON))
    mu = YOUNG / (2 * (1 + POISSON))
    if op == "diffusion":
        xq = torch.einsum("qa,ea->eq", N, x[..., 0])
        S = W * (1.0 + case.get("k2", 0.0) * xq * xq)
        A = torch.einsum("eqai,eqbi->eab", S[..., None, None] * G, G)
        return A[:, :, None, :, None], torch.einsum("eq,qa->ea", W, N)[..., None], None
    eye = torch.eye(3, dtype=F64, device=DEV)

    def products(c, L, R):  # sum_q c L_a (x) R_b as [e, a, i, b, j]
        q, a = L.shape[1], L.shape[2]
        left = (c[..., None, None] * L).reshape(-1, q, 3 * a)
        return torch.bmm(left.transpose(1, 2), R.reshape(-1, q, 3 * a)).reshape(-1, a, 3, a, 3)

    def swapped(M):  # [e, a, i, b, j] -> the block's transpose
        return M.permute(0, 1, 4, 3, 2)

    def traced(M):
        return torch.einsum("eaibi,cd->eacbd", M, eye)

    if op == "elasticity":
        M = products(W, G, G)
        A = lam * M + mu * swapped(M) + mu * traced(M)
        return A, torch.einsum("eq,qa->ea", W, N)[..., None].expand(-1, -1, 3), None
    H = torch.einsum("eai,eqaj->eqij", u, G)
    if op == "j2":
        sig, new, n, theta, bar = _return_map((H + H.transpose(-1, -2)) / 2, state)
        kappa = lam + 2 * mu / 3
        h = torch.einsum("eqij,eqaj->eqai", n, G)
        M = products(W * mu * theta, G, G)
        A = products(W * (kappa - 2 * mu * theta / 3), G, G) + swapped(M) + traced(M) - products(W * 2 * mu * bar, h, h)
        return A, torch.einsum("eq,eqij,eqaj->eai", W, sig, G), new
    F = H + eye
    det = (F[..., 0, :] * torch.linalg.cross(F[..., 1, :], F[..., 2, :])).sum(-1)
    T = torch.stack([torch.linalg.cross(F[..., 1, :], F[..., 2, :]), torch.linalg.cross(F[..., 2, :], F[..., 0, :]),
                     torch.linalg.cross(F[..., 0, :], F[..., 1, :])], -2) / det[..., None, None]  # F^-T
    lnJ = torch.log(det)
    h = torch.einsum("eqij,eqaj->eqai", T, G)
    A = lam * products(W, h, h) + swapped(products(W * (mu - lam * lnJ), h, h)) + traced(mu * products(W, G, G))
    A = A + torch.einsum("eq,qa,qb,cd->eacbd", case["mass"] * W, N, N, eye)
    P = mu * (F - T) + lam * lnJ[..., None, None] * T
    return A, torch.einsum("eq,eqij,eqaj->eai", W, P, G), None


def _graph(mesh):
    """Sorted keys node * N + neighbour of the node graph."""
    N, parts = mesh.n_nodes, None
    for _, conn in mesh.groups.values():
        for k in range(0, len(conn), 8 * _CHUNK):
            c = conn[k:k + 8 * _CHUNK].to(torch.int64)
            key = torch.unique((c[:, :, None] * N + c[:, None, :]).reshape(-1))
            parts = key if parts is None else torch.unique(torch.cat([parts, key]))
    return parts


def _assembled(case, mesh, u, state, d):
    N = mesh.n_nodes
    keys = _graph(mesh)
    row = torch.div(keys, N, rounding_mode="floor")
    first = torch.searchsorted(row, torch.arange(N + 1, device=DEV))
    deg = first[1:] - first[:-1]
    A = torch.zeros(d * d * len(keys), dtype=F64, device=DEV)
    b = torch.zeros((N, d), dtype=F64, device=DEV)
    new = torch.zeros_like(state) if state is not None else None
    comp = torch.arange(d, device=DEV)
    for t, (ids, conn) in mesh.groups.items():
        Nq, dN, w = _reference(t, case.get("tet_rule", 1) if case.get("op") not in ("j2", "neohooke") else 1)
        for k in range(0, len(ids), _CHUNK):
            e, c = ids[k:k + _CHUNK], conn[k:k + _CHUNK].to(torch.int64)
            Ae, be, se = _element_matrices(case, mesh.coords[c], u[c] if u is not None else None,
                                           state[e, :len(w)] if state is not None else None, Nq, dN, w)
            rank = torch.searchsorted(keys, c[:, :, None] * N + c[:, None, :]) - first[c][:, :, None]
            base = d * d * first[c][:, :, None] + d * comp * deg[c][:, :, None]  # [e, a, c]
            pos = base[:, :, :, None, None] + d * rank[:, :, None, :, None] + comp
            A.index_add_(0, pos.reshape(-1), Ae.reshape(-1))
            b.index_add_(0, c.reshape(-1), be.reshape(-1, d))
            if se is not None:
                new[e, :len(w)] = se
    return A, b.reshape(-1), new, keys, first, deg


def exact(case, seed):
    path = case["path"]
    if path == "batch":
        As, bs = [], []
        for mesh in _batch_meshes(case, seed):
            A, b = _assembled({"op": "elasticity"}, mesh, None, None, 3)[:2]
            pad = torch.zeros(1, dtype=F64, device=DEV)
            As += [A] + ([pad] if A.numel() & 1 else [])
            bs += [b] + ([pad] if b.numel() & 1 else [])
        return {"A": torch.cat(As), "b": torch.cat(bs)}
    if path == "pattern":
        return None  # whole numbers
    mesh, u, state = _inputs(case, seed)
    if path == "points":
        new, stress = _points(mesh, u, state)
        return {"state": new, "stress": stress}
    if path == "spmv":
        d = case["ndof"]
        op = {"op": "diffusion" if d == 1 else "elasticity"}
        A, _, _, keys, first, deg = _assembled(op, mesh, None, None, d)
        x = torch.randn(d * mesh.n_nodes, generator=_generator(seed + 1), dtype=F64, device=DEV).reshape(-1, d)
        node = torch.div(keys, mesh.n_nodes, rounding_mode="floor")
        col = keys - node * mesh.n_nodes
        y = torch.zeros((mesh.n_nodes, d), dtype=F64, device=DEV)
        at = d * d * first[node] + d * (torch.arange(len(keys), device=DEV) - first[node])
        for c in range(d):
            for k in range(d):
                y[:, c].index_add_(0, node, A[at + c * d * deg[node] + k] * x[col, k])
        return {"y": y.reshape(-1)}
    A, b, new = _assembled(case, mesh, u, state, 1 if case["op"] == "diffusion" else 3)[:3]
    out = {"A": A, "b": b}
    if new is not None:
        out["state"] = new
    return out
