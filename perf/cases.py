"""Performance cases: the work a user of the library has it do, through its public entry
points, with inputs made from a seed on the GPU and 64-bit reference values.

A case is a dict of plain values. `path` names the entry point (tabulate, assemble, pair,
rows, batch, adjoint, source, quadrature), `form` / `d` / `q` the form, the cell dimension
and the degree, `n` the structured mesh (2 n^2 triangles of the unit square or 6 n^3
tetrahedra of the unit cube, interior vertices jittered), `precision` the arithmetic.

`prepare` builds what a program holds before the call: mesh, dof map, pattern, slots, row
plan, form handle, coefficient fields. Meshes follow the library's conventions for local
and global dof order; the pattern is the one csr_pattern returns, made here on the GPU so
that inputs are quick to make.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_1112_0402_gb300 as ffc

FORMS = {"mass": ffc.MASS, "poisson": ffc.POISSON, "convection": ffc.NS_CONVECTION, "elasticity": ffc.ELASTICITY,
         "source": ffc.SOURCE}
MU, LAMBDA = 1.0, 1.25
BATCH_FORMS = (("elasticity", 1), ("elasticity", 2), ("elasticity", 3), ("poisson", 2))


def listed():
    return [
        # one small 2-D stiffness matrix from scratch, in the default precision: the smallest
        # call, where launches and latency count (the 64 x 64 x 2 P1 Poisson configuration)
        {"name": "tri_p1_poisson_assemble", "path": "assemble", "form": "poisson", "d": 2, "q": 1, "n": 64,
         "precision": "fp64"},
        # element tensors of a small 3-D mesh of odd size, for a program with its own insertion
        {"name": "tet_p2_poisson_tabulate_fp32", "path": "tabulate", "form": "poisson", "d": 3, "q": 2, "n": 13,
         "precision": "fp32"},
        # element tensors of high degree in the default precision, a large mesh
        {"name": "tet_p4_poisson_tabulate", "path": "tabulate", "form": "poisson", "d": 3, "q": 4, "n": 40,
         "precision": "fp64"},
        # a 3-D stiffness matrix from scratch in the default precision, odd size
        {"name": "tet_p3_poisson_assemble", "path": "assemble", "form": "poisson", "d": 3, "q": 3, "n": 31,
         "precision": "fp64"},
        # mass and stiffness of a low-degree space in one call (time stepping, eigenproblems)
        {"name": "tet_p2_pair_fp32", "path": "pair", "form": "mass+poisson", "d": 3, "q": 2, "n": 48,
         "precision": "fp32"},
        # the same by row-owner assembly, the route for high degrees: an odd-sized mesh, and
        # the largest configuration (48^3 x 6 cells, P4)
        {"name": "tet_p3_rows_pair_fp32", "path": "rows", "form": "mass+poisson", "d": 3, "q": 3, "n": 33,
         "precision": "fp32"},
        {"name": "tet_p4_rows_pair_fp32", "path": "rows", "form": "mass+poisson", "d": 3, "q": 4, "n": 48,
         "precision": "fp32"},
        # a form with a coefficient field, in the default precision (40^3 x 6 cells, vector P2)
        {"name": "convection_p2_tabulate", "path": "tabulate", "form": "convection", "d": 3, "q": 2, "n": 40,
         "precision": "fp64"},
        # many meshes and forms in one persistent launch, replayed as a graph: elasticity
        # P1-P3 and Poisson P2 on 32 meshes of uneven size
        {"name": "batch_32_meshes", "path": "batch", "form": "elasticity+poisson", "d": 3, "q": 3, "count": 32,
         "lo": 130, "hi": 25000, "precision": "fp32"},
        # forward and backward of a shape derivative through autograd (56^3 x 6 cells)
        {"name": "shape_gradient_p2", "path": "adjoint", "form": "poisson", "d": 3, "q": 2, "n": 56,
         "precision": "fp64"},
        # a load vector of high degree (48^3 x 6 cells)
        {"name": "source_p4_fp32", "path": "source", "form": "source", "d": 3, "q": 4, "n": 48, "precision": "fp32"},
        # element tensors on curved cells by the quadrature representation (40^3 x 6 cells)
        {"name": "curved_p2_poisson_tf32x3", "path": "quadrature", "form": "poisson", "d": 3, "q": 2, "n": 40,
         "precision": "tf32x3"},
    ]


def _mesh_size(rng, d, lo, hi):
    """n of a structured mesh whose cell count is log-uniform in [lo, hi]."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    n = round(math.sqrt(cells / 2)) if d == 2 else round((cells / 6) ** (1 / 3))
    return max(2, int(n))


def draw(rng):
    path = rng.choice(["tabulate", "tabulate", "assemble", "assemble", "pair", "rows", "rows", "batch", "adjoint",
                       "source", "quadrature", "quadrature"])
    d = 3 if path == "batch" else rng.choice([2, 3, 3, 3])
    precision = rng.choice(["fp64", "fp32"])
    if path in ("tabulate", "assemble"):
        form = rng.choice(["mass", "poisson", "convection", "elasticity"] if d == 3 else ["mass", "poisson"])
        q = rng.randint(1, {"convection": 2, "elasticity": 3}.get(form, 4))
        split = {"convection": (2,), "elasticity": (1, 2, 3), "poisson": (2, 3, 4), "mass": (3, 4)}[form]
        if d == 3 and q in split and rng.random() < 0.25:
            precision = rng.choice(["tf32x3", "bf16x3"])
    elif path in ("pair", "rows"):
        form, precision = "mass+poisson", "fp32" if path == "pair" else precision
        q = rng.randint(1, 2) if path == "pair" else rng.randint(2, 4)
    elif path == "batch":
        lo = rng.randint(60, 400)
        return {"path": path, "form": "elasticity+poisson", "d": 3, "q": 3, "count": rng.randint(3, 24), "lo": lo,
                "hi": lo * rng.randint(10, 60), "precision": "fp32"}
    elif path == "adjoint":
        form, q, precision = "poisson", rng.randint(1, 4), "fp64"
    elif path == "source":
        form, q = "source", rng.randint(1, 4)
    else:
        form, q = rng.choice(["mass", "poisson"]), rng.randint(1, 2)
        precision = rng.choice(["fp64", "fp32", "tf32x3", "bf16x3", "fp64_ozaki"])
    n_local = _n_scalar(d, q) * (d if form in ("convection", "elasticity") else 1)
    per_cell = n_local * n_local if path not in ("source",) else n_local
    most = {"tabulate": 3e8, "assemble": 1.5e8, "pair": 6e7, "rows": 3e8, "adjoint": 1e8, "source": 2e7,
            "quadrature": 3e7}[path]
    hi = max(2000.0, min(6e5, most / per_cell))
    return {"path": path, "form": form, "d": d, "q": q, "n": _mesh_size(rng, d, 500, hi), "precision": precision}


# ------------------------------------------------------------------ meshes and dof maps

def _n_scalar(d, q):
    return math.comb(q + d, d)


def _lattice(d, q):
    """Barycentric lattice indices in local dof order: by support (vertices, edges, faces,
    interior; subsets in lexicographic order), descending within a support."""
    out = []
    for m in range(d + 1):
        for support in itertools.combinations(range(d + 1), m + 1):
            pts = [k for k in itertools.product(range(q + 1), repeat=d + 1)
                   if sum(k) == q and tuple(j for j in range(d + 1) if k[j]) == support]
            out += sorted(pts, reverse=True)
    return np.array(out, dtype=np.int64)


def _grid(n, d):
    ax = torch.arange(n + 1, device="cuda")
    return torch.cartesian_prod(*([ax] * d))


def _cells(n, d):
    """int64 [n_elem, d+1]: two triangles a square, six Kuhn tetrahedra a cube."""
    ax = torch.arange(n, device="cuda")
    corner = torch.cartesian_prod(*([ax] * d))
    eye = torch.eye(d, dtype=torch.int64, device="cuda")

    def vid(c):
        v = c[:, 0]
        for a in range(1, d):
            v = v * (n + 1) + c[:, a]
        return v

    parts = []
    for p in itertools.permutations(range(d)):
        c = [corner]
        for a in p:
            c.append(c[-1] + eye[a])
        if d == 2 and p == (1, 0):
            c = [c[0], c[2], c[1]]
        parts.append(torch.stack([vid(x) for x in c], dim=1))
    return torch.stack(parts, dim=1).reshape(-1, d + 1)


def _vertices(lat, n, d, jitter, gen):
    x = lat.to(torch.float64) / n
    inside = ((lat > 0) & (lat < n)).all(dim=1)
    r = torch.rand(lat.shape, dtype=torch.float64, device="cuda", generator=gen)
    return x + inside[:, None] * (r * 2 - 1) * (jitter / n)


def _dofmap(cells, lat, n, d, q, vector=False):
    """int32 [n_elem, n_local] and the number of global dofs (lexicographic lattice ids)."""
    k = torch.from_numpy(_lattice(d, q)).cuda()
    corner = lat[cells]
    side = q * n + 1
    gid = torch.zeros((cells.shape[0], k.shape[0]), dtype=torch.int64, device="cuda")
    for a in range(d):
        pos = sum(corner[:, j, a][:, None] * k[None, :, j] for j in range(d + 1))
        gid = gid * side + pos
    if vector:
        gid = torch.cat([gid * d + c for c in range(d)], dim=1)
    return gid.to(torch.int32), side ** d * (d if vector else 1)


def _pattern(dofmap, n_dof, with_slots=True):
    """Sorted CSR pattern: row_ptr int64, col int32, slot int32 [n_elem, n, n] (or None)."""
    dm = dofmap.to(torch.int64)
    keys = (dm[:, :, None] * n_dof + dm[:, None, :]).reshape(-1)
    if with_slots:
        uniq, inv = torch.unique(keys, return_inverse=True)
        slot = inv.to(torch.int32).reshape(dm.shape[0], dm.shape[1], dm.shape[1])
        del inv
    else:
        uniq, slot = torch.unique(keys), None
    del keys
    row = torch.div(uniq, n_dof, rounding_mode="floor")
    col = (uniq - row * n_dof).to(torch.int32)
    row_ptr = torch.zeros(n_dof + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n_dof), 0)
    return row_ptr, col, slot


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _problem(case, n, form, q, gen):
    """Mesh, dof map and coefficients of one (mesh, form) problem."""
    d = case["d"]
    lat, cells = _grid(n, d), _cells(n, d)
    vector = form in ("convection", "elasticity")
    dofmap, n_dof = _dofmap(cells, lat, n, d, q, vector)
    p = {"cells": cells.to(torch.int32).contiguous(),
         "vertices": _vertices(lat, n, d, 0.2 if d == 2 else 0.15, gen).contiguous(),
         "dofmap": dofmap.contiguous(), "n_dof": n_dof, "coeffs": None}
    if form in ("convection", "source"):  # a global field, iid N(0, 1) per dof, gathered per cell
        w = torch.randn(n_dof, dtype=torch.float64, device="cuda", generator=gen)
        p["coeffs"] = w[dofmap.to(torch.int64)].contiguous()
    return p


def _curved(case, gen):
    """Quadratic-geometry cells: the P2 lattice of the straight mesh moved by a smooth
    field that vanishes on the boundary, with amplitude and direction from the seed."""
    d, n = case["d"], case["n"]
    lat, cells = _grid(n, d), _cells(n, d)
    nodes_of, n_nodes = _dofmap(cells, lat, n, d, 2)
    x = torch.cartesian_prod(*([torch.arange(2 * n + 1, device="cuda")] * d)).to(torch.float64) / (2 * n)
    v = torch.rand(d, dtype=torch.float64, device="cuda", generator=gen) * 2 - 1
    bump = torch.sin(math.pi * x).prod(dim=1)
    return {"cells": nodes_of.contiguous(), "nodes": (x + 0.08 * bump[:, None] * v / v.abs().max()).contiguous()}


def _batch_sizes(case):
    r = np.random.default_rng(4)
    t = np.exp(r.uniform(np.log(case["lo"]), np.log(case["hi"]), size=case["count"]))
    return [max(1, int(round((c / 6.0) ** (1.0 / 3.0)))) for c in t]


def _handle(form, d, q):
    return ffc.Form(FORMS[form], ffc.TRIANGLE if d == 2 else ffc.TETRAHEDRON, q, MU, LAMBDA)


def prepare(case, seed):
    gen = _generator(seed)
    path, form, d, q, prec = case["path"], case["form"], case["d"], case["q"], case["precision"]
    s = {"path": path, "precision": prec}
    if path == "batch":
        items = []
        forms = {}
        for m, n in enumerate(_batch_sizes(case)):
            f, fq = BATCH_FORMS[m % len(BATCH_FORMS)]
            p = _problem(case, n, f, fq, gen)
            _, col, slot = _pattern(p["dofmap"], p["n_dof"])
            if (f, fq) not in forms:
                forms[f, fq] = _handle(f, 3, fq)
            items.append({"form": forms[f, fq], "cells": p["cells"], "vertices": p["vertices"], "slot": slot,
                          "csr_val": torch.empty(col.numel(), dtype=torch.float64, device="cuda")})
        s["items"], s["batch"] = items, ffc.Batch(items)
        s["batch"].tune()
        return s
    if path == "quadrature":
        s.update(_curved(case, gen))
        s["form"] = ffc.QForm(FORMS[form], ffc.TRIANGLE if d == 2 else ffc.TETRAHEDRON, q, 2)
        return s
    if path in ("pair", "rows"):
        s.update(_problem(case, case["n"], "mass", q, gen))
        row_ptr, col, slot = _pattern(s["dofmap"], s["n_dof"], path == "pair")
        s["forms"] = [_handle("mass", d, q), _handle("poisson", d, q)]
        s["values"] = [torch.empty(col.numel(), dtype=torch.float64, device="cuda") for _ in range(2)]
        if path == "pair":
            s["slot"] = slot
        else:
            s["plan"] = ffc.RowPlan(s["dofmap"], s["n_dof"], row_ptr, col)
        return s
    s.update(_problem(case, case["n"], form, q, gen))
    s["form"] = _handle(form, d, q)
    if path == "assemble":
        _, col, s["slot"] = _pattern(s["dofmap"], s["n_dof"])
        s["csr_val"] = torch.empty(col.numel(), dtype=torch.float64, device="cuda")
    elif path == "source":
        s["b"] = torch.empty(s["n_dof"], dtype=torch.float64, device="cuda")
    elif path == "adjoint":  # L = u^T A v: the upstream gradient of every element tensor
        s["grad"] = _upstream(s, gen)
    return s


def _upstream(p, gen):
    u, v = (torch.randn(p["n_dof"], dtype=torch.float64, device="cuda", generator=gen) for _ in range(2))
    dm = p["dofmap"].to(torch.int64)
    return (u[dm][:, :, None] * v[dm][:, None, :]).contiguous()


def run(s):
    path, prec = s["path"], s["precision"]
    if path == "tabulate":
        return ffc.tabulate(s["form"], s["cells"], s["vertices"], coeffs=s["coeffs"], precision=prec)
    if path == "assemble":
        s["csr_val"].zero_()
        return ffc.assemble(s["form"], s["cells"], s["vertices"], s["slot"], s["csr_val"], coeffs=s["coeffs"],
                            precision=prec)
    if path == "pair":
        a, b = s["values"]
        a.zero_()
        b.zero_()
        return ffc.assemble_pair(*s["forms"], s["cells"], s["vertices"], s["slot"], a, b, precision=prec)
    if path == "rows":
        return ffc.assemble_rows_pair(*s["forms"], s["plan"], s["cells"], s["vertices"], *s["values"],
                                      precision=prec)
    if path == "batch":
        s["batch"].run(graph=True)
        return [it["csr_val"] for it in s["items"]]
    if path == "adjoint":
        from paper_1112_0402_gb300.autograd import element_tensors

        x = s["vertices"].detach().requires_grad_(True)
        A = element_tensors(s["form"], s["cells"], x)
        (dx,) = torch.autograd.grad(A, x, s["grad"])
        return A.detach(), dx
    if path == "source":
        s["b"].zero_()
        return ffc.assemble(s["form"], s["cells"], s["vertices"], s["dofmap"], s["b"], coeffs=s["coeffs"],
                            precision=prec)
    return ffc.tabulate_quadrature(s["form"], s["cells"], s["nodes"], precision=prec)


# ------------------------------------------------------------------ required work

def _counts(n, d, q):
    """Cells, vertices, scalar dofs and stored entries of the scalar P_q pattern. Two dofs
    share a cell when some simplex of the mesh is the join of their supports, so the
    entries are counted per simplex."""
    V, C = (n + 1) ** d, (2 if d == 2 else 6) * n ** d
    if d == 2:
        ent = [V, 2 * n * (n + 1) + n * n, C]
    else:
        E = 3 * n * (n + 1) ** 2 + 3 * n * n * (n + 1) + n ** 3
        ent = [V, E, 1 - V + E + C, 0]
        ent[2] = E + C + 1 - V
        ent[3] = C
    nnz = 0
    for m in range(d + 1):
        pts = [frozenset(j for j in range(m + 1) if k[j]) for k in itertools.product(range(q + 1), repeat=m + 1)
               if sum(k) == q]
        nnz += ent[m] * sum(len(a | b) == m + 1 for a in pts for b in pts)
    return C, V, (q * n + 1) ** d, nnz


def work(case):
    """Each input read once, each output written once; the contraction's multiply-adds."""
    path, d, q = case["path"], case["d"], case["q"]
    f64 = case["precision"] in ("fp64", "fp64_ozaki")
    if path == "batch":
        total = {"bytes": 0, "flops": 0}
        for m, n in enumerate(_batch_sizes(case)):
            f, fq = BATCH_FORMS[m % len(BATCH_FORMS)]
            w = work({"path": "assemble", "form": f, "d": 3, "q": fq, "n": n, "precision": "fp32"})
            total = {k: total[k] + w[k] for k in total}
        return total
    n = case["n"]
    C, V, dofs, nnz = _counts(n, d, q)
    ns = _n_scalar(d, q)
    form = case["form"]
    if path == "quadrature":
        points = math.ceil((2 * q + d + 1) / 2) ** d
        K = points * (1 if form == "mass" else d * (d + 1) // 2)
        ng = _n_scalar(d, 2)
        return {"bytes": C * (4 * ng + ns * ns * (8 if f64 else 4)) + 8 * d * (2 * n + 1) ** d,
                "flops": 2 * C * ns * ns * K}
    mesh = C * 4 * (d + 1) + V * 8 * d
    vec = d if form in ("convection", "elasticity") else 1
    nl = ns * vec
    per_entry = {"mass": 1, "poisson": d * (d + 1) // 2, "mass+poisson": 1 + d * (d + 1) // 2,
                 "convection": ns * d / d ** 2, "elasticity": d * d, "source": ns}[form]
    flops = 2 * C * (nl if form == "source" else nl * nl) * per_entry
    if path == "tabulate":
        return {"bytes": mesh + C * nl * nl * (8 if f64 else 4) + (C * nl * 8 if form == "convection" else 0),
                "flops": flops}
    if path == "adjoint":
        return {"bytes": 2 * mesh + 2 * C * nl * nl * 8 + V * 8 * d, "flops": 2 * flops}
    if path == "source":
        return {"bytes": mesh + C * nl * 12 + 8 * dofs, "flops": flops}
    if path == "rows":  # the pattern's part of the input is the dof map (the plan is its row view)
        return {"bytes": mesh + 4 * C * nl + 16 * nnz, "flops": flops}
    out = 16 * nnz if path == "pair" else 8 * nnz * vec * vec
    return {"bytes": mesh + 4 * C * nl * nl + out + (C * nl * 8 if form == "convection" else 0), "flops": flops}


# ------------------------------------------------------------------ values in 64 bits

def _poly(d, q):
    """The Lagrange P_q basis as polynomials in the d+1 barycentric coordinates: exponents
    [m][d+1], coefficients [n][m] and those of the reference gradients [d][n][m]."""
    expo = [k for k in itertools.product(range(q + 1), repeat=d + 1) if sum(k) <= q]
    at = {k: i for i, k in enumerate(expo)}
    one = []
    for m in range(q + 1):  # prod_{s<m} (q x - s) / (s + 1)
        c = np.array([1.0], dtype=np.longdouble)
        for s in range(m):
            c = np.convolve(c, np.array([-s, q], dtype=np.longdouble) / (s + 1))
        one.append(c)
    lat = _lattice(d, q)
    C = np.zeros((len(lat), len(expo)), dtype=np.longdouble)
    for i, k in enumerate(lat):
        for e in itertools.product(*[range(kj + 1) for kj in k]):
            C[i, at[e]] += np.prod([one[k[j]][e[j]] for j in range(d + 1)])
    D = np.zeros((d + 1,) + C.shape, dtype=np.longdouble)
    for e, m in at.items():
        for j in range(d + 1):
            if e[j]:
                D[j][:, at[e[:j] + (e[j] - 1,) + e[j + 1:]]] += e[j] * C[:, m]
    return np.array(expo), C, D[1:] - D[:1]


def _moment(e, d):
    f = [np.longdouble(math.factorial(i)) for i in range(64)]
    return np.prod([f[int(x)] for x in e]) / f[int(sum(e)) + d]


def _gram(expo, d):
    table = {}
    M = np.zeros((len(expo), len(expo)), dtype=np.longdouble)
    for i, a in enumerate(expo):
        for j, b in enumerate(expo):
            k = tuple(sorted(int(x) for x in a + b))
            if k not in table:
                table[k] = _moment(k, d)
            M[i, j] = table[k]
    return M


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _inverse(J):
    """K = J^-1 and |det J| by cofactors, J [..., d, d]."""
    d = J.shape[-1]
    if d == 2:
        adj = torch.stack([torch.stack([J[..., 1, 1], -J[..., 0, 1]], -1),
                           torch.stack([-J[..., 1, 0], J[..., 0, 0]], -1)], -2)
    else:
        r = [torch.linalg.cross(J[..., :, (a + 1) % 3], J[..., :, (a + 2) % 3], dim=-1) for a in range(3)]
        adj = torch.stack(r, -2)
    det = (adj[..., 0, :] * J[..., :, 0]).sum(-1)
    return adj / det[..., None, None], det.abs()


def _jacobian(x):
    """x [E, d+1, d] -> J [E, d, d], column c the edge x_{c+1} - x_0."""
    return (x[:, 1:] - x[:, :1]).transpose(1, 2)


class _Exact:
    """Element tensors of one form in 64 bits."""

    def __init__(self, form, d, q):
        self.form, self.d, self.ns = form, d, _n_scalar(d, q)
        expo, C, D = _poly(d, q)
        M = _gram(expo, d)
        if form in ("mass", "source"):
            self.A0 = _gpu(C @ M @ C.T)
        elif form in ("poisson", "elasticity"):
            self.A0 = _gpu(np.stack([D[a] @ M @ D[b].T for a in range(d) for b in range(d)]))  # [dd, n, n]
        else:
            T = np.array([[[_moment(a + b + c, d) for c in expo] for b in expo] for a in expo], dtype=np.longdouble)
            R = np.stack([np.tensordot(np.tensordot(np.tensordot(C, T, (1, 0)), C, (1, 1)), D[a], (1, 1))
                          for a in range(d)])  # [a, i, t, j]
            self.A0 = _gpu(R.transpose(2, 0, 1, 3).reshape(len(C) * d, -1))  # [(t, a), i j]

    def tensors(self, x, w=None):
        d, ns, E = self.d, self.ns, x.shape[0]
        K, det = _inverse(_jacobian(x))
        if self.form == "mass":
            return det[:, None, None] * self.A0
        if self.form == "source":
            return det[:, None] * (w @ self.A0.T)
        if self.form == "poisson":
            G = det[:, None, None] * (K @ K.transpose(1, 2))
            return (G.reshape(E, -1) @ self.A0.reshape(d * d, -1)).reshape(E, ns, ns)
        if self.form == "convection":
            H = det[:, None, None] * torch.einsum("eac,ect->eta", K, w.reshape(E, d, ns))
            B = (H.reshape(E, -1) @ self.A0).reshape(E, ns, ns)
            A = torch.zeros((E, d, ns, d, ns), dtype=torch.float64, device="cuda")
            for c in range(d):
                A[:, c, :, c, :] = B
        else:
            KK = K @ K.transpose(1, 2)
            A = torch.zeros((E, d, ns, d, ns), dtype=torch.float64, device="cuda")
            for c1 in range(d):
                for c2 in range(d):
                    G = MU * K[:, :, c2, None] * K[:, None, :, c1] + LAMBDA * K[:, :, c1, None] * K[:, None, :, c2]
                    if c1 == c2:
                        G = G + MU * KK
                    G = det[:, None] * G.reshape(E, -1)
                    A[:, c1, :, c2, :] = (G @ self.A0.reshape(d * d, -1)).reshape(E, ns, ns)
        return A.reshape(E, d * ns, d * ns)


def _assembled(form, d, q, p, slot, nnz):
    ex = _Exact(form, d, q)
    out = torch.zeros(nnz, dtype=torch.float64, device="cuda")
    E = p["cells"].shape[0]
    step = max(1, int(1e8 // max(1, slot[0].numel())))
    for e in range(0, E, step):
        x = p["vertices"][p["cells"][e:e + step].to(torch.int64)]
        w = None if p["coeffs"] is None else p["coeffs"][e:e + step]
        out.index_add_(0, slot[e:e + step].reshape(-1).to(torch.int64), ex.tensors(x, w).reshape(-1))
    return out


def _rule(d, degree):
    """Collapsed Gauss-Jacobi rule: points X [N][d] and weights, by the eigenvalues of the
    Jacobi matrix of the weight (1 - u)^k on [0, 1] in each direction."""
    m = math.ceil((degree + 1) / 2)
    dirs = []
    for k in range(d):
        n = np.arange(m, dtype=np.float64)
        a = (-k * k) / ((2 * n + k) * (2 * n + k + 2)) if k else np.zeros(m)
        n = n[1:]
        b = 4 * n * n * (n + k) ** 2 / ((2 * n + k) ** 2 * (2 * n + k + 1) * (2 * n + k - 1))
        x, v = np.linalg.eigh(np.diag(a) + np.diag(np.sqrt(b), 1) + np.diag(np.sqrt(b), -1))
        dirs.append(((x + 1) / 2, v[0] ** 2 / (k + 1)))
    X, W = [], []
    for idx in itertools.product(range(m), repeat=d):
        u = [dirs[k][0][idx[k]] for k in range(d)]
        X.append([u[k] * math.prod(1 - u[t] for t in range(k + 1, d)) for k in range(d)])
        W.append(math.prod(dirs[k][1][idx[k]] for k in range(d)))
    return np.array(X), np.array(W)


def _at_points(expo, C, X):
    lam = np.concatenate([1 - X.sum(1, keepdims=True), X], axis=1)
    mono = np.prod(lam[:, None, :] ** expo[None], axis=2)  # [N, m]
    return mono @ np.asarray(C, dtype=np.float64).T


def _exact_curved(case, seed):
    d, q = case["d"], case["q"]
    p = _curved(case, _generator(seed))
    X, W = _rule(d, 2 * q + d)
    expo, C, D = _poly(d, q)
    ge, _, GD = _poly(d, 2)
    dgeo = _gpu(np.stack([_at_points(ge, GD[a], X) for a in range(d)], -1))  # [N, n_g, d]
    if case["form"] == "mass":
        phi = _at_points(expo, C, X)
        B = _gpu(np.einsum("k,ki,kj->kij", W, phi, phi))
    else:
        dphi = np.stack([_at_points(expo, D[a], X) for a in range(d)], -1)
        B = _gpu(np.einsum("k,kia,kjb->kabij", W, dphi, dphi))
    ns, E, out = _n_scalar(d, q), p["cells"].shape[0], []
    for e in range(0, E, 32768):
        x = p["nodes"][p["cells"][e:e + 32768].to(torch.int64)]
        K, det = _inverse(torch.einsum("enr,kna->ekra", x, dgeo))
        G = det if case["form"] == "mass" else det[..., None, None] * (K @ K.transpose(-1, -2))
        out.append((G.reshape(x.shape[0], -1) @ B.reshape(-1, ns * ns)).reshape(-1, ns, ns))
    return torch.cat(out)


def exact(case, seed):
    path, d, q = case["path"], case["d"], case["q"]
    if path == "quadrature":
        return _exact_curved(case, seed)
    gen = _generator(seed)
    if path == "batch":
        out = []
        for m, n in enumerate(_batch_sizes(case)):
            f, fq = BATCH_FORMS[m % len(BATCH_FORMS)]
            p = _problem(case, n, f, fq, gen)
            _, col, slot = _pattern(p["dofmap"], p["n_dof"])
            out.append(_assembled(f, 3, fq, p, slot, col.numel()))
        return out
    if path in ("pair", "rows"):
        p = _problem(case, case["n"], "mass", q, gen)
        _, col, slot = _pattern(p["dofmap"], p["n_dof"])
        return tuple(_assembled(f, d, q, p, slot, col.numel()) for f in ("mass", "poisson"))
    p = _problem(case, case["n"], case["form"], q, gen)
    if path == "assemble":
        _, col, slot = _pattern(p["dofmap"], p["n_dof"])
        return _assembled(case["form"], d, q, p, slot, col.numel())
    if path == "source":
        return _assembled("source", d, q, p, p["dofmap"], p["n_dof"])
    ex = _Exact(case["form"], d, q)
    cells, E = p["cells"].to(torch.int64), p["cells"].shape[0]
    step = 16384
    A = torch.cat([ex.tensors(p["vertices"][cells[e:e + step]],
                              None if p["coeffs"] is None else p["coeffs"][e:e + step]) for e in range(0, E, step)])
    if path == "tabulate":
        return A
    grad = _upstream(p, gen)
    x = p["vertices"].detach().requires_grad_(True)
    Gbar = (grad.reshape(E, -1) @ ex.A0.reshape(d * d, -1).T).reshape(E, d, d)
    K, det = _inverse(_jacobian(x[cells]))
    (dx,) = torch.autograd.grad((det[:, None, None] * (K @ K.transpose(1, 2)) * Gbar).sum(), x)
    return A, dx
