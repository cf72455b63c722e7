"""Workloads by which changes to the kernels are judged: what they call, on which inputs, and what the results are in 64 bits.

Every case goes through the package's public calls (``assemble``, ``AssembleFn``, ``CsrMatrix.assemble``,
``BatchPlan.launch``) on seeded, perturbed structured meshes made on the GPU with the recipes of
``paper_1407_0904_gb300.meshgen`` (same grids, cells, node numbering, perturbation and coefficient ranges). The
sizes are those of the benchmark's workloads and of the test suite, or lie between them.

A case is a dict:
  op         "forward"  element matrices or vectors; with a float precision the coefficients are rounded, and for
                        degree 1 and the residual the coordinates split, in the same pass, as the benchmark does
             "adjoint"  one differentiable step: element matrices and the gradients of <A, dA>
             "csr"      global matrix values; the sparsity pattern and entry map belong to the mesh and are kept
             "batch"    mixed groups (form, degree) of one triangle and one tetrahedral mesh, planned once
  form, degree, cell, precision   the package's numbers
  ncells     cells (the mesh is the smallest cube or square that holds them, truncated)
  permute    whether the nodes of cell2dof are numbered at random
"""
import itertools
import math

import numpy as np
import torch

import paper_1407_0904_gb300 as coffee
from paper_1407_0904_gb300 import meshgen

MASS, HELMHOLTZ, ADVDIFF, BURGERS, RESIDUAL = range(5)
TRI, TET, PRISM = range(3)
FP64, TF32, TF32X3, BF16, BF16X3 = range(5)
NU = 0.01
DEV = "cuda"


def _case(op, form, degree, cell, precision, ncells, permute=False, name=None):
    c = {"op": op, "form": form, "degree": degree, "cell": cell, "precision": precision, "ncells": ncells,
         "permute": permute}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the smallest call: a 64 x 64 square of triangles in double, one short launch (a 2D test problem, one
        # matrix of a small Newton or time step)
        _case("forward", HELMHOLTZ, 1, TRI, FP64, 8192, name="helmholtz-p1-tri-fp64-small"),
        # the benchmark's headline: a large 3D Helmholtz problem in cubic elements, float results
        _case("forward", HELMHOLTZ, 3, TET, TF32X3, 1572864, name="helmholtz-p3-tet"),
        # the highest degree: 35 x 35 matrices, whose rows start at odd multiples of 4 bytes
        _case("forward", HELMHOLTZ, 4, TET, TF32X3, 196608, name="helmholtz-p4-tet"),
        # the same forms in double, the type that assemble() and the plain C entry point take by default
        _case("forward", HELMHOLTZ, 3, TET, FP64, 196608, name="helmholtz-p3-tet-fp64"),
        # advection-diffusion with P1 coefficients, 2^20 quadratic tetrahedra: transport of a scalar
        _case("forward", ADVDIFF, 2, TET, TF32X3, 1 << 20, name="advdiff-p2-tet"),
        # one Newton iteration of the viscous Burgers equation: its Jacobian, and its residual
        _case("forward", BURGERS, 2, TET, TF32X3, 1 << 20, name="burgers-p2-tet"),
        _case("forward", RESIDUAL, 2, TET, TF32X3, 1 << 20, name="burgers-residual-p2-tet"),
        # shape and parameter gradients: forward and backward of advection-diffusion in double (AssembleFn's
        # default), 2^19 quadratic tetrahedra
        _case("adjoint", ADVDIFF, 2, TET, FP64, 1 << 19, name="adjoint-advdiff-p2-tet"),
        # the global matrix of a quadratic Helmholtz problem in double (CsrMatrix.assemble's default)
        _case("csr", HELMHOLTZ, 2, TET, FP64, 196608, name="global-helmholtz-p2-tet-fp64"),
        # a mesh of many element types: 21 groups, 2^19 triangles and 2^19 tetrahedra
        _case("batch", HELMHOLTZ, 4, TET, TF32X3, 1 << 20, name="batch-mixed"),
        # layered meshes (ocean, atmosphere): twisted prisms, whose geometry varies inside the cell
        _case("forward", HELMHOLTZ, 3, PRISM, TF32X3, 55296, name="helmholtz-p3-prism"),
        # the Burgers Jacobian on them, which exists in double only
        _case("forward", BURGERS, 2, PRISM, FP64, 27648, name="burgers-p2-prism-fp64"),
    ]


def draw(rng):
    """One more case of the same ranges: any form, degree, cell, precision the package has, 300 cells or more."""
    while True:
        op = rng.choices(("forward", "adjoint", "csr", "batch"), (12, 3, 3, 1))[0]
        cell = rng.choices((TRI, TET, PRISM), (2, 4, 2))[0]
        form = rng.choices((MASS, HELMHOLTZ, ADVDIFF, BURGERS, RESIDUAL), (1, 3, 3, 2, 1))[0]
        degree = rng.randint(1, 4)
        precision = rng.choices((FP64, TF32X3, BF16X3, TF32, BF16), (6, 6, 1, 1, 1))[0]
        ncells = int(math.exp(rng.uniform(math.log(300), math.log(1600000))))
        permute = rng.random() < 0.25
        if op == "batch":
            case = _case(op, HELMHOLTZ, 4, TET, rng.choice((TF32X3, BF16X3)), max(4096, ncells // 2 * 2))
        else:
            case = _case(op, form, degree, cell, precision, ncells, permute)
            if op == "csr" and (form == RESIDUAL or not coffee.csr_supported(form, degree, cell, precision)):
                continue
            if op == "adjoint" and (cell == PRISM or form >= BURGERS):
                continue
            if not coffee.supported(form, degree, cell, precision):
                continue
            if op == "csr" and _rows(form, degree, cell) > 60:  # the pattern of longer rows is not built
                continue
        w = work(case)
        # no more than the largest listed cases: 2.6 GB, 0.2 TFLOP on the tensor cores, in double 20 GFLOP on
        # simplices and 3 GFLOP on prisms
        most = 200e9 if precision != FP64 or op == "batch" else 3e9 if cell == PRISM else 20e9
        if w["bytes"] <= (1e9 if op in ("csr", "adjoint") else 2.6e9) and w["flops"] <= most:
            return case


# ------------------------------------------------------------------ meshes (on the GPU)
_PERMS3 = list(itertools.permutations(range(3)))


def _dim(cell):
    return 2 if cell == TRI else 3


def _ns(cell, k):
    t = (k + 1) * (k + 2) // 2
    return t if cell == TRI else t * (k + 3) // 3 if cell == TET else t * (k + 1)


def _rows(form, degree, cell):
    return _ns(cell, degree) * (_dim(cell) if form >= BURGERS else 1)


def _nvc(cell):
    return (3, 4, 6)[cell]


def _shape(cell, ncells):
    """Cells per axis of the smallest square or cube that holds ncells cells."""
    per, d = (2, 6, 2)[cell], _dim(cell)
    n = max(1, round((ncells / per) ** (1.0 / d)) - 1)
    while per * n ** d < ncells:
        n += 1
    if cell == TET:  # fewer layers where the last ones would stay empty
        return n, n, -(-ncells // (per * n * n))
    return (n,) * d


def _corners(cell):
    """Integer offsets [cells per square or cube, vertices, d]."""
    if cell == TRI:
        return np.array([[(0, 0), (1, 0), (1, 1)], [(0, 0), (1, 1), (0, 1)]])
    if cell == TET:
        eye = np.eye(3, dtype=int)
        return np.array([[(0, 0, 0), eye[s[0]], eye[s[0]] + eye[s[1]], (1, 1, 1)] for s in _PERMS3])
    tris = (((0, 0, 0), (1, 0, 0), (1, 1, 0)), ((0, 0, 0), (1, 1, 0), (0, 1, 0)))
    return np.array([list(t) + [(x, y, 1) for x, y, _ in t] for t in tris])


class _Mesh:
    def __init__(self, cell, ncells, gen):
        self.cell, self.ncells, self.d = cell, ncells, _dim(cell)
        self.shape = _shape(cell, ncells)
        off = torch.from_numpy(_corners(cell)).to(DEV)
        e = torch.arange(ncells, device=DEV)
        cube, origin = e // off.shape[0], []
        for n in self.shape:
            origin.append(cube % n)
            cube = cube // n
        self.grid = torch.stack(origin, 1)[:, None, :] + off[e % off.shape[0]]  # [ncells, nvc, d]
        axes = [torch.arange(n + 1, device=DEV) for n in self.shape]
        pts = torch.stack(torch.meshgrid(*reversed(axes), indexing="ij")[::-1], -1).reshape(-1, self.d)
        n = torch.tensor(self.shape, device=DEV)
        inside = ((pts > 0) & (pts < n)).all(1, keepdim=True)
        p = 0.2 if cell == TRI else 0.15
        noise = (2 * torch.rand(pts.shape, generator=gen, device=DEV, dtype=torch.float64) - 1) * p
        self.coords = ((pts + noise * inside) / n).contiguous()
        self.cell2vert = self._number(self.grid, 1).to(torch.int32).contiguous()

    def _number(self, pts, k):
        ids, mult = torch.zeros(pts.shape[:-1], dtype=torch.int64, device=DEV), 1
        for a, n in enumerate(self.shape):
            ids += pts[..., a] * mult
            mult *= k * n + 1
        return ids

    def nodes(self, k, gen=None):
        """(cell2dof [ncells, ns] int32, number of nodes); numbered at random with gen."""
        V0 = self.grid[:, 0]
        cols = []
        for m in _lattice(self.cell, k):  # (a, b[, c]); on prisms E[2] leads to the top triangle
            x = k * V0
            for a, i in enumerate(m):
                if i:
                    x = x + i * (self.grid[:, a + 1] - V0)
            cols.append(self._number(x, k))
        ids, nn = torch.stack(cols, 1), math.prod(k * n + 1 for n in self.shape)
        if gen is not None:
            ids = torch.randperm(nn, generator=gen, device=DEV)[ids]
        return ids.to(torch.int32).contiguous(), nn


def _lattice(cell, k):
    tri = [(a, b) for b in range(k + 1) for a in range(k - b + 1)]
    if cell == TRI:
        return tri
    if cell == PRISM:
        return [(a, b, c) for c in range(k + 1) for a, b in tri]
    return [(a, b, c) for c in range(k + 1) for b in range(k - c + 1) for a in range(k - b - c + 1)]


def _inputs(case, seed):
    """Mesh, coefficient rows and their map, from the seed alone."""
    gen = torch.Generator(DEV).manual_seed(seed)
    mesh = _Mesh(case["cell"], case["ncells"], gen)
    coef = c2d = None
    f64 = {"generator": gen, "device": DEV, "dtype": torch.float64}
    if case["form"] == ADVDIFF:
        c2d, nn = mesh.nodes(1, gen if case["permute"] else None)
        eps = 0.5 + torch.rand(nn, 1, **f64)
        coef = torch.cat([eps, 2 * torch.rand(nn, mesh.d, **f64) - 1], 1).reshape(-1)
    elif case["form"] >= BURGERS:
        c2d, nn = mesh.nodes(case["degree"], gen if case["permute"] else None)
        coef = torch.randn(nn, mesh.d, **f64).reshape(-1)
    return mesh, coef, c2d, gen


def _batch_groups(case, seed):
    """Every (form, degree) of half the cells as triangles P1-P4 and half as tetrahedra P1-P3, Zipf counts."""
    half = case["ncells"] // 2
    got = []
    for cell, degrees, sd in ((TRI, (1, 2, 3, 4), 4), (TET, (1, 2, 3), 5)):
        sub = _case("forward", ADVDIFF, 1, cell, case["precision"], half)
        mesh, coef, c2d, _ = _inputs(sub, seed + cell)
        kinds = [(f, k) for k in degrees for f in (MASS, HELMHOLTZ, ADVDIFF)]
        counts = meshgen.zipf_counts(len(kinds), half, s=1.0, seed=sd)
        start = 0
        for (f, k), n in zip(kinds, counts):
            n = int(n)
            if n:
                got.append({"form": f, "degree": k, "cell": cell, "coords": mesh.coords,
                            "cell2vert": mesh.cell2vert[start:start + n].contiguous(),
                            "coef": coef if f == ADVDIFF else None,
                            "cell2dof": c2d[start:start + n].contiguous() if f == ADVDIFF else None})
            start += n
    return got


def _csr_pattern_input(case, mesh):
    l2g, nn = mesh.nodes(case["degree"])
    if case["form"] == BURGERS:
        l2g, nn = coffee.binding.vector_l2g(l2g, nn, mesh.d), nn * mesh.d
    return l2g, nn


# ------------------------------------------------------------------ what a program has in hand, and one pass
def prepare(case, seed):
    if case["op"] == "batch":
        groups = _batch_groups(case, seed)
        return {"op": "batch", "plan": coffee.BatchPlan(groups, precision=case["precision"])}
    mesh, coef, c2d, gen = _inputs(case, seed)
    form, degree, cell, precision = (case[k] for k in ("form", "degree", "cell", "precision"))
    n = _rows(form, degree, cell)
    odt = torch.float64 if precision == FP64 else torch.float32
    s = {"op": case["op"], "what": (form, degree, cell), "precision": precision, "coords": mesh.coords,
         "c2v": mesh.cell2vert, "coef": coef, "c2d": c2d}
    if case["op"] == "adjoint":
        s["coords"] = mesh.coords.requires_grad_()
        s["wrt"] = [s["coords"]]
        if coef is not None:
            s["wrt"].append(coef.requires_grad_())
        s["dout"] = torch.randn(case["ncells"], n, n, generator=gen, device=DEV, dtype=odt)
        return s
    if case["op"] == "csr":
        s["matrix"] = coffee.CsrMatrix(*_csr_pattern_input(case, mesh))
        s["vals"] = torch.empty(s["matrix"].nnz, device=DEV, dtype=odt)
        return s
    s["out"] = torch.empty((case["ncells"], n) if form == RESIDUAL else (case["ncells"], n, n), device=DEV, dtype=odt)
    s["cf"] = torch.empty(coef.shape, device=DEV) if coef is not None and precision != FP64 else None
    s["xs"] = None
    if precision != FP64 and cell != PRISM and (degree == 1 or form == RESIDUAL):
        s["xs"] = torch.empty(tuple(mesh.coords.shape) + (2,), device=DEV)
    return s


def run(s):
    if s["op"] == "batch":
        return s["plan"].launch()
    form, degree, cell = s["what"]
    if s["op"] == "adjoint":
        out = coffee.AssembleFn.apply(s["coords"], s["coef"], s["c2v"], s["c2d"], form, degree, cell, s["precision"])
        return [out.detach()] + list(torch.autograd.grad(out, s["wrt"], s["dout"]))
    if s["op"] == "csr":
        s["vals"].zero_()
        return s["matrix"].assemble(form, degree, cell, s["coords"], s["c2v"], s["coef"], s["c2d"],
                                    precision=s["precision"], vals=s["vals"])
    if s["xs"] is not None:
        coffee.split_coords(s["coords"], out=s["xs"])
    if s["cf"] is not None:
        coffee.round_coef(s["coef"], out=s["cf"])
    return coffee.assemble(form, degree, cell, s["coords"], s["c2v"], s["coef"], s["c2d"], precision=s["precision"],
                           out=s["out"], coords_split=s["xs"], coef_f32=s["cf"])


# ------------------------------------------------------------------ bytes and operations of one pass
def _cell_flops(form, degree, cell):
    """Operations of one cell's contraction with the quadrature summed beforehand (prisms: summed over the
    points direction by direction), which is what the results cannot do without on this path."""
    d, ns = _dim(cell), _ns(cell, degree)
    P = d * (d + 1) // 2
    if cell == PRISM:  # points x factors x (z pairs, then triangle pairs), one field per geometric factor
        b = form >= BURGERS
        q, t, z = ((3 * degree + 3) // 2 if b else degree + 2), (degree + 1) * (degree + 2) // 2, degree + 1
        fields = {MASS: 1, HELMHOLTZ: 7, ADVDIFF: 9, BURGERS: 18, RESIDUAL: 12}[form]
        if form == RESIDUAL:
            return 2 * fields * (q ** 3 * z + q * q * z * t)
        return 2 * fields * (q ** 3 * z * z + q * q * z * z * t * t)
    if form == RESIDUAL:
        return 2 * (ns * ns * (ns * d + P) + ns * ns * d)
    if form == BURGERS:
        return 2 * ns * ns * (d * d * ns * d + ns * d + P)
    return 2 * ns * ns * {MASS: 1, HELMHOLTZ: 1 + P, ADVDIFF: (d + 1) * P + (d + 1) * d}[form]


def work(case):
    if case["op"] == "batch":
        total = {"bytes": 0, "flops": 0}
        half = case["ncells"] // 2
        for cell, degrees in ((TRI, (1, 2, 3, 4)), (TET, (1, 2, 3))):  # Zipf counts: about the mean of the kinds
            kinds = [(f, k) for k in degrees for f in (MASS, HELMHOLTZ, ADVDIFF)]
            for f, k in kinds:
                w = work(_case("forward", f, k, cell, case["precision"], max(1, half // len(kinds))))
                total = {m: total[m] + w[m] for m in total}
        return total
    form, degree, cell, n = case["form"], case["degree"], case["cell"], case["ncells"]
    d, rows = _dim(cell), _rows(form, degree, cell)
    size = 8 if case["precision"] == FP64 else 4
    shape = _shape(cell, n)
    nverts = math.prod(m + 1 for m in shape)
    read = n * 4 * _nvc(cell) + 8 * d * nverts
    if form == ADVDIFF:
        read += n * 4 * _nvc(cell) + 8 * (d + 1) * nverts
    elif form >= BURGERS:
        read += n * 4 * _ns(cell, degree) + 8 * d * math.prod(degree * m + 1 for m in shape)
    flops = n * _cell_flops(form, degree, cell)
    entries = n * (rows if form == RESIDUAL else rows * rows)
    if case["op"] == "csr":  # the entry map, and every value once (about 0.55 values to an entry)
        return {"bytes": read + 4 * entries + size * 0.55 * entries, "flops": flops + entries}
    if case["op"] == "adjoint":  # dA read beside A written, the gradients written, two contractions
        grads = 8 * d * nverts + (8 * (d + 1) * nverts if form == ADVDIFF else 0)
        return {"bytes": 2 * read + 2 * size * entries + grads, "flops": 2 * flops}
    return {"bytes": read + size * entries, "flops": flops}


# ------------------------------------------------------------------ the same in 64 bits, by the definitions
def _gauss01(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1), 0.5 * w


def _simplex_rule(d, n):
    x, w = _gauss01(n)
    pts, wts = [], []
    for i in itertools.product(range(n), repeat=d):
        s, p, rest = float(np.prod(w[list(i)])), [], 1.0
        for a in range(d):  # Duffy's map: every coordinate takes its share of what the earlier ones left
            p.append(rest * x[i[a]])
            s *= rest if a else 1.0
            rest *= 1 - x[i[a]]
        # the measure of the map is the product of the remaining lengths
        pts.append(p)
        wts.append(s)
    return np.array(pts), np.array(wts)


def _monomials(exps, x):
    """Values [points, monomials] and derivatives [points, monomials, d]."""
    v = np.ones((len(x), len(exps)))
    g = np.zeros((len(x), len(exps), x.shape[1]))
    for j, e in enumerate(exps):
        v[:, j] = np.prod([x[:, a] ** e[a] for a in range(len(e))], axis=0)
        for a in range(len(e)):
            if e[a]:
                f = [m - (i == a) for i, m in enumerate(e)]
                g[:, j, a] = e[a] * np.prod([x[:, i] ** f[i] for i in range(len(f))], axis=0)
    return v, g


def _basis(cell, k, x):
    """Lagrange basis on the lattice nodes (the prism's: triangle lattice times the levels), by Vandermonde."""
    exps = _lattice(cell, k)
    C = np.linalg.inv(_monomials(exps, np.array(exps, dtype=float) / k)[0])
    v, g = _monomials(exps, x)
    return v @ C, np.einsum("qmd,mi->qid", g, C)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _adjugate(J):
    """(adjugate [.., d, d], det) of J, K = adj / det."""
    if J.shape[-1] == 2:
        a, b, c, d = J[..., 0, 0], J[..., 0, 1], J[..., 1, 0], J[..., 1, 1]
        return torch.stack([torch.stack([d, -b], -1), torch.stack([-c, a], -1)], -2), a * d - b * c
    c0, c1, c2 = J.unbind(-1)
    A = torch.stack([torch.linalg.cross(c1, c2), torch.linalg.cross(c2, c0), torch.linalg.cross(c0, c1)], -2)
    return A, (c0 * A[..., 0, :]).sum(-1)


def _pairs(d):
    return [(a, b) for a in range(d) for b in range(a, d)]


def _simplex_factors(form, mesh, coords, coef, c2d):
    """Per-cell factors [n, K] of the element matrix's terms (MASS, HELMHOLTZ, ADVDIFF)."""
    d = mesh.d
    X = coords[mesh.cell2vert.long()]
    adj, det = _adjugate((X[:, 1:] - X[:, :1]).transpose(1, 2))
    H = torch.stack([(adj[:, a] * adj[:, b]).sum(-1) / det.abs() for a, b in _pairs(d)], 1)
    if form == MASS:
        return det.abs()[:, None]
    if form == HELMHOLTZ:
        return torch.cat([det.abs()[:, None], H], 1)
    rows = coef.reshape(-1, d + 1)[c2d.long()]
    P = adj * torch.sign(det)[:, None, None]
    stiff = (rows[:, :, :1] * H[:, None, :]).reshape(len(H), -1)
    adv = torch.einsum("nar,nvr->nva", P, rows[:, :, 1:]).reshape(len(H), -1)
    return torch.cat([stiff, adv], 1)


def _simplex_tensor(form, k, cell):
    d = _dim(cell)
    x, w = _simplex_rule(d, k + 3)
    phi, g = _basis(cell, k, x)
    lam = _basis(cell, 1, x)[0]

    def stiff(wq):
        return [sum(np.einsum("q,qi,qj->ij", wq, g[:, :, p], g[:, :, r]) for p, r in {(a, b), (b, a)})
                for a, b in _pairs(d)]

    if form == MASS:
        T = [np.einsum("q,qi,qj->ij", w, phi, phi)]
    elif form == HELMHOLTZ:
        T = [np.einsum("q,qi,qj->ij", w, phi, phi)] + stiff(w)
    else:
        T = [t for v in range(d + 1) for t in stiff(w * lam[:, v])]
        T += [np.einsum("q,qi,qj->ij", w * lam[:, v], phi, g[:, :, a]) for v in range(d + 1) for a in range(d)]
    return _dev(np.stack(T).reshape(len(T), -1))


def _burgers_simplex(case, mesh, coords, coef, c2d):
    d, k, cell = mesh.d, case["degree"], case["cell"]
    ns = _ns(cell, k)
    x, w = _simplex_rule(d, (3 * k + 4) // 2 + 1)
    phi, g = _basis(cell, k, x)
    X = coords[mesh.cell2vert.long()]
    adj, det = _adjugate((X[:, 1:] - X[:, :1]).transpose(1, 2))
    P = adj * torch.sign(det)[:, None, None]
    u = coef.reshape(-1, d)[c2d.long()]  # [n, ns, d]
    nu_h = torch.stack([NU * (adj[:, a] * adj[:, b]).sum(-1) / det.abs() for a, b in _pairs(d)], 1)
    T1 = _dev(np.einsum("q,qra,qi,qj->raij", w, g, phi, phi).reshape(ns * d, -1))
    T2 = _dev(np.einsum("q,qr,qi,qja->raij", w, phi, phi, g).reshape(ns * d, -1))
    T3 = _dev(np.stack([sum(np.einsum("q,qi,qj->ij", w, g[:, :, p], g[:, :, r]) for p, r in {(a, b), (b, a)})
                        for a, b in _pairs(d)]).reshape(len(_pairs(d)), -1))
    n = len(X)
    C = torch.einsum("nrc,nac->nra", u, P).reshape(n, -1) @ T2 + nu_h @ T3
    if case["form"] == RESIDUAL:
        return torch.einsum("nis,nsc->nci", C.reshape(n, ns, ns), u).reshape(n, -1)
    out = torch.empty(n, d, ns, d, ns, device=DEV, dtype=torch.float64)
    for ci in range(d):
        for cj in range(d):
            F = (u[:, :, None, ci] * P[:, None, :, cj]).reshape(n, -1)
            B = F @ T1
            out[:, ci, :, cj, :] = (B + C if ci == cj else B).reshape(n, ns, ns)
    return out.reshape(n, d * ns, d * ns)


def _prism_points(n):
    x, w = _gauss01(n)
    pts = [(s, t * (1 - s), z) for z in x for s in x for t in x]
    wts = [ws * wt * wz * (1 - s) for wz in w for s, ws in zip(x, w) for wt in w]
    return np.array(pts), np.array(wts)


def _prism_geometry(X, x):
    """Adjugate and determinant [n, Q, ..] of the degree-1 map at the points x; the degree-1 functions there."""
    phi, g = _basis(PRISM, 1, x)
    adj, det = _adjugate(torch.einsum("nvr,qvc->nqrc", X, _dev(g)))
    return adj, det, _dev(phi)


def _prism(case, mesh, coords, coef, c2d):
    """Element matrices (vectors) by the rule that the package states for prisms, some cells at a time."""
    form, k = case["form"], case["degree"]
    x, w = _prism_points((3 * k + 3) // 2 if form >= BURGERS else k + 2)
    phi, g = _basis(PRISM, k, x)
    ns, Q, n = phi.shape[1], len(w), mesh.ncells
    W, ph, gr = _dev(w), _dev(phi), _dev(g)
    rows = _rows(form, k, PRISM)
    out = torch.empty((n, rows) if form == RESIDUAL else (n, rows, rows), device=DEV, dtype=torch.float64)
    pp = torch.einsum("qi,qj->qij", ph, ph).reshape(Q, -1)
    pg = torch.einsum("qi,qja->aqij", ph, gr).reshape(3, Q, -1)
    gg = [(torch.einsum("qi,qj->qij", gr[:, :, a], gr[:, :, b]) + (0 if a == b else torch.einsum(
        "qi,qj->qij", gr[:, :, b], gr[:, :, a]))).reshape(Q, -1) for a, b in _pairs(3)]
    step = max(1, int(2e8 // (Q * 30 + rows * rows)))
    for c0 in range(0, n, step):
        sel = slice(c0, c0 + step)
        adj, det, lam = _prism_geometry(coords[mesh.cell2vert[sel].long()], x)
        wd = W * det.abs()
        H = [W * (adj[:, :, a] * adj[:, :, b]).sum(-1) / det.abs() for a, b in _pairs(3)]
        P = adj * (W * torch.sign(det))[..., None, None]
        if form < BURGERS:
            if form == ADVDIFF:
                r = coef.reshape(-1, 4)[c2d[sel].long()]
                eps, b = r[..., 0] @ lam.T, torch.einsum("nvr,qv->nqr", r[..., 1:], lam)
                H = [h * eps for h in H]
                A = sum(torch.einsum("nqr,nqr->nq", P[:, :, a], b) @ pg[a] for a in range(3))
            else:
                A = wd @ pp
            if form != MASS:
                A = A + sum(h @ t for h, t in zip(H, gg))
            out[sel] = A.reshape(-1, ns, ns)
            continue
        u = coef.reshape(-1, 3)[c2d[sel].long()]
        uq = torch.einsum("qr,nrc->nqc", ph, u)
        du = torch.einsum("qra,nrc->nqca", gr, u)  # reference derivatives of the components
        M = torch.einsum("nqca,nqad->nqcd", du, P)  # w |det| d_cj u_ci
        beta = torch.einsum("nqac,nqc->nqa", P, uq)
        if form == RESIDUAL:
            adv = torch.einsum("nqcd,nqd->nqc", M, uq)
            V = torch.einsum("nqar,nqbr->nqab", adj, adj) * (W * NU / det.abs())[..., None, None]
            flux = torch.einsum("nqab,nqcb->nqca", V, du)
            R = torch.einsum("nqc,qi->nci", adv, ph) + torch.einsum("nqca,qia->nci", flux, gr)
            out[sel] = R.reshape(-1, rows)
            continue
        D = sum(beta[:, :, a] @ pg[a] for a in range(3)) + sum((NU * h) @ t for h, t in zip(H, gg))
        o = out[sel].view(-1, 3, ns, 3, ns)
        for ci in range(3):
            for cj in range(3):
                B = M[:, :, ci, cj].contiguous() @ pp
                o[:, ci, :, cj, :] = (B + D if ci == cj else B).reshape(-1, ns, ns)
    return out


def _matrices(case, mesh, coords, coef, c2d):
    if case["cell"] == PRISM:
        return _prism(case, mesh, coords, coef, c2d)
    if case["form"] >= BURGERS:
        return _burgers_simplex(case, mesh, coords, coef, c2d)
    G = _simplex_factors(case["form"], mesh, coords, coef, c2d)
    ns = _ns(case["cell"], case["degree"])
    return (G @ _simplex_tensor(case["form"], case["degree"], case["cell"])).reshape(-1, ns, ns)


class _Part:
    """The cells of one group of a batch, as the functions above take a mesh."""

    def __init__(self, g):
        self.d, self.cell2vert, self.ncells = _dim(g["cell"]), g["cell2vert"], g["cell2vert"].shape[0]


def exact(case, seed):
    if case["op"] == "batch":
        return [_matrices(g, _Part(g), g["coords"], g["coef"], g["cell2dof"]) for g in _batch_groups(case, seed)]
    mesh, coef, c2d, gen = _inputs(case, seed)
    if case["op"] == "adjoint":
        odt = torch.float64 if case["precision"] == FP64 else torch.float32
        n = _rows(case["form"], case["degree"], case["cell"])
        dout = torch.randn(mesh.ncells, n, n, generator=gen, device=DEV, dtype=odt).double()
        wrt = [mesh.coords.requires_grad_()] + ([coef.requires_grad_()] if coef is not None else [])
        A = _matrices(case, mesh, mesh.coords, coef, c2d)
        return [A.detach()] + list(torch.autograd.grad(A, wrt, dout))
    A = _matrices(case, mesh, mesh.coords, coef, c2d)
    if case["op"] == "forward":
        return A
    l2g, nn = _csr_pattern_input(case, mesh)
    # sorted (row, column) pairs, as a CSR matrix orders its values; some cells at a time
    l2g, uniq = l2g.long(), torch.empty(0, dtype=torch.int64, device=DEV)
    step = max(1, int(5e7 // l2g.shape[1] ** 2))
    keys = [(l2g[i:i + step, :, None] * nn + l2g[i:i + step, None, :]).reshape(-1) for i in range(0, len(l2g), step)]
    for key in keys:
        uniq = torch.unique(torch.cat([uniq, torch.unique(key)]))
    vals = torch.zeros(len(uniq), device=DEV, dtype=torch.float64)
    flat = A.reshape(-1)
    at = 0
    for key in keys:
        vals.index_add_(0, torch.searchsorted(uniq, key), flat[at:at + len(key)])
        at += len(key)
    return vals
