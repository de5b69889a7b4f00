"""Timed cases of the framework, each one pass through its public entry points.

A case is a dict of plain values.  Its ``kind`` says which entry points a pass
calls:

* ``forward64``  element matrices from FP64 coordinates, FP64 results
* ``step``       forward, then the adjoint of one mesh (one optimisation or
  training step): ``api`` "autograd" through ``Mesh.integrate`` and
  ``torch.autograd.grad``, "calls" through ``integrate_fwd`` /
  ``integrate_bwd`` with the buffers, the workspace and the saved determinant
  that a solver keeps
* ``assemble``   global sparse matrix of element matrices in hand
* ``curved``     forward and adjoint on non-affine (quadratic-geometry) elements
* ``batch``      forward and adjoint of many meshes of mixed forms in one call

Meshes are the library's own benchmark shapes: jittered unit squares (n x n
cells, 2 triangles each) and unit cubes (n^3 cells, 6 tetrahedra each), with
5% sliver elements where ``slivers`` says so, warped for the curved elements;
``order`` "shuffled" puts elements and vertices in random order, as a mesh
from an unstructured generator arrives.  They are made on the GPU from the
seed alone.  ``exact`` integrates the same inputs in 64 bits with plain torch.
"""
import itertools
import math

import torch

import paper_1103_0066_gb300 as fem

DEV = "cuda"
FORMS = {"P1": fem.LAPLACE_P1, "P2": fem.LAPLACE_P2, "ELASTIC": fem.ELASTIC_P1, "P1_W1": fem.LAPLACE_P1_W1,
         "P2_W1": fem.LAPLACE_P2_W1, "DIV_P2P1": fem.DIV_P2P1}
CURVED = {"P1": fem.LAPLACE_P1_ISO, "P2": fem.LAPLACE_P2_ISO}
CONTRACT = {"f32": fem.CONTRACT_F32, "bf16x3": fem.CONTRACT_BF16X3}


def listed():
    return [
        # the smallest use: a 2D model problem in double precision, bound by the call itself
        dict(name="tri_p1_f64_small", kind="forward64", dim=2, form="P1", n=64),
        # a small 3D mesh inside an optimisation loop, differentiated by autograd
        dict(name="tet_p1_autograd_small", kind="step", api="autograd", dim=3, form="P1", n=16, order="grid",
             slivers=0.05, coef=True, contract="f32"),
        # the headline: 12.6M tetrahedra with slivers, forward and adjoint
        dict(name="tet_p1_step_large", kind="step", api="calls", dim=3, form="P1", n=128, order="grid", slivers=0.05,
             coef=False, contract="f32"),
        # the same step on an unstructured mesh as its generator left it
        dict(name="tet_p1_step_shuffled", kind="step", api="calls", dim=3, form="P1", n=96, order="shuffled",
             slivers=0.05, coef=False, contract="f32"),
        # plane elasticity, an odd mesh of 2.1M triangles, coefficient gradient too
        dict(name="tri_elastic_step", kind="step", api="calls", dim=2, form="ELASTIC", n=1023, order="grid",
             slivers=0.0, coef=True, contract="f32"),
        # 3D elasticity with a material coefficient, ragged size
        dict(name="tet_elastic_step", kind="step", api="calls", dim=3, form="ELASTIC", n=61, order="grid",
             slivers=0.05, coef=True, contract="f32"),
        # second-order diffusion with a continuous coefficient field
        dict(name="tet_p2_w1_step", kind="step", api="calls", dim=3, form="P2_W1", n=72, order="grid", slivers=0.05,
             coef=True, contract="f32"),
        # global matrices of the three unknown layouts: vertices, vertices and edges, d x d blocks
        dict(name="assemble_p1", kind="assemble", dim=3, form="P1", n=96, order="grid"),
        dict(name="assemble_p2", kind="assemble", dim=3, form="P2", n=61, order="grid"),
        dict(name="assemble_elastic", kind="assemble", dim=3, form="ELASTIC", n=56, order="grid"),
        # second-order elements on curved geometry, shape derivatives included
        dict(name="curved_p2_step", kind="curved", dim=3, form="P2", n=64, order="grid", contract="f32"),
        # parameter study: many meshes of uneven size and mixed forms
        dict(name="batch_mixed", kind="batch", meshes=20, e_lo=1000, e_hi=800000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward64", "step", "step", "step", "assemble", "assemble", "curved", "batch"])
    dim = rng.choice([2, 3, 3])
    order = rng.choice(["grid", "grid", "shuffled"])
    if kind == "forward64":
        return dict(kind=kind, dim=dim, form=rng.choice(["P1", "P2", "ELASTIC"]),
                    n=_log_int(rng, 24, 400) if dim == 2 else _log_int(rng, 6, 32))
    if kind == "step":
        form = rng.choice(["P1", "P1", "P2", "ELASTIC", "P1_W1", "P2_W1", "DIV_P2P1"])
        contract = "f32"
        if dim == 3 and form in ("P2", "ELASTIC", "P2_W1"):
            contract = rng.choice(["f32", "bf16x3"])
        if dim == 2:
            n = _log_int(rng, 24, 2000 if form in ("P1", "P1_W1") else 1023)
        else:
            n = _log_int(rng, 6, 96 if form in ("P1", "P1_W1") else 61)
        return dict(kind=kind, api=rng.choice(["autograd", "calls"]), dim=dim, form=form, n=n, order=order,
                    slivers=rng.choice([0.0, 0.05]) if dim == 3 else 0.0,
                    coef=True if form.endswith("W1") else rng.choice([True, False]), contract=contract)
    if kind == "assemble":
        form = rng.choice(["P1", "P2", "ELASTIC"])
        return dict(kind=kind, dim=dim, form=form, order=order,
                    n=_log_int(rng, 32, 1000 if form == "P1" else 600) if dim == 2 else
                    _log_int(rng, 8, 80 if form == "P1" else 48))
    if kind == "curved":
        form = rng.choice(["P1", "P2"])
        return dict(kind=kind, dim=dim, form=form, order=order,
                    n=_log_int(rng, 24, 700) if dim == 2 else _log_int(rng, 6, 56),
                    contract=rng.choice(["f32", "bf16x3"]) if (dim, form) == (3, "P2") else "f32")
    return dict(kind=kind, meshes=rng.randint(6, 20), e_lo=1000, e_hi=_log_int(rng, 20000, 600000))


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _uniform(gen, *shape):
    return torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64)


def _square(n, gen):
    h = 1.0 / n
    i = torch.arange(n + 1, device=DEV)
    x = torch.stack([i.repeat(n + 1), i.repeat_interleave(n + 1)], 1).double() * h
    inner = ((x > 0.5 * h) & (x < 1 - 0.5 * h)).all(1, keepdim=True)
    x = x + inner * (0.4 * _uniform(gen, *x.shape) - 0.2) * h
    c = torch.arange(n, device=DEV)
    v = (c[:, None] * (n + 1) + c[None, :]).reshape(-1)
    tri = torch.stack([torch.stack([v, v + 1, v + n + 2], 1), torch.stack([v, v + n + 2, v + n + 1], 1)], 1)
    return x, tri.reshape(-1, 3)


def _cube(n, gen, slivers):
    h, m = 1.0 / n, n + 1
    i = torch.arange(m, device=DEV)
    k, j, i = torch.meshgrid(i, i, i, indexing="ij")
    x = torch.stack([i, j, k], -1).reshape(-1, 3).double() * h
    inner = ((x > 0.5 * h) & (x < 1 - 0.5 * h)).all(1, keepdim=True)
    x = (x + inner * (0.3 * _uniform(gen, *x.shape) - 0.15) * h).float().double()
    c = torch.arange(n, device=DEV)
    base = ((c[:, None, None] * m + c[None, :, None]) * m + c).reshape(-1)
    step = (1, m, m * m)
    tets = []
    for p in itertools.permutations(range(3)):
        v = [base, base + step[p[0]], base + step[p[0]] + step[p[1]], base + sum(step)]
        if sum(p[a] > p[b] for a in range(3) for b in range(a + 1, 3)) % 2:
            v[2], v[3] = v[3], v[2]
        tets.append(torch.stack(v, 1))
    conn = torch.stack(tets, 1).reshape(-1, 4)
    if slivers:
        E, V = conn.shape[0], x.shape[0]
        ns = int(round(slivers * E))
        el = torch.randperm(E, generator=gen, device=DEV)[:ns].sort().values
        loc = torch.randint(0, 4, (ns,), generator=gen, device=DEV)
        P = x[conn[el]]
        others = torch.tensor([[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]], device=DEV)[loc]
        a, b, c = (P[torch.arange(ns, device=DEV), others[:, q]] for q in range(3))
        y = P[torch.arange(ns, device=DEV), loc]
        nrm = torch.linalg.cross(b - a, c - a)
        nrm = nrm / nrm.norm(dim=1, keepdim=True)
        height = ((y - a) * nrm).sum(1, keepdim=True)
        r = 10.0 ** (-2 - 2 * _uniform(gen, ns, 1))
        x = torch.cat([x, y - (1 - r) * height * nrm])
        conn[el, loc] = V + torch.arange(ns, device=DEV)
    return x, conn


def _mesh(case, gen, slivers=0.0):
    """(coordinates FP64 [V][d], connectivity int32 [E][d+1]) of a case."""
    x, conn = _square(case["n"], gen) if case["dim"] == 2 else _cube(case["n"], gen, slivers)
    if case.get("order") == "shuffled":
        conn = conn[torch.randperm(conn.shape[0], generator=gen, device=DEV)]
        new = torch.randperm(x.shape[0], generator=gen, device=DEV)
        y = torch.empty_like(x)
        y[new] = x
        x, conn = y, new[conn]
    return x, conn.int().contiguous()


def _edges(d):
    return [(a, b) for a in range(d + 1) for b in range(a + 1, d + 1)]


def _curved_mesh(case, gen):
    def warp(x):
        s, o = torch.sin(math.pi * x), x.clone()
        for a in range(x.shape[-1]):
            o[..., a] += 0.05 * math.prod([s[..., b] for b in range(x.shape[-1]) if b != a])
        return o
    x, conn = _mesh(case, gen)
    P = x[conn.long()]
    mid = torch.stack([0.5 * (P[:, a] + P[:, b]) for a, b in _edges(case["dim"])], 1)
    return warp(x).float(), conn, warp(mid).float()


def _lognormal(gen, n):
    return torch.exp(torch.randn(n, generator=gen, device=DEV))


def _step_inputs(case, seed):
    gen = _gen(seed)
    x, conn = _mesh(case, gen, case["slivers"])
    x = x.float()
    coef = _lognormal(gen, x.shape[0] if case["form"].endswith("W1") else conn.shape[0]) if case["coef"] else None
    dA = torch.randn((conn.shape[0],) + _shape(case["form"], case["dim"]), generator=gen, device=DEV)
    return x, conn, coef, dA


def _assemble_inputs(case, seed):
    """Mesh and element matrices (64-bit integration, rounded once)."""
    gen = _gen(seed)
    x, conn = _mesh(case, gen)
    w = _lognormal(gen, conn.shape[0]).double()
    x = x.float()
    A = torch.empty((conn.shape[0],) + _shape(case["form"], case["dim"]), device=DEV)
    for s in _chunks(conn.shape[0]):
        A[s] = _affine(case["form"], x.double()[conn[s].long()], w[s]).float()
    return x, conn, A


def _batch_sizes(case):
    """Element counts, evenly spread over the logarithm, large and small ones mixed."""
    m = case["meshes"]
    t = [((q * 0.6180339887) % 1.0) for q in range(m)]
    return [int(round(case["e_lo"] * (case["e_hi"] / case["e_lo"]) ** x)) for x in t]


def _batch_inputs(case, seed):
    gen = _gen(seed)
    kinds = [(d, f) for d in (2, 3) for f in ("P1", "P2", "ELASTIC")]
    items = []
    for q, E in enumerate(_batch_sizes(case)):
        d, f = kinds[q % 6]
        n = math.ceil((E / 2) ** 0.5) if d == 2 else math.ceil((E / 6) ** (1 / 3) - 1e-9)
        x, conn = _mesh(dict(dim=d, n=max(n, 1)), gen)
        conn = conn[:E].contiguous()
        x = x[:int(conn.max()) + 1].float().contiguous()
        items.append((d, f, x, conn, _lognormal(gen, conn.shape[0]),
                      torch.randn((conn.shape[0],) + _shape(f, d), generator=gen, device=DEV)))
    return items


def prepare(case, seed):
    kind = case["kind"]
    if kind == "forward64":
        x, conn = _mesh(case, _gen(seed))
        return dict(kind=kind, x=x, conn=conn, form=FORMS[case["form"]])
    if kind == "step":
        x, conn, coef, dA = _step_inputs(case, seed)
        form = FORMS[case["form"]]
        mesh = fem.Mesh(x, conn)
        st = dict(kind=kind, api=case["api"], x=x, conn=conn, coef=coef, dA=dA, form=form, mesh=mesh,
                  contract=CONTRACT[case["contract"]], ws=mesh.workspace(form))
        if case["api"] == "autograd":
            for t in (x, coef):
                if t is not None:
                    t.requires_grad_(True)
        else:
            st["A"] = torch.empty_like(dA)
            st["det"] = torch.empty(conn.shape[0], device=DEV) if case["contract"] == "f32" else None
            st["dx"] = torch.empty_like(x)
            st["dw"] = torch.empty_like(coef) if coef is not None else None
        return st
    if kind == "assemble":
        x, conn, A = _assemble_inputs(case, seed)
        asm = fem.Assembly(x, conn, FORMS[case["form"]])
        return dict(kind=kind, asm=asm, A=A)
    if kind == "curved":
        gen = _gen(seed)
        x, conn, mid = _curved_mesh(case, gen)
        form = CURVED[case["form"]]
        dA = torch.randn((conn.shape[0],) + _shape(case["form"], case["dim"]), generator=gen, device=DEV)
        return dict(kind=kind, x=x, conn=conn, mid=mid, dA=dA, form=form, contract=CONTRACT[case["contract"]],
                    ws=fem.Mesh(x, conn).workspace(form), A=torch.empty_like(dA), dx=torch.empty_like(x),
                    dmid=torch.empty_like(mid))
    items = []
    for d, f, x, conn, coef, dA in _batch_inputs(case, seed):
        items.append(dict(coords=x, conn=conn, form=FORMS[f], coef=coef, dA=dA, A=torch.empty_like(dA),
                          dcoords=torch.empty_like(x), dcoef=torch.empty_like(coef)))
    return dict(kind=kind, items=items, batch=fem.Batch(items))


def run(st):
    kind = st["kind"]
    if kind == "forward64":
        return fem.integrate_fwd(st["x"], st["conn"], st["form"], out_dtype=torch.float64)
    if kind == "step" and st["api"] == "autograd":
        A = st["mesh"].integrate(st["form"], st["coef"], contract=st["contract"])
        wrt = [t for t in (st["x"], st["coef"]) if t is not None]
        return [A.detach(), *torch.autograd.grad(A, wrt, st["dA"])]
    if kind == "step":
        A = fem.integrate_fwd(st["x"], st["conn"], st["form"], st["coef"], out=st["A"], contract=st["contract"],
                              det_out=st["det"])
        dx, dw = fem.integrate_bwd(st["x"], st["conn"], st["form"], st["dA"], st["coef"], ws=st["ws"],
                                   need_dcoef=st["coef"] is not None, dcoords=st["dx"], dcoef=st["dw"], det=st["det"])
        return [A, dx] if dw is None else [A, dx, dw]
    if kind == "assemble":
        return st["asm"].assemble(st["A"])
    if kind == "curved":
        A = fem.integrate_fwd_iso(st["x"], st["conn"], st["mid"], st["form"], out=st["A"], contract=st["contract"])
        dx, dmid, _ = fem.integrate_bwd_iso(st["x"], st["conn"], st["mid"], st["form"], st["dA"], ws=st["ws"],
                                            dcoords=st["dx"], dmid=st["dmid"], contract=st["contract"])
        return [A, dx, dmid]
    st["batch"].run()
    return [it[k] for it in st["items"] for k in ("A", "dcoords", "dcoef")]


# ---------------------------------------------------------------- what a pass cannot do without

def _nb(form, d):
    return (d + 1) * (d + 2) // 2 if form.startswith("P2") else d + 1


def _shape(form, d):
    if form == "DIV_P2P1":
        return d + 1, d * _nb("P2", d)
    n = _nb(form, d) * (d if form == "ELASTIC" else 1)
    return n, n


def _counts(case):
    """(elements, vertices) of a case's mesh."""
    n, d = case["n"], case["dim"]
    E = 2 * n * n if d == 2 else 6 * n ** 3
    return E, (n + 1) ** d + int(round(case.get("slivers", 0.0) * E))


def work(case):
    kind, d = case["kind"], case.get("dim")
    if kind == "batch":
        b = f = 0
        kinds = [(d, f) for d in (2, 3) for f in ("P1", "P2", "ELASTIC")]
        for q, E in enumerate(_batch_sizes(case)):
            d, form = kinds[q % 6]
            n = math.prod(_shape(form, d))
            b += E * (4 * (d + 1) + 8 * n + 8) + 8 * (E // 2 if d == 2 else E // 6) * d
            f += E * 2 * n * d * (d + 1)
        return {"bytes": b, "flops": f}
    E, V = _counts(case)
    n = math.prod(_shape(case["form"], d))
    if kind == "forward64":
        return {"bytes": E * (4 * (d + 1) + 8 * n) + 8 * V * d, "flops": E * n * d * (d + 1)}
    if kind == "step":
        coef = 8 * (V if case["form"].endswith("W1") else E) * case["coef"]
        return {"bytes": E * (4 * (d + 1) + 8 * n) + 8 * V * d + coef, "flops": E * 2 * n * d * (d + 1)}
    if kind == "curved":
        ne = d * (d + 1) // 2
        return {"bytes": E * (4 * (d + 1) + 8 * n + 8 * ne * d) + 8 * V * d,
                "flops": E * 4 * n * d * _nb("P2", d)}
    # entries of the global matrix: pairs of unknowns that share an element
    c = case["n"]
    edges = 3 * c * c + 2 * c if d == 2 else 3 * c * (c + 1) ** 2 + 3 * c * c * (c + 1) + c ** 3
    if case["form"] == "P2":
        faces = E if d == 2 else 1 - V + edges + E
        nnz, rows = V + 7 * edges + 12 * faces + (6 * E if d == 3 else 0), V + edges
    else:
        nnz, rows = V + 2 * edges, V
    block = d * d if case["form"] == "ELASTIC" else 1
    return {"bytes": E * (4 * (d + 1) + 4 * n) + 4 * nnz * block + 4 * rows, "flops": E * n}


# ---------------------------------------------------------------- 64-bit results in plain torch

def _chunks(E, size=1 << 19):
    return [slice(s, min(s + size, E)) for s in range(0, E, size)]


def _simplex_monomial(d, powers):
    return math.prod(math.factorial(p) for p in powers) / math.factorial(d + sum(powers))


def _poly(form, d):
    """Basis functions as polynomials in the barycentric coordinates: {powers: value}."""
    unit = lambda *ks: tuple(sum(k == q for k in ks) for q in range(d + 1))
    if not form.startswith("P2"):
        return [{unit(i): 1.0} for i in range(d + 1)]
    return ([{unit(i, i): 2.0, unit(i): -1.0} for i in range(d + 1)] + [{unit(a, b): 4.0} for a, b in _edges(d)])


def _diff(p, d, mu):
    """Derivative along the reference coordinate mu (lambda_0 = 1 - sum, lambda_{mu+1} = xi_mu)."""
    out = {}
    for powers, v in p.items():
        for k, sign in ((mu + 1, 1.0), (0, -1.0)):
            if powers[k]:
                q = tuple(x - (a == k) for a, x in enumerate(powers))
                out[q] = out.get(q, 0.0) + sign * v * powers[k]
    return out


def _integral(d, *polys):
    terms = {(0,) * (d + 1): 1.0}
    for p in polys:
        terms_new = {}
        for a, x in terms.items():
            for b, y in p.items():
                c = tuple(s + t for s, t in zip(a, b))
                terms_new[c] = terms_new.get(c, 0.0) + x * y
        terms = terms_new
    return sum(v * _simplex_monomial(d, k) for k, v in terms.items())


_TENSORS = {}


def _reference(what, form, d):
    """Reference tensors by exact integration of barycentric monomials."""
    key = (what, form, d)
    if key not in _TENSORS:
        phi = _poly("P2" if form == "DIV_P2P1" else form, d)
        D = [[_diff(p, d, m) for m in range(d)] for p in phi]
        lam = _poly("P1", d)
        N, R, L = range(len(phi)), range(d), range(d + 1)
        if what == "K":
            t = [[[[_integral(d, D[i][m], D[j][v]) for v in R] for m in R] for j in N] for i in N]
        elif what == "K_w1":
            t = [[[[[_integral(d, lam[k], D[i][m], D[j][v]) for v in R] for m in R] for k in L] for j in N] for i in N]
        elif what == "K_iso":
            t = [[[[[[_integral(d, lam[k], lam[q], D[i][m], D[j][v]) for v in R] for q in L] for m in R] for k in L]
                  for j in N] for i in N]
        else:
            t = [[[_integral(d, lam[i], D[j][m]) for m in R] for j in N] for i in L]
        _TENSORS[key] = torch.tensor(t, dtype=torch.float64, device=DEV)
    return _TENSORS[key]


def _det_inv(J):
    """Determinant and inverse of [..][d][d] matrices by cofactors."""
    d = J.shape[-1]
    if d == 2:
        a, b, c, e = J[..., 0, 0], J[..., 0, 1], J[..., 1, 0], J[..., 1, 1]
        adj = torch.stack([torch.stack([e, -b], -1), torch.stack([-c, a], -1)], -2)
        det = a * e - b * c
    else:
        r = [J[..., q, :] for q in range(3)]
        cr = [torch.linalg.cross(r[(q + 1) % 3], r[(q + 2) % 3]) for q in range(3)]
        adj = torch.stack(cr, -1)
        det = (r[0] * cr[0]).sum(-1)
    return det, adj / det[..., None, None]


def _affine(form, P, w):
    """Element matrices [e][rows][cols] of vertex positions P [e][d+1][d] (FP64)."""
    e, _, d = P.shape
    Et = P[:, 1:] - P[:, :1]                    # Et[mu][c] = dx_c / dxi_mu
    det, inv = _det_inv(Et)                     # inv[c][mu] = dxi_mu / dx_c
    vol = det.abs()
    if form in ("P1", "P2"):
        K = _reference("K", form, d)
        G = torch.einsum("ecm,ecv->emv", inv, inv) * (vol * w)[:, None, None]
        return (G.reshape(e, -1) @ K.reshape(K.shape[0] ** 2, -1).T).reshape(e, K.shape[0], -1)
    if form.endswith("W1"):
        K = _reference("K_w1", form[:2], d)
        G = torch.einsum("ek,ecm,ecv->ekmv", w, inv, inv) * vol[:, None, None, None]
        return (G.reshape(e, -1) @ K.reshape(K.shape[0] ** 2, -1).T).reshape(e, K.shape[0], -1)
    if form == "DIV_P2P1":
        K = _reference("K_div", form, d)
        B = torch.einsum("ijm,ecm->eicj", K, inv) * (vol * w)[:, None, None, None]
        return B.reshape(e, d + 1, -1)
    # symmetric-gradient elasticity: 1/2 (grad u : grad v + grad u : grad v^T)
    g = torch.cat([-inv.sum(2, keepdim=True), inv], 2)          # g[c][i]: physical gradient of lambda_i
    s = (vol * w / math.factorial(d))[:, None, None, None, None]
    lap = torch.einsum("eai,eaj->eij", g, g)
    eye = torch.eye(d, dtype=P.dtype, device=P.device)
    A = 0.5 * s * (torch.einsum("cb,eij->ecibj", eye, lap) + torch.einsum("ebi,ecj->ecibj", g, g))
    return A.reshape(e, d * (d + 1), -1)


def _curved(form, P, M):
    """Non-affine Laplacian: inverse Jacobian interpolated from its vertex values, |det J| at the centroid."""
    e, _, d = P.shape
    nodes = torch.cat([P, M], 1)
    phi = _poly("P2", d)
    at = lambda p, x: sum(v * math.prod(a ** b for a, b in zip(x, k)) for k, v in p.items())
    def grad_at(x):
        return torch.tensor([[at(_diff(p, d, m), x) for m in range(d)] for p in phi], dtype=P.dtype, device=P.device)
    T = torch.stack([grad_at([float(q == k) for q in range(d + 1)]) for k in range(d + 1)])
    _, inv = _det_inv(torch.einsum("kam,eac->ekmc", T, nodes))  # [e][k][c][mu]
    detc, _ = _det_inv(torch.einsum("am,eac->emc", grad_at([1.0 / (d + 1)] * (d + 1)), nodes))
    K = _reference("K_iso", form, d)                             # [i][j][k][m][l][v]
    G = torch.einsum("ekcm,elcv->ekmlv", inv, inv) * detc.abs()[:, None, None, None, None]
    return (G.reshape(e, -1) @ K.reshape(K.shape[0] ** 2, -1).T).reshape(e, K.shape[0], -1)


def _value_and_gradients(fn, conn, dA, leaves, per_element):
    """A and the gradients of sum(dA * A): leaves indexed by vertex unless per_element says so."""
    leaves = [t.double() for t in leaves]
    grads = [torch.zeros_like(t) for t in leaves]
    A = torch.empty(dA.shape, dtype=torch.float64, device=DEV)
    for s in _chunks(conn.shape[0]):
        c = conn[s].long()
        local = [(t[s] if pe else t[c]).clone().requires_grad_(True) for t, pe in zip(leaves, per_element)]
        with torch.enable_grad():
            a = fn(*local)
            got = torch.autograd.grad(a, local, dA[s].double())
        A[s] = a.detach()
        for g, t, pe in zip(got, grads, per_element):
            if pe:
                t[s] = g
            else:
                t.index_add_(0, c.reshape(-1), g.reshape((-1,) + t.shape[1:]))
    return [A] + grads


def _exact_step(form, x, conn, coef, dA):
    one = lambda P: torch.ones(P.shape[0], dtype=torch.float64, device=DEV)
    if form == "P1_W1" or form == "P2_W1":
        return _value_and_gradients(lambda P, w: _affine(form, P, w), conn, dA, [x, coef], [False, False])
    if coef is None:
        return _value_and_gradients(lambda P: _affine(form, P, one(P)), conn, dA, [x], [False])
    return _value_and_gradients(lambda P, w: _affine(form, P, w), conn, dA, [x, coef], [False, True])


def _exact_assembly(form, d, n_vert, conn, A):
    dofs = conn.long()
    n_rows = n_vert
    if form == "P2":
        pairs = torch.stack([torch.stack([dofs[:, a], dofs[:, b]], 1) for a, b in _edges(d)], 1)
        key = pairs.min(2).values * n_vert + pairs.max(2).values
        uniq, inv = torch.unique(key, return_inverse=True)
        dofs = torch.cat([dofs, n_vert + inv], 1)
        n_rows = n_vert + uniq.numel()
    b = d if form == "ELASTIC" else 1
    n = dofs.shape[1]
    key = (dofs[:, :, None] * n_rows + dofs[:, None, :]).reshape(-1)
    uniq, inv = torch.unique(key, return_inverse=True)
    del key
    out = torch.zeros((uniq.numel(), b, b), dtype=torch.float64, device=DEV)
    for s in _chunks(conn.shape[0]):
        blocks = A[s].double().reshape(-1, b, n, b, n).permute(0, 2, 4, 1, 3).reshape(-1, b, b)
        out.index_add_(0, inv[s.start * n * n: s.stop * n * n], blocks)
    return out if b > 1 else out.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "forward64":
        x, conn = _mesh(case, _gen(seed))
        one = torch.ones(conn.shape[0], dtype=torch.float64, device=DEV)
        return torch.cat([_affine(case["form"], x[conn[s].long()], one[s]) for s in _chunks(conn.shape[0])])
    if kind == "step":
        x, conn, coef, dA = _step_inputs(case, seed)
        return _exact_step(case["form"], x, conn, coef, dA)
    if kind == "assemble":
        x, conn, A = _assemble_inputs(case, seed)
        return _exact_assembly(case["form"], case["dim"], x.shape[0], conn, A)
    if kind == "curved":
        gen = _gen(seed)
        x, conn, mid = _curved_mesh(case, gen)
        dA = torch.randn((conn.shape[0],) + _shape(case["form"], case["dim"]), generator=gen, device=DEV)
        return _value_and_gradients(lambda P, M: _curved(case["form"], P, M), conn, dA, [x, mid], [False, True])
    out = []
    for d, f, x, conn, coef, dA in _batch_inputs(case, seed):
        out += _exact_step(f, x, conn, coef, dA)
    return out
