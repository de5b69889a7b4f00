"""Chained kernels of every form, and of a batch, see the inputs of their own pass (-m gpu).

As in test_chained_launch.py, each pass's inputs are written into the same
buffers right before the library's calls, without a synchronisation between,
and a pass must leave what one with synchronisations leaves: here for both
dimensions, elasticity, the P1-coefficient forms, the curved and the coupling
forms with all their gradients, and for a batch whose meshes run on several
streams, eager and replayed from a CUDA graph."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
LP1, LP2, EP1 = 0, 1, 2
DEV = "cuda:0"
PASSES = 6


def _repeat(one_pass, outputs, how):
    """PASSES results of one_pass(scale, wait) with synchronisations, and without them."""
    scale = [torch.full((), 1.0 + 0.05 * k, device=DEV) for k in range(PASSES)]
    s = torch.ones((), device=DEV)
    want = []
    for k in range(PASSES):
        s.copy_(scale[k])
        one_pass(s, torch.cuda.synchronize)
        want.append([t.clone() for t in outputs])
    torch.cuda.synchronize()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    got = []
    with torch.cuda.stream(stream):
        if how == "graph":
            with torch.cuda.graph(graph, stream=stream):
                one_pass(s, lambda: None)
        for k in range(PASSES):
            s.copy_(scale[k])
            graph.replay() if how == "graph" else one_pass(s, lambda: None)
            got.append([t.clone() for t in outputs])
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        for g, w in zip(a, b):
            assert torch.equal(g, w)


def _mesh(dim):
    return mg.cube_tet_mesh(12, 0.15, mg.rng_for(95)) if dim == 3 else mg.square_tri_mesh(70, 0.2, mg.rng_for(95),
                                                                                         np.float32)


@pytest.mark.parametrize("how", ["stream", "graph"])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("form", ["LAPLACE_P1", "LAPLACE_P2", "ELASTIC_P1", "LAPLACE_P1_W1", "LAPLACE_P2_W1",
                                  "LAPLACE_P1_ISO", "LAPLACE_P2_ISO", "DIV_P2P1"])
def test_each_form_sees_its_own_inputs(gfem, how, dim, form):
    m = _mesh(dim)
    iso, w1, div = form.endswith("ISO"), form.endswith("W1"), form == "DIV_P2P1"
    cm, mid0 = mg.curved_mesh(m)
    form = getattr(gfem, form)
    conn = torch.from_numpy(m.conn).to(DEV)
    base, mid = (torch.from_numpy(t.astype(np.float32)).to(DEV) for t in (cm.coords, mid0))
    V, E = base.shape[0], conn.shape[0]
    c0 = 1 + torch.rand(V if w1 else E, generator=torch.Generator(DEV).manual_seed(1), device=DEV)
    x, md, c = base.clone(), mid.clone(), c0.clone()
    ws = gfem.Workspace(base, conn, form)
    A, dA = (torch.empty((E,) + gfem.form_shape(form, dim), device=DEV) for _ in range(2))
    dx, dm, dc = torch.empty_like(x), torch.empty_like(mid), torch.empty_like(c)
    asm = None if div else gfem.Assembly(base, conn, form)
    vals = torch.empty(0 if div else (asm.nnz,) + (asm.block,) * (2 if asm.block > 1 else 0), device=DEV)

    def one_pass(s, wait):
        for src, dst in ((base, x), (mid, md), (c0, c)):
            torch.mul(src, s, out=dst)
        wait()
        if iso:
            gfem.integrate_fwd_iso(x, conn, md, form, c, out=A)
        else:
            gfem.integrate_fwd(x, conn, form, c, out=A)
        wait()
        if asm:
            asm.assemble(A, out=vals)
        wait()
        torch.sin(A, out=dA)
        wait()
        if iso:
            gfem.integrate_bwd_iso(x, conn, md, form, dA, c, ws=ws, need_dcoef=True, dcoords=dx, dmid=dm, dcoef=dc)
        else:
            gfem.integrate_bwd(x, conn, form, dA, c, ws=ws, dcoords=dx, dcoef=dc)
        wait()

    _repeat(one_pass, [A, vals, dx, dc] + ([dm] if iso else []), how)


@pytest.mark.parametrize("how", ["stream", "graph"])
def test_batch_sees_its_own_inputs(gfem, how):
    items, base = [], []
    for k, (dim, n, form) in enumerate([(3, 9, LP1), (3, 12, LP1), (3, 7, LP2), (3, 8, EP1), (2, 40, LP1), (2, 33, LP2),
                                        (2, 50, EP1), (3, 5, LP1)]):
        m = (mg.cube_tet_mesh(n, 0.15, mg.rng_for(k)) if dim == 3 else
             mg.square_tri_mesh(n, 0.2, mg.rng_for(k), np.float32))
        x = torch.from_numpy(m.coords).to(DEV)
        conn = torch.from_numpy(m.conn).to(DEV)
        w = 1 + torch.rand(m.n_elem, device=DEV)
        A = torch.empty((m.n_elem,) + gfem.form_shape(form, dim), device=DEV)
        base.append((x, w))
        items.append(dict(coords=x.clone(), conn=conn, form=form, coef=w.clone(), A=A, dA=torch.empty_like(A),
                          dcoords=torch.empty_like(x), dcoef=torch.empty_like(w)))
    batch = gfem.Batch(items)
    batch.set_config(1, 1, gfem.BATCH_PHASED)

    def one_pass(s, wait):
        for it, (x, w) in zip(items, base):
            torch.mul(x, s, out=it["coords"])
            torch.mul(w, s, out=it["coef"])
        wait()
        batch.run(gfem.PHASE_FWD)
        wait()
        for it in items:
            torch.sin(it["A"], out=it["dA"])
        wait()
        batch.run(gfem.PHASE_BWD)
        wait()

    _repeat(one_pass, [it[k] for it in items for k in ("A", "dcoords", "dcoef")], how)
    assert batch.errors() == 0
