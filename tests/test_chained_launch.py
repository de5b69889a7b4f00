"""Kernels that may be set up while the stream's previous kernel ends (-m gpu).

Every pass's inputs are written, by kernels of others, into the same buffers
right before the library's calls, without a synchronisation between: each
pass must see its own inputs and leave what a pass with synchronisations
leaves, on the default stream, on another one and replayed from a CUDA graph."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
LP1, LP2, ISO2 = 0, 1, 6
DEV = "cuda:0"
PASSES = 12


@pytest.mark.parametrize("how", ["default", "stream", "graph"])
@pytest.mark.parametrize("form", [LP1, LP2, ISO2])
def test_each_pass_sees_its_own_inputs(gfem, how, form):
    m = mg.cube_tet_mesh(14, 0.15, mg.rng_for(95), 0.0, np.float32)
    cm, mid0 = mg.curved_mesh(m)
    conn = torch.from_numpy(m.conn).to(DEV)
    base, mid = torch.from_numpy(cm.coords).to(DEV), torch.from_numpy(mid0).to(DEV)
    scale = [torch.full((), 1.0 + 0.03 * k, device=DEV) for k in range(PASSES)]
    n = gfem.form_info(form, 3)[0]
    ws, asm = gfem.Workspace(base, conn, form), gfem.Assembly(base, conn, form)
    x, md, s = base.clone(), mid.clone(), torch.ones((), device=DEV)
    A, dA = (torch.empty((m.n_elem, n, n), device=DEV) for _ in range(2))
    det, dx, dm = torch.empty(m.n_elem, device=DEV), torch.empty_like(x), torch.empty_like(mid)
    vals = torch.empty(asm.nnz, device=DEV)

    def one_pass(sync):
        wait = torch.cuda.synchronize if sync else lambda: None
        torch.mul(base, s, out=x)
        torch.mul(mid, s, out=md)
        wait()
        if form == ISO2:
            gfem.integrate_fwd_iso(x, conn, md, form, out=A)
        else:
            gfem.integrate_fwd(x, conn, form, out=A, det_out=det)
        wait()
        asm.assemble(A, out=vals)
        wait()
        torch.sin(A, out=dA)
        wait()
        if form == ISO2:
            gfem.integrate_bwd_iso(x, conn, md, form, dA, ws=ws, dcoords=dx, dmid=dm)
        else:
            gfem.integrate_bwd(x, conn, form, dA, ws=ws, need_dcoef=False, dcoords=dx, det=det)
        wait()

    want = []
    for k in range(PASSES):
        s.copy_(scale[k])
        one_pass(True)
        want.append([t.clone() for t in (A, vals, dx)])
    torch.cuda.synchronize()
    stream = torch.cuda.default_stream() if how == "default" else torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        if how == "graph":
            with torch.cuda.graph(graph, stream=stream):
                one_pass(False)
        got = []
        for k in range(PASSES):
            s.copy_(scale[k])
            graph.replay() if how == "graph" else one_pass(False)
            got.append([t.clone() for t in (A, vals, dx)])
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        for g, w in zip(a, b):
            assert torch.equal(g, w)
