"""A forward into an output off the 16-byte boundary takes about as long as an aligned one (-m gpu).

Values: test_fwd_store.py.  The rolled scalar loop beside the wide stores took
1.24 to 1.39 times the aligned call's time on these shapes."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,form", [(2, "LAPLACE_P2_W1"), (3, "LAPLACE_P2"), (3, "ELASTIC_P1")])
def test_unaligned_output_time(gfem, dim, form):
    form = getattr(gfem, form)
    m = (mg.square_tri_mesh(500, 0.2, mg.rng_for(1), np.float32) if dim == 2 else
         mg.cube_tet_mesh(40, 0.15, mg.rng_for(1)))
    x, conn = torch.from_numpy(m.coords).cuda(), torch.from_numpy(m.conn).cuda()
    w = torch.ones(m.n_vert, device="cuda") if form == gfem.LAPLACE_P2_W1 else None
    shape = (m.n_elem,) + gfem.form_shape(form, dim)
    aligned = torch.empty(shape, device="cuda")
    off = torch.empty(aligned.numel() + 1, device="cuda")[1:].view(shape)

    def ms(out):
        best = 1e30
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(8):
                gfem.integrate_fwd(x, conn, form, w, out=out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    t, u = ms(aligned), ms(off)
    assert torch.equal(aligned, off)
    assert u < 1.2 * t


@pytest.mark.parametrize("dim", [2, 3])
def test_unaligned_curved_output_time(gfem, dim):
    """Curved P2: 1.36 and 1.44 times the aligned call with the rolled loop."""
    m = (mg.square_tri_mesh(1000, 0.2, mg.rng_for(1), np.float32) if dim == 2 else
         mg.cube_tet_mesh(56, 0.15, mg.rng_for(1)))
    cm, mid = mg.curved_mesh(m)
    x, conn, mid = (torch.from_numpy(t).cuda() for t in (cm.coords.astype(np.float32), m.conn, mid))
    shape = (m.n_elem,) + gfem.form_shape(gfem.LAPLACE_P2_ISO, dim)
    aligned = torch.empty(shape, device="cuda")
    off = torch.empty(aligned.numel() + 1, device="cuda")[1:].view(shape)

    def ms(out):
        best = 1e30
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(4):
                gfem.integrate_fwd_iso(x, conn, mid, gfem.LAPLACE_P2_ISO, out=out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    t, u = ms(aligned), ms(off)
    assert torch.equal(aligned, off)
    assert u < 1.3 * t
