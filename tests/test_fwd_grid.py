"""A grid given in CTAs per SM alone keeps the warps it had on every form (-m gpu).

The forms of 36 and 100 floats a row run one-warp CTAs on their own grid; a
caller's two CTAs per SM are two of four warps, which take less than twice the
default's time.  Two one-warp CTAs per SM take 2.6 to 3.3 times."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,form", [(2, "LAPLACE_P2"), (2, "ELASTIC_P1"), (3, "LAPLACE_P2_W1")])
def test_ctas_per_sm_alone(gfem, dim, form):
    form = getattr(gfem, form)
    m = (mg.square_tri_mesh(700, 0.2, mg.rng_for(1), np.float32) if dim == 2 else
         mg.cube_tet_mesh(48, 0.15, mg.rng_for(1)))
    x, conn = torch.from_numpy(m.coords).cuda(), torch.from_numpy(m.conn).cuda()
    w = torch.ones(m.n_vert, device="cuda") if form == gfem.LAPLACE_P2_W1 else None
    A, B = (torch.empty((m.n_elem,) + gfem.form_shape(form, dim), device="cuda") for _ in range(2))

    def us(ctas, out):
        best = 1e30
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(8):
                gfem.integrate_fwd(x, conn, form, w, out=out, ctas_per_sm=ctas)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    default, two = us(0, A), us(2, B)
    assert torch.equal(A, B)
    assert two < 2 * default
