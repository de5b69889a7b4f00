"""The adjoint's copy of the upstream matrices into its stage (-m gpu): ragged
last tiles of every residue that matters for 16-byte pieces, an aligned and an
unaligned dA.  The coefficient gradient belongs to one element, so it equals a
run over a few elements bit for bit; the vertex gradient does not depend on
where dA lies."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
LP1, LP2, EP1 = 0, 1, 2
DEV = "cuda:0"


@pytest.mark.parametrize("dim,form", [(2, LP1), (2, LP2), (2, EP1), (3, LP1), (3, LP2), (3, EP1)])
@pytest.mark.parametrize("tail", [1, 2, 3, 31, 32])
def test_dA_copy_aligned_unaligned_and_ragged(gfem, dim, form, tail):
    m = (mg.square_tri_mesh(60, 0.2, mg.rng_for(91), np.float32) if dim == 2
         else mg.cube_tet_mesh(11, 0.15, mg.rng_for(91), 0.02, np.float32))
    E = m.n_elem // 32 * 32 - 32 + tail
    x = torch.from_numpy(m.coords).to(DEV)
    conn = torch.from_numpy(m.conn[:E].copy()).to(DEV)
    w = torch.from_numpy(mg.lognormal_coef(mg.rng_for(92), E)).to(DEV)
    n = gfem.form_info(form, dim)[0]
    dA = torch.randn((E, n, n), generator=torch.Generator(device=DEV).manual_seed(5), device=DEV)
    shifted = torch.empty(dA.numel() + 1, device=DEV)[1:].view(E, n, n).copy_(dA)
    dx, dw = gfem.integrate_bwd(x, conn, form, dA, w)
    dx1, dw1 = gfem.integrate_bwd(x, conn, form, shifted, w)
    assert torch.isfinite(dx).all() and torch.equal(dx, dx1) and torch.equal(dw, dw1)
    for s in (slice(0, 32), slice(E - tail, E)):
        _, part = gfem.integrate_bwd(x, conn[s].contiguous(), form, dA[s].contiguous(), w[s].contiguous(),
                                     need_dcoords=False)
        assert torch.equal(part, dw[s])
