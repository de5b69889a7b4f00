"""The curved kernels over several tiles per warp (-m gpu).

An element's matrix and the gradients of its edge nodes and coefficient depend
on that element alone, so a mesh large enough that every warp walks several
tiles (the next tile's upstream matrices arriving under the current one's
arithmetic) must give, bit for bit, what a run over any few of its elements
gives; the last tile is ragged.  One invalid and one degenerate element sit in
tiles that are followed by others."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
ISO1, ISO2 = 5, 6
DEV = "cuda:0"


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("form", [ISO1, ISO2])
def test_tiles_do_not_touch_one_another(gfem, dim, form):
    base = (mg.square_tri_mesh(420, 0.2, mg.rng_for(61), np.float32) if dim == 2
            else mg.cube_tet_mesh(29, 0.15, mg.rng_for(61), 0.0, np.float32))
    cm, mid = mg.curved_mesh(base)
    E = cm.n_elem - 13
    conn = cm.conn[:E].copy()
    conn[40, 1] = cm.n_vert + 5        # invalid
    conn[70] = conn[70, 0]             # degenerate
    mid = mid[:E].copy()
    mid[70] = cm.coords[conn[70, 0]]
    x, c, m = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (cm.coords, conn, mid))
    w = torch.from_numpy(mg.lognormal_coef(mg.rng_for(62), E)).to(DEV)
    n = gfem.form_info(form, dim)[0]
    dA = torch.randn((E, n, n), generator=torch.Generator(device=DEV).manual_seed(3), device=DEV)
    ws = gfem.Workspace(x, c, form)
    A = gfem.integrate_fwd_iso(x, c, m, form, w)
    _, dm, dw = gfem.integrate_bwd_iso(x, c, m, form, dA, w, ws=ws, need_dcoef=True)
    assert torch.isfinite(A).all() and torch.isfinite(dm).all() and torch.isfinite(dw).all()
    assert not A[40].any() and not A[70].any() and not dm[40].any() and not dm[70].any()
    for s in (slice(0, 96), slice(E // 2 // 32 * 32, E // 2 // 32 * 32 + 64), slice(E - E % 32 - 64, E)):
        part = [t[s].contiguous() for t in (c, m, w, dA)]
        a = gfem.integrate_fwd_iso(x, part[0], part[1], form, part[2])
        _, pm, pw = gfem.integrate_bwd_iso(x, part[0], part[1], form, part[3], part[2],
                                           ws=gfem.Workspace(x, part[0], form), need_dcoef=True)
        assert torch.equal(a, A[s]) and torch.equal(pm, dm[s]) and torch.equal(pw, dw[s])
