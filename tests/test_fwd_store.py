"""The forward's tile stores (-m gpu): a ragged mesh over several tiles per
warp, written to an aligned and to an unaligned output, gives the same bits,
row by row those of a run over a few of its elements, and nothing around the
output is touched."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu
LP1, LP2, EP1, LP2W, ISO2 = 0, 1, 2, 4, 6
DEV = "cuda:0"


@pytest.mark.parametrize("dim,form", [(2, LP1), (2, LP2), (2, EP1), (2, ISO2), (3, LP1), (3, LP2), (3, EP1),
                                      (3, LP2W), (3, ISO2)])
@pytest.mark.parametrize("tail", [1, 31])
def test_store_aligned_unaligned_and_ragged(gfem, dim, form, tail):
    m = (mg.square_tri_mesh(420, 0.2, mg.rng_for(81), np.float32) if dim == 2
         else mg.cube_tet_mesh(27, 0.15, mg.rng_for(81), 0.02, np.float32))
    E = m.n_elem // 32 * 32 - 32 + tail
    conn = torch.from_numpy(m.conn[:E].copy()).to(DEV)
    w = torch.from_numpy(mg.lognormal_coef(mg.rng_for(82), m.n_vert if form == LP2W else E)).to(DEV)
    if form == ISO2:
        cm, mid = mg.curved_mesh(m)
        x, mid = torch.from_numpy(cm.coords).to(DEV), torch.from_numpy(mid[:E].copy()).to(DEV)
    else:
        x, mid = torch.from_numpy(m.coords).to(DEV), None

    def fwd(s, out):
        c, k = conn[s].contiguous(), (w if form == LP2W else w[s].contiguous())
        if form == ISO2:
            return gfem.integrate_fwd_iso(x, c, mid[s].contiguous(), form, k, out=out)
        return gfem.integrate_fwd(x, c, form, k, out=out)

    n = gfem.form_info(form, dim)[0]
    whole = slice(0, E)
    got = []
    for offset in (4, 1):
        buf = torch.full((E * n * n + 8,), 7.5, device=DEV)
        A = buf[offset:offset + E * n * n].view(E, n, n)
        fwd(whole, A)
        assert torch.all(buf[:offset] == 7.5) and torch.all(buf[offset + E * n * n:] == 7.5)
        got.append(A.clone())
    assert torch.isfinite(got[0]).all() and torch.equal(got[0], got[1])
    for s in (slice(0, 64), slice(E - tail - 64, E)):
        assert torch.equal(fwd(s, None), got[0][s])
