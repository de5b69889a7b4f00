"""P2 assembly where the chunks of incidences do not fit or a row is long.

The chunks lie in workspace that the built pattern leaves free, so the
workspace is that of the two graphs.  Values are float32 sums in element
order, compared bit for bit with np.add.at (-m gpu); and a mesh without room
for chunks, or with rows over the limit of a row buffer, takes about as long as
the same work elsewhere: one incidence after another takes twice as long."""
import numpy as np
import pytest
import torch

import __graft_entry__
from paper_1103_0066_gb300 import _native as nat
from paper_1103_0066_gb300 import meshgen as mg

LP2 = 1
DEV = "cuda:0"


def _p2_bytes(dim, E, V):
    """(workspace of both graphs, what the built pattern leaves free at most), padding to 256 bytes aside."""
    nv, n = dim + 1, (dim + 1) * (dim + 2) // 2
    rows = V + E * (n - nv)
    graph = [4 * (3 * (r + 1) + E * k + E * k * k) + E * k * k + 4 * (r // 1024 + 3) for r, k in ((V, nv), (rows, n))]
    tail = graph[0] + 4 * (V + 1)
    return graph[1] + tail + 4 * E * n, 4 * E * n * n + tail


@pytest.mark.parametrize("dim,E,V", [(3, 6 * 128**3, 129**3), (2, 2 * 1000**2, 1001**2), (3, 1000, 4000), (2, 1, 3)])
def test_chunks_take_no_room_of_their_own(dim, E, V):
    __graft_entry__.build()
    mesh = nat.FemMesh(dim=dim, n_elem=E, n_vert=V, coords=256, conn=256)
    got = nat.fem_assembly_workspace_size(mesh, LP2)
    assert got <= _p2_bytes(dim, E, V)[0] + 20 * 256


def _fans(dim, spokes, count):
    hub, ring = list(range(dim - 1)), [dim - 1 + k for k in range(spokes)]
    fan = np.array([hub + [ring[k], ring[(k + 1) % spokes]] for k in range(spokes)])
    n = dim - 1 + spokes
    return (fan + n * np.arange(count)[:, None, None]).reshape(-1, dim + 1), n * count


def _apart(dim, count):
    return np.arange(count * (dim + 1)).reshape(count, dim + 1), count * (dim + 1)


def _grid(dim, n):
    m = mg.square_tri_mesh(n, 0.0, mg.rng_for(3)) if dim == 2 else mg.cube_tet_mesh(n, 0.0, mg.rng_for(3), 0.0)
    return m.conn.astype(np.int64), m.n_vert


def _join(*meshes):
    conn, v = [], 0
    for c, n in meshes:
        conn.append(c + v)
        v += n
    return np.concatenate(conn), v


def _mesh(dim, shape):
    """Connectivity, vertices, whether the chunks fit, columns of the longest row."""
    # spokes of the hubs: the last of 160 columns or less (1 + 3 k, 3 + 4 k), the next, the most incidences
    a, b, c = (39, 40, 51) if dim == 3 else (53, 54, 84)
    grid = _grid(dim, 5 if dim == 3 else 40)
    if shape == "apart":
        return *_apart(dim, 700), False, None
    if shape == "apart, long":  # no chunks and rows over the limit
        return *_join(_apart(dim, 900), _fans(dim, c, 1)), False, 253 if dim == 2 else 207
    if shape == "long":  # rows over the limit beside short ones, several of them in a warp
        return *_join(grid, _fans(dim, b, 3), _fans(dim, c, 2)), True, 253 if dim == 2 else 207
    if shape == "limit":
        return *_join(_fans(dim, a, 3), grid), True, 160 if dim == 2 else 159
    return *grid, True, None


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("shape", ["apart", "apart, long", "long", "limit", "grid"])
@pytest.mark.parametrize("random", [False, True])
def test_p2_rows_bitwise(gfem, dim, shape, random):
    conn, V, fits, longest = _mesh(dim, shape)
    if random:
        conn = np.random.default_rng(4).permutation(V)[conn]
    conn = np.ascontiguousarray(conn.astype(np.int32))
    E, nv = conn.shape
    nb = nv * (nv + 1) // 2
    pairs = [(a, b) for a in range(nv) for b in range(a + 1, nv)]
    lo = np.stack([np.minimum(conn[:, a], conn[:, b]) for a, b in pairs], 1).astype(np.int64)
    hi = np.stack([np.maximum(conn[:, a], conn[:, b]) for a, b in pairs], 1)
    _, edge = np.unique(lo * V + hi, return_inverse=True)
    dofs = np.concatenate([conn, V + edge.reshape(E, -1)], 1)
    A = np.random.default_rng(5).standard_normal((E, nb, nb)).astype(np.float32)
    asm = gfem.Assembly(torch.zeros((V, dim), device=DEV), torch.from_numpy(conn).to(DEV), LP2)
    got = [asm.assemble(torch.from_numpy(A).to(DEV), out=torch.full((asm.nnz,), float("nan"), device=DEV)).cpu().numpy()
           for _ in range(2)]
    key = np.repeat(dofs, nb, axis=1).ravel().astype(np.int64) * asm.n_rows + np.tile(dofs, (1, nb)).ravel()
    uk, inv = np.unique(key, return_inverse=True)
    assert asm.nnz == len(uk) and np.array_equal(asm.col_idx.cpu().numpy(), uk % asm.n_rows)
    assert np.array_equal(asm.dofs.cpu().numpy(), dofs)
    # the mesh takes the path that it is here for
    chunks = int(((np.bincount(dofs.ravel()) + 3) // 4).sum())
    assert (4 * asm.nnz + chunks * (16 + 4 * nb) <= _p2_bytes(dim, E, V)[1]) == fits
    if longest:
        assert np.diff(asm.row_ptr.cpu().numpy()).max() == longest
    want = np.zeros(len(uk), np.float32)
    np.add.at(want, inv, A.ravel())
    assert np.array_equal(got[0], want) and np.array_equal(got[1], want)


def _us(gfem, conn, V):
    dim = conn.shape[1] - 1
    A = torch.randn((len(conn), (dim + 1) * (dim + 2) // 2, (dim + 1) * (dim + 2) // 2), device=DEV)
    asm = gfem.Assembly(torch.zeros((V, dim), device=DEV), torch.from_numpy(conn.astype(np.int32)).to(DEV), LP2)
    out = asm.assemble(A)
    best = 1e30
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            asm.assemble(A, out=out)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return 250 * best


@pytest.mark.gpu
def test_rows_over_the_limit_cost_no_chain(gfem):
    """Fans of 54 triangles (163 columns) against fans of 53 (160), the work being the same within 2%."""
    assert _us(gfem, *_fans(2, 54, 8000)) < 1.25 * _us(gfem, *_fans(2, 53, 8150))


@pytest.mark.gpu
def test_mesh_without_room_for_chunks(gfem):
    """Tets that share nothing: 10 rows and 100 values each, against a cube's 1.4 and 40."""
    E = 6 * 32**3
    assert _us(gfem, *_apart(3, E)) < 5 * _us(gfem, *_grid(3, 32))
