"""Row kernel of the assembly at the edges of its paths (-m gpu).

Meshes that make a row longer than the columns held in shared memory, rows of
one block that differ so much that the padded slots exceed their room, a last
block with few rows, empty rows, elements that list a vertex twice (blocks
only), and element matrices that are not 16-byte aligned.  The values are the
float32 sums of the given element matrices in the order that the library
defines, so they are compared bit for bit with numpy's unbuffered np.add.at."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
LP1, LP2, EP1 = 0, 1, 2
DEV = "cuda:0"


def _wheel(dim, spokes, first):
    """A closed fan of `spokes` elements around one vertex (triangles) or one edge (tets), vertices from `first` on."""
    hub = list(range(first, first + dim - 1))
    ring = [first + dim - 1 + k for k in range(spokes)]
    return [hub + [ring[k], ring[(k + 1) % spokes]] for k in range(spokes)], dim - 1 + spokes


def _mesh(dim, shape):
    if shape == "long":        # hubs of 41 and 42 columns (and of 32), other rows short
        a, n = _wheel(dim, 40, 3)
        b, m = _wheel(dim, 32 - (dim - 1), 3 + n)
        conn, V = a + b, 3 + n + m
    elif shape == "padded":    # each block of 32 rows holds one hub of 30 elements: 30 steps for rows of 2
        conn = [el for k in range(5) for el in _wheel(dim, 30, 32 * k)[0]]
        V = 32 * 5
    else:                      # "repeat": an element lists a vertex of its row twice, another one twice
        conn, V = _wheel(dim, 9, 0)
        conn[4][-1] = conn[4][0]
        conn[6][-1] = conn[6][-2]
    rng = np.random.default_rng(5)
    conn = np.array(conn, np.int32)[rng.permutation(len(conn))]
    return np.ascontiguousarray(conn), V + 2


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("form,shape", [(LP1, "long"), (LP1, "padded"), (EP1, "long"), (EP1, "padded"),
                                        (EP1, "repeat")])
@pytest.mark.parametrize("offset", [0, 1])
def test_row_paths_bitwise(gfem, dim, form, shape, offset):
    conn, V = _mesh(dim, shape)
    b = dim if form == EP1 else 1
    E, nv = conn.shape
    n = nv * b
    A = np.random.default_rng(6).standard_normal((E, n, n)).astype(np.float32)
    buf = torch.zeros(offset + A.size, device=DEV)
    buf[offset:] = torch.from_numpy(A.ravel()).to(DEV)
    At = buf[offset:].view(E, n, n)
    coords = torch.zeros((V, dim), device=DEV)
    asm = gfem.Assembly(coords, torch.from_numpy(conn).to(DEV), form)
    got = asm.assemble(At).cpu().numpy().reshape(asm.nnz, b, b)
    rows = np.repeat(conn, nv, axis=1).ravel().astype(np.int64)
    cols = np.tile(conn, (1, nv)).ravel()
    key = rows * V + cols
    uk, inv = np.unique(key, return_inverse=True)
    assert asm.nnz == len(uk)
    assert np.array_equal(asm.col_idx.cpu().numpy(), uk % V)
    blocks = A.reshape(E, b, nv, b, nv).transpose(0, 2, 4, 1, 3).reshape(-1, b, b)
    want = np.zeros((len(uk), b, b), np.float32)
    if b == 1:  # per 32-element tile in element order, then the tile sums in tile order
        tile = np.repeat(np.arange(E) // 32, nv * nv)
        keys, tinv = np.unique(tile * len(uk) + inv, return_inverse=True)
        part = np.zeros((len(keys), 1, 1), np.float32)
        np.add.at(part, tinv, blocks)
        np.add.at(want, keys % len(uk), part)
        assert asm.n_records == len(keys)
    else:
        np.add.at(want, inv, blocks)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("shape", ["long", "single", "wheels"])
@pytest.mark.parametrize("offset", [0, 1])
def test_p2_row_paths_bitwise(gfem, dim, shape, offset):
    """Vertex and edge unknowns: a vertex with more columns than a row buffer
    of the fast path holds beside short rows, elements that share nothing (one
    incidence per unknown: more chunks than their room), and closed fans."""
    nv, nb = dim + 1, (dim + 1) * (dim + 2) // 2
    if shape == "long":  # 60 triangles: 181 columns (45 tets around an edge: 231)
        conn = _wheel(dim, 60 if dim == 2 else 45, 0)[0] + [list(range(200, 200 + nv))]
        V = 210
    elif shape == "single":
        conn, V = [list(range(nv * e, nv * e + nv)) for e in range(2000)], nv * 2000 + 1
    else:
        conn, V = [el for k in range(7) for el in _wheel(dim, 5 + k, 16 * k)[0]], 16 * 8
    rng = np.random.default_rng(7)
    conn = np.ascontiguousarray(np.array(conn, np.int32)[rng.permutation(len(conn))])
    E = len(conn)
    A = rng.standard_normal((E, nb, nb)).astype(np.float32)
    buf = torch.zeros(offset + A.size, device=DEV)
    buf[offset:] = torch.from_numpy(A.ravel()).to(DEV)
    asm = gfem.Assembly(torch.zeros((V, dim), device=DEV), torch.from_numpy(conn).to(DEV), LP2)
    got = [asm.assemble(buf[offset:].view(E, nb, nb)).cpu().numpy() for _ in range(2)]
    pairs = [(a, b) for a in range(nv) for b in range(a + 1, nv)]
    lo = np.stack([np.minimum(conn[:, a], conn[:, b]) for a, b in pairs], 1).astype(np.int64)
    hi = np.stack([np.maximum(conn[:, a], conn[:, b]) for a, b in pairs], 1)
    _, edge = np.unique(lo * V + hi, return_inverse=True)
    dofs = np.concatenate([conn, V + edge.reshape(E, -1)], 1)
    assert np.array_equal(asm.dofs.cpu().numpy(), dofs)
    key = np.repeat(dofs, nb, axis=1).ravel().astype(np.int64) * asm.n_rows + np.tile(dofs, (1, nb)).ravel()
    uk, inv = np.unique(key, return_inverse=True)
    assert asm.nnz == len(uk) and np.array_equal(asm.col_idx.cpu().numpy(), uk % asm.n_rows)
    want = np.zeros(len(uk), np.float32)
    np.add.at(want, inv, A.ravel())
    assert np.array_equal(got[0], want) and np.array_equal(got[1], want)
