"""Assembly of the P1 forms and of elasticity on meshes unlike a cube (-m gpu).

Rows of a window that differ in length, vertices numbered at random or unused,
rows at the edges of the kinds (32, 33, 63, 64 columns, more than one range of
columns), several windows with a partial last one.  The values are float32 sums
in a defined order, so they are compared bit for bit with np.add.at.  And such
meshes take about as long per contribution as a cube of the same kind does: a
path that leaves the lanes of a warp idle takes ten times as long or more."""
import numpy as np
import pytest
import torch

from paper_1103_0066_gb300 import meshgen as mg

LP1, EP1 = 0, 2
DEV = "cuda:0"
RNG = np.random.default_rng


def _fan(dim, spokes, first):
    """A closed fan around one vertex (triangles) or one edge (tets): spokes + dim - 1 columns in the hub's row."""
    hub = list(range(first, first + dim - 1))
    ring = [first + dim - 1 + k for k in range(spokes)]
    return np.array([hub + [ring[k], ring[(k + 1) % spokes]] for k in range(spokes)]), dim - 1 + spokes


def _fans(dim, columns, gap=0):
    conn, v = [], 0
    for c in columns:
        el, n = _fan(dim, c - dim + 1, v)
        conn.append(el)
        v += n + gap
    return np.concatenate(conn), v


def _split(conn, n_vert):
    """Every element split at a new vertex of its own (barycentric split)."""
    c = n_vert + np.arange(len(conn))
    parts = []
    for i in range(conn.shape[1]):
        k = conn.copy()
        k[:, i] = c
        parts.append(k)
    return np.stack(parts, 1).reshape(-1, conn.shape[1]), n_vert + len(conn)


def _grid(dim, n):
    m = mg.square_tri_mesh(n, 0.0, mg.rng_for(3)) if dim == 2 else mg.cube_tet_mesh(n, 0.0, mg.rng_for(3), 0.0)
    return m.conn.astype(np.int64), m.n_vert


def _numbered(conn, n_vert, seed, elements=False):
    r = RNG(seed)
    conn = r.permutation(n_vert)[conn]
    return (conn[r.permutation(len(conn))] if elements else conn), n_vert


def _mesh(dim, shape):
    if shape == "edges":  # hubs at the edges of the kinds, each twice
        return _fans(dim, [31, 32, 33, 57, 58, 62, 63, 64, 65, 88, 110, 111] * 2)
    if shape == "unused":  # one row of 30 among unused vertices: no two in a block of any size
        return _fans(dim, [30] * 40, gap=40)
    if shape == "windows":  # hubs and ring vertices in random order, over several windows
        conn, v = _fans(dim, [5 + k % 28 for k in range(150)])
        return _numbered(conn, v, 4)
    if shape == "split":
        return _split(*_grid(dim, 5 if dim == 3 else 17))
    if shape == "split random":
        return _numbered(*_split(*_grid(dim, 5 if dim == 3 else 17)), 5)
    return _numbered(*_grid(dim, 11 if dim == 3 else 40), 6, elements=True)  # "shuffled"


def _windows_by_count(conn, V, b):
    """Which windows of short rows the build orders by incidence count (b: block size of the form)."""
    nv = conn.shape[1]
    slots = conn.ravel()
    count = np.bincount(slots, minlength=V)
    first = np.full(V, conn.size)
    np.minimum.at(first, slots, np.arange(conn.size))
    used = np.flatnonzero(count)
    pairs = used[:-1][np.diff(used) == 1]
    near = (np.abs(first[pairs + 1] - first[pairs]) <= 512).sum() * 2 >= len(pairs)
    cols = np.bincount(np.unique(np.repeat(conn, nv, axis=1).ravel() * V + np.tile(conn, (1, nv)).ravel()) // V,
                       minlength=V)
    rows = used if near else used[np.argsort(first[used])]
    rows = rows[(cols[rows] <= 32) & (count[rows] <= (32 if b == 1 else 255))]
    size, blocks = {1: (32, 31), 2: (8, 127), 3: (3, 251)}[b]
    out = []
    for w in range(0, len(rows), size * blocks):
        c = count[rows[w:w + size * blocks]]
        c = np.pad(c, (0, -len(c) % size)).reshape(-1, size)
        out.append(2 * size * c.max(1).sum() > 3 * c.sum())
    return out


SHAPES = ["edges", "unused", "windows", "split", "split random", "shuffled"]


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("form", [LP1, EP1])
def test_shapes_reach_both_orders(dim, form):
    by_count = [_windows_by_count(*_mesh(dim, shape), dim if form == EP1 else 1) for shape in SHAPES]
    assert any(any(w) for w in by_count) and any(not all(w) for w in by_count)
    assert any(len(w) > 1 for w in by_count)


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("form", [LP1, EP1])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("offset", [0, 1])
def test_irregular_rows_bitwise(gfem, dim, form, shape, offset):
    conn, V = _mesh(dim, shape)
    conn = np.ascontiguousarray(conn.astype(np.int32))
    b = dim if form == EP1 else 1
    E, nv = conn.shape
    A = RNG(6).standard_normal((E, nv * b, nv * b)).astype(np.float32)
    buf = torch.zeros(offset + A.size, device=DEV)
    buf[offset:] = torch.from_numpy(A.ravel()).to(DEV)
    asm = gfem.Assembly(torch.zeros((V, dim), device=DEV), torch.from_numpy(conn).to(DEV), form)
    out = [torch.full((asm.nnz,) if b == 1 else (asm.nnz, b, b), float("nan"), device=DEV) for _ in range(2)]
    got = [asm.assemble(buf[offset:].view(A.shape), out=o).cpu().numpy().reshape(-1, b, b) for o in out]
    key = np.repeat(conn, nv, axis=1).ravel().astype(np.int64) * V + np.tile(conn, (1, nv)).ravel()
    uk, inv = np.unique(key, return_inverse=True)
    assert asm.nnz == len(uk) and np.array_equal(asm.col_idx.cpu().numpy(), uk % V)
    blocks = A.reshape(E, b, nv, b, nv).transpose(0, 2, 4, 1, 3).reshape(-1, b, b)
    want = np.zeros((len(uk), b, b), np.float32)
    if b == 1:  # per 32-element tile in element order, then the tile sums in tile order
        keys, tinv = np.unique(np.repeat(np.arange(E) // 32, nv * nv) * len(uk) + inv, return_inverse=True)
        part = np.zeros((len(keys), 1, 1), np.float32)
        np.add.at(part, tinv, blocks)
        np.add.at(want, keys % len(uk), part)
        assert asm.n_records == len(keys)
    else:
        np.add.at(want, inv, blocks)
    assert np.array_equal(got[0], want) and np.array_equal(got[1], want)


def _ns_per_incidence(gfem, conn, V, form, dim):
    conn = torch.from_numpy(np.ascontiguousarray(conn.astype(np.int32))).to(DEV)
    n = gfem.form_info(form, dim)[0]
    A = torch.randn((conn.shape[0], n, n), device=DEV)
    asm = gfem.Assembly(torch.zeros((V, dim), device=DEV), conn, form)
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
    return best / conn.numel()


@pytest.mark.gpu
@pytest.mark.parametrize("form,dim,shape", [(LP1, 3, "split"), (LP1, 3, "split random"), (LP1, 3, "half"),
                                            (LP1, 2, "split random"), (EP1, 3, "split random"), (EP1, 2, "eighth")])
def test_irregular_mesh_costs_no_more_than_four_cubes(gfem, form, dim, shape):
    n = 40 if dim == 3 else 400
    conn, V = _grid(dim, n)
    cube = _ns_per_incidence(gfem, conn, V, form, dim)
    if shape == "half":
        conn, V = _numbered(conn, V, 7)
        conn = conn[:len(conn) // 2]
    elif shape == "eighth":  # corner vertices among many others that no element uses
        conn = RNG(8).permutation(8 * V)[:V][conn]
        V *= 8
    else:
        conn, V = _split(*_grid(dim, n * 5 // 8))
        if shape == "split random":
            conn, V = _numbered(conn, V, 9)
    assert _ns_per_incidence(gfem, conn, V, form, dim) < 4 * cube
