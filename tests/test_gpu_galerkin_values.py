"""The values of the multigrid hierarchy: the Galerkin operators of every coarse
level and the inverse of the last one, on blocks of odd extents that leave part
of the coarse grids inactive, with Dirichlet faces (also across the interior of
a coarse cell), hanging nodes, and a thin block.

Level 1, P^T K P in the matrix precision: each entry is a sum of at most n =
125 x 27 products taken in some order, so |error| <= n eps (|P|^T |K| |P|)
entry by entry.  The uniform levels below: the product is defined in whole
numbers (an entry of the finer operator rounded once, at 2^(56 - floor(log2(
8.000001 B))) with B the largest l1 norm of one of its rows; whole weights of 2^-3
a side), so it is recomputed in int64 and has to be the same bit for bit.  The inverse of
the last level, by elimination without pivoting on a symmetric positive definite
matrix: |error| <= 10 n cond eps of its largest entry, plus its rounding.
"""
import numpy as np
import pytest

from paper_2606_09275_gb300 import inputs
from test_gpu_resident_solve import config

pytestmark = pytest.mark.gpu


def interpolation(coord, fine, coarse, d_fine, d_coarse):
    """P (fine rows x coarse rows), trilinear on the grid of depth d_coarse."""
    import scipy.sparse as sp
    s, n = 1 << (d_fine - d_coarse), 1 << d_coarse
    row = {tuple(c): r for r, c in enumerate(coarse)}
    cell = np.minimum(coord // s, n - 1)
    t = (coord - cell * s) / s
    i, j, w = [], [], []
    for c in range(8):
        b = np.array([(c >> d) & 1 for d in range(3)])
        wc = np.prod(np.where(b, t, 1.0 - t), axis=1)
        for r in np.nonzero(wc)[0]:
            i.append(fine[r])
            j.append(row[tuple(cell[r] + b)])
            w.append(wc[r])
    return sp.csr_matrix((w, (i, j)), shape=(len(coord), len(coarse)))


def level_matrix(nodes, values, R, d):
    """The operator of a uniform level as a sparse matrix, values as stored."""
    import scipy.sparse as sp
    n, S1 = (1 << d) + 1, 2 * R + 1
    gid = np.full((n + 2 * R,) * 3, -1, dtype=np.int64)
    x, y, z = (nodes[:, k] + R for k in range(3))
    gid[x, y, z] = np.arange(len(nodes))
    i, j, v = [], [], []
    for o in range(S1 ** 3):
        off = np.array([o % S1, (o // S1) % S1, o // S1 ** 2]) - R
        col = gid[x + off[0], y + off[1], z + off[2]]
        on = np.nonzero(col >= 0)[0]
        assert not values[col < 0, o].any()  # nothing for a node that is not there
        for e in range(9):
            i.append(3 * on + e // 3)
            j.append(3 * col[on] + e % 3)
            v.append(values[on, o, e])
    return sp.csr_matrix((np.concatenate(v), (np.concatenate(i), np.concatenate(j))), shape=(3 * len(nodes),) * 2)


def fixed_rows(mask):
    return np.array([[(m >> c) & 1 for c in range(3)] for m in mask], dtype=bool).ravel()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("key,depth,block", [("indent", (5, 6), (19, 23, 11)), ("punch", (4, 6), (15, 9, 7)),
                                             ("indent", (4, 5), (13, 11, 2))])
def test_level_operators(key, depth, block, precision):
    import scipy.sparse as sp
    import torch
    from paper_2606_09275_gb300 import mpm
    cfg = config(key, depth, block)
    ctx = mpm.Context()
    pts = inputs.make_points(cfg)
    P = mpm.Points(pts, capacity=12 * len(pts["x"]) + 400000)
    bz = inputs.body_z(cfg, 1)
    mesh = mpm.octree_build(ctx, cfg, P, body_z=bz)
    nd = mesh.info()["ndof"]
    zero = torch.zeros(3 * nd, dtype=torch.float64, device="cuda")
    Kd = mpm.assemble(ctx, mesh, cfg, zero, precision=precision, body_z=bz)["K"]
    b = torch.from_numpy(np.random.default_rng(2).normal(size=3 * nd)).cuda()
    mpm.solve(ctx, mesh, cfg, Kd, b, precision=precision, tol=1e-6, maxit=2000, method=3, inner_tol=1e-4)
    eps = 2.0 ** -23 if precision else 2.0 ** -52
    store = np.float32 if precision else np.float64

    levels = [lv for lv in mesh.export("mg_levels") if lv[1]]
    nodes, values = mesh.export("mg_nodes"), mesh.export("mg_values")
    A, nn, at, an = [], [], 0, 0
    for d, rows, R, S in levels:
        nn.append(nodes[an:an + rows])
        A.append(level_matrix(nn[-1], values[at:at + 9 * S * rows].reshape(rows, S, 9), R, d))
        an, at = an + rows, at + 9 * S * rows

    # level 1
    dof, coord = mesh.export("node_dof"), mesh.export("node_coord")
    x = np.zeros((nd, 3), dtype=np.int64)
    x[dof[dof >= 0]] = coord[dof >= 0]
    K = sp.bsr_matrix((mpm.blocks(ctx, mesh, Kd, precision), mesh.export("col"), mesh.export("row_ptr")),
                      shape=(3 * nd, 3 * nd))
    free = sp.diags((~fixed_rows(mesh.export("bcmask"))).astype(float))
    p = sp.kron(interpolation(x, np.arange(nd), nn[0][:, :3], cfg["depth_max"], levels[0][0]), sp.eye(3)).tocsr()
    want = p.T @ (free @ K @ free) @ p
    bound = p.T @ abs(free @ K @ free) @ p
    fixed = fixed_rows(nn[0][:, 3])
    want = want + sp.diags(fixed.astype(float))
    over = abs(A[0] - want) - 125 * 27 * eps * bound
    assert over.max() <= 1e-300

    # the uniform levels
    for f in range(len(levels) - 1):
        d, c = levels[f], levels[f + 1]
        assert d[2] == c[2] == 2  # the gathered form
        fine = np.array(abs(A[f]).sum(axis=1)).reshape(-1, 3).sum(axis=1).max()
        ex = 56 - int(np.floor(np.log2(8.000001 * fine)))
        free = sp.diags((~fixed_rows(nn[f][:, 3])).astype(float))
        ints = (free @ A[f] @ free).tocsr()
        ints.data = np.rint(np.ldexp(ints.data, ex))
        ints = ints.astype(np.int64)
        w = interpolation(nn[f][:, :3], np.arange(d[1]), nn[f + 1][:, :3], d[0], c[0])
        w.data = np.rint(8.0 * w.data)
        w = sp.kron(w, sp.eye(3)).tocsr().astype(np.int64)
        want = (w.T @ ints @ w).tocsr()
        want = sp.csr_matrix((np.ldexp(want.data.astype(store).astype(np.float64), -ex - 6), want.indices, want.indptr),
                             shape=want.shape)
        want = want + sp.diags(fixed_rows(nn[f + 1][:, 3]).astype(float))
        assert abs(A[f + 1] - want).max() == 0.0

    # the inverse of the last level
    last = A[-1].toarray()
    n = len(last)
    got = values[at:].reshape(n, n)
    inv = np.linalg.inv(0.5 * (last + last.T))
    tol = (10 * n * np.linalg.cond(last) * 2.0 ** -53 + eps) * abs(inv).max() + abs(last - last.T).max() * abs(inv).max() ** 2 * n
    assert abs(got - inv).max() <= tol
