"""The one-launch Krylov solves of small and middle meshes, at the sizes where
their division of the rows can go wrong: fewer row quads than SMs, one slice
with padding rows, rows kept in and out of shared memory, several passes of a
block over its rows, and the two sides of the size limit.

Reference: the relative residual ||b - K x|| / ||b|| on the free components,
recomputed in FP64 on the host from the exported blocks.  The solves stop at a
recurrence residual of tol; the true one may exceed it by the rounding of the
recurrences, a few hundred iterations times 1e-16 times the norm ratio
|K||x|/|b| (at most about 1e5 on these meshes), far below the 0.2 tol allowed
at tol = 1e-8 in FP64.  The mixed path measures its residual itself.
"""
import numpy as np
import pytest

from paper_2606_09275_gb300 import inputs

pytestmark = pytest.mark.gpu


def config(name, depth, block):
    cfg = inputs.workload(name, depth_min=depth[0], depth_max=depth[1])
    h = cfg["L"] / (1 << depth[0])
    hi = tuple(n * h for n in block)
    cfg["bc"] = [(0, 0.0, 1), (0, hi[0], 1), (1, 0.0, 2), (1, hi[1], 2), (2, 0.0, 7)]
    cfg["points"].update(lo=(0, 0, 0), hi=hi, spacing=h / 2, jitter=0.05 * h, seed=3)
    cfg["dx_region"] = 2 * cfg["L"] / (1 << depth[1])
    if cfg["body"]:
        cfg["body"].update(cx=0.5 * hi[0], cy=0.5 * hi[1], z0=hi[2])
    return cfg


MESHES = {
    "one_slice": ("column", (1, 1), (2, 2, 2)),          # 27 rows: padding rows, 8 quads
    "few_quads": ("column", (2, 2), (3, 2, 3)),          # fewer quads than SMs
    "punch": ("punch", (3, 6), (8, 8, 4)),               # hanging nodes, rows of 27 to 180 blocks
    "block_13k": ("indent", (5, 6), (29, 27, 13)),       # K out of shared memory
    "block_100k": ("indent", (6, 7), (58, 50, 31)),      # several passes per block (FP32)
    "block_140k": ("indent", (6, 7), (61, 57, 39)),      # beyond the limit: launches per iteration
}


@pytest.fixture(scope="module")
def system():
    import torch
    import scipy.sparse as sp
    from paper_2606_09275_gb300 import mpm
    cache = {}

    def make(key):
        if key not in cache:
            cache.clear()
            cfg = config(*MESHES[key])
            ctx = mpm.Context()
            pts = inputs.make_points(cfg)
            n = len(pts["x"])
            P = mpm.Points(pts, capacity=2 * n if n > 500000 else 12 * n + 400000)
            bz = inputs.body_z(cfg, 1) if cfg["body"] else None
            mesh = mpm.octree_build(ctx, cfg, P, body_z=bz)
            nd = mesh.info()["ndof"]
            g = mpm.assemble(ctx, mesh, cfg, torch.zeros(3 * nd, dtype=torch.float64, device="cuda"),
                             body_z=bz)
            K = sp.bsr_matrix((mpm.blocks(ctx, mesh, g["K"]), mesh.export("col"), mesh.export("row_ptr")),
                              shape=(3 * nd, 3 * nd))
            mask = mesh.export("bcmask")
            free = np.array([[not (m >> c) & 1 for c in range(3)] for m in mask]).ravel()
            b = np.random.default_rng(7).normal(size=3 * nd)
            cache[key] = dict(mpm=mpm, torch=torch, cfg=cfg, ctx=ctx, mesh=mesh, Kd=g["K"], K=K, free=free, b=b)
        return cache[key]

    return make


@pytest.mark.parametrize("key", list(MESHES))
@pytest.mark.parametrize("method,precision", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_solution_residual(system, key, method, precision):
    s = system(key)
    mpm, torch = s["mpm"], s["torch"]
    cfg = s["cfg"]
    if method == 2:  # friction makes the mixed path choose BiCGStab
        cfg = dict(cfg, mu=0.3, contact=1)
    Kd = s["Kd"].float() if precision else s["Kd"]
    rhs = torch.from_numpy(s["b"]).cuda()
    tol = 1e-8
    x, st = mpm.solve(s["ctx"], s["mesh"], cfg, Kd, rhs, precision=precision, tol=tol, maxit=5000,
                      method=method, inner_tol=1e-4)
    assert st["status"] == 0 and 0 < st["iterations"] and st["relres"] <= tol
    K = s["K"] if precision == 0 else s["K"].astype(np.float32).astype(np.float64)
    bf = s["b"] * s["free"]
    r = (bf - K @ x.cpu().numpy()) * s["free"]
    assert np.linalg.norm(r) <= 1.2 * tol * np.linalg.norm(bf)
    # the same again, bit for bit
    y, st2 = mpm.solve(s["ctx"], s["mesh"], cfg, Kd, rhs, precision=precision, tol=tol, maxit=5000,
                       method=method, inner_tol=1e-4)
    assert st2 == st and torch.equal(x, y)


@pytest.mark.parametrize("method", [1, 2])
def test_iteration_cap_and_zero_rhs(system, method):
    s = system("punch")
    mpm, torch = s["mpm"], s["torch"]
    rhs = torch.from_numpy(s["b"]).cuda()
    with pytest.raises(mpm.MPMError) as e:
        mpm.solve(s["ctx"], s["mesh"], s["cfg"], s["Kd"], rhs, tol=1e-12, maxit=3, method=method)
    assert e.value.code == 4
    x, st = mpm.solve(s["ctx"], s["mesh"], s["cfg"], s["Kd"], torch.zeros_like(rhs), method=method)
    assert st["iterations"] == 0 and st["status"] == 0 and not x.any()
