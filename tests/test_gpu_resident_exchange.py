"""The exchange between the blocks of the one-launch Krylov solves.

A solve of one launch hands its vectors from block to block through grid sums;
a block that met an older value of another block's rows would change the
iterates.  Many solves of the same system therefore have to agree bit for bit,
on a mesh of short iterations (the exchange is all of the time) and on one
whose blocks keep K in global memory.
"""
import numpy as np
import pytest

from test_gpu_resident_solve import system  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("key", ["few_quads", "punch", "block_13k"])
@pytest.mark.parametrize("method,precision", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_every_solve_meets_the_same_vectors(system, key, method, precision):  # noqa: F811
    s = system(key)
    mpm, torch = s["mpm"], s["torch"]
    cfg = dict(s["cfg"], mu=0.3, contact=1) if method == 2 else s["cfg"]
    K = s["Kd"].float() if precision else s["Kd"]
    rhs = torch.from_numpy(s["b"]).cuda()
    run = lambda: mpm.solve(s["ctx"], s["mesh"], cfg, K, rhs, precision=precision, tol=1e-8, maxit=5000,  # noqa: E731
                            method=method, inner_tol=1e-4)
    x, st = run()
    for _ in range(25):
        y, st2 = run()
        assert st2 == st and torch.equal(x, y)
    assert np.isfinite(x.cpu().numpy()).all()


@pytest.mark.parametrize("method,precision", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_a_wait_that_runs_out_is_an_error(system, method, precision):  # noqa: F811
    # with one poll a wait ends before the other blocks can have answered: every
    # block leaves and the call says so; the next solve on the context is the usual one
    s = system("punch")
    mpm, torch = s["mpm"], s["torch"]
    cfg = dict(s["cfg"], mu=0.3, contact=1) if method == 2 else s["cfg"]
    K = s["Kd"].float() if precision else s["Kd"]
    rhs = torch.from_numpy(s["b"]).cuda()
    ctx = s["ctx"]
    run = lambda: mpm.solve(ctx, s["mesh"], cfg, K, rhs, precision=precision, tol=1e-8, maxit=5000,  # noqa: E731
                            method=method, inner_tol=1e-4)
    x, st = run()
    ctx.check(mpm.lib().mpm_wait_limit(ctx.h, 1))
    try:
        with pytest.raises(mpm.MPMError) as e:
            run()
    finally:
        ctx.check(mpm.lib().mpm_wait_limit(ctx.h, 0))
    assert e.value.code == 4 and "wait" in str(e.value)
    y, st2 = run()
    assert st2 == st and torch.equal(x, y)
    assert mpm.lib().mpm_wait_limit(ctx.h, -1) == 1


@pytest.mark.parametrize("method,precision,cls", [(1, 0, 1), (1, 1, 1), (2, 0, 9), (2, 1, 9)])
def test_the_profile_has_the_solve(system, method, precision, cls):  # noqa: F811
    import ctypes as C
    s = system("punch")
    mpm, torch, ctx = s["mpm"], s["torch"], s["ctx"]
    cfg = dict(s["cfg"], mu=0.3, contact=1) if method == 2 else s["cfg"]
    K = s["Kd"].float() if precision else s["Kd"]
    n, ms = (C.c_longlong * 17)(), (C.c_double * 17)()
    ctx.check(mpm.lib().mpm_profile(ctx.h, 1))
    _, st = mpm.solve(ctx, s["mesh"], cfg, K, torch.from_numpy(s["b"]).cuda(), precision=precision, tol=1e-8,
                      maxit=5000, method=method, inner_tol=1e-4)
    ctx.check(mpm.lib().mpm_profile_read(ctx.h, n, ms))
    ctx.check(mpm.lib().mpm_profile(ctx.h, 0))
    assert n[cls] == max(st["refinements"], 1) and ms[cls] > 0.0  # one launch a solve


@pytest.mark.parametrize("precision,shear", [(0, 0.02), (0, 1e-4), (1, 1e-4)])
def test_bicgstab_of_a_nonsymmetric_tangent(precision, shear):
    # non-associated Drucker-Prager under a shear that yields: the residual of the
    # solution in FP64 on the host, to the bound of test_gpu_resident_solve
    import scipy.sparse as sp
    import torch
    from paper_2606_09275_gb300 import inputs, mpm
    from test_gpu_resident_solve import config
    cfg = config("cone", (4, 6), (12, 11, 9))
    ctx = mpm.Context()
    pts = inputs.make_points(cfg)
    P = mpm.Points(pts, capacity=12 * len(pts["x"]) + 400000)
    bz = inputs.body_z(cfg, 1)
    mesh = mpm.octree_build(ctx, cfg, P, body_z=bz)
    nd = mesh.info()["ndof"]
    dof, coord, mask = mesh.export("node_dof"), mesh.export("node_coord"), mesh.export("bcmask")
    x = np.zeros((nd, 3))
    x[dof[dof >= 0]] = coord[dof >= 0] * (cfg["L"] / (1 << cfg["depth_max"]))
    free = np.array([[not (m >> c) & 1 for c in range(3)] for m in mask])
    u = shear * np.stack([x[:, 2], 0.3 * x[:, 2], -0.2 * x[:, 2]], axis=1) * free
    du = torch.from_numpy(u.ravel().copy()).cuda()
    Kd = mpm.assemble(ctx, mesh, cfg, du, precision=precision, body_z=bz)["K"]
    K = sp.bsr_matrix((mpm.blocks(ctx, mesh, Kd, precision), mesh.export("col"), mesh.export("row_ptr")),
                      shape=(3 * nd, 3 * nd)).tocsr()
    assert abs(K - K.T).max() > 1e-3 * abs(K).max()
    b = np.random.default_rng(7).normal(size=3 * nd)
    bf = b * free.ravel()
    tol = 1e-8
    y, st = mpm.solve(ctx, mesh, cfg, Kd, torch.from_numpy(b).cuda(), precision=precision, tol=tol, maxit=5000,
                      method=0 if precision else 2, inner_tol=1e-4)
    assert st["status"] == 0 and st["relres"] <= tol
    r = (bf - K @ y.cpu().numpy()) * free.ravel()
    assert np.linalg.norm(r) <= 1.2 * tol * np.linalg.norm(bf)


@pytest.mark.parametrize("method", [1, 2])
def test_blocks_that_take_their_rows_in_several_passes(method):
    # more than 512 rows to a block (FP32), just below the largest mesh of these
    # solves; the bound of test_gpu_resident_solve
    import scipy.sparse as sp
    import torch
    from paper_2606_09275_gb300 import inputs, mpm
    from test_gpu_resident_solve import config
    cfg = config("indent", (6, 7), (54, 52, 28))
    ctx = mpm.Context()
    P = mpm.Points(inputs.make_points(cfg), capacity=2500000)
    bz = inputs.body_z(cfg, 1)
    mesh = mpm.octree_build(ctx, cfg, P, body_z=bz)
    nd = mesh.info()["ndof"]
    assert 512 * 151 < nd <= 98304
    Kd = mpm.assemble(ctx, mesh, cfg, torch.zeros(3 * nd, dtype=torch.float64, device="cuda"), precision=mpm.MIXED,
                      body_z=bz)["K"]
    K = sp.bsr_matrix((mpm.blocks(ctx, mesh, Kd, mpm.MIXED), mesh.export("col"), mesh.export("row_ptr")),
                      shape=(3 * nd, 3 * nd))
    free = np.array([[not (m >> c) & 1 for c in range(3)] for m in mesh.export("bcmask")]).ravel()
    b = np.random.default_rng(7).normal(size=3 * nd)
    cfg = dict(cfg, mu=0.3, contact=1) if method == 2 else cfg
    n0 = _launches(mpm, ctx)
    x, st = mpm.solve(ctx, mesh, cfg, Kd, torch.from_numpy(b).cuda(), precision=mpm.MIXED, tol=1e-8, maxit=5000,
                      method=method, inner_tol=1e-4)
    assert st["status"] == 0 and _launches(mpm, ctx) - n0 < st["iterations"]  # (in one launch)
    r = (b * free - K @ x.cpu().numpy()) * free
    assert np.linalg.norm(r) <= 1.2e-8 * np.linalg.norm(b * free)


@pytest.mark.parametrize("method", [1, 2])
def test_a_right_hand_side_near_the_smallest(system, method):  # noqa: F811
    # r.z and r.r fall below the smallest normal number on the way, where a
    # reciprocal overflows; the residual keeps 1.2 tol at tol = 1e-6
    s = system("punch")
    mpm, torch = s["mpm"], s["torch"]
    cfg = dict(s["cfg"], mu=0.3, contact=1) if method == 2 else s["cfg"]
    b = np.ldexp(s["b"] / np.linalg.norm(s["b"]), -490)
    x, st = mpm.solve(s["ctx"], s["mesh"], cfg, s["Kd"], torch.from_numpy(b).cuda(), tol=1e-6, maxit=2000, method=method)
    assert st["status"] == 0
    r = np.ldexp(b * s["free"] - s["K"] @ x.cpu().numpy(), 490) * s["free"]
    assert np.linalg.norm(r) <= 1.2e-6 * np.linalg.norm(np.ldexp(b, 490) * s["free"])


def _launches(mpm, ctx):
    import ctypes as C
    n = C.c_longlong()
    ctx.check(mpm.lib().mpm_launch_count(ctx.h, C.byref(n)))
    return n.value
