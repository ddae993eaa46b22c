"""The work that programs have this library do, as timed cases: the calls of
one Newton iteration (residual, tangent, Krylov solve), the mesh rebuild, and
whole load steps, time steps and adjoint sweeps, each through the package's
public entry points, over the sizes of the workloads in `inputs.workload`.

A case names the call (`op`), the workload it belongs to (material, body,
boundary conditions) and its discretisation: the octree depths, the block in
depth_min cells (nx, ny, nz), the points per cell and axis (ppc), their jitter
in point spacings, and the width of the refined region in finest cells.
"""
import math

import numpy as np
import torch

from paper_2606_09275_gb300 import autodiff, inputs, mpm


def _case(name, op, workload, depth, block, ppc=2, jitter=0.25, region=2.0, **more):
    c = dict(name=name, op=op, workload=workload, depth_min=depth[0], depth_max=depth[1],
             nx=block[0], ny=block[1], nz=block[2], ppc=ppc, jitter=round(jitter, 4), region=region)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: the residual of the elastic column (8^3 cells, 4096
        # points), as a line search or an explicit check evaluates it
        _case("residual_column", "residual", "column", (3, 3), (8, 8, 8), jitter=0.0, strain=0.01),
        # the residual of the indentation block at full size (1.9 M points): every
        # line-search trial of every Newton iteration
        _case("residual_indent", "residual", "indent", (6, 7), (64, 64, 56), strain=0.02),
        # residual and FP64 tangent of the punch of the paper's size (depth 3 to 6)
        _case("tangent_punch_fp64", "tangent", "punch", (3, 6), (8, 8, 4), precision=0, jitter=0.125,
              strain=0.02),
        # residual and FP32 tangent of the cone in the frictional layer (depth 4 to
        # 8, non-symmetric)
        _case("tangent_cone_mixed", "tangent", "cone", (4, 8), (10, 10, 12), precision=1,
              strain=0.002),
        # the same at full size on the indentation block: one Newton iteration's
        # assembly of the mixed path
        _case("tangent_indent_mixed", "tangent", "indent", (6, 7), (64, 64, 56), precision=1,
              strain=0.02),
        # the mesh rebuild that opens a load step (octree, splits, nodes, basis,
        # pattern, ghost faces), with the residual that follows it
        _case("build_indent", "build", "indent", (6, 7), (64, 64, 56), strain=0.0),
        # FP64 block-Jacobi PCG on the punch mesh (about 10 k unknowns): launches
        # and latency
        _case("solve_pcg_punch_fp64", "solve", "punch", (3, 6), (8, 8, 4), precision=0, method=1,
              jitter=0.125, tol=1e-12, strain=0.004),
        # FP64 BiCGStab, the automatic choice for the frictional cone
        _case("solve_bicgstab_cone_fp64", "solve", "cone", (4, 8), (10, 10, 12), precision=0,
              method=0, tol=1e-12, strain=0.0001),
        # multigrid PCG, FP32 inside FP64 refinement, at full size: the solve of
        # the headline workload
        _case("solve_mg_indent_mixed", "solve", "indent", (6, 7), (64, 64, 56), precision=1,
              method=3, tol=1e-10, strain=0.004),
        # one Newmark time step of the rolling sphere (free rigid body, FP64)
        _case("timestep_sphere_fp64", "timestep", "rolling_sphere", (3, 5), (8, 2, 2),
              precision=0, method=0, jitter=0.0),
        # the adjoint of two load steps of the punch with lognormal stiffness
        _case("adjoint_punch", "adjoint", "adjoint", (3, 5), (8, 8, 4), jitter=0.125, steps=2,
              method=1),
        # one whole load step of the indentation at full size, mixed precision
        _case("step_indent_mixed", "step", "indent", (6, 7), (64, 64, 56), precision=1, method=3),
    ]


def _odd(rng, hi, lo=2):
    """An integer of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: the same calls on blocks of other (odd) sizes, depths,
    points per cell, jitters and materials."""
    op = rng.choice(["residual", "residual", "tangent", "tangent", "build", "solve", "solve",
                     "solve", "step", "timestep", "adjoint"])
    jitter = rng.uniform(0.05, 0.25)
    if op == "timestep":
        return _unnamed(op, "rolling_sphere", (3, rng.choice([4, 5])), (rng.randint(5, 8), rng.randint(2, 4), rng.randint(2, 3)),
                        2, 0.0, 2.0, precision=rng.choice([0, 1]), method=0)
    if op == "adjoint":
        d = rng.choice([3, 4])
        jitter *= 0.5
        n = 1 << d
        return _unnamed(op, "adjoint", (d, 5), (rng.randint(n - 2, n), rng.randint(n - 2, n), rng.randint(n // 2 - 1, n // 2)),
                        2, jitter, 2.0, steps=rng.choice([1, 2, 3]), method=1)
    if op == "step":
        w, d = rng.choice(["punch", "indent"]), rng.choice([3, 4])
        n, up = 1 << d, 1 if d > 3 else rng.choice([2, 3])
        block = (rng.randint(n - 3, n), rng.randint(n - 3, n), rng.randint(n // 2 - 1, n // 2 + 1))
        if d == 3:
            jitter *= 0.5
        p, meth = rng.choice([(0, 0), (1, 0), (1, 3)])
        return _unnamed(op, w, (d, d + up), block, 2, jitter, 2.0, precision=p, method=meth,
                        facets=rng.choice([0, 0, 8, 16]) if w == "punch" else 0)
    w = rng.choice(["column", "punch", "cone", "indent", "indent", "cpt"])
    if op == "solve" and w == "column":
        w = "punch"
    strain = {"column": 0.01, "punch": 0.02, "indent": 0.02, "cone": 0.002, "cpt": 0.002}[w]
    if w in ("cone", "cpt"):
        d = rng.choice([4, 5]) if op != "solve" else 4
        n, up = 1 << d, rng.choice([2, 3, 4]) if d == 4 else rng.choice([1, 2])
        block = (_odd(rng, n, 6), _odd(rng, n, 6), rng.randint(6, n - 2))
        if w == "cpt":  # (its cone stands on the cube's edge: no split may leave the cube)
            jitter *= 0.2
    elif w == "column":
        d, up = rng.choice([2, 3, 4, 5, 6]), 0
        n = 1 << d
        block = (n, n, n) if rng.random() < 0.5 else (_odd(rng, n), _odd(rng, n), _odd(rng, n))
    else:
        d = rng.choice([3, 4, 5, 6])
        n, up = 1 << d, (rng.choice([2, 3]) if d == 3 else 1 if d == 6 else rng.choice([1, 2]))
        block = (_odd(rng, n, n // 2), _odd(rng, n, n // 2), rng.randint(n // 4 + 1, n - 1))
        if d == 3:
            jitter *= 0.5
    ppc = rng.choice([2, 2, 3, 1]) if block[0] * block[1] * block[2] < 50000 else 2
    more = dict(strain=strain)
    if op == "tangent":
        more.update(precision=rng.choice([0, 1, 1]) if d < 6 else 1)
    if op == "solve":
        p = rng.choice([0, 1])
        sym = w in ("punch", "indent")
        meth = rng.choice([0, 1, 3] if sym else [0, 0, 4]) if d < 5 else (3 if sym else 0)
        if d == 6:
            p = 1
        if meth == 4 or w == "cpt":
            p = 0
        jitter *= 0.5
        more.update(precision=p, method=meth, tol=1e-12 if p == 0 else 1e-10,
                    strain=0.002 if sym else 0.0001)
        ppc = 2
    return _unnamed(op, w, (d, d + up), block, ppc, jitter, 2.0, **more)


def _unnamed(*a, **more):
    c = _case("", *a, **more)
    del c["name"]
    return c


# ---------------------------------------------------------------- configurations

def _config(case, seed):
    """The workload's parameters on the case's block and depths."""
    cfg = inputs.workload(case["workload"], depth_min=case["depth_min"], depth_max=case["depth_max"])
    h = cfg["L"] / (1 << case["depth_min"])
    hi = (case["nx"] * h, case["ny"] * h, case["nz"] * h)
    spacing = h / case["ppc"]
    top = cfg["points"]["hi"][2]
    cfg["bc"] = [(0, 0.0, inputs.ROLLER_X), (0, hi[0], inputs.ROLLER_X), (1, 0.0, inputs.ROLLER_Y),
                 (1, hi[1], inputs.ROLLER_Y), (2, 0.0, inputs.FIXED)]
    cfg["points"].update(lo=(0.0, 0.0, 0.0), hi=hi, spacing=spacing, jitter=case["jitter"] * spacing,
                         seed=1)
    cfg["dx_region"] = case["region"] * cfg["L"] / (1 << case["depth_max"])
    if cfg["body"]:
        b = cfg["body"]
        b["z0"] += hi[2] - top
        if case["workload"] == "rolling_sphere":
            v = 0.02 + 0.02 * np.random.default_rng(seed).random()  # rolling already
            b["cx"], b["cy"] = 1.0, 0.5 * hi[1]
            b["v"], b["w"] = (v, 0.0, 0.0), (0.0, v / b["r"], 0.0)
        if case.get("facets"):  # the punch as a triangulated prism, its vertices off the cell planes
            b.update(kind=3, mesh=inputs.cylinder_mesh(b["r"], 0.6, case["facets"], phase=0.5))
        if case["workload"] not in ("cpt", "rolling_sphere"):  # (the cpt's cone stands on the block's edge x = y = 0)
            b["cx"], b["cy"] = 0.5 * hi[0], 0.5 * hi[1]
    return cfg


def _initial(cfg, seed):
    """The initial points: a lattice that is the same for every seed (so that the
    mesh is), of lognormal Young's modulus."""
    pts = inputs.make_points(cfg)
    pts["E"] *= np.exp(np.random.default_rng(seed).normal(0.0, 0.2, len(pts["E"])))
    return pts


def _points(case, cfg, seed):
    """The points on the device, with room for the refined region's splits."""
    pts = _initial(cfg, seed)
    n = len(pts["x"])
    return mpm.Points(pts, capacity=2 * n if n > 500000 else 12 * n + 400000,
                      velocity=case["op"] == "timestep")


def _increment(case, cfg, mesh, seed):
    """A nodal increment as Newton meets them: a settlement under the body, of
    the given peak strain, on the free components, with a little noise."""
    nd = mesh.info()["ndof"]
    dof = torch.from_numpy(mesh.export("node_dof").astype(np.int64)).cuda()
    coord = torch.from_numpy(mesh.export("node_coord")).cuda().double()
    mask = torch.from_numpy(mesh.export("bcmask")).cuda()
    unit = cfg["L"] / (1 << cfg["depth_max"])
    x = torch.zeros((nd, 3), dtype=torch.float64, device="cuda")
    x[dof[dof >= 0]] = coord[dof >= 0] * unit
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = torch.rand(4, generator=g, device="cuda", dtype=torch.float64).tolist()
    hi = cfg["points"]["hi"]
    c = torch.tensor([hi[0] * (0.45 + 0.1 * rnd[0]), hi[1] * (0.45 + 0.1 * rnd[1]), hi[2]],
                     dtype=torch.float64, device="cuda")
    s = 0.25 * min(hi)
    a = case["strain"] * s * (0.9 + 0.2 * rnd[2])
    r = (x - c) / s
    w = torch.exp(-0.5 * (r * r).sum(1))
    u = torch.stack([0.3 * a * r[:, 0] * w, 0.3 * a * r[:, 1] * w, -a * w], dim=1)
    u += case["strain"] * 0.02 * unit * (torch.rand((nd, 3), generator=g, device="cuda",
                                                    dtype=torch.float64) - 0.5)
    free = torch.stack([(mask >> d) & 1 for d in range(3)], dim=1) == 0
    return (u * free).reshape(-1).contiguous()


# ---------------------------------------------------------------- the calls

def prepare(case, seed):
    cfg = _config(case, seed)
    ctx = mpm.Context()
    s = dict(case=case, cfg=cfg, ctx=ctx, bz=inputs.body_z(cfg, 1) if cfg["body"] else None)
    op = case["op"]
    if op == "adjoint":
        n = case["nx"] * case["ny"] * case["nz"] * case["ppc"] ** 3
        path = autodiff.LoadPath(ctx, cfg, _initial(cfg, seed), case["steps"],
                                 capacity=12 * n + 60000, method=case["method"])
        E = torch.from_numpy(path.points["E"]).cuda()
        ys = torch.from_numpy(path.points["ys"]).cuda()
        _, s["ckpts"], _ = path.run(E, ys)
        s["path"] = path
        return s
    s["points"] = _points(case, cfg, seed)
    if op in ("step", "timestep"):
        s["body"] = mpm.body_start(cfg) if op == "timestep" else None
        return s
    if op == "build":
        s["mesh"] = None
        return s
    s["mesh"] = mpm.octree_build(ctx, cfg, s["points"], body_z=s["bz"])
    s["du"] = _increment(case, cfg, s["mesh"], seed)
    if op == "solve":
        a = mpm.assemble(ctx, s["mesh"], cfg, s["du"], precision=mpm.FP64, body_z=s["bz"])
        # the mixed solve's matrix is the FP64 tangent rounded once
        s["K"] = a["K"].float() if case["precision"] == mpm.MIXED else a["K"]
        s["rhs"] = -a["R"]
    return s


def _residual(s, mesh, du, precision, tangent):
    a = mpm.assemble(s["ctx"], mesh, s["cfg"], du, precision=precision, tangent=tangent,
                     body_z=s["bz"])
    out = dict(R=a["R"], reaction=a["reaction"],
               norms=np.array([a["fint_norm"], a["fextc_norm"]]))
    if tangent:
        out["K"] = a["K"]
    return out


def run(s):
    case, cfg, ctx = s["case"], s["cfg"], s["ctx"]
    op = case["op"]
    if op == "residual":
        return _residual(s, s["mesh"], s["du"], mpm.FP64, False)
    if op == "tangent":
        return _residual(s, s["mesh"], s["du"], case["precision"], True)
    if op == "build":
        p = s["points"].clone()
        s["mesh"] = mpm.octree_build(ctx, cfg, p, body_z=s["bz"], mesh=s["mesh"])
        info = s["mesh"].info()
        du = torch.zeros(3 * info["ndof"], dtype=torch.float64, device="cuda")
        out = _residual(s, s["mesh"], du, mpm.FP64, False)
        out.update(info=np.array([info[k] for k in sorted(info)], dtype=np.int64),
                   x=p.t["x"][:p.count], lp=p.t["lp"][:p.count], V0=p.t["V0"][:p.count])
        return out
    if op == "solve":
        x, _ = mpm.solve(ctx, s["mesh"], cfg, s["K"], s["rhs"], precision=case["precision"],
                         tol=case["tol"], maxit=100000, method=case["method"], inner_tol=1e-4)
        return x
    if op == "adjoint":
        dE, dys, _ = s["path"].gradient(s["ckpts"], np.array([0.0, 0.0, 1.0]))
        return dict(dE=dE, dys=dys)
    p = s["points"].clone()
    kw = dict(tol=1e-11, lin_tol=1e-10, lin_maxit=100000, precision=case["precision"],
              method=case["method"], inner_tol=1e-4, mg_reuse=1)
    if op == "timestep":
        b = dict(s["body"])
        st = mpm.step(ctx, cfg, p, dt=cfg["dt"], body_state=b, **kw)
        extra = dict(v=p.t["v"][:p.count], q=st["body_q"], body_v=st["body_v"], body_w=st["body_w"])
    else:
        st = mpm.step(ctx, cfg, p, body_z=s["bz"], **kw)
        extra = {}
    n = p.count
    return dict(x=p.t["x"][:n], lp=p.t["lp"][:n], F=p.t["F"][:n], be=p.t["be"][:n],
                reaction=st["reaction"], sizes=np.array([st["npts"], st["ndof"], st["nnzb"]]), **extra)


# ---------------------------------------------------------------- minimal work

def _sizes(case):
    """Points, nodes and 3x3 blocks of the adapted mesh, estimated: the block's
    own cells, and for each finer level the cells around the body's footprint."""
    cfg = _config(case, 0)
    h = cfg["L"] / (1 << case["depth_min"])
    cells = float(case["nx"] * case["ny"] * case["nz"])
    P = cells * max(case["ppc"], 2) ** 3  # (one point per cell splits)
    nodes = (case["nx"] + 1.0) * (case["ny"] + 1.0) * (case["nz"] + 1.0)
    if cfg["body"]:
        quarter = 0.25 if case["workload"] == "cpt" else 1.0
        r = cfg["body"]["r"] * (0.3 if case["workload"] in ("cone", "cpt", "rolling_sphere") else 1.0)
        for lev in range(case["depth_min"] + 1, case["depth_max"] + 1):
            hl = cfg["L"] / (1 << lev)
            reach = r + (case["region"] + 3.0) * hl
            extra = quarter * min(3.14 * reach * reach * (case["region"] + 3.0) * hl, 0.5 * cells * h ** 3) / hl ** 3
            P += extra * 4.0
            nodes += extra * 0.45
    return P, nodes, (100.0 if case["jitter"] else 21.0) * nodes


def work(case):
    """Bytes that have to be read and written once, and operations: per point
    and support node (16 on average) 18 flops each for the deformation gradient
    and for the force, about 600 for the constitutive update, 54 per pair of
    support nodes of the tangent; per 3x3 block 18 flops of one product."""
    P, nodes, nnzb = _sizes(case)
    ns, op = 16.0, case["op"]
    point = P * 8.0 * (9 + 6 + 4)                  # b_e, constants in; F and stress state
    basis = P * ns * (4 * 8 + 4)                   # S, grad S and the support
    vec = nodes * 3 * 8.0
    res = dict(bytes=point + basis + 2 * vec, flops=P * (ns * 36.0 + 600.0))
    w = 4.0 if case.get("precision") else 8.0
    if op == "residual":
        return res
    if op == "tangent":
        return dict(bytes=res["bytes"] + 9 * w * nnzb, flops=res["flops"] + P * ns * ns * 54.0)
    if op == "build":
        return dict(bytes=res["bytes"] + basis + nnzb * 8.0 + P * 8.0 * 33,
                    flops=res["flops"] + P * ns * 4 * 20.0)
    if op == "solve":
        return dict(bytes=nnzb * (9 * w + 4) + 2 * vec, flops=nnzb * 18.0)
    n = case.get("steps", 1)
    return dict(bytes=n * (2 * res["bytes"] + basis + nnzb * (9 * w + 4) + P * 8.0 * 66),
                flops=n * (2 * res["flops"] + P * ns * ns * 54.0 + nnzb * 18.0))


# ---------------------------------------------------------------- 64-bit values

def exact(case, seed):
    """The residual of the elastic column on the full uniform grid, written out
    in plain torch: there the GIMP basis is a product of one-dimensional ones.
    The adapted octrees of the other cases have no such form."""
    n = 1 << case["depth_min"]
    if case["op"] != "residual" or case["workload"] != "column" or (case["nx"], case["ny"], case["nz"]) != (n, n, n) or n > 16:
        return None
    s = prepare(case, seed)  # (the inputs: points and increment)
    cfg, du = s["cfg"], s["du"].cpu()
    pts = {k: torch.from_numpy(v) for k, v in s["points"].numpy().items()}
    h = cfg["L"] / n
    # one-dimensional basis over the (at most 3) cells that a domain overlaps
    lo, hi = (pts["x"] - pts["lp"]) / h, (pts["x"] + pts["lp"]) / h
    for b in (lo, hi):
        near = torch.round(b)
        b[(b - near).abs() < 1e-9] = near[(b - near).abs() < 1e-9]
    V = hi - lo
    lo, hi = lo.clamp(min=0.0), hi.clamp(max=float(n))
    c0 = torch.floor(lo).clamp(max=n - 1)
    P = len(c0)
    S1 = torch.zeros((P, 3, 4), dtype=torch.float64)  # nodes c0 .. c0 + 3
    D1 = torch.zeros_like(S1)
    for k in range(3):
        a, e = torch.maximum(lo, c0 + k), torch.minimum(hi, c0 + k + 1)
        wk = ((e - a).clamp(min=0.0) / V)
        xi = 0.5 * (a + e) - (c0 + k)
        S1[..., k] += wk * (1.0 - xi)
        S1[..., k + 1] += wk * xi
        D1[..., k] -= wk / h
        D1[..., k + 1] += wk / h
    # sum of the weights per axis: gradients along one axis carry the others' values
    S = torch.einsum("pi,pj,pk->pkji", S1[:, 0], S1[:, 1], S1[:, 2]).reshape(P, 64)
    dS = torch.stack([torch.einsum("pi,pj,pk->pkji", D1[:, 0], S1[:, 1], S1[:, 2]).reshape(P, 64),
                      torch.einsum("pi,pj,pk->pkji", S1[:, 0], D1[:, 1], S1[:, 2]).reshape(P, 64),
                      torch.einsum("pi,pj,pk->pkji", S1[:, 0], S1[:, 1], D1[:, 2]).reshape(P, 64)], dim=2)
    o = torch.arange(4)
    ijk = torch.stack([o.repeat(16), o.repeat_interleave(4).repeat(4), o.repeat_interleave(16)], dim=1)
    node = (c0.long()[:, None, :] + ijk[None]).clamp(max=n)
    lin = node[..., 0] + (n + 1) * (node[..., 1] + (n + 1) * node[..., 2])
    # nodes are numbered along the Morton curve
    m = torch.arange(n + 1)
    z, y, x = torch.meshgrid(m, m, m, indexing="ij")
    key = torch.zeros_like(x)
    for b in range(8):
        key |= ((x >> b) & 1) << (3 * b) | ((y >> b) & 1) << (3 * b + 1) | ((z >> b) & 1) << (3 * b + 2)
    dof = torch.empty((n + 1) ** 3, dtype=torch.long)
    dof[torch.argsort(key.reshape(-1))] = torch.arange((n + 1) ** 3)
    d = dof[lin]
    u = du.reshape(-1, 3)[d]
    dF = torch.eye(3, dtype=torch.float64) + torch.einsum("pvi,pvj->pij", u, dS)
    be = pts["be"]
    B = torch.stack([be[:, 0], be[:, 3], be[:, 5], be[:, 3], be[:, 1], be[:, 4], be[:, 5], be[:, 4], be[:, 2]],
                    dim=1).reshape(P, 3, 3)
    lam, Q = torch.linalg.eigh(dF @ B @ dF.transpose(1, 2))
    eps = 0.5 * torch.log(lam)
    nu = cfg["nu"]
    mu = pts["E"] / (2 * (1 + nu))
    lm = pts["E"] * nu / ((1 + nu) * (1 - 2 * nu))
    tau = lm[:, None] * eps.sum(1, keepdim=True) + 2 * mu[:, None] * eps
    T = Q @ torch.diag_embed(tau) @ Q.transpose(1, 2)
    M = pts["V0"][:, None, None] * (T @ torch.linalg.inv(dF).transpose(1, 2))
    nd = (n + 1) ** 3
    fint = torch.zeros((nd, 3), dtype=torch.float64)
    fint.index_add_(0, d.reshape(-1), torch.einsum("pij,pvj->pvi", M, dS).reshape(-1, 3))
    g = torch.tensor(cfg["g"], dtype=torch.float64)
    fext = torch.zeros((nd, 3), dtype=torch.float64)
    fext.index_add_(0, d.reshape(-1), ((S * pts["mass"][:, None])[..., None] * g).reshape(-1, 3))
    return dict(R=(fint - fext).reshape(-1), reaction=None,
                norms=np.array([fint.norm().item(), fext.norm().item()]))
