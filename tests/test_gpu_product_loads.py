"""Products with the FP32 matrix and its FP16 copy on both sides of the size
from which they take streaming loads (values and columns in 3/4 of the L2):
multigrid PCG and BiCGStab, GMRES and the refinement residual.

Reference: the relative residual on the free components, in FP64 on the host
from the exported blocks rounded to FP32.  The refinement measures the same
residual in double-float arithmetic (about 48 bits) and stops at tol = 1e-8, so
it may differ by 2^-48 times |K||x|/|b| (at most about 1e5 here), far below the
0.2 tol allowed.
"""
import numpy as np
import pytest

from paper_2606_09275_gb300 import inputs
from test_gpu_resident_solve import config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("key,block", [("indent", (24, 24, 14)), ("indent", (32, 32, 24)), ("cone", (30, 30, 26))])
def test_mixed_solution_residual(key, block):
    import scipy.sparse as sp
    import torch
    from paper_2606_09275_gb300 import mpm
    cfg = config(key, (5, 6), block)
    ctx = mpm.Context()
    pts = inputs.make_points(cfg)
    P = mpm.Points(pts, capacity=12 * len(pts["x"]) + 400000)
    mesh = mpm.octree_build(ctx, cfg, P, body_z=inputs.body_z(cfg, 1))
    info = mesh.info()
    nd, l2 = info["ndof"], torch.cuda.get_device_properties(0).L2_cache_size
    assert (40 * info["nslot"] > 0.75 * l2) == (block[2] > 20)  # the side of the rule that is meant
    zero = torch.zeros(3 * nd, dtype=torch.float64, device="cuda")
    Kd = mpm.assemble(ctx, mesh, cfg, zero, precision=mpm.MIXED, body_z=inputs.body_z(cfg, 1))["K"]
    K = sp.bsr_matrix((mpm.blocks(ctx, mesh, Kd, mpm.MIXED), mesh.export("col"), mesh.export("row_ptr")),
                      shape=(3 * nd, 3 * nd))
    free = np.array([[not (m >> c) & 1 for c in range(3)] for m in mesh.export("bcmask")]).ravel()
    b = np.random.default_rng(5).normal(size=3 * nd)
    bf = b * free
    rhs = torch.from_numpy(b).cuda()
    for method in (3, 4):
        x, st = mpm.solve(ctx, mesh, cfg, Kd, rhs, precision=mpm.MIXED, tol=1e-8, maxit=5000, method=method,
                          inner_tol=1e-4)
        assert st["status"] == 0 and st["relres"] <= 1e-8
        r = (bf - K @ x.cpu().numpy()) * free
        assert np.linalg.norm(r) <= 1.2e-8 * np.linalg.norm(bf)
