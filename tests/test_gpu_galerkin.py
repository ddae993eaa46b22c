"""The Galerkin operators of the multigrid hierarchy, through the iteration
counts of the solves they precondition: on the small indentation block
(33,668 dofs, every level of stencil radius 2) the gathered products give the
counts that the scattered ones gave, 28 in FP64 and 38 mixed; an entry put at
a wrong offset or lost costs far more than the one iteration left for another
rounding of the operators.
"""
import numpy as np
import pytest

from paper_2606_09275_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision, count", [(0, 28), (1, 38)])
def test_iterations_with_the_gathered_products(precision, count):
    import torch
    from paper_2606_09275_gb300 import mpm
    cfg = inputs.workload("indent_small")
    pts = inputs.make_points(cfg)
    ctx = mpm.Context()
    P = mpm.Points(pts, capacity=64 * len(pts["x"]))
    mesh = mpm.octree_build(ctx, cfg, P)
    n = 3 * mesh.info()["ndof"]
    g = mpm.assemble(ctx, mesh, cfg, torch.zeros(n, device="cuda", dtype=torch.float64), precision=precision)
    b = torch.tensor(np.random.default_rng(1).standard_normal(n), device="cuda")
    x, st = mpm.solve(ctx, mesh, cfg, g["K"], b, tol=1e-10, maxit=500, method=3, precision=precision)
    assert st["status"] == 0
    assert abs(st["iterations"] - count) <= 1
