"""The tangent gather beyond the sizes of the parity meshes: supports of more
than 32 nodes (domains longer than a leaf, kept whole by a small beta), whose
columns past the 32nd take the gather's own loop, in both precisions and
against the oracle, with the tolerances of the assembly parity test (1e-10 in
FP64; 2e-6 in FP32, some 30 roundings of 6e-8 over the sums of a block).
"""
import numpy as np
import pytest

import oracle
from paper_2606_09275_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("model", [1, 2])
def test_supports_of_more_than_32_nodes(precision, model):
    import torch
    from paper_2606_09275_gb300 import mpm
    cfg = inputs.workload("column", beta=0.6, model=model, phi=0.5, psi=0.0,
                          points=dict(spacing=1.5 / 8, jitter=0.02, seed=4, ys=1e4))
    pts = inputs.make_points(cfg)
    ctx = mpm.Context()
    P = mpm.Points(pts)
    mesh = mpm.octree_build(ctx, cfg, P)
    assert mesh.info()["maxs"] > 32
    om = oracle.Model(cfg, pts)
    om.build()
    nd = om.counts()["ndof"]
    du = 2e-4 * np.random.default_rng(3).standard_normal(3 * nd)
    free = np.array([[not (m >> c) & 1 for c in range(3)] for m in om.bcmask()])
    du[~free.ravel()] = 0.0
    o = om.assemble(du, load=1.0)
    g = mpm.assemble(ctx, mesh, cfg, torch.tensor(du, device="cuda"), precision=precision)
    rp, col = om.pattern()
    row = np.repeat(np.arange(nd), np.diff(rp))
    keep = free[row][:, :, None] & free[col][:, None, :]
    Kg = mpm.blocks(ctx, mesh, g["K"], precision)
    tol = (1e-10 if precision == 0 else 2e-6) * np.abs(o["K"]).max()
    assert np.max(np.abs(np.where(keep, Kg - o["K"], 0))) <= tol
    assert np.max(np.abs(g["R"].cpu().numpy() - o["R"])) <= 1e-10 * np.abs(o["R"]).max()
