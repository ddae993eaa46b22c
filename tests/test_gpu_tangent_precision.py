"""The FP32 tangent against the FP64 one on the same mesh and increment.

An entry of K is a sum over some 64 sources at the most (the points that two
neighbouring nodes share), taken in order with one rounding of the sum a source:
a random walk of roundings of up to 2^-24 of a partial sum that grows with the
number of sources, in the rms 2^-24 / sqrt(3) sqrt(64 / 3) = 1.6e-7 of the entry,
and below 2e-7 with the roundings of the terms themselves (their own two or
three of 2^-24, averaged over the sources).  Three roundings of the sum a source
come to sqrt(3) times that.
"""
import pytest

from paper_2606_09275_gb300 import inputs
from test_gpu_resident_solve import config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("key,depth,block", [("indent", (5, 6), (32, 32, 16)), ("punch", (3, 6), (8, 8, 4))])
def test_mixed_tangent_error(key, depth, block):
    import torch
    from paper_2606_09275_gb300 import mpm
    cfg = config(key, depth, block)
    ctx = mpm.Context()
    pts = inputs.make_points(cfg)
    P = mpm.Points(pts, capacity=12 * len(pts["x"]) + 400000)
    bz = inputs.body_z(cfg, 1)
    mesh = mpm.octree_build(ctx, cfg, P, body_z=bz)
    n = 3 * mesh.info()["ndof"]
    g = torch.Generator(device="cuda").manual_seed(9)
    du = 1e-4 * cfg["L"] / (1 << depth[1]) * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    K = [mpm.assemble(ctx, mesh, cfg, du, precision=p, body_z=bz)["K"].double() for p in (mpm.FP64, mpm.MIXED)]
    assert ((K[1] - K[0]).norm() / K[0].norm()).item() <= 2e-7
