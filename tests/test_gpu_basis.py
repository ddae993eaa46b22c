"""The GIMP basis over domains from half a leaf to almost two leaves long: one
to 27 leaf intersections, whose corner values the kernel tabulates 16 at a
time, and supports up to the limit of 64 nodes.  The bounds are those of the
mesh parity test: a value is a sum of at most 27 terms of some eight roundings
each, 27 * 8 * 1.1e-16 = 2.4e-14 of a total of one.
"""
import numpy as np
import pytest

import oracle
from paper_2606_09275_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [0.5, 1.0, 1.5, 1.9])
def test_domains_of_up_to_27_leaves(length):
    from paper_2606_09275_gb300 import mpm
    cfg = inputs.workload("column", beta=0.4, points=dict(spacing=length / 8, jitter=0.02, seed=4, ys=1e4))
    pts = inputs.make_points(cfg)
    om = oracle.Model(cfg, pts)
    om.build(nosplit=True)
    mesh = mpm.octree_build(mpm.Context(), cfg, mpm.Points(pts), nosplit=True)
    nsup, sidx, S, dS = om.support()
    assert np.array_equal(mesh.export("nsup"), nsup)
    mask = np.arange(64)[None, :] < nsup[:, None]
    assert np.array_equal(np.where(mask, mesh.export("sidx"), -1), np.where(mask, sidx, -1))
    assert np.max(np.abs(np.where(mask, mesh.export("S") - S, 0))) < 1e-13
    scale = (1 << cfg["depth_max"]) / cfg["L"]
    assert np.max(np.abs(np.where(mask[..., None], mesh.export("dS") - dS, 0))) < 1e-13 * scale
    if length > 1.5:
        assert nsup.max() == 64


@pytest.mark.parametrize("length, longest", [(0.5, 125), (1.5, 294), (1.9, 256)])
def test_rows_around_256_columns(length, longest):
    """Rows beyond 256 columns take the pattern builder's large set, whole numbers throughout."""
    from paper_2606_09275_gb300 import mpm
    cfg = inputs.workload("column", beta=0.4, points=dict(spacing=length / 8, jitter=0.02, seed=4, ys=1e4))
    pts = inputs.make_points(cfg)
    om = oracle.Model(cfg, pts)
    om.build(nosplit=True)
    mesh = mpm.octree_build(mpm.Context(), cfg, mpm.Points(pts), nosplit=True)
    rp, col = om.pattern()
    assert np.array_equal(mesh.export("row_ptr"), rp)
    assert np.array_equal(mesh.export("col"), col)
    assert np.diff(rp).max() == longest
