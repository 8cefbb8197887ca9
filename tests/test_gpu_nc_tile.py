"""The non-circular forward's tile sums at the edges of their range, against the
FP64 oracle at the FP32 path's bound: axial footprints above and below a row
(lanes in step, taking turns, and the gather below half a row), few columns in
reach of a tile (columns taking turns), narrow and wide footprints, remainders."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import workloads as W
from gpu_util import TOL_F32, rel_l2

pytestmark = pytest.mark.gpu

# nx, ny, nz, nu, nv, du, dv (voxels 1.6 x 1.6 x 1.3 mm, magnification about 2)
SIZES = {
    "tall": (19, 22, 17, 70, 45, 2.1, 1.4),       # rows per voxel about 1.9
    "low": (17, 9, 33, 41, 37, 2.9, 3.6),         # about 0.7: neighbours share a row
    "lowest": (12, 13, 20, 33, 20, 2.9, 6.0),     # below half a row: the gather
    "coarse": (40, 37, 12, 9, 31, 9.0, 2.0),      # many columns to a cell
    "fine": (7, 6, 9, 150, 70, 0.9, 1.3),         # few columns to a tile, up to 8 cells wide
}


@pytest.mark.parametrize("proj", ["sf", "dd", "sftt"])
@pytest.mark.parametrize("size", SIZES)
def test_noncircular_forward_matches_oracle(size, proj):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_16741_gb300 as ct
    nx, ny, nz, nu, nv, du, dv = SIZES[size]
    nview = 35  # one more block of views than fits
    th = 0.1 + 2 * np.pi * np.arange(nview) / nview
    spec = W.GeometrySpec("noncirc3d", "flat", nx, ny, nz, 1.6, 1.6, 1.3, nu, nv, du, dv, nview, theta=th,
                          phi=0.09 * np.cos(2 * th), psi=0.02 * np.sin(3 * th), sad=320.0, sdd=640.0, x_src=1.2,
                          z_src=-2.0, u_ofst=-2.6, v_ofst=1.7, x_ofst=2.0, y_ofst=-1.0, z_ofst=1.5)
    g = ct.Geometry.from_spec(spec)
    x = torch.as_tensor(W.random_volume(spec, seed=2, batch=2) - 0.3, dtype=torch.float32).cuda()
    y = ct.forward(g, x, proj)
    for b in range(2):
        ref = oracle.forward(spec, proj, x[b].double().cpu().numpy())
        assert np.linalg.norm(ref) > 0 and rel_l2(y[b].cpu().numpy(), ref) <= TOL_F32
    assert torch.equal(y[1], ct.forward(g, x[1].contiguous(), proj))
    views = [0, 3, 34]
    assert torch.equal(ct.forward(g.subset(views), x, proj), y[:, views])


# du, dv: half of the views at magnification 2, half at 1.33
MIXED = {
    "kernels": (2.9, 3.6),  # axial footprints of about 0.7 and 0.48 rows: tile sums and the gather
    "cells": (1.6, 2.0),    # 6 and 4 cells
    "rows": (1.6, 1.25),    # 4 and 3 rows
}


@pytest.mark.parametrize("proj", ["sf", "dd", "sftt"])
@pytest.mark.parametrize("mix", MIXED)
def test_a_view_does_not_depend_on_the_others(mix, proj):
    """Views on either side of a dispatch rule: each has the same projection alone, among its like and in the mix."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_16741_gb300 as ct
    du, dv = MIXED[mix]
    nview = 38
    th = 0.1 + 2 * np.pi * np.arange(nview) / nview
    sad = np.where(np.arange(nview) % 2 == 0, 320.0, 480.0)
    spec = W.GeometrySpec("noncirc3d", "flat", 37, 33, 29, 1.6, 1.6, 1.3, 75, 50, du, dv, nview, theta=th,
                          phi=0.05 * np.cos(2 * th), psi=0.02 * np.sin(3 * th), sad=sad, sdd=640.0, x_src=1.2,
                          z_src=-2.0, u_ofst=-2.6, v_ofst=1.7, x_ofst=2.0, y_ofst=-1.0, z_ofst=1.5)
    g = ct.Geometry.from_spec(spec)
    x = torch.as_tensor(W.random_volume(spec, seed=3)[0] - 0.3, dtype=torch.float32).cuda()
    y = ct.forward(g, x, proj)
    assert rel_l2(y.cpu().numpy(), oracle.forward(spec, proj, x.double().cpu().numpy())) <= TOL_F32
    for views in (list(range(0, nview, 2)), list(range(1, nview, 2)), [4], [5]):
        assert torch.equal(ct.forward(g.subset(views), x, proj), y[views])


@pytest.mark.parametrize("proj", ["sf", "dd"])
def test_steep_views_near_the_source(proj):
    """Views whose footprints change by more than a cell along a column (a small volume close to the source, the
    detector rolled by 51 degrees) beside upright ones: either forward, in one scan."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_16741_gb300 as ct
    th = np.array([0.37, 1.2, 2.9, 4.4])
    spec = W.GeometrySpec("noncirc3d", "flat", 8, 8, 6, 1.6, 1.6, 1.96, 50, 44, 2.4, 2.5, 4, theta=th,
                          phi=np.array([0.115, 0.0, 0.115, 0.05]), psi=np.array([0.892, 0.0, 0.892, 0.02]),
                          sad=np.array([20.4, 30.0, 20.4, 30.0]), sdd=60.8)
    g = ct.Geometry.from_spec(spec)
    x = torch.as_tensor(W.random_volume(spec, seed=5)[0] - 0.3, dtype=torch.float32).cuda()
    y = ct.forward(g, x, proj)
    assert rel_l2(y.cpu().numpy(), oracle.forward(spec, proj, x.double().cpu().numpy())) <= TOL_F32
    for views in ([0, 2], [1, 3], [2]):
        assert torch.equal(ct.forward(g.subset(views), x, proj), y[views])
