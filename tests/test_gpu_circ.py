"""The circular cone-beam projection pair over its dispatch: taps of a footprint
(1 to 8 cells, and beyond), rows per voxel (below 1, 2, 4 and 8, and beyond),
chunks, patches, tiles and columns with remainders, views split over a cluster
and not, against the FP64 oracle at the FP32 path's bound."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import workloads as W
from gpu_util import TOL_F32, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ct():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2503_16741_gb300 as ct
    ct.load()
    return ct


# nx, ny, nz, nu, nv, views, du, dv (voxels 1.6 x 1.6 x 1.3 mm, magnification about 2)
SIZES = {
    "narrow-short": (19, 13, 16, 40, 30, 12, 7.0, 3.1),      # 2 cells (DD), sv < 1, one chunk
    "ragged": (17, 9, 37, 33, 47, 67, 3.4, 2.9),             # 3 / 4 cells, remainders, views split 8 ways
    "tall": (9, 22, 21, 45, 35, 9, 2.4, 1.6),                # 4 / 8 cells, sv in (1, 2), no split
    "taller": (10, 10, 45, 60, 70, 37, 1.3, 0.9),            # 8 cells, sv in (2, 4)
    "tallest": (9, 9, 13, 70, 90, 21, 1.3, 0.5),             # 8 cells, sv in (4, 8)
    "beyond": (6, 7, 5, 70, 60, 5, 0.7, 0.3),                # more than 8 cells, sv > 8: the general kernel
    "narrow-detector": (12, 12, 12, 7, 20, 8, 3.0, 3.0),     # fewer cells than a window
    "flat-volume": (12, 12, 3, 30, 40, 6, 2.6, 2.9),         # no z-major copy
    "large-detector": (11, 10, 37, 290, 130, 3, 0.9, 1.1),   # tiles of 64 rows, and of 290 = 9 x 32 + 2 cells
    "off": (24, 24, 140, 20, 40, 40, 2.2, 2.9),              # most of the volume beside the detector; 2 z-blocks
}


def _spec(det, nx, ny, nz, nu, nv, views, du, dv):
    return W.GeometrySpec("circ3d", det, nx, ny, nz, 1.6, 1.6, 1.3, nu, nv, du, dv, views,
                          theta=0.2 + 2 * np.pi * np.arange(views) / views, sad=320.0, sdd=640.0, x_src=1.2,
                          z_src=-2.0, u_ofst=-2.6, v_ofst=1.7, x_ofst=2.0, y_ofst=-1.0, z_ofst=1.5)


def _check(got, ref, what):
    assert np.linalg.norm(ref) > 0
    assert rel_l2(got, ref) <= TOL_F32, what


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("proj", ["sf", "dd", "voxel"])
def test_circ_back_matches_oracle(ct, det, size, proj):
    spec = _spec(det, *SIZES[size])
    g = ct.Geometry.from_spec(spec)
    y = W.random_sino(spec, seed=2, batch=2) - 0.3
    yd = torch.as_tensor(y, dtype=torch.float32).cuda()
    y = yd.double().cpu().numpy()  # the oracle's input is what the GPU was given
    x, r = ct.back(g, yd, proj), ct.back(g, yd, proj, mode="recon")
    for b in range(2):
        _check(x[b].cpu().numpy(), oracle.back(spec, proj, y[b]), "proj")
        _check(r[b].cpu().numpy(), oracle.back_recon(spec, y[b], proj), "recon")
    assert torch.equal(x[1], ct.back(g, yd[1].contiguous(), proj))


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("proj", ["sf", "dd", "voxel"])
def test_circ_forward_matches_oracle(ct, det, size, proj):
    spec = _spec(det, *SIZES[size])
    g = ct.Geometry.from_spec(spec)
    x = torch.as_tensor(W.random_volume(spec, seed=2, batch=2) - 0.3, dtype=torch.float32).cuda()
    y = ct.forward(g, x, proj)
    for b in range(2):
        _check(y[b].cpu().numpy(), oracle.forward(spec, proj, x[b].double().cpu().numpy()), "forward")
    assert torch.equal(y[1], ct.forward(g, x[1].contiguous(), proj))
    views = [0, 2]
    assert torch.equal(ct.forward(g.subset(views), x, proj), y[:, views])


@pytest.mark.parametrize("views", [31, 32, 67, 150])  # 1, 2, 4 and 8 blocks share the views
def test_sftt_back_with_shared_views_matches_oracle(ct, views):
    spec = _spec("flat", 17, 9, 37, 33, 47, views, 3.4, 2.9)
    g = ct.Geometry.from_spec(spec)
    yd = torch.as_tensor(W.random_sino(spec, seed=2, batch=2) - 0.3, dtype=torch.float32).cuda()
    x = ct.back(g, yd, "sftt")
    for b in range(2):
        _check(x[b].cpu().numpy(), oracle.back(spec, "sftt", yd[b].double().cpu().numpy()), "back")
    assert torch.equal(x[1], ct.back(g, yd[1].contiguous(), "sftt"))


@pytest.mark.parametrize("proj", ["sf", "dd", "voxel"])
def test_a_bad_cell_stays_where_its_rays_go(ct, proj):
    """An infinite detector cell reaches only voxels whose footprint is near it."""
    spec = _spec("flat", *SIZES["ragged"])
    g = ct.Geometry.from_spec(spec)
    y = torch.rand(g.sino_shape, device="cuda")
    clean = ct.back(g, y, proj)
    y[3, 40, 16] = float("inf")
    bad = ct.back(g, y, proj)
    ok = torch.isfinite(bad)
    assert torch.equal(bad[ok], clean[ok])
    mask = np.zeros(spec.sino_shape)
    mask[3, 38:43, 12:21] = 1.0
    assert not (~ok.cpu().numpy() & (oracle.back(spec, "sf", mask) == 0)).any()


def _weighs(spec, proj, cells):
    """Voxels with a weight on one of the cells (view, row, cell), positions on the detector uncertain by 1e-3 cell
    (FP32 positions are good to 1e-4)."""
    mask = np.zeros(spec.sino_shape)
    for c in cells:
        mask[c] = 1.0
    out = np.zeros(spec.vol_shape, dtype=bool)
    for su in (-1e-3, 0.0, 1e-3):
        for sv in (-1e-3, 0.0, 1e-3):
            moved = dataclasses.replace(spec, u_ofst=spec.u_ofst + su * spec.du, v_ofst=spec.v_ofst + sv * spec.dv)
            out |= oracle.back(moved, proj, mask) != 0
    return out


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("mode", ["proj", "recon"])
@pytest.mark.parametrize("size", ["tall", "taller", "tallest"])
@pytest.mark.parametrize("proj", ["sf", "dd", "voxel"])
def test_a_bad_cell_reaches_the_voxels_it_weighs(ct, det, mode, size, proj):
    """Voxels higher than a row read several rows; one that meets fewer of them is not reached by the others."""
    spec = _spec(det, *SIZES[size])
    g = ct.Geometry.from_spec(spec)
    y = torch.rand(g.sino_shape, device="cuda")
    clean = ct.back(g, y, proj, mode=mode)
    nu, nv = spec.nu, spec.nv
    cells = [(2, nv // 2, nu // 2), (3, nv // 2 + 5, 1), (4, nv // 2 - 5, nu - 2), (5, 1, nu // 2 + 3), (6, nv - 2, nu // 2)]
    for c in cells:
        y[c] = float("inf")
    bad = ct.back(g, y, proj, mode=mode)
    ok = torch.isfinite(bad)
    assert not ok.all() and torch.equal(bad[ok], clean[ok])
    assert not (~ok.cpu().numpy() & ~_weighs(spec, proj, cells)).any()


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("mode", ["proj", "recon"])
@pytest.mark.parametrize("proj", ["sf", "dd", "voxel"])
def test_a_bad_cell_near_the_detectors_end(ct, det, mode, proj):
    """Windows moved onto a truncating detector do not read further than others: footprints of up to 8 cells by less
    than a row take four cells (voxel-driven: its own two) and one row beyond their own."""
    spec = _spec(det, 24, 24, 40, 40, 40, 9, 1.3, 3.1)
    g = ct.Geometry.from_spec(spec)
    y = torch.rand(g.sino_shape, device="cuda")
    clean = ct.back(g, y, proj, mode=mode)
    cells, near = [(2, 20, 1), (3, 18, 5), (4, 22, 34), (5, 21, 38)], []
    for v, b, a in cells:
        y[v, b, a] = float("inf")
        w = 0 if proj == "voxel" else 3
        near += [(v, r, c) for r in (b - 1, b, b + 1) for c in range(max(a - w, 0), min(a + w, 39) + 1)]
    bad = ct.back(g, y, proj, mode=mode)
    ok = torch.isfinite(bad)
    assert not ok.all() and torch.equal(bad[ok], clean[ok])
    assert not (~ok.cpu().numpy() & ~_weighs(spec, proj, near)).any()


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("size", ["narrow-short", "tall"])
def test_an_infinite_voxel_stays_infinite(ct, det, size):
    """Voxel-driven forward: every cell that an infinite voxel weighs on is infinite, not NaN."""
    spec = _spec(det, *SIZES[size])
    g = ct.Geometry.from_spec(spec)
    x = torch.rand(g.vol_shape, device="cuda")
    clean = ct.forward(g, x, "voxel")
    at = (spec.nz // 2, spec.ny // 2, spec.nx // 2)
    x[at] = float("inf")
    one = np.zeros(spec.vol_shape)
    one[at] = 1.0
    w = oracle.forward(spec, "voxel", one)
    y = ct.forward(g, x, "voxel").cpu().numpy()
    assert np.isposinf(y[w > 1e-3 * w.max()]).all()
    assert np.array_equal(y[w == 0], clean.cpu().numpy()[w == 0])


# nx, ny, nz, nu, nv, views, du, dv, half voxel heights above and below half a row
WIDTHS = {
    "short": (33, 17, 9, 150, 7, 130, 1.0, 3.2),     # one tile of 8 rows
    "one-tile": (33, 17, 24, 150, 30, 130, 1.0, 3.2),  # one tile of 32 rows (64 when few)
    "large": (41, 23, 170, 150, 150, 104, 1.0, 3.2),   # tiles of 64 cells, 64 + 64 + 22 rows
    "tall": (41, 23, 60, 150, 150, 60, 1.0, 1.3),      # voxels of 1.9 to 2.2 rows
}


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("size", WIDTHS)
@pytest.mark.parametrize("proj,dtype", [("sf", torch.float32), ("dd", torch.float32), ("voxel", torch.float32),
                                        ("sf", torch.float16)], ids=["sf", "dd", "voxel", "sf-f16"])
def test_circ_forward_at_every_tile_width(ct, det, size, proj, dtype):
    """The width of a tile follows the number of views and changes nothing: all views, some and one agree bit for bit,
    and with the oracle."""
    spec = _spec(det, *WIDTHS[size])
    half = [0.5 * spec.dz * 640.0 / spec.dv / r for r in (320.0 + 45.0, 320.0 - 45.0)]  # in rows, farthest and nearest
    assert (half[1] < 0.5) == (size != "tall") and (size != "tall" or half[0] > 0.5)
    tiles = -(-spec.nu // 64) * -(-spec.nv // 64) * spec.nview
    assert size != "large" or tiles >= 2 * 3 * 152  # tiles of 64 cells
    g = ct.Geometry.from_spec(spec)
    x = torch.as_tensor(W.random_volume(spec, seed=2)[0] - 0.3, dtype=torch.float32).cuda().to(dtype)
    y = ct.forward(g, x, proj, out_dtype=torch.float32)
    _check(y.cpu().numpy(), oracle.forward(spec, proj, x.double().cpu().numpy()), "forward")
    for views in (list(range(0, spec.nview, 3)), [1], [spec.nview - 1]):
        assert torch.equal(ct.forward(g.subset(views), x, proj, out_dtype=torch.float32), y[views])


@pytest.mark.parametrize("proj", ["sf", "dd", "voxel"])
@pytest.mark.parametrize("du,dv", [(2.6, 3.2), (1.5, 1.5)])
def test_a_view_does_not_depend_on_the_others(ct, proj, du, dv):
    """Views at two magnifications: voxels below and above a row, footprints of different widths."""
    nview = 20
    sad = np.where(np.arange(nview) % 2 == 0, 320.0, 200.0)
    spec = dataclasses.replace(_spec("flat", 25, 19, 41, 70, 75, nview, du, dv), sad=sad)
    g = ct.Geometry.from_spec(spec)
    x = torch.as_tensor(W.random_volume(spec, seed=4)[0] - 0.3, dtype=torch.float32).cuda()
    y = ct.forward(g, x, proj)
    _check(y.cpu().numpy(), oracle.forward(spec, proj, x.double().cpu().numpy()), "forward")
    for views in (list(range(0, nview, 2)), list(range(1, nview, 2)), [4]):
        assert torch.equal(ct.forward(g.subset(views), x, proj), y[views])


@pytest.mark.parametrize("det", ["flat", "curved"])
def test_ray_forward_by_one_thread_or_four(ct, det):
    """A ray's runs of slabs, each by a thread of its own in small calls and all by one in large ones, add up alike."""
    spec = _spec(det, 41, 23, 60, 150, 150, 24, 1.0, 1.1)
    assert spec.nu * spec.nv * spec.nview >= 3 * 152 * 1024 > spec.nu * spec.nv * 8
    g = ct.Geometry.from_spec(spec)
    x = torch.as_tensor(W.random_volume(spec, seed=2)[0] - 0.3, dtype=torch.float32).cuda()
    y = ct.forward(g, x, "ray")
    _check(y.cpu().numpy(), oracle.forward(spec, "ray", x.double().cpu().numpy()), "forward")
    for views in (list(range(0, 24, 3)), [5], [23]):
        assert torch.equal(ct.forward(g.subset(views), x, "ray"), y[views])
