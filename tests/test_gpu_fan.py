"""The fan-beam kernels at the edges of their tiles (8 x 4 pixel patches, 32
cells, 8 view groups of 64 staged views, runs of slabs), against the FP64
oracle at the FP32 path's bound, in every projector and direction."""
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


# nx, ny, nu, views, cell size (mm): one pixel; single rows and columns; one past and one short of a tile; more
# views than one staging; wide footprints (5 to 8 cells, and beyond 8); a detector narrower than a footprint
SIZES = [(1, 1, 5, 1, 3.0), (33, 1, 31, 7, 2.0), (1, 29, 40, 9, 2.0), (8, 4, 32, 8, 1.5), (9, 5, 33, 65, 1.7),
         (40, 67, 129, 131, 1.9), (31, 31, 150, 12, 0.85), (12, 12, 160, 10, 0.4), (17, 16, 2, 6, 4.0)]


def _spec(det, nx, ny, nu, views, du):
    return W.GeometrySpec("fan2d", det, nx, ny, 1, 1.6, 1.6, 1.0, nu, 1, du, 1.0, views,
                          theta=0.2 + 2 * np.pi * np.arange(views) / views, sad=300.0, sdd=610.0, x_src=1.5,
                          u_ofst=0.7, x_ofst=-1.0, y_ofst=2.0)


def _same(got, ref, what):
    if np.linalg.norm(ref) == 0:
        assert float(np.abs(got).max()) == 0, what
    else:
        assert rel_l2(got, ref) <= TOL_F32, what


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("size", SIZES, ids=["x".join(map(str, s)) for s in SIZES])
@pytest.mark.parametrize("proj", ["sf", "dd", "voxel", "ray", "sftt"])
def test_fan_pair_matches_oracle(ct, det, size, proj):
    spec = _spec(det, *size)
    g = ct.Geometry.from_spec(spec)
    x, y = W.random_volume(spec, seed=1, batch=2), W.random_sino(spec, seed=2, batch=2)
    xd = torch.as_tensor(x[:, 0], dtype=torch.float32).cuda()
    yd = torch.as_tensor(y[:, :, 0], dtype=torch.float32).cuda()
    if proj == "sftt" and (det == "curved" or size[4] < 0.5):
        with pytest.raises(ct.CTError):
            ct.forward(g, xd, proj)
        return
    Ax, Aty = ct.forward(g, xd, proj), ct.back(g, yd, proj)
    for b in range(2):
        _same(Ax[b].cpu().numpy(), oracle.forward(spec, proj, x[b]).reshape(g.sino_shape), "forward")
        _same(Aty[b].cpu().numpy(), oracle.back(spec, proj, y[b]).reshape(g.vol_shape), "back")
    assert torch.equal(Ax[1], ct.forward(g, xd[1], proj)) and torch.equal(Aty[1], ct.back(g, yd[1], proj))


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("proj", ["voxel", "dd", "sf"])
def test_fan_recon_back_matches_oracle(ct, det, proj):
    spec = _spec(det, 40, 67, 129, 131, 1.9)
    g = ct.Geometry.from_spec(spec)
    q = W.random_sino(spec, seed=3)[0]
    got = ct.back(g, torch.as_tensor(q[:, 0], dtype=torch.float32).cuda(), proj, mode="recon")
    _same(got.cpu().numpy(), oracle.back_recon(spec, q, proj).reshape(g.vol_shape), proj)


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("mode", ["proj", "recon"])
@pytest.mark.parametrize("size", [(40, 33), (261, 259)], ids=["one-pixel", "two-pixels"])
def test_a_bad_edge_cell_stays_on_the_detector(ct, det, mode, size):
    """Voxel-driven back onto a detector that truncates the image: infinite cells at its ends reach only the pixels
    that project beside them, not those whose rays pass beyond its end."""
    spec = _spec(det, *size, 40, 12, size[0] * 1.6 / 40)
    g = ct.Geometry.from_spec(spec)
    y = torch.rand(g.sino_shape, device="cuda")
    clean = ct.back(g, y, "voxel", mode=mode)
    mask = np.zeros(spec.sino_shape)
    for v, a in ((2, 0), (5, 39)):
        y[v, a] = float("inf")
        mask[v, 0, max(a - 1, 0):a + 2] = 1.0  # one cell of slack
    bad = ct.back(g, y, "voxel", mode=mode)
    ok = torch.isfinite(bad)
    touched = oracle.back(spec, "voxel", mask).reshape(g.vol_shape) != 0
    assert not ok.all() and torch.equal(bad[ok], clean[ok])
    assert not (~ok.cpu().numpy() & ~touched).any()


@pytest.mark.parametrize("det", ["flat", "curved"])
@pytest.mark.parametrize("proj,mode", [("voxel", "proj"), ("voxel", "recon"), ("sf", "proj"), ("dd", "recon"), ("ray", "proj")])
def test_two_pixels_to_a_thread(ct, det, proj, mode):
    """Images of 65536 pixels and more, alone: patches of 8 x 8 with remainders of 3 columns and of 5 and 1 rows. The
    same image in a pair takes one pixel to a thread: equal bit for bit; footprints besides against the oracle (the
    other two read positions along the whole detector, whose rounding exceeds this bound at 300 cells)."""
    for nx, ny in ((259, 261), (259, 257)):
        assert nx * ny >= 65536
        spec = _spec(det, nx, ny, 300, 11, 259 * 1.6 * 2 * 0.9 / 300)
        g = ct.Geometry.from_spec(spec)
        q = W.random_sino(spec, seed=3)[0]
        y = torch.as_tensor(q[:, 0], dtype=torch.float32).cuda()
        got = ct.back(g, y, proj, mode=mode)
        assert torch.equal(got, ct.back(g, torch.stack([y, 1 - y]), proj, mode=mode)[0])
        if proj in ("sf", "dd"):
            ref = oracle.back(spec, proj, q) if mode == "proj" else oracle.back_recon(spec, q, proj)
            _same(got.cpu().numpy(), ref.reshape(g.vol_shape), proj)


@pytest.mark.parametrize("batch", [3, 5])
@pytest.mark.parametrize("tin,tout", [("f32", "f32"), ("f16", "f16"), ("f32", "bf16"), ("bf16", "f32")])
@pytest.mark.parametrize("proj", ["sf", "dd", "voxel", "ray"])
def test_the_item_after_the_pairs(ct, proj, tin, tout, batch):
    """Odd batches: pairs and one item alone, at its own offset for every storage type, each as by itself."""
    T = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
    g = ct.Geometry.from_spec(_spec("flat", 31, 45, 77, 9, 1.5))
    x = torch.rand((batch,) + g.vol_shape, device="cuda").to(T[tin])
    y = torch.rand((batch,) + g.sino_shape, device="cuda").to(T[tin])
    Ax, Aty = ct.forward(g, x, proj, out_dtype=T[tout]), ct.back(g, y, proj, out_dtype=T[tout])
    for b in range(batch):
        assert torch.equal(Ax[b], ct.forward(g, x[b].contiguous(), proj, out_dtype=T[tout]))
        assert torch.equal(Aty[b], ct.back(g, y[b].contiguous(), proj, out_dtype=T[tout]))
