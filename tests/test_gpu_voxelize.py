"""K1 where it could go wrong: quotients at voxel faces and at the ends of the
float range, and clouds on both sides of the shared-plane rule.  Bit-exact
against the oracle."""
import numpy as np
import pytest

from gridcheck import assert_same
from oracle import OracleGrid, OracleParams
from synth import body_pose

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def vg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13169_gb300 import build
    build.build()
    from paper_2112_13169_gb300 import vg as vgmod
    vgmod.load()
    return vgmod


def check_cloud(vg, n, vs, xyz, T, what):
    g = vg.Grid(n, vs, 60.0, 50.0, 6.0 * vs, 0, (0.0, 0.0, 0.0), flags=vg.VG_FLAG_STATS)
    o = OracleGrid(OracleParams(n, vs, 60.0, 50.0, 6.0 * vs, 0), (0.0, 0.0, 0.0))
    xyz = np.ascontiguousarray(xyz, np.float32)
    out = torch.empty(g.nvox, dtype=torch.uint8, device="cuda")
    for k in range(2):   # the second finds the planes as the first left them
        g.integrate_points(torch.from_numpy(xyz).cuda(), T)
        o.integrate_points(T, xyz)
        g.read(out)
        torch.cuda.synchronize()
        assert_same(out.cpu().numpy().reshape(g.shape), o.loc, "%s, cloud %d" % (what, k))
    points = g.stats()["points_in_grid"]
    g.close()
    return points


# 0.99999994: a significand of all ones, which divides by IEEE division
@pytest.mark.parametrize("vs", [0.05, 0.1, 1.0 / 3.0, 0.99999994, 1.0, 1.5, 3.0000002])
def test_points_at_voxel_faces(vg, vs):
    n = (41, 30, 21)
    rng = np.random.default_rng(int(vs * 1000))
    v = np.float32(vs)
    face = (rng.integers(-22, 23, (20000, 3)).astype(np.float32) * v).astype(np.float32)
    side = rng.integers(-1, 2, face.shape)
    xyz = np.where(side < 0, np.nextafter(face, np.float32(-np.inf)),
                   np.where(side > 0, np.nextafter(face, np.float32(np.inf)), face)).astype(np.float32)
    odd = np.array([0.0, -0.0, 1e-45, -1e-45, 1e-30, -1e-30, 1e-18, 3e38, -3e38, np.inf, np.nan, 1e19], np.float32)
    xyz[:3000] = rng.choice(odd, (3000, 3))
    xyz[3000:6000, 0] = rng.choice(odd, 3000)
    for T in (body_pose([0.0, 0.0, 0.0]), body_pose([0.3 * vs, -0.1, 0.0], 0.4, 0.2, -0.1)):
        assert check_cloud(vg, n, vs, xyz, T, "voxels of %r" % vs) > 0


@pytest.mark.parametrize("vs", [0.05, 0.99999994])
def test_pixels_of_any_depth(vg, vs):
    # depths from denormal to beyond the range, also on the image's centre lines
    n = (60, 50, 40)
    g = vg.Grid(n, vs, 80.0, 60.0, 20.0 * vs, 1)
    o = OracleGrid(OracleParams(n, vs, 80.0, 60.0, 20.0 * vs, 1), (0.0, 0.0, 0.0))
    rng = np.random.default_rng(5)
    out = torch.empty(g.nvox, dtype=torch.uint8, device="cuda")
    for w, h in ((65, 49), (64, 48)):
        d = (rng.uniform(0.0, 24.0, (h, w)) * vs).astype(np.float32)
        pick = rng.random((h, w))
        d[pick < 0.3] = rng.choice(np.array([1e-45, 1e-38, 1e-20, 1e-10, 1e-9, 1e9, 3e38, np.inf, np.nan, -1.0], np.float32),
                                   int((pick < 0.3).sum()))
        T = body_pose([0.0, 0.0, 0.0], rng.uniform(-1, 1), 0.1, 0.05)
        g.integrate_depth(torch.from_numpy(d).cuda(), T)
        o.integrate_depth(T, d)
        g.read(out)
        torch.cuda.synchronize()
        assert_same(out.cpu().numpy().reshape(g.shape), o.loc, "%dx%d depths" % (w, h))
    g.close()


# planes of 2,400 words, of 12,288 (the most that takes a shared plane) and of 12,416
@pytest.mark.parametrize("n", [(100, 30, 20), (128, 96, 32), (128, 97, 32)])
@pytest.mark.parametrize("more", [-1, 0, 1])
def test_clouds_around_the_shared_plane_rule(vg, n, more):
    words = 4 * n[1] * n[2]
    rng = np.random.default_rng(words + more)
    xyz = rng.uniform(-1.2, 1.2, (4 * words + more, 3)) * np.array(n)[[1, 2, 0]] * 0.05   # some outside
    xyz[: len(xyz) // 4] = xyz[0]          # many points of one voxel
    T = body_pose([0.02, 0.0, -0.01], 0.3, 0.0, 0.1)
    points = check_cloud(vg, n, 0.1, xyz, T, "%d points" % len(xyz))
    assert 0 < points < 2 * len(xyz)


# tiles of 32 x 32 pixels: one pixel, a tile less and more a pixel, rows that
# are and are not whole fours; a far noisy image fills a tile's table (1,024
# words where it has 256 slots), a flat one shares a few words
@pytest.mark.parametrize("w,h", [(1, 1), (31, 33), (32, 32), (36, 31), (68, 65), (97, 1), (1, 97)])
@pytest.mark.parametrize("dtype", [np.float32, np.uint16])
def test_images_around_tiles(vg, w, h, dtype):
    n, vs = (96, 120, 120), 0.1
    rng = np.random.default_rng(w * 100 + h)
    for off in (0, 1):   # the image's address whole and not whole fours of pixels
        g = vg.Grid(n, vs, 80.0, 70.0, 4.0, 0, (0.0, 0.0, 0.0), flags=vg.VG_FLAG_STATS)
        o = OracleGrid(OracleParams(n, vs, 80.0, 70.0, 4.0, 0), (0.0, 0.0, 0.0))
        out = torch.empty(g.nvox, dtype=torch.uint8, device="cuda")
        for flat in (False, True):
            d = rng.uniform(1.9 if flat else 0.4, 2.0 if flat else 5.9, (h, w))
            d[rng.random((h, w)) < 0.05] = 0
            d = np.rint(d * 1000).astype(dtype) if dtype == np.uint16 else d.astype(dtype)
            scale = 1e-3 if dtype == np.uint16 else 1.0
            buf = torch.zeros(w * h + off, dtype=torch.uint16 if dtype == np.uint16 else torch.float32, device="cuda")
            buf[off:] = torch.from_numpy(d.reshape(-1)).cuda()
            T = body_pose([0.0, 0.0, 0.0], rng.uniform(-3, 3), 0.2, 0.1)
            g.integrate_depth(buf[off:].view(h, w), T, scale)
            o.integrate_depth(T, d, scale)
            g.read(out)
            torch.cuda.synchronize()
            assert_same(out.cpu().numpy().reshape(g.shape), o.loc, "%dx%d, offset %d, flat %s" % (w, h, off, flat))
        g.close()


# rows that begin on every pixel of a whole four, whose fours reach into the
# rows before and after, and images that end inside one
@pytest.mark.parametrize("w,h", [(3, 3), (5, 2), (29, 35), (30, 33), (33, 34), (34, 5), (35, 7), (127, 40)])
@pytest.mark.parametrize("dtype", [np.float32, np.uint16])
def test_images_of_odd_widths(vg, w, h, dtype):
    n, vs = (96, 120, 120), 0.1
    rng = np.random.default_rng(w * 1000 + h)
    scale = 1e-3 if dtype == np.uint16 else 1.0
    for off in (0, 1):
        g = vg.Grid(n, vs, 80.0, 70.0, 4.0, 0, (0.0, 0.0, 0.0), flags=vg.VG_FLAG_STATS)
        o = OracleGrid(OracleParams(n, vs, 80.0, 70.0, 4.0, 0), (0.0, 0.0, 0.0))
        out = torch.empty(g.nvox, dtype=torch.uint8, device="cuda")
        for k in range(2):
            d = rng.uniform(0.4, 5.0, (h, w))
            d[rng.random((h, w)) < 0.05] = 0
            d = np.rint(d * 1000).astype(dtype) if dtype == np.uint16 else d.astype(dtype)
            # valid depths before and after the image, which must set nothing
            buf = torch.from_numpy(np.full(w * h + 9, 1000 if dtype == np.uint16 else 1.0, dtype)).cuda()
            at = 4 + off
            buf[at:at + w * h] = torch.from_numpy(d.reshape(-1)).cuda()
            T = body_pose([0.0, 0.0, 0.0], rng.uniform(-3, 3), 0.2, 0.1)
            g.integrate_depth(buf[at:at + w * h].view(h, w), T, scale)
            o.integrate_depth(T, d, scale)
            g.read(out)
            torch.cuda.synchronize()
            assert_same(out.cpu().numpy().reshape(g.shape), o.loc, "%dx%d, offset %d" % (w, h, off))
        assert 0 < g.stats()["points_in_grid"] <= 2 * w * h
        g.close()


# images of a few rows or columns, whose pixels K1 takes as they lie in memory,
# and one row or column more; page-locked images whose rows begin inside a
# unit of the host link; addresses and lengths that are no whole fours
@pytest.mark.parametrize("w,h", [(2000, 1), (1, 2000), (1025, 7), (7, 1025), (403, 8), (8, 403), (3, 3), (1024, 1), (65, 33)])
@pytest.mark.parametrize("dtype", [np.float32, np.uint16])
@pytest.mark.parametrize("host", [False, True])
def test_images_taken_as_they_lie(vg, w, h, dtype, host):
    n, vs = (96, 120, 120), 0.1
    rng = np.random.default_rng(w * 1000 + h)
    scale = 1e-3 if dtype == np.uint16 else 1.0
    for off in (0, 1):
        g = vg.Grid(n, vs, 80.0, 70.0, 4.0, 0, (0.0, 0.0, 0.0), flags=vg.VG_FLAG_STATS)
        o = OracleGrid(OracleParams(n, vs, 80.0, 70.0, 4.0, 0), (0.0, 0.0, 0.0))
        out = torch.empty(g.nvox, dtype=torch.uint8, device="cuda")
        for k in range(2):
            d = rng.uniform(0.4, 5.0, (h, w))
            d[rng.random((h, w)) < 0.05] = 0
            d = np.rint(d * 1000).astype(dtype) if dtype == np.uint16 else d.astype(dtype)
            # valid depths before and after the image, which must set nothing
            buf = torch.from_numpy(np.full(w * h + 9, 1000 if dtype == np.uint16 else 1.0, dtype))
            buf = buf.pin_memory() if host else buf.cuda()
            at = 4 + off
            buf[at:at + w * h] = torch.from_numpy(d.reshape(-1))
            T = body_pose([0.0, 0.0, 0.0], rng.uniform(-3, 3), 0.2, 0.1)
            g.integrate_depth(buf[at:at + w * h].view(h, w), T, scale)
            o.integrate_depth(T, d, scale)
            g.read(out)
            torch.cuda.synchronize()
            assert_same(out.cpu().numpy().reshape(g.shape), o.loc, "%dx%d, offset %d" % (w, h, off))
        assert 0 < g.stats()["points_in_grid"] <= 2 * w * h
        g.close()
