"""The gathered form of K3 and K4 (large frames) against the oracle, where it
could go wrong, and the scattered form at sizes that now take the gathered
one.  Bit-exact, like every parity test."""
import numpy as np
import pytest

from gridcheck import assert_same
from oracle import OracleGrid, OracleParams
from synth import body_pose, make

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


def pays(n, vs, fx, fy, depth):
    """The library's rule (gather_pays) with the whole grid as the box."""
    vd = round(depth / vs)
    rays = (2 * round(np.tan(np.radians(fx / 2)) * vd) + 1) * (2 * round(np.tan(np.radians(fy / 2)) * vd) + 1)
    return min(rays * vd / 3, n[0] * n[1] * n[2] / 2) >= 250e3


class Grids:
    def __init__(self, vg, n, vs, fx, fy, depth, r, pos, flags=0):
        self.g = vg.Grid(n, vs, fx, fy, depth, r, pos, flags=flags)
        self.o = OracleGrid(OracleParams(tuple(n), vs, fx, fy, depth, r), pos)
        self.out = torch.empty(self.g.nvox, dtype=torch.uint8, device="cuda")

    def check(self, what):
        origin = self.g.read(self.out)
        torch.cuda.synchronize()
        assert list(origin) == list(self.o.o), what
        assert_same(self.out.cpu().numpy().reshape(self.g.shape), self.o.loc, what)

    def depth(self, d, T, what):
        self.g.integrate_depth(torch.from_numpy(d).cuda(), T)
        self.o.integrate_depth(T, d)
        self.check(what)


def noise_image(rng, w, h, near, far, empty):
    """Blocks of like depth (surfaces with edges), speckled and with holes."""
    d = rng.uniform(near, far, (h // 8 + 1, w // 8 + 1)).repeat(8, 0).repeat(8, 1)[:h, :w]
    d = d * (1 + 0.02 * rng.standard_normal(d.shape))
    d[rng.random(d.shape) < empty] = 0
    return np.ascontiguousarray(d, np.float32)


# grid, voxel, fov x, fov y, range, radius, camera offset from the grid's centre
CASES = [
    ((171, 133, 67), 0.05, 87.0, 58.0, 5.0, 2, (0.0, 0.0, 0.0)),       # ragged rows, row groups and patches
    ((97, 250, 101), 0.05, 100.0, 101.0, 4.0, 1, (0.3, -0.2, 0.1)),    # rows of four words, wide views
    ((300, 300, 6), 0.05, 60.0, 50.0, 7.0, 3, (0.0, 0.0, 0.1)),        # six slices: thinner than the near box
    ((256, 200, 80), 0.05, 87.0, 58.0, 5.0, 0, (0.013, 0.0, -0.027)),  # no inflation: the raw plane's skin
    ((256, 200, 80), 0.05, 87.0, 58.0, 5.0, 6, (6.2, 0.0, 0.0)),       # camera at the grid's face
    ((200, 200, 100), 0.05, 87.0, 58.0, 6.0, 2, (-5.9, 1.0, 0.0)),     # camera outside the grid
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_gathered_frames(vg, case):
    n, vs, fx, fy, depth, r, off = CASES[case]
    assert pays(n, vs, fx, fy, depth)
    rng = np.random.default_rng(700 + case)
    P = Grids(vg, n, vs, fx, fy, depth, r, (0.0, 0.0, 0.0))
    for k in range(4):
        pos = np.array(off) + rng.uniform(-0.02, 0.02, 3)
        yaw = [0.0, np.pi / 2, rng.uniform(-3, 3), rng.uniform(-3, 3)][k]   # along the axes, then across
        if abs(off[0]) > 5:
            yaw = (np.pi if off[0] > 0 else 0.0) + rng.uniform(-0.4, 0.4)   # into the grid
        T = body_pose(pos, yaw, [0.0, 0.0, 0.4, -0.3][k], [0.0, 0.0, 0.2, -1.0][k])
        # near clutter, ordinary, nothing in range, all at one's nose
        d = noise_image(rng, 200, 150, *[(0.3, 2.0, 0.1), (0.5, 1.2 * depth, 0.1), (2 * depth, 3 * depth, 0.0),
                                         (0.05, 0.4, 0.5)][k])
        P.depth(d, T, "case %d frame %d" % (case, k))
        P.g.shift(pos + (0.3 * k, -0.1, 0.06))   # the next frame's merge clears what this brings in
        P.o.shift(pos + (0.3 * k, -0.1, 0.06))
    P.g.close()


def test_gathered_cloud_and_odd_poses(vg):
    # a cloud's occupied voxels lie anywhere, also behind the camera; a pose
    # that is no rotation and a camera far away take the scattered form
    rng = np.random.default_rng(77)
    P = Grids(vg, (200, 200, 100), 0.05, 87.0, 58.0, 5.0, 1, (0.0, 0.0, 0.0))
    xyz = rng.uniform(-4, 4, (20011, 3)).astype(np.float32)
    T = body_pose([0.0, 0.0, 0.0], 0.7, 0.1, 0.0)
    for cloud in (xyz, xyz[:0], xyz[:1]):
        P.g.integrate_points(torch.from_numpy(cloud).cuda(), T)
        P.o.integrate_points(T, cloud)
        P.check("cloud of %d points" % len(cloud))
    d = noise_image(rng, 160, 120, 0.5, 5.0, 0.1)
    T = T.copy()
    T[:3, :3] *= 1.2
    P.depth(d, T, "scaled rotation")
    T = body_pose([-300.0, 0.0, 0.0])
    P.depth(d, T, "far camera")
    P.g.close()


@pytest.mark.parametrize("lanes", [8, 16, 32])
def test_scattered_form_at_gathered_sizes(vg, lanes):
    # counting visits needs the walk
    w = make("seq", frames=2)
    g = w.grid
    P = Grids(vg, g.n, g.vox_size, w.cam.fov_x, w.cam.fov_y, g.depth, g.vox_inf, w.frames[0].robot_pos,
              flags=vg.VG_FLAG_STATS)
    P.g.tune(lanes)
    for k, f in enumerate(w.frames):
        P.depth(f.depth, f.T_wc, "scattered frame %d" % k)
        P.g.shift(f.robot_pos)
        P.o.shift(f.robot_pos)
    assert P.g.stats()["ray_visits"] > 0
    P.g.close()


@pytest.mark.parametrize("n", [(1, 5, 3), (7, 9, 4), (15, 4, 5), (16, 4, 4), (17, 6, 3), (33, 5, 5), (64, 3, 7)])
def test_reads_through_the_ring(vg, n):
    # rows shorter than a chunk, of a chunk, and ragged; every wrap position,
    # read with and without voxels that a re-centre brought in
    g = vg.Grid(n, 1.0, 60.0, 50.0, 3.0, 0, (0.0, 0.0, 0.0))
    o = OracleGrid(OracleParams(n, 1.0, 60.0, 50.0, 3.0, 0), (0.0, 0.0, 0.0))
    rng = np.random.default_rng(n[0])
    src = rng.integers(0, 4, (n[2], n[1], n[0])).astype(np.uint8)
    out = torch.full((g.nvox + 32,), 9, dtype=torch.uint8, device="cuda")
    g.write(src, g.origin)
    o.loc[:] = src
    pos = np.zeros(3)
    for k in range(20):
        pos = pos + rng.integers(-2, 3, 3)
        g.shift(pos)
        o.shift(pos)
        origin = g.read(out)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        assert list(origin) == list(o.o)
        assert_same(got[:g.nvox], o.loc, "read %d of %s" % (k, n))
        assert (got[g.nvox:] == 9).all()   # nothing past the grid
        if k % 5 == 4:
            o.loc[:] = src
            g.write(src, g.origin)
    g.close()


# points all round the robot: outside the rays' box, where the merge takes
# them, in words the box shares with the rays, and in what re-centres bring in
@pytest.mark.parametrize("n,r,off", [((200, 200, 100), 2, 0.0), ((211, 173, 61), 0, 0.0), ((400, 130, 70), 5, 0.0),
                                     ((200, 200, 100), 1, 4.9), ((200, 200, 100), 0, 60.0)])
def test_gathered_clouds_all_round(vg, n, r, off):
    rng = np.random.default_rng(sum(n) + r)
    P = Grids(vg, n, 0.05, 87.0, 58.0, 5.0, r, (0.0, 0.0, 0.0))
    half = np.array(n) * 0.05 / 2
    for k in range(4):
        # walls of a corridor, scattered points, and a few far outside the grid
        w = rng.uniform(-1, 1, (20_000, 3)) * half
        w[:8_000, 1] = np.sign(w[:8_000, 1])
        w[8_000:14_000, 2] = -0.42
        w[-500:] *= 3
        T = body_pose([off + 0.01, -0.02, 0.03], [0.0, 0.0, 2.2, -1.4][k] + (np.pi if 0 < off < 5 else 0.0), 0.1 * k, 0.05 * k)
        xyz = ((w - T[:3, 3]) @ T[:3, :3]).astype(np.float32)
        P.g.integrate_points(torch.from_numpy(xyz).cuda(), T)
        P.o.integrate_points(T, xyz)
        if k != 1:                                        # (frame 2 merges a pending re-centre)
            P.check("%s cloud %d" % (n, k))
        to = np.array([0.4, -0.3, 0.2]) * (k + 1)
        P.g.shift(to)
        P.o.shift(to)
    P.check("%s after the last re-centre" % (n,))
    P.g.close()


@pytest.mark.parametrize("n", [(1, 40, 3), (2, 3, 11), (3, 7, 7), (4, 9, 4), (5, 9, 4), (1, 1, 1), (2, 1, 37)])
def test_reads_of_narrow_rows_through_the_ring(vg, n):
    # rows read voxel by voxel (up to four), and one by runs; chunks that end
    # in a row, in a slice and past the grid
    test_reads_through_the_ring(vg, n)


def test_autotune_of_a_gathered_frame_leaves_the_walk_alone(vg):
    # lanes, K3's CTAs and K4's words do nothing on a gathered frame: their
    # candidates are not timed, and none is picked on noise
    w = make("seq", frames=1)
    g, f, reps = w.grid, w.frames[0], 2
    G = vg.Grid(g.n, g.vox_size, w.cam.fov_x, w.cam.fov_y, g.depth, g.vox_inf, f.robot_pos)
    best = G.autotune(torch.from_numpy(f.depth).cuda(), f.T_wc, reps=reps)
    assert (best["ctas_per_sm"], best["merge_words"]) == (0, 256) and best["lanes"] == 8
    # four tiles, K2's staging and its launch, each against the best so far,
    # reps and one frames of both
    frames = (4 + 1 + 1) * 2 * (reps + 1)
    launches = {k: v[2] for k, v in G.profile_read().items()}
    assert launches["voxelize"] == frames and launches["raytrace"] == 2 * frames
    G.close()


def test_autotune_of_a_gathered_batch_leaves_the_walk_alone(vg):
    w = make("seq", frames=1)
    g, f = w.grid, w.frames[0]
    grids = [vg.Grid(g.n, g.vox_size, w.cam.fov_x, w.cam.fov_y, g.depth, g.vox_inf, f.robot_pos) for _ in range(2)]
    d = torch.from_numpy(f.depth).cuda()
    batch = vg.Batch(2)
    best = batch.autotune([(G, d, f.T_wc, None, 1.0) for G in grids], reps=2)
    assert (best["lanes"], best["merge_words"], best["spread"]) == (0, 512, 1)
    batch.close()
    for G in grids:
        G.close()
