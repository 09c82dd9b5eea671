"""Which form of K3 and K4 a frame takes, walked or gathered, is asserted here
(a gathered frame launches two ray-trace kernels, a walked one one), for the
paths of either that other tests reach only by the sizes of their frames.
Bit-exact against the oracle."""
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


class Pair:
    """A library grid and the oracle's; every frame's form is asserted."""

    def __init__(self, vg, n, vs, fx, fy, depth, r, pos=(0.0, 0.0, 0.0), flags=0):
        self.g = vg.Grid(n, vs, fx, fy, depth, r, pos, flags=flags)
        self.o = OracleGrid(OracleParams(tuple(n), vs, fx, fy, depth, r), pos)
        self.out = torch.empty(self.g.nvox, dtype=torch.uint8, device="cuda")

    def frame(self, d, T, gathered, what):
        before = self.g.profile_read()["raytrace"][2]
        self.g.integrate_depth(torch.from_numpy(d).cuda(), T)
        self.o.integrate_depth(T, d)
        assert self.g.profile_read()["raytrace"][2] - before == (2 if gathered else 1), what
        self.check(what)

    def shift(self, pos):
        self.g.shift(pos)
        self.o.shift(pos)

    def check(self, what):
        origin = self.g.read(self.out)
        torch.cuda.synchronize()
        assert list(origin) == list(self.o.o), what
        assert_same(self.out.cpu().numpy().reshape(self.g.shape), self.o.loc, what)


def image(rng, w, h, near, far, empty=0.1):
    """Blocks of like depth, speckled and with holes."""
    d = rng.uniform(near, far, (h // 8 + 1, w // 8 + 1)).repeat(8, 0).repeat(8, 1)[:h, :w]
    d = d * (1 + 0.02 * rng.standard_normal(d.shape))
    d[rng.random(d.shape) < empty] = 0
    return np.ascontiguousarray(d, np.float32)


# ---------------------------------------------------------------------------
# gathered
# ---------------------------------------------------------------------------
def test_gathered_grid_thinner_than_the_box_around_the_camera(vg):
    rng = np.random.default_rng(3)
    P = Pair(vg, (900, 900, 6), 0.05, 60.0, 50.0, 20.0, 3)
    for k in range(4):
        T = body_pose(rng.uniform(-0.1, 0.1, 3), [0.0, 0.7, 2.4, -1.9][k], 0.0, [0.0, 0.0, 0.02, 1.5][k])
        P.frame(image(rng, 200, 150, *[(0.3, 2.0), (0.5, 24.0), (5.0, 19.0), (0.05, 0.4)][k]), T, True, "frame %d" % k)
        P.shift((0.3 * k, -0.1, 0.06))
    P.check("after the last re-centre")
    P.g.close()


# grid, fields of view, range, camera and its heading: coordinates of
# thousands of voxels, where the margin for rounding is 0.01 voxels and more
FAR = [((4000, 160, 120), 3.0, 2.4, 190.0, (-104.0, 0.1, 0.2), 0.0),
       ((160, 4000, 120), 3.0, 2.4, 190.0, (0.1, -104.0, -0.1), np.pi / 2),
       ((1200, 1200, 60), 3.0, 1.2, 200.0, (-120.0, -120.0, 0.0), np.pi / 4),
       ((2000, 2000, 20), 40.0, 1.0, 60.0, (-90.0, 5.0, 0.0), 0.05)]


@pytest.mark.parametrize("case", range(len(FAR)))
def test_gathered_far_from_the_origin(vg, case):
    n, fx, fy, depth, cam, yaw = FAR[case]
    rng = np.random.default_rng(50 + case)
    P = Pair(vg, n, 0.05, fx, fy, depth, 1)
    for k in range(3):
        pos = np.array(cam) + rng.uniform(-0.05, 0.05, 3)
        T = body_pose(pos, yaw + [0.0, 0.004, -0.003][k], [0.0, 0.002, -0.001][k], [0.0, 0.4, -2.0][k])
        P.frame(image(rng, 160, 120, 0.2 * depth, 1.1 * depth, 0.2), T, True, "case %d frame %d" % (case, k))
    P.g.close()


# ---------------------------------------------------------------------------
# walked, at sizes that are gathered unless visits are counted
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("tile", [1, 2, 3, 4])
@pytest.mark.parametrize("r", [1, 2, 3])
def test_walked_schedule_knobs_keep_results(vg, tile, r):
    # the four inflate tiles, K3 capped at few CTAs per SM, and K4's 256- and
    # 512-word units with re-centres
    w = make("robot", robot=90 + r, frames=3, spec=(640, 480, 0.05, (256, 120, 60), r))
    g = w.grid
    P = Pair(vg, g.n, g.vox_size, w.cam.fov_x, w.cam.fov_y, g.depth, g.vox_inf, w.frames[0].robot_pos, vg.VG_FLAG_STATS)
    P.g.set(vg.VG_TUNE_INFLATE_TILE, tile)
    P.g.set(vg.VG_TUNE_RT_CTAS_PER_SM, tile)
    P.g.set(vg.VG_TUNE_MERGE_WORDS, 512 if tile % 2 else 256)
    P.g.set(vg.VG_TUNE_INFLATE_TMA, 1 if r != 2 else 0)
    P.g.set(vg.VG_TUNE_EARLY_INFLATE, tile % 2)
    for k, f in enumerate(w.frames):
        P.frame(f.depth, f.T_wc, False, "tile %d r %d frame %d" % (tile, r, k))
        P.shift(f.robot_pos)
    P.check("after the last re-centre")
    P.g.close()


@pytest.mark.parametrize("lanes", [0, 1, 2, 4])
def test_walked_full_size_frames_by_lanes(vg, lanes):
    w = make("seq", frames=2)
    g = w.grid
    P = Pair(vg, g.n, g.vox_size, w.cam.fov_x, w.cam.fov_y, g.depth, g.vox_inf, w.frames[0].robot_pos, vg.VG_FLAG_STATS)
    P.g.tune(lanes)
    for k, f in enumerate(w.frames):
        P.frame(f.depth, f.T_wc, False, "%d lanes, frame %d" % (lanes, k))
        P.shift(f.robot_pos)
    P.g.close()


def test_walked_long_rays_take_more_lanes(vg):
    # 250 voxels of range: 32 lanes per ray of themselves
    rng = np.random.default_rng(41)
    P = Pair(vg, (200, 160, 90), 0.02, 87.0, 58.0, 5.0, 2, (0.01, -0.02, 0.03), vg.VG_FLAG_STATS)
    for k in range(2):
        d = rng.uniform(0.8, 5.5, size=(48, 64)).astype(np.float32)
        d[rng.random(d.shape) < 0.15] = 0
        P.frame(d, body_pose([0.01, -0.02, 0.03], rng.uniform(-np.pi, np.pi), rng.uniform(-0.3, 0.3)), False, "frame %d" % k)
    P.g.close()


@pytest.mark.parametrize("why", ["view", "pose", "side"])
def test_walked_where_the_gathered_form_has_limits(vg, why):
    # views of more than 105 degrees, poses that are no rotation, sides of
    # more than 4096 voxels
    rng = np.random.default_rng(43)
    n = (4100, 100, 40) if why == "side" else (200, 200, 100)
    P = Pair(vg, n, 0.05, 110.0 if why == "view" else 87.0, 58.0, 5.0, 2)
    for k in range(2):
        T = body_pose(rng.uniform(-0.1, 0.1, 3), rng.uniform(-3, 3), 0.1, 0.0)
        if why == "pose":
            T = T.copy()
            T[:3, :3] *= 1.01
        P.frame(image(rng, 200, 150, 0.3, 6.0), T, False, "%s frame %d" % (why, k))
    P.g.close()


# ---------------------------------------------------------------------------
# K2's tiles of 4 slices
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("n,r", [((200, 200, 100), 1), ((200, 200, 100), 3), ((100, 110, 100), 2)])
def test_inflate_tile_heights_of_clouds(vg, n, r):
    # one to four 8-slice tiles per SM take tiles 4 slices high.  A cloud's
    # tiles are the grid's: 325 of 8 words here, and 182 of 4
    rng = np.random.default_rng(sum(n) + r)
    P = Pair(vg, n, 0.05, 87.0, 58.0, 3.0, r)
    for k in range(2):
        xyz = rng.uniform(-1, 1, (4001, 3)) * np.array(n) * 0.03
        T = body_pose([0.01, 0.02, 0.03], rng.uniform(-3, 3), rng.uniform(-0.3, 0.3))
        before = P.g.profile_read()["inflate"][2]
        P.g.integrate_points(torch.from_numpy(xyz.astype(np.float32)).cuda(), T)
        P.o.integrate_points(T, xyz.astype(np.float32))
        assert P.g.profile_read()["inflate"][2] == before + 1
        P.check("cloud %d" % k)
    P.g.close()
