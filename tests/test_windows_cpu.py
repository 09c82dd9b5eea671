"""The windows of the gathered form's faces and voxels (vg_window.cuh) on the
CPU: the lists of (entry, ray) pairs made of them stay within 32 bits, and
every ray that crosses a face or voxel lies in its window."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from synth import body_pose

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def win(tmp_path_factory):
    from paper_2112_13169_gb300 import build
    out = str(tmp_path_factory.mktemp("windows") / "libwindows.so")
    cmd = [build.nvcc()] + build.ARCH + ["-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC,-ffp-contract=off",
           "-I", os.path.join(ROOT, "include"), "-I", build.CSRC, os.path.join(HERE, "windows.cu"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return C.CDLL(out)


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


# ---------------------------------------------------------------------------
# lists of pairs
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("rays", [1, 21201, (1 << 23) - 1, 1 << 23, 8388609, 67_000_000, 107_374_182, (1 << 27) - 1])
def test_a_round_of_windows_fits_32_bits(win, rays):
    # a round of the widest windows, and the strides of four loads per thread
    # past its end
    entries = win.w_round_entries(rays)
    assert 1 <= entries <= 256
    assert rays < win.w_max_rays()
    assert entries * rays + 4 * 256 < 1 << 32


def test_the_row_of_a_pair_is_exact(win):
    rng = np.random.default_rng(1)
    na = np.concatenate([np.arange(1, 300), rng.integers(1, 10651, 4000), [10651]]).astype(np.uint32)
    rows = rng.integers(1, 10651, (60, len(na)))
    rows[0], rows[1] = 1, 10650
    q = (rows * na.astype(np.int64)).ravel()     # the first ray of a row, and the last of the one before
    n2 = np.tile(na, 60)
    q, n2 = np.concatenate([q, q - 1, q + n2 // 2]).astype(np.uint32), np.tile(n2, 3)
    out = np.empty_like(q)
    for rays in (1 << 20, 113_000_000, (1 << 20) - 1):
        if rays < 1 << 20:                       # a window holds no more rays than the bundle
            q, n2, out = (v[q < rays].copy() for v in (q, n2, out))
        win.w_rows(C.c_int64(len(q)), ptr(q), ptr(n2), rays, ptr(out))
        assert np.array_equal(out, q // n2)
        # the device's quotient is within two units in the last place: the row
        # stays the same, or is put right
        f = (q.astype(np.float32) + np.float32(0.5)) / n2.astype(np.float32)
        for to in (np.float32(0), np.float32(np.inf)):
            row = np.nextafter(np.nextafter(f, to), to).astype(np.uint32)
            if rays >= 1 << 20:
                assert (row != q // n2).any()
                win.w_put_right(C.c_int64(len(q)), ptr(q), ptr(n2), ptr(row))
            assert np.array_equal(row, q // n2)


# ---------------------------------------------------------------------------
# windows
# ---------------------------------------------------------------------------
# grid, voxel, fov x, fov y, range, and the camera's voxel coordinates
FRAMES = [
    ((200, 200, 100), 0.05, 87.0, 58.0, 5.0, (100.2, 99.6, 50.5)),
    ((400, 400, 120), 0.05, 90.0, 60.0, 6.0, (200.9, 200.1, 60.0)),
    ((500, 500, 150), 0.02, 104.9, 104.9, 5.0, (230.5, 260.25, 75.7)),      # the widest
    ((100, 100, 20), 0.15, 85.0, 101.0, 6.5, (50.0, 3.5, 10.1)),
    ((4000, 300, 200), 0.05, 8.0, 6.0, 200.0, (-60.3, 150.5, 99.9)),        # far coordinates, long rays
    ((300, 4000, 200), 0.05, 8.0, 6.0, 200.0, (150.5, 3900.7, 99.9)),
]


def setup(win, frame, rng, yaw):
    n, vs, fx, fy, depth, cam = frame
    T = body_pose(np.array(cam) * vs, yaw, rng.uniform(-0.3, 0.3), rng.uniform(-3, 3))
    bundle, rays = np.zeros(3, np.int32), C.c_int64()
    on = win.w_setup(ptr(np.array(n, np.int32)), C.c_float(vs), C.c_float(fx), C.c_float(fy), C.c_float(depth),
                     ptr(np.ascontiguousarray(T, np.float64)), ptr(np.zeros(3, np.int32)), ptr(bundle), C.byref(rays))
    assert on == 1
    R, S = T[:3, :3].astype(np.float32).astype(np.float64), T[:3, 3] / np.float64(np.float32(vs))
    return R, S, bundle


def faces(win, i, k):
    i, k = np.ascontiguousarray(i, np.int32), np.ascontiguousarray(k, np.int32)
    out = np.zeros((len(i), 5), np.int32)
    win.w_faces(C.c_int64(len(i)), ptr(i), ptr(k), ptr(out))
    return out


def voxels(win, i):
    i = np.ascontiguousarray(i, np.int32)
    out = np.zeros((len(i), 5), np.int32)
    win.w_voxels(C.c_int64(len(i)), ptr(i), ptr(out))
    return out


@pytest.mark.parametrize("frame", range(len(FRAMES)))
def test_every_ray_through_a_face_lies_in_its_window(win, frame):
    rng = np.random.default_rng(40 + frame)
    n = np.array(FRAMES[frame][0])
    yaw = [0.4, -2.0, 1.1, 2.6, 0.02, -np.pi / 2 + 0.02][frame]
    R, S, (vd, hw, hh) = setup(win, FRAMES[frame], rng, yaw)
    m = 200_000
    a, b = rng.integers(-hw, hw + 1, m), rng.integers(-hh, hh + 1, m)
    a[: m // 10], b[m // 20 : m // 8] = hw, -hh          # the bundle's sides
    D = np.stack([a, b, np.full(m, vd)], 1) @ R.T
    i = np.floor(S + rng.uniform(0, 1, (m, 1)) * D).astype(np.int64)
    far = (i >= 0).all(1) & (i < n).all(1) & (np.abs(i - np.floor(S)).max(1) > 7)
    a, b, D, i = a[far], b[far], D[far], i[far]
    with np.errstate(divide="ignore", invalid="ignore"):
        t = np.where(i != np.floor(S), (np.where(D > 0, i, i + 1) - S) / D, -1.0)
    k = t.argmax(1)
    assert len(a) > 1000 and (t.max(1) > 0).all()
    for w in (faces(win, i, k), voxels(win, i)):
        assert ((w[:, 0] <= a) & (a <= w[:, 1]) & (w[:, 2] <= b) & (b <= w[:, 3])).all()
        kmin = (w[:, 4].astype(np.uint32) >> 2).view(np.float32)
        assert (kmin <= t.max(1) + 1e-6).all()


@pytest.mark.parametrize("frame", [0, 1, 2, 3, 5])   # (4: a camera before its grid)
def test_faces_beside_and_behind_the_camera_have_no_rays(win, frame):
    # a ray is at least two voxels along the optical axis when it leaves the
    # box of 15 voxels around the camera, even in the widest bundle
    rng = np.random.default_rng(60 + frame)
    n = np.array(FRAMES[frame][0])
    R, S, _ = setup(win, FRAMES[frame], rng, [0.0, 0.0, 0.7, -1.0, None, -np.pi / 2 + 0.01][frame])
    i = rng.integers(np.maximum(np.floor(S) - 60, 0), np.minimum(np.floor(S) + 60, n - 1) + 1, (100_000, 3))
    i = i[(np.abs(i - np.floor(S)).max(1) > 7) & (((i + 0.5 - S) @ R)[:, 2] < 1.0)]
    assert len(i) > 1000
    for k in range(3):
        w = faces(win, i, np.full(len(i), k))
        assert ((w[:, 0] > w[:, 1]) | (w[:, 2] > w[:, 3])).all()


def test_the_smallest_mixed_batch_is_gathered(win):
    # the frames of test_batch_of_both_forms_at_odd_sizes, one of each: the
    # batch has to take the gathered form, and one of its frames the walked
    from test_gpu_batch import BOTH
    win.w_gather_voxels.restype = win.w_batch_rule.restype = C.c_double
    voxels = []
    for k, (n, vs, fov, r, (w, h)) in enumerate(BOTH):
        pos = np.array((0.0, -0.2 * k, 0.1))
        origin = (np.floor(pos / np.float64(np.float32(vs))) - np.array(n) // 2).astype(np.int32)
        T = np.ascontiguousarray(body_pose(pos + 0.03, k), np.float64)
        voxels.append(win.w_gather_voxels(ptr(np.array(n, np.int32)), C.c_float(vs), C.c_float(fov), C.c_float(fov - 20),
                                          C.c_float(np.float32(0.45 * max(n) * vs)), r, ptr(T), ptr(origin), w, h))
    assert min(voxels) == 0.0 and sum(voxels) >= win.w_batch_rule()
