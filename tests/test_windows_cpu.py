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
    # the device's quotient is within two units in the last place: where it is
    # used, the row stays the same
    f = (q.astype(np.float32) + np.float32(0.5)) / n2.astype(np.float32)
    for to in (np.float32(0), np.float32(np.inf)):
        g = np.nextafter(np.nextafter(f, to), to)
        assert np.array_equal(g.astype(np.uint32), q // n2)
