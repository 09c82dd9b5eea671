// vg_window.cuh -- which rays of the bundle may cross a box of the grid: the
// windows of K3's faces and K4's voxels (vg_gather.cuh), and the lists of
// (entry, ray) pairs made of them.  Arithmetic only, for the host as well, so
// that its bounds can be checked without a device.
#pragma once

#include "vg_internal.cuh"

#include <cmath>
#include <cstring>

#define VG_BOTH __host__ __device__ __forceinline__

namespace vg {
namespace gather {

constexpr int kThreads = 256;

VG_BOTH float fma_rn(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fma(a, b, c);
#endif
}

// a / b within 2 ulp
VG_BOTH float quotient(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}

VG_BOTH uint32_t bits_of(float v) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(v);
#else
    uint32_t u;
    memcpy(&u, &v, sizeof(u));
    return u;
#endif
}

// A point in camera axes, voxels from the camera.
struct Place {
    float c0, c1, c2;
};

VG_BOTH Place place_of(const Gather &g, float rx, float ry, float rz) {
    Place p;
    p.c0 = fma_rn(g.M[2], rz, fma_rn(g.M[1], ry, g.M[0] * rx));
    p.c1 = fma_rn(g.M[5], rz, fma_rn(g.M[4], ry, g.M[3] * rx));
    p.c2 = fma_rn(g.M[8], rz, fma_rn(g.M[7], ry, g.M[6] * rx));
    return p;
}

// Whether a box around p with reaches e (sides +a, -a, +b, -b) and z may
// touch the bundle.
VG_BOTH bool in_bundle(const FrameArgs &a, const Place &p, const float e[4], float z) {
    const Gather &g = a.ga;
    return fma_rn(-g.ka, p.c2, p.c0) <= e[0] && fma_rn(-g.ka, p.c2, -p.c0) <= e[1] &&
           fma_rn(-g.kb, p.c2, p.c1) <= e[2] && fma_rn(-g.kb, p.c2, -p.c1) <= e[3] &&
           p.c2 + z + g.m >= 0.0f && p.c2 - z - g.m <= (float)a.vd;
}

struct Window {
    int32_t alo, ahi, blo, bhi;   // rays a in [alo, ahi], b in [blo, bhi]; empty if lo > hi
    uint32_t kmin;                // no ray enters the box with a key of kmin or less
    VG_BOTH int32_t count() const { return max(ahi - alo + 1, 0) * max(bhi - blo + 1, 0); }
};

// The window of a box with half sizes (hx, 1/2, 1/2) around p, z its reach
// along the optical axis: |a - fa| <= vd (its reach across the plane through
// the camera and its centre) / (its nearest depth).
VG_BOTH Window window_of(const FrameArgs &a, const Place &p, float hx, float z) {
    const Gather &g = a.ga;
    const float fvd = (float)a.vd, fw = (float)a.hw, fh = (float)a.hh;
    Window w;
    const float zn = p.c2 - z - g.m;
    w.kmin = bits_of(fminf(fmaxf(quotient(zn, fvd), 0.0f), 1.0f)) << 2;
    if (zn < 0.2f) {
        w.alo = -a.hw; w.ahi = a.hw; w.blo = -a.hh; w.bhi = a.hh;
        return w;
    }
    const float iz = quotient(1.0f, p.c2), k0 = p.c0 * iz, k1 = p.c1 * iz, q = quotient(fvd, zn);
    const float h0 = hx * fabsf(fma_rn(-k0, g.M[6], g.M[0])) +
                     0.5f * (fabsf(fma_rn(-k0, g.M[7], g.M[1])) + fabsf(fma_rn(-k0, g.M[8], g.M[2])));
    const float h1 = hx * fabsf(fma_rn(-k1, g.M[6], g.M[3])) +
                     0.5f * (fabsf(fma_rn(-k1, g.M[7], g.M[4])) + fabsf(fma_rn(-k1, g.M[8], g.M[5])));
    const float wa = fma_rn(h0 + g.m, q, g.m), wb = fma_rn(h1 + g.m, q, g.m);
    const float fa = k0 * fvd, fb = k1 * fvd;
    w.alo = (int32_t)ceilf(fmaxf(fa - wa, -fw));
    w.ahi = (int32_t)floorf(fminf(fa + wa, fw));
    w.blo = (int32_t)ceilf(fmaxf(fb - wb, -fh));
    w.bhi = (int32_t)floorf(fminf(fb + wb, fh));
    return w;
}

// The window of the face of voxel i that a walk enters through along axis k:
// the projections of its corners, the margin beyond its edges.  A word that
// touches the bundle may hold voxels beside and behind the camera, where
// corners have no projection: empty if the voxel lies outside the bundle.
VG_BOTH Window face_window(const FrameArgs &a, const float S[3], const int32_t v0[3], const int32_t i[3], int k) {
    const Gather &g = a.ga;
    const float fvd = (float)a.vd, fw = (float)a.hw, fh = (float)a.hh;
    const float span = 1.0f + 2.0f * g.m;
    float r[3];
#pragma unroll
    for (int j = 0; j < 3; ++j)
        r[j] = (j == k ? (float)(i[j] + (i[j] < v0[j])) : (float)i[j] - g.m) - S[j];
    const Place p = place_of(g, r[0], r[1], r[2]);
    const int k1 = k == 0 ? 1 : 0, k2 = k == 2 ? 1 : 2;
    const float u0 = span * g.M[k1], u1 = span * g.M[3 + k1], u2 = span * g.M[6 + k1];
    const float w0 = span * g.M[k2], w1 = span * g.M[3 + k2], w2 = span * g.M[6 + k2];
    Window w;
    const float zn = p.c2 + fminf(u2, 0.0f) + fminf(w2, 0.0f) - g.m;
    w.kmin = bits_of(fminf(fmaxf(quotient(zn, fvd), 0.0f), 1.0f)) << 2;
    if (zn < 0.2f) {
        if (!in_bundle(a, place_of(g, (float)i[0] + 0.5f - S[0], (float)i[1] + 0.5f - S[1], (float)i[2] + 0.5f - S[2]), g.ev,
                       g.zv))
            return Window{0, -1, 0, -1, 0};
        w.alo = -a.hw; w.ahi = a.hw; w.blo = -a.hh; w.bhi = a.hh;
        return w;
    }
    float alo = INFINITY, ahi = -INFINITY, blo = INFINITY, bhi = -INFINITY;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float x = p.c0 + (c & 1 ? u0 : 0.0f) + (c & 2 ? w0 : 0.0f), y = p.c1 + (c & 1 ? u1 : 0.0f) + (c & 2 ? w1 : 0.0f);
        const float q = quotient(fvd, p.c2 + (c & 1 ? u2 : 0.0f) + (c & 2 ? w2 : 0.0f));
        alo = fminf(alo, x * q);
        ahi = fmaxf(ahi, x * q);
        blo = fminf(blo, y * q);
        bhi = fmaxf(bhi, y * q);
    }
    const float m = fma_rn(2.5f * g.m, quotient(fvd, zn), g.m);
    w.alo = (int32_t)ceilf(fmaxf(alo - m, -fw));
    w.ahi = (int32_t)floorf(fminf(ahi + m, fw));
    w.blo = (int32_t)ceilf(fmaxf(blo - m, -fh));
    w.bhi = (int32_t)floorf(fminf(bhi + m, fh));
    return w;
}

// Entries of a list that a round of for_pairs takes.  A window holds at most
// the bundle's rays, fewer than 2^27 (kMaxRays), so the round's windows
// laid end to end number no more than 2^31, and neither their 32-bit sum nor
// the strides past its end wrap.  Bundles of 2^23 rays and more, ranges of
// 1,400 voxels both ways, take short rounds.
static_assert((int64_t)kMaxRays * 16 <= int64_t(1) << 31, "short rounds fit");
VG_BOTH uint32_t round_entries(int32_t rays) { return rays < (1 << 23) ? (uint32_t)kThreads : 16u; }

// q / na, the row of ray q of a window na rays wide.  (q + 1/2) / na lies at
// least 1 / (2 na) from a whole number and the quotient within 2^-22 of
// itself from it, so its whole part is exact below 2^21.  Windows of bundles
// of 2^20 rays and more (fewer than 2^27, so off by one at most) are put right.
VG_BOTH uint32_t put_right(uint32_t row, uint32_t q, uint32_t na) {
    const int32_t left = (int32_t)(q - row * na);
    return left < 0 ? row - 1u : row + (uint32_t)(left >= (int32_t)na);
}
VG_BOTH uint32_t row_of(uint32_t q, uint32_t na, int32_t rays) {
    const uint32_t row = (uint32_t)quotient((float)q + 0.5f, (float)na);
    return rays >> 20 ? put_right(row, q, na) : row;
}

}  // namespace gather
}  // namespace vg

#undef VG_BOTH
