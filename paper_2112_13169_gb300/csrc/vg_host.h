// vg_host.h -- host-side set-up arithmetic shared by every entry point of
// the library (vg_api.cu, vg_noalloc.cu, vg_server.cu), so that all of them
// give a frame exactly the same kernel arguments.
//
// Everything here runs in double on the host and is rounded once to float
// or integer (Sec. IV-A..IV-C):
//   origin_k   = floor(p_k / vox_size) - floor(N_k / 2)          (Sec. IV-A)
//   R^v_c      = R^w_c,  t^v_c = t^w_c - origin * vox_size       (Sec. IV-B)
//   vox_depth  = lround(depth / vox_size)                         (Sec. IV-C)
//   hw         = lround(tan(fov_x / 2) * vox_depth), hh likewise
//   fx         = (W / 2) / tan(fov_x / 2), cx = (W - 1) / 2, y likewise
// with fov/2 in radians taken as fov_deg * pi / 360.
#pragma once

#include "vg.h"
#include "vg_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace vg {
namespace host {

constexpr double kPi = 3.14159265358979323846;

inline int status_of(cudaError_t e) {
    if (e == cudaSuccess) return VG_OK;
    if (e == cudaErrorMemoryAllocation) return VG_ENOMEM;
    return VG_ECUDA;
}

inline double half_fov(float deg) { return (double)deg * kPi / 360.0; }

// Table I parameters that every kind of grid accepts (flags aside): sizes
// >= 1 with fewer than 2^31 voxels and fewer than 2^27 plane words (K3
// indexes plane bits with 32 bits; only Nx far below 32 nears that), a
// finite positive voxel size and range, fields of view in (0, 180) degrees,
// 0 <= vox_inf <= 15, and fewer than 10^6 voxels of range.
inline bool shape_ok(const vg_params *p) {
    if (!p) return false;
    int64_t nv = 1;
    for (int k = 0; k < 3; ++k) {
        if (p->grid_size[k] < 1) return false;
        nv *= p->grid_size[k];
        if (nv >= (int64_t(1) << 31)) return false;
    }
    if (!(std::isfinite(p->vox_size) && p->vox_size > 0.0f)) return false;
    if (!(p->fov_x_deg > 0.0f && p->fov_x_deg < 180.0f)) return false;
    if (!(p->fov_y_deg > 0.0f && p->fov_y_deg < 180.0f)) return false;
    if (!(std::isfinite(p->depth) && p->depth > 0.0f)) return false;
    if (p->vox_inf < 0 || p->vox_inf > kMaxInflate) return false;
    {
        int64_t w = (p->grid_size[0] + 31) / 32, wx = 4;
        while (wx < w) wx *= 2;
        if (wx * (int64_t)p->grid_size[1] * p->grid_size[2] >= (int64_t(1) << 27)) return false;
    }
    const double vd = (double)p->depth / (double)p->vox_size;
    return vd < 1.0e6;
}

inline PlaneGeom geom_of(const vg_params *p) {
    PlaneGeom g;
    g.nx = p->grid_size[0];
    g.ny = p->grid_size[1];
    g.nz = p->grid_size[2];
    const int32_t w = (g.nx + 31) / 32;
    g.wx = 4;
    while (g.wx < w) g.wx *= 2;
    g.words = (int64_t)g.wx * g.ny * g.nz;
    g.nvox = (int64_t)g.nx * g.ny * g.nz;
    return g;
}

// The ray bundle of Sec. IV-C: vox_depth and the half widths.
inline void bundle_of(const vg_params *p, int32_t &vd, int32_t &hw, int32_t &hh) {
    const long d = lround((double)p->depth / (double)p->vox_size);
    vd = (int32_t)d;
    hw = (int32_t)lround(tan(half_fov(p->fov_x_deg)) * (double)d);
    hh = (int32_t)lround(tan(half_fov(p->fov_y_deg)) * (double)d);
}

inline void origin_of(const vg_params *p, const double pos[3], int32_t o[3]) {
    for (int k = 0; k < 3; ++k)
        o[k] = (int32_t)floor(pos[k] / (double)p->vox_size) - p->grid_size[k] / 2;
}

// Composes T^v_c (Sec. IV-B) from T^w_c and the grid origin.  Rejects poses
// that are not finite, whose rotation block has an entry outside
// [-1.5, 1.5] (no rotation does), or whose camera lies 2^22 voxels or more
// from the grid corner: K3's walk length is bounded by the ray's length in
// voxels, and these limits keep it bounded and keep FP32 voxel
// coordinates exact to well below one voxel.
inline bool pose_vc(const double T_wc[16], const int32_t origin[3], float vox_size, Pose32 &T) {
    if (!T_wc) return false;
    for (int i = 0; i < 16; ++i)
        if (!std::isfinite(T_wc[i])) return false;
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c) {
            if (!(std::fabs(T_wc[r * 4 + c]) <= 1.5)) return false;
            T.R[r * 3 + c] = (float)T_wc[r * 4 + c];
        }
        const double t = T_wc[r * 4 + 3] - (double)origin[r] * (double)vox_size;
        if (!(std::fabs(t / (double)vox_size) < 4194304.0)) return false;
        T.t[r] = (float)t;
    }
    return true;
}

// A depth frame's shape and pixel type: 1 <= W, H with fewer than 2^31
// pixels, VG_DEPTH_F32 or VG_DEPTH_U16, and a finite positive scale for u16.
inline bool depth_frame_ok(int32_t width, int32_t height, int32_t dtype, float depth_scale) {
    if (width < 1 || height < 1 || (int64_t)width * height >= (int64_t(1) << 31)) return false;
    if (dtype != VG_DEPTH_F32 && dtype != VG_DEPTH_U16) return false;
    if (dtype == VG_DEPTH_U16 && !(std::isfinite(depth_scale) && depth_scale > 0.0f)) return false;
    return true;
}

// 1 / y rounded to nearest, for K1's divisions by a constant (units::div_by),
// or 0 where their correction step might not round correctly: y far from 1,
// or with a significand of all ones.
inline float reciprocal(float y) {
    uint32_t bits;
    std::memcpy(&bits, &y, sizeof(bits));
    if (!(y >= 1e-18f && y <= 1e18f) || (bits & 0x7fffffu) == 0x7fffffu) return 0.0f;
    return 1.0f / y;
}

// The kernel arguments of one measurement of a grid with parameters p and
// plane geometry g (planes, loc and stats are left for the caller).
// bundle: {vox_depth, hw, hh} where the caller has them.
inline FrameArgs frame_args(const vg_params *p, const PlaneGeom &g, const Pose32 &T, const int32_t *bundle = nullptr) {
    FrameArgs a;
    std::memset(&a, 0, sizeof(a));
    a.g = g;
    a.T = T;
    a.vs = p->vox_size;
    a.rvs = reciprocal(a.vs);
    a.depth_max = p->depth;
    if (bundle) {
        a.vd = bundle[0];
        a.hw = bundle[1];
        a.hh = bundle[2];
    } else {
        bundle_of(p, a.vd, a.hw, a.hh);
    }
    a.r = p->vox_inf;
    a.box = {0, g.wx, 0, g.ny, 0, g.nz};
    return a;
}

inline void depth_box(FrameArgs &a, const vg_params *p, double tx, double ty);

// Adds a depth frame's input and pinhole intrinsics to a.
inline void set_depth_frame(FrameArgs &a, const vg_params *p, const void *depth, int32_t width, int32_t height,
                            int32_t dtype, float depth_scale) {
    a.depth = depth;
    a.W = width;
    a.H = height;
    a.scale = (dtype == VG_DEPTH_U16) ? depth_scale : 1.0f;
    const double tx = tan(half_fov(p->fov_x_deg)), ty = tan(half_fov(p->fov_y_deg));
    a.fx = (float)(((double)width / 2.0) / tx);
    a.fy = (float)(((double)height / 2.0) / ty);
    a.rfx = reciprocal(a.fx);
    a.rfy = reciprocal(a.fy);
    a.cx = (float)(((double)width - 1.0) / 2.0);
    a.cy = (float)(((double)height - 1.0) / 2.0);
    // K1's tiles of 32 x 32 pixels leave most of a CTA idle where there are few
    // rows or columns: 307,200 pixels in one row K1 18.6 us as they lie in
    // memory, 26.9 in tiles; in one column 10.2 and 25
    a.linear = width < 8 || height < 8;
    depth_box(a, p, tx, ty);
}

// The image is read over the host link, in units of 32 bytes: a tile's rows
// that begin inside them read a fourth more, pixels as they lie do not (16-bit
// frames of 641x479: K1 14.4 us in tiles, 13.0 so; 640x480 12.1 and 12.4).
inline void over_link(FrameArgs &a) { a.linear = a.linear || a.W % 16 != 0; }

// Narrows a frame's box to a pyramid from the camera, of depth d voxels and
// half sides kx and ky there, with `spare` voxels more for rounding.  Poses
// whose rotation block is no rotation keep their linear map, so the corners
// bound it all the same.
inline void pyramid_box(FrameArgs &a, double d, double kx, double ky, double spare) {
    int32_t lo[3], hi[3];
    const int32_t n[3] = {a.g.nx, a.g.ny, a.g.nz};
    for (int k = 0; k < 3; ++k) {
        const double s = (double)a.T.t[k] / (double)a.vs;
        const double fwd = (double)a.T.R[k * 3 + 2] * d;
        const double side = std::fabs((double)a.T.R[k * 3]) * kx + std::fabs((double)a.T.R[k * 3 + 1]) * ky;
        const double m = spare + 1e-6 * (std::fabs(s) + std::fabs(fwd) + side);
        lo[k] = (int32_t)std::min(std::max(floor(s + std::min(0.0, fwd - side) - m), 0.0), (double)n[k]);
        hi[k] = (int32_t)std::min(std::max(ceil(s + std::max(0.0, fwd + side) + m), 0.0), (double)n[k]);
        if (hi[k] < lo[k]) hi[k] = lo[k];
    }
    if (lo[0] == hi[0] || lo[1] == hi[1] || lo[2] == hi[2]) {   // nothing of the grid: one word, for the launches
        a.box = {0, 1, 0, 1, 0, 1};
        return;
    }
    a.box = {lo[0] / 32, (hi[0] + 31) / 32 - lo[0] / 32, lo[1], hi[1] - lo[1], lo[2], hi[2] - lo[2]};
}

// A depth frame's box: what its pixels (inflated by vox_inf) and rays can
// reach (tx, ty: the tangents of half its fields of view).
inline void depth_box(FrameArgs &a, const vg_params *p, double tx, double ty) {
    const double d = std::max((double)a.vd, (double)p->depth / (double)p->vox_size);
    const double kx = std::max(tx, a.vd > 0 ? (double)a.hw / a.vd : 0.0) * d;
    const double ky = std::max(ty, a.vd > 0 ? (double)a.hh / a.vd : 0.0) * d;
    pyramid_box(a, d, kx, ky, a.r + 2.0);
}

// A cloud's box: what its rays can reach.  Its points lie anywhere.
inline void cloud_box(FrameArgs &a) {
    a.whole = 1;
    pyramid_box(a, a.vd, a.hw, a.hh, 2.0);
}

// Whether the gathered form of a frame (vg_gather.cuh) is the faster one:
// its voxels, the smaller of the bundle's pyramid and half its box, number
// kGatherVoxels or more.  Its kernels take about as long as the scattered
// ones of 10,700 rays of 71 voxels (252 k by this count; 640x480 frames of a
// 10 x 10 x 5 m grid: 36.1 against 36.0 us a frame with its read); below, the
// fixed cost of the lists and of one launch more is not made up (8,295 rays
// of 43 voxels: 28 against 22 us), above it is (21,201 of 100: 41.4 against
// 45.3; 33,221 of 125: 56 against 70; 132,525 of 250: 163 against 350).
constexpr double kGatherVoxels = 250e3;
inline double gather_voxels(const FrameArgs &a) {
    const double rays = (2.0 * a.hw + 1.0) * (2.0 * a.hh + 1.0);
    const double box = 32.0 * a.box.nw * a.box.ny * a.box.nz;
    return std::min(rays * a.vd / 3.0, box / 2.0);
}
inline bool gather_pays(const FrameArgs &a) { return gather_voxels(a) >= kGatherVoxels; }

// A batch's frames are gathered together or not at all (one gathered frame
// brings the launch a phase and a barrier more): from kBatchGatherVoxels in
// all, by the same count.  Measured, a step gathered against scattered: 4
// frames of 320x240 into 80 x 80 x 40 (185 k) 63 against 49 us, 8 (370 k) 70
// against 62, 12 (554 k) 68 against 70; into 100 x 100 x 20, 2 (200 k) 59
// against 48, 4 (400 k) 60 against 60, 8 (800 k) 65 against 75, 16 84 against
// 106; one 640x480 frame into 200 x 200 x 100 (707 k) 63 against 71.
constexpr double kBatchGatherVoxels = 450e3;

// Sets up the gathered form of a frame (vg_gather.cuh) in `bytes` bytes of
// device memory at base (256-byte aligned), or leaves it off: a.T, a.vs, the
// bundle and the geometry are set.  The form needs a rotation (within 1e-3:
// a voxel's inscribed sphere stays one), a bundle of at most 105 degrees (a
// wider one crosses voxels outside the near words at depths where windows are
// huge), a camera, grid and range within 4096 voxels, and room for its
// tables: 20 bytes a ray, 4 a tile of 64 and the near words.  Other frames
// take the scattered form.
//
// The margin.  With u = 2^-24, C1 = |S| + n and D the longest ray, a point's
// camera coordinates are off by at most 10 u C1 (the subtraction, the rounded
// matrix, five multiply-adds), a ray's direction by 9 u |D| (three products
// and two sums an axis), and the walk's crossings by 3 u |D| along the ray:
// together under 9e-7 C, C = C1 + |D|.  m = 0.002 + 1.7e-6 C is twice that (0.003
// at 10 m / 0.05 m, 0.03 at the limits).  A ray within 0.49 - m of a centre
// is 0.01 + m or more inside the voxel's faces there.
inline void gather_setup(FrameArgs &a, uint8_t *base, size_t bytes) {
    Gather &g = a.ga;
    g.on = 0;
    if (a.vd < 1 || a.vd > 4096 || a.hw > 1.3 * a.vd || a.hh > 1.3 * a.vd) return;
    const int32_t n[3] = {a.g.nx, a.g.ny, a.g.nz};
    double R[9], M[9];
    for (int k = 0; k < 9; ++k) R[k] = a.T.R[k];
    for (int i = 0; i < 3; ++i) {
        if (n[i] > 4096 || !(std::fabs(a.T.t[i] / a.vs) <= 4096.0f)) return;
        for (int j = 0; j < 3; ++j) {
            const double d = R[i] * R[j] + R[3 + i] * R[3 + j] + R[6 + i] * R[6 + j];
            if (!(std::fabs(d - (i == j ? 1.0 : 0.0)) <= 1e-3)) return;
        }
    }
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {   // adjugate
            const int i1 = (i + 1) % 3, i2 = (i + 2) % 3, j1 = (j + 1) % 3, j2 = (j + 2) % 3;
            M[j * 3 + i] = R[i1 * 3 + j1] * R[i2 * 3 + j2] - R[i1 * 3 + j2] * R[i2 * 3 + j1];
        }
    const double det = R[0] * M[0] + R[1] * M[3] + R[2] * M[6];
    for (int k = 0; k < 9; ++k) M[k] /= det;

    const int64_t rays = (2 * (int64_t)a.hw + 1) * (2 * (int64_t)a.hh + 1);
    const int64_t tiles = (int64_t)((2 * a.hw + 8) >> 3) * ((2 * a.hh + 8) >> 3);
    if (!base || rays * 20 + tiles * 4 + 2 * kNearWords * 4 > (int64_t)bytes || rays >= kMaxRays) return;
    g.rays = (int32_t)rays;
    g.inv = reinterpret_cast<float4 *>(base);
    g.hit = reinterpret_cast<uint32_t *>(g.inv + rays);
    g.tile = g.hit + rays;
    g.near_fr = g.tile + tiles;
    g.near_tr = g.near_fr + kNearWords;

    double smax = 0.0;
    for (int k = 0; k < 3; ++k) smax = std::max(smax, std::fabs((double)a.T.t[k] / a.vs) + n[k]);
    const double m = 0.002 + 1.7e-6 * (smax + std::sqrt((double)a.vd * a.vd + (double)a.hw * a.hw + (double)a.hh * a.hh));
    g.m = (float)m;
    g.sphere2 = (float)((0.49 - m) * (0.49 - m));
    const double ka = (double)a.hw / a.vd, kb = (double)a.hh / a.vd;
    g.ka = (float)ka;
    g.kb = (float)kb;
    for (int side = 0; side < 4; ++side) {
        const double *row = M + 3 * (side >> 1), k = (side >> 1 ? kb : ka) * (side & 1 ? -1.0 : 1.0);
        const double c[3] = {std::fabs(row[0] - k * M[6]), std::fabs(row[1] - k * M[7]), std::fabs(row[2] - k * M[8])};
        const double margin = m * (1.0 + std::fabs(k));
        g.ew[side] = (float)(16.0 * c[0] + 0.5 * c[1] + 0.5 * c[2] + margin);
        g.ep[side] = (float)(4.0 * c[0] + 2.0 * c[1] + 0.5 * c[2] + margin);
        g.ev[side] = (float)(0.5 * (c[0] + c[1] + c[2]) + margin);
    }
    for (int k = 0; k < 9; ++k) g.M[k] = (float)M[k];
    g.zp = (float)(4.0 * std::fabs(M[6]) + 2.0 * std::fabs(M[7]) + 0.5 * std::fabs(M[8]));
    g.zw = (float)(16.0 * std::fabs(M[6]) + 0.5 * std::fabs(M[7]) + 0.5 * std::fabs(M[8]));
    g.zv = (float)(0.5 * (std::fabs(M[6]) + std::fabs(M[7]) + std::fabs(M[8])));
    // |a - fa| <= vd (reach + margin) / (c2 - zv - margin) + margin, as in window_of
    const double reach = std::max(std::max(g.ev[0], g.ev[1]), std::max(g.ev[2], g.ev[3]));
    g.zr = (float)(a.vd * reach / (kLateReach - 0.5 - 2.0 * m) + g.zv + 2.0 * m);
    g.on = 1;
}

}  // namespace host
}  // namespace vg
