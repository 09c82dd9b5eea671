// Host entry points to the window arithmetic of vg_window.cuh, for
// test_windows_cpu.py: no device code runs here.
#include "vg_window.cuh"
#include "vg_host.h"

using namespace vg;

namespace {
FrameArgs g_a;
float g_S[3];
int32_t g_v0[3];
}  // namespace

extern "C" {

// The frame of a pose in a grid whose corner is at origin; whether the
// gathered form takes it (its tables are only addressed, never touched).
int w_setup(const int32_t n[3], float vs, float fx, float fy, float depth, const double T_wc[16], const int32_t origin[3],
            int32_t bundle[3], int64_t *rays) {
    vg_params p = {{n[0], n[1], n[2]}, vs, fx, fy, depth, 0, 0};
    Pose32 T;
    if (!host::shape_ok(&p) || !host::pose_vc(T_wc, origin, vs, T)) return -1;
    g_a = host::frame_args(&p, host::geom_of(&p), T);
    host::gather_setup(g_a, reinterpret_cast<uint8_t *>(256), (size_t)g_a.g.nvox + 16);
    for (int k = 0; k < 3; ++k) {
        g_S[k] = T.t[k] / vs;
        g_v0[k] = (int32_t)std::floor(g_S[k]);
    }
    bundle[0] = g_a.vd;
    bundle[1] = g_a.hw;
    bundle[2] = g_a.hh;
    *rays = g_a.ga.rays;
    return g_a.ga.on;
}

static void put(const gather::Window &w, int32_t *o) {
    o[0] = w.alo;
    o[1] = w.ahi;
    o[2] = w.blo;
    o[3] = w.bhi;
    o[4] = (int32_t)w.kmin;
}

// K3's windows of faces: voxels i[3 * m], axes k[m]; out[5 * m].
void w_faces(int64_t m, const int32_t *i, const int32_t *k, int32_t *out) {
    for (int64_t j = 0; j < m; ++j) put(gather::face_window(g_a, g_S, g_v0, i + 3 * j, k[j]), out + 5 * j);
}

// K4's windows of voxels.
void w_voxels(int64_t m, const int32_t *i, int32_t *out) {
    for (int64_t j = 0; j < m; ++j) {
        const int32_t *v = i + 3 * j;
        const gather::Place p = gather::place_of(g_a.ga, v[0] + 0.5f - g_S[0], v[1] + 0.5f - g_S[1], v[2] + 0.5f - g_S[2]);
        put(gather::window_of(g_a, p, 0.5f, g_a.ga.zv), out + 5 * j);
    }
}

// The voxels by which a depth frame of the same grid and pose counts for the
// gathered form (0: it is walked), and the sum from which a batch is gathered.
double w_gather_voxels(const int32_t n[3], float vs, float fx, float fy, float depth, int32_t r, const double T_wc[16],
                       const int32_t origin[3], int32_t w, int32_t h) {
    vg_params p = {{n[0], n[1], n[2]}, vs, fx, fy, depth, r, 0};
    Pose32 T;
    if (!host::shape_ok(&p) || !host::pose_vc(T_wc, origin, vs, T)) return -1.0;
    FrameArgs a = host::frame_args(&p, host::geom_of(&p), T);
    host::set_depth_frame(a, &p, reinterpret_cast<const void *>(256), w, h, VG_DEPTH_F32, 1.0f);
    host::gather_setup(a, reinterpret_cast<uint8_t *>(256), (size_t)a.g.nvox + 16);
    return a.ga.on ? host::gather_voxels(a) : 0.0;
}
double w_batch_rule() { return host::kBatchGatherVoxels; }

uint32_t w_round_entries(int32_t rays) { return gather::round_entries(rays); }
int32_t w_max_rays() { return kMaxRays; }
void w_rows(int64_t m, const uint32_t *q, const uint32_t *na, int32_t rays, uint32_t *out) {
    for (int64_t j = 0; j < m; ++j) out[j] = gather::row_of(q[j], na[j], rays);
}
void w_put_right(int64_t m, const uint32_t *q, const uint32_t *na, uint32_t *row) {
    for (int64_t j = 0; j < m; ++j) row[j] = gather::put_right(row[j], q[j], na[j]);
}

}  // extern "C"
