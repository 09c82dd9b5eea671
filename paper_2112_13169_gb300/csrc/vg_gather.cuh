// vg_gather.cuh -- K3 and K4 in their gathered form: occupied voxels tell
// the rays that cross them where they end, and every voxel then looks up the
// rays that may cross it.  Shared by the one-kernel-per-step launches
// (k_voxelize.cu, k_gather.cu) and the fused persistent launch (k_batch.cu).
//
// The walk of vg_rt.cuh visits voxel v on a ray exactly when, of v's faces,
// every entry crossing comes before every exit crossing of the serial order
// (by time, then axis) and the last entry crossing has t < 1: the walk is a
// merge of three sorted lists, and it stands in v after v's entry crossings
// and before its exit crossings.  The crossing times are the walk's own
// float expression, so this test (visits) gives the walk's answer bit for
// bit without walking.  A crossing's place in the order is one 32-bit key,
// event_key: the bits of its time, then its axis.  A ray's hit key is the
// key of the crossing by which it enters its first occupied voxel (0: the
// start voxel; kNoHit: it meets none).  A voxel entered with a key below the
// hit key is free by that ray, any other visited one traced.
//
// K3 (hits).  A ray's first occupied voxel is entered through a face whose
// other side is unoccupied and nearer to the camera's voxel, so only the
// occupied voxels with such a face (the skin the camera sees) are tested
// against the rays of their window, each hit key an atomicMin.
//
// Measured on a 640x480 frame into 200 x 200 x 100 voxels (21,201 rays of
// 100; ncu): K3 10 + 5 us and K4 16 us here, K3 40 and K4 7.4 us scattered; on
// 848x480 into 500 x 500 x 150 (132,525 rays of 250): 27 + 6 and 65 us against
// 269 and 22.  Both are bound by instruction issue and the latency of their
// phases, not by DRAM (1.1 MB a launch).
//
// K4 (gather).  About five rays cross each voxel of the bundle (3.4 M
// visits, 0.7 M voxels on a 200 x 200 x 100 grid at 5 m / 0.05 m), and the
// scattered form pays for every visit with a step of the walk and for about
// half of them with an L2 reduction.  Here a voxel is resolved once, mostly
// from the one ray nearest its centre, its word's 32 voxels by the 32 lanes
// of a warp, and the codes go straight into loc_grid: no free or traced
// plane, no reductions, and the merge is part of the same pass.
//
// Certain cases.  With p the voxel's centre and M the inverse rotation,
// M (p - S) = tau (a, b, vd) gives the voxel's place in the bundle.  If the
// nearest ray passes the centre within 0.49 - m voxels at the centre's
// depth, it crosses the voxel's inscribed sphere on a chord of 0.19 voxels or
// more, which is far beyond the rounding of the crossing times
// (gather_setup bounds it by m), so the walk visits the voxel; if its
// hit lies past the centre's depth the voxel is free; if its hit, and those
// of all rays around it that may reach the voxel (late_unit), lie before the
// voxel's nearest depth, it is traced.  All other voxels inside the bundle's sides are listed and
// resolved by testing every ray of their window with visits(); windows and
// culling leave the margin m for rounding.
//
// Voxels within kNear of the camera's would have windows of thousands of
// rays; there the rays mark the voxels they walk through (near_unit), 15
// words of 15 bits a slice.
#pragma once

#include "vg_units.cuh"
#include "vg_window.cuh"

#include <type_traits>

namespace vg {
namespace gather {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kNoHit = 0xffffffffu;
constexpr uint32_t kNone = 0xfffffffeu;   // no ray's key: no ray has a certain say
constexpr int kNear = kNearReach, kNearN = 2 * kNear + 1, kNearRows = kNearWords;
constexpr int kFlight = 4;     // loads in flight per thread
constexpr int kFaces = 4096;   // faces a round of K3 lists

__device__ __forceinline__ float cross_at(float b, float S, float inv) { return __fmul_rn(__fsub_rn(b, S), inv); }

// The place of the crossing of axis k at time t >= 0 in the walk's order;
// times of 1 and more, which are never walked, share the top keys.
__device__ __forceinline__ uint32_t event_key(float t, int k) {
    return (__float_as_uint(fminf(t, 1.0f)) << 2) + 1u + (uint32_t)k;
}

__device__ __forceinline__ void frame_start(const FrameArgs &a, float S[3], int32_t v0[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        S[k] = __fdiv_rn(a.T.t[k], a.vs);
        v0[k] = (int32_t)floorf(S[k]);
    }
}

// ---------------------------------------------------------------------------
// The ray table (with K1): 1/D of every ray in the walk's operation order,
// hits at kNoHit, and the words around the camera empty.  One ray per call;
// t counts from 0.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void table_thread(const FrameArgs &a, int64_t t) {
    if (t < 2 * kNearRows) a.ga.near_fr[t] = 0;
    if (t >= a.ga.rays) return;
    const uint32_t width = 2u * (uint32_t)a.hw + 1u, rb = (uint32_t)t / width;
    const float fa = (float)((int32_t)((uint32_t)t - rb * width) - a.hw), fb = (float)((int32_t)rb - a.hh),
                fvd = (float)a.vd;
    float inv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float d = __fadd_rn(__fadd_rn(__fmul_rn(a.T.R[k * 3 + 0], fa), __fmul_rn(a.T.R[k * 3 + 1], fb)),
                                  __fmul_rn(a.T.R[k * 3 + 2], fvd));
        inv[k] = 0.0f;
        if (d != 0.0f) {
            const float q = __frcp_rn(d);
            if (isfinite(q)) inv[k] = q;
        }
    }
    a.ga.inv[t] = make_float4(inv[0], inv[1], inv[2], 0.0f);
    a.ga.hit[t] = kNoHit;
}

// Threads the table needs (the near words alone may be more than the rays).
__host__ __device__ inline int64_t table_threads(const FrameArgs &a) {
    return a.ga.on ? (a.ga.rays > 2 * kNearRows ? a.ga.rays : 2 * kNearRows) : 0;
}

// ---------------------------------------------------------------------------
// Voxels and rays
// ---------------------------------------------------------------------------

// Whether the walk of the ray with reciprocals r visits voxel i, and the key
// E of the crossing it enters by (0: it starts there).
__device__ __forceinline__ bool visits(const float4 &r, const float S[3], const int32_t v0[3], const int32_t i[3],
                                       uint32_t &E) {
    const float inv[3] = {r.x, r.y, r.z};
    uint32_t in = 0, out = kNoHit;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int32_t d = i[k] - v0[k];
        const bool up = inv[k] > 0.0f, act = inv[k] != 0.0f;
        if (d != 0) {
            ok = ok && act && (d > 0) == up;
            in = max(in, event_key(cross_at((float)(i[k] + (up ? 0 : 1)), S[k], inv[k]), k));
        }
        if (act) out = min(out, event_key(cross_at((float)(i[k] + (up ? 1 : 0)), S[k], inv[k]), k));
    }
    E = in;
    return ok && in < out && in < (0x3f800000u << 2);   // t < 1
}

// Calls f(entry, ray, kmin, hit, inv) for every entry of a unit's list and every ray
// of the entry's window (window(entry)), a pair per thread: windows hold from
// one ray to several hundred (near the camera), and with an entry per thread
// or per warp a CTA would end with its widest.  In rounds of 256 entries (16
// of the widest bundles), whose windows are laid end to end.  CTA-cooperative.
struct PairSmem {
    uint32_t end[kThreads], first[kThreads], kmin[kThreads];
    uint16_t na[kThreads], entry[kThreads];
    uint32_t sums[kThreads / 32];
};

template <class L, class W, class F>
__device__ __forceinline__ void for_pairs(const FrameArgs &a, const uint16_t *list, uint32_t n, PairSmem &ps,
                                          W window, F f) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t width = 2u * (uint32_t)a.hw + 1u, round = round_entries(a.ga.rays);
    for (uint32_t l0 = 0; l0 < n; l0 += round) {
        uint32_t count = 0;
        if ((uint32_t)tid < round && l0 + tid < n) {
            const uint32_t e = list[l0 + tid];
            const Window w = window(e);
            count = (uint32_t)w.count();
            ps.entry[tid] = (uint16_t)e;
            ps.na[tid] = (uint16_t)max(w.ahi - w.alo + 1, 1);
            ps.first[tid] = (uint32_t)(w.blo + a.hh) * width + (uint32_t)(w.alo + a.hw);
            ps.kmin[tid] = w.kmin;
        }
        uint32_t end = count;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(kFull, end, d);
            if (lane >= d) end += o;
        }
        if (lane == 31) ps.sums[warp] = end;
        __syncthreads();
        uint32_t total = 0;
#pragma unroll
        for (int k = 0; k < kThreads / 32; ++k) {
            const uint32_t v = ps.sums[k];
            if (k < warp) end += v;
            total += v;
        }
        ps.end[tid] = end;
        __syncthreads();
        // kFlight pairs of each thread in flight: a look-up and a test are
        // chains of loads and latencies
        for (uint32_t t0 = tid; t0 < total; t0 += kThreads * kFlight) {
            uint32_t v[kFlight], ray[kFlight], hit[kFlight];
            float4 inv[kFlight];
#pragma unroll
            for (int k = 0; k < kFlight; ++k) {
                const uint32_t t = min(t0 + k * kThreads, total - 1u);
                uint32_t at = 0;   // the entry of pair t: the first whose pairs end past t
#pragma unroll
                for (int d = kThreads / 2; d > 0; d >>= 1)
                    if (ps.end[at + d - 1] <= t) at += d;
                const uint32_t q = t - (at ? ps.end[at - 1] : 0u), na = ps.na[at];
                const uint32_t row = row_of(q, na, a.ga.rays);
                v[k] = at;
                ray[k] = ps.first[at] + row * width + (q - row * na);
                hit[k] = L::ld(a.ga.hit + ray[k]);
                inv[k] = L::ld(a.ga.inv + ray[k]);
            }
#pragma unroll
            for (int k = 0; k < kFlight; ++k)
                if (t0 + k * kThreads < total) f((uint32_t)ps.entry[v[k]], ray[k], ps.kmin[v[k]], hit[k], inv[k]);
        }
        __syncthreads();
    }
}

// The words of a frame's box in groups of ROWS (4, or 1) rows of one word
// each: thread ROWS g + r has row r of its unit's group g.  The groups of a unit are spread
// evenly over the box: surfaces lie in few slices and rows (a floor is one
// slice) and the voxels near the camera, which many rays cross, close
// together, and units of neighbouring groups would have very different
// amounts of work.
template <int WPU, int ROWS>
__host__ __device__ inline uint32_t word_units(const WordBox &b) {
    const uint32_t groups = (uint32_t)b.nw * (uint32_t)((b.ny + ROWS - 1) / ROWS) * (uint32_t)b.nz;
    return (groups + WPU / ROWS - 1) / (WPU / ROWS);
}

// This thread's word of unit `unit` of `units`: its first voxel in i; false
// if there is none.
template <int ROWS>
__device__ __forceinline__ bool unit_word(const FrameArgs &a, uint32_t unit, uint32_t units, int32_t i[3]) {
    const WordBox &b = a.box;
    const uint32_t group = unit + (threadIdx.x / ROWS) * units;
    const uint32_t gy = (uint32_t)(b.ny + ROWS - 1) / ROWS, t = group / (uint32_t)b.nw, z = t / gy;
    i[0] = (b.w0 + (int32_t)(group - t * (uint32_t)b.nw)) * 32;
    i[1] = b.y0 + (int32_t)((t - z * gy) * ROWS + threadIdx.x % ROWS);
    i[2] = b.z0 + (int32_t)z;
    return z < (uint32_t)b.nz && i[1] < b.y0 + b.ny && i[0] < a.g.nx;
}

__device__ __forceinline__ uint32_t word_of(const PlaneGeom &g, const int32_t i[3]) {
    return ((uint32_t)i[2] * (uint32_t)g.ny + (uint32_t)i[1]) * (uint32_t)g.wx + (uint32_t)(i[0] >> 5);
}

// The word's bits that lie within kNear of the camera's voxel; ny, nz and dx
// place it among the near rows (bit b of a near row is its bit dx less).
__device__ __forceinline__ uint32_t near_bits(const int32_t v0[3], const int32_t i[3], uint32_t &row, int32_t &dx) {
    const uint32_t y = (uint32_t)(i[1] - v0[1] + kNear), z = (uint32_t)(i[2] - v0[2] + kNear);
    dx = i[0] - (v0[0] - kNear);
    row = z * kNearN + y;
    if (y >= (uint32_t)kNearN || z >= (uint32_t)kNearN || dx <= -32 || dx >= kNearN) return 0u;
    const uint32_t all = (1u << kNearN) - 1u;
    return dx >= 0 ? all >> dx : all << -dx;
}

// ---------------------------------------------------------------------------
// K3
// ---------------------------------------------------------------------------

// The voxels around the camera: 256 rays mark what they walk through within
// kNear of the camera's voxel, in shared memory, then in the frame's near
// words.  A ray meets its first hit there only after the voxels before it,
// which are there too, so the box decides for itself.  CTA-cooperative; sh:
// 3 * kNearRows words.
template <class L>
__device__ __forceinline__ void near_unit(const FrameArgs &a, const float S[3], const int32_t v0[3], int32_t unit,
                                          uint32_t *sh) {
    uint32_t *fr = sh, *tr = sh + kNearRows, *occ = sh + 2 * kNearRows;
    const int32_t xs = v0[0] - kNear;
    for (int i = threadIdx.x; i < kNearRows; i += kThreads) {
        const int32_t y = v0[1] - kNear + i % kNearN, z = v0[2] - kNear + i / kNearN;
        uint32_t v = 0;
        if ((unsigned)y < (unsigned)a.g.ny && (unsigned)z < (unsigned)a.g.nz) {
            const uint32_t *row = a.pl.occ_inf + ((uint32_t)z * (uint32_t)a.g.ny + (uint32_t)y) * (uint32_t)a.g.wx;
            const int32_t w = xs >> 5;
            const uint32_t lo = (unsigned)w < (unsigned)a.g.wx ? L::ld(row + w) : 0u;
            const uint32_t hi = (unsigned)(w + 1) < (unsigned)a.g.wx ? L::ld(row + w + 1) : 0u;
            v = __funnelshift_r(lo, hi, xs & 31);
        }
        occ[i] = v;
        fr[i] = 0;
        tr[i] = 0;
    }
    __syncthreads();
    const int64_t ray = (int64_t)unit * kThreads + threadIdx.x;
    if (ray < a.ga.rays) {
        const float4 r = L::ld(a.ga.inv + ray);
        const float inv[3] = {r.x, r.y, r.z};
        float nb[3], t[3], fs[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            fs[k] = inv[k] > 0.0f ? 1.0f : -1.0f;
            nb[k] = (float)(v0[k] + (inv[k] > 0.0f));
            t[k] = inv[k] != 0.0f ? cross_at(nb[k], S[k], inv[k]) : INFINITY;
        }
        const int32_t s0 = inv[0] > 0.0f ? 1 : -1, s1 = inv[1] > 0.0f ? 1 : -1, s2 = inv[2] > 0.0f ? 1 : -1;
        int32_t p0 = kNear, p1 = kNear, p2 = kNear;
        uint32_t key = 0, hit = kNoHit;
        for (;;) {
            const int32_t row = p2 * kNearN + p1;
            const uint32_t bit = 1u << p0;
            if (hit == kNoHit && (occ[row] & bit)) hit = key;
            uint32_t *to = (hit != kNoHit ? tr : fr) + row;
            if (!(*reinterpret_cast<volatile uint32_t *>(to) & bit)) atomicOr(to, bit);
            const float tm = fminf(t[0], fminf(t[1], t[2]));
            if (!(tm < 1.0f)) break;
            int32_t p;
            if (t[0] == tm) {
                p = p0 += s0;
                nb[0] = __fadd_rn(nb[0], fs[0]);
                t[0] = cross_at(nb[0], S[0], inv[0]);
                key = event_key(tm, 0);
            } else if (t[1] == tm) {
                p = p1 += s1;
                nb[1] = __fadd_rn(nb[1], fs[1]);
                t[1] = cross_at(nb[1], S[1], inv[1]);
                key = event_key(tm, 1);
            } else {
                p = p2 += s2;
                nb[2] = __fadd_rn(nb[2], fs[2]);
                t[2] = cross_at(nb[2], S[2], inv[2]);
                key = event_key(tm, 2);
            }
            if ((unsigned)p >= (unsigned)kNearN) break;
        }
        if (hit != kNoHit) atomicMin(a.ga.hit + ray, hit);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kNearRows; i += kThreads) {
        if (fr[i] & ~__ldcg(a.ga.near_fr + i)) atomicOr(a.ga.near_fr + i, fr[i]);
        if (tr[i] & ~__ldcg(a.ga.near_tr + i)) atomicOr(a.ga.near_tr + i, tr[i]);
    }
    __syncthreads();   // the shared memory may be reused right away
}

__host__ __device__ inline int32_t near_units_of(const FrameArgs &a) { return (a.ga.rays + kThreads - 1) / kThreads; }

struct SkinSmem {
    uint32_t at[kThreads];   // the word's place: x word, y, z in 7, 12 and 12 bits
    uint16_t list[kFaces];   // faces: (word slot * 32 + bit) * 4 + axis
    PairSmem pairs;
    uint32_t n, limit;
};

// K3 of one of `units` units of kThreads plane words.  A round lists at most
// kFaces faces; threads whose faces no longer fit wait for the next (a word
// has at most 96, so every round takes some).  CTA-cooperative.
template <class L>
__device__ __forceinline__ void skin_unit(const FrameArgs &a, const float S[3], const int32_t v0[3], uint32_t unit,
                                          uint32_t units, SkinSmem &sh) {
    const Gather &g = a.ga;
    const int tid = threadIdx.x;
    uint32_t skin[3] = {0, 0, 0};
    int32_t i[3];
    const bool any = unit_word<1>(a, unit, units, i);
    sh.at[tid] = (uint32_t)i[0] >> 5 | (uint32_t)i[1] << 7 | (uint32_t)i[2] << 19;
    if (any) {
        const uint32_t *p = a.pl.occ_inf + word_of(a.g, i);
        const uint32_t oc = L::ld(p);
        if (oc) {
            if (in_bundle(a, place_of(g, (float)(i[0] + 16) - S[0], (float)i[1] + 0.5f - S[1], (float)i[2] + 0.5f - S[2]),
                          g.ew, g.zw)) {
                // faces towards the camera whose other side is unoccupied (none
                // along an axis on which the voxel is level with the camera)
                uint32_t ny = kFull, nz = kFull;
                if (i[1] > v0[1]) ny = i[1] > 0 ? L::ld(p - a.g.wx) : 0u;
                if (i[1] < v0[1]) ny = i[1] + 1 < a.g.ny ? L::ld(p + a.g.wx) : 0u;
                if (i[2] > v0[2]) nz = i[2] > 0 ? L::ld(p - (int64_t)a.g.wx * a.g.ny) : 0u;
                if (i[2] < v0[2]) nz = i[2] + 1 < a.g.nz ? L::ld(p + (int64_t)a.g.wx * a.g.ny) : 0u;
                const uint32_t prev = i[0] > 0 ? L::ld(p - 1) : 0u;
                const uint32_t next = i[0] + 32 < 32 * a.g.wx ? L::ld(p + 1) : 0u;
                const int32_t c = v0[0] - i[0];   // the camera's bit of this word
                const uint32_t at = c >= 0 && c < 32 ? 1u << c : 0u;
                const uint32_t lt = c <= 0 ? 0u : (c >= 32 ? kFull : at - 1u);   // bits nearer x = 0 than the camera
                const uint32_t nx = (__funnelshift_l(prev, oc, 1) & ~lt) | (__funnelshift_r(oc, next, 1) & lt) | at;
                uint32_t row;
                int32_t dx;
                const uint32_t far = oc & ~near_bits(v0, i, row, dx);
                skin[0] = far & ~nx;
                skin[1] = far & ~ny;
                skin[2] = far & ~nz;
            }
        }
    }
    auto voxel = [&](uint32_t e, int32_t i[3]) {
        const uint32_t at = sh.at[e >> 7];
        i[0] = (int32_t)((at & 127u) * 32u + ((e >> 2) & 31u));
        i[1] = (int32_t)((at >> 7) & 4095u);
        i[2] = (int32_t)((at >> 19) & 4095u);
    };
    auto window = [&](uint32_t e) {
        int32_t i[3];
        voxel(e, i);
        return face_window(a, S, v0, i, (int)(e & 3u));
    };
    bool left;
    do {
        if (tid == 0) {
            sh.n = 0;
            sh.limit = kFaces;
        }
        __syncthreads();
        const uint32_t cnt = (uint32_t)(__popc(skin[0]) + __popc(skin[1]) + __popc(skin[2]));
        uint32_t pos = cnt ? atomicAdd(&sh.n, cnt) : 0u;
        left = pos + cnt > (uint32_t)kFaces;
        if (left) {
            atomicMin(&sh.limit, pos);   // later threads' faces do not fit either
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                for (uint32_t b = skin[k]; b; b &= b - 1)
                    sh.list[pos++] = (uint16_t)((tid * 32 + __ffs(b) - 1) * 4 + k);
                skin[k] = 0;
            }
        }
        left = __syncthreads_or(left);
        for_pairs<L>(a, sh.list, min(sh.n, sh.limit), sh.pairs, window,
                     [&](uint32_t e, uint32_t ray, uint32_t kmin, uint32_t h, const float4 &r) {
            // (an older value of the hit only costs an atomicMin too many)
            int32_t i[3];
            uint32_t E;
            voxel(e, i);
            if (h > kmin && visits(r, S, v0, i, E) && E < h) atomicMin(g.hit + ray, E);
        });
        __syncthreads();
    } while (left);
}

// The latest hit key of each tile of 8 x 8 rays, for wide windows, and the
// latest among the rays within kReach of each ray, into the fourth word of
// its inv entry: one look tells a voxel behind its nearest
// ray's hit that no ray that may reach it (its window, from depth zr on, lies
// within kReach - 1/2) hits later.  A tile of 32 x 8 rays per CTA.
constexpr int kLateW = 32, kLateH = 8, kReach = kLateReach;
struct LateSmem {
    uint32_t in[kLateH + 2 * kReach][kLateW + 2 * kReach], row[kLateH + 2 * kReach][kLateW];
};

__host__ __device__ inline int32_t tiles_x(const FrameArgs &a) { return (2 * a.hw + 8) >> 3; }
__host__ __device__ inline int32_t late_units_x(const FrameArgs &a) { return (2 * a.hw + kLateW) / kLateW; }
__host__ __device__ inline int32_t late_units(const FrameArgs &a) {
    return late_units_x(a) * ((2 * a.hh + kLateH) / kLateH);
}

template <class L>
__device__ __forceinline__ void late_unit(const FrameArgs &a, int32_t unit, LateSmem &sh) {
    const int32_t width = 2 * a.hw + 1, height = 2 * a.hh + 1, ux = late_units_x(a);
    const int32_t x0 = (unit % ux) * kLateW, y0 = (unit / ux) * kLateH;
    constexpr int kInW = kLateW + 2 * kReach, kInH = kLateH + 2 * kReach;
    for (int t = threadIdx.x; t < kInW * kInH; t += kThreads) {
        const int32_t x = x0 - kReach + t % kInW, y = y0 - kReach + t / kInW;
        uint32_t v = 0;
        if (x >= 0 && x < width && y >= 0 && y < height) v = L::ld(a.ga.hit + y * width + x);
        sh.in[t / kInW][t % kInW] = v;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < kLateW * kInH; t += kThreads) {
        const int x = t % kLateW, y = t / kLateW;
        uint32_t v = 0;
#pragma unroll
        for (int d = 0; d <= 2 * kReach; ++d) v = max(v, sh.in[y][x + d]);
        sh.row[y][x] = v;
    }
    __syncthreads();
    const int32_t lx = threadIdx.x % kLateW, ly = threadIdx.x / kLateW, x = x0 + lx, y = y0 + ly;
    uint32_t v = 0;
#pragma unroll
    for (int d = 0; d <= 2 * kReach; ++d) v = max(v, sh.row[ly + d][lx]);
    if (x < width && y < height) a.ga.inv[y * width + x].w = __uint_as_float(v);
    if (threadIdx.x < 4 * 32) {
        const int tx = threadIdx.x >> 5, l = threadIdx.x & 31;
        uint32_t m = 0;
#pragma unroll
        for (int k = 0; k < 2; ++k) m = max(m, sh.in[kReach + (l >> 3) + 4 * k][kReach + 8 * tx + (l & 7)]);
        m = __reduce_max_sync(kFull, m);
        if (l == 0 && x0 + 8 * tx < width) a.ga.tile[(y0 >> 3) * tiles_x(a) + (x0 >> 3) + tx] = m;
    }
    __syncthreads();   // the shared memory may be reused right away
}

// ---------------------------------------------------------------------------
// K4: every voxel's state, into loc_grid.
// ---------------------------------------------------------------------------
// Shared memory of a unit of WPU words: four rows by eight voxels make a
// patch, and byte p of the four words of a group are patch p's rows, so thread
// 4 g + p stands for word p and for patch p of group g.  Masks are kept as
// bytes [word][patch].
template <int WPU>
struct GatherSmem {
    uint32_t oc[WPU], need[WPU], fr[WPU], tr[WPU], ent[WPU];
    uint32_t at[WPU];          // the word's place: x word, y, z in 7, 12 and 12 bits
    Place first[WPU];          // the place of the patch's first voxel in camera axes
    uint32_t row[WPU];         // the first byte of the word's row in the ring-addressed loc_grid
    uint16_t list[WPU];        // patches that touch the bundle: well inside; from the end: at its edges
    uint16_t open[WPU * 32];   // voxels to resolve: patch * 32 + voxel; from the end: those the nearest ray traces
    uint16_t hard[WPU * 32];   // voxels that take every ray of their windows
    PairSmem pairs;
    uint32_t nlist, nopen, nhard;   // the first two: entries, and from bit 16 those from the end
};

// Appends this lane's value to a list in shared memory if `in`; all lanes of
// the warp call it.
__device__ __forceinline__ void push(uint16_t *list, uint32_t *n, bool in, uint32_t v) {
    const unsigned m = __ballot_sync(kFull, in);
    if (m == 0) return;
    const int lane = threadIdx.x & 31;
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(n, (uint32_t)__popc(m));
    at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (in) list[at] = (uint16_t)v;
}

// K4 of one of `units` units of WPU plane words: resolves the voxels, writes
// their codes through the ring (as merge_word does: unknown where a re-centre
// brought the voxel in and nothing marks it) and clears the occupancy words.
// CTA-cooperative.
// SPLIT: patches well inside the bundle and at its edges are resolved by loops
// of their own (a frame alone: 208 -> 193 us for three 1280x720 frames); the
// fused batch, whose code is larger than the instruction cache likes, keeps
// one (a step of 64 robots 550 us, 566 with two).
template <int WPU, bool SPLIT, class L>
__device__ __forceinline__ void gather_unit(const FrameArgs &a, const float S[3], const int32_t v0[3], uint32_t unit,
                                            uint32_t units, GatherSmem<WPU> &sh) {
    const Gather &g = a.ga;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float fvd = (float)a.vd;
    if (tid == 0) {
        sh.nlist = 0;
        sh.nopen = 0;
        sh.nhard = 0;
    }
    __syncthreads();

    // ---- the words: occupancy, near marks; the patches inside the bundle --
    static_assert(WPU % 32 == 0 && WPU <= kThreads, "a thread per word");
    if (tid < WPU) {
        uint32_t oc = 0, need = 0, nf = 0, nt = 0, ent = 0;
        int32_t i[3];
        if (unit_word<4>(a, unit, units, i)) {
            const uint32_t w = word_of(a.g, i);
            sh.row[tid] = (uint32_t)(units::ring_at(i[2], a.ring.r[2], a.g.nz) * a.g.ny +
                                     units::ring_at(i[1], a.ring.r[1], a.g.ny)) * (uint32_t)a.g.nx;
            oc = L::ld(a.pl.occ_inf + w);
            const int nbits = min(32, a.g.nx - i[0]);
            const uint32_t valid = nbits >= 32 ? kFull : ((1u << nbits) - 1u);
            ent = units::entering_bits(a.ring, i[0], i[1], i[2], nbits);
            uint32_t row;
            int32_t dx;
            const uint32_t near = near_bits(v0, i, row, dx) & valid;
            if (near) {
                const uint32_t f = L::ld(g.near_fr + row), t = L::ld(g.near_tr + row);
                nf = (dx >= 0 ? f >> dx : f << -dx) & valid;
                nt = (dx >= 0 ? t >> dx : t << -dx) & valid;
            }
            need = valid & ~oc & ~near;
            if (oc) {
                a.pl.occ_inf[w] = 0;
                a.pl.occ_raw[w] = 0;
            }
        }
        sh.oc[tid] = oc;
        sh.need[tid] = need;
        sh.fr[tid] = nf;
        sh.tr[tid] = nt;
        sh.ent[tid] = ent;
        sh.at[tid] = (uint32_t)i[0] >> 5 | (uint32_t)i[1] << 7 | (uint32_t)i[2] << 19;
        const Place p = place_of(g, (float)(i[0] + 8 * (tid & 3)) + 0.5f - S[0], (float)(i[1] - (tid & 3)) + 0.5f - S[1],
                                 (float)i[2] + 0.5f - S[2]);
        sh.first[tid] = p;
        const Place m = {__fmaf_rn(1.5f, g.M[1], __fmaf_rn(3.5f, g.M[0], p.c0)),
                         __fmaf_rn(1.5f, g.M[4], __fmaf_rn(3.5f, g.M[3], p.c1)),
                         __fmaf_rn(1.5f, g.M[7], __fmaf_rn(3.5f, g.M[6], p.c2))};
        const bool in = in_bundle(a, m, g.ep, g.zp);
        const bool inside = __fmaf_rn(-g.ka, m.c2, m.c0) <= -g.ep[0] && __fmaf_rn(-g.ka, m.c2, -m.c0) <= -g.ep[1] &&
                            __fmaf_rn(-g.kb, m.c2, m.c1) <= -g.ep[2] && __fmaf_rn(-g.kb, m.c2, -m.c1) <= -g.ep[3] &&
                            m.c2 - g.zp > 0.5f && m.c2 + g.zp < fvd;
        uint32_t some = need | __shfl_xor_sync(kFull, need, 1);   // the patch's columns, over its four rows
        some = ((some | __shfl_xor_sync(kFull, some, 2)) >> (8 * (tid & 3))) & 255u;
        const unsigned mi = __ballot_sync(kFull, in && some && inside), me = __ballot_sync(kFull, in && some && !inside);
        if (mi | me) {
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(&sh.nlist, (uint32_t)__popc(mi) + ((uint32_t)__popc(me) << 16));
            at = __shfl_sync(kFull, at, 0);
            const unsigned below = (1u << lane) - 1u;
            if ((mi >> lane) & 1u) sh.list[(at & 0xffffu) + __popc(mi & below)] = (uint16_t)tid;
            if ((me >> lane) & 1u) sh.list[WPU - 1 - (at >> 16) - __popc(me & below)] = (uint16_t)tid;
        }
    }
    __syncthreads();

    // ---- the certain cases, a patch per warp, a voxel per lane ------------
    const uint8_t *need8 = reinterpret_cast<const uint8_t *>(sh.need);
    uint8_t *fr8 = reinterpret_cast<uint8_t *>(sh.fr), *tr8 = reinterpret_cast<uint8_t *>(sh.tr);
    const float ivd = 1.0f / fvd, fw = (float)a.hw, fh = (float)a.hh;
    const float zmin = g.zv + g.m;
    const float lx = (float)(lane & 7), ly = (float)(lane >> 3);
    const float o0 = __fmaf_rn(ly, g.M[1], lx * g.M[0]), o1 = __fmaf_rn(ly, g.M[4], lx * g.M[3]),
                o2 = __fmaf_rn(ly, g.M[7], lx * g.M[6]);
    const int32_t width = 2 * a.hw + 1, centre = a.hh * width + a.hw;
    const uint32_t *hits = g.hit + centre;
    const uint32_t *latest = reinterpret_cast<const uint32_t *>(g.inv + centre) + 3;
    const uint32_t kzr = __float_as_uint(fminf((g.zr - zmin) * ivd, 1.5f)) << 2;   // (1.5: never)
    auto certain = [&](auto edge, uint32_t l0, uint32_t nlist) {
        const bool kEdge = edge;
        uint32_t patch[kFlight], hit[kFlight], late[kFlight], kmin[kFlight], kmid[kFlight];
        int32_t ray[kFlight];
        bool in[kFlight];
#pragma unroll
        for (int k = 0; k < kFlight; ++k) {
            const uint32_t l = min(l0 + k, nlist - 1u);
            patch[k] = sh.list[kEdge ? WPU - 1 - l : l];
            const Place q = sh.first[patch[k]];
            const Place p = {q.c0 + o0, q.c1 + o1, q.c2 + o2};
            in[k] = l0 + k < nlist && (((uint32_t)need8[4u * ((patch[k] & ~3u) + (uint32_t)(lane >> 3)) + (patch[k] & 3u)] >> (lane & 7)) & 1u);
            bool ranged = in[k];
            if (kEdge) {
                in[k] = in[k] && in_bundle(a, p, g.ev, g.zv);
                ranged = in[k] && p.c2 > 0.5f && p.c2 < fvd - g.m;
            }
            // the nearest ray, its indices by adding 1.5 * 2^23
            const float z = __fdividef(fvd, p.c2), tau = p.c2 * ivd;
            float fa = p.c0 * z, fb = p.c1 * z;
            if (kEdge) {
                fa = fminf(fmaxf(fa, -fw), fw);
                fb = fminf(fmaxf(fb, -fh), fh);
            }
            const float ma = fa + 12582912.0f, mb = fb + 12582912.0f;
            const float da = __fmaf_rn(12582912.0f - ma, tau, p.c0), db = __fmaf_rn(12582912.0f - mb, tau, p.c1);
            ray[k] = (__float_as_int(mb) - 0x4b400000) * width + (__float_as_int(ma) - 0x4b400000);
            kmin[k] = __float_as_uint(fmaxf((p.c2 - zmin) * ivd, 0.0f)) << 2;
            kmid[k] = __float_as_uint(tau) << 2 | 3u;
            hit[k] = kNone;
            if (ranged && __fmaf_rn(da, da, db * db) < g.sphere2) hit[k] = L::ld(hits + ray[k]);
        }
#pragma unroll
        for (int k = 0; k < kFlight; ++k) {
            late[k] = kNoHit;
            if (hit[k] < kmin[k] && kmin[k] >= kzr) late[k] = L::ld(latest + 4 * ray[k]);
        }
        // free: the hit lies past the centre; traced: before the voxel's
        // nearest depth, and final unless some ray that reaches the voxel
        // hits later
        unsigned mo[kFlight], mb[kFlight];
        uint32_t count = 0;   // of the open ones, and from bit 16 of those behind
#pragma unroll
        for (int k = 0; k < kFlight; ++k) {
            const bool free = hit[k] != kNone && hit[k] > kmid[k];
            const bool behind = hit[k] < kmin[k], traced = late[k] < kmin[k];
            const unsigned mf = __ballot_sync(kFull, free), mt = __ballot_sync(kFull, behind);
            mo[k] = __ballot_sync(kFull, in[k] && !free && !behind);
            mb[k] = __ballot_sync(kFull, behind && !traced);
            count += (uint32_t)__popc(mo[k]) + ((uint32_t)__popc(mb[k]) << 16);
            if ((lane & 7) == 0) {   // a row each
                const uint32_t byte = 4u * ((patch[k] & ~3u) + (uint32_t)(lane >> 3)) + (patch[k] & 3u);
                const uint32_t f = (mf >> lane) & 255u, t = (mt >> lane) & 255u;
                if (f) fr8[byte] |= (uint8_t)f;
                if (t) tr8[byte] |= (uint8_t)t;
            }
        }
        if (count) {
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(&sh.nopen, count);
            at = __shfl_sync(kFull, at, 0);
            const unsigned below = (1u << lane) - 1u;
            uint32_t po = at & 0xffffu, pb = WPU * 32 - 1 - (at >> 16);
#pragma unroll
            for (int k = 0; k < kFlight; ++k) {
                if ((mo[k] >> lane) & 1u) sh.open[po + __popc(mo[k] & below)] = (uint16_t)(patch[k] * 32 + lane);
                if ((mb[k] >> lane) & 1u) sh.open[pb - __popc(mb[k] & below)] = (uint16_t)(patch[k] * 32 + lane);
                po += __popc(mo[k]);
                pb -= __popc(mb[k]);
            }
        }
    };
    const uint32_t nin = sh.nlist & 0xffffu, nedge = sh.nlist >> 16;
    if (SPLIT) {
        for (uint32_t l0 = warp * kFlight; l0 < nin; l0 += kThreads / 32 * kFlight)
            certain(std::false_type(), l0, nin);
        // (the other way round, so that the warps that had a round less begin)
        for (uint32_t l0 = (kThreads / 32 - 1 - warp) * kFlight; l0 < nedge; l0 += kThreads / 32 * kFlight)
            certain(std::true_type(), l0, nedge);
    } else {
        const uint32_t rounds = (nin + kFlight - 1) / kFlight, all = rounds + (nedge + kFlight - 1) / kFlight;
        for (uint32_t l = warp; l < all; l += kThreads / 32) {
            const bool edge = l >= rounds;
            certain(edge, (edge ? l - rounds : l) * kFlight, edge ? nedge : nin);
        }
    }
    __syncthreads();

    // an entry's word and bit, voxel and place
    auto word_bit = [&](uint32_t e, uint32_t &bit) {
        bit = 1u << (((e >> 5) & 3u) * 8u + (e & 7u));
        return ((e >> 5) & ~3u) + ((e >> 3) & 3u);
    };
    auto voxel = [&](uint32_t e, int32_t i[3]) {
        const uint32_t at = sh.at[((e >> 5) & ~3u) + ((e >> 3) & 3u)];
        i[0] = (int32_t)((at & 127u) * 32u + ((e >> 5) & 3u) * 8u + (e & 7u));
        i[1] = (int32_t)((at >> 7) & 4095u);
        i[2] = (int32_t)((at >> 19) & 4095u);
    };
    auto place = [&](uint32_t e) {
        const Place q = sh.first[e >> 5];
        const float x = (float)(e & 7u), y = (float)((e >> 3) & 3u);
        return Place{__fmaf_rn(y, g.M[1], __fmaf_rn(x, g.M[0], q.c0)), __fmaf_rn(y, g.M[4], __fmaf_rn(x, g.M[3], q.c1)),
                     __fmaf_rn(y, g.M[7], __fmaf_rn(x, g.M[6], q.c2))};
    };
    auto window = [&](uint32_t e) { return window_of(a, place(e), 0.5f, g.zv); };

    // ---- traced ones that a later hit of some ray in their window may free
    const uint32_t nback = sh.nopen >> 16, nopen = sh.nopen & 0xffffu;
    for (uint32_t l0 = warp * 32; l0 < nback; l0 += kThreads) {
        uint32_t e = 0;
        bool hard = false;
        if (l0 + lane < nback) {
            e = sh.open[WPU * 32 - 1 - (l0 + lane)];
            const Window w = window(e);
            hard = true;
            // the latest hit of the window, ray by ray or of its tiles
            const bool tiled = w.count() > 12;
            const int32_t sh3 = tiled ? 3 : 0, pitch = tiled ? tiles_x(a) : width;
            const uint32_t *from = tiled ? g.tile : g.hit;
            const int32_t x0 = (w.alo + a.hw) >> sh3, x1 = (w.ahi + a.hw) >> sh3, y1 = (w.bhi + a.hh) >> sh3;
            uint32_t last = 0;
            for (int32_t y = (w.blo + a.hh) >> sh3; y <= y1; ++y) {
                const uint32_t *row = from + y * pitch;
                for (int32_t x = x0; x <= x1; x += 4) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) last = max(last, L::ld(row + min(x + k, x1)));
                }
            }
            hard = last > w.kmin;
        }
        push(sh.hard, &sh.nhard, hard, e);
    }

    // ---- the others by their nearest ray ----------------------------------
    for (uint32_t l0 = warp * 32; l0 < nopen; l0 += kThreads) {
        uint32_t e = 0;
        bool hard = false;
        if (l0 + lane < nopen) {
            e = sh.open[l0 + lane];
            const Place p = place(e);
            const float z = __fdividef(fvd, fmaxf(p.c2, 0.1f));
            const int32_t ra = (int32_t)rintf(fminf(fmaxf(p.c0 * z, -fw), fw));
            const int32_t rb = (int32_t)rintf(fminf(fmaxf(p.c1 * z, -fh), fh));
            const uint32_t h = L::ld(hits + rb * width + ra);
            int32_t i[3];
            uint32_t E;
            voxel(e, i);
            hard = true;
            const float4 v = L::ld(g.inv + (centre + rb * width + ra));
            if (visits(v, S, v0, i, E)) {
                // traced for good if no ray that reaches it hits later
                const uint32_t kmin = __float_as_uint(fmaxf((p.c2 - zmin) * ivd, 0.0f)) << 2;
                hard = E >= h;
                const bool last = hard && kmin >= kzr && __float_as_uint(v.w) < kmin;
                uint32_t bit;
                const uint32_t slot = word_bit(e, bit);
                atomicOr((hard ? sh.tr : sh.fr) + slot, bit);
                hard = hard && !last;
            }
        }
        push(sh.hard, &sh.nhard, hard, e);
    }
    __syncthreads();

    // ---- the rest by every ray of their windows ---------------------------
    for_pairs<L>(a, sh.hard, sh.nhard, sh.pairs, window, [&](uint32_t e, uint32_t, uint32_t kmin, uint32_t h,
                                                                      const float4 &r) {
        uint32_t bit;
        const uint32_t slot = word_bit(e, bit);
        volatile uint32_t *fr = sh.fr + slot, *tr = sh.tr + slot;
        if (*fr & bit) return;
        if (h <= kmin && (*tr & bit)) return;   // this ray could only trace it
        int32_t i[3];
        uint32_t E;
        voxel(e, i);
        if (!visits(r, S, v0, i, E)) return;
        if (E < h) atomicOr(&sh.fr[slot], bit);
        else if (!(*tr & bit)) atomicOr(&sh.tr[slot], bit);
    });

    // ---- codes through the ring: a word per 8 lanes, 4 voxels per lane ----
    for (uint32_t slot = tid >> 3; slot < (uint32_t)WPU; slot += kThreads / 8) {
        const int s = 4 * (lane & 7);
        const uint32_t oc = sh.oc[slot], f = sh.fr[slot], t = sh.tr[slot], en = sh.ent[slot];
        const uint32_t touch = ((oc | f | t | en) >> s) & 15u;
        if (touch == 0) continue;
        uint32_t hi, lo, known;
        units::code_masks(oc >> s, f >> s, t >> s, hi, lo, known);
        const uint32_t code = units::merge4(hi, lo, known, 0, 0u);
        const uint32_t at = sh.at[slot];
        uint8_t *rowp = a.loc + sh.row[slot];
        const int32_t x = (int32_t)(at & 127u) * 32 + s, xb = units::ring_at(x, a.ring.r[0], a.g.nx);
        uint8_t *p = rowp + xb;
        if (touch == 15u && xb + 4 <= a.g.nx && (reinterpret_cast<uintptr_t>(p) & 3u) == 0) {
            *reinterpret_cast<uint32_t *>(p) = code;
        } else {
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if ((touch >> b) & 1u) rowp[xb + b >= a.g.nx ? xb + b - a.g.nx : xb + b] = (uint8_t)(code >> (8 * b));
        }
    }
    __syncthreads();   // the shared memory may be reused right away
}

// What lies outside the frame's box, a word per thread; the box's own words
// are gather_unit's.  The voxels a re-centre brought in: words of the slabs it
// brought in along x, y and z (words in two slabs are written twice, alike).
// A cloud's points too (`whole`): all words of the grid.  Its box holds the
// rays alone, since gathering a word costs more than merging it: 300,000 points
// around the robot into 400 x 400 x 120 voxels took 65 us a frame with the grid
// as the box.
__host__ __device__ inline int64_t outside_words(const FrameArgs &a, int64_t part[3]) {
    const Ring &R = a.ring;
    const int64_t used = (a.g.nx + 31) / 32;
    const WordBox &b = a.box;
    part[0] = part[1] = part[2] = 0;
    if (b.w0 == 0 && b.nw >= used && b.ny == a.g.ny && b.nz == a.g.nz) return 0;
    if (a.whole) return used * a.g.ny * a.g.nz;
    part[0] = R.ehi[0] > R.elo[0] ? (int64_t)((R.ehi[0] + 31) / 32 - R.elo[0] / 32) * a.g.ny * a.g.nz : 0;
    part[1] = (int64_t)(R.ehi[1] - R.elo[1]) * used * a.g.nz;
    part[2] = (int64_t)(R.ehi[2] - R.elo[2]) * used * a.g.ny;
    return part[0] + part[1] + part[2];
}
__host__ __device__ inline int64_t outside_units(const FrameArgs &a, int threads) {
    int64_t part[3];
    return (outside_words(a, part) + threads - 1) / threads;
}

template <bool WHOLE>
__device__ __forceinline__ void outside_word(const FrameArgs &a, int64_t t) {
    const Ring &R = a.ring;
    int64_t part[3];
    if (t >= outside_words(a, part)) return;
    const uint32_t used = (uint32_t)(a.g.nx + 31) / 32u;
    int32_t i[3];
    if (WHOLE) {
        const uint32_t row = (uint32_t)t / used;   // grids hold fewer than 2^27 words
        i[0] = (int32_t)((uint32_t)t - row * used) * 32;
        i[2] = (int32_t)(row / (uint32_t)a.g.ny);
        i[1] = (int32_t)(row - (uint32_t)i[2] * (uint32_t)a.g.ny);
    } else if (t < part[0]) {
        const uint32_t nw = (uint32_t)((R.ehi[0] + 31) / 32 - R.elo[0] / 32), row = (uint32_t)t / nw;
        i[0] = (R.elo[0] / 32 + (int32_t)((uint32_t)t - row * nw)) * 32;
        i[2] = (int32_t)(row / (uint32_t)a.g.ny);
        i[1] = (int32_t)(row - (uint32_t)i[2] * (uint32_t)a.g.ny);
    } else {
        const bool in_y = t - part[0] < part[1];
        const uint32_t u = (uint32_t)(t - part[0] - (in_y ? 0 : part[1])), row = u / used;
        const int32_t lo = in_y ? R.elo[1] : R.elo[2];
        const uint32_t thick = (uint32_t)((in_y ? R.ehi[1] : R.ehi[2]) - lo), other = row / thick;
        const int32_t within = lo + (int32_t)(row - other * thick);
        i[0] = (int32_t)(u - row * used) * 32;
        i[1] = in_y ? within : (int32_t)other;
        i[2] = in_y ? (int32_t)other : within;
    }
    const WordBox &b = a.box;
    if ((uint32_t)((i[0] >> 5) - b.w0) < (uint32_t)b.nw && (uint32_t)(i[1] - b.y0) < (uint32_t)b.ny &&
        (uint32_t)(i[2] - b.z0) < (uint32_t)b.nz)
        return;
    const uint32_t w = word_of(a.g, i);
    const uint32_t oc = WHOLE ? a.pl.occ_inf[w] : 0u;
    const int nbits = min(32, a.g.nx - i[0]);
    const uint32_t touch = oc | units::entering_bits(R, i[0], i[1], i[2], nbits);
    if (touch == 0) return;
    uint32_t codes[9] = {};   // unknown
    if (WHOLE && oc) {
#pragma unroll
        for (int m = 0; m < 8; ++m) codes[m] = units::merge4(oc, 0u, oc, m, 0u);
        a.pl.occ_inf[w] = 0;
        a.pl.occ_raw[w] = 0;
    }
    uint8_t *rowp = a.loc + ((int64_t)units::ring_at(i[2], R.r[2], a.g.nz) * a.g.ny +
                             units::ring_at(i[1], R.r[1], a.g.ny)) * a.g.nx;
    const int32_t xb = units::ring_at(i[0], R.r[0], a.g.nx);
    const int n1 = min(nbits, a.g.nx - xb);
    units::store_codes(rowp + xb, 0, n1, codes, touch);
    if (n1 < nbits) units::store_codes(rowp, n1, nbits, codes, touch);
}

}  // namespace gather
}  // namespace vg
