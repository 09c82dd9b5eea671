// vg_units.cuh -- the work of K1, K2, K4 and K5 as device functions over one
// unit of work, shared by the one-kernel-per-step launches (k_*.cu) and the
// fused persistent launch (k_batch.cu).
//
// Loads of data that an earlier launch or phase wrote go through a load
// policy: LoadPlain (ordinary loads) or LoadL2 (loads that skip the SM's L1;
// ordinary ones see what was written before a grid barrier as well, by its
// fences).
// None take the read-only path: it is for data that nothing writes while the
// kernel lives, and the one-step kernels are dependent launches, alive while
// the kernel before them still writes.
#pragma once

#include "vg_internal.cuh"

namespace vg {
namespace units {

constexpr unsigned kFull = 0xffffffffu;

struct LoadPlain {
    template <class T>
    static __device__ __forceinline__ T ld(const T *p) { return *p; }
};

struct LoadL2 {
    template <class T>
    static __device__ __forceinline__ T ld(const T *p) { return __ldcg(p); }
};

// ---------------------------------------------------------------------------
// K1: transform and voxelize (Sec. IV-B, Alg. 1 before the inflation loops).
//
// Each thread reads four consecutive pixels of a row of a 32 x 32 tile of the
// depth image (one 16-byte float4 or 8-byte ushort4 load when aligned),
// back-projects the valid ones with the pinhole model, transforms them by
// T^v_c and sets their voxel's bit in the occ_raw plane.  The plane is
// bit-packed, so concurrent sets need an atomic, but neighbouring pixels, of
// a row and of a column, often land in the same 32-voxel word: a CTA gathers
// its tile's words in a small table in shared memory (WordTab) and sets each
// in the plane once.  (1280x720: 14.4 -> 9.2 us, 640x480 8.1 -> 7.2, against an
// OR-scan over a warp's row of 128 pixels and an atomic per run of lanes:
// 4.4 of the 14.4 us were the atomics.  About 4 us are a launch's with the
// ray table; the rest is issue, 150 instructions a pixel's warp.  256 slots;
// with 512, whose clearing and scanning cost more, 9.7 us.)
//
// Arithmetic follows the oracle's order with one IEEE rounding per operation
// (explicit __f*_rn intrinsics; the translation units are also built with
// -fmad=false):
//   xc = ((u - cx) * d) / fx,  yc = ((v - cy) * d) / fy,  zc = d
//   g_k = (((R_k0 xc + R_k1 yc) + R_k2 zc) + t_k) / vox_size
//   kept iff 0 <= g_k < N_k on every axis; voxel = floor(g).
// ---------------------------------------------------------------------------
constexpr uint32_t kNoWord = 0xffffffffu;

// x / y rounded to nearest, r = 1 / y rounded to nearest: Markstein's method
// (IBM J. Res. Dev. 34, 1990): two corrections by the exact remainder, the
// second of a quotient within an ulp, round as IEEE division does unless y's
// significand is all ones or the remainder underflows, which the callers
// exclude (r = 0, and |x| below 1e-18, take __fdiv_rn; x = 0 is exact).  K1
// divides five times a pixel by three constants: this way without the
// reciprocal unit, which its conversions keep busy (1280x720: 14.4 -> 13.8 us;
// 64 robots' phase, with the voxels floored by the conversion itself and the
// shorter warp_set_bits: a step 584 -> 550).
__device__ __forceinline__ float div_by(float x, float y, float r) {
    float q = __fmul_rn(x, r);
    q = __fmaf_rn(__fmaf_rn(-q, y, x), r, q);
    return __fmaf_rn(__fmaf_rn(-q, y, x), r, q);
}

// Returns the plane word of the point's voxel and its bit, or kNoWord.
__device__ __forceinline__ uint32_t point_word(const FrameArgs &a, float x, float y, float z, uint32_t &bit) {
    int32_t v[3];
    float g[3];
    const int32_t n[3] = {a.g.nx, a.g.ny, a.g.nz};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        g[k] = __fadd_rn(__fmul_rn(a.T.R[k * 3 + 0], x), __fmul_rn(a.T.R[k * 3 + 1], y));
        g[k] = __fadd_rn(g[k], __fmul_rn(a.T.R[k * 3 + 2], z));
        g[k] = __fadd_rn(g[k], a.T.t[k]);
    }
    if (a.rvs != 0.0f && fminf(fabsf(g[0]), fminf(fabsf(g[1]), fabsf(g[2]))) >= 1e-18f) {
#pragma unroll
        for (int k = 0; k < 3; ++k) g[k] = div_by(g[k], a.vs, a.rvs);
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) g[k] = __fdiv_rn(g[k], a.vs);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (!(g[k] >= 0.0f && g[k] < (float)n[k])) return kNoWord;
        v[k] = __float2int_rd(g[k]);
    }
    bit = 1u << (v[0] & 31);
    return (uint32_t)plane_word(a.g, v[0], v[1], v[2]);
}

__device__ __forceinline__ uint32_t pixel_word(const FrameArgs &a, float d, int32_t u, int32_t v, uint32_t &bit) {
    if (!(isfinite(d) && d > 0.0f && d <= a.depth_max)) return kNoWord;
    float xc = __fmul_rn(__fsub_rn((float)u, a.cx), d), yc = __fmul_rn(__fsub_rn((float)v, a.cy), d);
    // u - cx is 0 or at least a half, so the products are 0 or no smaller than d / 2
    if (a.rfx != 0.0f && a.rfy != 0.0f && d >= 1e-9f && d <= 1e9f) {
        xc = div_by(xc, a.fx, a.rfx);
        yc = div_by(yc, a.fy, a.rfy);
    } else {
        xc = __fdiv_rn(xc, a.fx);
        yc = __fdiv_rn(yc, a.fy);
    }
    return point_word(a, xc, yc, d, bit);
}

// ORs `bit` into plane[key] for every lane, with one atomicOr per run of
// consecutive lanes that share a word: an inclusive OR-scan over lanes that
// only pulls from lanes with the same key, after which the last lane of each
// run holds the run's bits.  Lanes whose keys match but are not adjacent may
// fold bits into each other; that is harmless, they name the same word.
// Every lane of the warp must call this (keys of idle lanes are kNoWord).
__device__ __forceinline__ void warp_set_bits(uint32_t *plane, uint32_t key, uint32_t bit) {
    const int lane = threadIdx.x & 31;
    uint32_t v = bit;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t kd = __shfl_up_sync(kFull, key, d);
        const uint32_t vd = __shfl_up_sync(kFull, v, d);
        if (lane >= d && kd == key) v |= vd;
    }
    const uint32_t knext = __shfl_down_sync(kFull, key, 1);
    if (key != kNoWord && (lane == 31 || knext != key)) atomicOr(plane + key, v);
}

// Adds the warp's number of in-grid points to the stats counter.  Every lane
// of the warp must call this.
__device__ __forceinline__ void count_points(const FrameArgs &a, unsigned kept) {
    if (!a.stats) return;
    const unsigned total = __reduce_add_sync(kFull, kept);
    if ((threadIdx.x & 31) == 0 && total) atomicAdd(a.stats + 1, (unsigned long long)total);
}

// A tile's words in shared memory: an open-addressed table from plane words
// to the bits to set there.
constexpr int kTabBits = 8, kTabSlots = 1 << kTabBits, kTabProbes = 4;
struct WordTab {
    uint32_t key[kTabSlots], bits[kTabSlots];
};

// 256 threads; the caller places the barriers.
__device__ __forceinline__ void tab_clear(WordTab &tab) {
    for (int i = threadIdx.x; i < kTabSlots; i += 256) {
        tab.key[i] = kNoWord;
        tab.bits[i] = 0;
    }
}

// Sets bits of a word in the table, or in the plane where its slots are taken.
__device__ __forceinline__ void tab_set(WordTab &tab, uint32_t *plane, uint32_t key, uint32_t bit) {
    uint32_t h = (key * 2654435769u) >> (32 - kTabBits);   // Knuth's multiplicative hashing
    for (int p = 0; p < kTabProbes; ++p) {
        uint32_t k = *reinterpret_cast<volatile uint32_t *>(&tab.key[h]);
        if (k == kNoWord) {
            k = atomicCAS(&tab.key[h], kNoWord, key);
            if (k == kNoWord) k = key;
        }
        if (k == key) {
            if (bit & ~*reinterpret_cast<volatile uint32_t *>(&tab.bits[h])) atomicOr(&tab.bits[h], bit);
            return;
        }
        h = (h + 1) & (kTabSlots - 1);
    }
    atomicOr(plane + key, bit);
}

// Sets the table's words in the plane and leaves it clear.
__device__ __forceinline__ void tab_flush(WordTab &tab, uint32_t *plane) {
    for (int i = threadIdx.x; i < kTabSlots; i += 256) {
        const uint32_t k = tab.key[i];
        if (k == kNoWord) continue;
        atomicOr(plane + k, tab.bits[i]);
        tab.key[i] = kNoWord;
        tab.bits[i] = 0;
    }
}

// The image in tiles of kTileW x kTileH pixels, four of a row to a thread, or
// (FrameArgs::linear) of kTilePixels pixels as they lie in memory.
constexpr int kTileW = 32, kTileH = 32, kTileLanes = kTileW / 4, kTilePixels = kTileW * kTileH;
static_assert(kTileLanes * kTileH == 256, "a thread per four pixels");
__host__ __device__ inline int32_t pixel_tiles_x(int32_t W) { return (W - 1) / kTileW + 1; }
__host__ __device__ inline int32_t pixel_tiles(const FrameArgs &a) {
    if (a.linear) return (int32_t)(((int64_t)a.W * a.H - 1) / kTilePixels + 1);
    return pixel_tiles_x(a.W) * ((a.H - 1) / kTileH + 1);
}

// Whether every whole four of the image's pixels can be loaded at once.
__host__ __device__ inline bool pixels_aligned(const void *depth, int bytes) {
    return reinterpret_cast<uintptr_t>(depth) % (4u * (unsigned)bytes) == 0;
}

// How K1 takes an image's pixels: in tiles one by one, in tiles by fours, or
// (kPixLinear) as they lie, by fours where the image's address allows it.
enum { kPixTile = 0, kPixTile4 = 1, kPixLinear = 2 };
__host__ __device__ inline int pixel_mode(const FrameArgs &a, int bytes) {
    if (a.linear) return kPixLinear;
    return a.W % 4 == 0 && pixels_aligned(a.depth, bytes) ? kPixTile4 : kPixTile;
}

// Four pixels at once.
template <int DT>
__device__ __forceinline__ void load_four(const FrameArgs &a, uint32_t p0, float d[4]) {
    if (DT == 0) {
        const float4 q = reinterpret_cast<const float4 *>(a.depth)[p0 >> 2];
        d[0] = q.x; d[1] = q.y; d[2] = q.z; d[3] = q.w;
    } else {
        const ushort4 q = reinterpret_cast<const ushort4 *>(a.depth)[p0 >> 2];
        d[0] = __fmul_rn((float)q.x, a.scale);
        d[1] = __fmul_rn((float)q.y, a.scale);
        d[2] = __fmul_rn((float)q.z, a.scale);
        d[3] = __fmul_rn((float)q.w, a.scale);
    }
}

// One pixel.
template <int DT>
__device__ __forceinline__ float load_one(const FrameArgs &a, uint32_t p) {
    if (DT == 0) return reinterpret_cast<const float *>(a.depth)[p];
    return __fmul_rn((float)reinterpret_cast<const uint16_t *>(a.depth)[p], a.scale);
}

// The depths of the thread's pixels u .. u+3 of row v of a tile (0 outside
// the image), or of the four from (u, v) on of a linear one.  DT: 0 = f32, 1 =
// u16.  MODE: pixel_mode.
template <int DT, int MODE>
__device__ __forceinline__ void load_depths(const FrameArgs &a, int32_t tile, int32_t &u, int32_t &v, float d[4]) {
    if (MODE == kPixLinear) {
        const uint32_t p = (uint32_t)tile * (uint32_t)kTilePixels + threadIdx.x * 4u, n = (uint32_t)a.W * (uint32_t)a.H;
        v = (int32_t)(p / (uint32_t)a.W);
        u = (int32_t)(p - (uint32_t)v * (uint32_t)a.W);
        if (p + 4u <= n && pixels_aligned(a.depth, DT == 0 ? 4 : 2)) {
            load_four<DT>(a, p, d);
            return;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) d[j] = p + j < n ? load_one<DT>(a, p + j) : 0.0f;
        return;
    }
    const int32_t tx = pixel_tiles_x(a.W), ty = tile / tx;
    u = (tile - ty * tx) * kTileW + (int32_t)(threadIdx.x % kTileLanes) * 4;
    v = ty * kTileH + (int32_t)(threadIdx.x / kTileLanes);
    const uint32_t p0 = (uint32_t)v * (uint32_t)a.W + (uint32_t)u;   // images hold fewer than 2^31 pixels
#pragma unroll
    for (int j = 0; j < 4; ++j) d[j] = 0.0f;
    if (v >= a.H) return;
    if (MODE == kPixTile4) {
        if (u < a.W) load_four<DT>(a, p0, d);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (u + j < a.W) d[j] = load_one<DT>(a, p0 + j);
    }
}

// Sets the thread's pixels, of depths d (outside the image: 0, which sets
// nothing), in the table.  LIN: they go on in the next row.  Warp-synchronous.
template <bool LIN>
__device__ __forceinline__ void voxelize_depths(const FrameArgs &a, int32_t u, int32_t v, const float d[4], WordTab &tab) {
    uint32_t key[4], bit[4];
    unsigned kept = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        bit[j] = 0;
        key[j] = pixel_word(a, d[j], LIN ? u : u + j, v, bit[j]);
        kept += (key[j] != kNoWord);
        if (LIN && ++u == a.W) {
            u = 0;
            ++v;
        }
    }
    // neighbouring pixels often share a word: once for a run of the thread's
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (key[j] == kNoWord) continue;
        if (j < 3 && key[j] == key[j < 3 ? j + 1 : 3]) {
            bit[j < 3 ? j + 1 : 3] |= bit[j];
            continue;
        }
        tab_set(tab, a.pl.occ_raw, key[j], bit[j]);
    }
    count_points(a, kept);
}

// One tile.  CTA-cooperative (256 threads).
template <int DT, int MODE>
__device__ __forceinline__ void voxelize_tile(const FrameArgs &a, int32_t tile, WordTab &tab) {
    float d[4];
    int32_t u, v;
    load_depths<DT, MODE>(a, tile, u, v, d);
    tab_clear(tab);
    __syncthreads();
    voxelize_depths<MODE == kPixLinear>(a, u, v, d, tab);
    __syncthreads();
    tab_flush(tab, a.pl.occ_raw);
}

// `tiles` tiles from `tile` on, each one's depths loaded while the one before
// is placed; finds the table clear and leaves it so.  CTA-cooperative.
template <int DT, int MODE>
__device__ __forceinline__ void voxelize_run(const FrameArgs &a, int32_t tile, int32_t tiles, WordTab &tab) {
    float d[4], next[4];
    int32_t u, v, un, vn;
    load_depths<DT, MODE>(a, tile, un, vn, next);
    for (int32_t k = 0; k < tiles; ++k) {
#pragma unroll
        for (int j = 0; j < 4; ++j) d[j] = next[j];
        u = un;
        v = vn;
        if (k + 1 < tiles) load_depths<DT, MODE>(a, tile + k + 1, un, vn, next);
        voxelize_depths<MODE == kPixLinear>(a, u, v, d, tab);
        __syncthreads();
        tab_flush(tab, a.pl.occ_raw);
        __syncthreads();
    }
}

// The word and bit of point i of the cloud (kNoWord past its end).
__device__ __forceinline__ uint32_t point_of_cloud(const FrameArgs &a, int64_t i, uint32_t &bit) {
    if (i >= a.npts) return kNoWord;
    const float x = a.xyz[3 * i + 0];
    const float y = a.xyz[3 * i + 1];
    const float z = a.xyz[3 * i + 2];
    if (!(isfinite(x) && isfinite(y) && isfinite(z))) return kNoWord;
    return point_word(a, x, y, z, bit);
}

// Point i of the cloud.  Warp-synchronous: every lane of the warp calls it.
__device__ __forceinline__ void voxelize_points_thread(const FrameArgs &a, int64_t i) {
    uint32_t bit = 0;
    const uint32_t key = point_of_cloud(a, i, bit);
    warp_set_bits(a.pl.occ_raw, key, bit);
    count_points(a, key != kNoWord);
}

// ---------------------------------------------------------------------------
// K2: inflation (Sec. IV-B, Alg. 1, the three nested loops around each
// point).  Stamping the cube of half side r around every occupied voxel is
// the Chebyshev dilation of occ_raw, which separates into three 1-D OR
// filters of width 2r+1 along x, y and z.  Clipping at the grid faces falls
// out of the zero fill outside the grid.
//
// One CTA produces a TXW x TY x TZ tile of 32-bit plane words.  It stages
// the tile plus its halo (one word each side in x, r rows in y, r slices in
// z) in shared memory, then runs the x pass (funnel shifts across word
// boundaries), the y pass and the z pass in shared memory and writes the
// tile of occ_inf once.  Bits beyond Nx are cleared so the plane's padding
// stays zero.  R > 0 is a compile-time radius (all index arithmetic folds);
// R == 0 takes the radius r_rt at run time.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t dilate_x(uint32_t prev, uint32_t cur, uint32_t next, int r) {
    uint32_t acc = cur;
#pragma unroll 4
    for (int d = 1; d <= r; ++d) {
        acc |= __funnelshift_r(cur, next, d);   // voxel x+d -> x
        acc |= __funnelshift_l(prev, cur, d);   // voxel x-d -> x
    }
    return acc;
}

template <int R, int TXW, int TY, int TZ>
__host__ __device__ constexpr size_t inflate_smem_words(int r) {
    return (size_t)(TZ + 2 * r) * (TY + 2 * r) * (TXW + 2) + (size_t)(TZ + 2 * r) * (TY + 2 * r) * TXW;
}

// The x, y and z passes of a tile whose raw words are staged in shared
// memory: word w0 - 1 + lx of row y0 - r + ly, slice z0 - r + lz at
// st[(lz * hy + ly) * sx + ox + lx], lx in [0, TXW + 2), with zeros outside
// the grid.  buf1 (hz * hy * TXW words) must not overlap the staged words;
// the y pass reuses the staged words' memory.  CTA-cooperative (256
// threads); ends with a barrier.  R > 0 is the radius, known to the compiler
// (1 to 3); R == 0 takes r_rt (4 or more).
template <int R, int TXW, int TY, int TZ>
__device__ __forceinline__ void inflate_passes(const PlaneGeom &g, uint32_t *out, const int r_rt, int tile_x,
                                               int tile_y, int tile_z, uint32_t *st, int sx, int ox, uint32_t *buf1) {
    const int r = R > 0 ? R : r_rt;
    const int hy = TY + 2 * r, hz = TZ + 2 * r;
    const int w0 = tile_x * TXW, y0 = tile_y * TY, z0 = tile_z * TZ;

    // x pass, clearing bits past the end of the row
    const int n1 = hz * hy * TXW;
    for (int i = threadIdx.x; i < n1; i += 256) {
        const int lx = i % TXW, row = i / TXW;
        const uint32_t *b = st + row * sx + ox + lx;
        uint32_t v = dilate_x(b[0], b[1], b[2], r);
        const int valid = g.nx - 32 * (w0 + lx);
        if (valid < 32) v &= valid > 0 ? ((1u << valid) - 1u) : 0u;
        buf1[i] = v;
    }
    __syncthreads();

    uint32_t *buf2 = st;
    if (R == 0) {
        // a radius of 4 to 15, at run time.  A window of 2r + 1 rows costs as
        // many loads an output, so threads share them: the TY (8) outputs of a
        // column have rows 7 .. 2r in common, and the rest is running ORs from
        // either end (2r + 8 loads for 8 outputs); in z two outputs share
        // all rows but one each.
        for (int i = threadIdx.x; i < hz * TXW; i += 256) {
            const uint32_t *b = buf1 + (i / TXW) * hy * TXW + i % TXW;
            uint32_t low[TY], mid = 0, up = 0;   // low[y]: rows y .. 6
            low[TY - 1] = 0;
#pragma unroll
            for (int y = TY - 2; y >= 0; --y) low[y] = low[y + 1] | b[y * TXW];
#pragma unroll 4
            for (int y = TY - 1; y <= 2 * r; ++y) mid |= b[y * TXW];
            uint32_t *o = buf2 + (i / TXW) * TY * TXW + i % TXW;
#pragma unroll
            for (int y = 0; y < TY; ++y) {
                if (y) up |= b[(2 * r + y) * TXW];
                o[y * TXW] = low[y] | mid | up;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < TZ / 2 * TY * TXW; i += 256) {
            const int c = i % (TY * TXW), lz = i / (TY * TXW) * 2, lx = c % TXW;
            const uint32_t *b = buf2 + lz * TY * TXW + c;
            uint32_t mid = 0;
#pragma unroll 4
            for (int d = 1; d <= 2 * r; ++d) mid |= b[d * TY * TXW];
            const int w = w0 + lx, y = y0 + c / TXW, z = z0 + lz;
            if (w >= g.wx || y >= g.ny) continue;
            if (z < g.nz) out[((int64_t)z * g.ny + y) * g.wx + w] = mid | b[0];
            if (z + 1 < g.nz) out[((int64_t)(z + 1) * g.ny + y) * g.wx + w] = mid | b[(2 * r + 1) * TY * TXW];
        }
        __syncthreads();   // the tile's shared memory may be reused right away
        return;
    }

    // y pass into the staged words' memory (now free): hz * TY * TXW
    const int n2 = hz * TY * TXW;
    for (int i = threadIdx.x; i < n2; i += 256) {
        const int lx = i % TXW, rest = i / TXW, ly = rest % TY, lz = rest / TY;
        const uint32_t *b = buf1 + (lz * hy + ly) * TXW + lx;
        uint32_t v = 0;
        for (int d = 0; d <= 2 * r; ++d) v |= b[d * TXW];
        buf2[i] = v;
    }
    __syncthreads();

    // z pass to global
    constexpr int n3 = TZ * TY * TXW;
    for (int i = threadIdx.x; i < n3; i += 256) {
        const int lx = i % TXW, rest = i / TXW, ly = rest % TY, lz = rest / TY;
        const int w = w0 + lx, y = y0 + ly, z = z0 + lz;
        if (w >= g.wx || y >= g.ny || z >= g.nz) continue;
        const uint32_t *b = buf2 + (lz * TY + ly) * TXW + lx;
        uint32_t v = 0;
        for (int d = 0; d <= 2 * r; ++d) v |= b[d * TY * TXW];
        out[((int64_t)z * g.ny + y) * g.wx + w] = v;
    }
    __syncthreads();   // the tile's shared memory may be reused right away
}

// CTA-cooperative: every thread of the (256-thread) CTA must call this.
// The threads stage the tile's raw words with halo themselves.
template <int R, int TXW, int TY, int TZ, class L>
__device__ __forceinline__ void inflate_tile(const PlaneGeom &g, const uint32_t *raw, uint32_t *out, const int r_rt,
                                             int tile_x, int tile_y, int tile_z, uint32_t *sm) {
    const int r = R > 0 ? R : r_rt;
    const int hx = TXW + 2, hy = TY + 2 * r, hz = TZ + 2 * r;
    uint32_t *buf0 = sm;                          // hz * hy * hx: raw with halo
    uint32_t *buf1 = sm + hz * hy * hx;           // hz * hy * TXW: x-dilated
    const int w0 = tile_x * TXW, y0 = tile_y * TY, z0 = tile_z * TZ;

    // stage raw words (zero outside the grid)
    const int n0 = hz * hy * hx;
#pragma unroll 8
    for (int i = threadIdx.x; i < n0; i += 256) {
        const int lx = i % hx, rest = i / hx, ly = rest % hy, lz = rest / hy;
        const int w = w0 + lx - 1, y = y0 + ly - r, z = z0 + lz - r;
        uint32_t v = 0;
        if (w >= 0 && w < g.wx && y >= 0 && y < g.ny && z >= 0 && z < g.nz)
            v = L::ld(raw + ((int64_t)z * g.ny + y) * g.wx + w);
        buf0[i] = v;
    }
    __syncthreads();
    inflate_passes<R, TXW, TY, TZ>(g, out, r_rt, tile_x, tile_y, tile_z, buf0, hx, 0, buf1);
}

// Starts the copies that stage a tile of radius R (zeros outside the grid):
// one commit group of this thread's, to be waited for.  They may go through
// the L1, so nothing on this SM may have read an older state of the plane in
// this launch.  CTA-cooperative.
template <int R, int TXW, int TY, int TZ>
__device__ __forceinline__ void inflate_stage(const PlaneGeom &g, const uint32_t *raw, int tile_x, int tile_y, int tile_z,
                                              uint32_t *st) {
    constexpr int hx = TXW + 2, hy = TY + 2 * R, hz = TZ + 2 * R;
    const int w0 = tile_x * TXW, y0 = tile_y * TY, z0 = tile_z * TZ;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(st);
    for (int i = threadIdx.x; i < hz * hy * hx; i += 256) {
        const int lx = i % hx, rest = i / hx, ly = rest % hy, lz = rest / hy;
        const int w = w0 + lx - 1, y = y0 + ly - R, z = z0 + lz - R;
        const bool in = (unsigned)w < (unsigned)g.wx && (unsigned)y < (unsigned)g.ny && (unsigned)z < (unsigned)g.nz;
        const uint32_t *src = in ? raw + ((int64_t)z * g.ny + y) * g.wx + w : raw;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4u * i), "l"(src), "r"(in ? 4 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// ---------------------------------------------------------------------------
// K4: merge the measurement grid into loc_grid (Sec. IV-D, Alg. 3).
//
// One 32-voxel plane word per thread.  The voxel's measurement state is
// resolved from the three planes with precedence
//   occupied (occ_inf) > free (fr) > unknown-and-traced (tr) > unknown,
// and Alg. 3 writes it to loc_grid wherever it is not unknown.  loc_grid is
// ring-addressed (Ring): a re-centre only moves the ring, and the voxels it
// brings into the grid are set to unknown by the next merge.  A word with no
// bit set in any plane and no voxel brought in touches neither loc_grid nor
// the planes, so the pass reads the bit planes everywhere but writes
// loc_grid only inside the measured frustum and the slabs a re-centre
// brought in, and never reads it.  Every plane word read non-zero is
// cleared, which leaves all planes zero for the next frame (occ_raw is a
// subset of occ_inf, so its non-zero words are cleared too).
// ---------------------------------------------------------------------------
// RAYS_LAST: the literal loc_grid reading, in which the rays' marks replace
// the measurement's occupied marks (free > traced > occupied).
//
// The resolve works on four voxels at once.  With the state codes
// OCC = 2, FREE = 1, TRACED = 3, a word's codes are two bit masks, hi (bit
// 1 of each code: occupied or traced) and lo (bit 0: free or traced), and
// known marks the voxels that are not unknown.  expand4 spreads a nibble
// into one 0/1 byte per bit (bit i times 2^(7i) lands on bit 8i; no other
// product of the multiply lands on a byte's low bit).  merge4 then writes
// the codes of voxels 4m..4m+3 over the four old bytes where known.
__device__ __forceinline__ uint32_t expand4(uint32_t nib) { return (nib * 0x00204081u) & 0x01010101u; }

template <bool RAYS_LAST = false>
__device__ __forceinline__ void code_masks(uint32_t oc, uint32_t f, uint32_t t, uint32_t &hi, uint32_t &lo,
                                           uint32_t &known) {
    uint32_t occ, fr, tr;
    if (!RAYS_LAST) {
        occ = oc;
        fr = f & ~oc;
        tr = t & ~(f | oc);
    } else {
        fr = f;
        tr = t & ~f;
        occ = oc & ~(f | t);
    }
    hi = occ | tr;
    lo = fr | tr;
    known = occ | fr | tr;
}

__device__ __forceinline__ uint32_t merge4(uint32_t hi, uint32_t lo, uint32_t known, int m, uint32_t old) {
    const int s = 4 * m;
    const uint32_t kb = expand4((known >> s) & 15u);
    const uint32_t code = (expand4((hi >> s) & 15u) << 1) | expand4((lo >> s) & 15u);
    return (old & ~(kb * 0xffu)) | code;
}

// The ring position of coordinate c (0 <= c < n) moved by r (0 <= r < n).
__device__ __forceinline__ int32_t ring_at(int32_t c, int32_t r, int32_t n) {
    const int32_t v = c + r;
    return v >= n ? v - n : v;
}

// Bits of the voxels of a row word (x0 .. x0 + nbits - 1, row (y, z)) that a
// re-centre brought into the grid: the whole word if its row did, else the
// part of it inside [elo[0], ehi[0]).
__device__ __forceinline__ uint32_t entering_bits(const Ring &R, int32_t x0, int32_t y, int32_t z, int nbits) {
    const uint32_t all = nbits >= 32 ? 0xffffffffu : ((1u << nbits) - 1u);
    if ((y >= R.elo[1] && y < R.ehi[1]) || (z >= R.elo[2] && z < R.ehi[2])) return all;
    const int32_t lo = max(R.elo[0] - x0, 0), hi = min(R.ehi[0] - x0, nbits);
    if (hi <= lo) return 0u;
    const uint32_t below_hi = hi >= 32 ? 0xffffffffu : ((1u << hi) - 1u);
    return below_hi & ~((1u << lo) - 1u);
}

// Writes codes[v] (byte v of the 8 words codes[0..7], codes[8] = 0) to
// p[v - v0] for the voxels v in [v0, v1) whose bit is set in touch: aligned
// 4-byte stores where all four bytes are this word's and touched, byte
// stores elsewhere, so that no store reaches a byte of another word.
__device__ __forceinline__ void store_codes(uint8_t *p, int v0, int v1, const uint32_t codes[9], uint32_t touch) {
    int v = v0;
    // head: bytes up to the first 4-byte boundary of the buffer
    while (v < v1 && (reinterpret_cast<uintptr_t>(p + (v - v0)) & 3u) != 0) {
        if ((touch >> v) & 1u) p[v - v0] = (uint8_t)(codes[v >> 2] >> (8 * (v & 3)));
        ++v;
    }
    for (; v + 4 <= v1; v += 4) {
        const uint32_t t4 = (touch >> v) & 15u;
        if (t4 == 0) continue;
        const uint32_t w = __funnelshift_r(codes[v >> 2], codes[(v >> 2) + 1], 8 * (v & 3));
        if (t4 == 15u) {
            *reinterpret_cast<uint32_t *>(p + (v - v0)) = w;
        } else {
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if ((t4 >> b) & 1u) p[v - v0 + b] = (uint8_t)(w >> (8 * b));
        }
    }
    for (; v < v1; ++v)
        if ((touch >> v) & 1u) p[v - v0] = (uint8_t)(codes[v >> 2] >> (8 * (v & 3)));
}

// K4 of one plane word w (the 32 voxels x0 .. x0 + 31 of one row of the
// grid in its own frame) into the ring-addressed loc: the measurement's
// codes where a plane marks a voxel, unknown where a re-centre brought the
// voxel in and no plane marks it, nothing elsewhere.  loc is only written,
// never read.  The row's voxels from x0 on sit at buffer x ring_at(x0, r[0])
// up to the row's end, the rest (when the ring wraps inside the word) from
// buffer x 0.  Clears the plane words it reads non-zero.
template <class L, bool RAYS_LAST = false>
__device__ __forceinline__ void merge_word(const PlaneGeom &g, const Planes &pl, uint8_t *loc, const Ring &R,
                                           int64_t w) {
    if (w >= g.words) return;
    // rows are a power of two of words; grids hold fewer than 2^31 voxels
    const int32_t wxi = (int32_t)(w & (g.wx - 1));
    const uint32_t row = (uint32_t)(w >> (__ffs(g.wx) - 1));
    const int32_t x0 = wxi * 32;
    if (x0 >= g.nx) return;   // padding word, always zero
    const uint32_t oc = L::ld(pl.occ_inf + w), f = L::ld(pl.fr + w), t = L::ld(pl.tr + w);
    const uint32_t any = oc | f | t;
    const int32_t y = (int32_t)(row % (uint32_t)g.ny), z = (int32_t)(row / (uint32_t)g.ny);
    const int nbits = min(32, g.nx - x0);
    const uint32_t ent = entering_bits(R, x0, y, z, nbits);
    if ((any | ent) == 0) return;
    uint32_t codes[9];
    codes[8] = 0;
    uint32_t touch = ent;
    if (any) {
        uint32_t hi, lo, known;
        code_masks<RAYS_LAST>(oc, f, t, hi, lo, known);
#pragma unroll
        for (int m = 0; m < 8; ++m) codes[m] = merge4(hi, lo, known, m, 0u);
        touch |= known;
    } else {
#pragma unroll
        for (int m = 0; m < 8; ++m) codes[m] = 0u;
    }
    uint8_t *rowp = loc + ((int64_t)ring_at(z, R.r[2], g.nz) * g.ny + ring_at(y, R.r[1], g.ny)) * g.nx;
    const int32_t xb = ring_at(x0, R.r[0], g.nx);
    const int n1 = min(nbits, g.nx - xb);
    store_codes(rowp + xb, 0, n1, codes, touch);
    if (n1 < nbits) store_codes(rowp, n1, nbits, codes, touch);   // voxel v at rowp[v - n1]
    if (oc) {
        pl.occ_inf[w] = 0;
        pl.occ_raw[w] = 0;
    }
    if (f) pl.fr[w] = 0;
    if (t) pl.tr[w] = 0;
}

// ---------------------------------------------------------------------------
// K5: loc_grid in its own frame (Sec. IV-E), out of the ring-addressed
// buffer: voxel (x, y, z) is the buffer's byte at the ring position of
// (x, y, z), or unknown where a re-centre brought the voxel in.  One 16-byte
// chunk of the output per call; dst is 16-byte aligned.
//
// A chunk is put together from runs: voxels of one row that lie contiguously
// in the buffer and are all old or all new.  Each run is read with as many
// bytes before it as the chunk already holds (five aligned words and funnel
// shifts), and replaces the chunk from its first byte on.  Of the 12.5
// chunks of a 200-voxel row two or three have more than one run (the row's
// end, the ring's wrap), so nearly every warp takes two or three rounds, where
// it used to walk such chunks byte by byte with one lane in ten: 200 x 200 x
// 100 voxels 10.0 -> 7.2 us, 400 x 400 x 120 23 -> 12, 500 x 500 x 150 42 -> 24
// (ncu; the instructions 4.0 -> 2.5, 18 -> 8, 37 -> 20 M).  The reads
// reach up to 15 bytes before the buffer and 19 past a run's start: the host
// leaves room on both sides.
//
// NARROW: voxel by voxel, for rows of which a chunk holds four or more.  By
// runs, rows of 1, 2, 3, 4 and 5 voxels (4 M in all) take 16.1, 14.0, 12.2, 8.0
// and 8.6 us, voxel by voxel 8.3, 6.8, 8.7, 6.0 and about 9.3.
// ---------------------------------------------------------------------------
constexpr int32_t kNarrowRow = 4;

template <class L, bool NARROW>
__device__ __forceinline__ void shift_chunk(const PlaneGeom &g, const Ring &R, const uint8_t *src, uint8_t *dst,
                                            int64_t chunk) {
    const int64_t i0 = chunk * 16;
    if (i0 >= g.nvox) return;
    // grids hold fewer than 2^31 voxels: 32-bit division
    const uint32_t yz = (uint32_t)i0 / (uint32_t)g.nx;
    int32_t x = (int32_t)((uint32_t)i0 - yz * (uint32_t)g.nx);
    int32_t z = (int32_t)(yz / (uint32_t)g.ny), y = (int32_t)(yz - (uint32_t)z * (uint32_t)g.ny);
    int32_t xr = ring_at(x, R.r[0], g.nx);
    const int32_t size = (int32_t)min((int64_t)16, g.nvox - i0);
    // the row's first byte in the buffer, and whether its voxels are old
    auto row_of = [&](bool &old) {
        old = !((y >= R.elo[1] && y < R.ehi[1]) || (z >= R.elo[2] && z < R.ehi[2]));
        return (ring_at(z, R.r[2], g.nz) * g.ny + ring_at(y, R.r[1], g.ny)) * g.nx;
    };
    // the run from (x, xr) on: its length, and 16 bytes that hold it from
    // byte `filled` on
    auto run = [&](int32_t row, bool old, int32_t filled, uint32_t w[4]) {
        int32_t len = min(g.nx - x, g.nx - xr);
        if (x < R.elo[0]) {
            len = min(len, R.elo[0] - x);
        } else if (x < R.ehi[0]) {
            len = min(len, R.ehi[0] - x);
            old = false;
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) w[m] = 0;
        if (old) {
            const int32_t sb = row + xr - filled;
            const uint32_t *from = reinterpret_cast<const uint32_t *>(src + (sb & ~3));
            uint32_t v[5];
#pragma unroll
            for (int m = 0; m < 5; ++m) v[m] = L::ld(from + m);
#pragma unroll
            for (int m = 0; m < 4; ++m) w[m] = __funnelshift_r(v[m], v[m + 1], (sb & 3) * 8);
        }
        return len;
    };
    uint32_t o[4];
    bool old;
    int32_t row = row_of(old);
    if (NARROW) {
#pragma unroll
        for (int m = 0; m < 4; ++m) o[m] = 0;
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            if (b < size && old && !(x >= R.elo[0] && x < R.ehi[0]))
                o[b >> 2] |= (uint32_t)L::ld(src + row + xr) << (8 * (b & 3));
            if (++xr == g.nx) xr = 0;
            if (++x == g.nx) {
                x = 0;
                xr = R.r[0];
                if (++y == g.ny) {
                    y = 0;
                    if (++z == g.nz) z = 0;   // past the end, where nothing is read
                }
                row = row_of(old);
            }
        }
    }
    int32_t len = NARROW ? size : run(row, old, 0, o), filled = len;
    while (filled < size) {
        x += len;
        xr += len;
        if (xr == g.nx) xr = 0;
        if (x == g.nx) {
            x = 0;
            xr = R.r[0];
            if (++y == g.ny) { y = 0; ++z; }
            row = row_of(old);
        }
        uint32_t w[4];
        len = run(row, old, filled, w);
#pragma unroll
        for (int m = 0; m < 4; ++m) {   // bytes `filled` and on
            const uint32_t mask = __funnelshift_lc(0u, 0xffffffffu, max(8 * filled - 32 * m, 0));
            o[m] = (o[m] & ~mask) | (w[m] & mask);
        }
        filled += len;
    }
    if (size == 16) {
        *reinterpret_cast<uint4 *>(dst + i0) = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
        for (int b = 0; b < size; ++b) dst[i0 + b] = (uint8_t)(o[b >> 2] >> (8 * (b & 3)));
    }
}

}  // namespace units
}  // namespace vg
