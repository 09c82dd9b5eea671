// k_batch.cu -- many measurements in one persistent, fused launch.
//
// One cooperative launch of k_batch runs, for every frame of a batch (each
// with its own grid, resolution, voxel size and radius), the whole path:
//   phase 1  K1 voxelize           tiles of 32 x 32 pixels; 256 rays of the table
//   phase 2  K2 inflate            8 (or 4) words x 8 rows x 8 (or 4)
//                                  slices (radius 1..3) of the frame's box
//   phase 3  K3 gathered           256 rays around the camera; 256 words
//            K3 scattered          groups of at most 256 / LPR rays (a
//                                  frame's rays spread over its units)
//   phase 3b K3 gathered           32 x 8 rays (their latest hits)
//   phase 4  K4 gathered           192 plane words of the box; 256 of slabs
//            K4 merge              512 plane words (256 if tuned)
// with a grid-wide barrier between phases (3b only if a frame is gathered; a
// batch without gathered frames takes a kernel without their phases).
// A batch whose frames that the gathered form can take (vg_gather.cuh) hold
// enough voxels together (kBatchGatherVoxels) has them gathered: many frames
// fill the device, so its fewer instructions count and the latency of its
// phases does not.  A frame's re-centre (K5) is not
// a phase: it moves its grid's ring, and that grid's next merge sets the
// voxels it brought in to unknown (Ring).
// Units of every frame are laid end to end per phase (BatchItem::off).  A
// CTA finds the frame of its first unit of a phase by binary search, steps
// forward through the frames as its units advance (see run_begin), and runs
// the same device code as the one-step kernels (vg_units.cuh, vg_rt.cuh).
// Reads of data an earlier phase wrote: the walked frames' merge skips the L1
// (LoadL2).  The inflation's and the rays' loads go through it, and the
// gathered phases' (hits, 1/D with the latest hits, tiles, near words), which
// loaded some of those lines before they were written: that they see the new
// state rests on the barrier's fences (vg_sync.cuh).
//
// With 32 warps to an SM the phases are bound by latency more than by issue
// (313 M warp instructions in 529 us, 54 % of the issue slots, for 64
// robots), so loads run ahead (the next unit's depths in phase 1, the next
// tile in phase 2) and the gathered units, whose cost differs most, are
// handed out as CTAs come free: phase 1 97 -> 88 us, phase 2 60 -> 55, and
// four steps with a read of every grid 2413 -> 2257 us (in turn: 2351); 192
// words a phase-4 unit instead of 128 gave 2138.
//
// The barrier waits with a deadline (BatchCtl::bar_ns, four seconds unless
// tuned): if the other CTAs do not all arrive in time, the waiting CTA sets
// BatchCtl::error and every CTA leaves the kernel, so the host sees
// VG_ETIMEOUT instead of a hung GPU.  The launch is cooperative, so all CTAs are resident together.
#include "vg_gather.cuh"
#include "vg_rt.cuh"
#include "vg_sync.cuh"

#include <type_traits>

namespace vg {
namespace {

using namespace rt;

// the scattered rays' buffers need kRtBuf columns, a gathered unit's lists a
// little more; four CTAs of this fit an SM
constexpr int kDynWords = 40 * kThreads;
static_assert(kDynWords >= kRtBuf * kThreads, "ray buffers fit");
// an inflate tile's staged words, twice, and its x pass
constexpr int kStageWords = 14 * 14 * 10;
static_assert(2 * kStageWords + 14 * 14 * 8 <= kDynWords, "inflate tiles of radius <= 3 fit");
constexpr int kGatherWords = kBatchGatherWords;
static_assert(sizeof(gather::GatherSmem<kGatherWords>) <= kDynWords * 4, "gathered words fit");
static_assert(sizeof(gather::SkinSmem) <= kDynWords * 4 && sizeof(gather::LateSmem) <= kDynWords * 4 &&
              3 * kNearWords <= kDynWords, "gathered K3 fits");
static_assert(sizeof(FrameArgs) % 4 == 0, "frame arguments copy as words");
static_assert(sizeof(BatchItem) <= 1024, "the served form's bound on a launch table");

__device__ __forceinline__ int find_item(const BatchItem *items, int n, int phase, int64_t u) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {   // last item whose offset is <= u
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&items[mid].off[phase]) <= u) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The first phase-3 unit whose weighted start (woff3 + its index in its
// frame x w3) is at least x, for 0 <= x <= ctl->wtotal3.
__device__ __forceinline__ int64_t weighted_unit(const BatchItem *items, int n, int64_t total, int64_t x) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {   // last item whose weighted offset is <= x
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&items[mid].woff3) <= x) lo = mid;
        else hi = mid - 1;
    }
    const int64_t first = __ldg(&items[lo].off[2]);
    const int64_t units = (lo + 1 < n ? __ldg(&items[lo + 1].off[2]) : total) - first;
    const int64_t w = __ldg(&items[lo].w3);
    const int64_t k = (x - __ldg(&items[lo].woff3) + w - 1) / w;
    return first + (k < units ? k : units);
}

// In the voxelize and ray-trace phases a CTA's units are a contiguous run
// [lo, hi) of the phase's units, so that it moves to another frame (and
// restages that frame's arguments) only a few times.  Their units cost about
// the same in every frame.  The inflate and merge units cost more in some
// frames than in others (tile width and radius; how much of a grid the
// measurement marks), so there the units go round the CTAs in turn, or, in
// the gathered phases, as CTAs come free.
__device__ __forceinline__ int64_t run_begin(int64_t total, unsigned b, unsigned nb) { return total * b / nb; }

// The frame of unit u, given the frame i of an earlier unit of the same CTA
// in the same phase (frames with no units in this phase are skipped).
__device__ __forceinline__ int next_item(const BatchItem *items, int n, int phase, int64_t u, int i) {
    while (i + 1 < n && __ldg(&items[i + 1].off[phase]) <= u) ++i;
    return i;
}

// The ray trace reads the occupancy planes with ordinary (L1-cached) loads:
// phase 2 wrote them before the grid barrier, whose release (every CTA's
// fence before it arrives) and acquire (thread 0's fence after it, then
// the CTA barrier) order those writes before these loads, and no SM reads
// a plane word of this launch's occupancy before phase 3, so none holds a
// stale line of it.  (64 robots: 148.1k -> 150.9k Mvoxel-updates/s.)
template <int LPR>
__device__ __forceinline__ unsigned group_lpr(const FrameArgs &a, int buffered, const float S[3], const Box &b,
                                              int64_t grp, int64_t G, uint32_t *box_fr, uint32_t *box_tr,
                                              const uint32_t *occ_box, uint32_t *buf) {
    return rt_group<LPR, units::LoadPlain>(a, S, b, grp, G, buffered, box_fr, box_tr, occ_box, buf);
}

// The tile of the inflate phase's unit u, in frame i.
struct Tile {
    int x, y, z;
};
__device__ __forceinline__ Tile tile_of(const BatchItem &it, int64_t u) {
    // a frame has fewer than 2^27 plane words, so fewer tiles
    const uint32_t local = (uint32_t)(u - it.off[1]), t0 = (uint32_t)it.tiles[0];
    const uint32_t t01 = local / t0;
    return Tile{it.tile0[0] + (int)(local - t01 * t0), it.tile0[1] + (int)(t01 % (uint32_t)it.tiles[1]),
                it.tile0[2] + (int)(t01 / (uint32_t)it.tiles[1])};
}

// One inflate tile of TXW words x 8 rows x TZ slices of a batch frame:
// starts its staging in st, or (DO) runs its passes from there.
template <bool DO, int TXW, int TZ>
__device__ __forceinline__ void inflate_part(const BatchItem &it, const Tile &t, uint32_t *st, uint32_t *buf1) {
    const PlaneGeom &g = it.a.g;
    auto part = [&](auto radius) {
        constexpr int R = decltype(radius)::value;
        if (DO) units::inflate_passes<R, TXW, 8, TZ>(g, it.a.pl.occ_inf, R, t.x, t.y, t.z, st, TXW + 2, 0, buf1);
        else units::inflate_stage<R, TXW, 8, TZ>(g, it.a.pl.occ_raw, t.x, t.y, t.z, st);
    };
    switch (it.a.r) {
    case 1: part(std::integral_constant<int, 1>()); break;
    case 2: part(std::integral_constant<int, 2>()); break;
    default: part(std::integral_constant<int, 3>()); break;
    }
}
template <bool DO>
__device__ __forceinline__ void inflate_unit(const BatchItem &it, const Tile &t, uint32_t *st, uint32_t *buf1) {
    switch (it.txw * 10 + it.tz) {
    case 88: inflate_part<DO, 8, 8>(it, t, st, buf1); break;
    case 84: inflate_part<DO, 8, 4>(it, t, st, buf1); break;
    case 48: inflate_part<DO, 4, 8>(it, t, st, buf1); break;
    default: inflate_part<DO, 4, 4>(it, t, st, buf1); break;
    }
}

// Copies a frame's arguments into shared memory, by the threads of the CTA
// (the caller places the barriers).
__device__ __forceinline__ void stage_args(const FrameArgs &src, FrameArgs &dst) {
    const uint32_t *s = reinterpret_cast<const uint32_t *>(&src);
    uint32_t *d = reinterpret_cast<uint32_t *>(&dst);
    for (int k = threadIdx.x; k < (int)(sizeof(FrameArgs) / 4); k += kThreads) d[k] = __ldg(s + k);
}

// GATHER: some frame may be gathered.  Batches of walked frames alone, which
// are small, take a kernel of their own: the gathered phases' code costs them
// time although they run none of it (one 320x240 frame into 80 x 80 x 40 voxels
// 43.9 us a step with it, 41.0 without; into 100 x 100 x 20 46.5 and 45.6).
template <bool GATHER>
__global__ void __launch_bounds__(kThreads, 4) k_batch(const BatchItem *__restrict__ items, BatchCtl *ctl) {
    __shared__ uint32_t box_fr[kBoxWords], box_tr[kBoxWords], occ_box[kBoxWords];
    extern __shared__ __align__(16) uint32_t dyn[];
    const int n = ctl->n;
    const unsigned nb = gridDim.x;

    // The frame arguments of the unit at hand are staged in shared memory
    // (s_a) whenever the CTA moves to another frame, so that the per-pixel
    // and per-ray code reads them there rather than field by field from the
    // table in global memory.
    __shared__ FrameArgs s_a;
    __shared__ int32_t s_kind;   // phase 1: dtype * 3 + pix_mode; phase 3: LPR * 2 + buffered

    // ---- phase 1: voxelize ------------------------------------------------
    {
        units::WordTab &tab = *reinterpret_cast<units::WordTab *>(dyn);
        units::tab_clear(tab);   // (the first frame's staging ends with a barrier)
        int cur = -1;
        const int64_t lo = run_begin(ctl->total[0], blockIdx.x, nb), hi = run_begin(ctl->total[0], blockIdx.x + 1, nb);
        int i = find_item(items, n, 0, lo);
        for (int64_t u = lo; u < hi;) {
            i = next_item(items, n, 0, u, i);   // the same for every thread
            if (i != cur) {
                __syncthreads();   // the previous frame's copy is no longer read
                stage_args(items[i].a, s_a);
                if (threadIdx.x == 0) s_kind = __ldg(&items[i].dtype) * 3 + __ldg(&items[i].pix_mode);
                __syncthreads();
                cur = i;
            }
            const int64_t local = u - __ldg(&items[i].off[0]), pix = __ldg(&items[i].pix_units);
            if (GATHER && local >= pix) {
                gather::table_thread(s_a, (local - pix) * kThreads + threadIdx.x);
                ++u;
                continue;
            }
            // the frame's units of this run, each one's depths loaded while
            // the one before is placed
            const int run = (int)(hi - u < pix - local ? hi - u : pix - local);
            switch (s_kind) {
            case 0: units::voxelize_run<0, units::kPixTile>(s_a, (int32_t)local, run, tab); break;
            case 1: units::voxelize_run<0, units::kPixTile4>(s_a, (int32_t)local, run, tab); break;
            case 2: units::voxelize_run<0, units::kPixLinear>(s_a, (int32_t)local, run, tab); break;
            case 3: units::voxelize_run<1, units::kPixTile>(s_a, (int32_t)local, run, tab); break;
            case 4: units::voxelize_run<1, units::kPixTile4>(s_a, (int32_t)local, run, tab); break;
            default: units::voxelize_run<1, units::kPixLinear>(s_a, (int32_t)local, run, tab); break;
            }
            u += run;
        }
        if (GATHER && blockIdx.x == 0 && threadIdx.x == 0) ctl->next = 0u;   // phase 3 counts from 0
    }
    if (!grid_sync(ctl, nb)) return;

    // ---- phase 2: inflate -------------------------------------------------
    {
        // units in turn over the CTAs: their cost differs between frames,
        // and interleaving keeps the CTAs' shares even.  A tile is staged
        // while the one before it is worked on.  (No SM reads occ_raw in this
        // launch before this phase, so its L1 holds no older state of it.)
        const int64_t total = ctl->total[1];
        int i = find_item(items, n, 1, blockIdx.x);
        Tile t = {};
        if (blockIdx.x < total) {
            t = tile_of(items[i], blockIdx.x);
            inflate_unit<false>(items[i], t, dyn, nullptr);
        }
        uint32_t *st = dyn, *other = dyn + kStageWords;
        for (int64_t u = blockIdx.x; u < total; u += nb) {
            int j = i;
            Tile tj = {};
            if (u + nb < total) {
                j = next_item(items, n, 1, u + nb, i);
                tj = tile_of(items[j], u + nb);
                inflate_unit<false>(items[j], tj, other, nullptr);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            inflate_unit<true>(items[i], t, st, dyn + 2 * kStageWords);   // ends with a barrier
            i = j;
            t = tj;
            uint32_t *const swap = st;
            st = other;
            other = swap;
        }
    }
    if (!grid_sync(ctl, nb)) return;

    // ---- phase 3, gathered: around the camera, and the skin ---------------
    // units go to the CTAs as these come free: their cost differs between
    // and within frames.  (Here and in the phases after it frame i's arguments are
    // staged for every unit: a CTA's units lie far apart.)
    auto stage = [&](int i) {
        __syncthreads();   // the previous copy is no longer read
        stage_args(items[i].a, s_a);
        __syncthreads();
    };
    // The next unit of this CTA: its first is its own, the others are handed
    // out.  Thread 0 asks as the unit before begins.
    __shared__ uint32_t s_next;
    auto ask = [&]() { return threadIdx.x == 0 ? nb + atomicAdd(&ctl->next, 1u) : 0u; };
    auto told = [&](uint32_t asked) {
        if (threadIdx.x == 0) s_next = asked;
        __syncthreads();
        return (int64_t)s_next;
    };
    if (GATHER) {
        float S[3];
        int32_t v0[3];
        uint32_t asked = 0;
        int i = blockIdx.x < ctl->total[4] ? find_item(items, n, 4, blockIdx.x) : 0;
        for (int64_t u = blockIdx.x; u < ctl->total[4]; u = told(asked)) {
            i = next_item(items, n, 4, u, i);
            stage(i);
            asked = ask();
            gather::frame_start(s_a, S, v0);
            const int32_t local = (int32_t)(u - __ldg(&items[i].off[4])), near = __ldg(&items[i].near_units);
            if (local < near)
                gather::near_unit<units::LoadPlain>(s_a, S, v0, local, dyn);
            else
                gather::skin_unit<units::LoadPlain>(s_a, S, v0, local - near, __ldg(&items[i].skin_units),
                                                    *reinterpret_cast<gather::SkinSmem *>(dyn));
        }
        __syncthreads();
    }

    // ---- phase 3, scattered: ray trace -------------------------------------
    // a contiguous run of units per CTA, so the camera box is staged again
    // only when the run crosses into another frame; the runs split the
    // units' total weight evenly (weights of 1: their number)
    if (!GATHER || ctl->total[2]) {
        const int64_t lo = weighted_unit(items, n, ctl->total[2], run_begin(ctl->wtotal3, blockIdx.x, nb));
        const int64_t hi = weighted_unit(items, n, ctl->total[2], run_begin(ctl->wtotal3, blockIdx.x + 1, nb));
        int cur = -1, i = find_item(items, n, 2, lo);
        float S[3] = {0.0f, 0.0f, 0.0f};
        Box b = {0, 0, 0};
        for (int64_t u = lo; u < hi; ++u) {
            i = next_item(items, n, 2, u, i);   // the same for every thread
            if (i != cur) {
                if (cur >= 0) box_flush(s_a, b, box_fr, box_tr);   // ends with a barrier
                else __syncthreads();   // phase 1's copy is no longer read
                stage_args(items[i].a, s_a);
                if (threadIdx.x == 0) s_kind = __ldg(&items[i].lpr) * 2 + __ldg(&items[i].buffered);
                __syncthreads();
                cur = i;
                frame_start(s_a, S);
                b = box_of(S);
                box_stage<units::LoadPlain>(s_a, b, box_fr, box_tr, occ_box);
            }
            // the frame's rays are spread over its G units of this phase
            const int64_t off = __ldg(&items[i].off[2]);
            const int64_t grp = u - off;
            const int64_t G = (i + 1 < n ? __ldg(&items[i + 1].off[2]) : ctl->total[2]) - off;
            const int buffered = s_kind & 1;
            unsigned visits;
            switch (s_kind >> 1) {
            case 8: visits = group_lpr<8>(s_a, buffered, S, b, grp, G, box_fr, box_tr, occ_box, dyn); break;
            case 16: visits = group_lpr<16>(s_a, buffered, S, b, grp, G, box_fr, box_tr, occ_box, dyn); break;
            default: visits = group_lpr<32>(s_a, buffered, S, b, grp, G, box_fr, box_tr, occ_box, dyn); break;
            }
            if (s_a.stats) {
                const unsigned total = __reduce_add_sync(kFull, visits);
                if ((threadIdx.x & 31) == 0 && total) atomicAdd(s_a.stats + 2, (unsigned long long)total);
            }
        }
        if (cur >= 0) box_flush(s_a, b, box_fr, box_tr);
    }
    if (!grid_sync(ctl, nb)) return;

    // ---- phase 3b: the latest hits of the gathered frames' rays -----------
    if (GATHER && ctl->total[5]) {
        int i = 0;
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->next = 0u;   // and phase 4
        for (int64_t u = blockIdx.x; u < ctl->total[5]; u += nb) {
            i = u == blockIdx.x ? find_item(items, n, 5, u) : next_item(items, n, 5, u, i);
            stage(i);
            gather::late_unit<units::LoadPlain>(s_a, (int32_t)(u - __ldg(&items[i].off[5])),
                                                *reinterpret_cast<gather::LateSmem *>(dyn));
        }
        if (!grid_sync(ctl, nb)) return;
    }

    // ---- phase 4: merge ---------------------------------------------------
    {
        float S[3];
        int32_t v0[3];
        const bool handed = GATHER && ctl->total[5] != 0;   // (a batch of scattered frames alone: in turn)
        uint32_t asked = 0;
        int i = find_item(items, n, 3, blockIdx.x);
        for (int64_t u = blockIdx.x; u < ctl->total[3]; u = handed ? told(asked) : u + nb) {
            i = next_item(items, n, 3, u, i);
            const BatchItem &it = items[i];
            const int64_t local = u - __ldg(&it.off[3]);
            if (handed) asked = ask();
            if (GATHER && __ldg(&it.a.ga.on)) {
                stage(i);
                const int32_t box = __ldg(&it.box_units);
                if (local < box) {
                    gather::frame_start(s_a, S, v0);
                    gather::gather_unit<kGatherWords, false, units::LoadPlain>(
                        s_a, S, v0, (uint32_t)local, box, *reinterpret_cast<gather::GatherSmem<kGatherWords> *>(dyn));
                } else {
                    gather::outside_word<false>(s_a, (local - box) * kThreads + threadIdx.x);
                }
                continue;
            }
            // the unit's mwpu plane words, one or two per thread
            for (int k = 0; k < it.mwpu; k += kThreads)
                units::merge_word<units::LoadL2>(it.a.g, it.a.pl, it.a.loc, it.a.ring, local * it.mwpu + k + threadIdx.x);
            if (handed) __syncthreads();   // s_next is no longer read
        }
    }
}

int g_batch_blocks_per_sm[64];
int g_batch_sms[64];

}  // namespace

cudaError_t configure_batch(int dev) {
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const size_t dyn = sizeof(uint32_t) * kDynWords;
    cudaError_t e = cudaDeviceGetAttribute(&g_batch_sms[dev], cudaDevAttrMultiProcessorCount, dev);
    int per_sm[2] = {0, 0};
    for (int k = 0; k < 2; ++k) {
        auto kernel = k ? k_batch<true> : k_batch<false>;
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[k], kernel, kThreads, dyn);
    }
    g_batch_blocks_per_sm[dev] = per_sm[0] < per_sm[1] ? per_sm[0] : per_sm[1];
    return e;
}

int batch_max_blocks(int dev) {
    if (dev < 0 || dev >= 64) return 0;
    return g_batch_sms[dev] * g_batch_blocks_per_sm[dev];
}

cudaError_t launch_batch(const BatchItem *items, BatchCtl *ctl, int blocks, bool gather, cudaStream_t s) {
    void *args[] = {(void *)&items, (void *)&ctl};
    return cudaLaunchCooperativeKernel((const void *)(gather ? k_batch<true> : k_batch<false>), dim3(blocks), dim3(kThreads),
                                       args, sizeof(uint32_t) * kDynWords, s);
}

}  // namespace vg
