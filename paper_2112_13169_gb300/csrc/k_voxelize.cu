// K1 as its own launch: a CTA per tile of pixels, a thread per point; the
// work itself is in vg_units.cuh.
#include "vg_gather.cuh"

#include <algorithm>

namespace vg {
namespace {

// K1 lets the frame's later kernels launch only once the work before the
// frame has completed: with `early` right after its own wait, so that K2's
// launch overlaps K1; without, when K1 completes, which leaves K1's SM
// slots to K3's CTAs, whose walk runs before they wait for K2 (a gathered
// frame's K3 does nothing before its wait).
//
// The first `ntab` CTAs write the gathered form's ray table instead.
template <int DT, int MODE>
__global__ void __launch_bounds__(256) k_voxelize_depth(const FrameArgs a, const int early, const int ntab) {
    __shared__ units::WordTab tab;
    pdl_wait();   // the depth image and the planes belong to earlier work
    if (early) pdl_trigger();
    if ((int)blockIdx.x < ntab) {
        gather::table_thread(a, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
        return;
    }
    const unsigned block = blockIdx.x - ntab;
    if (a.rt_next && block == 0 && threadIdx.x == 0) *a.rt_next = 0u;   // K3 of this frame counts from 0
    units::voxelize_tile<DT, MODE>(a, (int32_t)block, tab);
}

__global__ void __launch_bounds__(256) k_voxelize_points(const FrameArgs a, const int early, const int ntab) {
    pdl_wait();
    if (early) pdl_trigger();
    if ((int)blockIdx.x < ntab) {
        gather::table_thread(a, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
        return;
    }
    const unsigned block = blockIdx.x - ntab;
    if (a.rt_next && block == 0 && threadIdx.x == 0) *a.rt_next = 0u;
    units::voxelize_points_thread(a, (int64_t)block * blockDim.x + threadIdx.x);
}

// A cloud into a plane that fits shared memory: each CTA ORs its points into
// a plane of its own and then its words into occ_raw.  A cloud's points come in
// no order, so a warp's lanes seldom share a word, and the words of a near
// wall or of a floor's rows take a good part of all points: 300,000 points
// into 100 x 100 x 20 voxels queued at one L2 slice (68 % busy with atomics, the
// slices' mean 1.4 %).  Here a word is hit at most once per CTA.
constexpr int kDenseThreads = 1024;
__global__ void __launch_bounds__(kDenseThreads) k_voxelize_points_dense(const FrameArgs a, const int early,
                                                                         const int ntab) {
    extern __shared__ uint32_t plane[];
    pdl_wait();
    if (early) pdl_trigger();
    if ((int)blockIdx.x < ntab) {
        gather::table_thread(a, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
        return;
    }
    const unsigned block = blockIdx.x - ntab, blocks = gridDim.x - ntab;
    if (a.rt_next && block == 0 && threadIdx.x == 0) *a.rt_next = 0u;
    const int words = (int)a.g.words;
    for (int w = threadIdx.x; w < words; w += kDenseThreads) plane[w] = 0;
    __syncthreads();
    // whole warps stay in the loop: the points are counted warp by warp
    for (int64_t i0 = (int64_t)block * kDenseThreads; i0 < a.npts; i0 += (int64_t)blocks * kDenseThreads) {
        uint32_t bit = 0;
        const uint32_t key = units::point_of_cloud(a, i0 + threadIdx.x, bit);
        if (key != units::kNoWord && !(plane[key] & bit)) atomicOr(plane + key, bit);
        units::count_points(a, key != units::kNoWord);
    }
    __syncthreads();
    // from another word in every CTA, so that their atomics do not queue
    const int from = (int)((int64_t)words * block / blocks);
    for (int k = threadIdx.x; k < words; k += kDenseThreads) {
        const int w = from + k < words ? from + k : from + k - words;
        const uint32_t v = plane[w];
        if (v) atomicOr(a.pl.occ_raw + w, v);
    }
}

// Planes of up to 48 KB, the shared memory of a CTA without a set-up, and
// clouds of at least four points a word (a CTA clears and scans its plane).
constexpr int64_t kDenseWords = 12 * 1024;
constexpr int64_t kDenseBlocks = 152;   // one to an SM

}  // namespace

cudaError_t launch_voxelize_depth(const FrameArgs &a, int32_t dtype, cudaStream_t s, const Sched &sc) {
    const int ntab = (int)((gather::table_threads(a) + 255) / 256);
    const unsigned blocks = (unsigned)units::pixel_tiles(a) + ntab;
    auto run = [&](void (*k)(FrameArgs, int, int)) { return launch_pdl(k, blocks, 256, 0, s, a, (int)sc.early_inflate, ntab); };
    switch (dtype * 3 + units::pixel_mode(a, dtype == 0 ? 4 : 2)) {
    case 0: return run(k_voxelize_depth<0, units::kPixTile>);
    case 1: return run(k_voxelize_depth<0, units::kPixTile4>);
    case 2: return run(k_voxelize_depth<0, units::kPixLinear>);
    case 3: return run(k_voxelize_depth<1, units::kPixTile>);
    case 4: return run(k_voxelize_depth<1, units::kPixTile4>);
    default: return run(k_voxelize_depth<1, units::kPixLinear>);
    }
}

cudaError_t launch_voxelize_points(const FrameArgs &a, cudaStream_t s, const Sched &sc) {
    if (a.g.words <= kDenseWords && a.npts >= 4 * a.g.words) {
        const int ntab = (int)((gather::table_threads(a) + kDenseThreads - 1) / kDenseThreads);
        const unsigned blocks = (unsigned)std::min<int64_t>((a.npts + kDenseThreads - 1) / kDenseThreads, kDenseBlocks);
        return launch_pdl(k_voxelize_points_dense, blocks + ntab, kDenseThreads, (size_t)a.g.words * 4, s, a,
                          (int)sc.early_inflate, ntab);
    }
    // an empty cloud still takes a CTA, which zeroes K3's counter
    const int ntab = (int)((gather::table_threads(a) + 255) / 256);
    const unsigned blocks = (unsigned)std::max<int64_t>((a.npts + 255) / 256, 1) + ntab;
    return launch_pdl(k_voxelize_points, blocks, 256, 0, s, a, (int)sc.early_inflate, ntab);
}

}  // namespace vg
