// K3 and K4 in their gathered form as their own launches; the work itself is
// in vg_gather.cuh.
#include "vg_gather.cuh"

namespace vg {
namespace {

using namespace gather;

// The first `nnear` CTAs mark the voxels around the camera, the others test
// 256 words of occupied voxels each against the rays.
__global__ void __launch_bounds__(kThreads) k_rayhit(const FrameArgs a, const int nnear) {
    __shared__ union {
        uint32_t near[3 * kNearRows];
        SkinSmem skin;
    } sh;
    pdl_trigger();
    float S[3];
    int32_t v0[3];
    frame_start(a, S, v0);
    pdl_wait();
    if ((int)blockIdx.x < nnear) near_unit<units::LoadPlain>(a, S, v0, blockIdx.x, sh.near);
    else skin_unit<units::LoadPlain>(a, S, v0, blockIdx.x - nnear, gridDim.x - nnear, sh.skin);
}

__global__ void __launch_bounds__(kThreads) k_raylate(const FrameArgs a) {
    __shared__ LateSmem sh;
    pdl_trigger();
    pdl_wait();
    late_unit<units::LoadPlain>(a, blockIdx.x, sh);
}

// The first `nbox` CTAs take the words of the frame's box, the others what
// lies outside it: what a re-centre brought in, and a cloud's points.
// Four CTAs to an SM: without the bound, small changes elsewhere tip the
// compiler between 59 registers and 48 with spills, four CTAs and five.  Which
// is better goes with the number of CTAs: three headings of a 640x480 camera in
// 200 x 200 x 100 voxels take 163, 135 and 161 us for four frames with four,
// 148, 144 and 141 with five.
template <int WPU>
__global__ void __launch_bounds__(kThreads, 4) k_gather(const FrameArgs a, const int nbox) {
    __shared__ GatherSmem<WPU> sh;
    pdl_trigger();
    float S[3];
    int32_t v0[3];
    frame_start(a, S, v0);
    pdl_wait();
    if ((int)blockIdx.x < nbox) gather_unit<WPU, true, units::LoadPlain>(a, S, v0, blockIdx.x, nbox, sh);
    else if (a.whole) outside_word<true>(a, (int64_t)((int)blockIdx.x - nbox) * kThreads + threadIdx.x);
    else outside_word<false>(a, (int64_t)((int)blockIdx.x - nbox) * kThreads + threadIdx.x);
}

template <int WPU>
cudaError_t gather_words(const FrameArgs &a, cudaStream_t s) {
    const unsigned nbox = word_units<WPU, 4>(a.box);
    return launch_pdl(k_gather<WPU>, nbox + (unsigned)outside_units(a, kThreads), kThreads, 0, s, a, (int)nbox);
}

}  // namespace

// K3: the hits, then their latest of each tile and neighbourhood.
cudaError_t launch_rayhit(const FrameArgs &a, cudaStream_t s) {
    const int nnear = near_units_of(a);
    const cudaError_t e =
        launch_pdl(k_rayhit, nnear + word_units<kThreads, 1>(a.box), kThreads, 0, s, a, nnear);
    return e == cudaSuccess ? launch_pdl(k_raylate, late_units(a), kThreads, 0, s, a) : e;
}

// A CTA's words are taken a patch per warp and its listed voxels a thread
// each, one phase after another, so a CTA of few words ends sooner and one of
// many spends less on its barriers and rounds.  Measured (a frame with its
// read, CTAs of 64 / 128 / 256 words): a box of 40 k words 35 / 38 / 52 us, of
// 76 k 44 / 41 / 47, of 200 k 83 / 77 / 77, of 600 k 203 / 174 / 163.  CTAs of
// 128 threads, whose barriers hold fewer warps, and of 512 lose as well:
// three 640x480 frames with their read 157 to 189 and 170 us against 148.
cudaError_t launch_gather(const FrameArgs &a, cudaStream_t s) {
    const int64_t words = (int64_t)a.box.nw * a.box.ny * a.box.nz;
    if (words < 45000) return gather_words<64>(a, s);
    if (words < 250000) return gather_words<128>(a, s);
    return gather_words<256>(a, s);
}

}  // namespace vg
