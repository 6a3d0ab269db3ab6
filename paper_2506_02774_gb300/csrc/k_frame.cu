// k_frame.cu -- the start of a frame: its parameters and cleared tables.
//
// One kernel reads the frame's parameters from pinned host memory and clears
// what the frame counts into (counters, depth bins, tile counts, bucket cursors,
// digit groups) and the tile ranges.  It replaces a copy and three fills, each of
// which was a step of its own on the frame's critical path; the status block
// likewise goes to pinned host memory from the blend's last CTA instead of by two
// copies (about 15 us of a frame: 94 -> 80 on the 128 x 128 thumbnail, 112 -> 96 on
// the 60K-leaf window).  Bound by its launch and one round trip to the host.
#include "vgr_internal.cuh"
#include "vgr_launch.h"

namespace vgr {

constexpr int FB_THREADS = 256;

__device__ __forceinline__ void fill_words(uint4* p, size_t n16, uint32_t value) {
    const size_t stride = (size_t)gridDim.x * FB_THREADS;
    for (size_t i = (size_t)blockIdx.x * FB_THREADS + threadIdx.x; i < n16; i += stride)
        p[i] = make_uint4(value, value, value, value);
}

__global__ void __launch_bounds__(FB_THREADS) k_frame_begin(const FrameParams* host, FrameParams* dev, FrameClear c) {
    pdl_wait();
    static_assert(sizeof(FrameParams) % 4 == 0, "copied in words");
    constexpr uint32_t PW = sizeof(FrameParams) / 4;
    // the parameters by the last CTA, whose share of the fills is the smallest
    if (blockIdx.x == gridDim.x - 1u)
        for (uint32_t i = threadIdx.x; i < PW; i += FB_THREADS)
            reinterpret_cast<uint32_t*>(dev)[i] = reinterpret_cast<const volatile uint32_t*>(host)[i];
    fill_words(c.zero[0], c.zero16[0], 0u);
    fill_words(c.zero[1], c.zero16[1], 0u);
    fill_words(c.zero[2], c.zero16[2], 0u);
    const uint32_t stride = gridDim.x * FB_THREADS;
    for (uint32_t t = blockIdx.x * FB_THREADS + threadIdx.x; t < c.n_ranges; t += stride)
        c.ranges[t] = make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);  // (start, ~end), taken by minima
}

void launch_frame_begin(const FrameParams* host, FrameParams* dev, const FrameClear& c, int sms, cudaStream_t s) {
    launch_k(k_frame_begin, sms, FB_THREADS, s, host, dev, c);
}

}  // namespace vgr
