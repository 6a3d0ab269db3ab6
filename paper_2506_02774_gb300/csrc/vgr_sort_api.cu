// vgr_sort_api.cu -- the pair sort of the frame path (paper Sec. 3.1
// 'Sorting') as a standalone C-ABI call: stable LSD radix sort of u32
// (key, value) pairs on the device, 8-bit digits, a count and a scatter kernel
// per digit (k_sort.cu).  Scratch (digit counts, the ping-pong buffer of
// multi-pass sorts) comes from a per-device cache owned by the library.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>

#include "vgr.h"
#include "vgr_internal.cuh"
#include "vgr_launch.h"

namespace vgr {

size_t sort_row_words(uint64_t n) { return radix_row_words(n, 0, 8); }
size_t sort_group_words(uint64_t n, int passes) { return (size_t)passes * radix_group_words(n, 0, 8); }

int sort_passes(uint32_t key_bits) { return (int)((key_bits + 7u) / 8u); }

// Enqueue a sort on 's' with the given scratch; returns a CUDA error code.
cudaError_t sort_pairs_enqueue(const uint32_t* keys_in, const uint32_t* vals_in, uint32_t* keys_out,
                               uint32_t* vals_out, uint64_t n, int passes, uint16_t* rows, uint32_t* groups,
                               uint32_t* tmp_keys, uint32_t* tmp_vals, int sms, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(groups, 0, sort_group_words(n, passes) * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<uint64_t>(radix_grid(sms), radix_max_tiles(n));
    PdlScope pdl(true);  // the first kernel follows the clear in plain stream order
    // the last pass writes the output; earlier passes alternate backwards
    const uint32_t* kin = keys_in;
    const uint32_t* vin = vals_in;
    for (int p = 0; p < passes; ++p) {
        const bool to_out = ((passes - 1 - p) & 1) == 0;
        uint32_t* ko = to_out ? keys_out : tmp_keys;
        uint32_t* vo = to_out ? vals_out : tmp_vals;
        const RadixTab tab{rows, groups + sort_group_words(n, p)};
        launch_radix_count(kin, nullptr, nullptr, n, 8 * p, 8, tab, grid, s);
        launch_radix_scatter(kin, vin, ko, vo, nullptr, nullptr, n, 8 * p, 8, tab, 0u, false, grid, s);
        kin = ko;
        vin = vo;
    }
    return cudaGetLastError();
}

}  // namespace vgr

using namespace vgr;

namespace {

struct SortCache {
    std::mutex mu;
    uint16_t* rows = nullptr;
    size_t row_words = 0;
    uint32_t* groups = nullptr;
    size_t group_words = 0;
    uint32_t* tmp = nullptr;
    uint64_t tmp_n = 0;
    int sms = 0;
};

// Room for 'words' elements at p, growing it if there is less.
template <typename T>
cudaError_t sort_room(T*& p, size_t& have, size_t words) {
    if (words <= have) return cudaSuccess;
    if (p) cudaFree(p);
    p = nullptr;
    have = 0;
    const cudaError_t e = cudaMalloc(&p, words * sizeof(T));
    if (e == cudaSuccess) have = words;
    else p = nullptr;
    return e;
}

SortCache g_cache[64];

vgr_status sort_fail(vgr_status s, const char* msg, cudaError_t e = cudaSuccess) {
    char buf[512];
    snprintf(buf, sizeof(buf), "%s%s%s", msg, e != cudaSuccess ? ": " : "", e != cudaSuccess ? cudaGetErrorString(e) : "");
    set_last_error(buf);
    return s;
}

}  // namespace

extern "C" vgr_status vgr_sort_pairs(const uint32_t* keys_in, const uint32_t* vals_in, uint32_t* keys_out,
                                     uint32_t* vals_out, uint64_t n, uint32_t key_bits, void* stream) {
    if (key_bits < 1 || key_bits > 32) return sort_fail(VGR_E_INVALID, "key_bits must be in [1, 32]");
    if (n == 0) return VGR_OK;
    if (n >= 0xFFFFFFFFull) return sort_fail(VGR_E_INVALID, "n must be below 2^32 - 1");
    if (!keys_in || !vals_in || !keys_out || !vals_out) return sort_fail(VGR_E_INVALID, "null pointer");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) return sort_fail(VGR_E_CUDA, "cudaGetDevice", e);
    SortCache& c = g_cache[dev];
    std::lock_guard<std::mutex> lock(c.mu);
    if (!c.sms) {
        int sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        c.sms = std::max(1, sms);
    }
    const int passes = sort_passes(key_bits);
    if ((e = sort_room(c.rows, c.row_words, sort_row_words(n))) != cudaSuccess ||
        (e = sort_room(c.groups, c.group_words, sort_group_words(n, passes))) != cudaSuccess)
        return sort_fail(VGR_E_NOMEM, "sort digit counts", e);
    if (passes > 1 && n > c.tmp_n) {
        if (c.tmp) cudaFree(c.tmp);
        c.tmp = nullptr;
        c.tmp_n = 0;
        const uint64_t n_al = (n + 63u) & ~(uint64_t)63u;  // the value half starts 256-byte aligned
        if ((e = cudaMalloc(&c.tmp, 2 * n_al * sizeof(uint32_t))) != cudaSuccess)
            return sort_fail(VGR_E_NOMEM, "sort ping-pong buffer", e);
        c.tmp_n = n_al;
    }
    cudaStream_t s = (cudaStream_t)stream;
    e = sort_pairs_enqueue(keys_in, vals_in, keys_out, vals_out, n, passes, c.rows, c.groups, c.tmp,
                           c.tmp ? c.tmp + c.tmp_n : nullptr, c.sms, s);
    if (e != cudaSuccess) return sort_fail(VGR_E_CUDA, "sort launch", e);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return sort_fail(VGR_E_CUDA, "sort", e);
    return VGR_OK;
}
