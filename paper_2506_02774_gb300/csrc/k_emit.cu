// k_emit.cu -- emission of (tile, Gaussian) pairs in depth order with the
// tile-level preemptive alpha test, and the blend's tile order (which also
// finishes the per-tile ranges the last tile-sort pass records).
//
// Every visible Gaussian has a range of pair slots (one per candidate tile) in
// depth order; their first slots come with the depth order (k_depth.cu, or
// k_slot_scan after the radix passes: an exclusive scan of the counts by
// decoupled look-back over tiles of 4096), and so does, for every chunk of 1024
// slots, the depth rank that owns its first slot.  k_emit gives each CTA whole
// chunks, so a CTA's work does not depend on how the slots are spread over the
// Gaussians (a near one can have thousands): it marks the slots at which a
// Gaussian starts in a bitmap, a slot finds its Gaussian by counting the marks
// up to it, and reads its record (one 32-byte sector, shared through L1 with
// the Gaussian's other slots).  Chunks
// of 512 Gaussians before this left the CTA with the near ones running alone
// (SM cycles 43 % busy on average) and gathered three half-used sectors each;
// 1M-leaf box at 1080p (981K slots): 53 -> 18 us, city at 1080p (4.26M slots):
// 107 -> 52 us (with the records of two slots per lane in flight together; one: 56,
// all four, in CTAs of 512 threads: 68).  For each slot the tile-level form of
// Eq. 4 (paper Sec. 4.2) decides: a kept slot gets key = tile id, a dropped one
// all ones, which the tile sort's first pass leaves out (the others stay in
// depth order within a tile, the sort being stable).  The slot's
// value is the Gaussian's index in the in-front arrays << 8 | its row mask in
// that tile: bit w is set when the footprint box reaches one of the tile's
// pixel rows w MR .. w MR + MR - 1, MR = tile / 8 rows (1 for 8-pixel tiles);
// outside the box the Eq. 4 test fails at every pixel, so the blend reads only
// the records a strip needs, straight from the in-front arrays.  Indices
// therefore take 24 bits: a frame with more cut nodes in front of the camera
// reports an overflow.  The digit counts of the tile sort's first pass are
// written here as well, a row per chunk.
#include <cuda_fp16.h>

#include "vgr_internal.cuh"
#include "vgr_launch.h"
#include "vgr_tiletest.cuh"

namespace vgr {

constexpr int EM_THREADS = 256;
constexpr int EM_AHEAD = 2;                   // slots per lane whose records are in flight together
constexpr int EM_WARPS = EM_THREADS / 32;
constexpr uint32_t EM_SLOTS = EMIT_SLOTS;   // slots per chunk: 32 runs of a warp
constexpr uint32_t EM_GAUSS = EM_SLOTS + 1; // Gaussians that may be looked at for a chunk
static_assert(EM_SLOTS == 1024, "32 words of start bits, one per lane of the scanning warp");

uint32_t emit_owner_cap(uint64_t cap_pairs) { return (uint32_t)(cap_pairs / EMIT_SLOTS) + 1u; }

constexpr int SS_THREADS = 256;
constexpr int SS_ITEMS = 16;
constexpr int SS_TILE = SS_THREADS * SS_ITEMS;  // Gaussians per look-back tile of the slot scan

uint32_t slot_scan_tile() { return SS_TILE; }

// off[r] = candidate slots of the Gaussians of depth rank < r (r <= n_vis);
// off[n_vis] is the frame's candidate-slot count.
__global__ void __launch_bounds__(SS_THREADS) k_slot_scan(const uint32_t* __restrict__ order, uint32_t cap_vis,
                                                          const uint32_t* __restrict__ ntile,
                                                          uint32_t* __restrict__ off,
                                                          uint32_t* __restrict__ owner, uint64_t cap_pairs,
                                                          unsigned long long* __restrict__ status,
                                                          Counters* __restrict__ ctr,
                                                          const FrameParams* __restrict__ fp) {
    pdl_wait();
    __shared__ uint32_t s_scan[9];
    __shared__ uint32_t s_tile, s_prefix;
    const uint32_t n_vis = min(ctr->n_vis, cap_vis);
    const uint32_t ntiles = (n_vis + SS_TILE - 1) / SS_TILE;
    const uint32_t epoch = fp->epoch;
    if (blockIdx.x == 0 && threadIdx.x == 0 && ctr->n_front > MAX_RANKS) atomicOr(&ctr->flags, F_OVF_VIS);
    if (n_vis == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            off[0] = 0u;
            ctr->n_cand = 0ull;
        }
        return;
    }
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(&ctr->tickets[TK_EMIT], 1u);
        __syncthreads();
        const uint32_t tile = s_tile;
        if (tile >= ntiles) break;
        // thread t owns ranks tile * SS_TILE + SS_ITEMS t .. + SS_ITEMS - 1 (gathers in flight together)
        const uint32_t r0 = tile * SS_TILE + SS_ITEMS * threadIdx.x;
        uint32_t c[SS_ITEMS], vi[SS_ITEMS];
#pragma unroll
        for (int k = 0; k < SS_ITEMS; ++k) vi[k] = r0 + k < n_vis ? order[r0 + k] : NONE;
#pragma unroll
        for (int k = 0; k < SS_ITEMS; ++k) c[k] = vi[k] != NONE ? ntile[vi[k]] : 0u;
        uint32_t sum = 0;
#pragma unroll
        for (int k = 0; k < SS_ITEMS; ++k) sum += c[k];
        uint32_t total;
        uint32_t run = block_excl_scan<SS_THREADS / 32>(sum, s_scan, &total);
        if (threadIdx.x < 32) {
            // (test hook: tile 0 stays silent, so the others' bounded waits run out)
            const bool silent = tile == 0 && (fp->test_hooks & VGR_HOOK_WITHHOLD_LOOKBACK);
            const uint32_t pre = silent ? 0u : lookback_warp(status, 1, tile, total, epoch, &ctr->flags);
            if (threadIdx.x == 0) s_prefix = pre;
        }
        __syncthreads();
        run += s_prefix;
#pragma unroll
        for (int k = 0; k < SS_ITEMS; ++k) {
            if (r0 + k < n_vis) {
                off[r0 + k] = run;
                emit_owner(owner, (uint32_t)(cap_pairs / EMIT_SLOTS) + 1u, run, c[k], r0 + k);
            }
            run += c[k];
        }
        if (threadIdx.x == 0) {
            // the offsets wrap past 2^32, the frame's count does not.  A tile's own total wraps
            // only at 2^32 itself (4096 entries of 2^20 slots each)
            atomicAdd(&ctr->n_cand, total ? (unsigned long long)total : 1ull << 32);
            if (tile == ntiles - 1) off[n_vis] = s_prefix + total;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(EM_THREADS, 4) k_emit(const uint32_t* __restrict__ order, uint32_t cap_vis,
                                                     const float4* __restrict__ rec,
                                                     const uint32_t* __restrict__ slot_off,
                                                     const uint32_t* __restrict__ owner,
                                                     uint32_t* __restrict__ pair_key,
                                                     uint32_t* __restrict__ pair_val, uint64_t cap, int bits,
                                                     RadixTab tab, Counters* __restrict__ ctr,
                                                     const FrameParams* __restrict__ fp) {
    pdl_wait();
    __shared__ uint2 s_g[EM_GAUSS];   // per Gaussian: index in the in-front arrays, first slot
    __shared__ uint32_t s_bits[32];   // slots at which a Gaussian starts
    __shared__ uint32_t s_cnt[256];   // the chunk's kept slots by first digit
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, D = 1u << bits;
    const uint32_t n_vis = min(ctr->n_vis, cap_vis);
    // Slots that do not fit their buffers, or 32 bits, may have wrapped offsets, and a
    // slot scan that timed out leaves wrong ones: the owners then do not ascend, so
    // nothing is read through them.  Such a frame is replayed or refused.
    const uint64_t cand = ctr->n_cand;
    const bool timed_out = (ctr->flags & F_SPIN_TIMEOUT) != 0u;
    if (cand > cap || cand >= 0xFFFFFFFFull || timed_out) {
        if (blockIdx.x == 0 && threadIdx.x == 0 && !timed_out) atomicOr(&ctr->flags, F_OVF_PAIRS);
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctr->n_slots = cand;
    const uint32_t ns = (uint32_t)cand;
    const uint32_t nchunks = n_vis ? (ns + EM_SLOTS - 1u) / EM_SLOTS : 0u;
    const uint32_t TW = fp->tiles_x;
    const int T = (int)fp->tile;
    const int MR = T >= 8 ? T / 8 : 1;  // tile rows per row-mask bit (8 bits)
    const float Wf = fp->width_f, Hf = fp->height_f;
    const bool canonical = fp->filter == VGR_FILTER_CANONICAL;
    uint32_t kept = 0;
    for (uint32_t ck = blockIdx.x; ck < nchunks; ck += gridDim.x) {
        const uint32_t j0 = ck * EM_SLOTS, len = min(EM_SLOTS, ns - j0);
        const uint32_t g0 = owner[ck];
        const uint32_t g1 = ck + 1u < nchunks ? owner[ck + 1u] : n_vis - 1u;  // may start past the chunk
        const uint32_t m = min(g1 - g0 + 1u, EM_GAUSS);
        if (threadIdx.x < 32) s_bits[threadIdx.x] = threadIdx.x == 0 ? 1u : 0u;  // the chunk's first slot has an owner
        if (threadIdx.x < 256) s_cnt[threadIdx.x] = 0u;
        __syncthreads();
        for (uint32_t q = threadIdx.x; q < m; q += EM_THREADS) {
            const uint32_t o = slot_off[g0 + q];
            s_g[q] = make_uint2(order[g0 + q], o);
            if (o > j0 && o - j0 < len) atomicOr(&s_bits[(o - j0) >> 5], 1u << (o & 31u));  // j0 is a multiple of 32
        }
        __syncthreads();
        uint32_t total;
        const uint32_t bits_l = s_bits[lane];
        const uint32_t pre_l = warp_excl_scan(__popc(bits_l), &total);  // starts before word 'lane'
        for (uint32_t r0 = 0; r0 < EM_SLOTS / EM_THREADS; r0 += EM_AHEAD) {
            uint2 gvs[EM_AHEAD];
            float4 recA[EM_AHEAD], recB[EM_AHEAD];
#pragma unroll
            for (int r = 0; r < EM_AHEAD; ++r) {
                const uint32_t word = (r0 + r) * EM_WARPS + warp;
                const uint32_t bits = __shfl_sync(0xFFFFFFFFu, bits_l, word);
                const uint32_t before = __shfl_sync(0xFFFFFFFFu, pre_l, word);
                if (32u * word + lane < len) {
                    // the last Gaussian that starts at or before this slot
                    gvs[r] = s_g[before + __popc(bits & ((2u << lane) - 1u)) - 1u];
                    recA[r] = rec[2 * (size_t)gvs[r].x];
                    recB[r] = rec[2 * (size_t)gvs[r].x + 1];
                }
            }
#pragma unroll
            for (int r = 0; r < EM_AHEAD; ++r) {
                const uint32_t word = (r0 + r) * EM_WARPS + warp;
                const uint32_t j = j0 + 32u * word + lane;
                if (32u * word + lane < len) {
                    const uint2 gv = gvs[r];
                    const float4 A = recA[r], B = recB[r];
                    const uint32_t local = j - gv.y;
                    const uint32_t rc = __float_as_uint(B.z);
                    const uint32_t w = rc >> 20;
                    // local / w and local % w: local < 2^20 and w <= 2^10, so (local + 1/2) / w is
                    // at least 1 / 2^11 from an integer and its FP32 quotient floors exactly
                    const uint32_t qy = (uint32_t)(((float)local + 0.5f) * __frcp_rn((float)w));
                    const int tx = (int)(rc & 0x3FFu) + (int)(local - qy * w);
                    const int ty = (int)((rc >> 10) & 0x3FFu) + (int)qy;
                    bool keep = true;
                    uint32_t rows = 0xFFu;
                    if (!canonical) {
                        // the conic is stored pre-scaled (A = -a/2, B = -b, C = -c/2): exact to undo;
                        // edge optima dy* = (-b / c) dx, dx* = (-b / a) dy: an ulp or two of
                        // error moves rho_max by far less than the test's 2e-3 slack
                        const float ca = -2.0f * A.z, cb = -A.w, cc = -2.0f * B.x;
                        keep = tile_keep(A.x, A.y, ca, cb, cc, __fdividef(-cb, ca), __fdividef(-cb, cc), B.y - TILE_EPS,
                                         tx, ty, Wf, Hf, T);
                        // tile rows r with |row0 + r - v| <= half-height, as groups of MR rows
                        const float row0 = (float)(ty * T) + 0.5f;
                        const float hh = __half2float(__ushort_as_half((unsigned short)(__float_as_uint(B.w) & 0xFFFFu)));
                        const float rlo = fmaxf(0.f, ceilf(A.y - hh - row0));
                        const float rhi = fminf((float)(T - 1), floorf(A.y + hh - row0));
                        rows = 0u;
                        if (rlo <= rhi) {
                            const uint32_t w0 = (uint32_t)rlo / MR, w1 = (uint32_t)rhi / MR;
                            rows = ((2u << w1) - 1u) & ~((1u << w0) - 1u);
                        }
                    }
                    const uint32_t key = keep ? (uint32_t)ty * TW + (uint32_t)tx : NONE;
                    kept += keep;
                    pair_key[j] = key;
                    pair_val[j] = (gv.x << 8) | rows;
                    if (keep) atomicAdd(&s_cnt[key & (D - 1u)], 1u);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < D) {
            const uint32_t c = s_cnt[threadIdx.x];
            tab.rows[(size_t)ck * D + threadIdx.x] = (uint16_t)c;
            if (c) atomicAdd(&tab.groups[(size_t)(ck / RADIX_GROUP) * D + threadIdx.x], c);
        }
    }
    const uint32_t wk = __reduce_add_sync(0xFFFFFFFFu, kept);
    if (lane == 0 && wk) atomicAdd(&ctr->n_pairs, (unsigned long long)wk);
}

// The tile of every sorted pair (the debug view's array), from the ranges.
__global__ void k_debug_tiles(const uint2* __restrict__ ranges, uint32_t n_tiles, uint32_t* __restrict__ pair_tile,
                              uint64_t n_pairs) {
    for (uint32_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const uint2 r = ranges[t];
        for (uint64_t i = r.x + threadIdx.x; i < r.y && i < n_pairs; i += blockDim.x) pair_tile[i] = t;
    }
}

void launch_debug_tiles(const uint2* ranges, uint32_t n_tiles, uint32_t* pair_tile, uint64_t n_pairs, cudaStream_t s) {
    if (n_pairs) k_debug_tiles<<<1024, 128, 0, s>>>(ranges, n_tiles, pair_tile, n_pairs);
}

void launch_slot_scan(const uint32_t* order, uint32_t cap_vis, const VisBuffers& vis, uint32_t* slot_off,
                      uint32_t* owner, uint64_t cap_pairs, unsigned long long* status, Counters* ctr,
                      const FrameParams* fp, int grid, cudaStream_t s) {
    launch_k(k_slot_scan, grid, SS_THREADS, s, order, cap_vis, (const uint32_t*)vis.ntile, slot_off, owner, cap_pairs,
             status, ctr, fp);
}

void launch_emit(const uint32_t* order, uint32_t cap_vis, const VisBuffers& vis, const uint32_t* slot_off,
                 const uint32_t* owner, uint32_t* pair_key, uint32_t* pair_val, uint64_t cap_pairs, int bits,
                 RadixTab tab, Counters* ctr, const FrameParams* fp, int grid, cudaStream_t s) {
    launch_k(k_emit, grid, EM_THREADS, s, order, cap_vis, (const float4*)vis.rec, slot_off, owner, pair_key, pair_val,
             cap_pairs, bits, tab, ctr, fp);
}

// Blend order: tiles by descending pair count (classes of floor(log2(count+1)),
// heaviest class first), so the long tiles start in the first round and the
// short ones fill in behind them; the order inside a class does not matter
// (tiles are independent).  It also finishes the ranges the last tile-sort
// pass recorded as (start, ~end) by atomic minima from all ones: each becomes
// [start, end), or [0, 0) for a tile without pairs.  The class counts go to the
// frame's counters, for a batch's order over all its views.
// One cluster of 8 CTAs: each counts its tiles' classes in its own shared
// memory, the CTAs read each other's counts (distributed shared memory) for
// their places in the order, and place their tiles.  The few classes are
// counted and claimed once per run of equal classes in a warp (match
// instruction), not once per tile.  What bounds it is the chain load - count -
// barrier - place; one CTA walking all 8160 tiles of a 1080p image took 11 us,
// the cluster takes 6.
constexpr int TO_CTAS = 8;

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// word *p of the cluster's CTA 'rank'
__device__ __forceinline__ uint32_t cluster_load(const uint32_t* p, uint32_t rank) {
    uint32_t a, v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n"
                 : "=r"(a)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];\n" : "=r"(v) : "r"(a) : "memory");
    return v;
}

__global__ void __cluster_dims__(TO_CTAS, 1, 1) __launch_bounds__(1024)
    k_tile_order(uint2* __restrict__ ranges, uint32_t n_tiles, uint32_t* __restrict__ order,
                 Counters* __restrict__ ctr) {
    pdl_wait();
    __shared__ uint32_t s_cnt[33], s_start[33];
    const uint32_t lane = lane_id(), rank = blockIdx.x;  // one cluster: the CTA's rank is its index
    if (threadIdx.x < 33) s_cnt[threadIdx.x] = 0u;
    __syncthreads();
    const uint32_t first = rank * blockDim.x + (threadIdx.x & ~31u), stride = TO_CTAS * blockDim.x;
    for (uint32_t t0 = first; t0 < n_tiles; t0 += stride) {  // warp-uniform trips
        const uint32_t t = t0 + lane;
        uint32_t cls = 64u;  // past the end: no class
        if (t < n_tiles) {
            uint2 r = ranges[t];
            r = r.x == 0xFFFFFFFFu ? make_uint2(0u, 0u) : make_uint2(r.x, ~r.y);
            ranges[t] = r;  // read back below by this same thread
            cls = 32 - __clz(r.y - r.x + 1u);
        }
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, cls);
        if (cls < 33u && lane == (uint32_t)(__ffs(peers) - 1)) atomicAdd(&s_cnt[cls], (uint32_t)__popc(peers));
    }
    cluster_sync();
    if (threadIdx.x < 32) {
        // lane l takes class 32 - l (a count is below 2^32 - 1, so class 0 is
        // empty): its tiles in the whole image and in the CTAs before this one
        const uint32_t b = 32u - lane;
        uint32_t all = 0, before = 0;
#pragma unroll
        for (uint32_t c = 0; c < TO_CTAS; ++c) {
            const uint32_t v = cluster_load(&s_cnt[b], c);
            all += v;
            before += c < rank ? v : 0u;
        }
        uint32_t total;
        s_start[b] = warp_excl_scan(all, &total) + before;
        const uint32_t heavy = __reduce_add_sync(0xFFFFFFFFu, b >= BL_HEAVY_CLASS ? all : 0u);
        if (rank == 0) {
            ctr->tile_buckets[b] = all;
            if (lane == 0) ctr->n_heavy = heavy;
        }
    }
    cluster_sync();  // the counts have been read, the starts are there
    for (uint32_t t0 = first; t0 < n_tiles; t0 += stride) {
        const uint32_t t = t0 + lane;
        uint32_t cls = 64u;
        if (t < n_tiles) {
            const uint2 r = ranges[t];
            cls = 32 - __clz(r.y - r.x + 1u);
        }
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, cls);
        const int leader = __ffs(peers) - 1;
        uint32_t at = 0;
        if (cls < 33u && (int)lane == leader) at = atomicAdd(&s_start[cls], (uint32_t)__popc(peers));
        at = __shfl_sync(0xFFFFFFFFu, at, leader);
        if (cls < 33u) order[at + __popc(peers & lanemask_lt())] = t;
    }
}

void launch_tile_order(uint2* ranges, uint32_t n_tiles, uint32_t* order, Counters* ctr, cudaStream_t s) {
    launch_k(k_tile_order, TO_CTAS, 1024, s, ranges, n_tiles, order, ctr);
}

// The blend order of a batch: the tiles of all its views by class, heaviest
// first, each view's tiles of a class in that view's own order.  Class b of
// view v starts at off(b, v) = (tiles of every view in the classes above b)
// + (class-b tiles of the views before v); within view v's own order the
// class starts at start(b, v) = (v's tiles in the classes above b), so a tile
// at position p of v's order goes to p + off(b, v) - start(b, v): one CTA
// computes that difference per (class, view), then a grid places the tiles.
constexpr uint32_t BATCH_MAX_VIEWS = 1024;

__global__ void __launch_bounds__(1024) k_batch_offsets(const FrameParams* const* __restrict__ fps, uint32_t n_views,
                                                        uint32_t* __restrict__ delta,
                                                        uint32_t* __restrict__ n_heavy) {
    pdl_wait();
    __shared__ uint32_t s_scan[33];
    const uint32_t v = threadIdx.x;
    const Counters* c = v < n_views ? fps[v]->bl_ctr : nullptr;
    uint32_t run = 0, vstart = 0;
    for (int b = 32; b >= 0; --b) {
        const uint32_t cnt = c ? c->tile_buckets[b] : 0u;
        uint32_t total;
        const uint32_t pre = block_excl_scan<32>(cnt, s_scan, &total);
        if (c) delta[(size_t)b * n_views + v] = run + pre - vstart;
        vstart += cnt;
        run += total;
        if (v == 0u && b == (int)BL_HEAVY_CLASS) *n_heavy = run;
        __syncthreads();  // s_scan is reused by the next class
    }
}

__global__ void __launch_bounds__(256) k_batch_scatter(const FrameParams* const* __restrict__ fps, uint32_t n_views,
                                                       const uint32_t* const* __restrict__ orders,
                                                       const uint32_t* __restrict__ tile_base, uint32_t total,
                                                       const uint32_t* __restrict__ delta, uint32_t* __restrict__ work) {
    pdl_wait();
    for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        uint32_t lo = 0, hi = n_views;  // the view v with tile_base[v] <= g < tile_base[v + 1]
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (tile_base[mid] <= g) lo = mid; else hi = mid;
        }
        const uint32_t v = lo, p = g - tile_base[v];
        const uint32_t t = orders[v][p];
        const uint2 r = fps[v]->bl_ranges[t];
        const uint32_t b = 32 - __clz(r.y - r.x + 1u);
        work[p + delta[(size_t)b * n_views + v]] = (v << 20) | t;
    }
}

void launch_batch_order(const FrameParams* const* fps, uint32_t n_views, const uint32_t* const* orders,
                        const uint32_t* tile_base, uint32_t total_tiles, uint32_t* delta, uint32_t* work,
                        uint32_t* n_heavy, int grid, cudaStream_t s) {
    launch_k(k_batch_offsets, 1, BATCH_MAX_VIEWS, s, fps, n_views, delta, n_heavy);
    launch_k(k_batch_scatter, grid, 256, s, fps, n_views, orders, tile_base, total_tiles, (const uint32_t*)delta, work);
}

}  // namespace vgr
