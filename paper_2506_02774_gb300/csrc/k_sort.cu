// k_sort.cu -- stable LSD radix sort of (u32 key, u32 value) pairs, one or two
// kernels per digit of up to 8 bits: a count of the digits of every tile, and a
// scatter of the tiles.
//
// Sorts the emitted pairs by tile id (paper Sec. 3.1 'Sorting'), stable, so a
// tile's pairs keep their depth order; the depth keys of frames whose depths
// are too concentrated for the partition (k_depth.cu); and the pairs of the
// standalone calls.
//
// A pass's tables hold the digit counts of every tile (rows) and of every 32
// rows (groups).  A tile's base per digit is the sum of the groups and rows
// before it, which the scatter adds up for itself while the tile's keys are on
// their way: nothing waits for another tile.  (One kernel per pass whose tiles
// found their bases by look-back took 18-24 us for up to a million keys whatever
// the traffic: all the tiles were in flight at once, each digit's chain was as
// long as their number.)  The rows of the tile sort's first pass are written by
// the emission, so its count kernel is saved there.
//
// What bounds it: the instructions of the ranking.  Peers by one ballot per digit
// bit kept the ballots' pipe and half of the issue slots busy; lane masks OR-ed
// in shared memory take a third of the instructions, but lanes of one digit queue
// at its mask, so lane 0's are taken out by a ballot first.  4M random 32-bit
// keys: 174 us by ballots, 165 by masks alone, 167 with both; 7 different keys:
// 165, 178, 143; runs of 50 equal keys: 167, 186, 151 (match.any: 233, 138, 137).
// With the table-based passes the tile sort of 981K slots (1M-leaf box, 1080p) went
// from 47 to 29 us, of 4.26M (city, 1080p) from 85 to 71, of 235K (320 x 180, one
// pass) from 24 to 12, of 63K (801 x 603) to 18, the sort of 4M keys from 191 to
// 167.  Three CTAs an SM at 40 registers were no faster.
#include "vgr_internal.cuh"
#include "vgr_launch.h"

namespace vgr {

constexpr int RS_THREADS = RADIX_THREADS;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr uint32_t RS_TILE = RADIX_TILE;
constexpr int RS_ITEMS = RADIX_TILE / RADIX_THREADS, RS_ITEMS_SMALL = RADIX_TILE_SMALL / RADIX_THREADS;
static_assert(RS_TILE <= 0xFFFFu, "a row's counts and a tile's places fit 16 bits");

size_t radix_rows(uint64_t n, uint32_t row_len) {
    return (size_t)(row_len ? (n + row_len - 1) / row_len : radix_max_tiles(n));
}
size_t radix_groups(uint64_t n, uint32_t row_len) { return (radix_rows(n, row_len) + RADIX_GROUP - 1) / RADIX_GROUP; }
size_t radix_row_words(uint64_t n, uint32_t row_len, int bits) { return radix_rows(n, row_len) << bits; }
size_t radix_group_words(uint64_t n, uint32_t row_len, int bits) { return radix_groups(n, row_len) << bits; }

// Keys per thread: few keys go in small tiles over many SMs, since a tile's ranking is
// a chain over its keys per thread.  The line lies at one small tile per SM: per tile
// sort, 63K slots (801 x 603, two passes) took 22.9 us in tiles of 4096 and 18.4 in
// tiles of 1024, and 3.2K slots (one pass) 10.2 and 8.2, but 235K slots (one pass) 12.3
// and 13.3.
__device__ __forceinline__ int radix_items(uint32_t n) { return n > RADIX_SMALL_N ? RS_ITEMS : RS_ITEMS_SMALL; }

__device__ __forceinline__ uint32_t radix_n(const uint32_t* n32, const unsigned long long* n64, uint64_t cap) {
    uint64_t n = n32 ? (uint64_t)*n32 : n64 ? (uint64_t)*n64 : cap;
    return (uint32_t)(n < cap ? n : cap);
}

// Digit counts of every tile, and of every group of tiles.
__global__ void __launch_bounds__(RS_THREADS) k_radix_count(const uint32_t* __restrict__ keys,
                                                            const uint32_t* __restrict__ n32,
                                                            const unsigned long long* __restrict__ n64, uint64_t cap,
                                                            int shift, int bits, RadixTab tab) {
    pdl_wait();
    __shared__ uint32_t s_cnt[2][256];
    const uint32_t n = radix_n(n32, n64, cap);
    const int items = radix_items(n);
    const uint32_t tile_keys = items * RS_THREADS;
    const uint32_t ntiles = (uint32_t)(((uint64_t)n + tile_keys - 1) / tile_keys), D = 1u << bits, t = threadIdx.x;
    if (t < 256) s_cnt[0][t] = s_cnt[1][t] = 0u;
    __syncthreads();
    uint32_t flip = 0;
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, flip ^= 1u) {
        const uint32_t base = tile * tile_keys + t;  // n < 2^32, and so is a tile's end
        uint32_t key[RS_ITEMS];
#pragma unroll
        for (int k = 0; k < RS_ITEMS; ++k) {
            if (k >= items) break;
            const uint32_t i = base + k * RS_THREADS;
            key[k] = i < n ? keys[i] : 0u;
        }
#pragma unroll
        for (int k = 0; k < RS_ITEMS; ++k) {
            if (k >= items) break;
            if (base + k * RS_THREADS < n) atomicAdd(&s_cnt[flip][(key[k] >> shift) & (D - 1u)], 1u);
        }
        __syncthreads();
        if (t < D) {
            const uint32_t c = s_cnt[flip][t];
            s_cnt[flip][t] = 0u;  // used again after the next tile's barrier
            tab.rows[(size_t)tile * D + t] = (uint16_t)c;
            if (c) atomicAdd(&tab.groups[(size_t)(tile / RADIX_GROUP) * D + t], c);
        }
    }
}

// One digit pass over tiles of ITEMS pairs a thread (one row of the tables each, or
// as many rows of row_len pairs as it holds):
//  1. the tile's keys and values are requested; meanwhile the tables' entries
//     before the tile are added up (two digits per thread and load);
//  2. each warp ranks its contiguous share, an item per lane at a time: the peers
//     of lane 0 (same digit) by a ballot, the others' by the digits' lane masks in
//     shared memory, and the foremost peer advances the warp's counter of its digit;
//  3. a thread per digit turns the warps' counts into places in the tile;
//  4. the pairs are staged digit-sorted in shared memory and
//  5. stored, each digit's run contiguously.
// With DROP, pairs whose key is all ones are left out.  keys_out may be null.
// The last pass of the tile sort also records each tile's range: a CTA's staged
// elements are in final key order and each key's run is one contiguous stretch
// of global positions, so the first and last element of every run it holds give
// atomicMin updates of (start, ~end), from all ones.
template <uint32_t D>
struct RadixSmem {
    __align__(16) uint2 kv[RS_TILE];         // the tile staged digit-sorted: (key, value)
    __align__(16) uint16_t wc[RS_WARPS][D];  // per-warp digit counts, then per-warp places
    uint32_t gofs[D];                        // global index minus staged index, per digit
    uint32_t scan[2][RS_WARPS];
};

template <int BITS, bool DROP, int ITEMS>
__device__ __forceinline__ void radix_tiles(
    RadixSmem<1u << BITS>& sm, uint32_t n, const uint32_t* __restrict__ keys_in, const uint32_t* __restrict__ vals_in,
    uint32_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out, int shift, RadixTab tab, uint32_t row_len,
    uint2* __restrict__ ranges, uint32_t n_ranges) {
    constexpr uint32_t D = 1u << BITS, NQ = 2 * RS_THREADS / D;  // rows read at once, two digits a thread
    constexpr uint32_t tile_keys = ITEMS * RS_THREADS;
    static_assert(D <= RS_THREADS && 2 * RS_THREADS % D == 0 && RS_TILE >= 2 * RS_THREADS, "table layout");
    uint2* s_kv = sm.kv;
    uint16_t (*s_wc)[D] = sm.wc;
    uint32_t* s_gofs = sm.gofs;
    uint32_t (*s_scan)[RS_WARPS] = sm.scan;
    // the tables' partial sums lie under the staging buffer: groups, then rows
    uint32_t (*s_grp)[D] = reinterpret_cast<uint32_t (*)[D]>(s_kv);
    uint32_t (*s_row)[D] = reinterpret_cast<uint32_t (*)[D]>(s_kv + RS_THREADS);
    // and so do the warps' peer masks, behind them
    uint32_t (*s_mask)[D] = reinterpret_cast<uint32_t (*)[D]>(s_kv + 2 * RS_THREADS);
    static_assert(RS_WARPS * D * sizeof(uint32_t) <= (RS_TILE - 2 * RS_THREADS) * sizeof(uint2), "masks' place");
    const uint32_t ntiles = (uint32_t)(((uint64_t)n + tile_keys - 1) / tile_keys);
    const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    const uint32_t pair = t % (D / 2), q = t / (D / 2);
    if (blockIdx.x >= ntiles) return;
    const uint32_t row_tiles = row_len ? tile_keys / row_len : 1u;
    const uint32_t nrows = row_len ? (uint32_t)(((uint64_t)n + row_len - 1) / row_len) : ntiles;
    const uint32_t ngroups = (nrows + RADIX_GROUP - 1) / RADIX_GROUP;
    const uint2* groups2 = reinterpret_cast<const uint2*>(tab.groups);
    const uint32_t* rows2 = reinterpret_cast<const uint32_t*>(tab.rows);
    uint32_t run = 0;       // thread d: pairs of smaller digits, and of digit d in the groups before 'seen'
    uint32_t seen = 0;
    {
        uint2 tot = make_uint2(0u, 0u);
        for (uint32_t g = q; g < ngroups; g += NQ) {
            const uint2 v = groups2[(size_t)g * (D / 2) + pair];
            tot.x += v.x;
            tot.y += v.y;
        }
        reinterpret_cast<uint2*>(s_grp[q])[pair] = tot;
        __syncthreads();
        uint32_t c = 0, total;
        if (t < D) {
#pragma unroll
            for (uint32_t k = 0; k < NQ; ++k) c += s_grp[k][t];
        }
        run = block_excl_scan<RS_WARPS>(c, s_scan[0], &total);
        __syncthreads();
    }
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const uint32_t base = tile * tile_keys + warp * (32u * ITEMS) + lane;  // n < 2^32, and so is a tile's end
        uint32_t key[ITEMS], val[ITEMS], rank[ITEMS];
        const bool full = n - tile * tile_keys >= tile_keys;  // (uniform)
        if (full) {
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) key[it] = keys_in[base + it * 32u];
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) val[it] = vals_in ? vals_in[base + it * 32u] : base + it * 32u;
        } else {
#pragma unroll
            for (int it = 0; it < ITEMS; ++it) {
                const uint32_t idx = base + it * 32u;
                key[it] = idx < n ? keys_in[idx] : 0u;
                val[it] = idx < n ? (vals_in ? vals_in[idx] : idx) : 0u;
            }
        }
        const uint32_t r0 = tile * row_tiles, g0 = r0 / RADIX_GROUP;
        {
            uint2 a = make_uint2(0u, 0u), b = make_uint2(0u, 0u);
            for (uint32_t g = seen + q; g < g0; g += NQ) {
                const uint2 v = groups2[(size_t)g * (D / 2) + pair];
                a.x += v.x;
                a.y += v.y;
            }
            for (uint32_t r = g0 * RADIX_GROUP + q; r < r0; r += NQ) {
                const uint32_t v = rows2[(size_t)r * (D / 2) + pair];
                b.x += v & 0xFFFFu;
                b.y += v >> 16;
            }
            reinterpret_cast<uint2*>(s_grp[q])[pair] = a;
            reinterpret_cast<uint2*>(s_row[q])[pair] = b;
        }
        seen = g0;
        for (uint32_t i = t; i < RS_WARPS * D / 2; i += RS_THREADS) reinterpret_cast<uint32_t*>(&s_wc[0][0])[i] = 0u;
        for (uint32_t i = t; i < RS_WARPS * D / 4; i += RS_THREADS)
            reinterpret_cast<uint4*>(s_mask)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        uint32_t live = 0u;  // bit it: the pair takes part
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const uint32_t d = (key[it] >> shift) & (D - 1u);
            const bool valid = (full && !DROP) || (base + it * 32u < n && !(DROP && key[it] == NONE));
            live |= (uint32_t)valid << it;
            const uint32_t d0 = __shfl_sync(0xFFFFFFFFu, d, 0);
            const bool as_first = valid && d == d0;
            const uint32_t first = __ballot_sync(0xFFFFFFFFu, as_first);
            if (valid && !as_first) atomicOr(&s_mask[warp][d], 1u << lane);
            __syncwarp();
            const uint32_t peers = as_first ? first : valid ? s_mask[warp][d] : 1u << lane;
            __syncwarp();  // read before the foremost clears it
            const int foremost = __ffs(peers) - 1;
            uint32_t before = 0;
            if (valid && (int)lane == foremost) {
                before = s_wc[warp][d];
                s_wc[warp][d] = (uint16_t)(before + __popc(peers));
                s_mask[warp][d] = 0u;
            }
            before = __shfl_sync(0xFFFFFFFFu, before, foremost);
            rank[it] = before + __popc(peers & lanemask_lt());
            __syncwarp();  // the counters and masks as the next item's lanes read them
        }
        __syncthreads();
        uint32_t cnt = 0, ofs = 0, tile_n;
        if (t < D) {
#pragma unroll
            for (int w = 0; w < RS_WARPS; ++w) cnt += s_wc[w][t];
#pragma unroll
            for (uint32_t k = 0; k < NQ; ++k) {
                run += s_grp[k][t];
                ofs += s_row[k][t];
            }
        }
        const uint32_t lstart = block_excl_scan<RS_WARPS>(cnt, s_scan[1], &tile_n);
        if (t < D) {
            uint32_t p = lstart;
#pragma unroll
            for (int w = 0; w < RS_WARPS; ++w) {
                const uint32_t c = s_wc[w][t];
                s_wc[w][t] = (uint16_t)p;
                p += c;
            }
            s_gofs[t] = run + ofs - lstart;
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            if ((live >> it) & 1u)
                s_kv[s_wc[warp][(key[it] >> shift) & (D - 1u)] + rank[it]] = make_uint2(key[it], val[it]);
        }
        __syncthreads();
        for (uint32_t j = t; j < tile_n; j += RS_THREADS) {
            const uint2 kv = s_kv[j];
            const uint32_t pos = s_gofs[(kv.x >> shift) & (D - 1u)] + j;
            if (pos < n) {
                if (keys_out) keys_out[pos] = kv.x;
                vals_out[pos] = kv.y;
                if (ranges && kv.x < n_ranges) {
                    const uint32_t kp = j > 0u ? s_kv[j - 1u].x : ~kv.x;
                    const uint32_t kn = j + 1u < tile_n ? s_kv[j + 1u].x : ~kv.x;
                    if (kp != kv.x) atomicMin(&ranges[kv.x].x, pos);
                    if (kn != kv.x) atomicMin(&ranges[kv.x].y, ~(pos + 1u));
                }
            }
        }
        __syncthreads();  // the partial sums of the next tile go over the staged pairs
    }
}

template <int BITS, bool DROP>
__global__ void __launch_bounds__(RS_THREADS, 2) k_radix_scatter(
    const uint32_t* __restrict__ keys_in, const uint32_t* __restrict__ vals_in, uint32_t* __restrict__ keys_out,
    uint32_t* __restrict__ vals_out, const uint32_t* __restrict__ n32, const unsigned long long* __restrict__ n64,
    uint64_t cap, int shift, RadixTab tab, uint32_t row_len, uint2* __restrict__ ranges, uint32_t n_ranges) {
    pdl_wait();
    __shared__ RadixSmem<1u << BITS> sm;
    const uint32_t n = radix_n(n32, n64, cap);
    if (radix_items(n) == RS_ITEMS)
        radix_tiles<BITS, DROP, RS_ITEMS>(sm, n, keys_in, vals_in, keys_out, vals_out, shift, tab, row_len, ranges,
                                          n_ranges);
    else
        radix_tiles<BITS, DROP, RS_ITEMS_SMALL>(sm, n, keys_in, vals_in, keys_out, vals_out, shift, tab, row_len,
                                              ranges, n_ranges);
}

int radix_grid(int sms) { return 2 * sms; }

void launch_radix_count(const uint32_t* keys, const uint32_t* n32, const unsigned long long* n64, uint64_t cap,
                        int shift, int bits, RadixTab tab, int grid, cudaStream_t s) {
    launch_k(k_radix_count, grid, RS_THREADS, s, keys, n32, n64, cap, shift, bits, tab);
}

void launch_radix_scatter(const uint32_t* keys_in, const uint32_t* vals_in, uint32_t* keys_out, uint32_t* vals_out,
                          const uint32_t* n32, const unsigned long long* n64, uint64_t cap, int shift, int bits,
                          RadixTab tab, uint32_t row_len, bool drop, int grid, cudaStream_t s, uint2* ranges,
                          uint32_t n_ranges) {
#define VGR_SCATTER_D(B, DR)                                                                                          \
    launch_k(k_radix_scatter<B, DR>, grid, RS_THREADS, s, keys_in, vals_in, keys_out, vals_out, n32, n64, cap, shift, \
             tab, row_len, ranges, n_ranges)
#define VGR_SCATTER(B)                    \
    do {                                  \
        if (drop) VGR_SCATTER_D(B, true); \
        else VGR_SCATTER_D(B, false);     \
    } while (0)
    switch (bits) {
        case 5: VGR_SCATTER(5); break;
        case 6: VGR_SCATTER(6); break;
        case 7: VGR_SCATTER(7); break;
        default: VGR_SCATTER(8); break;
    }
#undef VGR_SCATTER
#undef VGR_SCATTER_D
}

}  // namespace vgr
