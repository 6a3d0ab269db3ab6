// k_depth.cu -- the depth order of the visible Gaussians (paper Sec. 3.1
// 'Sorting') by one partition and one sort per bucket, and each Gaussian's
// first pair slot.
//
// The order is (FP32 depth key, node id), i.e. (key, in-front index), and a
// pair (key, index) is unique, so no step needs to be stable and none needs a
// look-back chain:
//  * preprocess counts the visible keys in DEPTH_BINS bins of a monotone
//    function of the key (half of the bins logarithmic in z over the depths the
//    scene's bounds allow, half linear over those of its middle: depth_bin);
//  * k_depth_part scans the bins (every CTA for itself), joins neighbouring
//    bins into buckets of about s keys (bucket of a bin = its exclusive prefix
//    / s, so no bucket holds more than s + its largest bin), and
//    writes each (key, index << 8 | slot count) to its bucket, at a place
//    reserved with one atomic per CTA and bucket; the same atomic adds up the
//    bucket's candidate slots;
//  * k_depth_local gives each bucket to one CTA: a counting sort by 4096
//    sub-bins of the bucket's bins (finer steps of the same monotone function)
//    in shared memory leaves runs of one or two keys, whose members rank
//    themselves by (key, index); a bucket with a long run (many equal keys) is
//    sorted by a bitonic network instead.
//    The slot counts travel with the keys, so the CTA also writes the first
//    slot of each of its Gaussians (the sum of the earlier buckets' slots plus
//    a scan of its own).
// Four stable radix passes and a scan of the slot counts did this before; each
// pass was a chain of look-back round trips (15-21 us for 550K keys whatever
// the traffic).  Depth order and slots, 1M-leaf box at 1080p (552K visible):
// 96 -> 26 us; city at 1080p (2.67M visible): 153 -> 60 us.  Bound now by the
// shared-memory atomics and barriers of a CTA's steps (issue slots 35-50 %).
// A bucket that does not fit a CTA (F_SORT_SKEW: thousands of Gaussians in one
// bin) makes the host replay the frame with the radix passes of k_sort.cu, and
// order the view's next 63 frames by them: 82 us for 536K visible (26 here), 130 for
// 2M (47); the look-back passes of before took 74 and 98.
#include <algorithm>

#include "vgr_internal.cuh"
#include "vgr_launch.h"

namespace vgr {

constexpr int DP_THREADS = 512;
constexpr int DP_ITEMS = 16;
constexpr int DP_TILE = DP_THREADS * DP_ITEMS;  // entries a CTA partitions at a time
constexpr int DP_BPT = DEPTH_BINS / DP_THREADS;  // bins per thread
constexpr uint32_t DP_KEYS_MIN = 256, DP_KEYS_MAX = 4096;  // keys aimed at per bucket
constexpr uint32_t DP_ROUNDS = 3, DP_CTAS = 320;           // rounds of at most so many CTAs shared out evenly
// A bucket's cursor: its keys so far, and above them its candidate slots.  An entry has
// at most 2^20 slots, so a bucket that fits a CTA has less than 2^33, which one word
// holds; a tile's share of them is added up in 32 bits, entries of many slots apart.
constexpr int DP_KEY_BITS = 25;
constexpr uint32_t DP_FEW_SLOTS = 0xFFFFFFFFu / DP_TILE;
static_assert(MAX_RANKS < (1u << DP_KEY_BITS), "a cursor counts every key");
static_assert(DP_BPT % 4 == 0, "bins are read as uint4");

constexpr int DL_THREADS = 512;
constexpr int DL_WARPS = DL_THREADS / 32;
constexpr uint32_t DL_CAP = 6144;       // keys of a bucket sorted in shared memory
constexpr uint32_t DL_CAP_P2 = 8192;    // the bitonic network's size for DL_CAP keys
constexpr int DL_ITEMS = DL_CAP / DL_THREADS;
constexpr uint32_t DL_SUB_BITS = 12, DL_SUB = 1u << DL_SUB_BITS;
constexpr uint32_t DL_RUN_MAX = 48;     // longest run ranked by comparing its members
constexpr int DL_SPT = DL_SUB / DL_THREADS;

// The bucket of a key before which there are pre others (below 2^24) is the high word
// of pre times depth_step(...): pre / s rounded down, for s keys a bucket.  A bucket
// holds at most s keys and one bin more (s_max: the warps' largest bins), which has to
// fit its CTA.  Half of a bucket's time does not depend on its keys (sub-bins, scans,
// barriers), so the fewest whole rounds of k_depth_local's CTAs with buckets of up to
// DP_KEYS_MAX are shared out evenly, and past DP_ROUNDS rounds the buckets are full.
// Depth order of the city's frames with buckets of 2048 keys and as here: 5.1M visible
// 114 and 103 us, 2.9M 70 and 64, 1.4M 42 and 39, 0.94M 35 and 31, 0.67M 31 and 28.
__device__ __forceinline__ uint32_t depth_step(uint32_t n, const uint32_t* s_max) {
    const uint32_t ctas = min(gridDim.x, DP_CTAS);
    if (n < ctas * DP_KEYS_MIN) return 0xFFFFFFFFu / DP_KEYS_MIN + 1u;
    uint32_t most = 8u;  // for the rounding
#pragma unroll
    for (int w = 0; w < DP_THREADS / 32; ++w) most = max(most, s_max[w] + 8u);
    const uint32_t full = min(max(DL_CAP - min(most, DL_CAP), DP_KEYS_MAX / 2), DP_KEYS_MAX);
    uint32_t slots = ctas;
    while (slots < DP_ROUNDS * ctas && n > slots * full) slots += ctas;
    const uint32_t s = n > slots * full ? full : n / slots + 1u;
    return 0xFFFFFFFFu / s + 1u;  // 2^32 / s, rounded up
}

uint32_t depth_bucket_cap(uint32_t cap_vis) {
    return std::max(DP_ROUNDS * DP_CTAS, cap_vis / (DP_KEYS_MAX / 2)) + 2u;
}

__global__ void __launch_bounds__(DP_THREADS, 2) k_depth_part(const uint32_t* __restrict__ depth,
                                                              const uint32_t* __restrict__ ntile, uint32_t cap,
                                                              const uint32_t* __restrict__ bins,
                                                              uint2* __restrict__ bstart,
                                                              unsigned long long* __restrict__ cursor,
                                                              uint2* __restrict__ part, uint32_t cap_buckets,
                                                              Counters* __restrict__ ctr,
                                                              const FrameParams* __restrict__ fp) {
    pdl_wait();
    extern __shared__ uint32_t sm[];
    uint16_t* s_bucket = reinterpret_cast<uint16_t*>(sm);  // [DEPTH_BINS] bucket of each bin
    uint32_t* s_start = sm + DEPTH_BINS / 2;               // [nb + 1] first position of each bucket
    uint32_t* s_base = s_start + cap_buckets + 1;          // [nb] keys of this tile, then their first position
    uint32_t* s_slot = s_base + cap_buckets;               // [nb] candidate slots of this tile
    __shared__ uint32_t s_scan[DP_THREADS / 32];
    __shared__ uint32_t s_last[DP_THREADS], s_max[DP_THREADS / 32];
    const uint32_t t = threadIdx.x;
    const uint32_t n = min(ctr->n_front, cap);
    // contiguous chunks, whole rows of DP_THREADS entries
    uint32_t chunk = (n + gridDim.x - 1) / gridDim.x;
    chunk = max((chunk + DP_THREADS - 1) / DP_THREADS, 2u) * DP_THREADS;
    const uint32_t first = blockIdx.x * chunk;
    if (blockIdx.x == 0 && t == 0 && ctr->n_front > MAX_RANKS) atomicOr(&ctr->flags, F_OVF_VIS);
    if (blockIdx.x != 0 && first >= n) return;
    const uint32_t end = min(first + chunk, n);
    const DepthMap map = fp->depth;
    uint32_t key[DP_ITEMS];  // the first tile's keys are in flight during the scan of the bins
#pragma unroll
    for (int k = 0; k < DP_ITEMS; ++k) {
        const uint32_t i = first + k * DP_THREADS + t;
        key[k] = i < end ? depth[i] : NONE;
    }
    uint32_t total, nb;
    {
        uint32_t c[DP_BPT];
#pragma unroll
        for (int k = 0; k < DP_BPT / 4; ++k) {
            const uint4 v = reinterpret_cast<const uint4*>(bins)[t * (DP_BPT / 4) + k];
            c[4 * k] = v.x; c[4 * k + 1] = v.y; c[4 * k + 2] = v.z; c[4 * k + 3] = v.w;
        }
        uint32_t sum = 0, most = 0;
#pragma unroll
        for (int k = 0; k < DP_BPT; ++k) {
            sum += c[k];
            most = max(most, c[k]);
        }
        most = __reduce_max_sync(0xFFFFFFFFu, most);
        if (lane_id() == 0) s_max[t >> 5] = most;
        s_last[t] = c[DP_BPT - 1];
        uint32_t pre = block_excl_scan<DP_THREADS / 32>(sum, s_scan, &total);  // (and a barrier)
        const uint32_t step = depth_step(total, s_max);
        nb = min(__umulhi(total, step) + 1u, cap_buckets);
        if (blockIdx.x == 0 && t == 0) ctr->depth_nb = nb;
        // bucket ids above the previous bin's start at this bin
        uint32_t id = t == 0 ? NONE : min(__umulhi(pre - s_last[t - 1], step), nb - 1u);  // NONE + 1 == 0
#pragma unroll
        for (int k = 0; k < DP_BPT; ++k) {
            const uint32_t b = min(__umulhi(pre, step), nb - 1u);
            s_bucket[t * DP_BPT + k] = (uint16_t)b;
            while (id != b) {
                s_start[++id] = pre;
                if (blockIdx.x == 0) bstart[id] = make_uint2(pre, t * DP_BPT + k);
            }
            pre += c[k];
        }
        if (t == DP_THREADS - 1)
            while (id != nb) {
                s_start[++id] = total;
                if (blockIdx.x == 0) bstart[id] = make_uint2(total, DEPTH_BINS);
            }
    }
    for (uint32_t b = t; b < nb; b += DP_THREADS) s_base[b] = s_slot[b] = 0u;
    __syncthreads();
    if (blockIdx.x == 0) {
        bool skew = false;
        for (uint32_t b = t; b < nb; b += DP_THREADS) skew = skew || s_start[b + 1] - s_start[b] > DL_CAP;
        if (skew) atomicOr(&ctr->flags, F_SORT_SKEW);
    }
    for (uint32_t base = first;;) {
        uint32_t at[DP_ITEMS];         // bucket << 13 | place in this tile's share of it
        uint32_t cnt[DP_ITEMS / 4];    // slot counts, saturated at 255
#pragma unroll
        for (int k = 0; k < DP_ITEMS / 4; ++k) cnt[k] = 0u;
#pragma unroll
        for (int k = 0; k < DP_ITEMS; ++k) {
            const uint32_t i = base + k * DP_THREADS + t;
            at[k] = NONE;
            if (i < end && key[k] != NONE) {  // culled entries carry all ones
                const uint32_t b = s_bucket[depth_bin(map, key[k])];
                const uint32_t c = ntile[i];
                at[k] = (b << 13) | atomicAdd(&s_base[b], 1u);
                if (c <= DP_FEW_SLOTS) atomicAdd(&s_slot[b], c);
                else atomicAdd(&cursor[b], (unsigned long long)c << DP_KEY_BITS);
                cnt[k / 4] |= min(c, 255u) << (8 * (k % 4));
            }
        }
        __syncthreads();
        for (uint32_t b = t; b < nb; b += DP_THREADS) {
            const uint32_t c = s_base[b];
            if (c) {
                const unsigned long long add = (unsigned long long)s_slot[b] << DP_KEY_BITS | c;
                s_base[b] = s_start[b] + ((uint32_t)atomicAdd(&cursor[b], add) & ((1u << DP_KEY_BITS) - 1u));
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < DP_ITEMS; ++k) {
            if (at[k] != NONE) {
                const uint32_t i = base + k * DP_THREADS + t;
                const uint32_t pos = s_base[at[k] >> 13] + (at[k] & 8191u);
                part[pos] = make_uint2(key[k], (i << 8) | ((cnt[k / 4] >> (8 * (k % 4))) & 255u));
            }
        }
        base += DP_TILE;
        if (base >= end) break;
        __syncthreads();
        for (uint32_t b = t; b < nb; b += DP_THREADS) s_base[b] = s_slot[b] = 0u;
#pragma unroll
        for (int k = 0; k < DP_ITEMS; ++k) {
            const uint32_t i = base + k * DP_THREADS + t;
            key[k] = i < end ? depth[i] : NONE;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__global__ void __launch_bounds__(DL_THREADS, 2) k_depth_local(const uint2* __restrict__ part,
                                                               const uint2* __restrict__ bstart,
                                                               const unsigned long long* __restrict__ cursor,
                                                               const uint32_t* __restrict__ ntile, uint32_t cap_vis,
                                                               uint32_t* __restrict__ order,
                                                               uint32_t* __restrict__ off,
                                                               uint32_t* __restrict__ owner, uint64_t cap_pairs,
                                                               Counters* __restrict__ ctr,
                                                               const FrameParams* __restrict__ fp) {
    pdl_wait();
    extern __shared__ uint2 s_kv[];                                  // [DL_CAP] the bucket by sub-bin, then first slots
    uint32_t* s_off = reinterpret_cast<uint32_t*>(s_kv);
    uint32_t* s_sub = reinterpret_cast<uint32_t*>(s_kv + DL_CAP);    // [DL_SUB + 1] counts, then first places
    uint4* s_sub4 = reinterpret_cast<uint4*>(s_sub);
    uint32_t* s_fin = s_sub + DL_SUB + 4;                            // [DL_CAP] index << 8 | slots, in order
    __shared__ uint32_t s_scan[DL_WARPS], s_scan2[DL_WARPS];
    __shared__ unsigned long long s_sum[DL_WARPS];
    const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5;
    if (ctr->flags & F_SORT_SKEW) return;
    const DepthMap map = fp->depth;
    const uint32_t n_vis = min(ctr->n_vis, cap_vis);
    const uint32_t nb = ctr->depth_nb;
    const uint32_t cap_owner = (uint32_t)(cap_pairs / EMIT_SLOTS) + 1u;
    auto slots_of = [&](uint32_t v) -> uint32_t { return (v & 255u) < 255u ? v & 255u : ntile[v >> 8]; };
#pragma unroll
    for (int k = 0; k < DL_SPT / 4; ++k) s_sub4[k * DL_THREADS + t] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    unsigned long long slots = 0ull;  // candidate slots of the buckets before b
    uint32_t seen = 0;
    for (uint32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        const uint2 bs = bstart[b], be = bstart[b + 1];  // (first position, first bin)
        const uint32_t start = bs.x, n = min(be.x - bs.x, DL_CAP);
        if (n == 0u && b + 1u < nb) continue;
        // sub-bins: equal steps of the bin coordinate over the bucket's bins
        const float c0 = (float)bs.y, cs = __fdividef((float)DL_SUB, (float)max(be.y - bs.y, 1u));
        auto sub_of = [&](uint32_t key) -> uint32_t {
            return min(__float2uint_rz(__fmul_rn(__fsub_rn(depth_coord(map, key), c0), cs)), DL_SUB - 1u);
        };
        uint2 e[DL_ITEMS];
        uint32_t place[DL_ITEMS];  // sub-bin << 16 | place in it, in any order
#pragma unroll
        for (int k = 0; k < DL_ITEMS; ++k) {
            const uint32_t j = k * DL_THREADS + t;
            if (k * DL_THREADS >= n) break;
            if (j < n) e[k] = part[start + j];
        }
        unsigned long long sum = 0ull;
        for (uint32_t p = seen + t; p < b; p += DL_THREADS) sum += cursor[p] >> DP_KEY_BITS;
        seen = b;
#pragma unroll
        for (int k = 0; k < DL_ITEMS; ++k) {
            if (k * DL_THREADS >= n) break;
            if (k * DL_THREADS + t < n) {
                const uint32_t sub = sub_of(e[k].x);
                place[k] = sub << 16 | atomicAdd(&s_sub[sub], 1u);
            }
        }
        sum = warp_sum64(sum);
        if (lane == 0) s_sum[warp] = sum;
        __syncthreads();
        // first place of each sub-bin
        bool longrun = false;
        {
            uint32_t c[DL_SPT], s = 0, total;
#pragma unroll
            for (int k = 0; k < DL_SPT / 4; ++k) {
                const uint4 q = s_sub4[DL_SPT / 4 * t + k];
                c[4 * k] = q.x; c[4 * k + 1] = q.y; c[4 * k + 2] = q.z; c[4 * k + 3] = q.w;
            }
#pragma unroll
            for (int k = 0; k < DL_SPT; ++k) {
                longrun = longrun || c[k] > DL_RUN_MAX;
                s += c[k];
            }
            uint32_t pre = block_excl_scan<DL_WARPS>(s, s_scan, &total);
#pragma unroll
            for (int k = 0; k < DL_SPT / 4; ++k) {
                uint4 q;
                q.x = pre; pre += c[4 * k];
                q.y = pre; pre += c[4 * k + 1];
                q.z = pre; pre += c[4 * k + 2];
                q.w = pre; pre += c[4 * k + 3];
                s_sub4[DL_SPT / 4 * t + k] = q;
            }
            if (t == 0) s_sub[DL_SUB] = n;
        }
#pragma unroll
        for (int w = 0; w < DL_WARPS; ++w) slots += s_sum[w];
        longrun = __syncthreads_or(longrun);
#pragma unroll
        for (int k = 0; k < DL_ITEMS; ++k) {
            if (k * DL_THREADS >= n) break;
            if (k * DL_THREADS + t < n) s_kv[s_sub[place[k] >> 16] + (place[k] & 0xFFFFu)] = e[k];
        }
        __syncthreads();
        if (!longrun) {
            // the members of a run (a sub-bin) rank themselves by (key, index)
            for (uint32_t j = t; j < n; j += DL_THREADS) {
                const uint2 kv = s_kv[j];
                const uint32_t sub = sub_of(kv.x);
                const uint32_t r0 = s_sub[sub], r1 = s_sub[sub + 1];
                uint32_t at = r0;
                if (r1 - r0 > 1u)
                    for (uint32_t r = r0; r < r1; ++r) {
                        const uint2 o = s_kv[r];
                        at += (o.x < kv.x || (o.x == kv.x && o.y < kv.y)) ? 1u : 0u;
                    }
                s_fin[at] = kv.y;
            }
        } else {
            // many equal keys: a bitonic network over (key, index), padded with all ones
            uint32_t p2 = 1;
            while (p2 < n) p2 <<= 1;  // at most DL_CAP_P2: the padding may cover s_sub, which is done with
            for (uint32_t j = n + t; j < p2; j += DL_THREADS) s_kv[j] = make_uint2(NONE, NONE);
            for (uint32_t k = 2; k <= p2; k <<= 1)
                for (uint32_t d = k >> 1; d > 0; d >>= 1) {
                    __syncthreads();
                    for (uint32_t c = t; c < p2 / 2; c += DL_THREADS) {
                        const uint32_t i = 2u * c - (c & (d - 1u)), j = i + d;
                        const uint2 x = s_kv[i], y = s_kv[j];
                        const bool gt = x.x > y.x || (x.x == y.x && x.y > y.y);
                        if (gt == ((i & k) == 0u)) {
                            s_kv[i] = y;
                            s_kv[j] = x;
                        }
                    }
                }
            __syncthreads();
            for (uint32_t j = t; j < n; j += DL_THREADS) s_fin[j] = s_kv[j].y;
        }
        __syncthreads();
        // first slots: each thread an odd number of neighbours (no bank conflicts)
        const uint32_t per = ((n + DL_THREADS - 1u) / DL_THREADS) | 1u, jb = t * per, je = min(jb + per, n);
        uint32_t mine = 0, unused;
        for (uint32_t j = jb; j < je; ++j) mine += slots_of(s_fin[j]);
        uint32_t run = (uint32_t)slots + block_excl_scan<DL_WARPS>(mine, s_scan2, &unused);
        for (uint32_t j = jb; j < je; ++j) {
            const uint32_t c = slots_of(s_fin[j]);
            s_off[j] = run;
            emit_owner(owner, cap_owner, run, c, start + j);
            run += c;
        }
#pragma unroll
        for (int k = 0; k < DL_SPT / 4; ++k) s_sub4[k * DL_THREADS + t] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        for (uint32_t j = t; j < n; j += DL_THREADS) {
            order[start + j] = s_fin[j] >> 8;
            off[start + j] = s_off[j];
        }
        if (b == nb - 1u && t == 0) {
            const unsigned long long ns = slots + (cursor[b] >> DP_KEY_BITS);
            off[n_vis] = (uint32_t)ns;  // (past 2^32 these wrap, and the emission leaves the frame alone)
            ctr->n_cand = ns;
        }
        // (the next bucket writes s_kv and s_fin only after barriers that follow these reads)
    }
}

size_t depth_local_smem() { return DL_CAP * sizeof(uint2) + (DL_SUB + 4 + DL_CAP) * sizeof(uint32_t); }
static_assert(DL_CAP * 8 + (DL_SUB + 4) * 4 >= DL_CAP_P2 * 8, "the bitonic network fits in s_kv and s_sub");
size_t depth_part_smem(uint32_t cap_buckets) {
    return DEPTH_BINS * sizeof(uint16_t) + (3 * (size_t)cap_buckets + 1) * sizeof(uint32_t);
}

cudaError_t depth_sort_init() {
    cudaError_t e = cudaFuncSetAttribute(k_depth_local, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)depth_local_smem());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_depth_part, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)depth_part_smem(depth_bucket_cap(MAX_RANKS)));
    return e;
}

void launch_depth_sort(const VisBuffers& vis, uint32_t cap_vis, const uint32_t* bins, uint2* bstart,
                       unsigned long long* cursor, uint2* part, uint32_t* order, uint32_t* slot_off,
                       uint32_t* owner, uint64_t cap_pairs, Counters* ctr, const FrameParams* fp, int sms,
                       cudaStream_t s) {
    const uint32_t cap = cap_vis < MAX_RANKS ? cap_vis : MAX_RANKS;
    const uint32_t cb = depth_bucket_cap(cap);
    launch_ks(k_depth_part, 2 * sms, DP_THREADS, depth_part_smem(cb), s, (const uint32_t*)vis.depth,
              (const uint32_t*)vis.ntile, cap, bins, bstart, cursor, part, cb, ctr, fp);
    launch_ks(k_depth_local, 2 * sms, DL_THREADS, depth_local_smem(), s, (const uint2*)part, (const uint2*)bstart,
              (const unsigned long long*)cursor, (const uint32_t*)vis.ntile, cap, order, slot_off, owner, cap_pairs, ctr,
              fp);
}

}  // namespace vgr
