// k_blend.cu -- front-to-back alpha blending per 16x16 tile (paper
// Sec. 3.1 'Rasterization', Eq. 3) with the preemptive log-domain test of
// Sec. 4.2 (Eq. 4) in front of the exponential.
//
// A tile of T x T pixels (T = 8, 16 or 32, a tuning knob) is T T / 32
// strips of 32 / T rows x T columns; one warp shades one strip, one pixel per
// lane (k_blend), or half as many strips with two pixels per lane (k_blend_wide,
// for launches with many strips).  The kernels are persistent: their CTAs (a few
// per SM) take tiles one at a time from a work list ordered heaviest first --
// the tiles of one view, or of every view of a batch -- their first by block
// index, then through a global counter, and the CTA's warps
// claim the strips of the CTA's tiles from a shared counter, so a warp that
// finishes a light strip moves on to the next strip at once instead of idling
// until its tile's heaviest strip is done, and the strips of a tile run on
// one SM, sharing its pair values and records through L1.
//
// Each pair value carries the Gaussian's index in the in-front arrays and its
// row mask in the tile (set by the emission from the footprint box: outside
// the box rho < ln alpha* - ln theta holds with a margin, so a pair whose box
// misses the strip's rows would fail the Eq. 4 test at every one of its
// pixels); within a tile the pairs are in depth order.  The warp scans its
// tile's pair values (coalesced, a batch ahead), queues those with its row
// bit in a ring, and copies the 48-byte records (mean, conic, threshold,
// opacity, colour) of DEPTH queued hits at a time with cp.async into its own
// double-buffered slice of shared memory; the copies of the next chunk are in
// flight while the current one is walked, four records at a time: their reads
// and exponentials are independent, and only the transmittance runs through them
// in order.  Before the walk each lane rewrites its
// staged records for the strip's rows (the row offsets of the mean folded
// into the conic terms), so a pixel evaluates rho with one subtraction and
// two FMAs.  Records are read only for the pairs a strip needs, and the warps
// of a CTA, working on the strips of the same tiles, share them through L1.
// A warp leaves a strip when its 32 pixels have stopped; tiles crossing the
// horizon (tens of thousands of small distant Gaussians, each reaching one or
// two rows) cost each strip a scan of 4-byte values and a fraction of the
// records.  Per pixel:
//   rho   = A dx^2 + B dx dy + C dy^2      (A = -a/2, B = -b, C = -c/2)
//   skip if rho < ln alpha* - ln theta     (Eq. 4: alpha < alpha*, no exp)
//   alpha = min(0.99, theta e^rho)         (Eq. 3)
//   T'    = T (1 - alpha); stop when T' < 1e-4 (this Gaussian excluded)
//   C    += alpha T rgb; T = T'
// (the exact mode takes the same test and alpha in base 2 with ln theta
// folded into the exponent, see blend_prepare).  Modes: canonical (every
// record at every pixel of the tile, alpha first, then the alpha* test; for
// the filtered-vs-unfiltered comparison; its row masks are all ones) and the
// Eq. 5 lookup table for e^rho.  DEPTH (hits staged per chunk: 16, 32 or 48)
// and T are tuning knobs; the image does not depend on them.
//
// What bounds it: large images by their instructions (issue slots 75 % busy),
// small ones by the chunks of the longest strips (a horizon tile's 2000 to 3500
// hits).  Groups of four records, first tiles dealt out, two pixels per lane and
// parts of 32-pixel tiles as items of their own took the blend from 110 to 81 us
// (1M-leaf box, 1080p), 184 to 165 (city, 1080p), 347 to 156 (1440p, 32-pixel
// tiles), 81 to 48 and 56 (640 x 360 and 320 x 180 city views), 312 to 208
// (canonical mode, 960 x 540); that mode's pass over the staged records in order
// took it to 143.
#include <atomic>

#include "vgr_internal.cuh"
#include "vgr_launch.h"

namespace vgr {

constexpr int BL_THREADS = 256;          // 8 warps: a warp shades one strip of 32 pixels at a time
constexpr int BL_WARPS = BL_THREADS / 32;
constexpr int BL_SCAN = 128;   // pair values scanned per batch (4 per lane, loaded one batch ahead)
constexpr int BL_RING = 256;   // a warp's queue of pair values
constexpr int BL_GROUP = 4;    // records a pixel evaluates at a time
constexpr int BL_MIN_CTAS = 4; // resident CTAs per SM the register budget is set for (up to 64 registers)
// resident CTAs per SM of k_blend by tile side: with three (80 registers) a group's
// reads and the next group's slots are in flight together; strips of 4 rows read
// two words per record and are better off with four CTAs and neither
constexpr int bl_narrow_ctas(int tile) { return tile == 8 ? 4 : 3; }
constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t WORK_TILE_BITS = 20;  // work item = view << 20 | tile
constexpr uint32_t WORK_TILE_MASK = (1u << WORK_TILE_BITS) - 1u;

struct BlendPixel {
    float fxp;
    float T, cr, cg, cb;
    bool done;
    uint32_t contribs;
};

constexpr float LOG2E = 1.4426950408889634f;
constexpr float LOG2_ALPHA_MIN = -7.9943534368588578f;  // log2(1/255)

// A staged record, rewritten for the strip's SR pixel rows (dy_r the offset of
// the mean from the centre of row r):
//   X = (u, A, thr, theta),  R_r = (B dy_r, C dy_r^2)
// so that at a pixel of row r, dx = u - x:  rho = (A dx + B dy_r) dx + C dy_r^2,
// one subtraction and two FMAs (A = -a/2, B = -b, C = -c/2).  The exact mode
// works in base 2 with the opacity folded in: A, B, C scaled by log2 e and
// log2 theta added to the constant term, so that
//   rho' = (A' dx + B' dy_r) dx + (C' dy_r^2 + log2 theta) = log2(theta e^rho),
// Eq. 4 becomes rho' >= log2 alpha* (one constant) and Eq. 3 alpha =
// min(0.99, 2^rho'): X = (u, A', -, -).  R_0, R_1 replace the raw second
// record half in b; rows 2 and 3 (strips of 4 rows) go to b2.
//
// Returns the record's pixel mask in the strip: bit q (pixel q = row q / T,
// column q % T) is set when q lies in the footprint box, the axis-aligned
// box of {rho >= ln alpha* - ln theta - 2e-3} (with a margin) that preprocess
// stored as FP16 half-extents rounded up.  Outside it the Eq. 4 test fails,
// so the pixel need not look at the record.  The canonical mode (no Eq. 4
// before Eq. 3) and 'full' mark every pixel.
template <int MODE, int SR, int T>
__device__ __forceinline__ uint32_t blend_prepare(float4& a, float4& b, float4& b2, float theta, float row0,
                                                  float col0, bool full) {
    uint32_t pmask = 0xFFFFFFFFu;
    if (MODE != 1 && !full) {
        const uint32_t hw = __float_as_uint(b.w);
        const float by = __half2float(__ushort_as_half((unsigned short)(hw & 0xFFFFu))) + 0.01f;
        const float bx = __half2float(__ushort_as_half((unsigned short)(hw >> 16))) + 0.01f;
        // columns c with |col0 + c - u| <= bx, and rows of the strip likewise (conversions round and saturate)
        const int c0 = max(__float2int_ru(a.x - bx - col0), 0), c1 = min(__float2int_rd(a.x + bx - col0), T - 1);
        const int r0 = max(__float2int_ru(a.y - by - row0), 0), r1 = min(__float2int_rd(a.y + by - row0), SR - 1);
        pmask = 0u;
        if (c0 <= c1) {
            const uint32_t cols = (0xFFFFFFFFu >> (31 - c1)) & (0xFFFFFFFFu << c0);
#pragma unroll
            for (int r = 0; r < SR; ++r)
                if (r >= r0 && r <= r1) pmask |= cols << (r * T);
        }
    }
    float Bc, Cc, add;
    if (MODE == 0) {
        Bc = a.w * LOG2E;
        Cc = b.x * LOG2E;
        add = (LN_ALPHA_MIN - b.y) * LOG2E;  // b.y = ln alpha* - ln theta: log2 theta
    } else {
        Bc = a.w;
        Cc = b.x;
        add = 0.f;
    }
    const float v = a.y;
    float R[2 * SR];
#pragma unroll
    for (int r = 0; r < SR; ++r) {
        const float dy = v - (row0 + (float)r);
        R[2 * r] = Bc * dy;
        R[2 * r + 1] = MODE == 0 ? fmaf(Cc * dy, dy, add) : (Cc * dy) * dy;
    }
    if (MODE == 0 && SR <= 2) {  // one float4 per row: (u, A', B' dy_r, C' dy_r^2 + log2 theta)
        const float u = a.x, Ap = a.z * LOG2E;
        a = make_float4(u, Ap, R[0], R[1]);
        if (SR == 2) b = make_float4(u, Ap, R[2 % (2 * SR)], R[3 % (2 * SR)]);
        return pmask;
    }
    const float4 X = MODE == 0 ? make_float4(a.x, a.z * LOG2E, 0.f, 0.f) : make_float4(a.x, a.z, b.y, theta);
    a = X;
    b = make_float4(R[0], R[1], SR > 1 ? R[2 % (2 * SR)] : 0.f, SR > 1 ? R[3 % (2 * SR)] : 0.f);
    if (SR > 2) b2 = make_float4(R[4 % (2 * SR)], R[5 % (2 * SR)], R[6 % (2 * SR)], R[7 % (2 * SR)]);
    return pmask;
}

// Transpose of the 32 x 32 bit matrix held by a warp, lane l holding row l:
// afterwards lane q holds column q (bit l = bit q of lane l's row).  Five
// exchange steps, each swapping the off-diagonal blocks of half the size.
// The two larger ones move whole bytes.
template <uint32_t J, uint32_t M>
__device__ __forceinline__ uint32_t transpose_step(uint32_t x, uint32_t lane) {
    const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, J);
    const uint32_t up = lane & J;                      // 0: keep M and take the partner's M shifted up; J: the others
    const uint32_t m = __funnelshift_l(M, M, up);      // M, or ~M
    return (x & m) | (__funnelshift_l(y, y, J - 2u * up) & ~m);
}
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x) {
    const uint32_t lane = lane_id();
    x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 16), (lane & 16u) ? 0x3276u : 0x5410u);
    x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 8), (lane & 8u) ? 0x3715u : 0x6240u);
    x = transpose_step<4, 0x0F0F0F0Fu>(x, lane);
    x = transpose_step<2, 0x33333333u>(x, lane);
    return transpose_step<1, 0x55555555u>(x, lane);
}

// The staged slot of the foremost record in mm (bit 31 - l: slot 32 q + l), which
// leaves mm; slot DEPTH when there is none: a record that no pixel takes
// (dummy_part), so that a group of records needs no flags.
template <int DEPTH>
__device__ __forceinline__ uint32_t next_slot(uint32_t& mm, int q) {
    const uint32_t c = __clz(mm);
    mm &= ~(0x80000000u >> (c & 31u));
    if (DEPTH == 32) return c;
    return c < 32u ? 32u * q + c : (uint32_t)DEPTH;
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Opacity of a record at a pixel (Eq. 3), and whether it takes part (Eq. 4, or
// the alpha* test of the canonical mode).
template <int MODE>
__device__ __forceinline__ bool blend_alpha(const float4& X, float rho, const float* s_lut, uint32_t m, float lut_scale,
                                            float& alpha) {
    if (MODE == 0) {  // base 2, opacity folded in (see blend_prepare)
        alpha = fminf(ALPHA_MAX, ex2_approx(rho));
        return !(rho < LOG2_ALPHA_MIN);
    } else if (MODE == 1) {  // canonical: Eq. 3, then the alpha* test
        alpha = fminf(ALPHA_MAX, X.w * ex2_approx(rho * LOG2E));
        return !(alpha < ALPHA_MIN);
    } else {
        // Eq. 5: nearest of m intervals over [-5.55, 0] (the index is clamped for records that fail Eq. 4 too)
        const uint32_t idx = min(m, (uint32_t)__float2int_rn(rho * lut_scale));
        alpha = fminf(ALPHA_MAX, X.w * s_lut[idx]);
        return !(rho < X.z);
    }
}

// The staged X of slot i: only (u, A') in the exact mode.
template <int MODE>
__device__ __forceinline__ float4 load_x(const float4* wA, uint32_t i) {
    if (MODE == 0) {
        const float2 x = reinterpret_cast<const float2*>(wA)[2 * i];
        return make_float4(x.x, x.y, 0.f, 0.f);
    }
    return wA[i];
}

__device__ __forceinline__ float blend_rho(const BlendPixel& p, const float4& X, const float2& R) {
    const float dx = X.x - p.fxp;
    return fmaf(fmaf(X.y, dx, R.x), dx, R.y);
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// A warp's current item: where its strip reads and writes, copied from the
// view's frame parameters into shared memory when the warp takes the item and
// read from there at each use, so that neither the pointers nor the output
// location occupy registers during the walk; and the warp's blend statistics.
struct WarpItem {
    const uint32_t* pair_val;
    const float4* rec;
    const float4* rgb;
    float* image;
    float* host_image;
    Counters* ctr;           // statistics of the view below
    unsigned long long evals, contribs;
    uint32_t at;             // index of the strip's first pixel
    uint32_t width;          // image width
    uint32_t nx, ny;         // columns and rows of the strip inside the image
    uint32_t view;
};

// A CTA's claims: its warps take (slot, strip) items in order, a slot being a
// tile of the work list, or a part of one of at most BL_WARPS strips (so that a
// heavy tile of 32 x 32 pixels is not left to one CTA), claimed from the global
// counter and published in a ring of 4 entries.
constexpr int slot_strips(int ns) { return ns < BL_WARPS ? ns : BL_WARPS; }
struct ClaimRing {
    uint32_t claim;                        // next (slot, strip) item
    uint32_t tile[4], tag[4], read[4];     // per entry: the slot's global number, slot + 1, strips that have read it
    template <int TILE_STRIPS>
    __device__ __forceinline__ void init() {
        if (threadIdx.x == 0) claim = 0u;
        if (threadIdx.x < 4) {
            tag[threadIdx.x] = 0u;
            read[threadIdx.x] = slot_strips(TILE_STRIPS) - 1;
        }
    }
};

// The next (tile, strip) item of this warp's CTA: idx is the tile's place in the
// work list.  The CTA's first slot is number 'first' (NONE: a claimed one), later
// ones are base + the global counter *next.  The warp that takes strip 0 of a
// slot claims and publishes it; the other strips' warps wait for it.  False: a
// wait ran out (F_SPIN_TIMEOUT).
// First slots by block index deal the heaviest tiles out to the SMs one by one
// (blocks go to the SMs in turn); claimed, they went to whichever CTAs came first,
// and the SMs that got several finished last (240 tiles of a 320 x 180 view:
// 82 us, dealt out 62).
template <int TILE_STRIPS>
__device__ __forceinline__ bool claim_item(ClaimRing& ring, uint32_t* next, uint32_t first, uint32_t base,
                                           const FrameParams* fp0, uint32_t& idx_out, uint32_t& strip_out) {
    constexpr uint32_t NS = slot_strips(TILE_STRIPS), PARTS = TILE_STRIPS / NS;
    volatile uint32_t* slot_tile = ring.tile;
    volatile uint32_t* slot_tag = ring.tag;
    volatile uint32_t* slot_read = ring.read;
    uint32_t idx = 0, strip = 0;
    bool timed_out = false;
    if (lane_id() == 0) {
        const uint32_t k = atomicAdd(&ring.claim, 1u);
        const uint32_t slot = k / NS, e = slot & 3u;
        strip = k % NS;
        uint32_t spins = 0;
        if (strip == 0) {
            while (slot_read[e] < NS - 1) {  // the entry's last readers
                if (++spins > SPIN_LIMIT) { timed_out = true; break; }
                __nanosleep(32);
            }
            idx = slot == 0u && first != NONE ? first : base + atomicAdd(next, 1u);
            slot_read[e] = 0u;
            slot_tile[e] = idx;
            __threadfence_block();
            slot_tag[e] = slot + 1u;
        } else {
            while (slot_tag[e] != slot + 1u) {
                if (++spins > SPIN_LIMIT) { timed_out = true; break; }
                __nanosleep(32);
            }
            __threadfence_block();
            idx = slot_tile[e];
            atomicAdd(&ring.read[e], 1u);
        }
        if (timed_out) atomicOr(&fp0->bl_ctr->flags, F_SPIN_TIMEOUT);
    }
    idx = __shfl_sync(FULL, idx, 0);
    idx_out = idx / PARTS;
    strip_out = __shfl_sync(FULL, strip, 0) + idx % PARTS * NS;
    return !__shfl_sync(FULL, (uint32_t)timed_out, 0);
}

// The record in slot DEPTH of every staged part: at any pixel rho is far below
// every threshold (and theta 0), in the layout that blend_prepare leaves.
template <int MODE, int SR>
__device__ __forceinline__ float4 dummy_part(int part) {
    constexpr float LOW = -1e30f;
    if (MODE == 0 && SR <= 2) return make_float4(0.f, 0.f, 0.f, LOW);
    return part == 0 ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(0.f, LOW, 0.f, LOW);
}

__device__ __forceinline__ void init_item(WarpItem& it) {
    it.ctr = nullptr;
    it.evals = it.contribs = 0ull;
    it.view = 0xFFFFFFFFu;
}

// Lane 0: the statistics of the warp's last view.
__device__ __forceinline__ void flush_item(volatile WarpItem& it) {
    if (it.ctr && it.evals) {
        atomicAdd(&it.ctr->pix_evals, (unsigned long long)it.evals);
        atomicAdd(&it.ctr->pix_contribs, (unsigned long long)it.contribs);
    }
    it.evals = it.contribs = 0ull;
}

// The launch's last CTA to finish (every CTA calls this at its end) writes the
// status of the launch's views -- the head of their counters and their cut sizes
// -- to pinned host memory, where the host reads it once the launch has completed.
__device__ __forceinline__ void finish_blend(uint32_t* done, const FrameParams* fp0, const FrameParams* const* fps,
                                             uint32_t n_views) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();  // this CTA's statistics and flags before its count
        s_last = atomicAdd(done, 1u) == gridDim.x - 1u;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    constexpr uint32_t HEAD = COUNTERS_HEAD / 4, W = HEAD + 2;
    for (uint32_t i = threadIdx.x; i < W * (fps ? n_views : 1u); i += BL_THREADS) {
        const FrameParams* fp = fps ? fps[i / W] : fp0;
        const uint32_t w = i % W;
        if (w < HEAD) fp->host_status[w] = __ldcg(reinterpret_cast<const uint32_t*>(fp->bl_ctr) + w);
        else fp->host_n_cut[w - HEAD] = __ldcg(fp->n_cut + (w - HEAD));
    }
}

// Lane 0: the warp's item, a strip of nrows rows of T columns at (x0, y0) of the view.
__device__ __forceinline__ void fill_item(volatile WarpItem& it, const FrameParams* fp, uint32_t view, uint32_t x0,
                                          uint32_t y0, uint32_t T, uint32_t nrows) {
    if (view != it.view) {
        flush_item(it);
        it.view = view;
        it.ctr = fp->bl_ctr;
    }
    it.pair_val = fp->bl_pair_val;
    it.rec = fp->bl_rec;
    it.rgb = fp->bl_rgb;
    it.image = fp->bl_image;
    it.host_image = fp->host_image;
    it.at = y0 * fp->width + x0;
    it.width = fp->width;
    it.nx = min(T, fp->width - x0);
    it.ny = y0 < fp->height ? min(nrows, fp->height - y0) : 0u;
}

// Bits p0 .. p1 (0 <= p0, p1 < 32; none if p1 < p0)
__device__ __forceinline__ uint32_t pair_range(int p0, int p1) {
    return p1 < p0 ? 0u : (0xFFFFFFFFu >> (31 - p1)) & (0xFFFFFFFFu << p0);
}

// The blend, for tiles of T x T pixels.  A strip is SR = 32 / T rows of T
// columns (one warp, one pixel per lane); a tile has NS = T T / 32 strips.  A
// pair's 8-bit row mask has one bit per MR = max(1, T / 8) rows, and strip s
// needs the bits of its rows.  Work: a CTA claims the next tile of the work
// list from the global counter 'next'; the strips of the CTA's tiles are
// claimed by its warps from a shared counter, in (slot, strip) order.  The
// warp that takes strip 0 of a slot claims that slot's tile and publishes it
// in a ring of 4 entries; the other strips' warps wait for it.  Before it
// reuses an entry the publishing warp waits until the entry's previous readers
// have read it.  Every wait is on a claim made earlier in the CTA's order, so
// none can close a cycle; each is still bounded and reports F_SPIN_TIMEOUT.
//
// The strips of one warp, tiles from place 0 up to n_work of the work list.
// sbuf: staged records, [buffer][part: 0 = record A / X, 1 = colour, 2.. = record
// B / row terms][warp][slot]; ring: the warp's queue of hit pair values (at a
// strip's end its pixels); pm: the staged records' pixel masks.
template <int MODE, int DEPTH, int T>
__device__ __forceinline__ void blend_strips(float4 (*sbuf)[2 + (32 / T > 2 ? 2 : 1)][BL_WARPS][DEPTH + 1],
                                             uint32_t* ring,
                                             uint32_t* pm, volatile WarpItem& it, ClaimRing& claims,
                                             const FrameParams* __restrict__ fp0,
                                             const FrameParams* const* __restrict__ fps,
                                             const uint32_t* __restrict__ work, uint32_t n_work, uint32_t* next,
                                             uint32_t first, uint32_t base, const float* s_lut, uint32_t m,
                                             float lut_scale, bool full_walk) {
    constexpr int SR = 32 / T;                    // rows per strip
    constexpr int NS = T * T / 32;                // strips per tile
    constexpr int MR = T >= 8 ? T / 8 : 1;        // rows per mask bit
    constexpr int SB = SR >= MR ? SR / MR : 1;    // mask bits of one strip
    constexpr int NP = 2 + (SR > 2 ? 2 : 1);      // staged parts: X, colour, row terms
    constexpr bool AHEAD = SR <= 2;               // the next group's slots are found while one is evaluated
    constexpr int RING = BL_RING;                 // < DEPTH queued + BL_SCAN appended never exceeds it
    static_assert(T == 8 || T == 16 || T == 32, "tile size 8, 16 or 32");
    static_assert(DEPTH % 16 == 0 && DEPTH <= 48, "staging depth: 16, 32 or 48 hits");
    static_assert(DEPTH + BL_SCAN <= RING, "ring too small");
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    for (;;) {
        uint32_t idx, strip;
        if (!claim_item<NS>(claims, next, first, base, fp0, idx, strip) || idx >= n_work)
            break;
        uint2 rg;
        float rlo, clo;
        uint32_t wbits;
        bool inside;
        {
            const uint32_t item = work[idx];
            const uint32_t view = item >> WORK_TILE_BITS, tile = item & WORK_TILE_MASK;
            const FrameParams* fp = fps ? fps[view] : fp0;
            const uint32_t W = fp->width, H = fp->height, TW = fp->tiles_x;
            const uint32_t x0 = (tile % TW) * T, y0 = (tile / TW) * T + SR * strip;
            if (lane == 0) fill_item(it, fp, view, x0, y0, (uint32_t)T, (uint32_t)SR);
            rg = fp->bl_ranges[tile];
            inside = x0 + lane % T < W && y0 + lane / T < H;
            wbits = ((1u << SB) - 1u) << (SR * strip / MR);
            rlo = (float)y0 + 0.5f;  // centre of the strip's first row
            clo = (float)x0 + 0.5f;  // and column
            __syncwarp();
        }
        BlendPixel p;
        p.fxp = (float)(lane % T + it.at % it.width) + 0.5f;
        p.T = 1.f;
        p.cr = p.cg = p.cb = 0.f;
        p.contribs = 0;
        p.done = !inside;
        uint32_t evals = 0;
        // The strip's pairs (those whose row mask names its rows, in depth
        // order) pass through a ring of pair values: the range is scanned
        // BL_SCAN values at a time (loaded one batch ahead), hits are appended,
        // and records are staged DEPTH hits at a time, so staging and the walk
        // run on full chunks however sparse the strip's hits are among the
        // tile's pairs.
        uint32_t head = 0, tail = 0;
        uint32_t bp = rg.x;  // first pair value of the pending batch
        uint32_t pend[BL_SCAN / 32];
        {
            const uint32_t* pv = it.pair_val;
#pragma unroll
            for (int g = 0; g < BL_SCAN / 32; ++g) {
                const uint32_t j = bp + 32u * g + lane;
                pend[g] = j < rg.y ? pv[j] : 0u;
            }
        }
        auto refill = [&]() {
            while (tail - head < (uint32_t)DEPTH && bp < rg.y) {
#pragma unroll
                for (int g = 0; g < BL_SCAN / 32; ++g) {
                    const uint32_t v = pend[g];
                    const bool hit = (v & wbits) != 0u;  // entries past the range hold 0
                    const uint32_t hits = __ballot_sync(FULL, hit);
                    if (hit) ring[(tail + __popc(hits & lanemask_lt())) & (RING - 1)] = v;
                    tail += __popc(hits);
                }
                bp += BL_SCAN;
                const uint32_t* pv = it.pair_val;
#pragma unroll
                for (int g = 0; g < BL_SCAN / 32; ++g) {
                    const uint32_t j = bp + 32u * g + lane;
                    pend[g] = j < rg.y ? pv[j] : 0u;
                }
            }
            __syncwarp();
        };
        // stage up to DEPTH queued hits into buffer buf; returns their number
        auto issue = [&](int buf) -> uint32_t {
            const uint32_t nh = min((uint32_t)DEPTH, tail - head);
            const float4* rR = it.rec;
            const float4* rC = it.rgb;
#pragma unroll
            for (int q = 0; q < (DEPTH + 31) / 32; ++q) {
                const uint32_t sl = 32u * q + lane;
                if (sl < nh) {
                    const uint32_t gi = ring[(head + sl) & (RING - 1)] >> 8;
                    cp_async16(&sbuf[buf][0][warp][sl], rR + 2 * (size_t)gi);
                    cp_async16(&sbuf[buf][2][warp][sl], rR + 2 * (size_t)gi + 1);
                    cp_async16(&sbuf[buf][1][warp][sl], rC + gi);
                }
            }
            cp_async_commit();
            head += nh;
            return nh;
        };
        refill();
        uint32_t nh_cur = issue(0);
        int buf = 0;
        while (nh_cur > 0) {
            if (__all_sync(FULL, p.done)) break;
            refill();
            const uint32_t nh_next = issue(buf ^ 1);  // the next chunk in flight during this walk
            cp_async_wait<1>();  // this chunk's copies (all but the newest group)
            __syncwarp();
            float4* wA = sbuf[buf][0][warp];
            const float4* wC = sbuf[buf][1][warp];
            const uint32_t nh = nh_cur;
#pragma unroll
            for (int q = 0; q < (DEPTH + 31) / 32; ++q) {
                const uint32_t sl = 32u * q + lane;
                if (MODE == 1) {
                    if (sl < nh) {
                        blend_prepare<MODE, SR, T>(wA[sl], sbuf[buf][2][warp][sl], sbuf[buf][NP - 1][warp][sl],
                                                   wC[sl].w, rlo, clo, true);
                    } else if (sl < (uint32_t)DEPTH) {  // read with the last group
#pragma unroll
                        for (int part = 0; part < NP; ++part) sbuf[buf][part][warp][sl] = dummy_part<MODE, SR>(part);
                    }
                } else if (sl < (uint32_t)DEPTH)  // each lane its own slots; empty slots reach no pixel
                    pm[sl] = sl < nh ? blend_prepare<MODE, SR, T>(wA[sl], sbuf[buf][2][warp][sl],
                                                                           sbuf[buf][NP - 1][warp][sl],
                                                                           MODE != 0 ? wC[sl].w : 0.f, rlo, clo,
                                                                           full_walk)
                                             : 0u;
            }
            __syncwarp();
            // the records that can reach this lane's pixel, as slot bits in
            // depth order from bit 31 down: the transpose of the records' pixel masks
            uint32_t reach[(DEPTH + 31) / 32];
#pragma unroll
            for (int q = 0; q < (DEPTH + 31) / 32 && MODE != 1; ++q) {
                const uint32_t sl = 32u * q + 31u - lane;
                reach[q] = warp_transpose32(sl < (uint32_t)DEPTH ? pm[sl] : 0u);
            }
            if (!p.done) {
                // this lane's row r = lane / T.  Exact mode with strips of one or two
                // rows: the row's whole record is the float4 of part 0 (row 0) or 2
                // (row 1), one load per evaluation.  Otherwise X of part 0 and the
                // row's terms: float2 (r & 1) of part 2 + r / 2.
                const uint32_t r = lane / T;
                const float4* wY = sbuf[buf][r == 0 ? 0 : 2][warp];
                const float2* wR = reinterpret_cast<const float2*>(sbuf[buf][2 + r / 2][warp]) + (r & 1u);
                auto load = [&](uint32_t i, float4& X, float2& R) {
                    if constexpr (MODE == 0 && SR <= 2) {
                        X = wY[i];
                    } else {
                        X = load_x<MODE>(wA, i);
                        R = wR[2 * i];
                    }
                };
                auto rho_of = [&](const float4& X, const float2& R) -> float {
                    if constexpr (MODE == 0 && SR <= 2) {
                        const float dx = X.x - p.fxp;
                        return fmaf(fmaf(X.y, dx, X.z), dx, X.w);
                    } else {
                        return blend_rho(p, X, R);
                    }
                };
                if constexpr (MODE == 1) {
                    // Every record at every pixel, alpha first: the slots in order, several
                    // records' reads and exponentials together.  Of those that pass the alpha*
                    // test (one in twenty) only the bit is kept, and the walk below evaluates
                    // them again: 960 x 540, 108M evaluations, 143 us; with the rest of the
                    // blend behind a branch per record 161, as straight code for groups 203.
                    static_assert(DEPTH == 32, "one word of slots");
                    constexpr uint32_t G = 8;
                    evals += nh;
                    reach[0] = 0u;
                    for (uint32_t i = 0; i < nh; i += G) {
                        uint32_t word = 0u;
#pragma unroll
                        for (uint32_t g = 0; g < G; ++g) {
                            float4 X;
                            float2 R;
                            float alpha;
                            load(i + g, X, R);
                            if (blend_alpha<MODE>(X, rho_of(X, R), s_lut, m, lut_scale, alpha)) word |= 0x80000000u >> g;
                        }
                        reach[0] |= word >> i;
                    }
                }
#pragma unroll
                for (int q = 0; q < (DEPTH + 31) / 32; ++q) {
                    uint32_t mm = reach[q];  // bit 31 - l: slot 32 q + l
                    // BL_GROUP records at a time: their reads, rho and exponentials are
                    // independent of one another and go out together; only the
                    // transmittance runs through them in order
                    if (MODE != 1) evals += __popc(mm);
                    uint32_t at[BL_GROUP], nat[BL_GROUP];
                    auto take = [&](uint32_t* slots) {
#pragma unroll
                        for (int g = 0; g < BL_GROUP; ++g) slots[g] = next_slot<DEPTH>(mm, q);
                    };
                    auto advance = [&]() {
                        if constexpr (AHEAD) {
#pragma unroll
                            for (int g = 0; g < BL_GROUP; ++g) at[g] = nat[g];
                        } else {
                            take(at);
                        }
                    };
                    take(at);
                    while (at[0] != (uint32_t)DEPTH) {
                        float alpha[BL_GROUP], Tg[BL_GROUP];
                        bool use[BL_GROUP];
                        const uint32_t left = mm;  // behind this group
                        if constexpr (AHEAD) {
                            float4 X[BL_GROUP];
                            float2 R[BL_GROUP];
#pragma unroll
                            for (int g = 0; g < BL_GROUP; ++g) load(at[g], X[g], R[g]);
                            take(nat);
#pragma unroll
                            for (int g = 0; g < BL_GROUP; ++g)
                                use[g] = blend_alpha<MODE>(X[g], rho_of(X[g], R[g]), s_lut, m, lut_scale, alpha[g]);
                        } else {
#pragma unroll
                            for (int g = 0; g < BL_GROUP; ++g) {
                                float4 X;
                                float2 R;
                                load(at[g], X, R);
                                use[g] = blend_alpha<MODE>(X, rho_of(X, R), s_lut, m, lut_scale, alpha[g]);
                            }
                        }
                        float Tr = p.T;
#pragma unroll
                        for (int g = 0; g < BL_GROUP; ++g) {
                            Tg[g] = Tr;
                            if (use[g]) Tr = Tr * (1.f - alpha[g]);
                        }
                        // T never rises, so a group that ends at or above T_MIN stops nowhere
                        int last = BL_GROUP;  // records of the group before the pixel stops
                        if (Tr < T_MIN) {
#pragma unroll
                            for (int g = BL_GROUP - 1; g >= 0; --g)  // the first whose T falls below
                                if (use[g] && Tg[g] * (1.f - alpha[g]) < T_MIN) last = g;
                            p.done = true;
                            // not evaluated: what is left of this word, and the group's after the stop
                            if (MODE != 1) evals -= __popc(left);
#pragma unroll
                            for (int g = 0; g < BL_GROUP; ++g) {
                                if (MODE != 1 && g > last && at[g] != (uint32_t)DEPTH) --evals;
                                if (MODE == 1 && g == last) evals -= nh - (at[g] + 1u);
                                if (g >= last) use[g] = false;
                                if (g == last) Tr = Tg[g];
                            }
                        }
#pragma unroll
                        for (int g = 0; g < BL_GROUP; ++g) {
                            const float4 C4 = wC[at[g]];
                            if (use[g]) {
                                const float w = alpha[g] * Tg[g];
                                p.cr = fmaf(w, C4.x, p.cr);
                                p.cg = fmaf(w, C4.y, p.cg);
                                p.cb = fmaf(w, C4.z, p.cb);
                                ++p.contribs;
                            }
                        }
                        p.T = Tr;
                        if (p.done) break;
                        advance();
                    }
                    if (p.done) break;
                }
            }
            __syncwarp();  // the walk is done with this buffer before it is refilled
            buf ^= 1;
            nh_cur = nh_next;
        }
        cp_async_wait<0>();  // the chunk staged ahead, if the strip stopped early
        const uint32_t cx = lane % T, cy = lane / T;
        float* const host_image = it.host_image;
        // a whole strip whose rows start 16-byte aligned (image width a multiple of
        // 4): its 32 pixels staged in shared memory and stored as float4, SR rows
        // of 3T/4 float4 each (long aligned bursts over the host link)
        const bool whole = it.nx == (uint32_t)T && it.ny == (uint32_t)SR && (it.width & 3u) == 0u &&
                           ((reinterpret_cast<uintptr_t>(host_image) & 15u) == 0u);
        if (whole) {
            float* s = reinterpret_cast<float*>(ring);  // 96 of its words
            s[3 * lane + 0] = p.cr;
            s[3 * lane + 1] = p.cg;
            s[3 * lane + 2] = p.cb;
            __syncwarp();
            constexpr int F4_ROW = 3 * T / 4;
            if (lane < 24) {  // 96 floats = 24 float4
                const uint32_t r = lane / F4_ROW, c4 = lane % F4_ROW;
                const float4 val = reinterpret_cast<const float4*>(s)[lane];
                const size_t at4 = ((size_t)it.at + (size_t)r * it.width) * 3 + 4u * c4;
                *reinterpret_cast<float4*>(it.image + at4) = val;
                if (host_image) *reinterpret_cast<float4*>(host_image + at4) = val;  // pinned host buffer
            }
            __syncwarp();
        } else if (cx < it.nx && cy < it.ny) {
            const size_t at = ((size_t)it.at + (size_t)cy * it.width + cx) * 3;
            float* o = it.image + at;
            o[0] = p.cr;
            o[1] = p.cg;
            o[2] = p.cb;
            if (host_image) {  // the caller's pinned host buffer, over the host link
                float* q = host_image + at;
                q[0] = p.cr;
                q[1] = p.cg;
                q[2] = p.cb;
            }
        }
        const uint32_t ev_w = __reduce_add_sync(FULL, evals), co_w = __reduce_add_sync(FULL, p.contribs);
        if (lane == 0) {
            it.evals = it.evals + ev_w;
            it.contribs = it.contribs + co_w;
        }
        __syncwarp();  // every lane is done with the item before lane 0 rewrites it
    }
}

template <int MODE, int DEPTH, int T>
__global__ void __launch_bounds__(BL_THREADS, bl_narrow_ctas(T)) k_blend(const FrameParams* __restrict__ fp0,
                                                                   const FrameParams* const* __restrict__ fps,
                                                                   const uint32_t* __restrict__ work,
                                                                   uint32_t n_work, uint32_t* __restrict__ next,
                                                                   uint32_t* __restrict__ done, uint32_t n_views) {
    pdl_wait();
    __shared__ __align__(16) float4 sbuf[2][2 + (32 / T > 2 ? 2 : 1)][BL_WARPS][DEPTH + 1];
    __shared__ __align__(16) uint32_t s_ring[BL_WARPS][BL_RING];
    __shared__ uint32_t s_pm[BL_WARPS][DEPTH];
    __shared__ float s_lut[MODE == 2 ? 260 : 1];
    __shared__ WarpItem s_item[BL_WARPS];
    __shared__ ClaimRing s_claims;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    uint32_t m = 0;
    float lut_scale = 0.f;
    s_claims.init<T * T / 32>();
    if (lane == 0) init_item(s_item[warp]);
    constexpr int NP = 2 + (32 / T > 2 ? 2 : 1);
    if (lane < 2 * NP) sbuf[lane / NP][lane % NP][warp][DEPTH] = dummy_part<MODE, 32 / T>(lane % NP);
    if (MODE == 2) {  // the table mode runs on one view at a time
        m = fp0->lut_size;
        lut_scale = -(float)m / 5.55f;
        for (uint32_t i = threadIdx.x; i <= m; i += BL_THREADS) s_lut[i] = fp0->bl_lut[i];
    }
    __syncthreads();
    blend_strips<MODE, DEPTH, T>(sbuf, s_ring[warp], s_pm[warp], s_item[warp], s_claims, fp0, fps, work, n_work, next,
                                 blockIdx.x, gridDim.x, s_lut, m, lut_scale,
                                 (fp0->test_hooks & VGR_HOOK_FULL_STRIP_WALK) != 0u);
    if (lane == 0) flush_item(s_item[warp]);
    finish_blend(done, fp0, fps, n_views);
}

// The same blend for launches with many strips: tiles with few pairs take strips
// of 64 pixels (64 / T rows), two neighbours of one row per lane, and a record
// read for the lane serves both.  The arithmetic of a pixel is that of k_blend,
// so the image is the same bit for bit.  Exact exponential, tiles of 16 or 32
// pixels.  What it saves is the work per strip that does not depend on its pixels
// (claim, parameters, ranges, queue, copies, store: 47 of 114 us on the 1M-leaf
// box at 1080p with 32-pixel strips) and a part of the records' preparation; what
// it costs is the length of a heavy tile's strips, so with 16-pixel tiles the
// first *n_heavy tiles of the work list (BL_HEAVY_CLASS and up) keep strips of 32
// pixels, claimed first.
// next[0] counts those, next[1] the others.
template <int DEPTH, int T>
__global__ void __launch_bounds__(BL_THREADS, BL_MIN_CTAS) k_blend_wide(const FrameParams* __restrict__ fp0,
                                                                        const FrameParams* const* __restrict__ fps,
                                                                        const uint32_t* __restrict__ work,
                                                                        uint32_t n_work,
                                                                        const uint32_t* __restrict__ n_heavy,
                                                                        uint32_t* __restrict__ next,
                                                                        uint32_t* __restrict__ done,
                                                                        uint32_t n_views) {
    constexpr int SR = 64 / T;                    // rows per strip
    constexpr int NS = T * T / 64;                // strips per tile
    constexpr int MR = T / 8;                     // rows per mask bit
    constexpr int SB = SR >= MR ? SR / MR : 1;    // mask bits of one strip
    constexpr int HP = T / 2;                     // lanes (pixel pairs) per row
    constexpr int XR = SR > 2 ? SR - 2 : 0;       // row terms kept beside the raw records' slots
    constexpr int RING = BL_RING;
    constexpr int G = 2;                          // records a lane evaluates at a time, each at both pixels
    static_assert(T == 16 || T == 32, "tile size 16 or 32");
    static_assert(DEPTH % 16 == 0 && DEPTH <= 32, "staging depth: 16 or 32 hits");
    static_assert(DEPTH + BL_SCAN <= RING && RING >= 64 * 3, "ring too small");
    pdl_wait();
    // [buffer][part: 0 = record's first half / row 0, 1 = colour, 2 = second half / row 1][warp][slot]
    __shared__ __align__(16) float4 sbuf[2][3][BL_WARPS][DEPTH + 1];
    __shared__ __align__(16) float4 s_row[XR > 0 ? XR : 1][BL_WARPS][XR > 0 ? DEPTH + 1 : 1];  // rows 2 and 3
    __shared__ __align__(16) uint32_t s_ring[BL_WARPS][RING];  // queue of hit pair values; at the end the strip's pixels
    __shared__ WarpItem s_item[BL_WARPS];
    __shared__ uint2 s_pm[BL_WARPS][DEPTH];      // staged records' pixel masks: even and odd columns
    __shared__ ClaimRing s_heavy, s_light;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    s_heavy.init<T * T / 32>();
    s_light.init<NS>();
    if (lane == 0) init_item(s_item[warp]);
    if (lane < 6) sbuf[lane / 3][lane % 3][warp][DEPTH] = dummy_part<0, 2>(lane % 3);
    if (XR > 0 && lane < XR) s_row[lane][warp][XR > 0 ? DEPTH : 0] = dummy_part<0, 2>(0);
    __syncthreads();
    uint32_t* ring = s_ring[warp];
    volatile WarpItem& it = s_item[warp];
    const bool full_walk = (fp0->test_hooks & VGR_HOOK_FULL_STRIP_WALK) != 0u;
    // (strips of one row of a 32-pixel tile would all look at a mask bit's four rows)
    const uint32_t heavy = T == 16 ? min(*n_heavy, n_work) : 0u;
    // the first slots are dealt out over the whole list (heavy ones, then the
    // others), the rest of the heavy ones and the rest of the others are claimed
    constexpr uint32_t PARTS = NS / slot_strips(NS);  // slots of a tile (one for a heavy tile of 16 x 16)
    const uint32_t dealt = gridDim.x, mine = blockIdx.x;
    uint32_t light0 = mine;
    if constexpr (T == 16) {
        if (mine < heavy) light0 = NONE;
        if (heavy > 0u)
            blend_strips<0, DEPTH, T>(sbuf, ring, reinterpret_cast<uint32_t*>(s_pm[warp]), it, s_heavy, fp0, fps,
                                      work, heavy, next, mine < heavy ? mine : NONE, dealt, nullptr, 0u, 0.f,
                                      full_walk);
    }
    const uint32_t light_base = max(dealt, heavy);
    static_assert(T == 32 || PARTS == 1, "slots count tiles where some of them are heavy");
    const uint32_t row = lane / HP, col = 2u * (lane % HP);  // this lane's first pixel in the strip
    for (;;) {
        uint32_t idx, strip;
        if (!claim_item<NS>(s_light, next + 1, light0, light_base, fp0, idx, strip) || idx >= n_work) break;
        uint2 rg;
        float rlo, clo, fxa;
        uint32_t wbits;
        bool in_a, in_b;
        {
            const uint32_t item = work[idx];
            const uint32_t view = item >> WORK_TILE_BITS, tile = item & WORK_TILE_MASK;
            const FrameParams* fp = fps ? fps[view] : fp0;
            const uint32_t W = fp->width, H = fp->height, TW = fp->tiles_x;
            const uint32_t x0 = (tile % TW) * T, y0 = (tile / TW) * T + SR * strip;
            if (lane == 0) fill_item(it, fp, view, x0, y0, (uint32_t)T, (uint32_t)SR);
            rg = fp->bl_ranges[tile];
            in_a = x0 + col < W && y0 + row < H;
            in_b = x0 + col + 1u < W && y0 + row < H;
            wbits = ((1u << SB) - 1u) << (SR * strip / MR);
            rlo = (float)y0 + 0.5f;  // centre of the strip's first row
            clo = (float)x0 + 0.5f;  // and column
            fxa = (float)(col + x0) + 0.5f;
            __syncwarp();
        }
        const float fxb = fxa + 1.0f;  // exact
        float Ta = 1.f, ra = 0.f, ga = 0.f, ba = 0.f, Tb = 1.f, rb = 0.f, gb = 0.f, bb = 0.f;
        bool done_a = !in_a, done_b = !in_b;
        uint32_t evals = 0, contribs = 0;
        uint32_t head = 0, tail = 0;
        uint32_t bp = rg.x;  // first pair value of the pending batch
        uint32_t pend[BL_SCAN / 32];
        {
            const uint32_t* pv = it.pair_val;
#pragma unroll
            for (int g = 0; g < BL_SCAN / 32; ++g) {
                const uint32_t j = bp + 32u * g + lane;
                pend[g] = j < rg.y ? pv[j] : 0u;
            }
        }
        auto refill = [&]() {
            while (tail - head < (uint32_t)DEPTH && bp < rg.y) {
#pragma unroll
                for (int g = 0; g < BL_SCAN / 32; ++g) {
                    const uint32_t v = pend[g];
                    const bool hit = (v & wbits) != 0u;  // entries past the range hold 0
                    const uint32_t hits = __ballot_sync(FULL, hit);
                    if (hit) ring[(tail + __popc(hits & lanemask_lt())) & (RING - 1)] = v;
                    tail += __popc(hits);
                }
                bp += BL_SCAN;
                const uint32_t* pv = it.pair_val;
#pragma unroll
                for (int g = 0; g < BL_SCAN / 32; ++g) {
                    const uint32_t j = bp + 32u * g + lane;
                    pend[g] = j < rg.y ? pv[j] : 0u;
                }
            }
            __syncwarp();
        };
        uint32_t rows_next = 0;  // row-mask bits of the pair staged in this lane's slot
        auto issue = [&](int buf) -> uint32_t {
            const uint32_t nh = min((uint32_t)DEPTH, tail - head);
            if (lane < nh) {
                const float4* rR = it.rec;
                const float4* rC = it.rgb;
                const uint32_t v = ring[(head + lane) & (RING - 1)], gi = v >> 8;
                rows_next = v & wbits;
                cp_async16(&sbuf[buf][0][warp][lane], rR + 2 * (size_t)gi);
                cp_async16(&sbuf[buf][2][warp][lane], rR + 2 * (size_t)gi + 1);
                cp_async16(&sbuf[buf][1][warp][lane], rC + gi);
            }
            cp_async_commit();
            head += nh;
            return nh;
        };
        refill();
        uint32_t nh_cur = issue(0);
        int buf = 0;
        while (nh_cur > 0) {
            if (__all_sync(FULL, done_a && done_b)) break;
            const uint32_t rows = rows_next;
            refill();
            const uint32_t nh_next = issue(buf ^ 1);  // the next chunk in flight during this walk
            cp_async_wait<1>();  // this chunk's copies (all but the newest group)
            __syncwarp();
            if (lane < (uint32_t)DEPTH) {  // each lane its own slot; empty slots reach no pixel
                uint2 pm = make_uint2(0u, 0u);
                if (lane < nh_cur) {
                    const float4 a = sbuf[buf][0][warp][lane], b = sbuf[buf][2][warp][lane];
                    pm = make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);
                    if (!full_walk) {
                        const uint32_t hw = __float_as_uint(b.w);
                        const float by = __half2float(__ushort_as_half((unsigned short)(hw & 0xFFFFu))) + 0.01f;
                        const float bx = __half2float(__ushort_as_half((unsigned short)(hw >> 16))) + 0.01f;
                        const int c0 = max(__float2int_ru(a.x - bx - clo), 0);
                        const int c1 = min(__float2int_rd(a.x + bx - clo), T - 1);
                        int r0 = max(__float2int_ru(a.y - by - rlo), 0);
                        int r1 = min(__float2int_rd(a.y + by - rlo), SR - 1);
                        if (SB == 2) {  // rows whose mask bit is clear are out of reach
                            if (!(rows & (1u << (SR * strip / MR)))) r0 = max(r0, MR);
                            if (!(rows & (2u << (SR * strip / MR)))) r1 = min(r1, MR - 1);
                        }
                        // pairs p with c0 <= 2 p <= c1, and with c0 <= 2 p + 1 <= c1
                        const uint32_t ma = pair_range((c0 + 1) >> 1, c1 >> 1), mb = pair_range(c0 >> 1, (c1 - 1) >> 1);
                        pm = make_uint2(0u, 0u);
#pragma unroll
                        for (int r = 0; r < SR; ++r)
                            if (r >= r0 && r <= r1) {
                                pm.x |= ma << (r * HP);
                                pm.y |= mb << (r * HP);
                            }
                    }
                    // per row (u, A', B' dy_r, C' dy_r^2 + log2 theta), as blend_prepare computes them
                    const float Bc = a.w * LOG2E, Cc = b.x * LOG2E, add = (LN_ALPHA_MIN - b.y) * LOG2E;
                    const float Ap = a.z * LOG2E;
#pragma unroll
                    for (int r = 0; r < SR; ++r) {
                        const float dy = a.y - (rlo + (float)r);
                        const float4 Y = make_float4(a.x, Ap, Bc * dy, fmaf(Cc * dy, dy, add));
                        if (r == 0) sbuf[buf][0][warp][lane] = Y;
                        else if (r == 1) sbuf[buf][2][warp][lane] = Y;
                        else s_row[XR > 0 ? r - 2 : 0][warp][XR > 0 ? lane : 0] = Y;
                    }
                }
                s_pm[warp][lane] = pm;
            }
            __syncwarp();
            // the records that can reach this lane's pixels, as slot bits in depth
            // order from bit 31 down: the transposes of the records' pixel masks
            uint32_t reach_a, reach_b;
            {
                const uint32_t sl = 31u - lane;
                const uint2 pm = sl < (uint32_t)DEPTH ? s_pm[warp][sl] : make_uint2(0u, 0u);
                reach_a = warp_transpose32(pm.x);
                reach_b = warp_transpose32(pm.y);
            }
            if (done_a) reach_a = 0u;
            if (done_b) reach_b = 0u;
            evals += __popc(reach_a) + __popc(reach_b);
            uint32_t mm = reach_a | reach_b;
            const float4* wY = row == 0u ? sbuf[buf][0][warp] : row == 1u ? sbuf[buf][2][warp]
                                                                          : s_row[XR > 1 ? row - 2u : 0u][warp];
            const float4* wC = sbuf[buf][1][warp];
            while (mm != 0u) {
                uint32_t at[G];
                bool ua[G], ub[G];
                float aa[G], ab[G];
#pragma unroll
                for (int g = 0; g < G; ++g) at[g] = next_slot<DEPTH>(mm, 0);
                // a record that only the neighbour's reach holds is not this pixel's, whatever
                // its rho: outside the box Eq. 4 fails, but the rounding of rho can pass it for
                // Gaussians hundreds of pixels long and one wide (a pixel that is done reaches none)
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const float4 X = wY[at[g]];
                    const float da = X.x - fxa, db = X.x - fxb;
                    const float rho_a = fmaf(fmaf(X.y, da, X.z), da, X.w), rho_b = fmaf(fmaf(X.y, db, X.z), db, X.w);
                    aa[g] = fminf(ALPHA_MAX, ex2_approx(rho_a));
                    ab[g] = fminf(ALPHA_MAX, ex2_approx(rho_b));
                    const uint32_t bit = 0x80000000u >> (at[g] & 31u);  // (slot DEPTH passes at no rho)
                    ua[g] = !(rho_a < LOG2_ALPHA_MIN) && (reach_a & bit) != 0u;
                    ub[g] = !(rho_b < LOG2_ALPHA_MIN) && (reach_b & bit) != 0u;
                }
                float ta[G], tb[G], Na = Ta, Nb = Tb;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    ta[g] = Na;
                    tb[g] = Nb;
                    if (ua[g]) Na = Na * (1.f - aa[g]);
                    if (ub[g]) Nb = Nb * (1.f - ab[g]);
                }
                // T never rises, so a group that ends at or above T_MIN stops nowhere
                if (Na < T_MIN) {
                    uint32_t after = 0;  // slots behind the stop, which are not evaluated
                    bool go = true;
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        if (go && ua[g] && ta[g] * (1.f - aa[g]) < T_MIN) {
                            go = false;
                            Na = ta[g];
                            after = 0x7FFFFFFFu >> at[g];
                        }
                        if (!go) ua[g] = false;
                    }
                    done_a = true;
                    evals -= __popc(reach_a & after);
                    reach_a = 0u;
                }
                if (Nb < T_MIN) {
                    uint32_t after = 0;
                    bool go = true;
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        if (go && ub[g] && tb[g] * (1.f - ab[g]) < T_MIN) {
                            go = false;
                            Nb = tb[g];
                            after = 0x7FFFFFFFu >> at[g];
                        }
                        if (!go) ub[g] = false;
                    }
                    done_b = true;
                    evals -= __popc(reach_b & after);
                    reach_b = 0u;
                }
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const float4 C4 = wC[at[g]];
                    if (ua[g]) {
                        const float w = aa[g] * ta[g];
                        ra = fmaf(w, C4.x, ra);
                        ga = fmaf(w, C4.y, ga);
                        ba = fmaf(w, C4.z, ba);
                        ++contribs;
                    }
                    if (ub[g]) {
                        const float w = ab[g] * tb[g];
                        rb = fmaf(w, C4.x, rb);
                        gb = fmaf(w, C4.y, gb);
                        bb = fmaf(w, C4.z, bb);
                        ++contribs;
                    }
                }
                Ta = Na;
                Tb = Nb;
                mm &= reach_a | reach_b;
            }
            __syncwarp();  // the walk is done with this buffer before it is refilled
            buf ^= 1;
            nh_cur = nh_next;
        }
        cp_async_wait<0>();  // the chunk staged ahead, if the strip stopped early
        float* const host_image = it.host_image;
        // a whole strip whose rows start 16-byte aligned: its pixels through shared
        // memory, SR rows of 3T/4 float4 (long aligned bursts over the host link)
        const bool whole = it.nx == (uint32_t)T && it.ny == (uint32_t)SR && (it.width & 3u) == 0u &&
                           ((reinterpret_cast<uintptr_t>(host_image) & 15u) == 0u);
        if (whole) {
            float2* s = reinterpret_cast<float2*>(ring) + 3u * lane;
            s[0] = make_float2(ra, ga);
            s[1] = make_float2(ba, rb);
            s[2] = make_float2(gb, bb);
            __syncwarp();
            constexpr uint32_t F4_ROW = 3 * T / 4;
            for (uint32_t i = lane; i < 48u; i += 32u) {  // 192 floats
                const float4 val = reinterpret_cast<const float4*>(ring)[i];
                const size_t at4 = ((size_t)it.at + (size_t)(i / F4_ROW) * it.width) * 3 + 4u * (i % F4_ROW);
                *reinterpret_cast<float4*>(it.image + at4) = val;
                if (host_image) *reinterpret_cast<float4*>(host_image + at4) = val;  // pinned host buffer
            }
            __syncwarp();
        } else if (in_a) {
            const size_t at = ((size_t)it.at + (size_t)row * it.width + col) * 3;
            const float px[6] = {ra, ga, ba, rb, gb, bb};
            const int n = in_b ? 6 : 3;
            for (int k = 0; k < n; ++k) {
                it.image[at + k] = px[k];
                if (host_image) host_image[at + k] = px[k];  // the caller's pinned host buffer, over the host link
            }
        }
        const uint32_t ev_w = __reduce_add_sync(FULL, evals), co_w = __reduce_add_sync(FULL, contribs);
        if (lane == 0) {
            it.evals = it.evals + ev_w;
            it.contribs = it.contribs + co_w;
        }
        __syncwarp();  // every lane is done with the item before lane 0 rewrites it
    }
    if (lane == 0) flush_item(it);
    finish_blend(done, fp0, fps, n_views);
}

template <int MODE, int DEPTH, int T>
void launch_blend_t(const FrameParams* fp0, const FrameParams* const* fps, const uint32_t* work, uint32_t n_work,
                    uint32_t* next, uint32_t* done, uint32_t n_views, int grid, cudaStream_t s) {
    launch_k(k_blend<MODE, DEPTH, T>, grid, BL_THREADS, s, fp0, fps, work, n_work, next, done, n_views);
}

// Two pixels per lane when the launch has 32-pixel strips for every resident warp
// BL_WIDE_ROUNDS times over; with fewer, the longest strips decide.  Blend with
// and without: 801 x 603 (15.5K strips, 3.2 rounds) 21.7 and 26.4 us, 640 x 360
// (7.4K, 1.5 rounds; long horizon tiles) 49.5 and 47.6, 320 x 180 (1.9K) 58.2 and
// 55.7.  Tiles of 32 pixels always: a strip of one row would stage the hits of
// the four rows of its mask bit (1440p: 156 us, 347 before).
constexpr uint32_t BL_WIDE_ROUNDS = 2;

bool blend_wide(uint32_t filter, uint32_t exp_mode, uint32_t depth, uint32_t tile, uint32_t n_work, int sms) {
    if (filter != VGR_FILTER_PREEMPTIVE || exp_mode != VGR_EXP_EXACT || depth > 32 || tile < 16) return false;
    const uint64_t strips = (uint64_t)n_work * (tile * tile / 32);
    return tile == 32 || strips >= (uint64_t)BL_WIDE_ROUNDS * sms * BL_MIN_CTAS * BL_WARPS;
}

template <int DEPTH, int T>
void launch_blend_wide(const FrameParams* fp0, const FrameParams* const* fps, const uint32_t* work, uint32_t n_work,
                       const uint32_t* n_heavy, uint32_t* next, uint32_t* done, uint32_t n_views, int sms,
                       cudaStream_t s) {
    // resident CTAs per SM, queried once (or by each of the threads that come first: the
    // answer is the same, on every device that the library runs on)
    static std::atomic<int> cached{0};
    int ctas = cached.load(std::memory_order_relaxed);
    if (!ctas) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, k_blend_wide<DEPTH, T>, BL_THREADS, 0);
        ctas = ctas > 0 ? ctas : 1;
        cached.store(ctas, std::memory_order_relaxed);
    }
    launch_k(k_blend_wide<DEPTH, T>, sms * ctas, BL_THREADS, s, fp0, fps, work, n_work, n_heavy, next, done, n_views);
}

// The default mode at every (depth, tile) of the tuner; the canonical and
// table modes at depth 32.
template <int T>
void launch_blend_tile(const FrameParams* fp0, const FrameParams* const* fps, const uint32_t* work, uint32_t n_work,
                       uint32_t* next, uint32_t* done, uint32_t n_views, int grid, uint32_t filter, uint32_t exp_mode,
                       uint32_t depth, cudaStream_t s) {
    if (filter == VGR_FILTER_CANONICAL) launch_blend_t<1, 32, T>(fp0, fps, work, n_work, next, done, n_views, grid, s);
    else if (exp_mode == VGR_EXP_LUT) launch_blend_t<2, 32, T>(fp0, fps, work, n_work, next, done, n_views, grid, s);
    else if (depth == 16) launch_blend_t<0, 16, T>(fp0, fps, work, n_work, next, done, n_views, grid, s);
    else if (depth == 48 && T != 8)
        launch_blend_t<0, (T != 8 ? 48 : 32), T>(fp0, fps, work, n_work, next, done, n_views, grid, s);
    else launch_blend_t<0, 32, T>(fp0, fps, work, n_work, next, done, n_views, grid, s);
}

template <int MODE, int DEPTH, int T>
int occupancy() {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_blend<MODE, DEPTH, T>, BL_THREADS, 0);
    return n > 0 ? n : 1;
}

static int blend_ctas_per_sm(uint32_t filter, uint32_t exp_mode, uint32_t depth, uint32_t tile) {
    // [mode][depth][tile], queried once each (as in launch_blend_wide)
    static std::atomic<int> cache[3][3][3] = {};
    const int md = filter == VGR_FILTER_CANONICAL ? 1 : exp_mode == VGR_EXP_LUT ? 2 : 0;
    const int d = md != 0 ? 1 : depth == 16 ? 0 : (depth == 48 && tile != 8) ? 2 : 1;
    const int t = tile == 8 ? 0 : tile == 32 ? 2 : 1;
    int c = cache[md][d][t].load(std::memory_order_relaxed);
    if (!c) {
        switch (md * 9 + d * 3 + t) {
            case 0: c = occupancy<0, 16, 8>(); break;
            case 1: c = occupancy<0, 16, 16>(); break;
            case 2: c = occupancy<0, 16, 32>(); break;
            case 3: c = occupancy<0, 32, 8>(); break;
            case 4: c = occupancy<0, 32, 16>(); break;
            case 5: c = occupancy<0, 32, 32>(); break;
            case 7: c = occupancy<0, 48, 16>(); break;
            case 8: c = occupancy<0, 48, 32>(); break;
            case 12: c = occupancy<1, 32, 8>(); break;
            case 13: c = occupancy<1, 32, 16>(); break;
            case 14: c = occupancy<1, 32, 32>(); break;
            case 21: c = occupancy<2, 32, 8>(); break;
            case 22: c = occupancy<2, 32, 16>(); break;
            case 23: c = occupancy<2, 32, 32>(); break;
            default: c = 1; break;
        }
        cache[md][d][t].store(c, std::memory_order_relaxed);
    }
    return c;
}

void launch_blend(const FrameParams* fp0, const FrameParams* const* fps, const uint32_t* work, uint32_t n_work,
                  const uint32_t* n_heavy, uint32_t* next, uint32_t* done, uint32_t n_views, int sms, uint32_t filter,
                  uint32_t exp_mode, uint32_t depth, uint32_t tile, cudaStream_t s) {
    if (blend_wide(filter, exp_mode, depth, tile, n_work, sms)) {
        auto wide = tile == 32 ? (depth == 16 ? launch_blend_wide<16, 32> : launch_blend_wide<32, 32>)
                               : (depth == 16 ? launch_blend_wide<16, 16> : launch_blend_wide<32, 16>);
        wide(fp0, fps, work, n_work, n_heavy, next, done, n_views, sms, s);
        return;
    }
    const int grid = sms * blend_ctas_per_sm(filter, exp_mode, depth, tile);
    auto narrow = tile == 8 ? launch_blend_tile<8> : tile == 32 ? launch_blend_tile<32> : launch_blend_tile<16>;
    narrow(fp0, fps, work, n_work, next, done, n_views, grid, filter, exp_mode, depth, s);
}

}  // namespace vgr
