// k_lod.cu -- LoD cut finding on the GPU (paper Sec. 3.1 'Cut Finding',
// Sec. 4.1 'Temporal-Aware LoD Search', Algorithm 1).
//
// The cut is written as a bitmap over node ids (plus a second bitmap of the
// cut nodes in front of the near plane), then compacted into ascending id
// lists.  Two producers:
//  * k_lod_update: the temporal update.  Each node n of the previous cut
//    tests itself and its parent against the current camera:
//      parent does not expand  -> collapse: climb to the highest ancestor whose
//                                 parent expands (or the root); it joins the cut
//      n expands               -> expand: explore n's subtree depth-first;
//                                 non-expanding nodes reached join the cut
//      otherwise               -> n stays in the cut.
//    This is Algorithm 1 with single nodes in place of height-2 subtrees:
//    TOP (collapse) moves to the parent, BOTTOM (expand) to the children.
//    The result equals the top-down cut whenever the test is monotone
//    (a child expands only if its parent does), which the nested radii
//    guarantee; a violation raises F_NONMONOTONE.  A thread that would
//    explore more than the budget sets F_LOD_FALLBACK and the host redoes
//    the frame top-down.  The node's (mean, radius^2) and its parent's are
//    stored together in one 32-byte record per node (built at load), so a
//    cut node costs one sector and one round instead of waiting for the
//    parent's id first; the id itself is read only when the node collapses.
//  * k_lod_dense: the cut without a previous one (frame 0, tau change, reset,
//    fallback), in one pass over the nodes.
//  * k_lod_level: one level of the from-scratch, top-down traversal, for coarse
//    cuts of large trees (DENSE_ANY_NODES in vgr_capi.cu) and for views whose test
//    turned out not monotone; frontiers are appended with one atomic per warp after
//    a warp scan of the child counts.
#include "vgr_internal.cuh"
#include "vgr_launch.h"

namespace vgr {

constexpr int CC_TILE_WORDS = 256;             // bitmap words per tile of the compaction
constexpr int CC_TILE_IDS = CC_TILE_WORDS * 32;
// words between the tiles' counters: a line each, since the warps in flight
// count into neighbouring tiles (in one line their atomics queue at one L2
// slice: +24 us on the city)
constexpr int CC_COUNT_STRIDE = 32;

// A cut node joins the cut bitmap, and the potentially-visible bitmap when
// its FP32 depth key is beyond the near plane (the same key and test as
// preprocess) and its footprint can reach the image.  The footprint test is
// a bound on the one preprocess applies: preprocess's box half-width is
//   bx = r sqrt(S'00) * 1.0001 + 1e-3,  r^2 = 2 (ln theta - ln alpha*) + 2 slack
//   <= 3.33 (slack included),  S'00 = m0^T S m0 + 0.3,  m0 = fx/z (R0 - tx R2),
// and |m0|^2 = (fx/z)^2 (1 + tx^2) <= (fx/z)^2 (1 + limx^2) while
// m0^T S m0 <= lambda_max(S) |m0|^2 <= L |m0|^2, L the largest absolute row
// sum of S (Gershgorin, stored per node at load); so with
//   Bx = 3.34 sqrt(L (fx/z)^2 (1 + limx^2) + 0.3) + 0.01
// a Gaussian with u + Bx < 0.5 or u - Bx > T tiles_x - 0.5 (or likewise in
// v) has no candidate tile in preprocess and can be left out here.  The
// canonical mode's 3-sigma box is bounded the same way.
// Node n's record in one 32-byte load: its (mean, radius^2) entry and its parent's.
__device__ __forceinline__ void load_lodr(const float4* __restrict__ lodr, uint32_t n, float4& c, float4& p) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
        : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w), "=f"(p.x), "=f"(p.y), "=f"(p.z), "=f"(p.w)
        : "l"(lodr + 2 * (size_t)n));
}

// Set bit n of two bitmaps in the lanes where in_a and in_b hold (in_b implies
// in_a), one atomic per word: the lanes that hit the same word (the match
// instruction; a warp's nodes are few words) OR their bits together and the lowest
// of them stores them.  All 32 lanes call it.
__device__ __forceinline__ void warp_bitmap_set(uint32_t* a, uint32_t* b, uint32_t n, bool in_a, bool in_b) {
    const uint32_t w = in_a ? n >> 5 : 0xFFFFFFFFu;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, w);
    const uint32_t bit = 1u << (n & 31u);
    const uint32_t bits_a = __reduce_or_sync(peers, in_a ? bit : 0u);
    const uint32_t bits_b = __reduce_or_sync(peers, in_b ? bit : 0u);
    if (in_a && lane_id() == (uint32_t)(__ffs(peers) - 1)) {
        atomicOr(&a[w], bits_a);
        if (bits_b) atomicOr(&b[w], bits_b);
    }
}

// With weight interpolation the rendered Gaussian of a cut node n is not n's
// own: its mean lies on the segment from n's centre to its parent's and its
// covariance is a convex combination of theirs, so its largest eigenvalue is
// at most max(L_n, L_p).  When both centres are beyond the near plane the
// whole segment is, its projection is the segment between the two projected
// centres and its depth is at least the smaller of theirs: the union of the
// two boxes, widened for max(L_n, L_p) at that depth, bounds the footprint.
// A segment across the near plane is kept; one wholly behind it is dropped.
struct CutOut {
    uint32_t* cut_bm;
    uint32_t* front_bm;
    uint32_t* counts;  // bits set per bitmap tile: cut | in front << 16
    const float* lmax;
    const float4* cr;
    const uint32_t* parent;
    float R0, R1, R2, R3, R4, R5, R6, R7, R8, Cx, Cy, Cz, z_near;
    float fx, fy, cx, cy, kx, ky, umax, vmax;
    bool canonical;
    bool interp;  // weight interpolation: bound the interpolated Gaussian, not the node's own
    // an ancestor that several nodes may report: the one that sets a bit counts it
    __device__ __forceinline__ void add_shared(uint32_t n, float4 c) const {
        const uint32_t bit = 1u << (n & 31u);
        uint32_t fresh = (atomicOr(&cut_bm[n >> 5], bit) & bit) ? 0u : 1u;
        if (visible(n, c, lmax[n]) && !(atomicOr(&front_bm[n >> 5], bit) & bit)) fresh |= 1u << 16;
        if (fresh) atomicAdd(&counts[n / CC_TILE_IDS * CC_COUNT_STRIDE], fresh);
    }
    // a node that only this thread reports (unless the previous cut held one of
    // its ancestors as well: see k_cut_compact); its counts are held back in
    // (tile, held) while the thread stays in one tile (a subtree's nodes do)
    __device__ __forceinline__ void add(uint32_t n, float4 c, uint32_t& tile, uint32_t& held) const {
        const uint32_t bit = 1u << (n & 31u);
        atomicOr(&cut_bm[n >> 5], bit);
        uint32_t one = 1u;
        if (visible(n, c, lmax[n])) {
            atomicOr(&front_bm[n >> 5], bit);
            one |= 1u << 16;
        }
        if (n / CC_TILE_IDS != tile) {
            flush(tile, held);
            tile = n / CC_TILE_IDS;
        }
        held += one;
    }
    __device__ __forceinline__ void flush(uint32_t tile, uint32_t& held) const {
        if (held) atomicAdd(&counts[tile * CC_COUNT_STRIDE], held);
        held = 0u;
    }
    // may the Gaussian rendered for cut node n (centre c, lm = lmax[n]) reach the image?
    __device__ __forceinline__ bool visible(uint32_t n, float4 c, float lm) const {
        if (!interp) return in_front(c, lm);
        const uint32_t p = parent[n];
        if (p == NONE) return in_front(c, lm);
        return in_front_segment(c, lm, cr[p], lmax[p]);
    }
    __device__ __forceinline__ float depth(float4 c) const {
        const float dx = __fsub_rn(c.x, Cx), dy = __fsub_rn(c.y, Cy), dz = __fsub_rn(c.z, Cz);
        return __fadd_rn(__fadd_rn(__fmul_rn(R6, dx), __fmul_rn(R7, dy)), __fmul_rn(R8, dz));
    }
    __device__ __forceinline__ void project(float4 c, float z, float& u, float& v) const {
        const float dx = __fsub_rn(c.x, Cx), dy = __fsub_rn(c.y, Cy), dz = __fsub_rn(c.z, Cz);
        const float x = fmaf(R0, dx, fmaf(R1, dy, R2 * dz));
        const float y = fmaf(R3, dx, fmaf(R4, dy, R5 * dz));
        const float iz = 1.0f / z;
        u = fmaf(fx, x * iz, cx);
        v = fmaf(fy, y * iz, cy);
    }
    __device__ __forceinline__ void half_box(float lm, float z, float& bx, float& by) const {
        const float iz = 1.0f / z;
        const float t = lm * iz * iz;
        if (!canonical) {
            bx = 3.34f * sqrtf(fmaf(t, kx, 0.3f)) + 0.01f;
            by = 3.34f * sqrtf(fmaf(t, ky, 0.3f)) + 0.01f;
        } else {
            bx = by = 3.01f * sqrtf(fmaf(t, kx + ky, 1.0f)) + 1.01f;
        }
    }
    __device__ __forceinline__ bool in_front_segment(float4 cn, float lmn, float4 cp, float lmp) const {
        const float zn = depth(cn), zp = depth(cp);
        const float zeps = 1e-2f;  // far above the FP32 error of the interpolated mean's depth
        if (zn <= z_near - zeps && zp <= z_near - zeps) return false;
        if (!(zn > z_near + zeps) || !(zp > z_near + zeps)) return true;
        float un, vn, up, vp, bx, by;
        project(cn, zn, un, vn);
        project(cp, zp, up, vp);
        half_box(fmaxf(lmn, lmp), fminf(zn, zp), bx, by);
        const float ulo = fminf(un, up), uhi = fmaxf(un, up), vlo = fminf(vn, vp), vhi = fmaxf(vn, vp);
        const float su = 1e-5f * fmaxf(fabsf(ulo), fabsf(uhi)) + 1e-2f;
        const float sv = 1e-5f * fmaxf(fabsf(vlo), fabsf(vhi)) + 1e-2f;
        return !(uhi + bx < 0.5f - su || ulo - bx > umax + su || vhi + by < 0.5f - sv || vlo - by > vmax + sv);
    }
    // may node (centre c, lm = lmax[n]) reach the image in front of the near plane?
    __device__ __forceinline__ bool in_front(float4 c, float lm) const {
        const float dx = __fsub_rn(c.x, Cx), dy = __fsub_rn(c.y, Cy), dz = __fsub_rn(c.z, Cz);
        const float z = __fadd_rn(__fadd_rn(__fmul_rn(R6, dx), __fmul_rn(R7, dy)), __fmul_rn(R8, dz));
        if (!(z > z_near)) return false;
        const float x = fmaf(R0, dx, fmaf(R1, dy, R2 * dz));
        const float y = fmaf(R3, dx, fmaf(R4, dy, R5 * dz));
        const float iz = 1.0f / z;
        const float u = fmaf(fx, x * iz, cx), v = fmaf(fy, y * iz, cy);
        const float t = lm * iz * iz;
        float bx, by;
        if (!canonical) {
            bx = 3.34f * sqrtf(fmaf(t, kx, 0.3f)) + 0.01f;
            by = 3.34f * sqrtf(fmaf(t, ky, 0.3f)) + 0.01f;
        } else {
            // canonical: ceil(3 sqrt(lam)), lam <= S'00 + S'11 + 0.32 (its sqrt(max(0.1, .)) floor)
            bx = by = 3.01f * sqrtf(fmaf(t, kx + ky, 1.0f)) + 1.01f;
        }
        const float su = 1e-5f * fabsf(u) + 1e-2f, sv = 1e-5f * fabsf(v) + 1e-2f;  // FP32 slack
        return !(u + bx < 0.5f - su || u - bx > umax + su || v + by < 0.5f - sv || v - by > vmax + sv);
    }
};

// Count the warp's nodes n[0..U) that join the cut (and of those the ones in
// front) per bitmap tile: one atomic per tile, and a warp's nodes are mostly in
// one.  All 32 lanes call it; every node is reported once.
template <int U>
__device__ __forceinline__ void warp_tile_count(uint32_t* counts, const uint32_t* n, const bool* in_cut,
                                                const bool* in_front) {
    uint32_t left[U], vis[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        left[u] = __ballot_sync(0xFFFFFFFFu, in_cut[u]);
        vis[u] = __ballot_sync(0xFFFFFFFFu, in_front[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        while (left[u]) {  // uniform: every lane takes part in every shuffle and ballot
            const int lead = __ffs(left[u]) - 1;
            const uint32_t tile = __shfl_sync(0xFFFFFFFFu, n[u] / CC_TILE_IDS, lead);
            uint32_t c = 0;
#pragma unroll
            for (int v = u; v < U; ++v) {
                const uint32_t same = __ballot_sync(0xFFFFFFFFu, n[v] / CC_TILE_IDS == tile) & left[v];
                left[v] &= ~same;
                c += (uint32_t)__popc(same) | ((uint32_t)__popc(vis[v] & same) << 16);
            }
            if ((int)lane_id() == lead) atomicAdd(&counts[tile * CC_COUNT_STRIDE], c);
        }
    }
}

template <bool IP>
__device__ __forceinline__ CutOut make_cut_out(const FrameParams* fp, const SceneDev& sc, uint32_t* cut_bm,
                                               uint32_t* front_bm, uint32_t* counts) {
    CutOut o;
    o.counts = counts;
    o.cut_bm = cut_bm;
    o.front_bm = front_bm;
    o.lmax = sc.lmax;
    o.cr = sc.cr;
    o.parent = sc.parent;
    o.R0 = fp->R[0]; o.R1 = fp->R[1]; o.R2 = fp->R[2];
    o.R3 = fp->R[3]; o.R4 = fp->R[4]; o.R5 = fp->R[5];
    o.R6 = fp->R[6]; o.R7 = fp->R[7]; o.R8 = fp->R[8];
    o.Cx = fp->pos[0]; o.Cy = fp->pos[1]; o.Cz = fp->pos[2];
    o.z_near = fp->z_near;
    o.fx = fp->fx; o.fy = fp->fy; o.cx = fp->cx; o.cy = fp->cy;
    o.kx = fp->fx * fp->fx * (1.0f + fp->limx * fp->limx);
    o.ky = fp->fy * fp->fy * (1.0f + fp->limy * fp->limy);
    o.umax = (float)(fp->tile * fp->tiles_x) - 0.5f;
    o.vmax = (float)(fp->tile * fp->tiles_y) - 0.5f;
    o.canonical = fp->filter == VGR_FILTER_CANONICAL;
    o.interp = IP;  // a compile-time constant: the other form's code is not generated
    return o;
}

constexpr int LOD_UNROLL = 2;  // previous-cut nodes per thread and round

template <bool FR, bool IP>
__global__ void __launch_bounds__(256) k_lod_update(const uint32_t* __restrict__ prev_cut,
                                                    const uint32_t* __restrict__ n_prev_p, uint32_t cap_prev,
                                                    SceneDev sc, const FrameParams* __restrict__ fp,
                                                    uint32_t* __restrict__ bitmap, uint32_t* __restrict__ front,
                                                    uint32_t* __restrict__ counts, Counters* __restrict__ ctr) {
    pdl_wait();
    const uint32_t n_prev = min(*n_prev_p, cap_prev);
    const float px = fp->pos[0], py = fp->pos[1], pz = fp->pos[2], k = fp->k;
    const uint32_t budget = fp->lod_budget, max_depth = fp->max_depth;
    const CutOut out = make_cut_out<IP>(fp, sc, bitmap, front, counts);
    LodFrustum fr;
    if (FR) fr.load(fp, sc.box);
    // the granularity test, and in the frustum-aware variant the box test
    auto expand = [&](uint32_t node, float4 c) -> bool {
        if (!lod_expand(c, px, py, pz, k)) return false;
        if constexpr (FR) return fr.meets(node);
        return true;
    };
    uint32_t evals = 0, flags = 0;
    const uint32_t stride = gridDim.x * blockDim.x;
    // one previous-cut node: stay, collapse or expand
    // (a staying node is only reported: its bits are set warp-aggregated below).
    // cp is the parent's entry (w = +inf at the root); the parent's id p is
    // loaded with it by the frustum and interpolation variants (which test its
    // box or read its extent), else only when n collapses
    constexpr bool WITH_P = FR || IP;
    auto visit = [&](uint32_t n, float4 cn, uint32_t p, float4 cp) -> bool {
        const bool en = expand(n, cn);
        bool ep = true;
        ++evals;
        if (cp.w != INFINITY) { ep = expand(p, cp); ++evals; }
        if (!ep) {
            if (en) flags |= F_NONMONOTONE;
            // collapse: climb while the parent of a does not expand
            uint32_t a = WITH_P ? p : sc.parent[n];
            float4 ca = cp;
            for (uint32_t steps = 0;; ++steps) {
                const uint32_t pa = sc.parent[a];
                if (pa == NONE) break;
                ++evals;
                const float4 cpa = sc.cr[pa];
                if (expand(pa, cpa)) break;
                a = pa;
                ca = cpa;
                if (steps > max_depth) { flags |= F_LOD_FALLBACK; break; }
            }
            out.add_shared(a, ca);
        } else if (en) {
            // expand: depth-first over n's subtree, children ranges on a stack
            uint32_t nxt[MAX_TREE_DEPTH], end[MAX_TREE_DEPTH];
            const uint32_t c0 = sc.child[n];
            nxt[0] = c0 & CHILD_MASK;
            end[0] = nxt[0] + (c0 >> CHILD_SHIFT);
            int sp = 1;
            uint32_t local = 0, tile = NONE, held = 0;
            while (sp > 0) {
                if (nxt[sp - 1] == end[sp - 1]) { --sp; continue; }
                const uint32_t m = nxt[sp - 1]++;
                if (++local > budget) { flags |= F_LOD_FALLBACK; break; }
                const float4 cm = sc.cr[m];
                if (expand(m, cm)) {
                    if (sp == MAX_TREE_DEPTH) { flags |= F_LOD_FALLBACK; break; }
                    const uint32_t chm = sc.child[m];
                    nxt[sp] = chm & CHILD_MASK;
                    end[sp] = nxt[sp] + (chm >> CHILD_SHIFT);
                    ++sp;
                } else {
                    out.add(m, cm, tile, held);
                }
            }
            out.flush(tile, held);
            evals += local;
        } else {
            return true;  // stay
        }
        return false;
    };
    // LOD_UNROLL nodes per thread and round, their loads in flight together;
    // warp-uniform rounds so the staying nodes' bits can be set per warp
    const uint32_t lane = lane_id();
    const uint32_t first = (blockIdx.x * blockDim.x + threadIdx.x) & ~31u;
    uint32_t nx[LOD_UNROLL];  // the next round's node ids, loaded one round ahead
#pragma unroll
    for (int u = 0; u < LOD_UNROLL; ++u) {
        const uint32_t i = first + u * stride + lane;
        nx[u] = i < n_prev ? prev_cut[i] : 0u;
    }
    for (uint32_t b0 = first; b0 < n_prev; b0 += LOD_UNROLL * stride) {
        uint32_t nn[LOD_UNROLL], pp[LOD_UNROLL];
        float4 cc[LOD_UNROLL], qq[LOD_UNROLL];
        float ll[LOD_UNROLL];
        bool ok[LOD_UNROLL], in_cut[LOD_UNROLL], in_front[LOD_UNROLL];
#pragma unroll
        for (int u = 0; u < LOD_UNROLL; ++u) {
            const uint32_t i = b0 + u * stride + lane;
            ok[u] = i < n_prev;
            nn[u] = nx[u];
            const uint32_t inext = i + LOD_UNROLL * stride;
            nx[u] = inext < n_prev ? prev_cut[inext] : 0u;
        }
#pragma unroll
        for (int u = 0; u < LOD_UNROLL; ++u) {
            load_lodr(sc.lodr, nn[u], cc[u], qq[u]);  // its entry and the parent's
            ll[u] = sc.lmax[nn[u]];
            pp[u] = WITH_P ? sc.parent[nn[u]] : NONE;
        }
#pragma unroll
        for (int u = 0; u < LOD_UNROLL; ++u) {
            const bool stay = ok[u] && visit(nn[u], cc[u], pp[u], qq[u]);
            bool vis = false;
            if (stay) {
                if (!out.interp || pp[u] == NONE) vis = out.in_front(cc[u], ll[u]);
                else vis = out.in_front_segment(cc[u], ll[u], qq[u], sc.lmax[pp[u]]);
            }
            warp_bitmap_set(bitmap, front, nn[u], stay, vis);
            in_cut[u] = stay;
            in_front[u] = vis;
        }
        warp_tile_count<LOD_UNROLL>(counts, nn, in_cut, in_front);
    }
    // one atomic per warp for the statistics
    uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, evals);
    uint32_t wflags = __reduce_or_sync(0xFFFFFFFFu, flags);
    if (lane_id() == 0) {
        if (wsum) atomicAdd(&ctr->nodes_eval, (unsigned long long)wsum);
        if (wflags) atomicOr(&ctr->flags, wflags);
    }
}

// The cut without a previous one, in a single pass over all the nodes: where
// the test is monotone (a child expands only if its parent does), a node is
// reached exactly when its parent expands, so it is in the cut when its parent
// expands and it does not, and no level waits for the one above.  A node that
// expands under a parent that does not raises F_NONMONOTONE, and the host redoes
// the frame with k_lod_level.  A warp takes runs of 4 bitmap words and stores each
// from a ballot, with no atomics but one count per run.  Bound by HBM (the 32-byte
// node-and-parent records in order, 5.6 TB/s of them):
// 23 us on the 1M-leaf box against 130 for 12 level kernels, 181 us on the city
// at tau = 3 against 550 for 16 (tau = 24: 153 and 141, 48: 148 and 106).
constexpr int LOD_DENSE_UNROLL = 4;
constexpr uint32_t LOD_DENSE_RUN = 4;  // words

template <bool FR, bool IP>
__global__ void __launch_bounds__(256, FR || IP ? 2 : 4) k_lod_dense(SceneDev sc, const FrameParams* __restrict__ fp,
                                                   uint32_t* __restrict__ bitmap, uint32_t* __restrict__ front,
                                                   uint32_t* __restrict__ counts, Counters* __restrict__ ctr) {
    pdl_wait();
    const uint32_t N = sc.n_nodes;
    const float px = fp->pos[0], py = fp->pos[1], pz = fp->pos[2], k = fp->k;
    const CutOut out = make_cut_out<IP>(fp, sc, bitmap, front, counts);
    LodFrustum fr;
    if (FR) fr.load(fp, sc.box);
    constexpr bool WITH_P = FR || IP;
    constexpr int U = LOD_DENSE_UNROLL;
    constexpr uint32_t RUN = LOD_DENSE_RUN;
    static_assert(RUN % U == 0 && CC_TILE_WORDS % RUN == 0, "a run lies in one tile");
    const uint32_t lane = lane_id();
    const uint32_t nruns = (N + 32u * RUN - 1u) / (32u * RUN), nwarps = (gridDim.x * blockDim.x) >> 5;
    uint32_t evals = 0;
    bool bad = false;
    for (uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < nruns; r += nwarps) {
        uint32_t total = 0;  // of the run: cut | in front << 16
        for (uint32_t w0 = r * RUN; w0 < (r + 1u) * RUN; w0 += U) {
            float4 c[U], q[U];
            uint32_t p[U];
            bool ok[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t n = 32u * (w0 + u) + lane, at = min(n, N - 1u);
                ok[u] = n < N;
                load_lodr(sc.lodr, at, c[u], q[u]);
                p[u] = WITH_P ? sc.parent[at] : NONE;
            }
            bool in_cut[U];
            float lm[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t n = 32u * (w0 + u) + lane;
                bool en = ok[u] && lod_expand(c[u], px, py, pz, k);
                bool ep = ok[u] && (q[u].w == INFINITY || lod_expand(q[u], px, py, pz, k));
                if constexpr (FR) {
                    if (en) en = fr.meets(n);
                    if (ep && p[u] != NONE) ep = fr.meets(p[u]);
                }
                evals += ep;
                bad = bad || (en && !ep);
                in_cut[u] = ep && !en;
                lm[u] = in_cut[u] ? sc.lmax[n] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                bool vis = false;
                if (in_cut[u]) {
                    if (!IP || p[u] == NONE) vis = out.in_front(c[u], lm[u]);
                    else vis = out.in_front_segment(c[u], lm[u], q[u], sc.lmax[p[u]]);
                }
                const uint32_t cw = __ballot_sync(0xFFFFFFFFu, in_cut[u]), fw = __ballot_sync(0xFFFFFFFFu, vis);
                total += (uint32_t)__popc(cw) | ((uint32_t)__popc(fw) << 16);
                // (words without bits are zero already)
                if (lane == 0 && cw) bitmap[w0 + u] = cw;
                if (lane == 1 && fw) front[w0 + u] = fw;
            }
        }
        if (lane == 0 && total) atomicAdd(&counts[r * RUN / CC_TILE_WORDS * CC_COUNT_STRIDE], total);
    }
    const uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, evals);
    const bool wbad = __any_sync(0xFFFFFFFFu, bad);
    if (lane == 0) {
        if (wsum) atomicAdd(&ctr->nodes_eval, (unsigned long long)wsum);
        if (wbad) atomicOr(&ctr->flags, F_NONMONOTONE);
    }
}

// One level of the top-down traversal.  Level 0 starts from the root.
template <bool FR, bool IP>
__global__ void __launch_bounds__(256) k_lod_level(int level, const uint32_t* __restrict__ fin,
                                                   uint32_t* __restrict__ fout, uint32_t cap, SceneDev sc,
                                                   const FrameParams* __restrict__ fp,
                                                   uint32_t* __restrict__ bitmap, uint32_t* __restrict__ front,
                                                   uint32_t* __restrict__ counts, Counters* __restrict__ ctr) {
    pdl_wait();
    const uint32_t n_in = level == 0 ? 1u : min(ctr->frontier_n[level], cap);
    uint32_t* n_out = &ctr->frontier_n[level + 1];
    const float px = fp->pos[0], py = fp->pos[1], pz = fp->pos[2], k = fp->k;
    const CutOut out = make_cut_out<IP>(fp, sc, bitmap, front, counts);
    LodFrustum fr;
    if (FR) fr.load(fp, sc.box);
    const uint32_t lane = lane_id();
    const uint32_t warp_global = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    uint32_t evals = 0;
    for (uint32_t base = warp_global * 32u; base < n_in; base += nwarps * 32u) {
        const uint32_t i = base + lane;
        uint32_t cnt = 0, first = 0, n = 0;
        bool is_cut = false, in_front = false;
        if (i < n_in) {
            n = level == 0 ? 0u : fin[i];
            const float4 cn = sc.cr[n];
            const float lm = sc.lmax[n];
            ++evals;
            if (lod_expand(cn, px, py, pz, k) && (!FR || fr.meets(n))) {
                const uint32_t c = sc.child[n];
                first = c & CHILD_MASK;
                cnt = c >> CHILD_SHIFT;
            } else {
                is_cut = true;
                in_front = out.visible(n, cn, lm);
            }
        }
        // one atomic per bitmap word and warp (a node's siblings are neighbours)
        warp_bitmap_set(bitmap, front, n, is_cut, in_front);
        warp_tile_count<1>(counts, &n, &is_cut, &in_front);
        uint32_t total;
        const uint32_t off = warp_excl_scan(cnt, &total);
        uint32_t basepos = 0;
        if (lane == 0 && total) basepos = atomicAdd(n_out, total);
        basepos = __shfl_sync(0xFFFFFFFFu, basepos, 0);
        for (uint32_t j = 0; j < cnt; ++j) {
            const uint32_t pos = basepos + off + j;
            if (pos < cap) fout[pos] = first + j;
            else atomicOr(&ctr->flags, F_OVF_FRONTIER);
        }
    }
    uint32_t wsum = __reduce_add_sync(0xFFFFFFFFu, evals);
    if (lane == 0 && wsum) atomicAdd(&ctr->nodes_eval, (unsigned long long)wsum);
}

// Bitmaps -> ascending id lists (the cut, and its in-front part), clearing
// both bitmaps for the next frame.  The LoD kernels count the bits they set per
// tile of 256 words, so a tile's place in the lists is the sum of the counts
// before it: no count is waited for, and the CTAs take tiles in any order.  The
// counts are the bits' as long as every node is reported once.  Where the test is
// not monotone, an update can leave a node and its descendant in the cut without
// any of its tests showing it, and the next update then reports nodes twice; so a
// tile checks its count against its bits, and where they differ F_LOD_FALLBACK has
// the host replay the frame from the root (one word per tile; until then the lists
// hold some earlier frame's ids in places, all of them nodes).  A
// warp takes a row of 32 words: a scan of their bit counts gives every word its
// place, and the warp goes through the words that have bits, lane l storing the
// id of bit l if it is set (contiguous stores, no barrier, no staging).  Bound by
// those instructions (a bit count per word, at a quarter of the issue rate) and, on
// small scenes, by the kernel's three round trips.  The words and their places come
// as broadcasts from shared memory, two words per load: by two shuffles per word the
// 1M-leaf box took 10 us, now 8.5, the city (26.5M nodes) 32, now 28.  Tiles of 1024
// words on a look-back chain, their ids unpacked in shared memory bit by bit, took
// 28 and 41 us (while counting adds 10 to the 119 us of the city's LoD update).
constexpr int CC_THREADS = 256;
constexpr int CC_WARPS = CC_THREADS / 32;
static_assert(CC_TILE_WORDS == CC_THREADS, "one row of 32 words per warp");

// Store the ids of a row's set bits (lane l holds word l, first id id0 + 32 l)
// from out[at] on.  s_row: the warp's, for the words and places as broadcasts.
__device__ __forceinline__ void cc_row(uint32_t word, uint32_t pre, uint32_t id0, uint32_t* __restrict__ out,
                                       uint32_t cap, uint2* s_row) {
    const uint32_t lane = lane_id(), below = lanemask_lt();
    uint32_t some = __ballot_sync(0xFFFFFFFFu, word != 0u);
    if (__popc(some) >= 12) {  // most words have bits: all of them, independent of one another
        s_row[lane] = make_uint2(word, pre);
        __syncwarp();
        const uint4* two = reinterpret_cast<const uint4*>(s_row);
        const uint32_t id = id0 + lane;
#pragma unroll
        for (int w = 0; w < 16; ++w) {
            const uint4 q = two[w];
            const uint32_t p0 = q.y + __popc(q.x & below), p1 = q.w + __popc(q.z & below);
            if (((q.x >> lane) & 1u) && p0 < cap) out[p0] = id + 64u * w;
            if (((q.z >> lane) & 1u) && p1 < cap) out[p1] = id + 64u * w + 32u;
        }
        __syncwarp();  // read before the next row's words
        return;
    }
    while (some) {
        const int w = __ffs(some) - 1;
        some &= some - 1u;
        const uint32_t bits = __shfl_sync(0xFFFFFFFFu, word, w);
        const uint32_t p = __shfl_sync(0xFFFFFFFFu, pre, w) + __popc(bits & below);
        if (((bits >> lane) & 1u) && p < cap) out[p] = id0 + 32u * w + lane;
    }
}

__global__ void __launch_bounds__(CC_THREADS) k_cut_compact(uint32_t* __restrict__ bitmap, uint32_t* __restrict__ front,
                                                            const uint32_t* __restrict__ counts, uint32_t n_words,
                                                            uint32_t* __restrict__ cut,
                                                            uint32_t* __restrict__ front_list, uint32_t cap,
                                                            uint32_t* __restrict__ n_cut_out,
                                                            Counters* __restrict__ ctr) {
    pdl_wait();
    __shared__ uint2 s_sum[2][CC_WARPS];
    __shared__ uint32_t s_scan[2][CC_WARPS];
    __shared__ __align__(16) uint2 s_row[CC_WARPS][32];
    const uint32_t ntiles = n_words / CC_TILE_WORDS;  // the bitmaps are padded to whole tiles
    const uint32_t t = threadIdx.x, warp = t >> 5, lane = lane_id();
    uint32_t oa = 0, ob = 0, seen = 0, flip = 0;  // ids in the tiles before 'seen'
    for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, flip ^= 1u) {
        const uint32_t wi = tile * CC_TILE_WORDS + t;
        const uint32_t a = bitmap[wi], b = front[wi];
        const uint32_t said = t == 0 ? counts[tile * CC_COUNT_STRIDE] : 0u;
        uint32_t sa = 0, sb = 0;
        for (uint32_t j = seen + t; j < tile; j += CC_THREADS) {
            const uint32_t c = counts[j * CC_COUNT_STRIDE];
            sa += c & 0xFFFFu;
            sb += c >> 16;
        }
        seen = tile;
        sa = __reduce_add_sync(0xFFFFFFFFu, sa);
        sb = __reduce_add_sync(0xFFFFFFFFu, sb);
        if (lane == 0) s_sum[flip][warp] = make_uint2(sa, sb);
        uint32_t total;  // both counts packed: at most 8192 each
        const uint32_t pre = block_excl_scan<CC_WARPS>(__popc(a) | (__popc(b) << 16), s_scan[flip], &total);
#pragma unroll
        for (int w = 0; w < CC_WARPS; ++w) {
            const uint2 c = s_sum[flip][w];
            oa += c.x;
            ob += c.y;
        }
        const uint32_t id0 = (tile * CC_TILE_WORDS + 32u * warp) * 32u;
        cc_row(a, oa + (pre & 0xFFFFu), id0, cut, cap, s_row[warp]);
        cc_row(b, ob + (pre >> 16), id0, front_list, cap, s_row[warp]);
        if (a) bitmap[wi] = 0u;
        if (b) front[wi] = 0u;
        if (t == 0 && said != total) atomicOr(&ctr->flags, F_LOD_FALLBACK);  // a node was reported twice
        if (tile == ntiles - 1 && t == 0) {
            const uint32_t n = oa + (total & 0xFFFFu);
            *n_cut_out = n;
            ctr->n_front = ob + (total >> 16);
            if (n > cap) atomicOr(&ctr->flags, F_OVF_CUT);
        }
        // (the shared words of this tile are written again two barriers from here)
    }
}

// ------------------------------------------------------------ launchers
void launch_lod_update(const SceneDev& sc, const uint32_t* prev_cut, const uint32_t* n_prev, uint32_t cap_prev,
                       const FrameParams* fp, uint32_t* bitmap, uint32_t* front, uint32_t* counts, Counters* ctr, int grid,
                       bool frustum, bool interp, cudaStream_t s) {
#define VGR_LOD_UPDATE(FR, IP) \
    launch_k(k_lod_update<FR, IP>, grid, 256, s, prev_cut, n_prev, cap_prev, sc, fp, bitmap, front, counts, ctr)
    if (frustum) {
        if (interp) VGR_LOD_UPDATE(true, true);
        else VGR_LOD_UPDATE(true, false);
    } else {
        if (interp) VGR_LOD_UPDATE(false, true);
        else VGR_LOD_UPDATE(false, false);
    }
#undef VGR_LOD_UPDATE
}

void launch_lod_dense(const SceneDev& sc, const FrameParams* fp, uint32_t* bitmap, uint32_t* front, uint32_t* counts,
                      Counters* ctr, int grid, bool frustum, bool interp, cudaStream_t s) {
#define VGR_LOD_DENSE(FR, IP) launch_k(k_lod_dense<FR, IP>, grid, 256, s, sc, fp, bitmap, front, counts, ctr)
    if (frustum) {
        if (interp) VGR_LOD_DENSE(true, true);
        else VGR_LOD_DENSE(true, false);
    } else {
        if (interp) VGR_LOD_DENSE(false, true);
        else VGR_LOD_DENSE(false, false);
    }
#undef VGR_LOD_DENSE
}

void launch_lod_level(int level, const SceneDev& sc, const uint32_t* fin, uint32_t* fout, uint32_t cap,
                      const FrameParams* fp, uint32_t* bitmap, uint32_t* front, uint32_t* counts, Counters* ctr, int grid,
                      bool frustum, bool interp, cudaStream_t s) {
#define VGR_LOD_LEVEL(FR, IP) \
    launch_k(k_lod_level<FR, IP>, grid, 256, s, level, fin, fout, cap, sc, fp, bitmap, front, counts, ctr)
    if (frustum) {
        if (interp) VGR_LOD_LEVEL(true, true);
        else VGR_LOD_LEVEL(true, false);
    } else {
        if (interp) VGR_LOD_LEVEL(false, true);
        else VGR_LOD_LEVEL(false, false);
    }
#undef VGR_LOD_LEVEL
}

void launch_cut_compact(uint32_t* bitmap, uint32_t* front, const uint32_t* counts, uint32_t n_words, uint32_t* cut,
                        uint32_t* front_list, uint32_t cap, uint32_t* n_cut_out, Counters* ctr, int grid,
                        cudaStream_t s) {
    launch_k(k_cut_compact, grid, CC_THREADS, s, bitmap, front, counts, n_words, cut, front_list, cap, n_cut_out, ctr);
}

uint32_t cut_compact_tile_words() { return CC_TILE_WORDS; }
uint32_t cut_compact_count_words(uint32_t n_words) { return n_words / CC_TILE_WORDS * CC_COUNT_STRIDE; }

}  // namespace vgr
