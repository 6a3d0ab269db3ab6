// vgr_launch.h -- host-side launchers of the frame-path kernels (internal).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vgr {

// vgr_capi.cu: the thread-local message returned by vgr_last_error()
void set_last_error(const char* msg);

// Kernels of a frame are launched with programmatic stream serialization:
// a kernel's CTAs may be scheduled while the previous kernel drains, and each
// kernel waits (griddepcontrol.wait, its first statement) until the previous
// one has completed and its writes are visible, so ordering is unchanged and
// only the launch latency overlaps.  That wait covers a preceding kernel only:
// a kernel that follows copies, memsets or event records in the stream (the first
// of a frame) is launched in plain stream order (PdlScope), so it cannot start before them.
// VGR_PDL=0 in the environment turns it off everywhere.
bool pdl_enabled();
struct PdlState {
    bool on = true;          // frame kernels may use it (off while stage events sit between kernels)
    bool plain_next = false; // the next launch follows a non-kernel operation
};
PdlState& pdl_state();  // per host thread
// For the kernels of one frame: the first launch in plain order, PDL for the
// rest unless 'on' is false; restores the defaults when it ends.
struct PdlScope {
    explicit PdlScope(bool on) {
        pdl_state().on = on;
        pdl_state().plain_next = true;
    }
    ~PdlScope() { pdl_state() = PdlState{}; }
};
template <typename... KArgs, typename... Args>
inline void launch_ks(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                      Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    PdlState& st = pdl_state();
    cfg.numAttrs = pdl_enabled() && st.on && !st.plain_next ? 1 : 0;
    st.plain_next = false;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline void launch_k(void (*kernel)(KArgs...), unsigned grid, unsigned block, cudaStream_t s, Args... args) {
    launch_ks(kernel, grid, block, 0, s, args...);
}

struct SceneDev;
struct FrameParams;
struct Counters;

// k_frame.cu
// What a frame starts from: up to three regions of zeros (16-byte units) and the
// tile ranges, all ones.
struct FrameClear {
    uint4* zero[3];
    size_t zero16[3];
    uint2* ranges;
    uint32_t n_ranges;
};
// host: the parameters in pinned host memory, as the device sees it
void launch_frame_begin(const FrameParams* host, FrameParams* dev, const FrameClear& c, int sms, cudaStream_t s);

// k_lod.cu
void launch_lod_update(const SceneDev& sc, const uint32_t* prev_cut, const uint32_t* n_prev, uint32_t cap_prev,
                       const FrameParams* fp, uint32_t* bitmap, uint32_t* front, uint32_t* counts, Counters* ctr, int grid,
                       bool frustum, bool interp, cudaStream_t s);
// the whole from-scratch cut in one pass (F_NONMONOTONE: to be redone level by level)
void launch_lod_dense(const SceneDev& sc, const FrameParams* fp, uint32_t* bitmap, uint32_t* front, uint32_t* counts,
                      Counters* ctr, int grid, bool frustum, bool interp, cudaStream_t s);
void launch_lod_level(int level, const SceneDev& sc, const uint32_t* fin, uint32_t* fout, uint32_t cap,
                      const FrameParams* fp, uint32_t* bitmap, uint32_t* front, uint32_t* counts, Counters* ctr, int grid,
                      bool frustum, bool interp, cudaStream_t s);
void launch_cut_compact(uint32_t* bitmap, uint32_t* front, const uint32_t* counts, uint32_t n_words, uint32_t* cut,
                        uint32_t* front_list, uint32_t cap, uint32_t* n_cut_out, Counters* ctr, int grid,
                        cudaStream_t s);
uint32_t cut_compact_tile_words();
uint32_t cut_compact_count_words(uint32_t n_words);  // words of the tiles' counters

// k_preprocess.cu
// Per in-front entry i (the entry's node id is the in-front list's entry i)
struct VisBuffers {
    uint32_t* depth;
    uint32_t* ntile;
    // 2 float4 per entry, one 32-byte sector: u v A B (rho = A dx^2 + B dx dy + C dy^2), then C, thr, the candidate
    // tiles (pack_rect) and the footprint box's half-height | half-width << 16 (FP16 bits, rounded up)
    float4* rec;
    float4* rgb;    // r g b theta
    float* lw;      // parent weight of the interpolated Gaussian (weight interpolation only)
};
void launch_preprocess(const SceneDev& sc, const uint32_t* front, const uint32_t* n_front, uint32_t cap,
                       const FrameParams* fp, VisBuffers vis, Counters* ctr, uint32_t* depth_bins, bool interp,
                       int grid, cudaStream_t s);
// The records of n entries as vgr_debug_buffers lays them out
void launch_debug_records(const VisBuffers& vis, uint32_t n, uint2* rect, float4* recA, float4* recB, float4* rgb,
                          cudaStream_t s);
// the culled entries of order[n_vis .. n)
void launch_debug_culled(const VisBuffers& vis, uint32_t n, uint32_t n_vis, uint32_t* order, cudaStream_t s);
void prepare_scene(float4* covB, uint32_t n, cudaStream_t s);
void prepare_scene_half(float4* covB, uint32_t n, cudaStream_t s);

// k_depth.cu
// Depth order of the visible entries and their first pair slots: order[r] is
// the in-front index of depth rank r, slot_off[r] its first slot (r <= n_vis).
uint32_t depth_bucket_cap(uint32_t cap_vis);  // bucket ids a frame of cap_vis entries can have, plus one
cudaError_t depth_sort_init();                // once per device: the kernels' shared-memory limits
void launch_depth_sort(const VisBuffers& vis, uint32_t cap_vis, const uint32_t* bins, uint2* bstart,
                       unsigned long long* cursor, uint2* part, uint32_t* order, uint32_t* slot_off,
                       uint32_t* owner, uint64_t cap_pairs, Counters* ctr, const FrameParams* fp, int sms,
                       cudaStream_t s);

// k_sort.cu
// Tables of one digit pass: digit counts per row (a tile's keys, or a part of
// it) and per RADIX_GROUP rows; the groups are cleared before they are counted.
struct RadixTab {
    uint16_t* rows;
    uint32_t* groups;
};
// (row_len: keys per row of the tables, or 0 for one row per tile, of whichever size)
size_t radix_row_words(uint64_t n, uint32_t row_len, int bits);    // 16-bit words of the rows
size_t radix_group_words(uint64_t n, uint32_t row_len, int bits);  // 32-bit words of the groups
int radix_grid(int sms);
// one row per tile
void launch_radix_count(const uint32_t* keys, const uint32_t* n32, const unsigned long long* n64, uint64_t cap,
                        int shift, int bits, RadixTab tab, int grid, cudaStream_t s);
// bits: 5 to 8; row_len: RADIX_TILE_SMALL or a divisor of it, or 0 for the rows of launch_radix_count; the element
// count is *n32, *n64 or (both null) cap, and at most cap
void launch_radix_scatter(const uint32_t* keys_in, const uint32_t* vals_in, uint32_t* keys_out, uint32_t* vals_out,
                          const uint32_t* n32, const unsigned long long* n64, uint64_t cap, int shift, int bits,
                          RadixTab tab, uint32_t row_len, bool drop, int grid, cudaStream_t s, uint2* ranges = nullptr,
                          uint32_t n_ranges = 0);

// k_emit.cu
// slot offsets in depth order, into slot_off[cap_vis + 1], after a radix depth sort
void launch_slot_scan(const uint32_t* order, uint32_t cap_vis, const VisBuffers& vis, uint32_t* slot_off,
                      uint32_t* owner, uint64_t cap_pairs, unsigned long long* status, Counters* ctr,
                      const FrameParams* fp, int grid, cudaStream_t s);
uint32_t emit_owner_cap(uint64_t cap_pairs);  // entries of the owner table (first rank of each emission chunk)
// 'tab' receives the counts of the keys' low 'bits' bits, one row per EMIT_SLOTS slots; dropped slots (key all ones)
// are not counted
void launch_emit(const uint32_t* order, uint32_t cap_vis, const VisBuffers& vis, const uint32_t* slot_off,
                 const uint32_t* owner, uint32_t* pair_key, uint32_t* pair_val, uint64_t cap_pairs, int bits,
                 RadixTab tab, Counters* ctr, const FrameParams* fp, int grid, cudaStream_t s);
// the tile of every sorted pair, from the ranges
void launch_debug_tiles(const uint2* ranges, uint32_t n_tiles, uint32_t* pair_tile, uint64_t n_pairs, cudaStream_t s);
uint32_t slot_scan_tile();
void launch_tile_order(uint2* ranges, uint32_t n_tiles, uint32_t* order, Counters* ctr, cudaStream_t s);
constexpr uint32_t BATCH_VIEWS_MAX = 1024;  // views of one batch blend (k_batch_offsets: one thread each)

// k_blend.cu: the persistent blend over a work list of (view << 20 | tile)
// items in blend order; fps == null: every item is of the view of fp0.  next[0..1]
// (zero before the launch) hand out the list's tiles; *n_heavy: how many of
// them, from the start, are of BL_HEAVY_CLASS or above.  The last CTA writes the
// status of fp0's view, or of the n_views views of fps, to their host buffers;
// *done (zero before the launch) finds it.  depth: hits staged per
// chunk (16, 32, 48; 48 needs tiles of 16 or 32); tile: 8, 16 or 32 pixels.
constexpr uint32_t BL_HEAVY_CLASS = 11;  // class floor(log2(pairs + 1)) + 1: 1023 pairs and more
void launch_blend(const FrameParams* fp0, const FrameParams* const* fps, const uint32_t* work, uint32_t n_work,
                  const uint32_t* n_heavy, uint32_t* next, uint32_t* done, uint32_t n_views, int sms, uint32_t filter,
                  uint32_t exp_mode, uint32_t depth, uint32_t tile, cudaStream_t s);
// k_emit.cu: the order of a batch's tiles over all its views (heaviest class
// first), from each view's tile order and class counts
void launch_batch_order(const FrameParams* const* fps, uint32_t n_views, const uint32_t* const* orders,
                        const uint32_t* tile_base, uint32_t total_tiles, uint32_t* delta, uint32_t* work,
                        uint32_t* n_heavy, int grid, cudaStream_t s);

// vgr_sort_api.cu: enqueue a standalone pair sort on caller-provided scratch
size_t sort_row_words(uint64_t n);                  // 16-bit words
size_t sort_group_words(uint64_t n, int passes);    // 32-bit words
int sort_passes(uint32_t key_bits);
cudaError_t sort_pairs_enqueue(const uint32_t* keys_in, const uint32_t* vals_in, uint32_t* keys_out,
                               uint32_t* vals_out, uint64_t n, int passes, uint16_t* rows, uint32_t* groups,
                               uint32_t* tmp_keys, uint32_t* tmp_vals, int sms, cudaStream_t s);

// k_store.cu
void convert_sh_half(const float* src, uint32_t n, uint32_t k3, void* dst, uint32_t stride, cudaStream_t s);
void convert_cov_bf16(const float* src6, uint32_t n, void* dst, cudaStream_t s);

}  // namespace vgr
