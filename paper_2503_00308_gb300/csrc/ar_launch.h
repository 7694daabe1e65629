// ar_launch.h -- host launchers of the per-M kernels (instantiated for the
// numbers of pose variables M in {1, 4, 6} carried by the linear forms).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ar {

struct CallConst;
struct PixBox;

struct RenderLaunch {
    float *recs;                      // FP32 records
    const double *recs64 = nullptr;   // FP64 records (plain renderer only)
    const PixBox *boxes;
    const uint32_t *seg_start, *seg_end, *seg_order, *ent_ev, *ev_val;
    // full-list lengths where the lists are depth prefixes (the first binning
    // phase), else null; a segment whose sweep needs more than its prefix is
    // abandoned like one that leaves its window
    const uint32_t *seg_total = nullptr;
    const uint32_t *cell_ev = nullptr;  // [n_cells + 1] first sorted event of each cell (for sweep_hist's depth part)
    // windowed rounds (FP32 renderer): segments active[0, *n_active) are swept;
    // one that needs entries beyond `window` is appended to next_active
    const uint32_t *active = nullptr, *n_active = nullptr;
    uint32_t *next_active = nullptr, *n_next = nullptr;
    uint32_t window = 0xffffffffu;
    uint32_t *sweep_hist = nullptr;   // optional [256]: completed segments by entries swept / 32, then (with
                                      // cell_ev) [64] 64-bit: their full lengths by where in the cell's
                                      // depth order they stopped, and [64] their counts
    const uint64_t *ev_key;
    int W, H, ntx, n_tiles, n_cells;
    uint64_t n_entries = 0;           // of the segments' full lists
    uint64_t n_events = 0;            // of all cells
    bool dense = false;               // (see dense_boxes)
    int64_t n_gauss;
    float k_open;                     // 1 / (1 - largest opacity), rounded up
    float fp64_dev = 3.0e38f;         // opacity evaluations whose FP32 deviation estimate exceeds this
                                      // are taken again in FP64 (pixel_alpha_fp64)
    float *out_lo, *out_hi;
    unsigned long long *counters;     // optional: [0] opacity evaluations, [1] re-evaluations,
                                      // [5] segments abandoned for a wider window ([2]-[4]: record build),
                                      // [6] evaluations taken again in FP64, [7] segments swept again for them
    unsigned int *work;               // segment counter of the persistent grid (zeroed before the first round)
    int rel = 0;                      // 1: relational upper transmittance (AR_BLEND_RELATIONAL)
    int ch = 16;                      // events per staged chunk of the FP32 sweep (8, 16 or 32 at tile 16)
    // interleave: the first round's FP32 sweep (whose active list is all n_seg
    // segments) launches one CTA per work item (direct) instead of persistent
    // CTAs, so that work on a higher-priority stream can take SMs as they free
    int interleave = 0, direct = 0;
    // the windowed rounds' state of the segments, zeroed before the first (see
    // render_kernel), and the most entries that a part of each swept
    int round_no = 0;
    uint32_t *seg_state = nullptr, *seg_swept = nullptr;
    // precision: the FP32 sweep appends a segment that needs an FP64
    // evaluation to precise, with the mask of the pixels that do in
    // precise_mask[segment * TS * TS / 32 ...] and the number of its first
    // work item in precise_first; *n_precise: the segments
    // (high word) and their work items; render_fp64_kernel takes them
    // (work_fp64: its item counter)
    uint32_t *precise = nullptr, *precise_mask = nullptr, *precise_first = nullptr;
    unsigned long long *n_precise = nullptr;
    unsigned int *work_fp64 = nullptr;
};

// Whether a screen box holds many pixels of each tile that it meets: DENSE_PX or more
// on average (triples: pixels in boxes; a box has two entries per tile).  The
// relational sweep of few segments at six pose variables takes halves of tiles only
// then (see Part).
constexpr uint64_t DENSE_PX = 32;
inline bool dense_boxes(uint64_t n_triples, uint64_t n_entries) { return 2 * n_triples >= DENSE_PX * n_entries; }

size_t cell_data_bytes(int M);
int rec_width(int M);
struct ZeroWords {  // n words to be set to 0
    uint32_t *p = nullptr;
    uint32_t n = 0;
};
// the cells' forms, and (vN non-null) the Gaussians' v and N; za and zb are zeroed
int launch_call_prep(int M, const double *lo, const double *hi, const CallConst &cc, void *cells, const float *uw_lo,
                     const float *uw_hi, const double *Mw, double *vN, cudaStream_t st, ZeroWords za = {},
                     ZeroWords zb = {});
// list, count (optional): cull the certain drops first and run the FP64
// decision chain over the list of the other pairs (cull_kernel)
int launch_record_prep(int M, const double *vN, const void *gp,
                       const CallConst &cc, const void *cells, int TS, float *recs, PixBox *boxes, double *keys,
                       unsigned long long *counters, cudaStream_t st, uint32_t *list = nullptr,
                       uint32_t *count = nullptr);
int launch_render(int M, int TS, const RenderLaunch &a, cudaStream_t st, int *launches);
int launch_record_prep64(int M, const double *vN, const void *gp,
                         const CallConst &cc, const void *cells, int TS, double *recs, PixBox *boxes, double *keys,
                         unsigned long long *counters, cudaStream_t st);
int launch_render_plain(int M, int TS, const RenderLaunch &a, cudaStream_t st);
// union of the bounds of n_cells cells of n floats each (k_union.cu); acc: fold
// the current outputs in too
int launch_bounds_union(const float *lo, const float *hi, int n_cells, size_t n, float *out_lo, float *out_hi,
                        bool acc, cudaStream_t st);
// out = out intersected with [lo, hi] elementwise (k_union.cu)
int launch_bounds_intersect(const float *lo, const float *hi, size_t n, float *out_lo, float *out_hi, cudaStream_t st);
// part[c * blocks + b] = partial sum of (hi - lo) over cell c (k_union.cu); the
// host adds the partials in order, so the sums are deterministic
int launch_width_partials(const float *lo, const float *hi, int n_cells, size_t n, int blocks, double *part,
                          cudaStream_t st);
// value parts of the records listed in work[0, *count); counters: [0] fallbacks, [1] built, [2] split.
// split_list (list_cap >= *count entries), split_count and khigh_count (zeroed by the caller): pairs whose
// MatrixInv fails on the cell, and from the back pairs whose Taylor order exceeds the default, which a last
// kernel finishes.  launches (optional) is advanced by the kernels launched.
int launch_record_build(int M, const double *vN, const CallConst &cc, const void *cells, int64_t n_gauss,
                        const uint32_t *work, const uint32_t *count, float *recs, unsigned long long *counters,
                        uint32_t *split_list, uint32_t *split_count, uint32_t list_cap, uint32_t *khigh_count,
                        cudaStream_t st, int *launches);
// concrete render (k_concrete.cu)
size_t concrete_pose_bytes();
int concrete_rec_width();
int launch_concrete_pose(const double *delta, const CallConst &cc, void *pose, cudaStream_t st);
int launch_concrete_prep(const float *uw, const double *Mw, const double *tau, const float *opac, const float *rgb,
                         const CallConst &cc, const void *pose, int TS, double *recs, PixBox *boxes, double *keys,
                         unsigned long long *counters, cudaStream_t st);
int launch_concrete_render(const double *recs, const PixBox *boxes, const uint32_t *seg_start, const uint32_t *seg_end,
                           const uint32_t *ent_ev, const uint32_t *ev_val, const uint64_t *ev_key, const void *pose,
                           int W, int H, int ntx, int n_tiles, float *out, cudaStream_t st);
int launch_scene_prep(const float *logscale, const float *quat, const float *opacity, int64_t n, double *Mw,
                      double *tau, cudaStream_t st);
int launch_gparam(const float *o_lo, const float *o_hi, const float *c_lo, const float *c_hi, int64_t n, void *gp,
                  cudaStream_t st);

}  // namespace ar
