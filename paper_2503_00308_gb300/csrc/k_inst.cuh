// k_inst.cuh -- instantiation of the per-M kernels; included once per M by
// k_m1.cu, k_m4.cu, k_m6.cu with AR_M defined.
#include "ar.h"
#include "ar_launch.h"
#include "k_prep.cuh"
#include "k_render.cuh"

#define AR_CAT2(a, b) a##b
#define AR_CAT(a, b) AR_CAT2(a, b)

namespace ar {

size_t AR_CAT(cell_data_bytes_m, AR_M)() { return sizeof(CellData<AR_M>); }
int AR_CAT(rec_width_m, AR_M)() { return Rec<AR_M>::WIDTH; }
int AR_CAT(rec_scalar_offset_m, AR_M)() { return Rec<AR_M>::SC; }

int AR_CAT(launch_call_prep_m, AR_M)(const double *lo, const double *hi, const CallConst &cc, void *cells,
                                     const float *uw_lo, const float *uw_hi, const double *Mw, double *vN,
                                     cudaStream_t st, ZeroWords za, ZeroWords zb)
{
    const unsigned cb = (unsigned)((cc.n_cells + CALL_PREP_T / 32 - 1) / (CALL_PREP_T / 32));
    const unsigned gb = vN ? (unsigned)((cc.n_gauss + CALL_PREP_T - 1) / CALL_PREP_T) : 0u;
    call_prep_kernel<AR_M><<<cb + gb, CALL_PREP_T, 0, st>>>(lo, hi, cc, (CellData<AR_M> *)cells, cb, uw_lo, uw_hi, Mw, vN,
                                                            za, zb);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int AR_CAT(launch_record_prep_m, AR_M)(const double *vN, const void *gp,
                                       const CallConst &cc, const void *cells, int TS, float *recs,
                                       PixBox *boxes, double *keys, unsigned long long *counters,
                                       cudaStream_t st, uint32_t *list, uint32_t *count)
{
    const int T = 128;
    const CellData<AR_M> *cd = (const CellData<AR_M> *)cells;
    const unsigned gb = (unsigned)((cc.n_gauss + T - 1) / T);
    // all cells of a range of Gaussians together (their vN rows stay in L2),
    // where the grid's y can hold the Gaussian blocks
    const int cf = gb <= 65535u ? 1 : 0;
    const dim3 grid = cf ? dim3((unsigned)cc.n_cells, gb) : dim3(gb, (unsigned)cc.n_cells);
    // decision part only: the value parts are built by the renderer on demand
    if (!list) {
        record_prep_kernel<AR_M, float, false><<<grid, T, 0, st>>>(vN, (const GParam *)gp, cc, cd, TS, recs, boxes,
                                                                   keys, counters, cf);
        return cudaGetLastError() == cudaSuccess ? 0 : 1;
    }
    if (cudaMemsetAsync(count, 0, sizeof(uint32_t), st) != cudaSuccess) return 1;
    cull_kernel<AR_M><<<grid, T, 0, st>>>(vN, (const GParam *)gp, cc, cd, boxes, list, count, cf);
    const uint64_t pairs = (uint64_t)cc.n_gauss * (uint64_t)cc.n_cells;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    uint64_t lg = (pairs + T - 1) / T;
    if (lg > (uint64_t)sms * 32u) lg = (uint64_t)sms * 32u;
    record_prep_list_kernel<AR_M, float, false><<<(unsigned)(lg ? lg : 1), T, 0, st>>>(
        vN, (const GParam *)gp, cc, cd, TS, recs, boxes, keys, counters, list, count);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int AR_CAT(launch_record_prep64_m, AR_M)(const double *vN, const void *gp,
                                         const CallConst &cc, const void *cells, int TS, double *recs,
                                         PixBox *boxes, double *keys, unsigned long long *counters,
                                         cudaStream_t st)
{
    const int T = 128;
    dim3 grid((unsigned)((cc.n_gauss + T - 1) / T), (unsigned)cc.n_cells);
    record_prep_kernel<AR_M, double><<<grid, T, 0, st>>>(vN, (const GParam *)gp, cc, (const CellData<AR_M> *)cells,
                                                         TS, recs, boxes, keys, counters, 0);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

template <int TS>
static int launch_render_plain_ts(const RenderLaunch &a, cudaStream_t st)
{
    const uint32_t nseg = (uint32_t)a.n_cells * (uint32_t)a.n_tiles;
    render_plain_kernel<AR_M, TS, 32><<<nseg, TS * TS, 0, st>>>(a.recs64, a.boxes, a.seg_start, a.seg_end, a.ent_ev,
                                                                a.ev_val, a.ev_key, a.W, a.H, a.ntx, a.n_tiles,
                                                                a.n_gauss, a.out_lo, a.out_hi);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int AR_CAT(launch_render_plain_m, AR_M)(int TS, const RenderLaunch &a, cudaStream_t st)
{
    return TS == 16 ? launch_render_plain_ts<16>(a, st) : launch_render_plain_ts<8>(a, st);
}

template <int TS, bool REL, int CH, int PARTS, int CTAS>
static int launch_render_parts(const RenderLaunch &a, cudaStream_t st)
{
    // double-buffered chunks of CH events (16 unless the autotuner picks 8 or
    // 32 at tile 16: the exit vote, taken once per chunk,
    // stops a part sooner with short chunks, while long chunks take fewer
    // barriers) and a ring of 4 (rings of 3-8 measured: 4 keeps the ring's
    // shared memory small)
    constexpr int RING = 4, NT = Part<TS, PARTS>::NT;
    typedef RenderSmem<AR_M, NT, CH, RING> SM;
    auto kern = render_kernel<AR_M, TS, CH, RING, REL, PARTS, CTAS>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM::BYTES) != cudaSuccess)
        return 1;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, SM::BYTES) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    // work items: the parts of every segment
    const uint64_t items = (uint64_t)a.n_cells * (uint64_t)a.n_tiles * PARTS;
    uint32_t grid = (uint32_t)(sms * per_sm);
    if (grid > items) grid = (uint32_t)items;
    // direct launches (a.direct: the active list holds every segment) take
    // one CTA per item
    if (a.direct) grid = (uint32_t)items;
    kern<<<grid, NT, SM::BYTES, st>>>(a.recs, a.boxes, a.seg_start, a.seg_end, a.seg_total, a.cell_ev,
                                      a.active, a.n_active, a.window, a.round_no,
                                      a.next_active, a.n_next, a.seg_state, a.seg_swept, a.precise, a.n_precise,
                                      a.precise_mask, a.precise_first, a.sweep_hist, a.ent_ev, a.ev_val,
                                      a.ev_key, a.W, a.H, a.ntx, a.n_tiles, a.n_gauss, a.k_open, a.fp64_dev, a.out_lo,
                                      a.out_hi, a.counters, a.work, a.direct);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

// the parts of a tile that a render sweeps, over all its rounds (see Part; the
// grid of a direct launch has one CTA per part, so their number stays below 2^31)
static int render_parts(int TS, const RenderLaunch &a)
{
    const uint64_t n_seg = (uint64_t)a.n_cells * (uint64_t)a.n_tiles;
    if (TS != 16 || n_seg < HALVES_SEGMENTS || n_seg >= (1ull << 30) || a.n_entries < HALVES_ENTRIES * n_seg) return 1;
    const bool small_rel = a.rel && AR_M > 4 && !a.dense;
    return (middle_on_edge(a.H) && n_seg < EDGE_SEGMENTS) || (small_rel && n_seg < SMALL_REL_SEGMENTS) ? 1 : 2;
}

template <int TS, bool REL, int CH = 16>
static int launch_render_ts(const RenderLaunch &a, cudaStream_t st)
{
    if constexpr (TS == 16)
        return render_parts(TS, a) == 2 ? launch_render_parts<TS, REL, CH, 2, 4>(a, st)
                                        : launch_render_parts<TS, REL, CH, 1, 2>(a, st);
    else
        return (uint64_t)a.n_cells * (uint64_t)a.n_tiles >= SIX_SEGMENTS ? launch_render_parts<TS, REL, CH, 1, 6>(a, st)
                                                                         : launch_render_parts<TS, REL, CH, 1, 4>(a, st);
}

// the FP64-capable sweep of the segments listed in a.precise (it stages 16
// entries at a time whatever the FP32 sweep's chunk is), in the form that its
// items ask for
template <int TS, bool REL, bool FULL>
static int launch_render_fp64_form(const RenderLaunch &a, uint32_t full_from, cudaStream_t st, int *launches)
{
    constexpr int CH = 16, RING = 4;
    typedef PreciseSmem<AR_M, CH, RING, FULL> SM;
    auto kern = render_fp64_kernel<AR_M, TS, CH, RING, REL, FULL>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SM)) != cudaSuccess) return 1;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32, sizeof(SM)) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const uint64_t items = (uint64_t)a.n_cells * (uint64_t)a.n_tiles * (uint64_t)(TS * TS / PRECISE_PX);
    uint32_t grid = (uint32_t)(sms * per_sm);
    if (grid > items) grid = (uint32_t)items;
    kern<<<grid, 32, sizeof(SM), st>>>(a.recs, a.boxes, a.seg_start, a.seg_end, a.seg_total, a.precise,
                                       a.precise_first, a.n_precise, a.seg_state, render_parts(TS, a), a.window,
                                       a.round_no, a.next_active, a.n_next, a.precise_mask, a.ent_ev, a.ev_val, a.ev_key,
                                       a.W, a.H, a.ntx, a.n_tiles, a.n_gauss, a.k_open, a.fp64_dev, a.out_lo, a.out_hi,
                                       a.counters, a.work_fp64, full_from);
    ++*launches;
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

template <int TS, bool REL>
static int launch_render_fp64_ts(const RenderLaunch &a, cudaStream_t st, int *launches)
{
    if (!(a.fp64_dev < AR_FP64_ALPHA_DEFAULT)) return launch_render_fp64_form<TS, REL, false>(a, 0u, st, launches);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint32_t full_from = FULL_ITEMS * (uint32_t)sms * PRECISE_CTAS;
    if (launch_render_fp64_form<TS, REL, false>(a, full_from, st, launches)) return 1;
    return launch_render_fp64_form<TS, REL, true>(a, full_from, st, launches);
}

// the deferred pairs (the counts stay on the device)
int AR_CAT(launch_finish_build_m, AR_M)(const double *vN, const CallConst &cc, const void *cells, int64_t n_gauss,
                                        const uint32_t *split_list, const uint32_t *split_count, uint32_t list_cap,
                                        const uint32_t *khigh_count, float *recs, unsigned long long *counters,
                                        cudaStream_t st)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto fin = finish_build_kernel<AR_M>;
    const int fin_smem = (int)sizeof(double) * FINISH_GROUPS * Coop<AR_M>::STRIDE;
    if (cudaFuncSetAttribute(fin, cudaFuncAttributeMaxDynamicSharedMemorySize, fin_smem) != cudaSuccess) return 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fin, FINISH_T, fin_smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    fin<<<sms * per_sm, FINISH_T, fin_smem, st>>>(vN, cc.fx, cc.fy, cc.cx, cc.cy, (const CellData<AR_M> *)cells, n_gauss,
                                                  split_list, split_count, list_cap, khigh_count, recs, counters);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int AR_CAT(launch_record_build_m, AR_M)(const double *vN, const CallConst &cc, const void *cells, int64_t n_gauss,
                                        const uint32_t *work, const uint32_t *count, float *recs,
                                        unsigned long long *counters, uint32_t *split_list, uint32_t *split_count,
                                        uint32_t list_cap, uint32_t *khigh_count, cudaStream_t st, int *launches)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const CellData<AR_M> *cd = (const CellData<AR_M> *)cells;
    // the list's length is on the device: a short list is the group builder's,
    // a long one the one-thread builder's (not launched where the pairs are too few
    // for one)
    auto coop = record_build_coop_kernel<AR_M>;
    const int coop_smem = (int)sizeof(double) * (COOP_T / 4) * Coop<AR_M>::STRIDE;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, coop, COOP_T, coop_smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int coop_most = (int)(COOP_MAX / (COOP_T / 4));
    coop<<<sms * per_sm < coop_most ? sms * per_sm : coop_most, COOP_T, coop_smem, st>>>(
        vN, cc.fx, cc.fy, cc.cx, cc.cy, cd, n_gauss, work, count, recs, counters, split_list, split_count);
    if (cudaGetLastError() != cudaSuccess) return 1;
    int n = 2;
    if (list_cap > COOP_MAX) {
        ++n;
        auto kern = record_build_kernel<AR_M>;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 128, 0) != cudaSuccess || per_sm < 1) per_sm = 1;
        kern<<<sms * per_sm, 128, 0, st>>>(vN, cc.fx, cc.fy, cc.cx, cc.cy, cd, n_gauss, work, count, recs, counters,
                                           split_list, split_count, list_cap, khigh_count);
        if (cudaGetLastError() != cudaSuccess) return 1;
    }
    if (launches) *launches += n;
    return AR_CAT(launch_finish_build_m, AR_M)(vN, cc, cells, n_gauss, split_list, split_count, list_cap, khigh_count,
                                               recs, counters, st);
}

int AR_CAT(launch_debug_alpha_m, AR_M)(const float *recs, int n, const int64_t *gi, const int32_t *px,
                                       const int32_t *py, int precision, float fp64_dev, double *out,
                                       cudaStream_t st)
{
    debug_alpha_kernel<AR_M><<<(n + 63) / 64, 64, 0, st>>>(recs, n, gi, px, py, precision, fp64_dev, out);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int AR_CAT(launch_render_m, AR_M)(int TS, const RenderLaunch &a, cudaStream_t st, int *launches)
{
    int r;
    if (TS == 8) r = a.rel ? launch_render_ts<8, true>(a, st) : launch_render_ts<8, false>(a, st);
    else if (a.ch == 8) r = a.rel ? launch_render_ts<16, true, 8>(a, st) : launch_render_ts<16, false, 8>(a, st);
    else if (a.ch == 32) r = a.rel ? launch_render_ts<16, true, 32>(a, st) : launch_render_ts<16, false, 32>(a, st);
    else r = a.rel ? launch_render_ts<16, true>(a, st) : launch_render_ts<16, false>(a, st);
    if (r) return r;
    ++*launches;
    // the segments where some pixel met an evaluation needing FP64 (window
    // abandons go to the same next list)
    if (TS == 8)
        return a.rel ? launch_render_fp64_ts<8, true>(a, st, launches) : launch_render_fp64_ts<8, false>(a, st, launches);
    return a.rel ? launch_render_fp64_ts<16, true>(a, st, launches) : launch_render_fp64_ts<16, false>(a, st, launches);
}

}  // namespace ar
