// k_concrete.cu -- the concrete GSplat render (Algorithm 1, blended as in
// BlendInd, Algorithm 4) at sampled poses, in FP64, for soundness checks of
// the abstract bounds on the device.
//
// Per pose: concrete_pose_kernel builds R_wc(delta) and t; concrete_prep_kernel
// projects every Gaussian (d, up, Mp, X, Conic, W = Conic Mp, the pixel box
// of the ellipse m <= tau, the near plane and the frustum guard band); the
// Gaussians are binned into depth-ordered tile lists by the abstract
// renderer's binning (each Gaussian gives two events with equal keys, the
// second ignored); concrete_render_kernel blends each pixel front to back,
// Gaussians of equal depth as one group (Ind(0) = 0), until the transmittance
// is below CONC_T_STOP, which bounds the colour left out.
//
// The render is bound by the FP64 pipe (1/64 of the FP32 rate, and a warp
// instruction costs the same whatever lanes it serves), so it spends FP64 on
// full warps of (pixel, Gaussian) pairs that can matter: an FP32 test drops the
// pairs certainly beyond the cutoff, the others are listed per warp and their
// opacities taken 32 at a time, and only the blend itself runs per pixel.
#include "ar_common.cuh"
#include "ar_launch.h"
#include "k_prep.cuh"

namespace ar {

constexpr double CONC_T_STOP = 1e-13;

// record (20 doubles): d^2, d up (2), W0c (3), W1c (3), o, tau, c0, c1, c2, then
// the FP32 cutoff test's 8 floats: the projected mean as two-float sums (x hi,
// x lo, y hi, y lo) and the quadratic form A, 2 B, C of m around it, tau rounded
// up (A = B = C = 0: the test drops nothing)
constexpr int CR_D2 = 0, CR_P = 1, CR_W0 = 3, CR_W1 = 6, CR_O = 9, CR_TAU = 10, CR_COL = 11, CR_F32 = 14;
constexpr int CR_WIDTH = 20;

// e^x for x in [-CONC_XMAX, 0] by table (Tang, ACM TOMS 15(2), 1989): with
// h = ln 2 / 256 and k the integer nearest x / h, e^x = 2^(k/256) e^r, |r| <=
// h/2 = 1.4e-3, where the degree-4 Taylor polynomial of e^r leaves 4e-17.
// Eight FP64 operations against about twenty of the library call; x = -m/2
// with m <= tau <= 2 ln 255, so the table needs no other range.
constexpr double CONC_XMAX = 5.56;
constexpr int CONC_TAB = 2056;  // 2^(-j/256), j = 0 .. CONC_TAB - 1 (CONC_XMAX / h = 2053.4)

struct ConcretePose {
    double Rwc[9];
    double t[3];
    double exp_tab[CONC_TAB];
};

// R_wc(delta) = R_delta^T R0 with R_delta = Rx Ry Rz, t = t0 + delta_t
__global__ void concrete_pose_kernel(const double *__restrict__ delta, CallConst cc, ConcretePose *__restrict__ out)
{
    for (int j = threadIdx.x; j < CONC_TAB; j += blockDim.x) out->exp_tab[j] = exp2(-(double)j / 256.0);
    if (threadIdx.x != 0) return;
    double X[9], Y[9], Z[9], D[9], T[9], Rd[9], RdT[9];
    rot3(0, delta[3], X, D);
    rot3(1, delta[4], Y, D);
    rot3(2, delta[5], Z, D);
    mat3(X, Y, T);
    mat3(T, Z, Rd);
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) RdT[3 * i + j] = Rd[3 * j + i];
    mat3(RdT, cc.R0, out->Rwc);
    for (int k = 0; k < 3; ++k) out->t[k] = dadd(cc.t0[k], delta[k]);
}

// One thread per Gaussian.  counters: [2] Gaussians present, [3] tile entries.
__global__ void __launch_bounds__(128) concrete_prep_kernel(
    const float *__restrict__ uw, const double *__restrict__ Mw, const double *__restrict__ tau_g,
    const float *__restrict__ opacity, const float *__restrict__ rgb, CallConst cc,
    const ConcretePose *__restrict__ pose, int TS, double *__restrict__ recs, PixBox *__restrict__ boxes,
    double *__restrict__ keys, unsigned long long *__restrict__ counters)
{
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    uint32_t valid = 0, tiles = 0;
    if (g < cc.n_gauss) {
        PixBox box = {-1, -1, -1, -1};
        const double *Rwc = pose->Rwc;
        double uc[3], Mc[9];
        for (int a = 0; a < 3; ++a) {
            const double d0 = dsub((double)uw[3 * g], pose->t[0]);
            const double d1 = dsub((double)uw[3 * g + 1], pose->t[1]);
            const double d2 = dsub((double)uw[3 * g + 2], pose->t[2]);
            uc[a] = dadd(dadd(dmul(Rwc[3 * a], d0), dmul(Rwc[3 * a + 1], d1)), dmul(Rwc[3 * a + 2], d2));
        }
        mat3(Rwc, Mw + 9 * g, Mc);
        const double d = uc[2];
        const double o = opacity[g], tau = tau_g[g];
        const double up0 = dadd(dmul((double)cc.fx, uc[0]), dmul((double)cc.cx, d));
        const double up1 = dadd(dmul((double)cc.fy, uc[1]), dmul((double)cc.cy, d));
        // J = [[fx d, 0, -fx uc0], [0, fy d, -fy uc1]] (d^2 times the projection Jacobian)
        const double J[6] = {dmul((double)cc.fx, d), 0.0, dmul(-(double)cc.fx, uc[0]),
                             0.0, dmul((double)cc.fy, d), dmul(-(double)cc.fy, uc[1])};
        double Mp[6];
        for (int r = 0; r < 2; ++r)
            for (int c = 0; c < 3; ++c)
                Mp[3 * r + c] = dadd(dadd(dmul(J[3 * r], Mc[c]), dmul(J[3 * r + 1], Mc[3 + c])),
                                     dmul(J[3 * r + 2], Mc[6 + c]));
        double X[4];
        for (int r = 0; r < 2; ++r)
            for (int s = 0; s < 2; ++s)
                X[2 * r + s] = dadd(dadd(dmul(Mp[3 * r], Mp[3 * s]), dmul(Mp[3 * r + 1], Mp[3 * s + 1])),
                                    dmul(Mp[3 * r + 2], Mp[3 * s + 2]));
        const double det = dsub(dmul(X[0], X[3]), dmul(X[1], X[2]));
        bool alive = (d > (double)cc.near_plane) && (det > 0) && (o > 0) && (tau >= 0);
        double mux = 0, muy = 0;
        if (alive) {
            // frustum guard band (3DGS convention)
            const double gx = dmul(GUARD, (double)cc.W), gy = dmul(GUARD, (double)cc.H);
            mux = dadd((double)cc.cx, dmul((double)cc.fx, uc[0]) / d);
            muy = dadd((double)cc.cy, dmul((double)cc.fy, uc[1]) / d);
            alive = mux >= dsub((double)cc.cx, gx) && mux <= dadd((double)cc.cx, gx) &&
                    muy >= dsub((double)cc.cy, gy) && muy <= dadd((double)cc.cy, gy);
        }
        if (alive) {
            // pixel box of the ellipse m <= tau: half-extents sqrt(tau X_rr) / d^2
            const double d2 = dmul(d, d);
            const double rx = sqrt(dmul(tau, X[0])) / d2, ry = sqrt(dmul(tau, X[3])) / d2;
            double xl = dsub(mux, rx), xh = dadd(mux, rx), yl = dsub(muy, ry), yh = dadd(muy, ry);
            xl = dsub(xl, dmul(BOX_SLACK, dadd(1.0, fabs(xl))));
            xh = dadd(xh, dmul(BOX_SLACK, dadd(1.0, fabs(xh))));
            yl = dsub(yl, dmul(BOX_SLACK, dadd(1.0, fabs(yl))));
            yh = dadd(yh, dmul(BOX_SLACK, dadd(1.0, fabs(yh))));
            double fx0 = fmax(ceil(dsub(xl, 0.5)), 0.0), fx1 = fmin(floor(dsub(xh, 0.5)), (double)(cc.W - 1));
            double fy0 = fmax(ceil(dsub(yl, 0.5)), 0.0), fy1 = fmin(floor(dsub(yh, 0.5)), (double)(cc.H - 1));
            if (xh >= xl && yh >= yl && fx0 <= fx1 && fy0 <= fy1) {
                box = PixBox{(int)fx0, (int)fx1, (int)fy0, (int)fy1};
                const double conic[4] = {X[3] / det, -X[1] / det, -X[2] / det, X[0] / det};
                double *rec = recs + g * CR_WIDTH;
                rec[CR_D2] = d2;
                rec[CR_P] = dmul(d, up0);
                rec[CR_P + 1] = dmul(d, up1);
                for (int c = 0; c < 3; ++c) {
                    rec[CR_W0 + c] = dadd(dmul(conic[0], Mp[c]), dmul(conic[1], Mp[3 + c]));
                    rec[CR_W1 + c] = dadd(dmul(conic[2], Mp[c]), dmul(conic[3], Mp[3 + c]));
                }
                rec[CR_O] = o;
                rec[CR_TAU] = tau;
                for (int k = 0; k < 3; ++k) rec[CR_COL + k] = rgb[3 * g + k];
                // m = A x^2 + 2 B x y + C y^2 around the mean: A, B, C are d^4
                // times the conic.  Not tested where the covariance is so
                // ill-conditioned that the FP64 evaluation of m from W could
                // differ from this form by more than the test's margin.
                float *f = reinterpret_cast<float *>(rec + CR_F32);
                const double d4 = dmul(d2, d2);
                const bool test = dmul(X[0], X[3]) <= 1e6 * det;
                f[0] = (float)mux;
                f[1] = (float)dsub(mux, (double)f[0]);
                f[2] = (float)muy;
                f[3] = (float)dsub(muy, (double)f[2]);
                f[4] = test ? (float)dmul(d4, conic[0]) : 0.f;
                f[5] = test ? (float)dmul(2.0, dmul(d4, conic[1])) : 0.f;
                f[6] = test ? (float)dmul(d4, conic[3]) : 0.f;
                f[7] = __double2float_ru(tau);
                keys[2 * g] = d;
                keys[2 * g + 1] = d;
                valid = 1;
                tiles = (uint32_t)(box.x1 / TS - box.x0 / TS + 1) * (uint32_t)(box.y1 / TS - box.y0 / TS + 1);
            }
        }
        boxes[g] = box;
    }
    const uint32_t v = __reduce_add_sync(0xffffffffu, valid);
    const uint32_t e = __reduce_add_sync(0xffffffffu, tiles);
    if ((threadIdx.x & 31) == 0) {
        if (v) atomicAdd(&counters[2], (unsigned long long)v);
        if (e) atomicAdd(&counters[3], (unsigned long long)e);
    }
}

// One CTA per 16 x 16 tile, out is [H][W][3] of this pose; each warp blends an
// 8 x 4 block of its pixels over the tile's Gaussians, CH at a time:
//   - per Gaussian, the lanes whose pixel lies in its box and is not certainly
//     beyond the cutoff (FP32) list their (Gaussian, pixel) pair;
//   - the listed pairs' opacities in FP64, one pair per lane whatever pixel it
//     belongs to;
//   - each pixel blends its own pairs in depth order.
// FP64 operations per pair: 25 on full warps, 5 in the blend (56 in all before,
// on warps a third of whose lanes lay outside the box or beyond the cutoff).
// Four poses of 300k Gaussians at 800 x 800, projection and binning included:
// 84.9 -> 34.8 ms.
constexpr int CONC_CH = 32;
struct ConcSmem {
    double tab[CONC_TAB];
    double rec[CONC_CH][CR_WIDTH];
    double a[8][CONC_CH * 32];
    PixBox box[CONC_CH];
    uint32_t rid[CONC_CH];
    uint32_t new_key;  // bit j: Gaussian j's depth differs from the one before
    uint16_t pair[8][CONC_CH * 32];
};

__global__ void __launch_bounds__(256, 2) concrete_render_kernel(
    const double *__restrict__ recs, const PixBox *__restrict__ boxes, const uint32_t *__restrict__ seg_start,
    const uint32_t *__restrict__ seg_end, const uint32_t *__restrict__ entry_ev, const uint32_t *__restrict__ ev_val,
    const uint64_t *__restrict__ ev_key, const ConcretePose *__restrict__ pose, int W, int H, int ntx,
    float *__restrict__ out)
{
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ConcSmem &sm = *reinterpret_cast<ConcSmem *>(smem_raw);
    const int tid = threadIdx.x, ln = tid & 31, wp = tid >> 5;
    const int tile = blockIdx.x;
    // 8 x 4 pixels per warp
    const int x0 = tile % ntx * 16 + (wp & 1) * 8, y0 = tile / ntx * 16 + (wp >> 1) * 4;
    const int px = x0 + (ln & 7), py = y0 + (ln >> 3);
    const bool inside = px < W && py < H;
    const uint32_t below = (1u << ln) - 1u;
    // a Gaussian's two events have equal keys and follow one another: Gaussian
    // j of the list is entry b0 + 2 j
    const uint32_t b0 = seg_start[tile], n = (seg_end[tile] - b0) / 2u;
    if (n)
        for (int j = tid; j < CONC_TAB; j += 256) sm.tab[j] = pose->exp_tab[j];
    uint16_t *pair = sm.pair[wp];
    double *opac = sm.a[wp];
    // T: transmittance in front of the current group of equal depths, Tg: behind it
    double T = 1.0, Tg = 1.0, pc[3] = {0.0, 0.0, 0.0};
    bool done = !inside;
    for (uint32_t base = 0; base < n; base += CONC_CH) {
        if (!done && T < CONC_T_STOP) done = true;
        if (__syncthreads_and(done)) break;
        const int cnt = (int)min((uint32_t)CONC_CH, n - base);
        if (wp == 0) {
            bool nk = false;
            if (ln < cnt) {
                const uint32_t i = b0 + 2u * (base + (uint32_t)ln);
                const uint32_t e = entry_ev[i];
                nk = i == b0 || ev_key[entry_ev[i - 1]] != ev_key[e];
                const uint32_t rid = ev_val[e] >> 1;
                sm.rid[ln] = rid;
                sm.box[ln] = boxes[rid];
            }
            const uint32_t m = __ballot_sync(FULL, nk);
            if (ln == 0) sm.new_key = m;
        }
        __syncthreads();
        for (int t = tid; t < cnt * (CR_WIDTH / 2); t += 256) {
            const int e = t / (CR_WIDTH / 2), q = t - e * (CR_WIDTH / 2);
            reinterpret_cast<double2 *>(sm.rec[e])[q] =
                reinterpret_cast<const double2 *>(recs + (size_t)sm.rid[e] * CR_WIDTH)[q];
        }
        __syncthreads();
        if (__all_sync(FULL, done)) continue;
        // the pairs to evaluate
        uint32_t mine = 0, my_off = 0, my_mask = 0;  // this pixel's Gaussians; Gaussian ln's first pair and its lanes
        int total = 0;
        for (int j = 0; j < cnt; ++j) {
            const PixBox bx = sm.box[j];
            bool in = !done && px >= bx.x0 && px <= bx.x1 && py >= bx.y0 && py <= bx.y1;
            if (in) {
                // |dx|, |dy| to 2^-22 and the form's terms to 2^-21, far inside the margin
                const float4 mu = *reinterpret_cast<const float4 *>(&sm.rec[j][CR_F32]);
                const float4 q = *reinterpret_cast<const float4 *>(&sm.rec[j][CR_F32 + 2]);
                const float dx = (px + 0.5f - mu.x) - mu.y, dy = (py + 0.5f - mu.z) - mu.w;
                const float xx = q.x * dx * dx, xy = q.y * dx * dy, yy = q.z * dy * dy;
                in = !(xx + xy + yy > q.w + 1e-3f + 1e-5f * (xx + fabsf(xy) + yy));
            }
            const uint32_t m = __ballot_sync(FULL, in);
            if (in) {
                pair[total + __popc(m & below)] = (uint16_t)(j << 5 | ln);
                mine |= 1u << j;
            }
            if (ln == j) {
                my_off = (uint32_t)total;
                my_mask = m;
            }
            total += __popc(m);
        }
        __syncwarp();
        for (int i = ln; i < total; i += 32) {
            const int code = pair[i], pl = code & 31;
            const double *r = sm.rec[code >> 5];
            const double ux = x0 + (pl & 7) + 0.5, uy = y0 + (pl >> 3) + 0.5;
            const double D0 = fma(r[CR_D2], ux, -r[CR_P]), D1 = fma(r[CR_D2], uy, -r[CR_P + 1]);
            double m = 0.0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double q = fma(D0, r[CR_W0 + c], D1 * r[CR_W1 + c]);
                m = c ? fma(q, q, m) : q * q;
            }
            const double tau = r[CR_TAU];
            // the cutoff: near it, decided on the separately rounded operations
            // of the definition
            if (fabs(m - tau) <= 1e-9 * (1.0 + tau)) {
                const double E0 = dsub(dmul(r[CR_D2], ux), r[CR_P]), E1 = dsub(dmul(r[CR_D2], uy), r[CR_P + 1]);
                double md = 0.0;
                for (int c = 0; c < 3; ++c) {
                    const double q = dadd(dmul(E0, r[CR_W0 + c]), dmul(E1, r[CR_W1 + c]));
                    md = dadd(md, dmul(q, q));
                }
                m = md > tau ? 2.0 * tau + 1.0 : fmin(m, tau);
            }
            double a = 0.0;
            if (m <= tau) {
                constexpr double MAGIC = 6755399441055744.0;                  // 1.5 2^52: rounds to an integer
                const double kd = fma(m, 184.6649652337873, MAGIC);           // (m / 2) (256 / ln 2)
                const int k = __double2loint(kd);
                const double kf = kd - MAGIC;
                // r = -m/2 + k ln 2 / 256, the product in two parts
                double x = fma(kf, 0x1.62e42fefa2p-9, -0.5 * m);
                x = fma(kf, 0x1.9ef35793c7673p-49, x);
                double p = fma(x, 1.0 / 24.0, 1.0 / 6.0);
                p = fma(p, x, 0.5);
                p = fma(p, x, 1.0);
                const double t = r[CR_O] * sm.tab[k];
                a = fma(t * x, p, t);
            }
            opac[i] = a;
        }
        __syncwarp();
        // blend, front to back
        const uint32_t nk = sm.new_key;
        uint32_t passed = 0;  // the Gaussians up to the last blended one
        while (__any_sync(FULL, mine != 0u)) {
            const int j = mine ? __ffs(mine) - 1 : 0;
            const uint32_t off = __shfl_sync(FULL, my_off, j), m = __shfl_sync(FULL, my_mask, j);
            if (mine) {
                mine &= mine - 1u;
                // a new depth since the last blended Gaussian: its group is in front now
                const uint32_t upto = (2u << j) - 1u;
                if (nk & upto & ~passed) T = Tg;
                passed = upto;
                const double a = opac[off + __popc(m & below)];
                const double Ta = T * a;
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) pc[ch] = fma(Ta, sm.rec[j][CR_COL + ch], pc[ch]);
                Tg = fma(-Tg, a, Tg);
            }
        }
        if (nk & ~passed) T = Tg;
        __syncwarp();
    }
    if (inside) {
        float *o = out + ((size_t)py * W + px) * 3;
        for (int ch = 0; ch < 3; ++ch) o[ch] = (float)fmin(1.0, fmax(0.0, pc[ch]));
    }
}

int launch_concrete_pose(const double *delta, const CallConst &cc, void *pose, cudaStream_t st)
{
    concrete_pose_kernel<<<1, 1024, 0, st>>>(delta, cc, (ConcretePose *)pose);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
size_t concrete_pose_bytes() { return sizeof(ConcretePose); }
int concrete_rec_width() { return CR_WIDTH; }

int launch_concrete_prep(const float *uw, const double *Mw, const double *tau, const float *opac, const float *rgb,
                         const CallConst &cc, const void *pose, int TS, double *recs, PixBox *boxes, double *keys,
                         unsigned long long *counters, cudaStream_t st)
{
    const int T = 128;
    concrete_prep_kernel<<<(unsigned)((cc.n_gauss + T - 1) / T), T, 0, st>>>(
        uw, Mw, tau, opac, rgb, cc, (const ConcretePose *)pose, TS, recs, boxes, keys, counters);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

int launch_concrete_render(const double *recs, const PixBox *boxes, const uint32_t *seg_start, const uint32_t *seg_end,
                           const uint32_t *ent_ev, const uint32_t *ev_val, const uint64_t *ev_key, const void *pose,
                           int W, int H, int ntx, int n_tiles, float *out, cudaStream_t st)
{
    if (cudaFuncSetAttribute(concrete_render_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(ConcSmem)) != cudaSuccess)
        return 1;
    concrete_render_kernel<<<n_tiles, 256, sizeof(ConcSmem), st>>>(recs, boxes, seg_start, seg_end, ent_ev, ev_val,
                                                                   ev_key, (const ConcretePose *)pose, W, H, ntx, out);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}

}  // namespace ar
