// FP64-accurate operators on one tile (one detector, up to 4096 samples) per CTA: the normal operator
// acc += P^T N^-1 P x, the right-hand side acc += P^T N^-1 d and N^-1 alone (Furax paper: the estimator
// A = (H.T @ N.I @ H).I @ H.T @ N.I of the Software Design listing, with the block decomposition
// P^T N^-1 P = sum_i P_i^T N_i^-1 P_i of "Algebraic reductions"), for FURAX_F64 and FURAX_PREC_F32X2.
//
// Each CTA forms the tile's samples with their 63-sample halos in registers, applies the band on the tensor
// cores (band_tc.cuh) and scatters y (1, cos 2psi, sin 2psi) in time order as whole FP64 pixel records; the
// pointing is read a second time for the scatter (from L2), which leaves the shared memory to the digits.
// What bounds it: the L2's FP64 reductions (3 per sample, 18,000 cycles per tile and SM at the rate of
// furax_probe_l2 kind 5) and the latency of the phases before them (fill 4,000 from data, 21,000 through a map;
// digits and sums 4,000; products 9,000; accumulators to y 5,000-7,000 cycles), which two CTAs per SM overlap in part.
// Each CTA has 512 threads at 64 registers: with 256 at 128 the same phases took 5,000 / 26,000, 4,000, 9,000 and
// 6,000-10,000 cycles and the scatter 33,000 instead of 23,000. Measured (GB300): FP64 FMAs (double-FP32 for the
// right-hand side), 256 threads, now:
//   normal operator, 32 x 262,147 samples, nside 256, FP64 cache   2277, 329, 284 us
//   right-hand side, 128 x 524,288 FP32 samples, mixed cache       3440, 1730, 1428 us
//   N^-1 alone, 32 x 131,071 samples                               1011, 61, 64 us
// (277, 1387 and 58 us before every block of outputs was checked and the taps had eight digits, band_tc.cuh.)
#include "tc_sample.cuh"
#include "tpl_eval.cuh"

namespace fx {

// Template correction of the right-hand side, y -= (W T) b for amplitudes b already solved from d: in the
// interior of a stream a cubic in the offset j of the sample from the middle of the tile's own samples
// (no extrapolation in tau), summed term by term near the stream's ends.
struct TplCorr {
    double e[4];
    __device__ __forceinline__ void init(const TplView &tv, const Tile &tl, const ObsInfo &ob, int64_t gdet)
    {
        const double h = ob.nsamp > 1 ? 2.0 / (double)(ob.nsamp - 1) : 0.0;
        const double2 m = tv.mom[gdet];
        const double bv[4] = {tv.b[4 * gdet], tv.b[4 * gdet + 1], tv.b[4 * gdet + 2], tv.b[4 * gdet + 3]};
        double c[4];
        tpl_cubic(m.x, m.y * h * h * 0.5, bv, c);
        cubic_shift(c, tpl_tau_ref(tl.t0 + (tl.len >> 1), ob.nsamp), h, e);
    }
    __device__ __forceinline__ double apply(double y, const NoiseView &nv, const TplView &tv, const Tile &tl,
                                            const ObsInfo &ob, int64_t gdet, int k) const
    {
        const int64_t t = tl.t0 + k;
        if (tpl_interior(tv, t, ob.nsamp)) {
            const double j = (double)(k - (tl.len >> 1));
            return y - fma(fma(fma(e[3], j, e[2]), j, e[1]), j, e[0]);
        }
        double w[4];
        wt_eval<double>(nv, tv, gdet, ob.nsamp, t, w);
#pragma unroll
        for (int l = 0; l < 4; ++l) y -= tv.b[4 * gdet + l] * w[l];
        return y;
    }
};

// FROM_TOD: samples d, else P x. TPL (FROM_TOD only): with the template correction.
template <int MODE, bool FROM_TOD, bool TPL, typename DT>
__global__ void __launch_bounds__(TT, 2) tc_operator_kernel(const Tile *__restrict__ tiles, PointingView pv, NoiseView nv,
                                                            const double4_32a *__restrict__ x, const DT *__restrict__ d,
                                                            double *__restrict__ acc64, unsigned *__restrict__ err,
                                                            bool f64, TplView tv, const unsigned *__restrict__ done, unsigned n_obs)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ TplCorr corr;
    if (done && *done == n_obs) return;
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = pv.obs[tl.obs];
    const int64_t gdet = ob.det_off + tl.det;
    const DetOffset psi(pv, gdet);
    tc_begin(sm, nv, gdet, err);
    if constexpr (TPL)
        if (threadIdx.x == 0) corr.init(tv, tl, ob, gdet);
    {
        double v[kTcPer];
        const TcSlots sl(tl, ob);
        auto fill = [&](double (&w)[kTcPer]) {
            if constexpr (FROM_TOD) tc_fill_tod(w, sl, d);
            else tc_fill_map<MODE, false>(sm, w, sl, pv, ob, tl, psi, x, d);
        };
        fill(v);
        bool ok;
        if constexpr (MODE == 0 && !FROM_TOD)   // the recipe costs more than the registers
            ok = tc_band(sm, v, nv, gdet, err, f64, tl.len, TcKeep{v});
        else
            ok = tc_band<!FROM_TOD || sizeof(DT) == 8>(sm, v, nv, gdet, err, f64, tl.len, fill);
        if (!ok) return;
    }
    const double *ys = tc_ys(sm);
    double *rec = acc64 + 3 * ob.map_off;
    tc_each<MODE == 0 && !FROM_TOD ? kTcKept : MODE, TT, 4>(pv, ob, tl, psi, [](int, int32_t) { return TcNone{}; },
                         [&](int k, int32_t pix, double c, double s, TcNone) {
        double y = pix >= 0 ? ys[spos(k)] : 0.0;
        if constexpr (TPL)
            if (pix >= 0) y = corr.apply(y, nv, tv, tl, ob, gdet, k);
        const double v[3] = {y, y * c, y * s};
        red_add_f64_records_warp<3, double>(rec, pix, v, tc_stage(sm), tc_stage_pix(sm));
    });
}

// White noise: no neighbours, so each sample goes straight from the gather to its records.
template <int MODE, bool FROM_TOD, bool TPL, typename DT>
__global__ void __launch_bounds__(FT) white_operator_kernel(const Tile *__restrict__ tiles, PointingView pv, NoiseView nv,
                                                            const double4_32a *__restrict__ x, const DT *__restrict__ d,
                                                            double *__restrict__ acc64, TplView tv,
                                                            const unsigned *__restrict__ done, unsigned n_obs)
{
    __shared__ double stage[FT / 32][96];
    __shared__ int32_t spix[FT / 32][32];
    __shared__ TplCorr corr;
    if (done && *done == n_obs) return;
    const Tile tl = tile_part(tiles[blockIdx.x]);
    if (tl.len <= 0) return;
    const ObsInfo ob = pv.obs[tl.obs];
    const int64_t gdet = ob.det_off + tl.det;
    const DetOffset psi(pv, gdet);
    if constexpr (TPL) {
        if (threadIdx.x == 0) corr.init(tv, tl, ob, gdet);
        __syncthreads();
    }
    const double w = nv.p64[gdet];
    const DT *row = d + ob.tod_off + (int64_t)tl.det * ob.nsamp + tl.t0;
    double *rec = acc64 + 3 * ob.map_off;
    const int warp = threadIdx.x >> 5;
    struct In {   // map record or datum
        TcPix m;
        DT d;
    };
    tc_each<MODE, FT, 4>(pv, ob, tl, psi, [&](int k, int32_t pix) {
        In in;
        if constexpr (FROM_TOD) in.d = __ldg(row + k);
        else in.m.load(x, ob.map_off + max(pix, 0));
        return in;
    }, [&](int k, int32_t pix, double c, double s, const In &in) {
        double y = 0.0;
        if (pix >= 0) {
            if constexpr (FROM_TOD) y = tod_f64(in.d) * w;
            else y = in.m.project(pix, c, s) * w;
            if constexpr (TPL) y = corr.apply(y, nv, tv, tl, ob, gdet, k);
        }
        const double v[3] = {y, y * c, y * s};
        red_add_f64_records_warp<3, double>(rec, pix, v, stage[warp], spix[warp]);
    });
}

// out = N^-1 in on an FP64 TOD, banded.
__global__ void __launch_bounds__(TT, 2) tc_ninv_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                        NoiseView nv, const double *__restrict__ in,
                                                        double *__restrict__ out, unsigned *__restrict__ err, bool f64)
{
    extern __shared__ __align__(128) unsigned char sm[];
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    const int64_t gdet = ob.det_off + tl.det;
    const int64_t row = ob.tod_off + (int64_t)tl.det * ob.nsamp;
    tc_begin(sm, nv, gdet, err);
    double v[kTcPer];
    const TcSlots sl(tl, ob);
    tc_fill_tod(v, sl, in);
    const bool ok = tc_band(sm, v, nv, gdet, err, f64, tl.len, [&](double (&w)[kTcPer]) { tc_fill_tod(w, sl, in); });
    const double *ys = tc_ys(sm);   // NaN where there are no results: this handle's status may never be asked for
    for (int k = threadIdx.x; k < tl.len; k += TT) out[row + tl.t0 + k] = ok ? ys[spos(k)] : __longlong_as_double(-1LL);
}

furax_status launch_ninv_tc(const furax_noise *n, const double *in, double *out, bool f64, unsigned *err, cudaStream_t st)
{
    if (n->n_tiles == 0) return FURAX_OK;
    furax_status rc = launch_dyn(tc_ninv_kernel, (unsigned)n->n_tiles, TT, kTcSmem, st, n->d_tiles, n->d_obs, n->view(), in, out,
                                 err, f64);
    if (rc) return rc;
    count_launches(1);
    return check_launch("N^-1 apply (FP64, banded)");
}

template <int MODE, bool FROM_TOD, bool TPL, typename DT>
static furax_status run_tc(const furax_pointing *p, const furax_noise *n, const double4_32a *x, const DT *d, double *a64,
                           bool f64, const TplView &tv, const unsigned *done, cudaStream_t st)
{
    if constexpr (MODE == 0 && !FROM_TOD) {
        if (n->kind == FURAX_NOISE_BANDED)
            return each_kept_chunk(p, [&](const Tile *tiles, unsigned g, const PointingView &pv) {
                return launch_dyn(tc_operator_kernel<MODE, FROM_TOD, TPL, DT>, g, TT, kTcSmem, st, tiles, pv, n->view(), x, d, a64,
                                  p->d_err, f64, tv, done, (unsigned)p->n_obs);
            });
    }
    if (n->kind == FURAX_NOISE_BANDED)
        return launch_dyn(tc_operator_kernel<MODE, FROM_TOD, TPL, DT>, (unsigned)p->n_tiles, TT, kTcSmem, st, p->d_tiles,
                          p->view(), n->view(), x, d, a64, p->d_err, f64, tv, done, (unsigned)p->n_obs);
    white_operator_kernel<MODE, FROM_TOD, TPL, DT><<<tile_grid(p), FT, 0, st>>>(p->d_tiles, p->view(), n->view(), x,
                                                                                         d, a64, tv, done,
                                                                                         (unsigned)p->n_obs);
    return FURAX_OK;
}

template <bool FROM_TOD, bool TPL, typename DT>
static furax_status dispatch_tc(const furax_pointing *p, const furax_noise *n, const double4_32a *x, const DT *d, double *a64,
                                bool f64, const TplView &tv, const unsigned *done, cudaStream_t st)
{
    if (p->n_tiles == 0) return FURAX_OK;
    furax_status rc;
    switch (p->mode) {
    case FURAX_POINTING_ON_THE_FLY: rc = run_tc<0, FROM_TOD, TPL, DT>(p, n, x, d, a64, f64, tv, done, st); break;
    case FURAX_POINTING_CACHE_F32: rc = run_tc<1, FROM_TOD, TPL, DT>(p, n, x, d, a64, f64, tv, done, st); break;
    case FURAX_POINTING_CACHE_MIXED: rc = run_tc<3, FROM_TOD, TPL, DT>(p, n, x, d, a64, f64, tv, done, st); break;
    default: rc = run_tc<2, FROM_TOD, TPL, DT>(p, n, x, d, a64, f64, tv, done, st);
    }
    if (rc) return rc;
    count_launches(1);
    return check_launch(FROM_TOD ? "right-hand side P^T N^-1 d" : "fused P^T N^-1 P (FP64)");
}

__global__ void pack_x4_kernel(const double *__restrict__ x, const uint8_t *__restrict__ valid, double4_32a *__restrict__ x4,
                               int64_t np)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
        const bool ok = !valid || valid[i];
        x4[i] = ok ? double4_32a{x[3 * i], x[3 * i + 1], x[3 * i + 2], 0.0} : double4_32a{0.0, 0.0, 0.0, 0.0};
    }
}

furax_status launch_pack_x4(const furax_pointing *p, const double *x, const uint8_t *valid, cudaStream_t st)
{
    furax_pointing *pm = const_cast<furax_pointing *>(p);
    const int64_t np = p->npix_total;
    furax_status rc = ensure_ws(pm, (void **)&pm->ws_x4, sizeof(double4_32a) * (size_t)np);
    if (rc) return rc;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((np + 255) / 256, 8LL * p->n_sm));
    pack_x4_kernel<<<g, 256, 0, st>>>(x, valid, pm->ws_x4, np);
    count_launches(1);
    return check_launch("pack FP64 map");
}

furax_status launch_fused_tc_packed(const furax_pointing *p, const furax_noise *n, double *a64, bool f64,
                                    const unsigned *done, cudaStream_t st)
{
    return dispatch_tc<false, false, double>(p, n, p->ws_x4, nullptr, a64, f64, TplView{}, done, st);
}

furax_status launch_fused_tc(const furax_pointing *p, const furax_noise *n, const double *x, const uint8_t *valid, double *a64,
                             bool f64, cudaStream_t st)
{
    furax_status rc = launch_pack_x4(p, x, valid, st);
    if (rc) return rc;
    return launch_fused_tc_packed(p, n, a64, f64, nullptr, st);
}

furax_status launch_rhs_tc(const furax_pointing *p, const furax_noise *n, const void *d, int d_t, double *a64, bool f64,
                           cudaStream_t st, const furax_templates *tp)
{
    const double *d64 = (const double *)d;
    const float *d32 = (const float *)d;
    if (tp) {
        const TplView tv = tp->view();
        return d_t == FURAX_F64 ? dispatch_tc<true, true, double>(p, n, nullptr, d64, a64, f64, tv, nullptr, st)
                                : dispatch_tc<true, true, float>(p, n, nullptr, d32, a64, f64, tv, nullptr, st);
    }
    return d_t == FURAX_F64 ? dispatch_tc<true, false, double>(p, n, nullptr, d64, a64, f64, TplView{}, nullptr, st)
                            : dispatch_tc<true, false, float>(p, n, nullptr, d32, a64, f64, TplView{}, nullptr, st);
}

// Digits of a detector's taps (one CTA each): 63-bit integers relative to 2^ec, balanced base-256
// digits, stored as the distinct core matrices of the operand (band_tc.cuh): [digit][matrix h][row r][column e]
// is the tap of lag index 8 h - 8 + e - r (0 .. 126).
__global__ void __launch_bounds__(128) tap_digits_kernel(const double *__restrict__ taps, int ntaps,
                                                         unsigned char *__restrict__ out, int32_t *__restrict__ exps,
                                                         float *__restrict__ weights)
{
    __shared__ double c[MAXTAPS];
    const int64_t det = blockIdx.x;
    if (threadIdx.x < MAXTAPS) c[threadIdx.x] = threadIdx.x < ntaps ? taps[det * ntaps + threadIdx.x] : 0.0;
    __syncthreads();
    double m = 0.0;   // largest tap
    bool finite = true;
    for (int k = 0; k < MAXTAPS; ++k) {
        m = fmax(m, fabs(c[k]));
        finite = finite && isfinite(c[k]);
    }
    bool ok = finite && m > 0.0;
    // |c| 2^(63 - ec) <= 0x7f7f7f7f7f7f7f7f, the largest integer of eight balanced digits
    int ec = ok ? ilogb(m) + 1 : 0;
    if (scalbn(m, -ec) > 0.99) ++ec;
    // Weight m: the smallest tap between sample block o + m and output block o (tap index 8 m - 7 .. 8 m + 7).
    __shared__ float w[kTcWeights];
    if (threadIdx.x < kTcWeights - 1) {
        double v = m;
        for (int j = 8 * (int)threadIdx.x - 7; j <= 8 * (int)threadIdx.x + 7; ++j)
            v = j < 0 || j >= kBand ? 0.0 : fmin(v, fabs(c[j < kHalo ? kHalo - j : j - kHalo]));
        w[threadIdx.x] = ok ? (float)scalbn(v, -ec) : 0.f;
        weights[det * kTcWeights + threadIdx.x] = w[threadIdx.x];
    }
    // The same for groups of 32 samples: the smallest sum, over the 32 places an output can have, of the smallest tap of
    // each group that lies within its band (three or four).
    __shared__ double place[32];
    if (threadIdx.x < 32) {
        double sum = 0.0;
        for (int j0 = (32 - (int)threadIdx.x) % 32; j0 + 32 <= kBand; j0 += 32) {
            double v = m;
            for (int j = j0; j < j0 + 32; ++j) v = fmin(v, fabs(c[j < kHalo ? kHalo - j : j - kHalo]));
            sum += v;
        }
        place[threadIdx.x] = sum;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = place[0];
        for (int i = 1; i < 32; ++i) v = fmin(v, place[i]);
        weights[det * kTcWeights + kTcWeights - 1] = ok ? (float)scalbn(v, -ec) : 0.f;
    }
    // Gaussian samples have sums of 6.4 sigma = 1.6 X where X = 4 sigma; twice that over the line on average leaves few
    // blocks of ordinary noise below it.
    float sum = 0.f;
    for (int i = 0; i < kTcWeights - 1; ++i) sum += w[i];
    ok = ok && 1.6f * sum >= ldexpf(2.f, -kTcRange);
    if (threadIdx.x == 0) exps[det] = ok ? ec : finite ? kTcNoTaps : kTcBadTaps;
    __half *o = reinterpret_cast<__half *>(out + det * kTcDetBytes);
    for (int i = threadIdx.x; i < kTcCores * 64; i += 128) {
        const int j = 8 * (i >> 6) - 8 + (i & 7) - ((i >> 3) & 7);
        const int lag = j < kHalo ? kHalo - j : j - kHalo;
        const double v = ok && j >= 0 && j < kBand ? scalbn(c[lag], 63 - ec) : 0.0;
        const uint64_t d = (uint64_t)__double2ll_rn(v) + 0x8080808080808080ull;
        for (int g = 0; g < kTcCDig; ++g)
            o[g * kTcCores * 64 + i] = __int2half_rn((int)((d >> (8 * (kTcCDig - 1 - g))) & 0xff) - 128);
    }
}

size_t tc_taps_bytes(int64_t ndet) { return (size_t)kTcDetBytes * (size_t)ndet; }
size_t tc_weights_bytes(int64_t ndet) { return sizeof(float) * kTcWeights * (size_t)ndet; }

furax_status prepare_noise_tc(furax_noise *n, cudaStream_t st)
{
    furax_status rc;
    const size_t nd = (size_t)n->ndet_total;
    if ((rc = allow_smem((const void *)tc_ninv_kernel, kTcSmem))) return rc;
    tap_digits_kernel<<<(unsigned)nd, 128, 0, st>>>(n->p64, n->ntaps, n->tc_taps, n->tc_exp, n->tc_w);
    count_launches(1);
    return check_launch("tap digits");
}

template <int MODE>
static furax_status prep_tc_mode()
{
    furax_status rc = FURAX_OK;
    if (!rc) rc = allow_smem((const void *)tc_operator_kernel<MODE, false, false, double>, kTcSmem);
    if (!rc) rc = allow_smem((const void *)tc_operator_kernel<MODE, true, false, double>, kTcSmem);
    if (!rc) rc = allow_smem((const void *)tc_operator_kernel<MODE, true, false, float>, kTcSmem);
    if (!rc) rc = allow_smem((const void *)tc_operator_kernel<MODE, true, true, double>, kTcSmem);
    if (!rc) rc = allow_smem((const void *)tc_operator_kernel<MODE, true, true, float>, kTcSmem);
    return rc;
}

furax_status prepare_fused_tc()
{
    furax_status rc = prep_tc_mode<0>();
    if (!rc) rc = prep_tc_mode<1>();
    if (!rc) rc = prep_tc_mode<2>();
    if (!rc) rc = prep_tc_mode<3>();
    return rc;
}

furax_status prepare_kernels()
{
    static furax_status done = 1;
    if (done == FURAX_OK) return FURAX_OK;
    furax_status rc = prepare_fused_f32();
    if (!rc) rc = prepare_fused_tc();
    done = rc;
    return rc;
}

}  // namespace fx
