// chi^2 = r^T N^-1 r, r = d - P m, with its gradients -2 P^T N^-1 r in the map and -2 sum (N^-1 r) 2 (U c - Q s)
// in the detectors' polarisation angles (the paper's differentiability, "Summary"), FP64-accurate, for
// FURAX_F64 and FURAX_PREC_F32X2: the tile skeleton of fused_tc.cu, the band on the tensor cores.
//
// r stays in the registers it was formed in until y is known; the map records are gathered a second time for the
// angle gradient. Bound by the FP64 pipe (9 instructions per sample and 8 more for angle offsets, where the FMA chain
// took 127 for the band alone) and the phases' latency: 128 x 131,072 samples, nside 256, FP64 cache: 4561 us with the
// chain, 919 us with r formed a second time beside y and 256 threads, 857 us now.
#include "tc_sample.cuh"

namespace fx {

// White noise has no phases to overlap: half as many threads and four CTAs per SM, so that small observations end in one
// round (16 x 131,072 samples, mixed cache: 105 us with 512 threads, 101 so, 91 with two FP64 instructions less).
template <bool BANDED> constexpr int kChiThreads = BANDED ? TT : 256;

template <int MODE, bool BANDED, typename DT>
__global__ void __launch_bounds__(kChiThreads<BANDED>, BANDED ? 2 : 4) chi2_tc_kernel(const Tile *__restrict__ tiles, PointingView pv, NoiseView nv,
                                                        const DT *__restrict__ d, const double4_32a *__restrict__ m,
                                                        double *__restrict__ chi2, double *__restrict__ grad_map,
                                                        double *__restrict__ grad_psi, unsigned *__restrict__ err, bool f64)
{
    extern __shared__ __align__(128) unsigned char sm[];
    constexpr int NT = kChiThreads<BANDED>;
    __shared__ double red[2][NT / 32];
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = pv.obs[tl.obs];
    const int64_t gdet = ob.det_off + tl.det;
    const DetOffset psi(pv, gdet);
    const DT *row = d + ob.tod_off + (int64_t)tl.det * ob.nsamp;
    double w = 0.0, *stage;
    int32_t *spix;
    double part_chi2 = 0.0, part_psi = 0.0;
    const double *ys = tc_ys(sm);
    if constexpr (BANDED) {
        stage = tc_stage(sm);
        spix = tc_stage_pix(sm);
        tc_begin(sm, nv, gdet, err);
        double v[kTcPer];
        const TcSlots sl(tl, ob);
        tc_fill_map<MODE, true>(sm, v, sl, pv, ob, tl, psi, m, d);
        if (!tc_band(sm, v, nv, gdet, err, f64, tl.len, TcKeep{v})) return;
        // r^T N^-1 r over this thread's own slots: r is still at hand
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) {
            const int t = sl.slot(k) - kHalo;
            if (t >= 0 && t < tl.len) part_chi2 = fma(v[k], ys[spos(t)], part_chi2);
        }
    } else {
        __shared__ double wstage[NT / 32][96];
        __shared__ int32_t wpix[NT / 32][32];
        stage = wstage[threadIdx.x >> 5];
        spix = wpix[threadIdx.x >> 5];
        w = -2.0 * nv.p64[gdet];
    }
    double *rec = grad_map ? grad_map + 3 * ob.map_off : nullptr;
    struct In {
        TcPix m;
        DT d;
    };
    tc_each<MODE == 0 && BANDED ? kTcKept : MODE, NT, 2>(pv, ob, tl, psi, [&](int k, int32_t pix) {
        In in;
        in.m.load(m, ob.map_off + max(pix, 0));
        if constexpr (!BANDED) in.d = __ldg(row + tl.t0 + k);
        return in;
    }, [&](int k, int32_t pix, double c, double s, const In &in) {
        double g = 0.0;   // -2 N^-1 r; part_chi2 (white) and part_psi are sums of it, and halved below
        if (k < tl.len) {
            if constexpr (BANDED) {
                g = -2.0 * ys[spos(k)];
            } else {
                const double r = tod_f64(in.d) - in.m.project(pix, c, s);
                g = r * w;
                part_chi2 = fma(r, g, part_chi2);
            }
            if (pix < 0) g = 0.0;
        }
        const double gc = g * c, gs = g * s;
        if (pix >= 0) part_psi = fma(in.m.u, gc, fma(-in.m.q, gs, part_psi));
        if (rec) {
            const double v[3] = {g, gc, gs};
            red_add_f64_records_warp<3, double>(rec, pix, v, stage, spix);
        }
    });
    // d(weights)/d delta = 2 (-s, c), or its opposite when a half-wave plate reflects the weights
    part_psi *= ob.hwp ? 1.0 : -1.0;
    if constexpr (!BANDED) part_chi2 *= -0.5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        part_chi2 += __shfl_down_sync(0xffffffffu, part_chi2, o);
        part_psi += __shfl_down_sync(0xffffffffu, part_psi, o);
    }
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = part_chi2; red[1][threadIdx.x >> 5] = part_psi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int i = 0; i < NT / 32; ++i) { a += red[0][i]; b += red[1][i]; }
        red_add_f64(chi2 + tl.obs, a);
        if (grad_psi) red_add_f64(grad_psi + gdet, -2.0 * b);
    }
}

template <int MODE, typename DT>
static furax_status run_chi2_tc(const furax_pointing *p, const furax_noise *n, const DT *d, const double4_32a *m, double *chi2,
                                double *gm, double *gp, bool f64, cudaStream_t st)
{
    if constexpr (MODE == 0) {
        if (n->kind == FURAX_NOISE_BANDED)
            return each_kept_chunk(p, [&](const Tile *tiles, unsigned g, const PointingView &pv) {
                return launch_dyn(chi2_tc_kernel<MODE, true, DT>, g, TT, kTcSmem, st, tiles, pv, n->view(), d, m, chi2, gm, gp,
                                  p->d_err, f64);
            });
    }
    if (n->kind == FURAX_NOISE_BANDED)
        return launch_dyn(chi2_tc_kernel<MODE, true, DT>, (unsigned)p->n_tiles, TT, kTcSmem, st, p->d_tiles, p->view(),
                          n->view(), d, m, chi2, gm, gp, p->d_err, f64);
    return launch_dyn(chi2_tc_kernel<MODE, false, DT>, (unsigned)p->n_tiles, kChiThreads<false>, 0, st, p->d_tiles, p->view(),
                      n->view(), d, m, chi2, gm, gp, p->d_err, f64);
}

template <typename DT>
static furax_status dispatch_chi2_tc(const furax_pointing *p, const furax_noise *n, const DT *d, const double4_32a *m,
                                     double *chi2, double *gm, double *gp, bool f64, cudaStream_t st)
{
    switch (p->mode) {
    case FURAX_POINTING_ON_THE_FLY: return run_chi2_tc<0, DT>(p, n, d, m, chi2, gm, gp, f64, st);
    case FURAX_POINTING_CACHE_F32: return run_chi2_tc<1, DT>(p, n, d, m, chi2, gm, gp, f64, st);
    case FURAX_POINTING_CACHE_MIXED: return run_chi2_tc<3, DT>(p, n, d, m, chi2, gm, gp, f64, st);
    default: return run_chi2_tc<2, DT>(p, n, d, m, chi2, gm, gp, f64, st);
    }
}

furax_status launch_chi2_tc(const furax_pointing *p, const furax_noise *n, const void *d, int d_t, const double *m,
                            double *chi2, double *grad_map, double *grad_psi, bool f64, cudaStream_t st)
{
    furax_status rc = launch_pack_x4(p, m, nullptr, st);
    if (rc) return rc;
    return d_t == FURAX_F64 ? dispatch_chi2_tc<double>(p, n, (const double *)d, p->ws_x4, chi2, grad_map, grad_psi, f64, st)
                            : dispatch_chi2_tc<float>(p, n, (const float *)d, p->ws_x4, chi2, grad_map, grad_psi, f64, st);
}

}  // namespace fx
