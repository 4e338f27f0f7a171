// Gap filling by constrained Gaussian realisation, the use the Furax paper gives its symmetric
// band Toeplitz operator besides noise weighting (SymmetricBandToeplitzOperator, Table 2). With N
// the noise covariance (a symmetric band per detector), d the data, v the observed samples, g the
// gaps and n an unconstrained realisation of covariance N (supplied by the caller: the random
// draws of the method),
//     d_g <- n_g + N_gv N_vv^-1 (d_v - n_v),    d_v unchanged.
// N_vv^-1 is applied by conjugate gradients run for every detector at once: the operator is the
// band product (direct, or overlap-save for long bands) between two applications of the mask,
// and each detector keeps its own scalars (per-CTA partial sums reduced into them).
#include "tc_sample.cuh"
#include "dfloat.cuh"

namespace fx {

struct GfDet {
    double rr, rr0, pq, rr_new, alpha, beta;
    int32_t done, iters;
    uint32_t count, pad;   // tiles of the detector that have arrived (fused iteration)
};

__device__ __forceinline__ double cta_sum_d(double v)
{
    __shared__ double red[FT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < FT / 32; ++w) s += red[w];
    return s;
}

__device__ __forceinline__ int64_t tod_index(const ObsInfo &ob, const Tile &tl, int u)
{
    return ob.tod_off + (int64_t)tl.det * ob.nsamp + tl.t0 + u;
}

// r = S (d - n), p = r, y = 0; rr[det] += |r|^2.
template <typename DT>
__global__ void __launch_bounds__(FT) gf_init_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                     const DT *__restrict__ d, const DT *__restrict__ nr,
                                                     const uint8_t *__restrict__ valid, double *__restrict__ y,
                                                     double *__restrict__ r, double *__restrict__ p,
                                                     GfDet *__restrict__ sc)
{
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    double acc = 0.0;
    for (int u = threadIdx.x; u < tl.len; u += FT) {
        const int64_t i = tod_index(ob, tl, u);
        const double rv = valid[i] ? (double)d[i] - (double)nr[i] : 0.0;
        r[i] = rv;
        p[i] = rv;
        y[i] = 0.0;
        acc += rv * rv;
    }
    acc = cta_sum_d(acc);
    if (threadIdx.x == 0) red_add_f64(&sc[ob.det_off + tl.det].rr, acc);
}

__global__ void gf_start_kernel(int64_t ndet, GfDet *__restrict__ sc)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ndet) return;
    GfDet &s = sc[i];
    s.rr0 = s.rr;
    s.done = s.rr0 > 0.0 ? 0 : 1;
    s.iters = 0;
    s.pq = 0.0;
    s.rr_new = 0.0;
    s.beta = 0.0;
    s.count = 0u;
}

// FP32 copy of an FP64 TOD (the operand of the FP32 band product).
__global__ void __launch_bounds__(FT) gf_to_f32_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                       const double *__restrict__ x, float *__restrict__ x32)
{
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    for (int u = threadIdx.x; u < tl.len; u += FT) {
        const int64_t i = tod_index(ob, tl, u);
        x32[i] = f64_to_f32_bits(x[i]);
    }
}

// q = S (N p) (the band product nq, FP64 or FP32); pq[det] += p . q. The FP64 q is stored (in
// place over nq); the FP32 one is recomputed from nq by the update, which saves a stored vector.
template <typename QT>
__global__ void __launch_bounds__(FT) gf_pq_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                   const uint8_t *__restrict__ valid, const double *__restrict__ p,
                                                   const QT *__restrict__ nq, double *__restrict__ q,
                                                   GfDet *__restrict__ sc)
{
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    if (sc[ob.det_off + tl.det].done) return;
    double acc = 0.0;
    for (int u = threadIdx.x; u < tl.len; u += FT) {
        const int64_t i = tod_index(ob, tl, u);
        double qv = 0.0;
        if (valid[i]) {
            if constexpr (sizeof(QT) == 8) qv = nq[i];
            else qv = f32_to_f64_bits(nq[i]);   // exact, and no FP64 conversion issued
        }
        if constexpr (sizeof(QT) == 8) q[i] = qv;
        acc += p[i] * qv;
    }
    acc = cta_sum_d(acc);
    if (threadIdx.x == 0) red_add_f64(&sc[ob.det_off + tl.det].pq, acc);
}

__global__ void gf_alpha_kernel(int64_t ndet, GfDet *__restrict__ sc)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ndet) return;
    GfDet &s = sc[i];
    s.alpha = (!s.done && s.pq > 0.0) ? s.rr / s.pq : 0.0;
    s.rr_new = 0.0;
}

// y += alpha p; r -= alpha q; rr_new[det] += |r|^2. q is the stored FP64 S N p, or S applied to the
// FP32 band product.
template <typename QT>
__global__ void __launch_bounds__(FT) gf_update_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                       const uint8_t *__restrict__ valid, const double *__restrict__ p,
                                                       const QT *__restrict__ q, double *__restrict__ y,
                                                       double *__restrict__ r, GfDet *__restrict__ sc)
{
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    const GfDet s = sc[ob.det_off + tl.det];
    if (s.done) return;
    double acc = 0.0;
    for (int u = threadIdx.x; u < tl.len; u += FT) {
        const int64_t i = tod_index(ob, tl, u);
        y[i] += s.alpha * p[i];
        double qv;
        if constexpr (sizeof(QT) == 8) qv = q[i];
        else qv = valid[i] ? f32_to_f64_bits(q[i]) : 0.0;
        const double rv = r[i] - s.alpha * qv;
        r[i] = rv;
        acc += rv * rv;
    }
    acc = cta_sum_d(acc);
    if (threadIdx.x == 0) red_add_f64(&sc[ob.det_off + tl.det].rr_new, acc);
}

__global__ void gf_beta_kernel(int64_t ndet, double tol2, GfDet *__restrict__ sc)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ndet) return;
    GfDet &s = sc[i];
    s.pq = 0.0;
    if (s.done) { s.beta = 0.0; return; }
    s.beta = s.rr > 0.0 ? s.rr_new / s.rr : 0.0;
    s.rr = s.rr_new;
    s.iters += 1;
    if (s.rr <= tol2 * s.rr0) s.done = 1;
}

// p = r + beta p (detectors still iterating), and its FP32 copy for the next FP32 band product.
__global__ void __launch_bounds__(FT) gf_dir_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                    const double *__restrict__ r, double *__restrict__ p,
                                                    float *__restrict__ x32, const GfDet *__restrict__ sc)
{
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    const GfDet s = sc[ob.det_off + tl.det];
    if (s.done) return;
    for (int u = threadIdx.x; u < tl.len; u += FT) {
        const int64_t i = tod_index(ob, tl, u);
        const double pv = r[i] + s.beta * p[i];
        p[i] = pv;
        if (x32) x32[i] = f64_to_f32_bits(pv);
    }
}

// ------------------------------------------------------------------------------------
// The FP64-accurate iteration for short bands in two passes: the direction is formed where the band product
// loads it, the product is masked and dotted where it leaves, and the detector's last tile forms the scalar that
// the next pass reads. (With a pass per step: 113 B per sample and iteration and five launches; here 82 B and two. 32 x
// 131,071 samples: 115 us an iteration before, 90 us now: 62 us the product, bound by its phases' latency (fused_tc.cu),
// 28 us the step, 7.3 TB/s of its 48 B per sample. Of the product's outputs only those of observed samples must keep
// their accuracy: the check of the blocks asks the mask.)
// ------------------------------------------------------------------------------------

// Sum over the CTA's TT threads added to *sum; true in every thread of the detector's last tile.
template <int NT>
__device__ __forceinline__ bool gf_arrive(double v, double *sum, uint32_t *count, int64_t nsamp)
{
    __shared__ double red[NT / 32];
    __shared__ bool last;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < NT / 32; ++w) s += red[w];
        red_add_f64(sum, s);
        __threadfence();
        const uint32_t n = (uint32_t)((nsamp + TILE - 1) / TILE);
        last = atomicAdd(count, 1u) == n - 1u;
        if (last) *count = 0u;
        __threadfence();
    }
    __syncthreads();
    return last;
}

// p = r + beta p_old; q = S N p; pq[det] += p . q; alpha. p and p_old are different arrays: a tile's halo
// belongs to its neighbours.
__global__ void __launch_bounds__(TT, 2) gf_apply_tc_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                            NoiseView nv, const uint8_t *__restrict__ valid,
                                                            const double *__restrict__ r, const double *__restrict__ p_old,
                                                            double *__restrict__ p, double *__restrict__ q, GfDet *sc,
                                                            unsigned *__restrict__ err, bool f64)
{
    extern __shared__ __align__(128) unsigned char sm[];
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    const int64_t gdet = ob.det_off + tl.det;
    GfDet &s = sc[gdet];
    if (s.done) return;
    const double beta = s.beta;
    tc_begin(sm, nv, gdet, err);
    double v[kTcPer];
    const TcSlots sl(tl, ob);
#pragma unroll
    for (int k = 0; k < kTcPer; ++k) v[k] = __ldg(r + sl.index(k));
    if (beta != 0.0) {   // the first direction is the residual itself
        double po[kTcPer];
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) po[k] = __ldg(p_old + sl.index(k));
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) v[k] = fma(beta, po[k], v[k]);
    }
#pragma unroll
    for (int k = 0; k < kTcPer; ++k)
        if (!sl.in(k)) v[k] = 0.0;
    const int64_t row = sl.row + kHalo;
    const bool ok = tc_band(sm, v, nv, gdet, err, f64, tl.len, TcKeep{v}, [&](int t) {   // outputs in gaps are not used
        bool any = false;
        for (int k = t; k < min(t + 8, tl.len); ++k) any = any || valid[row + k];
        return any;
    });
    if (!ok) return;   // the host sees the error word
    const double *ys = tc_ys(sm);
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < kTcPer; ++k) {
        const int t = sl.slot(k) - kHalo;
        if (t >= 0 && t < tl.len) {
            const int64_t i = sl.row + sl.slot(k);
            const double qv = valid[i] ? ys[spos(t)] : 0.0;
            p[i] = v[k];
            q[i] = qv;
            acc = fma(v[k], qv, acc);
        }
    }
    if (gf_arrive<TT>(acc, &s.pq, &s.count, ob.nsamp) && threadIdx.x == 0) {
        const double pq = __ldcg(&s.pq);
        s.alpha = pq > 0.0 ? s.rr / pq : 0.0;
        s.rr_new = 0.0;
    }
}

// y += alpha p; r -= alpha q; rr_new[det] += |r|^2; beta and convergence. Four samples per thread in flight.
__global__ void __launch_bounds__(FT) gf_step_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                     const double *__restrict__ p, const double *__restrict__ q,
                                                     double *__restrict__ y, double *__restrict__ r, GfDet *sc, double tol2)
{
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    GfDet &s = sc[ob.det_off + tl.det];
    if (s.done) return;
    const double alpha = s.alpha;
    double acc = 0.0;
    for (int u0 = threadIdx.x; u0 < tl.len; u0 += 4 * FT) {
        double pv[4], qv[4], yv[4], rv[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int64_t i = tod_index(ob, tl, min(u0 + b * FT, tl.len - 1));
            pv[b] = p[i];
            qv[b] = q[i];
            yv[b] = y[i];
            rv[b] = r[i];
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (u0 + b * FT >= tl.len) break;
            const int64_t i = tod_index(ob, tl, u0 + b * FT);
            y[i] = fma(alpha, pv[b], yv[b]);
            const double rn = fma(-alpha, qv[b], rv[b]);
            r[i] = rn;
            acc = fma(rn, rn, acc);
        }
    }
    if (gf_arrive<FT>(acc, &s.rr_new, &s.count, ob.nsamp) && threadIdx.x == 0) {
        const double rr = __ldcg(&s.rr_new);
        s.pq = 0.0;
        s.beta = s.rr > 0.0 ? rr / s.rr : 0.0;
        s.rr = rr;
        s.iters += 1;
        if (rr <= tol2 * s.rr0) s.done = 1;
    }
}

// out = d on observed samples, n + (N y) in the gaps. out may be d (documented in-place use), so
// neither carries __restrict__.
template <typename DT, typename QT>
__global__ void __launch_bounds__(FT) gf_fill_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                     const DT *d, const DT *__restrict__ nr,
                                                     const uint8_t *__restrict__ valid, const QT *__restrict__ ny,
                                                     DT *out)
{
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    for (int u = threadIdx.x; u < tl.len; u += FT) {
        const int64_t i = tod_index(ob, tl, u);
        out[i] = valid[i] ? d[i] : (DT)((double)nr[i] + (double)ny[i]);
    }
}

furax_status gapfill(const furax_noise *n, const void *d, const uint8_t *valid, const void *nr, void *out, int dtype,
                     int maxiter, double tol, int precision, int32_t *iters_out, cudaStream_t st)
{
    const bool f32 = precision == FURAX_F32;   // band product in FP32, vectors and scalars in FP64
    // N y, of which the gaps' outputs are used, however far they lie from observed samples: every block is checked (7 of
    // a tile's 512 formed again with 4 % of the samples in gaps of 120)
    auto ninv64 = [&](const double *in, double *o) {
        return long_band(n) ? launch_ninv(n, in, o, FURAX_F64, st) : launch_ninv_tc(n, in, o, precision == FURAX_F64, n->gf_err(), st);
    };
    const int64_t ns = n->nsamp_total, nd = n->ndet_total;
    if (ns == 0 || nd == 0) return FURAX_OK;
    const unsigned g = (unsigned)n->n_tiles;
    const unsigned dg = (unsigned)((nd + 127) / 128);
    furax_noise *nm = const_cast<furax_noise *>(n);   // workspaces live in the handle
    furax_status rc = FURAX_OK;
    auto ensure = [&](void **ptr, size_t bytes) {
        if (!rc && !*ptr && (rc = check_cuda(cudaMalloc(ptr, bytes), "gap-filling workspace"))) *ptr = nullptr;
    };
    ensure((void **)&nm->gf_y, sizeof(double) * ns);
    ensure((void **)&nm->gf_r, sizeof(double) * ns);
    ensure((void **)&nm->gf_p, sizeof(double) * ns);
    const bool fused = !f32 && !long_band(n);
    if (fused) ensure((void **)&nm->gf_p2, sizeof(double) * ns);
    if (!f32) ensure((void **)&nm->gf_q, sizeof(double) * ns);   // FP32 band product: q is not stored
    ensure(&nm->gf_sc, sizeof(GfDet) * nd);
    if (f32) {
        ensure((void **)&nm->gf_x32, sizeof(float) * ns);
        ensure((void **)&nm->gf_n32, sizeof(float) * ns);
    }
    double *y = nm->gf_y, *r = nm->gf_r, *p = nm->gf_p, *q = nm->gf_q;
    GfDet *sc = (GfDet *)nm->gf_sc;
    float *x32 = nm->gf_x32, *n32 = nm->gf_n32;
    std::vector<GfDet> h(nd);
    bool all_done = false;
    unsigned gave_up = 0;
    if (!rc) rc = check_cuda(cudaMemsetAsync(sc, 0, sizeof(GfDet) * nd, st), "memset");
    if (!rc) rc = check_cuda(cudaMemsetAsync(n->gf_err(), 0, sizeof gave_up, st), "clear");
    if (!rc) {
        if (dtype == FURAX_F64)
            gf_init_kernel<double><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, (const double *)d, (const double *)nr, valid,
                                                      y, r, p, sc);
        else
            gf_init_kernel<float><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, (const float *)d, (const float *)nr, valid,
                                                     y, r, p, sc);
        gf_start_kernel<<<dg, 128, 0, st>>>(nd, sc);
        count_launches(2);
        if (f32) {   // the first direction's FP32 copy; later ones come from gf_dir
            gf_to_f32_kernel<<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, p, x32);
            count_launches(1);
        }
        rc = check_launch("gap filling (start)");
    }
    for (int it = 0; !rc && it < maxiter && !all_done && !gave_up; ++it) {
        if (f32) {   // N p in FP32
            if ((rc = launch_ninv(n, x32, n32, FURAX_F32, st))) break;
            gf_pq_kernel<float><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, valid, p, n32, nullptr, sc);
            gf_alpha_kernel<<<dg, 128, 0, st>>>(nd, sc);
            gf_update_kernel<float><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, valid, p, n32, y, r, sc);
        } else if (fused) {
            if ((rc = launch_dyn(gf_apply_tc_kernel, g, TT, kTcSmem, st, n->d_tiles, n->d_obs, n->view(), valid, r,
                                 it % 2 ? p : nm->gf_p2, it % 2 ? nm->gf_p2 : p, q, sc, n->gf_err(), precision == FURAX_F64)))
                break;
            gf_step_kernel<<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, it % 2 ? nm->gf_p2 : p, q, y, r, sc, tol * tol);
            count_launches(2);
        } else {
            if ((rc = ninv64(p, q))) break;
            gf_pq_kernel<double><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, valid, p, q, q, sc);
            gf_alpha_kernel<<<dg, 128, 0, st>>>(nd, sc);
            gf_update_kernel<double><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, valid, p, q, y, r, sc);
        }
        if (!fused) {
            gf_beta_kernel<<<dg, 128, 0, st>>>(nd, tol * tol, sc);
            gf_dir_kernel<<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, r, p, f32 ? x32 : nullptr, sc);
            count_launches(5);
        }
        if ((rc = check_launch("gap filling (iteration)"))) break;
        if ((it + 1) % 16 == 0 || it + 1 == maxiter) {
            if ((rc = check_cuda(cudaMemcpyAsync(h.data(), sc, sizeof(GfDet) * nd, cudaMemcpyDeviceToHost, st), "read")))
                break;
            if ((rc = check_cuda(cudaMemcpyAsync(&gave_up, n->gf_err(), sizeof gave_up, cudaMemcpyDeviceToHost, st), "read")))
                break;
            if ((rc = check_cuda(cudaStreamSynchronize(st), "gap filling"))) break;
            all_done = true;
            for (const GfDet &s : h) all_done = all_done && s.done;
        }
    }
    if (!rc && f32) {   // N y
        gf_to_f32_kernel<<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, y, x32);
        count_launches(1);
        rc = launch_ninv(n, x32, n32, FURAX_F32, st);
    } else if (!rc) {
        rc = ninv64(y, q);
    }
    if (!rc) {
        if (dtype == FURAX_F64 && f32)
            gf_fill_kernel<double, float><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, (const double *)d, (const double *)nr,
                                                             valid, n32, (double *)out);
        else if (dtype == FURAX_F64)
            gf_fill_kernel<double, double><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, (const double *)d, (const double *)nr,
                                                              valid, q, (double *)out);
        else if (f32)
            gf_fill_kernel<float, float><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, (const float *)d, (const float *)nr,
                                                            valid, n32, (float *)out);
        else
            gf_fill_kernel<float, double><<<g, FT, 0, st>>>(n->d_tiles, n->d_obs, (const float *)d, (const float *)nr,
                                                             valid, q, (float *)out);
        count_launches(1);
        rc = check_launch("gap filling (fill)");
    }
    if (!rc) rc = check_cuda(cudaMemcpyAsync(h.data(), sc, sizeof(GfDet) * nd, cudaMemcpyDeviceToHost, st), "read");
    if (!rc) rc = check_cuda(cudaMemcpyAsync(&gave_up, n->gf_err(), sizeof gave_up, cudaMemcpyDeviceToHost, st), "read");
    if (!rc) rc = check_cuda(cudaStreamSynchronize(st), "gap filling");
    if (rc) return rc;
    if (gave_up) return set_error(FURAX_ETIMEOUT, "a bounded device-side wait gave up during gap filling");
    all_done = true;
    for (int64_t i = 0; i < nd; ++i) {
        all_done = all_done && h[i].done;
        if (iters_out) iters_out[i] = h[i].iters;
    }
    return all_done ? FURAX_OK : FURAX_ENOTCONVERGED;
}

}  // namespace fx
