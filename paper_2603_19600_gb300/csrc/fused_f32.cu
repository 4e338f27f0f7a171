// Fused tile kernels of the map-making operator (Furax paper: the estimator
// A = (H.T @ N.I @ H).I @ H.T @ N.I in the Software Design listing, with the block
// decomposition P^T N^-1 P = sum_i P_i^T N_i^-1 P_i of "Algebraic reductions").
//
// One CTA owns one tile: one detector, TILE consecutive samples. It
//   1. gathers the projected map P x for the tile plus a 63-sample halo on each side into
//      shared memory (samples outside the detector stream are zeros: finite section),
//   2. applies N^-1 (white scale, or the 127-term symmetric band, register-blocked),
//   3. scatters y (1, cos 2psi, sin 2psi) into per-pixel accumulators with L2 reductions.
// The time-ordered data never leaves the SM. The same skeleton gives the standalone N^-1,
// the right-hand side P^T N^-1 d and chi^2 with its gradients.
#include "tile.cuh"

namespace fx {

// ------------------------------------------------------------------------------------
// FP32 fused apply: acc += P^T N^-1 P x32  (x32: padded FP32 map, zero on masked pixels)
// ------------------------------------------------------------------------------------
// On the FP64 cache (FP32 weights are read by the pipelined kernels).
template <int ACC, bool BANDED>
__global__ void __launch_bounds__(FT, 3) fused_f32_kernel(const Tile *__restrict__ tiles, PointingView pv, NoiseView nv,
                                                          const float4 *__restrict__ x32, float4 *__restrict__ acc_hi,
                                                          float4 *__restrict__ acc_lo, double *__restrict__ acc64)
{
    extern __shared__ float fsm[];
    float *xs = fsm;                           // [XS] projected map P x over the tile and its halos
    float *taps = xs + XS;                     // [MAXTAPS]
    float *sc = taps + MAXTAPS;                // [XS] cos 2psi of the same samples
    float *ss = sc + XS;                       // [XS] sin 2psi
    int32_t *spix = reinterpret_cast<int32_t *>(ss + XS);   // [XS] pixel (-1: none)

    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = pv.obs[tl.obs];
    const int64_t gdet = ob.det_off + tl.det;
    constexpr int halo = BANDED ? kHalo : 0;
    if constexpr (BANDED) load_taps<float>(nv, gdet, taps);
    const int nload = tl.len + 2 * halo;
    const int64_t t_first = tl.t0 - halo;

    for (int u = threadIdx.x; u < nload; u += FT) {
        const int64_t t = t_first + u;
        float v = 0.f, c = 0.f, s = 0.f;
        int32_t pix = -1;
        if (t >= 0 && t < ob.nsamp) {
            pix = get_sample<FURAX_POINTING_CACHE_F64, float>(pv, ob, tl.det, t, c, s);
            if (pix >= 0) {
                const float4 m = __ldg(x32 + ob.map_off + pix);
                v = fmaf(m.z, s, fmaf(m.y, c, m.x));
            }
        }
        xs[spos(u)] = v;
        spix[spos(u)] = pix;
        sc[spos(u)] = c;
        ss[spos(u)] = s;
    }
    __syncthreads();

    // N^-1 on the tile, then the scatter of y (1, c, s).
    const int base = threadIdx.x * FR;
    if (base >= tl.len) return;
    float y[FR];
    if constexpr (BANDED) {
        band_product<float, FR>(xs, taps, base, y);
    } else {
        const float w = white_scale<float>(nv, gdet);
#pragma unroll
        for (int r = 0; r < FR; ++r) y[r] = xs[spos(base + r)] * w;
    }
#pragma unroll
    for (int r = 0; r < FR; ++r) {
        const int k = base + r;
        if (k >= tl.len) break;
        const int u = k + halo;
        const int32_t pix = spix[spos(u)];
        if (pix < 0) continue;
        const float c = sc[spos(u)], s = ss[spos(u)];
        const int64_t gp = ob.map_off + pix;
        const float4 v = make_float4(y[r], y[r] * c, y[r] * s, 0.f);
        if constexpr (ACC == FURAX_ACC_F32) red_add_v4(acc_hi + gp, v);
        else if constexpr (ACC == FURAX_ACC_F32_KAHAN)
            kahan_add_v4(acc_hi + kKahanStride * gp, acc_lo + kKahanStride * gp, v);
        else {
            red_add_f64(acc64 + 3 * gp + 0, (double)v.x);
            red_add_f64(acc64 + 3 * gp + 1, (double)v.y);
            red_add_f64(acc64 + 3 * gp + 2, (double)v.z);
        }
    }
}

template <bool BANDED>
static furax_status dispatch_fused_f32_acc(const furax_pointing *p, const furax_noise *n, const float4 *x32, int acc,
                                           float4 *hi, float4 *lo, double *a64, cudaStream_t st)
{
    const unsigned g = (unsigned)p->n_tiles;
    const PointingView pv = p->view();
    const NoiseView nv = n->view();
    if (acc == FURAX_ACC_F32)
        return launch_dyn(fused_f32_kernel<FURAX_ACC_F32, BANDED>, g, FT, kF32Smem, st, p->d_tiles, pv, nv, x32,
                          hi, lo, a64);
    if (acc == FURAX_ACC_F32_KAHAN)
        return launch_dyn(fused_f32_kernel<FURAX_ACC_F32_KAHAN, BANDED>, g, FT, kF32Smem, st, p->d_tiles, pv, nv,
                          x32, hi, lo, a64);
    return launch_dyn(fused_f32_kernel<FURAX_ACC_F64, BANDED>, g, FT, kF32Smem, st, p->d_tiles, pv, nv, x32, hi,
                      lo, a64);
}

static furax_status dispatch_fused_f32(const furax_pointing *p, const furax_noise *n, const float4 *x32, int acc,
                                       float4 *hi, float4 *lo, double *a64, cudaStream_t st)
{
    if (n->kind == FURAX_NOISE_BANDED) return dispatch_fused_f32_acc<true>(p, n, x32, acc, hi, lo, a64, st);
    return dispatch_fused_f32_acc<false>(p, n, x32, acc, hi, lo, a64, st);
}

// On the fly: the certified pointing (pointing_fast.cu) of a chunk of tiles goes to a workspace, and the
// pipelined operator of the cached pointing reads it from there, chunk by chunk. One kernel that did both per tile
// had to be 72 KB of shared memory and 80 registers wide and ran its phases (pointing, exact recipe, gather, band,
// scatter) one after the other. 64 x 262,144 samples, nside 512: 768 us that way, 648 us this way (626 us since the sums go straight into the output, 617 us with dependent launches) with 32 tiles per SM
// and chunk; with 16 some 60 us more, with 8, which stay in L2, 130 us more: the last round of every launch costs more than the 24
// bytes per sample through memory. The workspace (250 MB) is all that on-the-fly pointing ever holds. The three kernels
// of a chunk are dependent launches, each placed while the one before ends: 3 x 9001 samples with FP32 sums take 60 us in one kernel,
// 64 us in ordinary launches and 58 us so (300 x 1000: 45, 50, 43 us).
static int64_t chunk_tiles(const furax_pointing *p) { return std::min<int64_t>(p->n_tiles, 32LL * p->n_sm); }

// The same workspace holds the FP64 pointing of half as many tiles (fused_tc.cu, chi2_tc.cu).
int64_t kept_tiles(const furax_pointing *p) { return std::min<int64_t>(p->n_tiles, 16LL * p->n_sm); }

furax_status ensure_local_ws(const furax_pointing *p)
{
    furax_pointing *pm = const_cast<furax_pointing *>(p);
    const size_t pix = sizeof(float) * kLocalTile * (size_t)chunk_tiles(p);
    const size_t w = std::max(pix, sizeof(double) * TILE * (size_t)kept_tiles(p));
    furax_status rc = ensure_ws(pm, (void **)&pm->ws_local_pix, pix);
    if (!rc) rc = ensure_ws(pm, (void **)&pm->ws_local_c, w);
    if (!rc) rc = ensure_ws(pm, (void **)&pm->ws_local_s, w);
    return rc;
}

int64_t on_the_fly_launches(const furax_pointing *p)
{
    const int64_t c = chunk_tiles(p);
    return c ? 1 + 2 * ((p->n_tiles + c - 1) / c) : 0;
}

static furax_status apply_on_the_fly(const furax_pointing *p, const furax_noise *n, const float4 *x32, int acc, float4 *hi,
                                     float4 *lo, double *a64, cudaStream_t st, const unsigned *done)
{
    furax_pointing *pm = const_cast<furax_pointing *>(p);
    const int64_t c = chunk_tiles(p);
    furax_status rc;
    if ((rc = ensure_local_ws(p)) || (rc = launch_bore_rows(p, st))) return rc;
    TmaChunk chunk{0, 0, p->view()};
    chunk.pv.pix = p->ws_local_pix;
    chunk.pv.c32 = p->ws_local_c;
    chunk.pv.s32 = p->ws_local_s;
    for (; chunk.tile0 < p->n_tiles; chunk.tile0 += c) {
        chunk.n = std::min(c, p->n_tiles - chunk.tile0);
        if ((rc = launch_expand_local(p, chunk.tile0, chunk.n, pm->ws_local_pix, pm->ws_local_c, pm->ws_local_s, st))) return rc;
        if ((rc = launch_fused_tma(p, n, x32, acc, hi, lo, a64, st, nullptr, done, &chunk))) return rc;
        count_launches(1);
    }
    count_launches(-1);   // the caller counts one
    return FURAX_OK;
}

bool fused_f32_projects_templates(const furax_pointing *p)
{
    return p->mode == FURAX_POINTING_CACHE_F32 || p->mode == FURAX_POINTING_CACHE_MIXED;
}

furax_status launch_fused_f32(const furax_pointing *p, const furax_noise *n, const float4 *x32, int acc, float4 *hi,
                              float4 *lo, double *a64, cudaStream_t st, const FusedTpl *ft, const unsigned *done)
{
    if (p->n_tiles == 0) return FURAX_OK;
    furax_status rc;
    if (ft && !fused_f32_projects_templates(p))
        return set_error(FURAX_EINVAL, "template work is fused only for the cached FP32 pointing");
    if (p->mode == FURAX_POINTING_ON_THE_FLY) rc = apply_on_the_fly(p, n, x32, acc, hi, lo, a64, st, done);
    else if ((p->mode == FURAX_POINTING_CACHE_F32 || p->mode == FURAX_POINTING_CACHE_MIXED) && !ft &&
             sorted_active(p) && !long_band(n))
        rc = launch_fused_sorted(p, n, x32, acc, hi, lo, a64, st);   // pixel-sorted schedule
    else if (p->mode == FURAX_POINTING_CACHE_F32 || p->mode == FURAX_POINTING_CACHE_MIXED)  // FP32 weights: hi
        rc = launch_fused_tma(p, n, x32, acc, hi, lo, a64, st, ft, done);
    else rc = dispatch_fused_f32(p, n, x32, acc, hi, lo, a64, st);
    if (rc) return rc;
    count_launches(1);
    return check_launch("fused P^T N^-1 P (FP32)");
}

template <bool B>
static furax_status prep_f32_band()
{
    furax_status rc = FURAX_OK;
    if (!rc) rc = allow_smem((const void *)fused_f32_kernel<FURAX_ACC_F32, B>, kF32Smem);
    if (!rc) rc = allow_smem((const void *)fused_f32_kernel<FURAX_ACC_F32_KAHAN, B>, kF32Smem);
    if (!rc) rc = allow_smem((const void *)fused_f32_kernel<FURAX_ACC_F64, B>, kF32Smem);
    return rc;
}

furax_status prepare_fused_f32()
{
    furax_status rc = prepare_fused_tma();
    if (!rc) rc = prepare_fused_sorted();
    if (!rc) rc = prep_f32_band<true>();
    if (!rc) rc = prep_f32_band<false>();
    return rc;
}

}  // namespace fx
