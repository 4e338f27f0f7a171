// Fast pointing expansion for the FP32 cache (PointingOperator, "Map-making classes": the
// pointing is expanded from the quaternions; HEALPix RING pixels, "Landscape types").
//
// GB300 runs FP64 ~70x slower than FP32, and the exact FP64 recipe of pointing_math.cuh costs
// ~150 FP64 operations per sample. Here each sample is computed on the FP32 pipes and the
// exact recipe runs only where the FP32 result could differ from it:
//   * R(q_bore(t)) is formed once per boresight sample in FP64 and stored as double-FP32
//     (hi + lo, 18 floats of an 80-byte row); the detector axes R(q_det) z^, R(q_det) x^ once per tile.
//     d = R(q_bore) d_det and o = R(q_bore) o_det are then evaluated with exact FP32 products
//     and two-sums, so the FP32 line of sight and orientation are within ~1 ulp of the exact
//     values (R(a (x) b) = R(a) R(b) for unit quaternions).
//   * The RING lookup is done in FP32 (atan2f: at most 3 ulp). Every floor() argument is
//     accepted only if it lies farther from an integer than a bound on its FP32 error
//     (derived below); the zone test, facet edges and the neighbourhood of the poles likewise.
//     An accepted floor equals the floor of the exact value, hence the FP64 recipe's floor.
//   * Samples that fail any test are queued in shared memory and recomputed with the exact
//     FP64 recipe by the whole CTA (dense, no divergence). Non-unit or non-finite quaternions
//     always take the exact path, which gives them pixel -1 where the recipe does.
// Pixels are therefore identical to the FP64 recipe's; weights are FP32 (relative error a few
// 1e-7 away from the poles).
//
// Error budget (u = 2^-24): |d - d_exact|, |o - o_exact| <= 6u per component (rounding of the
// double-FP32 result plus |q|^2 within 4u of 1). phi: <= 8.5u/rho + 24u (atan2f) + 8u (2 pi
// wrap); tt = 2 phi/pi: <= 5.4u/rho + 24.4u. Belt arguments N(1/2 + tt -/+ 3z/4): <= 44 N u;
// cap arguments tp s, (1 - tp) s with s = N sqrt(3 (1-|z|)): <= 51 N u; cap in-ring argument
// tt * ir: <= 47 N u + 5.4u/rho. The margins used are about twice these.
#include "internal.cuh"
#include "pointing_math.cuh"
#include "pointing_fast.cuh"
#include "tile.cuh"

namespace fx {

// Boresight rows: M_t = R(q_bore(t)) in the layout of kBoreRow; [0] = NaN marks a boresight quaternion
// that must take the exact path (not finite, or |q|^2 not within 4u of 1).
__global__ void bore_matrix_kernel(const double *__restrict__ q_bore, int64_t n, float *__restrict__ m)
{
    let_next_start();
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const Quat q = load_quat(q_bore, t);
        const double off = fabs(q.w * q.w + q.x * q.x + q.y * q.y + q.z * q.z - 1.0);
        float4 *o = reinterpret_cast<float4 *>(m + kBoreRow * t);
        if (!(off <= kUnitTol)) {
            o[0] = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
            continue;
        }
        const double xx = q.x * q.x, yy = q.y * q.y, zz = q.z * q.z;
        const double xy = q.x * q.y, xz = q.x * q.z, yz = q.y * q.z;
        const double wx = q.w * q.x, wy = q.w * q.y, wz = q.w * q.z;
        // columns of rows 0 and 1 in pairs, then row 2
        const double r[9] = {1.0 - 2.0 * (yy + zz), 2.0 * (xy + wz), 2.0 * (xy - wz), 1.0 - 2.0 * (xx + zz),
                             2.0 * (xz + wy), 2.0 * (yz - wx), 2.0 * (xz - wy), 2.0 * (yz + wx), 1.0 - 2.0 * (xx + yy)};
        float h[9], l[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            h[k] = f64_to_f32_bits(r[k]);   // conversions off the FP64 pipe, which bounds this kernel
            l[k] = f64_to_f32_bits(r[k] - f32_to_f64_bits(h[k]));
        }
        o[0] = make_float4(h[0], h[1], h[2], h[3]);
        o[1] = make_float4(h[4], h[5], l[0], l[1]);
        o[2] = make_float4(l[2], l[3], l[4], l[5]);
        o[3] = make_float4(h[6], h[7], h[8], l[6]);
        o[4] = make_float4(l[7], l[8], 0.f, 0.f);
    }
}

// Bound by FP32 issue (the certified evaluation) and the FP64 pipe (the exact recipe for 1.56 % of the samples
// at nside 512, half of the pipe's time). A refresh of 28.8 M samples: 637 us with scalar two-sums, 4-byte loads of the
// boresight matrices and integer remainders; 537 us packed, with 16-byte loads and without remainders. Smaller
// blocks (128 threads: 545 us; 64: 681 us) load the detector axes more often. Tighter margins would send fewer samples
// to the exact recipe, but those would change their weights' rounding.
// HALO: 0 for the cache (flat time-ordered index), else the halo on both sides of each tile, which is written to
// its own block of kLocalTile samples (slot u = sample t0 - HALO + u).
template <int HALO>
__global__ void __launch_bounds__(256, 4) expand_fast_kernel(const Tile *__restrict__ tiles, const ObsInfo *__restrict__ obs,
                                                          const double *__restrict__ q_bore, const double *__restrict__ q_det,
                                                          const float *__restrict__ bm, const double2 *__restrict__ hwp_cs,
                                                          int32_t *__restrict__ pix_out,
                                                          float *__restrict__ c_out, float *__restrict__ s_out,
                                                          unsigned long long *__restrict__ n_invalid)
{
    __shared__ int qn, sdet_ok;
    __shared__ float sdet[12];   // detector axes: d hi, d lo, o hi, o lo
    __shared__ int32_t queue[TILE + 2 * HALO];
    const Tile tl = tiles[blockIdx.x];
    const ObsInfo ob = obs[tl.obs];
    const int64_t gdet = ob.det_off + tl.det;
    const Quat qd = load_quat(q_det, gdet);
    // detector axes in double-FP32, formed once per tile (FP64 work: one thread, not every thread)
    if (threadIdx.x == 0) {
        sdet_ok = det_axes_df(qd, sdet);
        qn = 0;
    }
    __syncthreads();
    if constexpr (HALO > 0) {
        let_next_start();
        prior_done();   // the boresight rows are written; the operator is done with the previous chunk
    }
    const DetAxes ax(sdet);
    const bool det_ok = sdet_ok != 0;
    const int64_t row = HALO ? (int64_t)blockIdx.x * kLocalTile - (tl.t0 - HALO) : ob.tod_off + tl.det * ob.nsamp;
    for (int k = threadIdx.x; k < tl.len + 2 * HALO; k += blockDim.x) {
        const int64_t t = tl.t0 - HALO + k;
        if (HALO && (t < 0 || t >= ob.nsamp)) continue;
        int32_t p = -1;
        float c = 1.f, s = 0.f;
        bool ok = det_ok && certified_sample(bm + kBoreRow * (ob.bore_off + t), ax, (int32_t)ob.nside, p, c, s);
        if (ok && hwp_cs) apply_hwp<float>(c, s, hwp_cs[ob.bore_off + t]);
        if (ok) {
            pix_out[row + t] = p;
            c_out[row + t] = c;
            s_out[row + t] = s;
        } else {
            queue[atomicAdd(&qn, 1)] = k;
        }
    }
    __syncthreads();
    // exact FP64 recipe for the queued samples, densely
    const int nq = qn;
    int bad = 0;
    for (int j = threadIdx.x; j < nq; j += blockDim.x) {
        const int64_t t = tl.t0 - HALO + queue[j];
        const SampleF64 r = point_f64(load_quat(q_bore, ob.bore_off + t), qd, ob.nside);
        double c = r.c, s = r.s;
        if (hwp_cs && r.pix >= 0) apply_hwp<double>(c, s, hwp_cs[ob.bore_off + t]);
        pix_out[row + t] = r.pix;
        c_out[row + t] = (float)c;
        s_out[row + t] = (float)s;
        bad += r.pix < 0;
    }
    if (n_invalid) {
        bad = __reduce_add_sync(0xffffffffu, bad);
        if ((threadIdx.x & 31) == 0 && bad) atomicAdd(n_invalid, (unsigned long long)bad);
    }
}

// The boresight rows from the handle's current quaternions.
furax_status launch_bore_rows(const furax_pointing *p, cudaStream_t st)
{
    furax_pointing *pm = const_cast<furax_pointing *>(p);
    furax_status rc = ensure_ws(pm, (void **)&pm->ws_bore_m, sizeof(float) * kBoreRow * std::max<int64_t>(1, p->nbore_total));
    if (rc) return rc;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((p->nbore_total + 255) / 256, 16LL * p->n_sm));
    bore_matrix_kernel<<<g, 256, 0, st>>>(p->q_bore, p->nbore_total, pm->ws_bore_m);
    count_launches(1);
    return check_launch("boresight matrices");
}

furax_status launch_expand_local(const furax_pointing *p, int64_t tile0, int64_t n, int32_t *pix, float *c, float *s,
                                 cudaStream_t st)
{
    furax_status rc = launch_behind(expand_fast_kernel<kHalo>, (unsigned)n, 256, 0, st, p->d_tiles + tile0, p->d_obs, p->q_bore,
                                    p->q_det, p->ws_bore_m, p->has_hwp ? p->d_hwp_cs : nullptr, pix, c, s, nullptr);
    if (rc) return rc;
    count_launches(1);
    return check_launch("pointing of a chunk of tiles");
}

furax_status launch_expand_fast(const furax_pointing *p, unsigned long long *n_invalid, cudaStream_t st)
{
    furax_status rc = launch_bore_rows(p, st);
    if (rc) return rc;
    if (p->n_tiles == 0) return FURAX_OK;
    expand_fast_kernel<0><<<(unsigned)p->n_tiles, 256, 0, st>>>(p->d_tiles, p->d_obs, p->q_bore, p->q_det, p->ws_bore_m,
                                                                p->has_hwp ? p->d_hwp_cs : nullptr, p->pix, p->c32,
                                                                p->s32, n_invalid);
    count_launches(1);
    return check_launch("fast pointing expansion");
}

}  // namespace fx
