// Certified FP32 evaluation of the pointing (PointingOperator, "Map-making classes"; HEALPix RING
// pixels, "Landscape types"), shared by the cache fill (pointing_fast.cu) and the on-the-fly FP32
// operator (fused_f32.cu). The design, the error budget and the margins are described at the top
// of pointing_fast.cu: a sample whose FP32 decisions the margins cannot certify returns false and
// is recomputed by the caller with the exact FP64 recipe, so pixels equal the recipe's.
#pragma once
#include "pointing_math.cuh"
#include "stencil.cuh"

namespace fx {

constexpr float kU = 5.9604645e-8f;   // 2^-24

// Boresight rotation matrices in double-FP32, kBoreRow floats per boresight sample: hi words of rows 0 and 1
// as pairs (m00, m10), (m01, m11), (m02, m12), their lo words, row 2 hi, row 2 lo. [0] NaN marks a quaternion for the exact path.
constexpr int kBoreRow = 20;
constexpr double kUnitTol = 4.0 * 5.9604644775390625e-8;       // |q|^2 within this of 1: FP32 path

__device__ __forceinline__ unsigned long long f2_neg(unsigned long long a) { return a ^ 0x8000000080000000ull; }
// Two dot products of three terms in double-FP32 (exact products of the hi parts, two-sums), rounded to
// FP32: packed, so that the six of a sample are three of these (half the instructions, the same roundings).
__device__ __forceinline__ unsigned long long dot3_df_x2(const unsigned long long (&mh)[3], const unsigned long long (&ml)[3],
                                                         const unsigned long long (&vh)[3], const unsigned long long (&vl)[3])
{
    unsigned long long s = f2_mul(mh[0], vh[0]);
    unsigned long long err = f2_fma(mh[0], vl[0], f2_fma(ml[0], vh[0], f2_fma(mh[0], vh[0], f2_neg(s))));
#pragma unroll
    for (int j = 1; j < 3; ++j) {
        const unsigned long long p = f2_mul(mh[j], vh[j]);
        const unsigned long long e = f2_fma(mh[j], vh[j], f2_neg(p));
        const unsigned long long t = f2_add(s, p);
        const unsigned long long bv = f2_sub(t, s);
        const unsigned long long te = f2_add(f2_sub(s, f2_sub(t, bv)), f2_sub(p, bv));
        s = t;
        err = f2_fma(mh[j], vl[j], f2_fma(ml[j], vh[j], f2_add(err, f2_add(te, e))));
    }
    return f2_add(s, err);
}

__device__ __forceinline__ float frac_dist(float v)
{
    const float f = v - floorf(v);
    return fminf(f, 1.f - f);
}

// FP32 RING lookup with certified floors; false if any decision is within its error bound.
// Integer work is 32-bit (every index stays below 12 * 8192^2 < 2^31): conversions between FP32
// and 64-bit integers would run on the FP64 pipe.
__device__ __forceinline__ bool fast_ring_pixel(float dx, float dy, float dz, int32_t nside, int32_t &pix)
{
    const float rho2 = fmaf(dx, dx, dy * dy);
    if (!(rho2 >= 0.0025f)) return false;              // within ~3 deg of a pole (or NaN)
    const float za = fabsf(dz);
    if (fabsf(za - 0.6666667f) <= 64.f * kU) return false;   // zone decision
    const float N = (float)nside;
    float phi = atan2f(dy, dx);
    if (phi < 0.f) phi += 6.2831855f;
    const float tt = phi * 0.63661977f;
    if (za <= 0.6666667f) {
        const float t1 = N * (0.5f + tt), t2 = N * (dz * 0.75f);
        const float a1 = t1 - t2, a2 = t1 + t2;
        const float m = 96.f * N * kU + 16.f * kU;
        if (frac_dist(a1) <= m || frac_dist(a2) <= m) return false;
        const int32_t jp = (int32_t)floorf(a1), jm = (int32_t)floorf(a2);
        const int32_t ir = nside + 1 + jp - jm;
        const int32_t kshift = 1 - (ir & 1);
        const int32_t nl4 = 4 * nside;
        int32_t ip = (jp + jm - nside + kshift) >> 1;   // an even number in [-2, 8 nside]
        if (ip >= nl4) ip -= nl4;
        if (ip < 0) ip += nl4;
        const int32_t p = 2 * nside * (nside - 1) + (ir - 1) * nl4 + ip;
        if (p < 0 || p >= 12 * nside * nside) return false;
        pix = p;
        return true;
    }
    const float rho = sqrtf(rho2);
    const float ft = tt - floorf(tt);
    if (fminf(ft, 1.f - ft) <= 16.f * kU / rho + 64.f * kU) return false;   // facet edge
    const float tmp = N * sqrtf(3.f * (rho2 / (1.f + za)));
    const float b1 = ft * tmp, b2 = (1.f - ft) * tmp;
    const float mc = 112.f * N * kU + 16.f * kU;
    if (frac_dist(b1) <= mc || frac_dist(b2) <= mc) return false;
    const int32_t jp = (int32_t)floorf(b1), jm = (int32_t)floorf(b2);
    const int32_t ir = jp + jm + 1;
    const float b3 = tt * (float)ir;
    if (frac_dist(b3) <= 96.f * N * kU + 16.f * kU / rho + 64.f * kU) return false;
    int32_t ip = (int32_t)floorf(b3);
    const int32_t nl = 4 * ir;
    if (ip >= nl) ip -= nl;
    if (ip < 0) ip += nl;
    const int32_t p = dz > 0.f ? 2 * ir * (ir - 1) + ip : 12 * nside * nside - 2 * ir * (ir + 1) + ip;
    if (p < 0 || p >= 12 * nside * nside) return false;
    pix = p;
    return true;
}

// Third and first columns of R(q_det) (line of sight and orientation of the detector) in
// double-FP32: out = d hi[3], d lo[3], o hi[3], o lo[3]. False if |q_det|^2 is not within 4u of 1 (every
// sample of that detector then takes the exact recipe). FP64: call once per detector.
__device__ __forceinline__ bool det_axes_df(const Quat &qd, float *out)
{
    const double n2 = qd.w * qd.w + qd.x * qd.x + qd.y * qd.y + qd.z * qd.z;
    const double xx = qd.x * qd.x, yy = qd.y * qd.y, zz = qd.z * qd.z;
    const double xy = qd.x * qd.y, xz = qd.x * qd.z, yz = qd.y * qd.z;
    const double wx = qd.w * qd.x, wy = qd.w * qd.y, wz = qd.w * qd.z;
    const double dv[3] = {2.0 * (xz + wy), 2.0 * (yz - wx), 1.0 - 2.0 * (xx + yy)};
    const double ov[3] = {1.0 - 2.0 * (yy + zz), 2.0 * (xy + wz), 2.0 * (xz - wy)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float h = (float)dv[k], g = (float)ov[k];
        out[k] = h;
        out[3 + k] = (float)(dv[k] - (double)h);
        out[6 + k] = g;
        out[9 + k] = (float)(ov[k] - (double)g);
    }
    return fabs(n2 - 1.0) <= kUnitTol;
}

// The detector's axes as the packed operands of dot3_df_x2.
struct DetAxes {
    unsigned long long dh[3], dl[3], oh[3], ol[3], bh[3], bl[3];   // (d, d), (o, o), (d, o): hi and lo words
    __device__ __forceinline__ explicit DetAxes(const float *ax)
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            dh[k] = pack_f32x2(ax[k], ax[k]);
            dl[k] = pack_f32x2(ax[3 + k], ax[3 + k]);
            oh[k] = pack_f32x2(ax[6 + k], ax[6 + k]);
            ol[k] = pack_f32x2(ax[9 + k], ax[9 + k]);
            bh[k] = pack_f32x2(ax[k], ax[6 + k]);
            bl[k] = pack_f32x2(ax[3 + k], ax[9 + k]);
        }
    }
};

// Pixel and FP32 weights (cos 2psi, sin 2psi) of one sample from its boresight row m and the detector
// axes; false if the exact recipe must decide. No half-wave plate or offset rotation.
__device__ __forceinline__ bool certified_sample(const float *m, const DetAxes &ax, int32_t nside, int32_t &pix, float &c,
                                                 float &s)
{
    const float4 *q = reinterpret_cast<const float4 *>(m);
    const float4 q0 = __ldg(q), q1 = __ldg(q + 1), q2 = __ldg(q + 2), q3 = __ldg(q + 3), q4 = __ldg(q + 4);
    if (isnan(q0.x)) return false;
    const unsigned long long ph[3] = {pack_f32x2(q0.x, q0.y), pack_f32x2(q0.z, q0.w), pack_f32x2(q1.x, q1.y)};
    const unsigned long long pl[3] = {pack_f32x2(q1.z, q1.w), pack_f32x2(q2.x, q2.y), pack_f32x2(q2.z, q2.w)};
    const unsigned long long zh[3] = {pack_f32x2(q3.x, q3.x), pack_f32x2(q3.y, q3.y), pack_f32x2(q3.z, q3.z)};
    const unsigned long long zl[3] = {pack_f32x2(q3.w, q3.w), pack_f32x2(q4.x, q4.x), pack_f32x2(q4.y, q4.y)};
    float dx, dy, dz, ox, oy, oz;
    unpack_f32x2(dot3_df_x2(ph, pl, ax.dh, ax.dl), dx, dy);
    unpack_f32x2(dot3_df_x2(ph, pl, ax.oh, ax.ol), ox, oy);
    unpack_f32x2(dot3_df_x2(zh, zl, ax.bh, ax.bl), dz, oz);
    if (!fast_ring_pixel(dx, dy, dz, nside, pix)) return false;
    // psi from local north through east (same convention as the exact recipe)
    const float rho2 = fmaf(dx, dx, dy * dy);
    const float a = fmaf(-dz, fmaf(ox, dx, oy * dy), rho2 * oz);
    const float b = fmaf(oy, dx, -ox * dy);
    const float n2 = fmaf(a, a, b * b);
    const float inv = 1.f / n2;
    c = (a * a - b * b) * inv;
    s = 2.f * a * b * inv;
    return true;
}

// Boresight rows for certified_sample ([n][kBoreRow], pointing_fast.cu).
__global__ void bore_matrix_kernel(const double *__restrict__ q_bore, int64_t n, float *__restrict__ m);

}  // namespace fx
