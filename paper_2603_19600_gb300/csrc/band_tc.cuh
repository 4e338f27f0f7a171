// The symmetric band product y_t = sum_{|k|<64} c_|k| x_{t+k} of one 4096-sample tile in FP64 accuracy
// on the tensor cores (SymmetricBandToeplitzOperator, Table 2 of the Furax paper).
//
// The FP64 pipe of this GPU runs ~70x below its FP32 pipes, and 127 FP64 FMAs per sample are what
// bounds every FP64 band product (4.0 Gsamples/s), even in double-FP32 on the FP32 pipes (~25
// Gsamples/s). The product is a contraction with exact integer arithmetic available at tensor-core
// rate, so it is computed without rounding (Ozaki, Ogita, Oishi & Rump 2012, error-free splitting;
// integer digits in FP16 with FP32 accumulators):
//   * the tile's samples become 62-bit integers relative to the tile's largest magnitude, and those
//     eight balanced base-256 digits (values in [-128, 128], exact in FP16); the taps, once per noise
//     handle, 55-bit integers relative to the largest tap and seven digits;
//   * y is a sum over digit pairs (i, j) of weight 256^-(i+j); all pairs of one weight d = i + j share
//     one FP32 accumulator per output: at most 7 pairs x 127 taps x 2^14 < 2^24, so every partial sum
//     is an integer that FP32 holds exactly, in any order. Weights d <= 7 are kept (35 pairs);
//   * the eight accumulators are combined as an 82-bit integer and rounded to FP64 once.
// Error: the dropped weights d >= 8 are ~2^-57 and the taps' rounding ~2^-52.6 of a typical output, and
// the samples are kept to 2^-62 of the tile's maximum. Measured against extended precision (Gaussian
// samples, the 1/f band): N^-1 1.5e-16 relative where the FP64 FMA chain is at 3.8e-16; the normal operator
// 1.3e-16 - 2.2e-16 (chain 1.7e-16 - 2.9e-16, double-FP32 1.3e-14 - 3.9e-14).
//
// As a matrix product: D[m][n] = sum_k A[m][k] B[n][k], row m = outputs 16 m .. 16 m + 15, A[m][k] =
// digit of x[16 m + k] (k < 144: 16 outputs + 126 halo, padded), B[n][k] = digit of c_|k - n - 63|. Both
// operands use the unswizzled K-major core-matrix layout (8 rows x 16 bytes). Consecutive rows of A
// are shifted by 16 samples = two 16-byte units, so the overlapping rows need no copies: the even
// and the odd units of the stream form two planes in which row m + 1 follows row m, the two 8-wide
// halves of a K = 16 step lie one plane apart, and the next step starts one unit further on. A
// core matrix of B depends only on (k - n) / 8, so a digit of the taps is 19 distinct core matrices in
// global memory; the two 8-output halves of a row are swapped (columns 0-7: outputs 8-15) so that
// each half is a window of 18 consecutive ones, copied to shared memory by bulk copies. Digit i of
// x multiplies the digits 0 .. min(6, 7 - i) of c in one instruction: their columns stand side by side
// (16 per digit), and so do the accumulators of the weights i, i + 1, ... in TMEM.
//
// Integers relative to the tile's maximum do not resolve outputs that are far smaller than it. Tiles that
// hold such outputs take a floating-point product instead, decided per tile inside the kernel: the FP64
// FMA chain, or, where the caller asked for no more, the compensated double-FP32 dot product. These are
// tiles where a 32-sample group of the stream is zero or more than 2^6 (2^8) below the tile's maximum (up to
// there the digits' error stays below that of the product they replace, relative to the quiet samples),
// tiles with infinities, NaNs or extreme exponents, and all tiles of bands with fewer than 8 taps or almost
// without weight off the diagonal, where an output can be as small as one sample.
#pragma once
#include <cuda_fp16.h>
#include "tile.cuh"
#include "mbarrier.cuh"

namespace fx {

constexpr int kTcXDig = 8, kTcCDig = 7;                 // digits of the samples and of the taps
constexpr int kTcDiag = 8;                              // weights kept
constexpr int kTcOut = 16;                              // outputs per row (columns per weight)
constexpr int kTcSteps = 9;                             // K = 144 in steps of 16
constexpr int TT = 512;                                 // threads per CTA
constexpr int TR = TILE / TT;                           // outputs per thread
constexpr int kTcSlots = TILE + 128;                    // samples read by the 256 rows
constexpr int kTcPer = (kTcSlots + TT - 1) / TT;        // samples per thread
constexpr int kTcPitch = kTcSlots / 16 * 16 + 32;       // bytes per plane; +32 spreads the planes over the banks
constexpr int kTcRun = 18 * 128;                        // one digit, one half: 18 core matrices
constexpr int kTcCores = 19;                            // distinct core matrices per digit
constexpr int kTcDetBytes = kTcCDig * kTcCores * 128;   // per detector in global memory
constexpr int kTcOffX = kTcCDig * 2 * kTcRun;           // shared memory: taps, then sample digits
constexpr int kTcOffCtl = kTcOffX + kTcXDig * 2 * kTcPitch;
constexpr int kTcRange = 6, kTcRangeDot2 = 8;           // log2 of the largest range taken (see above)
constexpr int kTcNoTaps = -(1 << 20);                   // exponent of taps that have no digits
constexpr int kTcMinTaps = 8;                           // shorter bands take the chain (see above)
constexpr unsigned kTcTmemCols = 256;                   // 2 row blocks x 8 weights x 16 columns
static_assert(TT == 512 && TR == 8 && kTcOut == 2 * TR, "each of 16 warps owns half of 32 rows");
static_assert(kTcOffX % 128 == 0 && kTcPitch % 16 == 0 && kTcRun % 16 == 0, "16-byte units");
static_assert(7 * 127 * 128 * 128 < (1 << 24), "accumulators must stay exact in FP32");
static_assert(sizeof(double) * XS + (sizeof(double) * 96 + 128) * (TT / 32) <= kTcOffCtl - kTcOffX,
              "the samples' region also holds y and the record staging afterwards");

struct TcCtl {
    uint64_t taps_full, mma_done;
    uint32_t tmem;
    unsigned wmax[TT / 32], wmin[TT / 32];
};
constexpr size_t kTcSmem = kTcOffCtl + sizeof(TcCtl);
// Two CTAs per SM (one loads and scatters while the other multiplies) and no more: each holds half of TMEM.
static_assert(2 * (kTcSmem + 1024) <= 228 * 1024 && 3 * kTcSmem > 228 * 1024, "two CTAs per SM");

// Behind the digits' region once the product is done: y (skewed), then one staging area per warp.
__device__ __forceinline__ double *tc_ys(unsigned char *sm) { return reinterpret_cast<double *>(sm + kTcOffX); }
__device__ __forceinline__ double *tc_stage(unsigned char *sm)
{
    return reinterpret_cast<double *>(sm + kTcOffX) + XS + 1 + (threadIdx.x >> 5) * 112;
}
__device__ __forceinline__ int32_t *tc_stage_pix(unsigned char *sm) { return reinterpret_cast<int32_t *>(tc_stage(sm) + 96); }

// Start of the CTA: TMEM, barriers and the copy of the detector's tap digits. Every thread calls it.
__device__ __forceinline__ void tc_begin(unsigned char *sm, const NoiseView &nv, int64_t gdet)
{
    TcCtl &C = *reinterpret_cast<TcCtl *>(sm + kTcOffCtl);
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&C.tmem)),
                     "r"(kTcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
        mbar_init(&C.taps_full, 1);
        mbar_init(&C.mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&C.taps_full)),
                     "r"(kTcCDig * 2 * kTcRun)
                     : "memory");
        const unsigned char *src = nv.tc_taps + gdet * kTcDetBytes;
        for (int j = 0; j < kTcCDig; ++j)
            for (int h = 0; h < 2; ++h)
                bulk_copy_g2s(sm + (2 * j + h) * kTcRun, src + j * kTcCores * 128 + h * 128, kTcRun, &C.taps_full, false, 0);
    }
}

// Unswizzled K-major operand: lead = bytes between the two 8-wide halves of a K step, stride =
// bytes between 8-row groups (both and the address in 16-byte units; bit 46: this descriptor's version).
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lead, uint32_t stride)
{
    return (uint64_t)(addr >> 4) | ((uint64_t)(lead >> 4) << 16) | ((uint64_t)(stride >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, int ndig, bool add)
{
    // FP32 accumulators, FP16 operands, both K-major, N = 16 ndig, M = 128
    const uint32_t idesc = (1u << 4) | ((uint32_t)(2 * ndig) << 17) | (8u << 24);
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)add)
        : "memory");
}

// All digit products of the tile, issued by one thread: two blocks of 128 rows, nine K steps each.
__device__ __forceinline__ void tc_issue(unsigned char *sm, uint32_t tmem)
{
    const uint32_t t0 = smem_u32(sm), x0 = t0 + kTcOffX;
    for (int q = 0; q < kTcSteps; ++q) {
        const uint64_t b = tc_desc(t0 + 256 * q, 128, kTcRun);
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const uint32_t d = tmem + 128 * mt;
#pragma unroll
            for (int i = 0; i < kTcXDig; ++i) {
                const uint64_t a = tc_desc(x0 + 2 * i * kTcPitch + 16 * (128 * mt + q), kTcPitch, 128);
                const int nj = i == 0 ? kTcCDig : kTcDiag - i;
                if (i == 1 && q == 0) {   // weight 7 starts here: the others add to what digit 0 wrote
                    tc_mma(d + 16, a, b, 6, true);
                    tc_mma(d + 112, a, tc_desc(t0 + 12 * kTcRun, 128, kTcRun), 1, false);
                } else {
                    tc_mma(d + 16 * i, a, b, nj, !(q == 0 && i == 0));
                }
            }
        }
    }
}

__device__ __forceinline__ void tc_load4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// (H 2^32 + L) 2^e rounded to the nearest FP64 value (up to a dropped sticky bit), from the encoding on the
// integer pipes: three FP64 additions per output would occupy the FP64 pipe three times as long as
// everything else this kernel does with the integers. |H|, |L| < 2^50.
__device__ __forceinline__ double tc_value(long long H, long long L, int e)
{
    long long hi = H + (L >> 32);
    uint32_t lo = (uint32_t)L;
    const uint32_t sign = (uint32_t)(hi >> 63) & 0x80000000u;
    if (sign) {
        hi = ~hi + (lo == 0u);
        lo = 0u - lo;
    }
    // the leading one to bit 63: at most 32 of the low word's bits fit below 2^50's
    const int z = __clzll(hi);
    const uint64_t frac = z <= 32 ? (uint64_t)lo >> (32 - z) : (uint64_t)lo << (z - 32);
    uint64_t m = z < 64 ? ((uint64_t)hi << z) | frac : 0u;
    int x = 1023 + 63 + 32 - z + e;
    if (z == 64) {   // |value| < 2^32
        const int zl = __clz((int)lo);
        m = zl < 32 ? (uint64_t)lo << (32 + zl) : 0u;
        x = 1023 + 31 - zl + e;
    }
    if (m == 0u) return 0.0;
    m = (m >> 11) + ((m >> 10) & 1u);   // bit 52 is the implicit one; a carry moves into the exponent
    const uint64_t b = ((uint64_t)(uint32_t)(x - 1) << 52) + m;
    return __hiloint2double((int)((uint32_t)(b >> 32) | sign), (int)(uint32_t)b);
}

// One digit pair: half2(1024 + a, 1024 + b) from two bytes of w (offset digits), minus 1152.
__device__ __forceinline__ void tc_put2(unsigned char *p, uint32_t w, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(0x64646464u), "r"(sel));
    const __half2 h = __hsub2(*reinterpret_cast<const __half2 *>(&r), __half2half2(__ushort_as_half(0x6480)));
    *reinterpret_cast<__half *>(p) = __low2half(h);
    *reinterpret_cast<__half *>(p + 2 * kTcPitch) = __high2half(h);
}

constexpr int kTcChainTaps = 16;   // bands up to this long take the chain in either precision

// The FP64 FMA chain over the skewed samples xs, taps from global memory, y over the samples: tiles the
// digits do not take.
// With finite samples the zeros past the band's last tap add nothing and are skipped.
static __device__ __noinline__ void tc_chain(double *xs, const double *__restrict__ c, int ntaps, bool finite)
{
    const int base = threadIdx.x * TR;
    double y[TR];
#pragma unroll
    for (int r = 0; r < TR; ++r) y[r] = 0.0;
    const int skip = finite ? kHalo + 1 - ntaps : 0;
#pragma unroll 1
    for (int j = skip; j < kBand - skip; ++j) {
        const int k = j < kHalo ? kHalo - j : j - kHalo;
        const double t = k < ntaps ? c[k] : 0.0;
#pragma unroll
        for (int r = 0; r < TR; ++r) y[r] = fma(t, xs[spos(base + r + j)], y[r]);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < TR; ++r) xs[spos(base + r)] = y[r];
}

// Compensated dot product in double-FP32 on output pairs (y_i, y_{i+4}) (Ogita, Rump & Oishi 2005,
// algorithm Dot2; packed FP32): every product of the high words is split exactly by an FMA, the products
// are summed with Knuth's two-sum, and errors and cross terms gather in a second word; the product is
// negated once so that no packed negation is needed. C4[j] = (c_hi, c_hi, -c_hi, -c_hi) and CL2[j] =
// (c_lo, c_lo) hold the band in tap order (j < 127). The taps are walked in rolled blocks of 8: a fully
// unrolled body overflows the instruction cache.
constexpr int kDfJB = 8;

__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long f2_sub(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ void dot2_step_x2(unsigned long long ch, unsigned long long nch, unsigned long long cl,
                                             unsigned long long x, unsigned long long &S, unsigned long long &E)
{
    const unsigned long long np = f2_mul(nch, x);          // -p
    const unsigned long long e = f2_fma(ch, x, np);        // ch x - p exactly
    const unsigned long long s = f2_sub(S, np);            // S + p
    const unsigned long long bv = f2_sub(s, S);
    const unsigned long long t2 = f2_sub(S, f2_sub(s, bv));
    const unsigned long long err = f2_sub(t2, f2_add(np, bv));   // (S - (s - bv)) + (p - bv)
    S = s;
    E = f2_fma(cl, x, f2_add(E, f2_add(err, e)));
}

template <int R>
__device__ __forceinline__ void band_product_dfx2(const float *__restrict__ xs, const float *__restrict__ xl,
                                                  const float4 *__restrict__ C4, const float2 *__restrict__ CL2, int base,
                                                  float (&S)[R], float (&E)[R])
{
    constexpr int H = R / 2;
    unsigned long long W[H], WL[H], SS[H], EE[H];   // W[i] = (x[base+i+j], x[base+i+H+j]) at tap j
#pragma unroll
    for (int i = 0; i < H; ++i) {
        W[i] = pack_f32x2(xs[spos(base + i)], xs[spos(base + i + H)]);
        WL[i] = pack_f32x2(xl[spos(base + i)], xl[spos(base + i + H)]);
        SS[i] = 0ull;
        EE[i] = 0ull;
    }
#pragma unroll 1
    for (int j0 = 0; j0 < kBandPad; j0 += kDfJB) {
#pragma unroll
        for (int jj = 0; jj < kDfJB; ++jj) {
            const int j = j0 + jj;
            if (j < kBand) {
                const float4 c4 = C4[j];
                const float2 c2 = CL2[j];
                const unsigned long long ch = pack_f32x2(c4.x, c4.y), nch = pack_f32x2(c4.z, c4.w);
                const unsigned long long cl = pack_f32x2(c2.x, c2.y);
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    dot2_step_x2(ch, nch, cl, W[i], SS[i], EE[i]);
                    EE[i] = f2_fma(ch, WL[i], EE[i]);
                }
                if (j < kBand - 1) {
                    float lo0, hi0;
                    unpack_f32x2(W[0], lo0, hi0);
                    const unsigned long long wl = pack_f32x2(hi0, xs[spos(base + R + j)]);
#pragma unroll
                    for (int i = 0; i < H - 1; ++i) W[i] = W[i + 1];
                    W[H - 1] = wl;
                    {
                        unpack_f32x2(WL[0], lo0, hi0);
                        const unsigned long long wll = pack_f32x2(hi0, xl[spos(base + R + j)]);
#pragma unroll
                        for (int i = 0; i < H - 1; ++i) WL[i] = WL[i + 1];
                        WL[H - 1] = wll;
                    }
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
        unpack_f32x2(SS[i], S[i], S[i + H]);
        unpack_f32x2(EE[i], E[i], E[i + H]);
    }
}

// The compensated product over the samples in the digits' region (high words, then low words, skewed),
// y over them in FP64.
static __device__ __noinline__ void tc_dot2(float *xh, const double *__restrict__ c, int ntaps)
{
    float *xl = xh + XS + 1;
    float4 *C4 = reinterpret_cast<float4 *>(xh + 2 * XS + 4);
    float2 *CL2 = reinterpret_cast<float2 *>(C4 + kBandPad);
    if (threadIdx.x < kBandPad) {
        const int j = threadIdx.x, k = j < kHalo ? kHalo - j : j - kHalo;
        const double t = j < kBand && k < ntaps ? c[k] : 0.0;
        const float h = (float)t, l = (float)(t - (double)h);
        C4[j] = make_float4(h, h, -h, -h);
        CL2[j] = make_float2(l, l);
    }
    __syncthreads();
    float S[TR], E[TR];
    const int base = threadIdx.x * TR;
    band_product_dfx2<TR>(xh, xl, C4, CL2, base, S, E);
    __syncthreads();
    double *ys = reinterpret_cast<double *>(xh);
#pragma unroll
    for (int r = 0; r < TR; ++r) ys[spos(base + r)] = (double)S[r] + (double)E[r];
}
static_assert((2 * XS + 4) % 4 == 0 && sizeof(float) * (2 * XS + 4) + (16 + 8) * kBandPad <= kTcOffCtl - kTcOffX,
              "the compensated product fits the samples' region");

// tc_ys(sm)[spos(t)] = sum_k c_|k| x_{t+k} for the tile's outputs t. v[k]: the sample of slot u = threadIdx.x +
// 512 k (slot 63 is the tile's first output; zero past the loaded samples). Every thread calls it after
// tc_begin; on return the results are visible to the CTA and no TMEM is held. Slots [in0, in1) lie in the
// stream. f64: FP64 accuracy of every output (else that of the compensated product). MASKED: zero
// samples are masked ones whose own outputs are not used (the vectors of gap filling): all-zero groups do not
// count as quiet.
template <bool MASKED>
__device__ __forceinline__ void tc_band(unsigned char *sm, const double (&v)[kTcPer], const NoiseView &nv, int64_t gdet,
                                        unsigned *err, bool f64, int in0, int in1)
{
    TcCtl &C = *reinterpret_cast<TcCtl *>(sm + kTcOffCtl);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // largest and smallest nonzero 32-sample group maximum (high words of |x| order like the values)
    unsigned gmax = 0u, gmin = 0xffffffffu;
#pragma unroll
    for (int k = 0; k < kTcPer; ++k) {
        const unsigned m = __reduce_max_sync(0xffffffffu, (unsigned)__double2hiint(v[k]) & 0x7fffffffu);
        gmax = max(gmax, m);
        const int u0 = 32 * warp + k * TT;
        if (MASKED ? m != 0u : u0 >= in0 && u0 + 32 <= in1) gmin = min(gmin, m);   // whole groups of the stream
    }
    if (lane == 0) { C.wmax[warp] = gmax; C.wmin[warp] = gmin; }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < TT / 32; ++w) { gmax = max(gmax, C.wmax[w]); gmin = min(gmin, C.wmin[w]); }
    const int emax = (int)(gmax >> 20), ec = nv.tc_exp[gdet];
    const int ey = emax - 1022 + ec - 69;   // y = (H 2^32 + L) 2^ey
    const int range = f64 ? kTcRange : kTcRangeDot2;
    const bool digits = emax >= 123 && emax < 2047 && emax - (int)(gmin >> 20) <= range && ec > -900 && ec < 900 && ey > -900 && ey < 900;
    const uint32_t tmem = C.tmem;
    if (digits) {
        unsigned char *px = sm + kTcOffX;
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) {
            const int u = threadIdx.x + k * TT;
            if (u < kTcSlots) {
                // 62-bit integer x 2^(62 - ex) with |x| < 2^ex, then offset digits (byte = digit + 128)
                const uint32_t hi = (uint32_t)__double2hiint(v[k]), lo = (uint32_t)__double2loint(v[k]);
                const int e = (int)(hi >> 20) & 0x7ff;
                uint64_t m = (((uint64_t)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo) << 9;
                m >>= min(emax - e, 63);
                const uint64_t w = ((int32_t)hi < 0 ? 0ull - m : m) + 0x8080808080808080ull;
                unsigned char *p = px + ((u >> 3) & 1) * kTcPitch + (u >> 4) * 16 + (u & 7) * 2;
                const uint32_t wh = (uint32_t)(w >> 32), wl = (uint32_t)w;
                tc_put2(p, wh, 0x4243);
                tc_put2(p + 4 * kTcPitch, wh, 0x4041);
                tc_put2(p + 8 * kTcPitch, wl, 0x4243);
                tc_put2(p + 12 * kTcPitch, wl, 0x4041);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the digits, for the tensor core's reads
        __syncthreads();
        const long long budget = wait_budget(err);
        if (threadIdx.x == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (mbar_wait(&C.taps_full, 0, err, budget)) tc_issue(sm, tmem);
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_u32(&C.mma_done))
                         : "memory");
        }
        __syncwarp();
        mbar_wait(&C.mma_done, 0, err, budget);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // warps 4 b .. 4 b + 3 hold the 128 rows of block b & 1, one lane each, and half b >> 1 of their columns
        const int half = warp >> 3, r0 = 128 * ((warp >> 2) & 1) + 32 * (warp & 3) + lane;
        const uint32_t at = tmem + ((uint32_t)(warp & 3) << 21) + 128u * ((warp >> 2) & 1) + 8u * half;
        double *ys = tc_ys(sm) + spos(kTcOut * r0);   // a row's 16 slots are consecutive
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t d[kTcDiag][4];
#pragma unroll
            for (int w = 0; w < kTcDiag; ++w) tc_load4(at + 16 * w + 4 * h, d[w]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                int q[kTcDiag];
#pragma unroll
                for (int w = 0; w < kTcDiag; ++w) q[w] = __float2int_rn(__uint_as_float(d[w][r]));
                const long long H = (long long)q[0] * (1 << 24) + ((long long)q[1] * (1 << 16) + ((long long)q[2] * 256 + q[3]));
                const long long L = (long long)q[4] * (1 << 24) + ((long long)q[5] * (1 << 16) + ((long long)q[6] * 256 + q[7]));
                ys[8 * (1 - half) + 4 * h + r] = tc_value(H, L, ey);
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
    } else {
        // Dot2 well inside FP32's range, and for bands of which the chain's 2 ntaps - 1 FP64 FMAs cost more than its
        // 127 x 10 FP32 operations (right-hand side of 2.1 M samples and 4 taps: 219 us with Dot2, 72 us with the chain)
        const bool dot2 = !f64 && emax > 1023 - 80 && emax < 1023 + 100 && nv.ntaps > kTcChainTaps;
        double *xs = tc_ys(sm);
        float *xh = reinterpret_cast<float *>(xs);
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) {
            const int u = threadIdx.x + k * TT;
            if (u < TILE + 2 * kHalo) {
                if (dot2) {
                    const float h = (float)v[k];
                    xh[spos(u)] = h;
                    xh[XS + 1 + spos(u)] = (float)(v[k] - (double)h);
                } else {
                    xs[spos(u)] = v[k];
                }
            }
        }
        if (threadIdx.x == 0) mbar_wait(&C.taps_full, 0, err, wait_budget(err));   // no copy in flight at exit
        __syncthreads();
        if (dot2) tc_dot2(xh, nv.p64 + gdet * nv.ntaps, nv.ntaps);
        else tc_chain(xs, nv.p64 + gdet * nv.ntaps, nv.ntaps, emax < 2047);
        __syncthreads();
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols));
}

}  // namespace fx
