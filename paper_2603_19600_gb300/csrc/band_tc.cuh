// The symmetric band product y_t = sum_{|k|<64} c_|k| x_{t+k} of one 4096-sample tile in FP64 accuracy
// on the tensor cores (SymmetricBandToeplitzOperator, Table 2 of the Furax paper).
//
// The FP64 pipe of this GPU runs ~70x below its FP32 pipes, and 127 FP64 FMAs per sample are what
// bounds every FP64 band product (4.0 Gsamples/s), even in double-FP32 on the FP32 pipes (~25
// Gsamples/s). The product is a contraction with exact integer arithmetic available at tensor-core
// rate, so it is computed without rounding (Ozaki, Ogita, Oishi & Rump 2012, error-free splitting;
// integer digits in FP16 with FP32 accumulators):
//   * the tile's samples become 62-bit integers relative to the tile's largest magnitude, and those
//     eight balanced base-256 digits (values in [-128, 127], exact in FP16); the taps, once per noise
//     handle, 63-bit integers relative to the largest tap and eight digits;
//   * y is a sum over digit pairs (i, j) of weight 256^-(i+j); all pairs of one weight d = i + j share
//     one FP32 accumulator per output: at most 8 pairs x 127 taps x 2^14 < 2^24, so every partial sum
//     is an integer that FP32 holds exactly, in any order. Weights d <= 7 are kept (36 pairs);
//   * the eight accumulators are combined as an 82-bit integer and rounded to FP64 once.
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
// Error: with X and C the powers of two above the tile's largest sample and the detector's largest tap, an
// output is off by the dropped weights d >= 8, at most 2^-53.2 X C and in practice 2^-59.7 X C (rms; they are sums
// of some 700 digit products of either sign), and by its one rounding. Small beside |c| * |x|, the scale of an FP64 FMA
// chain's error, only where the band reaches samples that are not too far below X. So every block of 8
// outputs is checked: sums of |x| over blocks of 8 samples, weighted with the smallest |tap| that joins the
// two blocks, bound |c| * |x| of its outputs from below (within a factor of 2 for the 1/f band), and blocks for
// which that is under 2^-kTcRange X C are formed again by the FP64 FMA chain. (Ordinary noise passes by a coarser bound of the
// same kind, over groups of 32 samples, without the blocks: right-hand side of 67 M samples 1456 -> 1426 us.) Up to the line the
// digits' error is at most 9 u |c| * |x| in emulation (u = 2^-53; rms 0.3 u on Gaussian samples), that of the chain up to 14 u
// (rms 2 u). An output whose band holds only zeros is exact in digits too. Where the caller asked for no more
// than the compensated double-FP32 product, the line is kTcRangeDot2, and many blocks take that product.
// A few loud samples (glitches, a planet, infinities and NaNs) are left out of the digits, and every block whose band
// reaches one is formed again (tc_band). Tiles with extreme exponents, tiles mostly below the line, and bands whose
// small or missing taps would send ordinary noise to the chain (tap_digits_kernel) form every block that way.
// Measured (FP64 data, 32 x 131,071 samples, N^-1 alone, all tiles alike): 64 us in digits (58 without the checks), 126 us
// with a glitch per tile (895 with the chain for the whole tile), 524 us with half of each tile 2^16 louder.
#pragma once
#include <cuda_fp16.h>
#include <type_traits>
#include "tile.cuh"
#include "mbarrier.cuh"

namespace fx {

constexpr int kTcXDig = 8, kTcCDig = 8;                 // digits of the samples and of the taps
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
constexpr int kTcRange = 9, kTcRangeDot2 = 12;          // -log2 of the smallest |c| * |x| / (X C) taken (see above)
constexpr int kTcNoTaps = -(1 << 20);                   // "exponent" of taps that are not used in digits,
constexpr int kTcBadTaps = -(1 << 21);                  // of taps that are not finite
constexpr int kTcBlocks = kTcSlots / 8;                 // blocks of 8 samples
constexpr int kTcReach = 17;                            // blocks that the band joins to a block of 8 outputs
constexpr int kTcWeights = 16;                          // floats per detector: weights of the first 15, then that of groups of 32
constexpr int kTcSumRows = 64 + kTcReach - 1;
constexpr uint32_t kTcOut28 = 1u << 28;                 // marks a sample above the cut in a sum of 25-bit magnitudes
constexpr int kTcChainTaps = 16;                        // bands up to this long take the chain in either precision
constexpr int kTcLoud = 12;                             // groups of 32 samples that may lie above the cut
constexpr unsigned kTcTmemCols = 256;                   // 2 row blocks x 8 weights x 16 columns
static_assert(TT == 512 && TR == 8 && kTcOut == 2 * TR, "each of 16 warps owns half of 32 rows");
static_assert(kTcOffX % 128 == 0 && kTcPitch % 16 == 0 && kTcRun % 16 == 0, "16-byte units");
static_assert(kTcDiag * 127 * 128 * 128 < (1 << 24), "accumulators must stay exact in FP32");
static_assert(kTcDiag == kTcCDig, "the first digit's instruction writes every weight");
static_assert(TILE / 8 == TT, "one block of outputs per thread");
static_assert(sizeof(double) * XS <= kTcOffX, "the taps' region also holds the samples afterwards");
static_assert(sizeof(double) * XS + (sizeof(double) * 96 + 128) * (TT / 32) <= kTcOffCtl - kTcOffX,
              "the samples' region also holds y and the record staging afterwards");

struct TcCtl {
    uint64_t taps_full, mma_done;
    uint32_t tmem;
    unsigned nlist, gave_up, held;
    __align__(16) unsigned ctl[kCtlWords];   // the handle's control block, copied with the taps
    unsigned gmax[kTcPer * (TT / 32)];   // largest |x| (high word) of each 32 samples
    __align__(16) float w[kTcWeights];   // the detector's weights
    uint32_t least[TT / 32];             // per warp: smallest sum of |x| over 32 samples
    union {
        float sum[kTcSumRows][9];        // sum of |x| over 8 samples (tc_put_sum)
        uint16_t list[TILE / 8];         // blocks of outputs that are formed again
    };
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
__device__ __forceinline__ void tc_begin(unsigned char *sm, const NoiseView &nv, int64_t gdet, const unsigned *err)
{
    TcCtl &C = *reinterpret_cast<TcCtl *>(sm + kTcOffCtl);
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&C.tmem)),
                     "r"(kTcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x < kTcWeights) C.w[threadIdx.x] = __ldg(nv.tc_w + gdet * kTcWeights + threadIdx.x);
    if (threadIdx.x == 0) {
        C.nlist = C.gave_up = C.held = 0u;
        mbar_init(&C.taps_full, 1);
        mbar_init(&C.mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&C.taps_full)),
                     "r"(kTcCDig * 2 * kTcRun + (int)sizeof C.ctl)
                     : "memory");
        bulk_copy_g2s(C.ctl, err, sizeof C.ctl, &C.taps_full, false, 0);
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
                tc_mma(d + 16 * i, a, b, kTcDiag - i, !(q == 0 && i == 0));
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

// Compensated dot product in double-FP32 on output pairs (y_i, y_{i+4}) (Ogita, Rump & Oishi 2005,
// algorithm Dot2; packed FP32): every product of the high words is split exactly by an FMA, the products
// are summed with Knuth's two-sum, and errors and cross terms gather in a second word; the product is
// negated once so that no packed negation is needed. C4[j] = (c_hi, c_hi, -c_hi, -c_hi) and CL2[j] =
// (c_lo, c_lo) hold the band in tap order (j < 127). The taps are walked in rolled blocks of 8: a fully
// unrolled body overflows the instruction cache.
constexpr int kDfJB = 8;

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

// LOW: the samples have low words (FP32 data has none).
template <int R, bool LOW>
__device__ __forceinline__ void band_product_dfx2(const float *__restrict__ xs, const float *__restrict__ xl,
                                                  const float4 *__restrict__ C4, const float2 *__restrict__ CL2, int base,
                                                  float (&S)[R], float (&E)[R])
{
    constexpr int H = R / 2;
    unsigned long long W[H], WL[H], SS[H], EE[H];   // W[i] = (x[base+i+j], x[base+i+H+j]) at tap j
#pragma unroll
    for (int i = 0; i < H; ++i) {
        W[i] = pack_f32x2(xs[spos(base + i)], xs[spos(base + i + H)]);
        if constexpr (LOW) WL[i] = pack_f32x2(xl[spos(base + i)], xl[spos(base + i + H)]);
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
                    if constexpr (LOW) EE[i] = f2_fma(ch, WL[i], EE[i]);
                }
                if (j < kBand - 1) {
                    float lo0, hi0;
                    unpack_f32x2(W[0], lo0, hi0);
                    const unsigned long long wl = pack_f32x2(hi0, xs[spos(base + R + j)]);
#pragma unroll
                    for (int i = 0; i < H - 1; ++i) W[i] = W[i + 1];
                    W[H - 1] = wl;
                    if constexpr (LOW) {
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

// Outputs of the n blocks in C.list again, from the samples in the taps' region (skewed; see tc_put_samples).

// FP64 FMA chain. A warp per block, four lanes to the band of an output, or a thread per block, whose eight outputs share
// the loads: whichever takes fewer FP64 instructions of a warp (17 blocks of 64 taps: 578 against 1016; 512 blocks of 4 taps:
// 2048 against 896, which is 316 against 178 us of a normal operator).
static __device__ __noinline__ void tc_redo_chain(unsigned char *sm, int n, const double *__restrict__ c, int ntaps)
{
    const TcCtl &C = *reinterpret_cast<const TcCtl *>(sm + kTcOffCtl);
    const double *xs = reinterpret_cast<const double *>(sm);
    const int lane = threadIdx.x & 31, part = lane & 3, skip = kHalo + 1 - ntaps;
    if ((n + 31) / 32 * 8 * (2 * ntaps - 1) <= n * ((2 * ntaps + 2) / 4 + 2)) {
        if ((int)threadIdx.x >= n) return;
        const int base = 8 * (int)C.list[threadIdx.x];
        double y[TR];
#pragma unroll
        for (int r = 0; r < TR; ++r) y[r] = 0.0;
#pragma unroll 1
        for (int j = skip; j < kBand - skip; ++j) {
            const double t = __ldg(c + (j < kHalo ? kHalo - j : j - kHalo));
#pragma unroll
            for (int r = 0; r < TR; ++r) y[r] = fma(t, xs[spos(base + r + j)], y[r]);
        }
#pragma unroll
        for (int r = 0; r < TR; ++r) tc_ys(sm)[spos(base + r)] = y[r];
        return;
    }
#pragma unroll 1
    for (int i = threadIdx.x >> 5; i < n; i += TT / 32) {
        const int t = 8 * (int)C.list[i] + (lane >> 2);
        double y = 0.0;
#pragma unroll 4
        for (int j = skip + part; j < kBand - skip; j += 4)
            y = fma(__ldg(c + (j < kHalo ? kHalo - j : j - kHalo)), xs[spos(t + j)], y);
        y += __shfl_xor_sync(0xffffffffu, y, 1);
        y += __shfl_xor_sync(0xffffffffu, y, 2);
        if (part == 0) tc_ys(sm)[spos(t)] = y;
    }
}

// The compensated product, a thread per block.
template <bool LOW>
static __device__ __noinline__ void tc_redo_dot2(unsigned char *sm, int n, const double *__restrict__ c, int ntaps)
{
    const TcCtl &C = *reinterpret_cast<const TcCtl *>(sm + kTcOffCtl);
    const float *xh = reinterpret_cast<const float *>(sm), *xl = xh + XS + 1;
    float4 *C4 = reinterpret_cast<float4 *>(sm + kTcOffCtl) - kBandPad;   // behind y and the staging
    float2 *CL2 = reinterpret_cast<float2 *>(C4) - kBandPad;
    if (threadIdx.x < kBandPad) {
        const int j = threadIdx.x, k = j < kHalo ? kHalo - j : j - kHalo;
        const double t = j < kBand && k < ntaps ? c[k] : 0.0;
        const float h = (float)t, l = (float)(t - (double)h);
        C4[j] = make_float4(h, h, -h, -h);
        CL2[j] = make_float2(l, l);
    }
    __syncthreads();
    if ((int)threadIdx.x >= n) return;
    float S[TR], E[TR];
    const int base = 8 * (int)C.list[threadIdx.x];
    band_product_dfx2<TR, LOW>(xh, xl, C4, CL2, base, S, E);
    double *ys = tc_ys(sm);
#pragma unroll
    for (int r = 0; r < TR; ++r) ys[spos(base + r)] = (double)S[r] + (double)E[r];
}
static_assert(TR == 8 && sizeof(float) * 2 * (XS + 1) <= kTcOffX && kTcOffCtl % 16 == 0 &&
                  sizeof(double) * XS + (sizeof(double) * 96 + 128) * (TT / 32) + (16 + 8) * kBandPad <= kTcOffCtl - kTcOffX,
              "samples in the taps' region, the compensated product's taps behind y and the staging");

// This thread's samples into the taps' region: FP64, or high and low words for the compensated product.
__device__ __forceinline__ void tc_put_samples(unsigned char *sm, const double (&v)[kTcPer], bool dot2)
{
    float *xh = reinterpret_cast<float *>(sm);
    double *xs = reinterpret_cast<double *>(sm);
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
}

// Sum over the 8 lanes of an aligned group of a[0] .. a[7]: lane l gets that of a[l & 7] (7 exchanges instead of 24).
__device__ __forceinline__ uint32_t tc_sum8(const uint32_t (&a)[kTcPer])
{
    const int lane = threadIdx.x & 31;
    uint32_t b[4], c[2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        b[i] = (lane & 4 ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, lane & 4 ? a[i] : a[i + 4], 4);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        c[i] = (lane & 2 ? b[i + 2] : b[i]) + __shfl_xor_sync(0xffffffffu, lane & 2 ? b[i] : b[i + 2], 2);
    return (lane & 1 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, lane & 1 ? c[0] : c[1], 1);
}

// Sum of block 64 k + at: row `at`, so that neither the writing lanes (four rows, eight k) nor the reading ones (a row each)
// share a bank, and once more behind the last row, so that a block's successors are the rows that follow.
__device__ __forceinline__ void tc_put_sum(TcCtl &C, int at, int k, uint32_t s)
{
    const float f = s >= kTcOut28 ? __int_as_float(0x7f800000) : (float)s;
    C.sum[at][k] = f;
    if (at < kTcReach - 1 && k > 0) C.sum[64 + at][k - 1] = f;
}

// True if the band may reach too little for block o of 8 outputs to keep its accuracy in digits (see above), or reaches
// a sample above the cut.
__device__ __forceinline__ bool tc_quiet(const TcCtl &C, int o, float line)
{
    const float *x = &C.sum[o & 63][o >> 6];
    float s = 0.f, any = 0.f;
#pragma unroll
    for (int m = 0; m < kTcReach; ++m) {
        any = fmaxf(any, x[9 * m]);
        if (m < kTcWeights - 1) s = fmaf(C.w[m], x[9 * m], s);
    }
    return any > 0.f && (s < line || any > 1e30f);
}
static_assert(TILE / 8 + kTcReach - 1 == kTcBlocks, "every sample of the band belongs to a block");

struct TcKeep {   // for a caller that needs its samples afterwards
    const double (&v)[kTcPer];
    __device__ __forceinline__ void operator()(double (&w)[kTcPer]) const
    {
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) w[k] = v[k];
    }
};

struct TcAll {   // every output is used
    __device__ __forceinline__ bool operator()(int) const { return true; }
};

// tc_ys(sm)[spos(t)] = sum_k c_|k| x_{t+k} for the tile's len outputs t. v[k]: the sample of slot u = threadIdx.x +
// 512 k (slot 63 is the tile's first output; zero outside the stream and past the loaded samples). Every thread
// calls it after tc_begin; on return the results are visible to the CTA and no TMEM is held. f64: FP64 accuracy of
// every output (else that of the compensated product). LOW: samples may be wider than FP32. False if a wait gave up: there are no results then, and the error
// word is set. again(w): w = v once more, for outputs that are formed again
// (to keep v in registers past the products cost N^-1 alone 109 -> 121 us of 8.4 M samples). used(t): false if outputs
// t .. t + 7 are not used.
template <bool LOW = true, class Again, class Used = TcAll>
__device__ __forceinline__ bool tc_band(unsigned char *sm, const double (&v)[kTcPer], const NoiseView &nv, int64_t gdet,
                                        unsigned *err, bool f64, int len, Again &&again, Used &&used = Used{})
{
    TcCtl &C = *reinterpret_cast<TcCtl *>(sm + kTcOffCtl);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // largest magnitude of each 32 samples (high words of |x| order like the values)
#pragma unroll
    for (int k = 0; k < kTcPer; ++k) {
        const unsigned m = __reduce_max_sync(0xffffffffu, (unsigned)__double2hiint(v[k]) & 0x7fffffffu);
        if (lane == 0) C.gmax[k * (TT / 32) + warp] = m;
    }
    __syncthreads();
    const int range = f64 ? kTcRange : kTcRangeDot2, ec = nv.tc_exp[gdet];
    constexpr int G = (kTcPer * (TT / 32) + 31) / 32;
    unsigned g[G], gmax = 0u;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        g[i] = lane + 32 * i < kTcPer * (TT / 32) ? C.gmax[lane + 32 * i] : 0u;
        gmax = max(gmax, g[i]);
    }
    gmax = __reduce_max_sync(0xffffffffu, gmax);
    auto groups = [&](auto &&f) {   // groups with f(their exponent)
        int n = 0;
#pragma unroll
        for (int i = 0; i < G; ++i) n += __popc(__ballot_sync(0xffffffffu, g[i] != 0u && f((int)(g[i] >> 20))));
        return n;
    };
    int emax = (int)(gmax >> 20);   // exponent of the largest sample in digits
    bool digits = true;
    // Much of the tile is far below its largest sample. If that is up to kTcLoud groups' doing (glitches, a planet, NaNs),
    // these groups' loud samples stay out of the digits and all that the band joins to them is formed again. If the tile is
    // below the line all the same, the products are not worth forming.
    if (emax == 2047 || groups([&](int e) { return e + range - 5 < emax; }) > kTcLoud) {
        int lo = 0, hi = 2047;   // smallest exponent with no more than kTcLoud groups above it
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (groups([&](int e) { return e > mid; }) <= kTcLoud) hi = mid;
            else lo = mid + 1;
        }
        if (lo + 4 <= emax) emax = lo;
        digits = groups([&](int e) { return e + range < emax; }) <= 100;
    }
    const int ey = emax - 1022 + ec - 69;   // y = (H 2^32 + L) 2^ey
    digits = digits && emax >= 123 && emax < 2047 && ec > -900 && ec < 900 && ey > -900 && ey < 900;
    // the compensated product, well inside FP32's range
    const bool may_dot2 = !f64 && nv.ntaps > kTcChainTaps && emax > 1023 - 80 && (int)(gmax >> 20) < 1023 + 100;
    const uint32_t tmem = C.tmem;
    // The chain takes 565 cycles a block with 64 taps, the compensated product, which walks 127 taps whatever their number,
    // 15,000 for any few and 150 a block for many (normal operator with 8 taps: 282 us with the chain, 459 us).
    constexpr int kDot2From = 32;
    int nredo = 0;
    if (digits) {
        unsigned char *px = sm + kTcOffX;
        const int top = (emax + 1) << 20;   // high words from here on stay out
        uint32_t a[kTcPer];   // 2^25 |x| / X rounded down, at least 1 unless x is zero
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) {
            const int u = threadIdx.x + k * TT;
            const uint32_t hi = (uint32_t)__double2hiint(v[k]), lo = (uint32_t)__double2loint(v[k]);
            const int ah = (int)(hi & 0x7fffffffu);
            // 62-bit integer x 2^(62 - ex) with |x| < 2^ex, then offset digits (byte = digit + 128)
            const int e = ah >> 20;
            uint64_t m = (((uint64_t)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo) << 9;
            m = ah >= top ? 0ull : m >> min(emax - e, 63);
            a[k] = ah >= top ? kTcOut28 : (uint32_t)(m >> 32) >> 5 | (uint32_t)((ah | lo) != 0);
            if (u < kTcSlots) {
                const uint64_t w = ((int32_t)hi < 0 ? 0ull - m : m) + 0x8080808080808080ull;
                unsigned char *p = px + ((u >> 3) & 1) * kTcPitch + (u >> 4) * 16 + (u & 7) * 2;
                const uint32_t wh = (uint32_t)(w >> 32), wl = (uint32_t)w;
                tc_put2(p, wh, 0x4243);
                tc_put2(p + 4 * kTcPitch, wh, 0x4041);
                tc_put2(p + 8 * kTcPitch, wl, 0x4243);
                tc_put2(p + 12 * kTcPitch, wl, 0x4041);
            }
        }
        auto block_sums = [&] {
            // sums over blocks: slot u = threadIdx.x + 512 k is of block 64 k + threadIdx.x / 8
            static_assert(kTcPer == 9 && TT == 512, "eight samples at once, then the ninth");
            const int at = threadIdx.x >> 3;
            tc_put_sum(C, at, lane & 7, tc_sum8(a));
            if (512 + at < kTcBlocks) {   // whole warps
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) a[8] += __shfl_xor_sync(0xffffffffu, a[8], o);
                if ((lane & 7) == 0) tc_put_sum(C, at, 8, a[8]);
            }
        };
        // Smallest sum over 32 samples, by which ordinary noise is accepted; vectors with gaps are not.
        constexpr bool kQuick = std::is_same_v<std::decay_t<Used>, TcAll>;
        uint32_t least = 0xffffffffu;
        if constexpr (kQuick) {
#pragma unroll
            for (int k = 0; k < kTcPer; ++k)
                if (k < kTcPer - 1 || warp < (kTcSlots - TT * (kTcPer - 1)) / 32)
                    least = min(least, __reduce_add_sync(0xffffffffu, a[k]));
            if (lane == 0) C.least[warp] = least;
        } else {
            block_sums();
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the digits, for the tensor core's reads
        __syncthreads();
        const long long budget = wait_budget(err);
        if (threadIdx.x == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const bool taps = mbar_wait(&C.taps_full, 0, err, budget);
            if (taps && C.ctl[1]) {
                C.held = 1u;   // nothing is issued, and the waits run out
            } else {
                if (taps) tc_issue(sm, tmem);
                else C.gave_up = 1u;
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 smem_u32(&C.mma_done))
                             : "memory");
            }
        }
        __syncwarp();
        // While the products run: which blocks of outputs the digits do not resolve. None if no 32 samples are quiet enough
        // for three groups of them to be (ordinary noise, except at the ends of streams).
        const float line = ldexpf(1.f, 25 - range);
        if constexpr (kQuick) least = __reduce_min_sync(0xffffffffu, C.least[lane % (TT / 32)]);
        if (!kQuick || emax < (int)(gmax >> 20) || (float)least * C.w[kTcWeights - 1] < line) {
            if constexpr (kQuick) {
                block_sums();
                __syncthreads();
            }
            const int t8 = 8 * threadIdx.x;
            const bool redo = t8 < len && tc_quiet(C, threadIdx.x, line) && used(t8);
            nredo = __syncthreads_count(redo);
            if (redo) C.list[atomicAdd(&C.nlist, 1u)] = (uint16_t)threadIdx.x;
        }
        if (!mbar_wait(&C.mma_done, 0, err, budget)) C.gave_up = 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (nredo) {
            double w[kTcPer];
            again(w);
            tc_put_samples(sm, w, may_dot2 && nredo > kDot2From);
            __syncthreads();   // `again` may use the region of y
        }
    } else {
        if (threadIdx.x == 0 && !mbar_wait(&C.taps_full, 0, err, wait_budget(err))) C.gave_up = 1u;   // written over below
        C.list[threadIdx.x] = (uint16_t)threadIdx.x;
        nredo = (len + 7) / 8;
        bool zero = gmax == 0u && ec != kTcBadTaps;
        if (zero) {   // no sample, no output
            bool any = false;
#pragma unroll
            for (int k = 0; k < kTcPer; ++k) any = any || __double2loint(v[k]) != 0;
            zero = !__syncthreads_or(any);
        }
        if (zero) {
            nredo = 0;
#pragma unroll
            for (int r = 0; r < TR; ++r) tc_ys(sm)[spos(TR * threadIdx.x + r)] = 0.0;
        }
        __syncthreads();
        if (nredo) tc_put_samples(sm, v, may_dot2 && nredo > kDot2From);
    }
    if (digits) {   // sums that are not complete are dropped below
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
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    const bool bad = C.gave_up != 0u;
    if (bad) {   // what is in flight gets as long again to end before its memory is given back
        if (threadIdx.x == 0) {
            mbar_wait(&C.taps_full, 0, err, wait_budget(err));
            if (digits && !C.held) mbar_wait(&C.mma_done, 0, err, wait_budget(err));
        }
        __syncthreads();
    } else if (nredo) {
        const double *c = nv.p64 + gdet * nv.ntaps;
        if (may_dot2 && nredo > kDot2From) tc_redo_dot2<LOW>(sm, nredo, c, nv.ntaps);
        else tc_redo_chain(sm, nredo, c, nv.ntaps);
        __syncthreads();
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols));
    return !bad;
}

}  // namespace fx
