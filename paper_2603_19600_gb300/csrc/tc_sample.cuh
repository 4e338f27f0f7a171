// Per-sample pointing and data in FP64 for the tensor-core tile kernels (fused_tc.cu, chi2_tc.cu). The
// loads of a sample are unconditional (clamped indices), so that a thread's samples can be in flight
// together; FP32 words widen on the integer pipe.
#pragma once
#include "band_tc.cuh"

namespace fx {

template <typename DT>
__device__ __forceinline__ double tod_f64(DT v)
{
    if constexpr (sizeof(DT) == 8) return v;
    else return f32_to_f64_bits(v);
}

// One pixel of an FP64 map padded to 32-byte records (I, Q, U, 0): one 32-byte load and one L2 sector per
// random gather, where a 24-byte record takes two or three loads and 1.5 sectors (fill phase of the normal
// operator, 256 threads: 43,600 cycles per tile with three loads, sample by sample; 30,200 with two and the batches
// below; 25,700 with this, 21,300 with 512 threads; the pass that packs the map costs 8 us at nside 256).
struct TcPix {
    double i, q, u;
    __device__ __forceinline__ void load(const double4_32a *__restrict__ x4, int64_t gp)
    {
        double pad;
        asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(i), "=d"(q), "=d"(u), "=d"(pad) : "l"(x4 + gp));
    }
    __device__ __forceinline__ double project(int32_t pix, double c, double s) const
    {
        return pix >= 0 ? fma(u, s, fma(q, c, i)) : 0.0;
    }
};

// The tile's slots that lie in the stream: [tc_in0, tc_in1).
__device__ __forceinline__ int tc_in0(const Tile &tl) { return tl.t0 < kHalo ? (int)(kHalo - tl.t0) : 0; }
__device__ __forceinline__ int tc_in1(const Tile &tl, const ObsInfo &ob)
{
    return (int)min((int64_t)(tl.len + 2 * kHalo), ob.nsamp - tl.t0 + kHalo);
}

// This thread's slot k and the sample it stands for, clamped into the tile's loaded range.
struct TcSlots {
    int64_t row;   // flat index of slot 0
    int in0, in1;
    __device__ __forceinline__ TcSlots(const Tile &tl, const ObsInfo &ob)
        : row(ob.tod_off + (int64_t)tl.det * ob.nsamp + tl.t0 - kHalo), in0(tc_in0(tl)), in1(tc_in1(tl, ob))
    {
    }
    __device__ __forceinline__ int slot(int k) const { return (int)threadIdx.x + k * TT; }
    __device__ __forceinline__ bool in(int k) const { return slot(k) >= in0 && slot(k) < in1; }
    __device__ __forceinline__ int64_t index(int k) const { return row + max(in0, min(slot(k), in1 - 1)); }
};

// v[k] = time-ordered data of this thread's slots (zero outside the stream): every load in flight at once.
template <typename DT>
__device__ __forceinline__ void tc_fill_tod(double (&v)[kTcPer], const TcSlots &sl, const DT *__restrict__ d)
{
    DT raw[kTcPer];
#pragma unroll
    for (int k = 0; k < kTcPer; ++k) raw[k] = __ldg(d + sl.index(k));
#pragma unroll
    for (int k = 0; k < kTcPer; ++k) v[k] = sl.in(k) ? tod_f64(raw[k]) : 0.0;
}

// v[k] = (P x)_t, or d_t - (P x)_t with RESID, of this thread's slots. Cached pointing: every pixel index is
// loaded first, then weights, data and map records a few samples at a time (registers). On the fly: one
// sample at a time (the FP64 recipe is too long to unroll), through shared memory; the recipe's results of the tile's own
// samples are kept for the scatter in this CTA's block of pv.pix, c64, s64 (tc_each<kTcKept>), which stay in L2
// until then.
template <int MODE, bool RESID, typename DT>
__device__ __forceinline__ void tc_fill_map(unsigned char *sm, double (&v)[kTcPer], const TcSlots &sl, const PointingView &pv,
                                            const ObsInfo &ob, const Tile &tl, const DetOffset &psi,
                                            const double4_32a *__restrict__ x, const DT *__restrict__ d)
{
    if constexpr (MODE == 0) {
        double *tmp = tc_ys(sm);   // read back by the thread that wrote it
#pragma unroll 1
        for (int k = 0; k < kTcPer; ++k) {
            double r = 0.0;
            if (sl.in(k)) {
                double c, s;
                const int32_t pix = get_sample<0, double>(pv, ob, tl.det, tl.t0 - kHalo + sl.slot(k), c, s);
                const int t = sl.slot(k) - kHalo;
                if (t >= 0 && t < tl.len) {
                    const int64_t i = (int64_t)blockIdx.x * TILE + t;
                    __stcg(const_cast<int32_t *>(pv.pix) + i, pix);
                    __stcg(const_cast<double *>(pv.c64) + i, c);
                    __stcg(const_cast<double *>(pv.s64) + i, s);
                }
                TcPix m;
                m.load(x, ob.map_off + max(pix, 0));
                r = m.project(pix, c, s);
                if constexpr (RESID) r = tod_f64(__ldg(d + sl.index(k))) - r;
            }
            tmp[sl.slot(k)] = r;
        }
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) v[k] = tmp[sl.slot(k)];
    } else {
        constexpr int B = 3;
        int32_t pix[kTcPer];
#pragma unroll
        for (int k = 0; k < kTcPer; ++k) pix[k] = __ldg(pv.pix + sl.index(k));
#pragma unroll
        for (int k0 = 0; k0 < kTcPer; k0 += B) {
            RawWeights<MODE> w[B];
            TcPix m[B];
            DT dd[B];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = k0 + b;
                if (k < kTcPer) {
                    w[b] = load_weights<MODE>(pv, sl.index(k));
                    m[b].load(x, ob.map_off + max(pix[k], 0));
                    if constexpr (RESID) dd[b] = __ldg(d + sl.index(k));
                }
            }
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = k0 + b;
                if (k < kTcPer) {
                    double c, s;
                    widen_weights<MODE>(w[b], psi, c, s);
                    double r = m[b].project(pix[k], c, s);
                    if constexpr (RESID) r = tod_f64(dd[b]) - r;
                    v[k] = sl.in(k) ? r : 0.0;
                }
            }
        }
    }
}
static_assert(sizeof(double) * kTcPer * TT <= kTcOffCtl - kTcOffX, "the on-the-fly fill fits the samples' region");

// Core samples of the tile in time order, 32 consecutive ones per warp: f(k, pix, c, s, more(k, pix)) for every
// lane of a warp together (pix = -1 past the tile or without a pixel). Cached pointing: the loads of B samples per
// thread (of NT), and what `more` loads for them (k clamped into the tile), are issued before the first is used.
// kTcKept: as left by tc_fill_map<0> of the same CTA, offsets applied.
constexpr int kTcKept = 4;

template <int MODE, int NT, int B, typename G, typename F>
__device__ __forceinline__ void tc_each(const PointingView &pv, const ObsInfo &ob, const Tile &tl, const DetOffset &psi,
                                        G &&more, F &&f)
{
    const int64_t row = ob.tod_off + (int64_t)tl.det * ob.nsamp + tl.t0;
    if constexpr (MODE == 0) {
#pragma unroll 1
        for (int k = threadIdx.x; k - (int)(threadIdx.x & 31) < tl.len; k += NT) {
            double c = 0.0, s = 0.0;
            const int32_t pix = k < tl.len ? get_sample<0, double>(pv, ob, tl.det, tl.t0 + k, c, s) : -1;
            f(k, pix, c, s, more(min(k, tl.len - 1), pix));
        }
    } else if constexpr (MODE == kTcKept) {
        const int64_t at = (int64_t)blockIdx.x * TILE;
#pragma unroll 1
        for (int k = threadIdx.x; k - (int)(threadIdx.x & 31) < tl.len; k += NT) {
            const int64_t i = at + min(k, tl.len - 1);
            const int32_t pix = __ldcg(pv.pix + i);
            const double c = __ldcg(pv.c64 + i), s = __ldcg(pv.s64 + i);
            f(k, k < tl.len ? pix : -1, c, s, more(min(k, tl.len - 1), pix));
        }
    } else {
#pragma unroll 1
        for (int k0 = threadIdx.x; k0 - (int)(threadIdx.x & 31) < tl.len; k0 += B * NT) {
            int32_t pix[B];
            RawWeights<MODE> w[B];
            decltype(more(0, 0)) g[B];
#pragma unroll
            for (int b = 0; b < B; ++b) pix[b] = __ldg(pv.pix + row + min(k0 + b * NT, tl.len - 1));
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = min(k0 + b * NT, tl.len - 1);
                w[b] = load_weights<MODE>(pv, row + k);
                g[b] = more(k, pix[b]);
            }
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int k = k0 + b * NT;
                double c, s;
                widen_weights<MODE>(w[b], psi, c, s);
                f(k, k < tl.len ? pix[b] : -1, c, s, g[b]);
            }
        }
    }
}

struct TcNone {};

// Launches f(tiles, number, view) for chunks of tiles whose FP64 pointing is kept in the on-the-fly workspace.
template <typename F>
furax_status each_kept_chunk(const furax_pointing *p, F &&f)
{
    furax_status rc = ensure_local_ws(p);
    PointingView pv = p->view();
    pv.pix = p->ws_local_pix;
    pv.c64 = reinterpret_cast<const double *>(p->ws_local_c);
    pv.s64 = reinterpret_cast<const double *>(p->ws_local_s);
    const int64_t c = kept_tiles(p);
    for (int64_t t = 0; !rc && t < p->n_tiles; t += c) {
        rc = f((const Tile *)p->d_tiles + t, (unsigned)std::min(c, p->n_tiles - t), pv);
        if (t > 0) count_launches(1);   // the caller counts one
    }
    return rc;
}

}  // namespace fx
