// nsli_map.cuh -- device code shared by the dense Map and Reduce kernels:
// storage types and their decoding, warp folds, and the reduce-and-step of
// one 32-column block.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <cfloat>
#include <cmath>

#include "nsli.h"
#include "nsli_internal.h"
#include "nsli_async.cuh"

namespace nsli {

// ---------------------------------------------------------------- traits ----

template <int S> struct Traits;
template <> struct Traits<NSLI_F64> {
    using acc = double;
    using meta = RowMeta64;
    static constexpr int EPV = 2;   // elements per 16-byte vector
    static constexpr int BYTES = 8;
};
template <> struct Traits<NSLI_F32> {
    using acc = float;
    using meta = RowMeta32;
    static constexpr int EPV = 4;
    static constexpr int BYTES = 4;
};
template <> struct Traits<NSLI_BF16> {
    using acc = float;
    using meta = RowMeta32;
    static constexpr int EPV = 8;
    static constexpr int BYTES = 2;
};
template <> struct Traits<NSLI_FP8E4M3> {
    using acc = float;
    using meta = RowMeta32;
    static constexpr int EPV = 16;
    static constexpr int BYTES = 1;
};

__device__ __forceinline__ float meta_scale(const RowMeta32 &m) { return m.scale; }
__device__ __forceinline__ double meta_scale(const RowMeta64 &) { return 1.0; }

__device__ __forceinline__ void fp8x2_to_float2(unsigned int pair, float &lo, float &hi)
{
    __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(pair & 0xffffu), __NV_E4M3);
    const float2 f = __half22float2(__half2(hr));
    lo = f.x;
    hi = f.y;
}

// Decode one 16-byte vector of stored elements into the accumulation type.
template <int S>
__device__ __forceinline__ void decode(const uint4 q, typename Traits<S>::acc (&a)[Traits<S>::EPV]);

template <> __device__ __forceinline__ void decode<NSLI_F64>(const uint4 q, double (&a)[2])
{
    a[0] = __hiloint2double((int)q.y, (int)q.x);
    a[1] = __hiloint2double((int)q.w, (int)q.z);
}
template <> __device__ __forceinline__ void decode<NSLI_F32>(const uint4 q, float (&a)[4])
{
    a[0] = __uint_as_float(q.x);
    a[1] = __uint_as_float(q.y);
    a[2] = __uint_as_float(q.z);
    a[3] = __uint_as_float(q.w);
}
template <> __device__ __forceinline__ void decode<NSLI_BF16>(const uint4 q, float (&a)[8])
{
    const unsigned int w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        a[2 * k] = __uint_as_float(w[k] << 16);
        a[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
}
template <> __device__ __forceinline__ void decode<NSLI_FP8E4M3>(const uint4 q, float (&a)[16])
{
    const unsigned int w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        fp8x2_to_float2(w[k], a[4 * k], a[4 * k + 1]);
        fp8x2_to_float2(w[k] >> 16, a[4 * k + 2], a[4 * k + 3]);
    }
}

template <typename T> __device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// d0 += a0 * b0 and d1 += a1 * b1 with one packed binary32x2 FMA
// (round to nearest; the same result as two scalar fmaf).
__device__ __forceinline__ void fma2(float &d0, float &d1, float a0, float a1, float b0, float b1)
{
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "mov.b64 rd, {%0, %1};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rd;\n\t"
        "mov.b64 {%0, %1}, rd;\n\t}"
        : "+f"(d0), "+f"(d1)
        : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
__device__ __forceinline__ void fma2(double &d0, double &d1, double a0, double a1, double b0, double b1)
{
    d0 = fma(a0, b0, d0);
    d1 = fma(a1, b1, d1);
}

template <typename T> __device__ __forceinline__ T neg_inf();
template <> __device__ __forceinline__ float neg_inf<float>() { return -INFINITY; }
template <> __device__ __forceinline__ double neg_inf<double>() { return -INFINITY; }

// Sum v[0..RG) over the warp with one folded butterfly; returns, in lane l,
// the warp total of row l / (32 / RG).
template <int RG, typename T> __device__ __forceinline__ T warp_fold_rows(const T (&v)[RG], int lane)
{
    if constexpr (RG == 1) {
        return warp_sum(v[0]);
    } else if constexpr (RG == 2) {
        const bool hi = (lane & 16) != 0;
        T keep = hi ? v[1] : v[0];
        const T send = hi ? v[0] : v[1];
        keep += __shfl_xor_sync(0xffffffffu, send, 16);
#pragma unroll
        for (int off = 8; off > 0; off >>= 1)
            keep += __shfl_xor_sync(0xffffffffu, keep, off);
        return keep;
    } else if constexpr (RG == 8) {
        // lanes [4q, 4q + 4) end with row q: three exchange levels, then a
        // butterfly over four lanes (the pairing of every level as in the
        // one-row butterfly)
        const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0, b2 = (lane & 4) != 0;
        T k[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const T keep = b4 ? v[q + 4] : v[q];
            const T send = b4 ? v[q] : v[q + 4];
            k[q] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
        T m0 = b3 ? k[2] : k[0], m1 = b3 ? k[3] : k[1];
        const T t0 = b3 ? k[0] : k[2], t1 = b3 ? k[1] : k[3];
        m0 += __shfl_xor_sync(0xffffffffu, t0, 8);
        m1 += __shfl_xor_sync(0xffffffffu, t1, 8);
        T keep = b2 ? m1 : m0;
        const T send = b2 ? m0 : m1;
        keep += __shfl_xor_sync(0xffffffffu, send, 4);
        keep += __shfl_xor_sync(0xffffffffu, keep, 2);
        keep += __shfl_xor_sync(0xffffffffu, keep, 1);
        return keep;
    } else {
        static_assert(RG == 4, "row groups of 1, 2, 4 or 8");
        const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0;
        T k0 = b4 ? v[2] : v[0], k1 = b4 ? v[3] : v[1];
        const T s0 = b4 ? v[0] : v[2], s1 = b4 ? v[1] : v[3];
        k0 += __shfl_xor_sync(0xffffffffu, s0, 16);
        k1 += __shfl_xor_sync(0xffffffffu, s1, 16);
        T keep = b3 ? k1 : k0;
        const T send = b3 ? k0 : k1;
        keep += __shfl_xor_sync(0xffffffffu, send, 8);
#pragma unroll
        for (int off = 4; off > 0; off >>= 1)
            keep += __shfl_xor_sync(0xffffffffu, keep, off);
        return keep;
    }
}

// ---------------------------------------------------- reduce and update ----
//
// Block = 256 threads = 8 groups x 32 columns.  Group q sums partial rows
// g = q, q + 8, ... of its column in the accumulation type, and the 8 group
// sums are added in binary64: in order 0..7 for binary32 storage; for
// binary64 storage, whose dependent operations are slow on GB300, as four
// running sums per group and trees.  Every block recomputes h and the maxima
// from the per-CTA records (exact integer sum / exact maxima), so all blocks
// take the same decision.  The last block to finish (ticket) completes the
// step.
template <int NGRP> struct ReduceSharedT {
    double part[NGRP][32];
    double red[NGRP];
    long long h;
    double mv, mn, mb;
    int last;
};
using ReduceShared = ReduceSharedT<8>;

__device__ __forceinline__ unsigned long long red_ord_enc(double d)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(d);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double red_ord_dec(unsigned long long u)
{
    const unsigned long long bits = (u >> 63) ? (u & 0x7fffffffffffffffull) : ~u;
    return __longlong_as_double((long long)bits);
}

// Barrier of the threads that run one reduce item: the whole block
// (bar_id < 0) or the named barrier bar_id of nthr threads.
__device__ __forceinline__ void sub_sync(int bar_id, int nthr)
{
    if (bar_id < 0)
        __syncthreads();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(nthr) : "memory");
}

template <typename SH>
__device__ __forceinline__ void reduce_stats(const PartStat *ps, int G, SH &sh, int tid = threadIdx.x)
{
    const int lane = tid & 31;
    // maxima as order-preserving integers: exact, and no binary64 compare
    // (a long dependency chain on GB300) on the way
    if (tid < 32) {
        long long h = 0;
        unsigned long long mv = red_ord_enc(-INFINITY), mn = mv, mb = red_ord_enc(0.0);
#pragma unroll 4
        for (int g = lane; g < G; g += 32) {
            const PartStat q = ps[g];
            h += q.h;
            mv = max(mv, red_ord_enc(q.maxviol));
            mn = max(mn, red_ord_enc(q.maxnorm));
            mb = max(mb, red_ord_enc(q.maxb));
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            h += __shfl_xor_sync(0xffffffffu, h, off);
            mv = max(mv, __shfl_xor_sync(0xffffffffu, mv, off));
            mn = max(mn, __shfl_xor_sync(0xffffffffu, mn, off));
            mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, off));
        }
        if (lane == 0) {
            sh.h = h;
            sh.mv = red_ord_dec(mv);
            sh.mn = red_ord_dec(mn);
            sh.mb = red_ord_dec(mb);
        }
    }
}

// Column block `blk` of `nblk` of one problem's reduce-and-step, by a block
// of NGRP warps (NGRP groups of partial rows per column: 8 in the
// reduce kernels, 2 in the persistent serving kernel).
template <typename Acc, int NGRP = 8>
__device__ __forceinline__ void reduce_body(const ReduceArgs &p, const int blk, const int nblk,
                                            ReduceSharedT<NGRP> &sh, const int tid, const int bar_id)
{
    // tid / bar_id: the thread's index within the NGRP warps that run this
    // item and their barrier (-1: the whole block; else the named barrier
    // bar_id of NGRP * 32 threads)
    const int nthr = NGRP * 32;
    DevState *st = p.st;
    if (*(volatile int *)&st->done)
        return;
    const int lane = tid & 31, grp = tid >> 5;
    reduce_stats(p.part_stat, p.G, sh, tid);
    sub_sync(bar_id, nthr);
    const long long h = sh.h;
    const double mv = sh.mv, mn = sh.mn, mb = sh.mb;
    const int stop = st->stop;
    const double eps = st->eps;
    const bool force = st->force_step != 0;
    const bool pass = !force && ((stop != NSLI_STOP_NONE && h == 0) || (stop == NSLI_STOP_EPSMEM && mn < eps) ||
                                 (stop == NSLI_STOP_MAXVIOL_REL && mv <= eps * mb));
    const bool at_max = !pass && (st->it >= st->max_iter);
    const bool step = !pass && !at_max;
    const int rule = st->rule;
    const double lambda = st->lambda;
    const long long j = (long long)blk * kReduceCols + lane;

    if (step) {
        double yj = 0.0;
        if (j < p.ld) {
            const Acc *py = static_cast<const Acc *>(p.part_y);
            // the partial rows g = grp, grp + NGRP, ... added in that order
            // in the accumulation type (binary64 is slow on this part), the
            // NGRP group sums then in binary64
            if constexpr (sizeof(Acc) == 8) {
                // binary64: four running sums (g = grp + NGRP (4c + u)),
                // added in a tree; a dependent binary64 add costs about 300
                // cycles on a full SM (64 on an idle one)
                double a[4] = {0.0, 0.0, 0.0, 0.0};
                for (int g = grp; g < p.G; g += 4 * NGRP) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (g + NGRP * u < p.G)
                            a[u] += py[(long long)(g + NGRP * u) * p.ld + j];
                }
                yj = (a[0] + a[1]) + (a[2] + a[3]);
            } else {
                Acc t = Acc(0);
#pragma unroll 8
                for (int g = grp; g < p.G; g += NGRP)
                    t += py[(long long)g * p.ld + j];
                yj = (double)t;
            }
        }
        sh.part[grp][lane] = yj;
    }
    sub_sync(bar_id, nthr);
    if (step && grp == 0) {
        // the NGRP group sums added pairwise (adjacent pairs, log2 NGRP
        // levels): a chain of dependent binary64 adds costs about 300 cycles a
        // link on a full SM
        static_assert((NGRP & (NGRP - 1)) == 0, "a power-of-two number of groups");
        double v[NGRP];
#pragma unroll
        for (int q = 0; q < NGRP; ++q)
            v[q] = sh.part[q][lane];
#pragma unroll
        for (int w = NGRP / 2; w >= 1; w /= 2) {
#pragma unroll
            for (int q = 0; q < w; ++q)
                v[q] = v[2 * q] + v[2 * q + 1];
        }
        const double y = v[0];
        double val = 0.0;
        if (j < p.ld) {
            if (rule == NSLI_RULE_MODAP) {
                p.ybuf[j] = y;
                val = y * y;
            } else {
                const double s = h > 0 ? (p.rtab ? __ldg(p.rtab + h) : lambda / (double)h) : 0.0;
                const double xo = p.x64[j];
                const double xn = xo - s * y;
                p.x64[j] = xn;
                static_cast<Acc *>(p.x)[j] = (Acc)xn;
                const double d = xn - xo;
                val = d * d;
            }
        }
        val = warp_sum(val);
        if (lane == 0)
            p.part_dx[blk] = val;
    }
    __threadfence();
    sub_sync(bar_id, nthr);
    if (tid == 0) {
        const unsigned int t = atomicAdd(&st->ticket, 1u);
        sh.last = (t == (unsigned int)nblk - 1) ? 1 : 0;
    }
    sub_sync(bar_id, nthr);
    if (!sh.last)
        return;
    __threadfence();

    double dx2 = 0.0, ynorm = 0.0;
    if (step) {
        if (grp == 0) {
            // four running sums per lane (blocks q = lane + 32 (4c + u)),
            // added pairwise: a quarter of the dependent binary64 adds
            double v4[4] = {0.0, 0.0, 0.0, 0.0};
            for (int q = lane; q < nblk; q += 128) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (q + 32 * u < nblk)
                        v4[u] += __ldcg(p.part_dx + q + 32 * u);
            }
            double v = (v4[0] + v4[1]) + (v4[2] + v4[3]);
            v = warp_sum(v);
            if (lane == 0)
                sh.red[0] = v;
        }
        sub_sync(bar_id, nthr);
        const double tot = sh.red[0];
        if (rule == NSLI_RULE_MODAP) {
            ynorm = sqrt(tot);
            const double s = ynorm > 0.0 ? lambda / ynorm : 0.0;
            Acc *x = static_cast<Acc *>(p.x);
            double v = 0.0;
            for (long long q = tid; q < p.ld; q += nthr) {
                const double xo = p.x64[q];
                const double xn = xo - s * __ldcg(p.ybuf + q);
                p.x64[q] = xn;
                x[q] = (Acc)xn;
                const double d = xn - xo;
                v += d * d;
            }
            v = warp_sum(v);
            sub_sync(bar_id, nthr);
            if (lane == 0)
                sh.red[grp] = v;
            sub_sync(bar_id, nthr);
            double t = 0.0;
            for (int q = 0; q < NGRP; ++q)
                t += sh.red[q];
            dx2 = t;
        } else {
            dx2 = tot;
        }
    }
    if (tid == 0) {
        st->h = h;
        st->maxviol = mv;
        st->maxnorm = mn;
        st->maxb = mb;
        if (pass) {
            st->status = ST_CANDIDATE;
            st->done = 1;
        } else if (at_max) {
            st->status = NSLI_NOT_CONVERGED;
            st->done = 1;
        } else {
            st->it += 1;
            if (!st->hold_tick)
                st->tick += 1;
            st->dx2 = dx2;
            st->y_norm = ynorm;
            if (stop == NSLI_STOP_STEP && step_norm_below(dx2, eps)) {
                st->status = NSLI_OK;
                st->done = 1;
            }
        }
        st->force_step = 0;
        st->ticket = 0u;
    }
}

}  // namespace nsli
