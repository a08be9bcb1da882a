// nsli_sumsq.cuh -- ||a_i||^2 of stored rows with little binary64 work.
//
// GB300 executes binary64 at a small fraction of its binary32 rate, and a
// plain binary64 sum of squares (one conversion and one binary64 FMA per
// entry) bounds the set-up and row-update kernels.  Every stored value of a
// binary32 / bf16 / FP8 row is a binary32 number, so each thread instead
// keeps an unevaluated pair s + c of binary32 numbers ("double-float"):
//   v^2 = p + e exactly (p = fl(v v), e = fma(v, v, -p)),
//   s + p = t + err exactly (two-sum),
//   c += err + e, then (s, c) = fast-two-sum(t, c), so |c| <= ulp(s) / 2.
// Every 8 entries the pair is added to a binary64 accumulator (two binary64
// additions for 8 entries instead of 16 operations).  The pair carries about
// 48 significant bits, so each group of 8 is summed to within a few units of
// 2^-48 relative and the result agrees with a binary64 sum to about 1e-14.
// The quick norm (SumSq2) has no periodic fold: each thread keeps two such
// pairs, for its even and its odd entries, side by side in packed binary32x2
// instructions (13 for two entries instead of 26: the row updates are bound by
// their instructions; 32768 x 16384 rows updated: binary32 747 -> 636 us, bf16
// 724 -> 590 us), and sumsq_block_total adds the pairs of a block as
// double-floats and converts the row total once.
// Values whose square could leave the binary32 normal range (|v| outside
// [2^-60, 2^60]) are squared and added in binary64 directly.  The order is
// fixed per thread, so the set-up kernel and the row-update kernel, which
// both use this, give identical norms for identical rows.  Every operation is
// an explicit round-to-nearest intrinsic so no multiply-add is contracted.
#pragma once

#include <cuda_runtime.h>

namespace nsli {

struct SumSq {
    double acc;
    float s, c;
    int k;
};

__device__ __forceinline__ SumSq sumsq_init()
{
    SumSq q;
    q.acc = 0.0;
    q.s = 0.0f;
    q.c = 0.0f;
    q.k = 0;
    return q;
}

__device__ __forceinline__ void sumsq_flush(SumSq &q)
{
    q.acc = __dadd_rn(q.acc, (double)q.s);
    q.acc = __dadd_rn(q.acc, (double)q.c);
    q.s = 0.0f;
    q.c = 0.0f;
    q.k = 0;
}

// One entry.  FOLD = 8: folded into binary64 every 8 entries (accurate to
// ~1e-14: the binary64 norms); FOLD = 0: never (the quick norm of FP8 rows,
// whose conversions leave no room for the packed form's moves: 32768 x 16384
// rows updated in 1090 us against 1128 us packed).  The range takes one
// integer comparison instead of three (1086 -> 1054 us).
template <int FOLD = 8> __device__ __forceinline__ void sumsq_add(SumSq &q, float v)
{
    // |v| outside [2^-60, 2^60] (one comparison): 0, or in binary64
    const unsigned int u = __float_as_uint(v) & 0x7fffffffu;
    if (u - 0x21800000u > 0x3c000000u) {
        if (u != 0u)
            q.acc = __fma_rn((double)v, (double)v, q.acc);
        return;
    }
    const float p = __fmul_rn(v, v);
    const float e = __fmaf_rn(v, v, -p);          // p + e = v^2 exactly
    const float t = __fadd_rn(q.s, p);            // two-sum: s + p = t + err
    const float bp = __fsub_rn(t, q.s);
    const float err = __fadd_rn(__fsub_rn(q.s, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    const float c = __fadd_rn(q.c, __fadd_rn(err, e));
    const float s2 = __fadd_rn(t, c);             // fast-two-sum (|t| >= |c|)
    q.c = __fsub_rn(c, __fsub_rn(s2, t));
    q.s = s2;
    if (FOLD > 0 && ++q.k == FOLD)
        sumsq_flush(q);
}

__device__ __forceinline__ double sumsq_value(SumSq &q)
{
    sumsq_flush(q);
    return q.acc;
}

// Packed binary32x2 arithmetic, each half rounded to nearest as the scalar
// instruction rounds it.
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi)
{
    return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ float f2_lo(unsigned long long v) { return __uint_as_float((unsigned int)v); }
__device__ __forceinline__ float f2_hi(unsigned long long v) { return __uint_as_float((unsigned int)(v >> 32)); }
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// a - b (the product with -1 is exact, so the sum is rounded once)
__device__ __forceinline__ unsigned long long f2_sub(unsigned long long a, unsigned long long b)
{
    return f2_fma(b, 0xbf800000bf800000ull, a);
}
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Two running double-float sums, of a thread's even and odd entries.
struct SumSq2 {
    double acc;              // squares outside the binary32 range
    unsigned long long s, c;
};
__device__ __forceinline__ SumSq2 sumsq2_init() { return SumSq2{0.0, 0ull, 0ull}; }

// The next two entries (0 for one that does not exist: a zero changes
// neither pair, since s is the rounding of s + c).
__device__ __forceinline__ void sumsq2_add(SumSq2 &q, float v0, float v1)
{
    // |v| outside [2^-60, 2^60] and not 0: in binary64
    const unsigned int u0 = __float_as_uint(v0) & 0x7fffffffu, u1 = __float_as_uint(v1) & 0x7fffffffu;
    const bool out0 = u0 - 0x21800000u > 0x3c000000u && u0 != 0u, out1 = u1 - 0x21800000u > 0x3c000000u && u1 != 0u;
    if (out0 || out1) {
        if (out0) {
            q.acc = __fma_rn((double)v0, (double)v0, q.acc);
            v0 = 0.0f;
        }
        if (out1) {
            q.acc = __fma_rn((double)v1, (double)v1, q.acc);
            v1 = 0.0f;
        }
    }
    const unsigned long long v = f2_pack(v0, v1);
    const unsigned long long p = f2_mul(v, v);
    const unsigned long long e = f2_fma(v, v, p ^ 0x8000000080000000ull);
    const unsigned long long t = f2_add(q.s, p);
    const unsigned long long bp = f2_sub(t, q.s);
    const unsigned long long err = f2_add(f2_sub(q.s, f2_sub(t, bp)), f2_sub(p, bp));
    const unsigned long long c = f2_add(q.c, f2_add(err, e));
    const unsigned long long s2 = f2_add(t, c);
    q.c = f2_sub(c, f2_sub(s2, t));
    q.s = s2;
}

// The quick norm's accumulator, and its next two entries.
template <bool PACKED> struct QuickSumType;
template <> struct QuickSumType<true> { using type = SumSq2; };
template <> struct QuickSumType<false> { using type = SumSq; };
template <bool PACKED> using QuickSum = typename QuickSumType<PACKED>::type;
__device__ __forceinline__ void quick_init(SumSq2 &q) { q = sumsq2_init(); }
__device__ __forceinline__ void quick_init(SumSq &q) { q = sumsq_init(); }
__device__ __forceinline__ void quick_add(SumSq2 &q, float v0, float v1) { sumsq2_add(q, v0, v1); }
__device__ __forceinline__ void quick_add(SumSq &q, float v0, float v1)
{
    sumsq_add<0>(q, v0);
    sumsq_add<0>(q, v1);
}

// (s, c) += (s2, c2) for two double-float pairs of non-negative sums:
// two-sum of the heads (its error is exact, so the result does not depend
// on the order of the operands), the tails and that error added, and a
// fast-two-sum to renormalise (the head dominates: all terms are >= 0).
__device__ __forceinline__ void sumsq_pair_add(float &s, float &c, float s2, float c2)
{
    const float t = __fadd_rn(s, s2);
    const float bp = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(s2, bp));
    const float cc = __fadd_rn(__fadd_rn(c, c2), err);
    const float s3 = __fadd_rn(t, cc);
    c = __fsub_rn(cc, __fsub_rn(s3, t));
    s = s3;
}

// The block total of the per-thread quick sums, for blocks of NW warps: a
// thread's two pairs are added, then the threads' as double-floats in an xor
// tree within each warp and then in warp order by
// thread 0, and converted to binary64 once; the binary64 parts (squares
// outside the binary32 range) are added in binary64 only when some thread
// has one.  Binary32 work instead of a binary64 tree: GB300's binary64 pipe
// takes a whole warp instruction for each binary64 operation.  Every thread
// of the block calls it; the result is valid in thread 0.  spair and sacc
// are shared arrays of NW entries.
__device__ __forceinline__ void quick_pair(const SumSq2 &a, float &s, float &c, double &acc)
{
    s = f2_lo(a.s);
    c = f2_lo(a.c);
    sumsq_pair_add(s, c, f2_hi(a.s), f2_hi(a.c));
    acc = a.acc;
}
__device__ __forceinline__ void quick_pair(const SumSq &a, float &s, float &c, double &acc)
{
    s = a.s;
    c = a.c;
    acc = a.acc;
}
template <int NW, typename Q>
__device__ __forceinline__ double sumsq_block_total(const Q &q, float2 *spair, double *sacc)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float s, c;
    double acc_in;
    quick_pair(q, s, c, acc_in);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float s2 = __shfl_xor_sync(0xffffffffu, s, off);
        const float c2 = __shfl_xor_sync(0xffffffffu, c, off);
        sumsq_pair_add(s, c, s2, c2);
    }
    const bool wide = __syncthreads_or(acc_in != 0.0) != 0;   // block-uniform
    double acc = 0.0;
    if (wide) {
        acc = acc_in;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            acc += __shfl_xor_sync(0xffffffffu, acc, off);
    }
    if (lane == 0) {
        spair[wid] = make_float2(s, c);
        sacc[wid] = acc;
    }
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0) {
        float S = spair[0].x, Cc = spair[0].y;
        for (int w = 1; w < NW; ++w)
            sumsq_pair_add(S, Cc, spair[w].x, spair[w].y);
        t = __dadd_rn((double)S, (double)Cc);
        if (wide) {
            double a = 0.0;
            for (int w = 0; w < NW; ++w)
                a = __dadd_rn(a, sacc[w]);
            t = __dadd_rn(t, a);
        }
    }
    return t;
}

}  // namespace nsli
