// nsli_handover.h -- which words the iterations of one launch hand over in
// (nsli_dense.cu), when and how many of them, and how row counts are summed over a
// warp: plain functions, also compiled for the host by the tests.
#pragma once

#ifdef __CUDACC__
#define NSLI_HD __host__ __device__
#else
#define NSLI_HD
#endif

namespace nsli {

// The records of a one-launch run alternate between two halves by the parity
// of the iteration.  One half would not do: a CTA writes the column blocks'
// dx^2 and max |dx_j| of step k on its way into hand-over B or after it has
// announced itself there, waiting for nobody, while a slower CTA may still be
// reading those of step k - 1 for the step rule.  With two, the words that
// step k writes were last read in iteration k - 1, and every CTA has left
// that iteration's reads behind when hand-over A of iteration k is through.
NSLI_HD constexpr int stat_half(int k) { return k & 1; }             // the CTAs' counts and maxima of Map k
NSLI_HD constexpr int dx_half_written(int k) { return k & 1; }       // dx of the step of iteration k
NSLI_HD constexpr int dx_half_read(int k) { return (k - 1) & 1; }    // ... as read in iteration k >= 1

// Iterations per launch for a matrix of `bytes` bytes: at most 64 GiB of it are
// read (some 10 ms) unless one iteration reads more, so that other streams get
// their turn and a solve its polls; at most 1024.  (A launch's ring slots, of
// 16 bytes or more and over two blocks or more, then number below 2^32.)
NSLI_HD constexpr int iterations_of(long long bytes)
{
    const long long k = (64ll << 30) / bytes;
    return (int)(k < 1 ? 1 : (k > 1024 ? 1024 : k));
}

// Does the one-launch form serve a system of nblk column blocks on G CTAs?  A
// CTA reduces its own nblk / G blocks, one after another beyond a few, where
// the Reduce kernel has a thread block for each: with few rows of many columns
// that outweighs the launches saved.  Per iteration, one launch against Map
// and Reduce launches, by blocks per CTA: binary32 4.0 8.9 / 13.1 us (64 x
// 8192), 6.7 13.5 / 16.5 (76 x 16384), 8.0 10.4 / 9.6 to 11.5 / 12.5 (4 x 1024,
// 32 x 8192), 10.7 13.9 / 12.2 (24 x 8192), 32 27.4 / 12.3 (8 x 8192); binary64,
// whose chains are longer, 2.6 20.7 / 23.7 us (100 x 8192), 2.7 14.4 / 13.8 (24 x
// 2048), 4.0 18.1 / 16.1 (8 x 1024), 8.0 30.2 / 20.9 (32 x 8192).  bf16 and FP8 as
// binary32.
NSLI_HD constexpr bool one_launch_pays(int nblk, int G, bool f64) { return nblk <= (f64 ? 3 : 7) * G; }

// A count of rows in two parts whose sums over 32 lanes fit 32 bits, so that
// two 32-bit warp reductions add counts of up to 2^53 rows a lane exactly (one
// would wrap where more than 2^31 - 1 rows of a system are violated).
struct CountParts {
    unsigned int lo, hi;
};
NSLI_HD constexpr CountParts count_parts(long long h)
{
    return CountParts{(unsigned int)(h & 0x3ffffff), (unsigned int)(h >> 26)};
}
NSLI_HD constexpr long long count_join(unsigned int lo_sum, unsigned int hi_sum)
{
    return ((long long)hi_sum << 26) + (long long)lo_sum;
}

}  // namespace nsli
