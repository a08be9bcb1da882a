// nsli_handover.h -- which words the iterations of one launch hand over in
// (nsli_dense.cu): plain functions, also compiled for the host by the tests.
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

}  // namespace nsli
