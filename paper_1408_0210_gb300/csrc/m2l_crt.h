// m2l_crt.h -- launcher of the FP64 M2L on the tensor cores (m2l_crt.cu).
#pragma once
#include "internal.h"

namespace eifmm {

// Step 4 of one level: g[I][r] = sum_J K^delta W[J][r] on FP64 arrays
// [box (Morton)][R][d].
struct CrtJob {
  int level;
  const CrtImage* img;
  const double* W;
  double* g;
};
// Bytes of scratch the jobs of levels 2..depth use at most (img: per level);
// levels whose planes exceed the library's limit run in slabs and columns.
size_t crt_scratch_bytes(int depth, const CrtImage* const* img, int R);
// All jobs on stream s, in `buf` (buf_bytes from crt_scratch_bytes); wmax:
// [kMaxLevel + 1][R] words; err: error word of the bounded waits.
eifmm_status launch_m2l_crt(int njobs, const CrtJob* jobs, int R, void* buf, size_t buf_bytes,
                            unsigned long long* wmax, int nsm, int* err, cudaStream_t s);
// The residue image of an operator stack kdT ([343][l][m'], d x d).
eifmm_status build_crt_image(const double* kdT, int d, CrtImage* img, cudaStream_t s);
// How much the operators of a level amplify rounding: the largest, over the
// offsets, of max_{m'} sum_l |T_{m'l}| |K(x_l, y)| over max_{m'} |K(y_{m'}, y +
// delta)| for a unit charge at the first node y of the box, whose W is K(x_l, y)
// and whose g is K(y_{m'}, y + delta).
eifmm_status crt_kappa(int kern, const LevelOps& v, double lk, double* kappa, cudaStream_t s);
void free_crt_image(CrtImage* img);

}  // namespace eifmm
