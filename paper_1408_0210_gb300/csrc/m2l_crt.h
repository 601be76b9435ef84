// m2l_crt.h -- launcher of the FP64 products on the tensor cores (m2l_crt.cu).
#pragma once
#include "internal.h"

namespace eifmm {

// One level of a product g[I][r] = add[I][r] + sum_J T^{IJ} W[J][r] on FP64
// arrays [box (Morton)][R][rank], `level` the level of the target boxes I.
enum CrtMode {
  kCrtM2L = 0,  // J in the interaction list, 343 operators by offset
  kCrtM2M = 1,  // J the 8 children, 8 operators by octant
  kCrtL2L = 2,  // J the parent, 8 operators by octant
  kCrtBox = 3,  // J = I, one operator (Delta^t at the leaf level)
};
struct CrtJob {
  CrtMode mode;
  int level;
  const CrtImage* img;
  const double* W;
  double* g;
  const double* add;
};
// Words for the largest |W| of the units that share a scale (a level of the M2L
// and its boxes, a box of a tree of this depth elsewhere) and the marks of the
// M2L's second part.
size_t crt_max_words(int depth, int R);
// Scratch for the jobs of one call (M2L jobs run together, others one by one);
// jobs beyond the library's limit run in slabs and columns.
size_t crt_scratch_bytes(int njobs, const CrtJob* jobs, int R);
// Whether the kernel falls off so steeply within an interaction list that the M2L
// of this level stays on the FP32 or FP64 pipes.  The operators of all offsets
// share one scale per row, 60 bits for its largest entry; between the closest
// separated points, a box width w apart, and the farthest, 4 sqrt(3) w, 1/r falls
// to 2^-2.8 and an entry keeps 57 bits, exp(-r^2) at w = 1/2 to 2^-17.  53 bits
// are left down to 2^-7.
bool crt_steep(int kern, double L, int level);
// Whether a job of this image can run in `bytes` of scratch.
bool crt_ready(CrtMode mode, int level, const CrtImage& img, int R, size_t bytes);
// M2L jobs, or one job of another mode, on stream s, in `buf` (buf_bytes from
// crt_scratch_bytes); wmax: crt_max_words(depth, R) words; err: error word of the
// bounded waits.
eifmm_status launch_crt(int njobs, const CrtJob* jobs, int R, void* buf, size_t buf_bytes, unsigned long long* wmax,
                        int nsm, int* err, cudaStream_t s);
// The residue image of an operator stack [nslots][l < dl][m' < d].
eifmm_status build_crt_image(const double* kdT, int nslots, int dl, int d, CrtImage* img, cudaStream_t s);
// The residue image of Delta^t of a level, from Gamma and B in double-double.
// An operator set too ill conditioned for its 104 bits sets img->refused.
eifmm_status build_crt_delta_image(const LevelOps& v, CrtImage* img, cudaStream_t s);
// How much the operators of a level amplify rounding: the largest, over the
// offsets, of max_{m'} sum_l |T_{m'l}| |K(x_l, y)| over max_{m'} |K(y_{m'}, y +
// delta)| for a unit charge at the first node y of the box, whose W is K(x_l, y)
// and whose g is K(y_{m'}, y + delta).
eifmm_status crt_kappa(int kern, const LevelOps& v, double lk, double* kappa, cudaStream_t s);
void free_crt_image(CrtImage* img);

}  // namespace eifmm
