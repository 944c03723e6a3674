// rows_family.cuh -- register-resident row passes for one row length N, for
// plans whose column direction runs the recursive column solve (no column
// kernels are compiled for these lengths; see run_rows_shape). Each
// rows_family_<k>.cu instantiates a few lengths in FP32 and each
// rows_family16_<k>.cu the same lengths in 16 bits, so the library builds in
// parallel; solve_fast.cu lists them.
#pragma once

#include "fast_kernels.cuh"

namespace gfc {

// Row lengths: X(N, R1, R2, F), N = R1 R2 with R2 threads per transform and F
// transforms per block (about 128 threads, within the shared memory of 2 forward
// blocks and 3 inverse blocks per SM, 4 and 4 for N <= 512). Short lengths take
// blocks of about 64 threads with few idle lanes, bands of at most 22 rows (with
// their recursions in registers up to 18, tri_solve_band) that a square image fills
// with little left over; each F is
// the faster of two to four tried, in ps a pixel of a solve: N = 42 F 16 23.8,
// 9 14.6; 56 F 16 14.4, 8 11.6; 72 F 14 11.9, 7 9.2; 90 F 12 9.4, 6 8.2; 112 F 9
// 7.2, 4 7.9. R2 dividing R1 keeps every thread in both stages and won wherever N
// allows it at these sizes: 98 as 14 x 7 against 7 x 14 8.4 -> 6.6, 128 as 16 x 8
// 7.4 -> 5.8, 882 as 42 x 21 6.8 -> 5.8 (adjoint 10.0 -> 8.2), 1200 as 60 x 20 6.8 ->
// 6.35. Images narrower than 23 pixels (N < 32) keep the generic passes.
#define GFC_ROWS_S(X)                                                                                        \
  X(32, 4, 8, 8) X(36, 6, 6, 5) X(40, 5, 8, 6) X(42, 6, 7, 9) X(48, 6, 8, 7) X(50, 5, 10, 11)            \
  X(54, 6, 9, 6) X(56, 7, 8, 8) X(60, 6, 10, 9) X(64, 8, 8, 8)
#define GFC_ROWS_T(X)                                                                                        \
  X(70, 7, 10, 6) X(72, 8, 9, 7) X(80, 8, 10, 6) X(84, 7, 12, 10) X(90, 9, 10, 6) X(96, 8, 12, 8)        \
  X(98, 14, 7, 9)
#define GFC_ROWS_U(X)                                                                                        \
  X(100, 10, 10, 6) X(112, 8, 14, 9) X(120, 10, 12, 10) X(126, 9, 14, 9) X(128, 16, 8, 8)
#define GFC_ROWS_A(X) X(140, 10, 14, 9) X(160, 10, 16, 8) X(180, 12, 15, 8) X(200, 20, 10, 6) X(224, 14, 16, 8)
#define GFC_ROWS_B(X) X(252, 14, 18, 7) X(294, 14, 21, 6) X(320, 16, 20, 6) X(360, 18, 20, 6) X(400, 20, 20, 6)
#define GFC_ROWS_C(X) X(448, 16, 28, 4) X(500, 20, 25, 5) X(560, 20, 28, 4) X(630, 21, 30, 4) X(700, 25, 28, 4)
#define GFC_ROWS_D(X) X(784, 28, 28, 4) X(882, 42, 21, 6) X(980, 28, 35, 3) X(1080, 30, 36, 3)
#define GFC_ROWS_E(X) X(1120, 32, 35, 3) X(1200, 60, 20, 5) X(1372, 28, 49, 4) X(1400, 35, 40, 4)
#define GFC_ROWS_F(X) X(1536, 32, 48, 3) X(1750, 35, 50, 3) X(1960, 40, 49, 2) X(2058, 42, 49, 2)

#define GFC_ROW_SHAPE(N_, R1_, R2_, F_)                                                                          \
  cudaError_t fast_rows_run_##N_(gfc_plan* P, const Bufs& bf, int mode, const void* in0, const void* in1,       \
                                 void* out0, void* out1, int nf, cudaStream_t st, const EditArgs* ed) {         \
    return run_rows_shape<RowShape<N_, R1_, R2_, F_>, float>(P, bf, mode, in0, in1, out0, out1, nf, st, ed);     \
  }                                                                                                             \
  size_t fast_rows_zbuf_##N_(int H) { return fast_zbuf_elems_for<RowShape<N_, R1_, R2_, F_>>(H); }              \
  int fast_rows_items_##N_() { return F_; }

#define GFC_ROW_SHAPE16(N_, R1_, R2_, F_)                                                                        \
  cudaError_t fast_rows_run16_##N_(gfc_plan* P, const Bufs& bf, int mode, const void* in0, const void* in1,     \
                                   void* out0, void* out1, int nf, cudaStream_t st, const EditArgs* ed) {       \
    using RS = RowShape<N_, R1_, R2_, F_>;                                                                      \
    return P->dtype == GFC_F16 ? run_rows_shape<RS, __half>(P, bf, mode, in0, in1, out0, out1, nf, st, ed)       \
                               : run_rows_shape<RS, __nv_bfloat16>(P, bf, mode, in0, in1, out0, out1, nf, st, ed); \
  }

}  // namespace gfc
