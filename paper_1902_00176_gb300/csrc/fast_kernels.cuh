// fast_kernels.cuh -- register-resident GFC passes for transform lengths with a
// two-stage schedule (Eq. 23, Algorithm B; the same three passes as solve.cu).
// Each supported size pair is instantiated in its own translation unit
// (fast_<M>x<N>.cu) so the library builds in parallel.
//
// Hand-offs between the passes:
//   pass L  (edited solves, some 16-bit Laplacians, or rows too wide to stage) writes
//           the packed rows z[pair][j] = L[2 pair][j] + i L[2 pair+1][j];
//   pass A  stages the gradient rows of an item by bulk copy and forms L itself
//           (or stages z, or the adjoint's grad_out rows), and writes the row
//           spectrum column-major, spec[l][r] (l < N/2+1 Hermitian columns), one
//           2F-row column segment at a time: the transpose is folded into the
//           two-for-one split it does through shared memory anyway;
//   pass B  loads whole columns of spec straight into registers and writes its
//           result row-major, Y[i][l] (image rows i < H; H + 1 for the
//           adjoint), straight from registers, into the buffer that held z;
//   pass C  stages the rows of Y an item needs by bulk copy (the adjoint's
//           inverse row pass likewise) and writes the cropped output.
//
// Row transforms (length N = R1 R2, T = R2 threads per transform, F transforms
// per block): stage 1 is one radix-R1 DFT per thread on x[t + R2 r]; one
// shared-memory exchange; stage 2 has R1 radix-R2 DFTs with the twiddles
// w_N^(r j): R1/R2 per thread when R2 divides R1, else one for each of the
// first R1 threads (R1 < R2). Column transforms (M = R1 R2, R1 <= R2, T = R2 threads
// per column): forward stage 1 radix-R1, exchange, forward stage 2 radix-R2;
// each thread then holds the bins t + R1 s, multiplies them by the Green
// spectrum and runs the inverse's first stage (radix-R2, no twiddles) on the
// same registers; one more exchange and the inverse's radix-R1 stage.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <mutex>
#include <type_traits>

#include "fft_reg.cuh"
#include "gfc_internal.h"
#include "tma.cuh"

namespace gfc {

// The register-resident schedules assume Algorithm A's pad of 4.
constexpr int kP = 4;

// smallest image width that pads to row length N under the SMOOTH policy (pad
// kP): the row kernels skip the crop test for columns below it
constexpr int cx_min_width(int N) {
  int lo = N;
  for (int n = N; n > 2 * kP && cx_row_policy(n) >= N; --n)
    if (cx_row_policy(n) == N) lo = n;
  return lo - 2 * kP;
}

// Column schedule placeholder of a shape compiled for its row length only.
struct NoCols {
  static constexpr int C = 1;
};

struct FastArgs {
  int H, W, p, M, N, Nh, ldM;
  int nrows, ncols;  // support of L (from torus row/col p): H+1, W+1 (gradient) or H, W
  int npairs, ldz;   // packed row pairs of L, and the stride of a packed row (>= N, zero padded)
  int zpairs;        // packed rows per field (npairs rounded up to whole groups, extra rows zero)
  int ngroups;       // row-pair groups per field (pass A) / output row-pair groups (pass C)
  int nparts;        // pass B column blocks per field (u[0,0] partial sums)
  int nf;            // fields in this chunk
  int ldY;           // row stride of the row-major spectrum Y (complex elements)
  int* err;          // the plan's device error word (bounded waits that run out)
  // recursive column solve (row-major spectrum S, bands of 2F rows from torus row p)
  int srows;         // rows of S per field (2 zpairs; rows past the support are zero)
  int G;             // bands per field
  size_t tri_field;  // complex elements per field of the band scratch
  int stage_out;     // inverse row pass: output rows staged in shared memory, stored by bulk copy
  double invM, invN; // 1 / M, 1 / N (FP64 divisions are slow on this part)
  int overlap;       // the kernels after the first may start while the one ahead ends (launch_after)
  int adj;           // the recursive column solve runs the adjoint (half-bands, the sum term at row 0)
  int l2res;         // the chunks' spectrum hand-off fits the L2: evict-first streams, evict-last spectrum,
                     // the inverse row pass drops the spectrum lines it has read
};

// Band scratch of one field (recursive column solve), complex elements:
//   carries [G][2][ldY]: row 0 of band g the causal carry into the band, row 1
//           the anticausal carry from below it (the sweep; read by pass C);
//   sums    [nkb][G][2][32]: the bands' causal and anticausal sums with zero
//           carries (pass A), in tiles of 32 columns, so that a tile is one
//           contiguous copy for the sweep;
//   col0    srows floats: the real parts of column 0 of S (pass A).
// The row-major spectrum S holds 2F rows per band; the sweep writes column 0's
// exact solution into it.
// (The plan sizes this per field in tri_field.)
constexpr int kTriCols = 32;
// Slots of a field's FP64 partial-sum area used by the recursive column solve:
// [0, nkb) the sweep blocks' partials of u[0,0]; kTriCnt a counter of sweep
// blocks done (reset by the row pass, which runs first); kTriU00 u[0,0] itself,
// combined by the last sweep block of the field.
constexpr int kTriCnt = 150, kTriU00 = 151;
__device__ __forceinline__ float2* tri_sums(float2* tri, int field, const FastArgs& A) {
  return tri + (size_t)field * A.tri_field + (size_t)2 * A.G * A.ldY;
}
__device__ __forceinline__ float* tri_col0(float2* tri, int field, const FastArgs& A) {
  const size_t nkb = (size_t)(A.ldY + kTriCols - 1) / kTriCols;
  return reinterpret_cast<float*>(tri_sums(tri, field, A) + nkb * 2 * A.G * kTriCols);
}
// s + v with its rounding error added to err (Knuth's TwoSum, explicitly
// rounded so the compiler cannot reassociate it); returns the rounded sum
__device__ __forceinline__ float two_sum_acc(float s, float v, float& err) {
  const float t = __fadd_rn(s, v);
  const float bp = __fsub_rn(t, s);
  err = __fadd_rn(err, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(v, bp)));
  return t;
}

// one step of y <- x + a y with a = 1 - delta, as (x + y) - delta y: delta is
// held to full relative precision, so the pole near DC is not rounded away
__device__ __forceinline__ float2 tri_step(float2 x, float2 y, float delta) {
  return __ffma2_rn(make_float2(-delta, -delta), y, cadd(x, y));  // packed pair arithmetic
}

// one step of the carry sweep, t <- e + T t with T = 1 - D, the same way: bands of
// a few rows have T next to 1, and its rounding would add up over the bands
__device__ __forceinline__ float2 tri_carry(float2 e, float2 t, float D) { return tri_step(e, t, D); }

__device__ __forceinline__ float f_to_f(float x) { return x; }
__device__ __forceinline__ float f_to_f(__half x) { return __half2float(x); }
__device__ __forceinline__ float f_to_f(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T f_from_f(float x);
template <> __device__ __forceinline__ float f_from_f<float>(float x) { return x; }
template <> __device__ __forceinline__ __half f_from_f<__half>(float x) { return __float2half_rn(x); }
template <> __device__ __forceinline__ __nv_bfloat16 f_from_f<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

template <typename T>
__device__ __forceinline__ float ldz(const T* __restrict__ g, int i, int j, int H, int W) {
  return (i >= 0 && i < H && j >= 0 && j < W) ? f_to_f(g[(size_t)i * W + j]) : 0.0f;
}

template <typename T>
__device__ __forceinline__ float4 ld4(const T* __restrict__ g, int i, int j, int W);
template <>
__device__ __forceinline__ float4 ld4<float>(const float* __restrict__ g, int i, int j, int W) {
  return __ldg(reinterpret_cast<const float4*>(g + (size_t)i * W + j));
}
template <>
__device__ __forceinline__ float4 ld4<__half>(const __half* __restrict__ g, int i, int j, int W) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(g + (size_t)i * W + j));
  const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
  const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}
template <>
__device__ __forceinline__ float4 ld4<__nv_bfloat16>(const __nv_bfloat16* __restrict__ g, int i, int j, int W) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(g + (size_t)i * W + j));
  const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}

template <int N_, int R1_, int R2_, int F_>
struct RowShape {
  static constexpr int N = N_, R1 = R1_, R2 = R2_, F = F_;
  static constexpr int T = R2;                            // threads per transform
  static constexpr int J2 = (R1 >= R2) ? R1 / R2 : 1;     // stage-2 butterflies per thread
  static constexpr int JSPAN = (R1 >= R2) ? R2 : R1;      // stage-2 butterflies j = t + R2 jj, t < JSPAN
  // exchange stride of a thread's R1 stage-1 outputs: odd, so that the threads'
  // 8-byte accesses spread over the banks
  static constexpr int R1P = (R1 % 2 == 0) ? R1 + 1 : R1 + 2;
  static constexpr int NP = (N / R1) * R1P;               // padded transform buffer
  static constexpr int THREADS = ((F * T + 31) / 32) * 32;
  static_assert(R1 % R2 == 0 || R1 < R2, "row schedule needs R2 | R1 or R1 < R2");
  static constexpr int NO = N + 1;        // stage-2 output buffer stride (natural order)
  static constexpr int WMIN = cx_min_width(N);
  static constexpr int LDY_ = ((N / 2 + 1) + 3) & ~3;  // row stride of Y and S (complex)
  static constexpr size_t smem_bytes() { return (size_t)(R1 * R2 + F * NP) * sizeof(float2); }
  static constexpr int CBUF = ((R1 * R2 + F * NP) + 1) & ~1;  // 16-byte aligned offset of the carry rows
  static constexpr size_t smem_bytes_tri_inv() { return (size_t)(CBUF + 2 * LDY_) * sizeof(float2); }
  static constexpr size_t smem_bytes_fwd() { return (size_t)(R1 * R2 + F * NP + F * NO) * sizeof(float2); }
  // blocks per SM the register allocation must allow: long rows fill shared
  // memory at 2 (3 for the inverse pass); short rows leave room for 4. Wider
  // blocks and long stage-2 radices get fewer, so that the transforms keep
  // their values in registers (at least ~200 registers a thread in the forward
  // passes, ~160 in the inverse one; stage-2 radices >= 48 take 2 blocks)
  static constexpr bool SHORT = N <= 512;
  static constexpr int cx_blocks(int cap, int regs) {
    const int b = 65536 / (THREADS * regs);
    return b < 1 ? 1 : (b > cap ? cap : b);
  }
  static constexpr int MINB_FWD = SHORT ? 4 : cx_blocks(2, 200);
  static constexpr int MINB_INV = SHORT ? 4 : cx_blocks(R2 >= 48 ? 2 : 3, 160);
  static constexpr int MINB_ADJ = SHORT ? 4 : cx_blocks(2, 200);
  // the adjoint's column solve writes the transforms' inputs (tri_solve_half)
  // where a block's threads have about a column each: with far fewer columns than
  // threads the work moves from all threads to those that own a column, and with
  // several columns a thread the solve's chains grow. The adjoint in ps a pixel,
  // packed against not: N = 50 18.0 / 15.3, 64 11.1 / 12.1, 72 10.0 / 11.4, 100
  // 8.6 / 9.4, 180 7.2 / 7.7, 270 7.5 / 7.9, 500 6.9 / 7.3, 784 8.1 / 8.1, 1080
  // 9.9 / 9.6, 1568 9.4 / 8.8
  static constexpr bool PACK_ADJ = SHORT && N >= 56;
  // adjoint inverse row pass: twiddles, exchange, the factor table
  // 1 - exp(2 pi i l / N) for l <= N/2, then (16-byte aligned) the F + 1 rows of
  // Y an item needs, LDY complex each
  static constexpr int LDY = LDY_;
  static constexpr size_t adj_stage_offset() {
    return (((size_t)(R1 * R2 + F * NP + (N / 2 + 1)) * sizeof(float2)) + 15) / 16 * 16;
  }
  static constexpr size_t smem_bytes_adj() { return adj_stage_offset() + (size_t)(F + 1) * LDY * sizeof(float2); }
  // the recursive column solve's adjoint also stages the half-band's two carries
  static constexpr size_t smem_bytes_adj_tri() { return adj_stage_offset() + (size_t)(F + 3) * LDY * sizeof(float2); }
  // The exchange stores each run of R1 elements at a stride of R1P (element
  // m = t R1 + s at t R1P + s, conflict-free stage-1 writes); the kernels use
  // the closed forms t R1P + s for m = t R1 + s and j + R1P r for m = j + R1 r.
};

// Shared-memory wavefronts of the column pass's four exchange accesses for a
// per-column stride MP (8-byte elements, thread tid = t C + c, each half-warp
// one request): forward write t R1 + s, forward read t + R1 r (t < R1),
// inverse write t (R2 + 1) + s (t < R1), inverse read t + (R2 + 1) r (t < R2).
constexpr int cols_exchange_wavefronts(int C, int R1, int R2, int threads, int MP) {
  int total = 0;
  for (int h = 0; h < threads / 16; ++h) {
    for (int pat = 0; pat < 4; ++pat) {
      int addr[16] = {}, n = 0;
      for (int L = 0; L < 16; ++L) {
        const int tid = 16 * h + L, c = tid % C, t = tid / C;
        const int tmax = (pat == 1 || pat == 2) ? R1 : R2;
        if (t >= tmax) continue;
        const int stride = pat == 0 ? R1 : (pat == 2 ? R2 + 1 : 1);
        const int a = c * MP + t * stride;
        bool seen = false;
        for (int k = 0; k < n; ++k) seen = seen || addr[k] == a;
        if (!seen) addr[n++] = a;
      }
      int worst = 0;
      for (int b = 0; b < 16; ++b) {
        int cnt = 0;
        for (int k = 0; k < n; ++k) cnt += ((addr[k] % 16) == b) ? 1 : 0;
        worst = cnt > worst ? cnt : worst;
      }
      total += worst;
    }
  }
  return total;
}
// the smallest stride >= lo with the fewest wavefronts among the next 32
constexpr int cols_exchange_stride(int C, int R1, int R2, int threads, int lo) {
  int best = lo, bw = cols_exchange_wavefronts(C, R1, R2, threads, lo);
  for (int mp = lo + 1; mp < lo + 32; ++mp) {
    const int w = cols_exchange_wavefronts(C, R1, R2, threads, mp);
    if (w < bw) { bw = w; best = mp; }
  }
  return best;
}

template <int M_, int R1_, int R2_, int C_>
struct ColShape {
  static constexpr int M = M_, R1 = R1_, R2 = R2_, C = C_;
  static constexpr int T = R2;             // threads per column
  static constexpr int THREADS = ((C * T + 31) / 32) * 32;
  // blocks per SM the registers must allow (short columns leave room for 4)
  static constexpr int MINB = (M <= 512 && THREADS <= 160) ? 4 : ((THREADS <= 256) ? 2 : 1);
  static_assert(R1 <= R2, "column schedule needs R1 <= R2");
  static_assert(C <= 32, "the u[0,0] partial of a block is gathered in one warp");
  // per-column exchange stride: the inverse exchange keeps one spare slot every
  // R2 elements (t (R2 + 1) + s, t + (R2 + 1) r), so it needs M + R1 - 1
  static constexpr int MP = cols_exchange_stride(C, R1, R2, THREADS, M + R1 - 1);
  static constexpr int TWF_STRIDE = (R2 % 2 == 0) ? R2 + 1 : R2;
  static constexpr int TWI_STRIDE = (R1 % 2 == 0) ? R1 + 1 : R1;
  static constexpr int GS = ((M + 3) / 4) * 4;  // floats per staged Green column (16-byte multiple)
  static constexpr size_t smem_bytes() {
    return (size_t)C * GS * sizeof(float) + (size_t)(R1 * TWF_STRIDE + R2 * TWI_STRIDE + C * MP) * sizeof(float2);
  }
};

// ---------------------------------------------------------------------------
// pass L: divergence (Eq. 3) or copy of the given Laplacian, packed two rows per
// complex value: z[pair][j] = L[2 pair][j] + i L[2 pair + 1][j], j < ncols
// (image columns; the pad is implicit). Streams gx, gy once.
// ---------------------------------------------------------------------------
template <typename T, int MODE>
__global__ void __launch_bounds__(512) k_fast_div(const T* __restrict__ in0, const T* __restrict__ in1,
                                                  float2* __restrict__ z, float* __restrict__ partial, FastArgs A) {
  // grid: x = groups of 4 padded columns, y = packed rows (zpairs), z = fields.
  // Packed row `pair`, padded column c holds L[2 pair][c - p] + i L[2 pair + 1][c - p],
  // zero outside the support, so the row pass can load it without range checks.
  // MODE 2 (adjoint) packs grad_out like a Laplacian and also sums it: one
  // block covers a whole packed row and writes that row pair's FP64 sum.
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  const int pair = blockIdx.y, field = blockIdx.z;
  const bool inq = q < A.ldz / 4;
  if (MODE != 2 && !inq) return;
  const int c0 = 4 * q, j0 = c0 - kP;
  float la[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lb[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (inq && pair < A.npairs && j0 + 3 >= 0 && j0 < A.ncols) {
    const bool vec4 = (A.W % 4) == 0 && j0 >= 0;
    const size_t fe = (size_t)A.H * A.W;
    const T* a = in0 + field * fe;
    const T* b = (MODE == 0) ? in1 + field * fe : nullptr;
    const int ia = 2 * pair, ib = ia + 1;
    if (MODE == 0) {
      float xa[5], xb[5], ya[4], yb[4], ym[4];  // gx rows ia, ib at j0-1..j0+3; gy rows ia, ib, ia-1
      const bool ina = ia < A.H, inb = ib < A.H, inm = ia >= 1 && ia - 1 < A.H;
      if (vec4 && j0 + 3 < A.W) {
        const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const float4 ga = ina ? ld4(a, ia, j0, A.W) : z4, gb = inb ? ld4(a, ib, j0, A.W) : z4;
        const float4 ha = ina ? ld4(b, ia, j0, A.W) : z4, hb = inb ? ld4(b, ib, j0, A.W) : z4;
        const float4 hm = inm ? ld4(b, ia - 1, j0, A.W) : z4;
        xa[1] = ga.x; xa[2] = ga.y; xa[3] = ga.z; xa[4] = ga.w;
        xb[1] = gb.x; xb[2] = gb.y; xb[3] = gb.z; xb[4] = gb.w;
        ya[0] = ha.x; ya[1] = ha.y; ya[2] = ha.z; ya[3] = ha.w;
        yb[0] = hb.x; yb[1] = hb.y; yb[2] = hb.z; yb[3] = hb.w;
        ym[0] = hm.x; ym[1] = hm.y; ym[2] = hm.z; ym[3] = hm.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          xa[e + 1] = ldz(a, ia, j0 + e, A.H, A.W);
          xb[e + 1] = ldz(a, ib, j0 + e, A.H, A.W);
          ya[e] = ldz(b, ia, j0 + e, A.H, A.W);
          yb[e] = ldz(b, ib, j0 + e, A.H, A.W);
          ym[e] = ldz(b, ia - 1, j0 + e, A.H, A.W);
        }
      }
      xa[0] = ldz(a, ia, j0 - 1, A.H, A.W);
      xb[0] = ldz(a, ib, j0 - 1, A.H, A.W);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        la[e] = (xa[e + 1] - xa[e]) + (ya[e] - ym[e]);
        lb[e] = (xb[e + 1] - xb[e]) + (yb[e] - ya[e]);
      }
    } else {
      if (vec4 && j0 + 3 < A.W) {
        const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const float4 ga = ia < A.H ? ld4(a, ia, j0, A.W) : z4, gb = ib < A.H ? ld4(a, ib, j0, A.W) : z4;
        la[0] = ga.x; la[1] = ga.y; la[2] = ga.z; la[3] = ga.w;
        lb[0] = gb.x; lb[1] = gb.y; lb[2] = gb.z; lb[3] = gb.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          la[e] = ldz(a, ia, j0 + e, A.H, A.W);
          lb[e] = ldz(a, ib, j0 + e, A.H, A.W);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const bool inj = j0 + e >= 0 && j0 + e < A.ncols;
      la[e] = (inj && ia < A.nrows) ? la[e] : 0.0f;
      lb[e] = (inj && ib < A.nrows) ? lb[e] : 0.0f;
    }
  }
  if (inq) {
    float4* dst = reinterpret_cast<float4*>(z + ((size_t)field * A.zpairs + pair) * A.ldz + c0);
    dst[0] = make_float4(la[0], lb[0], la[1], lb[1]);
    dst[1] = make_float4(la[2], lb[2], la[3], lb[3]);
  }
  if (MODE == 2) {
    // a thread's 8 values summed in FP32 (error a few ulp of their magnitudes),
    // the block's in FP64: FP64 arithmetic is scarce on this GPU
    const float s8 = ((la[0] + la[1]) + (la[2] + la[3])) + ((lb[0] + lb[1]) + (lb[2] + lb[3]));
    double v = (double)s8;
    __shared__ double red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
      reinterpret_cast<double*>(partial)[(size_t)field * (kMaxRowBlocks / 2) + pair] = t;
    }
  }
}

// Pass L with a gradient edit applied as the gradient is loaded (Sec. 3.2.3
// thresholding, Eq. 26 merging): the same packed rows as k_fast_div<T, 0> on
// the edited field, bit for bit, without the edited field ever being stored.
// Every edited pixel is computed once: a thread owns 4 columns and walks down
// kEditPairs row pairs, keeping the edited gy of the row above in registers;
// the edited gx of the column to its left comes from the neighbouring lane
// (lane 0 edits that one pixel itself).
constexpr int kEditPairs = 8;

template <typename T, int EDIT>
__device__ __forceinline__ void edit_row4(const T* __restrict__ a, const T* __restrict__ b,
                                          const T* __restrict__ e, int i, int j0, const FastArgs& A, float t2,
                                          float alpha, float* ex, float* ey) {
  if (i < 0 || i >= A.H || j0 + 3 < 0 || j0 >= A.W) {
#pragma unroll
    for (int k = 0; k < 4; ++k) ex[k] = ey[k] = 0.0f;
    return;
  }
  if ((A.W % 4) == 0 && j0 >= 0 && j0 + 3 < A.W) {
    const float4 x = ld4(a, i, j0, A.W), y = ld4(b, i, j0, A.W);
    float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w}, cs[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (EDIT == kEditMerge) {
      const float4 c = ld4(e, i, j0, A.W);
      cs[0] = c.x; cs[1] = c.y; cs[2] = c.z; cs[3] = c.w;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (EDIT == kEditThreshold) {
        const bool drop = edit_mag2(xs[k], ys[k]) < t2;
        ex[k] = drop ? 0.0f : xs[k];
        ey[k] = drop ? 0.0f : ys[k];
      } else {
        const float sc = edit_merge_scale(xs[k], ys[k], cs[k], alpha);
        ex[k] = edit_round(__fmul_rn(xs[k], sc), a);
        ey[k] = edit_round(__fmul_rn(ys[k], sc), a);
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 v = edit_pixel<T, EDIT>(a, b, e, i, j0 + k, A.H, A.W, t2, alpha);
      ex[k] = v.x;
      ey[k] = v.y;
    }
  }
}

template <typename T, int EDIT>
__global__ void __launch_bounds__(512) k_fast_div_edit(const T* __restrict__ gx, const T* __restrict__ gy,
                                                       const T* __restrict__ edges, const float* __restrict__ t2s,
                                                       float alpha, float2* __restrict__ z, FastArgs A) {
  // grid: x = groups of 4 padded columns (whole warps), y = blocks of kEditPairs
  // packed rows, z = fields. Every lane stays to the end (warp shuffles).
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  const int field = blockIdx.z, lane = threadIdx.x & 31;
  const bool inq = q < A.ldz / 4;
  const int c0 = 4 * q, j0 = c0 - kP;
  const size_t fe = (size_t)A.H * A.W;
  const T* a = gx + field * fe;
  const T* b = gy + field * fe;
  const T* e = (EDIT == kEditMerge) ? edges + field * fe : nullptr;
  const float t2 = (EDIT == kEditThreshold) ? t2s[field] : 0.0f;
  const int p0 = blockIdx.y * kEditPairs;
  const int p1 = min(p0 + kEditPairs, A.zpairs);
  // edited gy of the row above the first row of the block
  float ym[4], scratch[4];
  edit_row4<T, EDIT>(a, b, e, 2 * p0 - 1, j0, A, t2, alpha, scratch, ym);
  for (int pair = p0; pair < p1; ++pair) {
    float L[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = 2 * pair + h;
      float ex[4], ey[4];
      edit_row4<T, EDIT>(a, b, e, i, j0, A, t2, alpha, ex, ey);
      float left = __shfl_up_sync(0xffffffffu, ex[3], 1);
      if (lane == 0) left = edit_pixel<T, EDIT>(a, b, e, i, j0 - 1, A.H, A.W, t2, alpha).x;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float xl = (k == 0) ? left : ex[k - 1];
        const bool in = j0 + k >= 0 && j0 + k < A.ncols && i < A.nrows && pair < A.npairs;
        L[h][k] = in ? (ex[k] - xl) + (ey[k] - ym[k]) : 0.0f;
        ym[k] = ey[k];
      }
    }
    if (inq) {
      float4* dst = reinterpret_cast<float4*>(z + ((size_t)field * A.zpairs + pair) * A.ldz + c0);
      dst[0] = make_float4(L[0][0], L[1][0], L[0][1], L[1][1]);
      dst[1] = make_float4(L[0][2], L[1][2], L[0][3], L[1][3]);
    }
  }
}

// ---------------------------------------------------------------------------
// Recursive column solve, pass A side: the item's 2F rows of the spectrum, from
// the F packed transforms in buf2 (two-for-one split), stored row-major
// (S[row][l], row = image-relative torus row), and per column l the item's
// band sums with zero carries,
//   e  = sum_r a^(nb-1-r) X[r]   (causal recursion y = X + a y run down the band)
//   e' = sum_r a^r X[r]          (anticausal recursion run up the band),
// over the nb band rows that lie on the torus. Thread t takes columns t, t +
// blockDim, ...: the row stores and sums are coalesced across threads.
// ---------------------------------------------------------------------------
// HALF (the adjoint): the sums are taken per half-band of F rows (half-bands
// 2g and 2g + 1; A.G counts half-bands), so that the inverse pass can solve F
// rows at a time.
template <class S, bool HALF = false>
__device__ __forceinline__ void tri_store_item(const float2* buf2, float2* __restrict__ spec, float2* __restrict__ tri,
                                               const float* __restrict__ cc, int field, int g, const FastArgs& A) {
  constexpr int RW = 2 * S::F;
  float2* Sr = spec + ((size_t)field * A.srows + (size_t)g * RW) * A.ldY;
  float2* sums = tri_sums(tri, field, A);
  const int nb = min(RW, A.M - A.p - g * RW);
  for (int k = threadIdx.x; k < A.Nh; k += blockDim.x) {
    float2* te = sums + ((size_t)(k / kTriCols) * A.G + g) * 2 * kTriCols + (k % kTriCols);  // tile of column k
    float2* tp = te + kTriCols;
    const int km = k == 0 ? 0 : S::N - k;
    float2 x[RW];
#pragma unroll
    for (int q = 0; q < S::F; ++q) {
      // X_a = (Z[k] + conj Z[N-k]) / 2, X_b = -i (Z[k] - conj Z[N-k]) / 2, in packed pair arithmetic
      const float2 zk = buf2[q * S::NO + k], zm = buf2[q * S::NO + km];
      const float2 zc = make_float2(zm.x, -zm.y);
      x[2 * q] = cscale(cadd(zk, zc), 0.5f);
      const float2 d = csub(zk, zc);
      x[2 * q + 1] = cscale(make_float2(d.y, -d.x), 0.5f);
    }
    if (!HALF && A.l2res) {  // the inverse row pass reads these rows next: last out of the L2
      const uint64_t pol = l2_policy_evict_last();
#pragma unroll
      for (int r = 0; r < RW; ++r) st_global_hint(Sr + (size_t)r * A.ldY + k, x[r], pol);
    } else {
#pragma unroll
      for (int r = 0; r < RW; ++r) Sr[(size_t)r * A.ldY + k] = x[r];
    }
    if (k == 0) {
      float* c0 = tri_col0(tri, field, A) + (size_t)g * RW;
#pragma unroll
      for (int r = 0; r < RW; ++r) c0[r] = x[r].x;
    }
    const float dl = __ldg(cc + (size_t)k * 8);
    if constexpr (HALF) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h * S::F >= nb) break;  // the second half lies past the torus
        float2 e = make_float2(0.0f, 0.0f), ep = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int r = h * S::F; r < (h + 1) * S::F; ++r)
          if (r < nb) e = tri_step(x[r], e, dl);
#pragma unroll
        for (int r = (h + 1) * S::F - 1; r >= h * S::F; --r)
          if (r < nb) ep = tri_step(x[r], ep, dl);
        float2* th = sums + ((size_t)(k / kTriCols) * A.G + 2 * g + h) * 2 * kTriCols + (k % kTriCols);
        th[0] = e;
        th[kTriCols] = ep;
      }
    } else {
      float2 e = make_float2(0.0f, 0.0f), ep = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int r = 0; r < RW; ++r)
        if (r < nb) e = tri_step(x[r], e, dl);
#pragma unroll
      for (int r = RW - 1; r >= 0; --r)
        if (r < nb) ep = tri_step(x[r], ep, dl);
      *te = e;
      *tp = ep;
    }
  }
}

// ---------------------------------------------------------------------------
// pass A: forward row transforms of the packed rows + two-for-one split +
// transposed store. Persistent over (field, group of F row pairs). The F packed
// rows of an item are one contiguous bulk copy into the exchange buffer,
// completed on an mbarrier; the copy for the next item is issued as soon as
// this item's stage-2 inputs are read, so it overlaps the stage-2 transforms
// and the transposed store of the spectrum.
// ---------------------------------------------------------------------------
template <class S, bool TRI>
__global__ void __launch_bounds__(S::THREADS, S::MINB_FWD) k_fast_rows_fwd(const float2* __restrict__ z,
                                                                 float2* __restrict__ spec,
                                                                 const float2* __restrict__ twg, FastArgs A,
                                                                 float2* __restrict__ tri,
                                                                 const float* __restrict__ cc,
                                                                 float* __restrict__ partial = nullptr) {
  extern __shared__ __align__(16) float2 sm[];
  float2* tw2 = sm;                   // [R1][R2]: w_N^(r j)
  float2* buf = sm + S::R1 * S::R2;   // staged packed rows [F][ldz], then the exchange (m -> m + m / R1)
  float2* buf2 = buf + S::F * S::NP;  // [F][NO] stage-2 output, natural order
  __shared__ __align__(8) uint64_t bar;
  const int tid = threadIdx.x;
  const int f = tid / S::T, t = tid - f * S::T;
  const bool act = f < S::F;
  for (int i = tid; i < S::R1 * S::R2; i += blockDim.x) {
    const int j = i / S::R2, r = i - j * S::R2;
    tw2[i] = twg[r * j];
  }
  float2* mybuf = buf + (act ? f : 0) * S::NP;
  float2* mybuf2 = buf2 + (act ? f : 0) * S::NO;
  // unpack mapping: thread (uf, uk0) takes the bins k = uk0 + T s of transform uf
  const int uf = tid % S::F, uk0 = tid / S::F;
  const bool uact = tid < S::F * S::T;
  const int items = A.nf * A.ngroups;
  // one thread: stage the packed rows of item w (zero padded, whole rows);
  // prefetch: only start fetching them into L2, for the copy one item later
  auto issue = [&](int w, bool prefetch) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    const float2* zs = z + ((size_t)field * A.zpairs + (size_t)g * S::F) * A.ldz;
    const unsigned nb = (unsigned)(S::F * A.ldz * sizeof(float2));
    if (prefetch)
      l2_prefetch(zs, nb);
    else
      bulk_load(buf, zs, nb, &bar);
  };
  if (tid == 0) mbar_init(&bar, 1);
  __syncthreads();
  if (tid == 0 && (int)blockIdx.x < items) issue(blockIdx.x, false);
  if (tid == 0 && (int)(blockIdx.x + gridDim.x) < items) issue(blockIdx.x + gridDim.x, true);
  unsigned phase = 0;
#pragma unroll 1
  for (int w = blockIdx.x; w < items; w += gridDim.x, phase ^= 1u) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    if (TRI && w + (int)gridDim.x >= items) dependents_may_start();  // the block's last item
    if (TRI && g == 0 && tid == 0)  // the sweep's count of finished blocks for this field starts at 0
      reinterpret_cast<unsigned*>(reinterpret_cast<double*>(partial) + (size_t)field * (kMaxRowBlocks / 2) + kTriCnt)[0] = 0u;
    const bool landed = mbar_wait(&bar, phase);
    if (__syncthreads_or(!landed)) {  // the copy never completed: report, let it drain, stop
      if (tid == 0) atomicExch(A.err, kErrBulkWait);
      mbar_wait(&bar, phase);
      return;
    }
    float2 v[S::R1];
    if (act) {
      const float2* zr = buf + (size_t)f * A.ldz + t;
#pragma unroll
      for (int r = 0; r < S::R1; ++r) v[r] = zr[S::R2 * r];
    }
    __syncthreads();  // every staged row read: buf becomes the exchange buffer
    if (act) {
      dft_reg<S::R1, -1>(v);
      // Stockham stage 1 writes t R1 + s; its padded index is t R1P + s
#pragma unroll
      for (int s2 = 0; s2 < S::R1; ++s2) mybuf[t * S::R1P + s2] = v[s2];
    }
    __syncthreads();  // stage-1 results visible; previous unpack done with buf2
    const bool act2 = act && t < S::JSPAN;
#pragma unroll
    for (int jj = 0; jj < S::J2; ++jj) {
      const int j = t + S::R2 * jj;  // j < R1, so the padded index of j + R1 r is j + R1P r
      float2 u[S::R2];
      if (act2) {
        u[0] = mybuf[j];
#pragma unroll
        for (int r = 1; r < S::R2; ++r) u[r] = cmul(mybuf[j + S::R1P * r], tw2[j * S::R2 + r]);
      }
      if (jj == S::J2 - 1) {
        fence_proxy_async_smem();  // this thread's accesses of buf precede the next bulk copy into it
        __syncthreads();           // buf free
        if (tid == 0 && w + (int)gridDim.x < items) issue(w + gridDim.x, false);
        if (tid == 0 && w + 2 * (int)gridDim.x < items) issue(w + 2 * gridDim.x, true);
      }
      if (act2) {
        dft_reg<S::R2, -1>(u);
#pragma unroll
        for (int s2 = 0; s2 < S::R2; ++s2) mybuf2[j + S::R1 * s2] = u[s2];
      }
    }
    __syncthreads();  // stage-2 results visible
    if constexpr (TRI) {
      tri_store_item<S>(buf2, spec, tri, cc, field, g, A);
      continue;
    }
    if (g == 0) {
      // rows of every column outside the support [p, p + nrows) are zero, so the
      // column pass loads whole columns without range checks
      float2* Sz = spec + (size_t)field * A.Nh * A.ldM;
      const int nz = A.M - A.nrows;
      for (int idx = tid; idx < A.Nh * nz; idx += blockDim.x) {
        const int k = idx / nz, q = idx - k * nz;
        Sz[(size_t)k * A.ldM + (q < kP ? q : q + A.nrows)] = make_float2(0.0f, 0.0f);
      }
    }
    // X_a[k] = (Z[k] + conj Z[N-k]) / 2, X_b[k] = -i (Z[k] - conj Z[N-k]) / 2, stored at spec[k][p + row]
    const int ra = g * 2 * S::F + 2 * uf;
    if (uact && ra < A.nrows) {
      float2* Sp = spec + (size_t)field * A.Nh * A.ldM + A.p + ra;
      const float2* zb = buf2 + uf * S::NO;
      const bool two = ra + 1 < A.nrows, vec = ((A.p + ra) & 1) == 0;
      for (int k = uk0; k < A.Nh; k += S::T) {
        const float2 zk = zb[k], zm = zb[k == 0 ? 0 : S::N - k];
        const float2 xa = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
        const float2 xb = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
        float2* dst = Sp + (size_t)k * A.ldM;
        if (two && vec) {
          *reinterpret_cast<float4*>(dst) = make_float4(xa.x, xa.y, xb.x, xb.y);
        } else {
          dst[0] = xa;
          if (two) dst[1] = xb;
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// pass L folded into pass A: the input rows an item needs arrive by bulk copy in
// the exchange buffers and each thread forms its packed values
// L[2 pair][j] + i L[2 pair + 1][j] from shared memory with the same arithmetic
// as pass L, so the packed rows never go through HBM. IN = kInGrad: 2F gx rows
// and 2F + 1 gy rows (gy from the row above the item's first pair), Eq. 3;
// kInLap: 2F rows of a given Laplacian; kInAdj: the adjoint's first step,
// z = Crop^T(grad_out) from 2F rows of grad_out, with each row pair's FP64 sum
// written where pass B reads it for the -(sum grad_out) e_00 term (as
// k_fast_div<T, 2>). The rest is k_fast_rows_fwd. The next item's rows are
// requested once this item's spectrum is stored (the staging area spans both
// exchange buffers).
// The rows of an item are one contiguous run of global memory, so rows of any
// length are staged: the copy starts at the 16-byte boundary at or below the
// first element and ends at the one at or above the last, and the row pointers
// start at the remainder. Only a run that ends at the end of the whole input
// stops at the boundary below, and its last elements (fewer than 16 bytes) are
// loaded one by one.
// ---------------------------------------------------------------------------
enum FwdIn { kInGrad = 0, kInLap = 1, kInAdj = 2 };

// shared memory of one staged run of n elements: at most 15 bytes of another
// run in front, whole 16-byte units
template <typename T>
__host__ __device__ constexpr size_t run_bytes(size_t n) {
  return (n * sizeof(T) + 15 + 15) / 16 * 16;
}
// the item's input rows as staged: gradient 2F gx rows, then 2F + 1 gy rows;
// Laplacian and adjoint 2F rows
template <class S, typename T>
__host__ __device__ constexpr size_t fused_stage_bytes(int W, int in = kInGrad) {
  return run_bytes<T>((size_t)2 * S::F * W) + (in == kInGrad ? run_bytes<T>((size_t)(2 * S::F + 1) * W) : 0);
}
template <class S>
__host__ __device__ constexpr size_t fused_exchange_bytes() {
  return (size_t)(S::F * S::NP + S::F * S::NO) * sizeof(float2);
}

// a run of n > 0 elements at src of an input that ends at `end`, as it is copied
template <typename T>
struct Run {
  const char* from;  // 16-byte aligned, at or below src
  unsigned bytes;    // whole 16-byte units copied
  int lead;          // elements between `from` and src
  int tail;          // last elements of the run that the copy does not reach
  __device__ __forceinline__ Run(const T* src, unsigned n, const T* end) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(src), e = a + (uintptr_t)n * sizeof(T), b = a & ~(uintptr_t)15;
    uintptr_t stop = (e + 15) & ~(uintptr_t)15;
    if (stop > reinterpret_cast<uintptr_t>(end)) stop = e & ~(uintptr_t)15;
    from = reinterpret_cast<const char*>(b);
    bytes = stop > b ? (unsigned)(stop - b) : 0u;
    lead = (int)((a - b) / sizeof(T));
    tail = e > stop ? (int)((e - (stop > a ? stop : a)) / sizeof(T)) : 0;
  }
};

// Store n contiguous elements from shared memory to dst, by one warp: the
// 16-byte units of dst that the run covers by bulk copy, the elements before
// and after them one by one. src is at dst's remainder from a 16-byte boundary.
// The caller's lane 0 waits for the copy; the lanes' reads of shared memory are
// ordered before later asynchronous writes to it.
template <typename T>
__device__ __forceinline__ void store_run(T* dst, const T* src, unsigned n, int lane) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(dst), e = a + (uintptr_t)n * sizeof(T);
  uintptr_t b = (a + 15) & ~(uintptr_t)15, stop = e & ~(uintptr_t)15;
  if (stop < b) b = stop = e;  // no whole unit
  const unsigned head = (unsigned)((b - a) / sizeof(T)), last = (unsigned)((stop - a) / sizeof(T));
  if (lane == 0 && stop > b) bulk_store(dst + head, src + head, (unsigned)(stop - b));
  if (lane < (int)head) dst[lane] = src[lane];
  if (lane < (int)(n - last)) dst[last + lane] = src[last + lane];
  fence_proxy_async_smem();
  __syncwarp();
}

// EDIT = kEditThreshold (Sec. 3.2.3) zeroes, in the staged rows, every pixel whose
// gradient magnitude is below the field's threshold (t2s: squared thresholds of
// the chunk's fields), with the keep/drop decision of the standalone threshold
// kernel, before the divergence is formed; the gy row above the item takes its
// decision from gx of that row, read from global memory ahead of the staging.
template <class S, typename T, int IN, bool TRI, int EDIT = kEditNone>
__global__ void __launch_bounds__(S::THREADS, S::MINB_FWD) k_fast_rows_fwd_div(const T* __restrict__ gx,
                                                                     const T* __restrict__ gy,
                                                                     float2* __restrict__ spec,
                                                                     const float2* __restrict__ twg,
                                                                     float* __restrict__ partial, FastArgs A,
                                                                     float2* __restrict__ tri,
                                                                     const float* __restrict__ cc,
                                                                     const float* __restrict__ t2s = nullptr) {
  constexpr bool ADJ = IN == kInAdj;
  static_assert(EDIT == kEditNone || (EDIT == kEditThreshold && IN == kInGrad), "only the threshold edit is staged");
  extern __shared__ __align__(16) float2 sm[];
  float2* tw2 = sm;
  float2* buf = sm + S::R1 * S::R2;
  float2* buf2 = buf + S::F * S::NP;
  constexpr int RW = 2 * S::F;  // image rows per item
  static_assert((S::R1 * S::R2) % 2 == 0, "the staging area is 16-byte aligned");
  // gx rows (else the only input's rows) r0 .. r0 + RW - 1; gy rows from the one above
  T* const stx = reinterpret_cast<T*>(buf);
  T* const sty = reinterpret_cast<T*>(reinterpret_cast<char*>(buf) + run_bytes<T>((size_t)RW * A.W));
  __shared__ __align__(8) uint64_t bar;
  __shared__ float2 red[ADJ ? S::F * S::T : 1];  // ADJ: per-thread compensated sums (sum, error) of the row pairs
  const int tid = threadIdx.x;
  const int f = tid / S::T, t = tid - f * S::T;
  const bool act = f < S::F;
  for (int i = tid; i < S::R1 * S::R2; i += blockDim.x) {
    const int j = i / S::R2, r = i - j * S::R2;
    tw2[i] = twg[r * j];
  }
  float2* mybuf = buf + (act ? f : 0) * S::NP;
  float2* mybuf2 = buf2 + (act ? f : 0) * S::NO;
  const int uf = tid % S::F, uk0 = tid / S::F;
  const bool uact = tid < S::F * S::T;
  const int items = A.nf * A.ngroups;
  const size_t fe = (size_t)A.H * A.W;
  const T* const xend = gx + (size_t)A.nf * fe;
  // rows of whole 16-byte units start every run at a boundary (so do the fields)
  const bool whole = (A.W * sizeof(T)) % 16 == 0;
  const T* const yend = IN == kInGrad ? gy + (size_t)A.nf * fe : nullptr;
  // the runs of item w: rows r0 .. r0 + nx - 1 of gx (nx may be 0), rows y0 .. y1 - 1 of gy
  auto rows_x = [&](int r0) { return (A.H - r0) < RW ? (A.H - r0) : RW; };
  auto run_x = [&](int field, int r0, int nx) { return Run<T>(gx + field * fe + (size_t)r0 * A.W, (unsigned)(nx * A.W), xend); };
  auto run_y = [&](int field, int r0) {
    const int y0 = r0 > 0 ? r0 - 1 : 0, y1 = (A.H < r0 + RW) ? A.H : r0 + RW;
    return Run<T>(gy + field * fe + (size_t)y0 * A.W, (unsigned)((y1 - y0) * A.W), yend);
  };
  // one thread: stage the input rows of item w (prefetch: only start fetching
  // the same rows into L2, for the copy one item later)
  auto issue = [&](int w, bool prefetch) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    const int r0 = g * RW, nx = rows_x(r0);  // (with the recursive column solve the last band may hold no row)
    const char* xs = nullptr;
    const char* ys = nullptr;
    unsigned xb = 0, yb = 0;
    if (nx > 0) {
      const Run<T> q = run_x(field, r0, nx);
      xs = q.from;
      xb = q.bytes;
    }
    if constexpr (IN == kInGrad) {
      const Run<T> q = run_y(field, r0);
      ys = q.from;
      yb = q.bytes;
    }
    if (prefetch) {
      if (xb) l2_prefetch(xs, xb);
      if (yb) l2_prefetch(ys, yb);
      return;
    }
    mbar_expect_tx(&bar, xb + yb);
    if (IN != kInAdj && A.l2res) {  // read once: first out of the L2, so that the spectrum stays
      const uint64_t pol = l2_policy_evict_first();
      if (xb) bulk_copy_hint(stx, xs, xb, &bar, pol);
      if (yb) bulk_copy_hint(sty, ys, yb, &bar, pol);
    } else {
      if (xb) bulk_copy(stx, xs, xb, &bar);
      if (yb) bulk_copy(sty, ys, yb, &bar);
    }
  };
  if (tid == 0) mbar_init(&bar, 1);
  __syncthreads();
  if (tid == 0 && (int)blockIdx.x < items) issue(blockIdx.x, false);
  if (tid == 0 && (int)(blockIdx.x + gridDim.x) < items) issue(blockIdx.x + gridDim.x, true);
  unsigned phase = 0;
  constexpr int kEdW = (S::N + S::THREADS - 1) / S::THREADS;  // gx values of the row above, per thread
#pragma unroll 1
  for (int w = blockIdx.x; w < items; w += gridDim.x, phase ^= 1u) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    if (TRI && !ADJ && w + (int)gridDim.x >= items) dependents_may_start();  // the block's last item
    if (TRI && !ADJ && g == 0 && tid == 0)  // the sweep's count of finished blocks for this field starts at 0
      reinterpret_cast<unsigned*>(reinterpret_cast<double*>(partial) + (size_t)field * (kMaxRowBlocks / 2) + kTriCnt)[0] = 0u;
    float gxa[EDIT == kEditThreshold ? kEdW : 1];
    if constexpr (EDIT == kEditThreshold) {
      const int r0 = g * RW;
      const T* src = gx + field * fe + (size_t)(r0 > 0 ? r0 - 1 : 0) * A.W;
#pragma unroll
      for (int q = 0; q < kEdW; ++q) {
        const int j = tid + q * S::THREADS;
        gxa[q] = (r0 > 0 && j < A.W) ? f_to_f(src[j]) : 0.0f;
      }
    }
    const bool landed = mbar_wait(&bar, phase);
    if (__syncthreads_or(!landed)) {  // the copies never completed: report, let them drain, stop
      if (tid == 0) atomicExch(A.err, kErrBulkWait);
      mbar_wait(&bar, phase);
      return;
    }
    // the staged rows: sgx row i is image row r0 + i, sgy row i image row r0 - 1 + i
    T* sgx = stx;
    T* sgy = sty - (IN == kInGrad && g == 0 ? A.W : 0);  // (there is no row -1; it is not read)
    if (!whole) {
      const int r0 = g * RW, nx = rows_x(r0);
      int xt = 0, yt = 0;
      if (nx > 0) {
        const Run<T> q = run_x(field, r0, nx);
        sgx += q.lead;
        xt = q.tail;
        if (tid < xt) sgx[nx * A.W - xt + tid] = gx[field * fe + (size_t)(r0 + nx) * A.W - xt + tid];
      }
      if constexpr (IN == kInGrad) {
        const Run<T> q = run_y(field, r0);
        const int y0 = r0 > 0 ? r0 - 1 : 0, y1 = (A.H < r0 + RW) ? A.H : r0 + RW;
        yt = q.tail;
        if (tid < yt) sty[q.lead + (y1 - y0) * A.W - yt + tid] = gy[field * fe + (size_t)y1 * A.W - yt + tid];
        sgy += q.lead;
      }
      if (xt + yt > 0) __syncthreads();  // the input's last elements are in place
    }
    if constexpr (EDIT == kEditThreshold) {
      const float t2 = t2s[field];
      const int r0 = g * RW, nx = (A.H - r0) < RW ? (A.H - r0) : RW;
      const T zero = f_from_f<T>(0.0f);
      // staged pixels (r0 + i, j): gx in sgx row i, gy in sgy row i + 1; 16 bytes (VE
      // pixels) at a time where rows are 16-byte multiples
      constexpr int VE = 16 / (int)sizeof(T);
      const int wv = A.W / VE;
      if (A.W % VE != 0) {  // rows at odd remainders: one pixel at a time
        for (int idx = tid; idx < nx * A.W; idx += S::THREADS) {
          T* yp = sgy + A.W + idx;
          if (edit_mag2(f_to_f(sgx[idx]), f_to_f(*yp)) < t2) sgx[idx] = *yp = zero;
        }
      } else {
      for (int idx = tid; idx < nx * wv; idx += S::THREADS) {
        const int i = idx / wv, jv = idx - i * wv;
        uint4* xp = reinterpret_cast<uint4*>(sgx + (size_t)i * A.W) + jv;
        uint4* yp = reinterpret_cast<uint4*>(sgy + (size_t)(i + 1) * A.W) + jv;
        uint4 xv = *xp, yv = *yp;
        T* xe = reinterpret_cast<T*>(&xv);
        T* ye = reinterpret_cast<T*>(&yv);
        bool any = false;
#pragma unroll
        for (int e2 = 0; e2 < VE; ++e2)
          if (edit_mag2(f_to_f(xe[e2]), f_to_f(ye[e2])) < t2) {
            xe[e2] = zero;
            ye[e2] = zero;
            any = true;
          }
        if (any) {
          *xp = xv;
          *yp = yv;
        }
      }
      }
      if (r0 > 0) {  // gy of the row above (sgy row 0)
#pragma unroll
        for (int q = 0; q < kEdW; ++q) {
          const int j = tid + q * S::THREADS;
          if (j < A.W && edit_mag2(gxa[q], f_to_f(sgy[j])) < t2) sgy[j] = zero;
        }
      }
      __syncthreads();
    }
    float2 v[S::R1];
    if (IN != kInGrad && act) {
      // the given Laplacian, or z = Crop^T(grad_out): rows ia, ib at torus rows p + ia, p + ib, columns
      // j < W at p + j; and the row pair's sum for the (sum grad_out) e_00 term,
      // compensated in FP32 (Knuth's TwoSum: the sum and the exact rounding
      // errors), so no FP64 work (scarce on this part) runs per value
      const int ia = g * RW + 2 * f, ib = ia + 1;
      const bool ha = ia < A.H, hb = ib < A.H;
      const T* xa = sgx + (size_t)(2 * f) * A.W;
      const T* xb = xa + A.W;
      float sum = 0.0f, err = 0.0f;
#pragma unroll
      for (int r = 0; r < S::R1; ++r) {
        const int j = t + S::R2 * r - kP;
        const bool sure = (S::R2 * r >= kP) && (S::R2 * r + S::R2 - 1 - kP < S::WMIN);
        const bool c1 = sure || (j >= 0 && j < A.W);
        const float a = (ha && c1) ? f_to_f(xa[j]) : 0.0f, b = (hb && c1) ? f_to_f(xb[j]) : 0.0f;
        v[r] = make_float2(a, b);
        if constexpr (ADJ) {
          sum = two_sum_acc(sum, a, err);
          sum = two_sum_acc(sum, b, err);
        }
      }
      if constexpr (ADJ) red[tid] = make_float2(sum, err);
    } else if (act) {
      const int r0 = g * RW, ia = r0 + 2 * f, ib = ia + 1;
      const bool ha = ia < A.H, hb = ib < A.H, hm = ia >= 1;  // rows present (ia - 1 < H always)
      const bool sa = ia < A.nrows, sb = ib < A.nrows;         // rows inside the support
      const T* xa = sgx + (size_t)(2 * f) * A.W;
      const T* xb = xa + A.W;
      const T* ym = sgy + (size_t)(2 * f) * A.W;  // gy row ia - 1
      const T* ya = ym + A.W;
      const T* yb = ya + A.W;
#pragma unroll
      for (int r = 0; r < S::R1; ++r) {
        const int j = t + S::R2 * r - kP;
        // columns j - 1 .. j inside [0, W) for every t and every width padding to N
        const bool sure = (S::R2 * r >= kP + 1) && (S::R2 * r + S::R2 - 1 - kP < S::WMIN);
        const bool c1 = sure || (j >= 0 && j < A.W), c0 = sure || (j >= 1 && j - 1 < A.W);
        const bool inj = sure || (j >= 0 && j < A.ncols);
        const float xa1 = (ha && c1) ? f_to_f(xa[j]) : 0.0f, xa0 = (ha && c0) ? f_to_f(xa[j - 1]) : 0.0f;
        const float xb1 = (hb && c1) ? f_to_f(xb[j]) : 0.0f, xb0 = (hb && c0) ? f_to_f(xb[j - 1]) : 0.0f;
        const float ya1 = (ha && c1) ? f_to_f(ya[j]) : 0.0f, yb1 = (hb && c1) ? f_to_f(yb[j]) : 0.0f;
        const float ym1 = (hm && c1) ? f_to_f(ym[j]) : 0.0f;
        const float la = (xa1 - xa0) + (ya1 - ym1);
        const float lb = (xb1 - xb0) + (yb1 - ya1);
        v[r] = make_float2((sa && inj) ? la : 0.0f, (sb && inj) ? lb : 0.0f);
      }
    }
    __syncthreads();  // every staged row read: the buffers become the exchange buffers
    if (ADJ && act && t == 0) {
      // the row pair's sum over its threads in order (compensated), stored in FP64
      float sp = 0.0f, ep = 0.0f;
      for (int k = 0; k < S::T; ++k) {
        const float2 e = red[f * S::T + k];
        sp = two_sum_acc(sp, e.x, ep);
        ep = __fadd_rn(ep, e.y);
      }
      reinterpret_cast<double*>(partial)[(size_t)field * (kMaxRowBlocks / 2) + g * S::F + f] = (double)sp + (double)ep;
    }
    if (act) {
      dft_reg<S::R1, -1>(v);
#pragma unroll
      for (int s2 = 0; s2 < S::R1; ++s2) mybuf[t * S::R1P + s2] = v[s2];
    }
    __syncthreads();
    if (act && t < S::JSPAN) {
#pragma unroll
      for (int jj = 0; jj < S::J2; ++jj) {
        const int j = t + S::R2 * jj;
        float2 u[S::R2];
        u[0] = mybuf[j];
#pragma unroll
        for (int r = 1; r < S::R2; ++r) u[r] = cmul(mybuf[j + S::R1P * r], tw2[j * S::R2 + r]);
        dft_reg<S::R2, -1>(u);
#pragma unroll
        for (int s2 = 0; s2 < S::R2; ++s2) mybuf2[j + S::R1 * s2] = u[s2];
      }
    }
    __syncthreads();  // stage-2 results visible
    if constexpr (TRI) {
      tri_store_item<S, ADJ>(buf2, spec, tri, cc, field, g, A);
    } else {
    if (g == 0) {
      float2* Sz = spec + (size_t)field * A.Nh * A.ldM;
      const int nz = A.M - A.nrows;
      for (int idx = tid; idx < A.Nh * nz; idx += blockDim.x) {
        const int k = idx / nz, q = idx - k * nz;
        Sz[(size_t)k * A.ldM + (q < kP ? q : q + A.nrows)] = make_float2(0.0f, 0.0f);
      }
    }
    const int ra = g * 2 * S::F + 2 * uf;
    if (uact && ra < A.nrows) {
      float2* Sp = spec + (size_t)field * A.Nh * A.ldM + A.p + ra;
      const float2* zb = buf2 + uf * S::NO;
      const bool two = ra + 1 < A.nrows, vec = ((A.p + ra) & 1) == 0;
      for (int k = uk0; k < A.Nh; k += S::T) {
        const float2 zk = zb[k], zm = zb[k == 0 ? 0 : S::N - k];
        const float2 xa = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
        const float2 xb = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
        float2* dst = Sp + (size_t)k * A.ldM;
        if (two && vec) {
          *reinterpret_cast<float4*>(dst) = make_float4(xa.x, xa.y, xb.x, xb.y);
        } else {
          dst[0] = xa;
          if (two) dst[1] = xb;
        }
      }
    }
    }
    fence_proxy_async_smem();  // this thread's accesses of the buffers precede the next bulk copies
    __syncthreads();
    if (tid == 0 && w + (int)gridDim.x < items) issue(w + gridDim.x, false);
    if (tid == 0 && w + 2 * (int)gridDim.x < items) issue(w + 2 * gridDim.x, true);
  }
}

// ---------------------------------------------------------------------------
// pass B: column transform, Green multiply, inverse column transform, over
// items (field, block of C columns); persistent. Thread tid = t C + c works on
// column c of the block, so a warp's loads and stores cover whole 32-byte
// sectors of C neighbouring columns: the spectrum columns are read straight
// into registers (the next item's columns are prefetched into L2 meanwhile)
// and the result rows p .. p+H-1 (adjoint: p .. p+H) are written row-major
// straight from registers. The block's Green columns arrive by bulk copy,
// issued one item ahead.
// ---------------------------------------------------------------------------
// adjoint: sum(grad_out) of each field from its row-pair FP64 sums, lane-strided
// then a fixed shuffle tree (the same order on every call), into the field's
// slot kAdjTotal for the column pass; one warp per field
constexpr int kAdjTotal = kMaxRowBlocks / 2 - 1;
static __global__ void __launch_bounds__(32) k_adj_total(double* __restrict__ partial, int zpairs) {
  double* pp = partial + (size_t)blockIdx.x * (kMaxRowBlocks / 2);
  double a = 0.0;
  for (int i = threadIdx.x; i < zpairs; i += 32) a += pp[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (threadIdx.x == 0) pp[kAdjTotal] = a;
}

// the same sum, by one warp of the carry sweep (every lane gets it)
__device__ __forceinline__ float adj_total(const double* partial, int field, const FastArgs& A) {
  const double* pp = partial + (size_t)field * (kMaxRowBlocks / 2);
  double a = 0.0;
  for (int i = threadIdx.x & 31; i < A.zpairs; i += 32) a += __ldcg(pp + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return (float)a;
}

// ---------------------------------------------------------------------------
// Recursive column solve, between the row passes: the carry sweep. A block
// takes 32 columns (one per lane) of one field; its kTriSeg warps cut the G
// bands into segments. With T_g = a^(rows of band g):
//   causal:     the carry into band g is c_g, c_{g+1} = e_g + T_g c_g around the
//               cycle, where the rows after the last band (tail) and above band 0
//               (pad) are zero: a^tail (c_G - prod T c_0) = (1 - a^M) y[M-1] -
//               ..., i.e. with P the sweep of the e_g from a zero carry,
//               y[M-1] = a^tail P_G / (1 - a^M) and c_0 = a^p y[M-1];
//   anticausal: the carry from below band g is q_g, q_{g-1} = e'_g + T_g q_g,
//               q_{G-1} = a^tail y'[0], y'[0] = a^p Q_{-1} / (1 - a^M) with Q the
//               sweep from a zero carry.
// Each warp sweeps its segment from zero carries (both directions); warps 0
// and 1 then sweep the segment totals (segment transfers a^(2F n) from the
// plan's FP64 power table) and close the cycle; every warp re-sweeps its
// segment from its true carries and writes c_g, q_g (the band sums are read
// twice, the second time from cache). Row 0 of the solved spectrum (a padding
// row, X = 0) is U[0][l] = C_l (a y[M-1] + y'[0]): the block's FP64 sum of
// w_l Re U[0][l] (w = 1 at l = N/2, else 2) is its partial of u[0,0], added in
// block order by the inverse row pass. Column 0 (b = 2, singular) is the 1D
// periodic Poisson problem with its mean removed (the reading G[0,0] = 0): one
// more block per field solves it exactly in FP64 and writes it into S.
// ---------------------------------------------------------------------------
constexpr int kTriSeg = kTriSegments;  // band segments (warps) per sweep block
constexpr int kTriTileMaxG = 160;      // bands whose sums a sweep block stages (80 KB)

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Inclusive scan of one FP64 value per thread over NW warps (the whole block when
// NW > 1, through ws[NW]); the last thread's value, the total, in `total`.
template <int NW>
__device__ __forceinline__ double scan_d(double v, double* ws, double& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  if constexpr (NW == 1) {
    total = __shfl_sync(0xffffffffu, v, 31);
    return v;
  }
  if (lane == 31) ws[warp] = v;
  __syncthreads();
  double base = 0.0, t = 0.0;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    const double x = ws[w];
    if (w < warp) base += x;
    t += x;
  }
  __syncthreads();
  total = t;
  return v + base;
}

// Column 0 of one field (FP64, by NW warps): d[r] = u[r+1] - u[r] has
// d[r] - d[r-1] = f[r] - mean(f); periodicity fixes d[-1] = D = -sum_r G[r] / M
// with G the prefix sums of f - mean(f); u[0] = 0 (any constant is removed with
// u[0,0]: column 0 adds w_0 U[0][0] = u[0] / N = 0 to it). f(r) gives torus row
// r's value; each thread takes a contiguous run of rows: one pass for its sums
// P = sum f and Q = sum of f's running sums, two scans over the threads, one pass
// that rebuilds u. put(r, u[r] / N) for every torus row. FP64 runs at a small
// fraction of the FP32 rate here, so the passes do eight FP64 instructions a
// row; one warp at thirteen a row, on the sweep's critical path, was 12 of the
// 24 us of a sweep of 3 fields of 801x1200 and 36 of 101 for 2048 of 256x256.
template <int NW, class F, class Put>
__device__ __forceinline__ void column0_solve(F f, Put put, double* ws, int M, double invM, double invN) {
  const int run = (M + 32 * NW - 1) / (32 * NW);
  const int me = NW == 1 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  const int r0 = min(me * run, M), r1 = min(r0 + run, M), n = r1 - r0;
  double P = 0.0, Q = 0.0;  // sum of f, sum over the run's rows of the running sum
  for (int r = r0; r < r1; ++r) {
    P += (double)f(r);
    Q += P;
  }
  double sum, gsum;
  const double Pi = scan_d<NW>(P, ws, sum);
  const double mean = sum * invM;
  const double off = (Pi - P) - mean * (double)r0;                       // G just above the run
  const double Gs = Q + (double)n * (off - mean * (0.5 * (double)(n + 1)));  // sum of G over the run
  const double Gi = scan_d<NW>(Gs, ws, gsum);
  const double D = -gsum * invM;
  double u = ((Gi - Gs) + D * (double)r0) * invN, g = (off + D) * invN;
  const double mN = mean * invN;
  for (int r = r0; r < r1; ++r) {
    put(r, (float)u);
    g += fma((double)f(r), invN, -mN);
    u += g;
  }
}

static __global__ void __launch_bounds__(32 * kTriSeg) k_tri_carries(float2* __restrict__ spec,
                                                                          float2* __restrict__ tri,
                                                                          const float* __restrict__ cc,
                                                                          const float* __restrict__ powc,
                                                                          double* __restrict__ partial, FastArgs A) {
  __shared__ float2 seg_e[kTriSeg][kTriCols], seg_q[kTriSeg][kTriCols];  // segment totals, then carries
  __shared__ float2 y0s[kTriCols];
  __shared__ float yls[2 * kTriCols];
  __shared__ __align__(8) uint64_t tbar;
  __shared__ float sadj_s;
  __shared__ double ws[kTriSeg];
  extern __shared__ __align__(16) float2 tile[];  // the block's band sums when they fit (staged)
  const int nkb = gridDim.x - 1;  // column blocks; one more block for column 0
  const int kb = blockIdx.x, field = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k = kb * kTriCols + lane;
  const bool col_ok = k >= 1 && k < A.Nh;
  wait_for_predecessor();
  dependents_may_start();
  if (kb == nkb) {
    const float sadj = A.adj ? adj_total(partial, field, A) : 0.0f;  // (every warp for itself)
    const int nr = min(A.srows, A.M - A.p);
    const float* c0 = tri_col0(tri, field, A);
    float2* col = spec + (size_t)field * A.srows * A.ldY;
    column0_solve<kTriSeg>(
        [&](int r) { return r == 0 ? -sadj : (r >= A.p && r < A.p + nr ? __ldcg(c0 + (r - A.p)) : 0.0f); },
        [&](int r, float u) {
          if (r >= A.p && r < A.p + nr) col[(size_t)(r - A.p) * A.ldY] = make_float2(u, 0.0f);
        },
        ws, A.M, A.invM, A.invN);
    return;
  }
  const float2* gsums = tri_sums(tri, field, A) + (size_t)kb * 2 * A.G * kTriCols;  // [g][2][32], contiguous
  const bool staged = A.G <= kTriTileMaxG;
  const float2* sums = (staged ? tile : gsums) + lane;
  float2* carry = tri + (size_t)field * A.tri_field + k;  // [g][2][ldY]
  if (staged) {  // the whole tile of band sums by one bulk copy
    if (tid == 0) {
      mbar_init(&tbar, 1);
      bulk_load(tile, gsums, (unsigned)(2 * A.G * kTriCols * sizeof(float2)), &tbar);
    }
    if (A.adj && warp == 1) {
      const float t = adj_total(partial, field, A);
      if (lane == 0) sadj_s = t;
    }
    __syncthreads();
    const bool landed = mbar_wait(&tbar, 0);
    if (__syncthreads_or(!landed)) {  // the copy never completed: report, let it drain, stop
      if (tid == 0) atomicExch(A.err, kErrBulkWait);
      mbar_wait(&tbar, 0);
      return;
    }
  } else if (A.adj) {
    if (warp == 1) {
      const float t = adj_total(partial, field, A);
      if (lane == 0) sadj_s = t;
    }
    __syncthreads();
  }
  // the adjoint's z has -(sum grad_out) at torus (0, 0): -s in every column of row 0
  const float sadj = A.adj ? sadj_s : 0.0f;
  float4 c03 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), c47 = c03;
  if (col_ok) {
    c03 = __ldg(reinterpret_cast<const float4*>(cc + (size_t)k * 8));
    c47 = __ldg(reinterpret_cast<const float4*>(cc + (size_t)k * 8) + 1);
  }
  const float a = c03.y, C = c03.z, Db = c03.w, Dl = c47.x, Tp = c47.y, inv = c47.z, Tt = c47.w;
  const int per = (A.G + kTriSeg - 1) / kTriSeg;
  const int g0 = min(warp * per, A.G), g1 = min(g0 + per, A.G);
  // phase 1: each segment from zero carries
  if (warp < kTriSeg) {
    float2 t = make_float2(0.0f, 0.0f), q = t;
    if (col_ok) {
#pragma unroll 4
      for (int g = g0; g < g1; ++g) {
        const float D = (g == A.G - 1) ? Dl : Db;
        const float2 e = sums[(size_t)g * 2 * kTriCols];
        t = tri_carry(e, t, D);
      }
#pragma unroll 4
      for (int g = g1 - 1; g >= g0; --g) {
        const float D = (g == A.G - 1) ? Dl : Db;
        const float2 e = sums[(size_t)g * 2 * kTriCols + kTriCols];
        q = tri_carry(e, q, D);
      }
    }
    seg_e[warp][lane] = t;
    seg_q[warp][lane] = q;
  }
  __syncthreads();
  // phase 2: the segment totals around the cycle (warp 0 causal, warp 1 anticausal)
  if (warp < 2 && col_ok) {
    float Ts[kTriSeg];  // transfer of segment s: a^(rows of its bands), all loaded at once
#pragma unroll
    for (int s2 = 0; s2 < kTriSeg; ++s2) {
      const int b0 = min(s2 * per, A.G), b1 = min(b0 + per, A.G);
      Ts[s2] = (b1 <= b0) ? 1.0f
                          : (b1 < A.G ? __ldg(powc + (size_t)(b1 - b0) * A.ldY + k)
                                      : __ldg(powc + (size_t)(b1 - b0 - 1) * A.ldY + k) * (1.0f - Dl));
    }
    auto seg_T = [&](int s2) { return Ts[s2]; };
    if (warp == 0) {
      float2 t = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int s = 0; s < kTriSeg; ++s) {
        const float T = seg_T(s);
        const float2 e = seg_e[s][lane];
        t = make_float2(fmaf(T, t.x, e.x), fmaf(T, t.y, e.y));
      }
      const float2 yl = make_float2(Tt * t.x * inv, Tt * t.y * inv);  // y[M-1]
      float2 c = make_float2(Tp * yl.x, Tp * yl.y);                   // y[p-1]: carry into band 0
      if (A.adj) c.x -= (Tp / a) * sadj * inv;  // row 0's -s, carried a^(p-1) down
#pragma unroll
      for (int s = 0; s < kTriSeg; ++s) {
        const float T = seg_T(s);
        const float2 e = seg_e[s][lane];
        seg_e[s][lane] = c;
        c = make_float2(fmaf(T, c.x, e.x), fmaf(T, c.y, e.y));
      }
      yls[lane] = yl.x;
    } else {
      float2 q = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int s = kTriSeg - 1; s >= 0; --s) {
        const float T = seg_T(s);
        const float2 e = seg_q[s][lane];
        q = make_float2(fmaf(T, q.x, e.x), fmaf(T, q.y, e.y));
      }
      float2 y0 = make_float2(Tp * q.x * inv, Tp * q.y * inv);  // y'[0]
      if (A.adj) y0.x = (Tp * q.x - sadj) * inv;
      float2 c = make_float2(Tt * y0.x, Tt * y0.y);                   // carry from below the last band
#pragma unroll
      for (int s = kTriSeg - 1; s >= 0; --s) {
        const float T = seg_T(s);
        const float2 e = seg_q[s][lane];
        seg_q[s][lane] = c;
        c = make_float2(fmaf(T, c.x, e.x), fmaf(T, c.y, e.y));
      }
      y0s[lane] = y0;
    }
  }
  __syncthreads();
  // phase 3: each segment again from its true carries; the carries go out
  if (warp < kTriSeg && col_ok) {
    float2 c = seg_e[warp][lane];
#pragma unroll 4
    for (int g = g0; g < g1; ++g) {
      const float D = (g == A.G - 1) ? Dl : Db;
      const float2 e = sums[(size_t)g * 2 * kTriCols];
      carry[(size_t)(2 * g) * A.ldY] = c;
      c = tri_carry(e, c, D);
    }
    float2 q = seg_q[warp][lane];
#pragma unroll 4
    for (int g = g1 - 1; g >= g0; --g) {
      const float D = (g == A.G - 1) ? Dl : Db;
      const float2 e = sums[(size_t)g * 2 * kTriCols + kTriCols];
      carry[(size_t)(2 * g + 1) * A.ldY] = q;
      q = tri_carry(e, q, D);
    }
  }
  if (warp == 0 && !A.adj) {  // u[0,0] (the adjoint has no offset)
    double acc = 0.0;
    if (col_ok) acc = (2 * k == A.N ? 1.0 : 2.0) * (double)(C * fmaf(a, yls[lane], y0s[lane].x));
    acc = warp_sum_d(acc);
    double* pp = partial + (size_t)field * (kMaxRowBlocks / 2);
    unsigned done = 0;
    if (lane == 0) {
      pp[kb] = acc;
      __threadfence();  // this partial is visible before the count says so
      done = atomicAdd(reinterpret_cast<unsigned*>(pp + kTriCnt), 1u);
    }
    done = __shfl_sync(0xffffffffu, done, 0);
    if (done == (unsigned)nkb - 1) {
      // the field's last sweep block: u[0,0] from every block's partial,
      // lane-strided then a fixed shuffle tree (the same order on every call)
      __threadfence();
      double s2 = 0.0;
      for (int i = lane; i < nkb; i += 32) s2 += __ldcg(pp + i);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s2 += __shfl_down_sync(0xffffffffu, s2, o);
      if (lane == 0) pp[kTriU00] = s2;
    }
  }
}

// The carry sweep for fields of at most kTriRegG bands: one warp per (field,
// block of 32 columns), one column per lane, all of the block's band sums in
// registers (one round of loads per direction), each direction swept from a
// zero carry and then from the true carries, as above; no shared-memory
// staging and no block barriers. One more warp per field solves column 0 exactly,
// and each field's last warp to finish combines the u[0,0] partials.
constexpr int kTriRegG = 32;
constexpr int kTriRegWarps = 8;
// MAXG: the loops' length; short columns run a shorter one at twice the blocks per
// SM (12288 warps of 72-row columns of 5 bands: 37 us with the loops of 32, 55 with
// loops of 48).
template <int MAXG>
__global__ void __launch_bounds__(32 * kTriRegWarps, MAXG <= 16 ? 4 : 2) k_tri_carries_reg(
    float2* __restrict__ spec, float2* __restrict__ tri, const float* __restrict__ cc, double* __restrict__ partial,
    FastArgs A, int nkb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int task = blockIdx.x * kTriRegWarps + warp;
  wait_for_predecessor();
  dependents_may_start();
  if (task >= A.nf * (nkb + 1)) return;
  const int field = task / (nkb + 1), kb = task - field * (nkb + 1);
  const int k = kb * kTriCols + lane;
  const bool col_ok = k >= 1 && k < A.Nh;
  const int G = A.G;
  // the adjoint's z has -(sum grad_out) at torus (0, 0): -s in every column of row 0
  const float sadj = A.adj ? adj_total(partial, field, A) : 0.0f;
  if (kb == nkb) {
    const int nr = min(A.srows, A.M - A.p);
    const float* c0 = tri_col0(tri, field, A);
    float2* col = spec + (size_t)field * A.srows * A.ldY;
    column0_solve<1>(
        [&](int r) { return r == 0 ? -sadj : (r >= A.p && r < A.p + nr ? __ldcg(c0 + (r - A.p)) : 0.0f); },
        [&](int r, float u) {
          if (r >= A.p && r < A.p + nr) col[(size_t)(r - A.p) * A.ldY] = make_float2(u, 0.0f);
        },
        nullptr, A.M, A.invM, A.invN);
    return;
  }
  const float2* sums = tri_sums(tri, field, A) + (size_t)kb * 2 * G * kTriCols + lane;  // [g][2][32]
  float2* carry = tri + (size_t)field * A.tri_field + k;                                 // [g][2][ldY]
  double acc = 0.0;
  if (col_ok) {
    const float4 c03 = __ldg(reinterpret_cast<const float4*>(cc + (size_t)k * 8));
    const float4 c47 = __ldg(reinterpret_cast<const float4*>(cc + (size_t)k * 8) + 1);
    const float a = c03.y, C = c03.z, Db = c03.w, Dl = c47.x, Tp = c47.y, inv = c47.z, Tt = c47.w;
    float2 yl, y0;
    {  // causal: the band sums in registers, from a zero carry, close the cycle, carries out
      float2 e[MAXG];
#pragma unroll
      for (int g = 0; g < MAXG; ++g)
        if (g < G) e[g] = sums[(size_t)g * 2 * kTriCols];
      float2 t = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int g = 0; g < MAXG; ++g)
        if (g < G) {
          const float D = (g == G - 1) ? Dl : Db;
          t = tri_carry(e[g], t, D);
        }
      yl = make_float2(Tt * t.x * inv, Tt * t.y * inv);  // y[M-1]
      float2 c = make_float2(Tp * yl.x, Tp * yl.y);     // carry into band 0
      if (A.adj) c.x -= (Tp / a) * sadj * inv;          // row 0's -s, carried a^(p-1) down
#pragma unroll
      for (int g = 0; g < MAXG; ++g)
        if (g < G) {
          const float D = (g == G - 1) ? Dl : Db;
          carry[(size_t)(2 * g) * A.ldY] = c;
          c = tri_carry(e[g], c, D);
        }
    }
    {  // anticausal, the same way up the bands
      float2 ep[MAXG];
#pragma unroll
      for (int g = 0; g < MAXG; ++g)
        if (g < G) ep[g] = sums[(size_t)g * 2 * kTriCols + kTriCols];
      float2 q = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int g = MAXG - 1; g >= 0; --g)
        if (g < G) {
          const float D = (g == G - 1) ? Dl : Db;
          q = tri_carry(ep[g], q, D);
        }
      y0 = make_float2(Tp * q.x * inv, Tp * q.y * inv);  // y'[0]
      if (A.adj) y0.x = (Tp * q.x - sadj) * inv;
      float2 c = make_float2(Tt * y0.x, Tt * y0.y);     // carry from below the last band
#pragma unroll
      for (int g = MAXG - 1; g >= 0; --g)
        if (g < G) {
          const float D = (g == G - 1) ? Dl : Db;
          carry[(size_t)(2 * g + 1) * A.ldY] = c;
          c = tri_carry(ep[g], c, D);
        }
    }
    acc = (2 * k == A.N ? 1.0 : 2.0) * (double)(C * fmaf(a, yl.x, y0.x));
  }
  acc = warp_sum_d(acc);
  double* pp = partial + (size_t)field * (kMaxRowBlocks / 2);
  if (A.adj) return;  // u[0,0]: the adjoint has no offset
  unsigned done = 0;
  if (lane == 0) {
    pp[kb] = acc;
    __threadfence();  // this partial is visible before the count says so
    done = atomicAdd(reinterpret_cast<unsigned*>(pp + kTriCnt), 1u);
  }
  done = __shfl_sync(0xffffffffu, done, 0);
  if (done == (unsigned)nkb - 1) {
    // the field's last warp: u[0,0] from every column block's partial,
    // lane-strided then a fixed shuffle tree (the same order on every call)
    __threadfence();
    double s2 = 0.0;
    for (int i = lane; i < nkb; i += 32) s2 += __ldcg(pp + i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_down_sync(0xffffffffu, s2, o);
    if (lane == 0) pp[kTriU00] = s2;
  }
}

template <class S, int MODE>
__global__ void __launch_bounds__(S::THREADS, S::MINB) k_fast_cols(const float2* __restrict__ spec, float2* __restrict__ Y,
                                                          const float* __restrict__ GT, const float2* __restrict__ twg,
                                                          float* __restrict__ partial, FastArgs A) {
  extern __shared__ __align__(16) float2 sm[];
  float* gsm = reinterpret_cast<float*>(sm);                       // [C][GS] Green columns of the item
  float2* twF = reinterpret_cast<float2*>(gsm + S::C * S::GS);     // [R1][TWF_STRIDE]: w_M^(r j), j < R1, r < R2
  float2* twI = twF + S::R1 * S::TWF_STRIDE;                       // [R2][TWI_STRIDE]: w_M^(r j), j < R2, r < R1
  float2* xbuf = twI + S::R2 * S::TWI_STRIDE;                      // [C][MP] exchange
  __shared__ __align__(8) uint64_t bar;
  const int tid = threadIdx.x;
  const int c = tid % S::C, t = tid / S::C;
  const bool act = t < S::R2, act2 = t < S::R1;
  const int items = A.nf * A.nparts;
  const int yrows = (MODE == 2) ? A.H + 1 : A.H;
  float2* mybuf = xbuf + c * S::MP;
  const float* gcol = gsm + c * S::GS;
  auto ncols_of = [&](int blk) { return (A.Nh - blk * S::C) < S::C ? (A.Nh - blk * S::C) : S::C; };
  auto issue_green = [&](int w) {  // one thread
    const int blk = w % A.nparts;
    const unsigned gb = (unsigned)(ncols_of(blk) * A.ldM * sizeof(float));
    bulk_load(gsm, GT + (size_t)blk * S::C * A.ldM, gb, &bar);
  };
  auto prefetch_spec = [&](int w) {  // one thread: the item's spectrum columns into L2
    const int field = w / A.nparts, blk = w - field * A.nparts;
    l2_prefetch(spec + ((size_t)field * A.Nh + (size_t)blk * S::C) * A.ldM,
                (unsigned)(ncols_of(blk) * A.ldM * sizeof(float2)));
  };
  for (int i = tid; i < S::R1 * S::R2; i += blockDim.x) {
    const int j = i / S::R2, r = i - j * S::R2;
    twF[j * S::TWF_STRIDE + r] = twg[r * j];
  }
  for (int i = tid; i < S::R2 * S::R1; i += blockDim.x) {
    const int j = i / S::R1, r = i - j * S::R1;
    twI[j * S::TWI_STRIDE + r] = twg[r * j];
  }
  if (tid == 0) {
    mbar_init(&bar, 1);
    if ((int)blockIdx.x < items) issue_green(blockIdx.x);
  }
  __syncthreads();  // barrier initialised, twiddles in place
  unsigned phase = 0;
#pragma unroll 1
  for (int w = blockIdx.x; w < items; w += gridDim.x, phase ^= 1u) {
    const int field = w / A.nparts, blk = w - field * A.nparts;
    const int l = blk * S::C + c;
    const bool colok = l < A.Nh;
    if (tid == 0 && w + (int)gridDim.x < items) prefetch_spec(w + gridDim.x);
    // rows outside the support were zeroed by the row pass
    float2 v[S::R1];
    {
      const float2* col = spec + ((size_t)field * A.Nh + (colok ? l : 0)) * A.ldM;
#pragma unroll
      for (int r = 0; r < S::R1; ++r) v[r] = (act && colok) ? col[t + S::R2 * r] : make_float2(0.0f, 0.0f);
    }
    if (MODE == 2) {
      // adjoint: z = Crop^T(grad_out) - (sum grad_out) e_00; the row DFT of the
      // second term is -sum in every column, at torus row 0 (the sum from
      // k_adj_total); the threads with t = 0 are lanes 0 .. C-1 of warp 0.
      if (t == 0) {
        const double a = reinterpret_cast<const double*>(partial)[(size_t)field * (kMaxRowBlocks / 2) + kAdjTotal];
        v[0] = make_float2((float)(-a), 0.0f);
      }
    }
    if (act) dft_reg<S::R1, -1>(v);
    __syncthreads();  // the previous item's reads of the exchange are done
    if (act) {
#pragma unroll
      for (int s2 = 0; s2 < S::R1; ++s2) mybuf[t * S::R1 + s2] = v[s2];
    }
    __syncthreads();
    float2 u[S::R2];
    if (act2) {
      u[0] = mybuf[t];
#pragma unroll
      for (int r = 1; r < S::R2; ++r) u[r] = cmul(mybuf[t + S::R1 * r], twF[t * S::TWF_STRIDE + r]);
      dft_reg<S::R2, -1>(u);
    }
    const bool landed = mbar_wait(&bar, phase);
    if (act2) {
      // bins k = t + R1 s: multiply by the real Green spectrum (Eq. 23)
#pragma unroll
      for (int s2 = 0; s2 < S::R2; ++s2) u[s2] = cscale(u[s2], gcol[t + S::R1 * s2]);
      // inverse stage 1 (span 1): butterfly t takes exactly the bins t + R1 r held here
      dft_reg<S::R2, +1>(u);
    }
    fence_proxy_async_smem();  // this thread's reads of the Green columns precede the next bulk copy
    if (__syncthreads_or(!landed)) {  // the copy never completed: report, let it drain, stop
      if (tid == 0) atomicExch(A.err, kErrBulkWait);
      mbar_wait(&bar, phase);
      return;
    }
    if (tid == 0 && w + (int)gridDim.x < items) issue_green(w + gridDim.x);
    if (act2) {
#pragma unroll
      for (int s2 = 0; s2 < S::R2; ++s2) mybuf[t * (S::R2 + 1) + s2] = u[s2];  // pad(t R2 + s2), s2 < R2
    }
    __syncthreads();
    if (act) {
      // pad(t + R2 r) = t + (R2 + 1) r for t < R2
      v[0] = mybuf[t];
#pragma unroll
      for (int r = 1; r < S::R1; ++r) v[r] = cmul(mybuf[t + (S::R2 + 1) * r], cconj(twI[t * S::TWI_STRIDE + r]));
      dft_reg<S::R1, +1>(v);
    }
    if (MODE != 2 && tid < 32) {
      // u[0,0] = sum over the row-0 spectrum, weight 1 at l = 0 and N/2, 2
      // elsewhere; FP64, columns added in order (an error in u[0,0] shifts
      // every output pixel)
      const double cv = (tid < S::C && colok) ? ((l == 0 || 2 * l == A.N) ? (double)v[0].x : 2.0 * (double)v[0].x)
                                              : 0.0;
      double s2 = 0.0;
#pragma unroll
      for (int cc = 0; cc < S::C; ++cc) s2 += __shfl_sync(0xffffffffu, cv, cc);
      if (tid == 0) reinterpret_cast<double*>(partial)[(size_t)field * (kMaxRowBlocks / 2) + blk] = s2;
    }
    if (act && colok) {
      float2* Yc = Y + (size_t)field * yrows * A.ldY + l;
#pragma unroll
      for (int r = 0; r < S::R1; ++r) {
        const int i = t + S::R2 * r - A.p;  // image row of torus row t + R2 r
        if (i >= 0 && i < yrows) Yc[(size_t)i * A.ldY] = v[r];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// pass C: inverse row transforms of the row-major spectrum Y with the
// Hermitian extension formed on load, offset, crop and cast. Persistent over
// (field, group of F output row pairs). The 2F rows of Y an item needs are one
// contiguous bulk copy into the exchange buffer, completed on an mbarrier; the
// copy for the next item is issued as soon as this item's stage-2 inputs are
// in registers, so it overlaps the stage-2 transforms and the output stores.
// ---------------------------------------------------------------------------
// Recursive column solve, pass C side: the 2F staged rows of band g (row-major
// spectrum S) become the inputs of the band's F inverse transforms in place. Per
// column l >= 1, from the band's two staged carries: the causal recursion down the
// band and the anticausal one up it, U = C_l (y + y' - X); column 0 already holds
// its exact solution. Of each row pair (a, b) the column's thread has both values,
// so it forms the transform's inputs A + i B at l and, by the Hermitian extension,
// at N - l, and leaves them in the pair's two slots of column l: row 2f the one at
// l, row 2f + 1 the one at N - l. The transforms then read one value per input;
// with U left in the rows they read both rows for every input, and y crossed
// shared memory once more (six passes over the band against three; these kernels
// are bound by shared-memory wavefronts): the inverse pass of 100 fields of
// 801x1200 227 -> 204 us, of 2048 bf16 fields of 256x256 315 -> 281 us. Rows past
// the torus (band rows >= nb) hold zeros and stay so.
template <class S>
__device__ __forceinline__ void tri_pack_pair(float2 ya, float2 yb, bool edge, float2& lo, float2& hi) {
  if (edge) ya.y = yb.y = 0.0f;  // bins 0 and N/2 are real in a real transform
  lo = make_float2(ya.x - yb.y, ya.y + yb.x);
  hi = make_float2(ya.x + yb.y, yb.x - ya.y);
}

template <class S>
__device__ __forceinline__ void tri_solve_band(float2* buf, const float2* cbuf, const float* __restrict__ cc, int g,
                                               const FastArgs& A) {
  constexpr int RW = 2 * S::F;
  const int nb = min(RW, A.M - A.p - g * RW);
  if constexpr (S::SHORT) {
    // short rows: one column per thread (the band's RW values of a column pair
    // would not fit the registers of four blocks per SM); y stays in registers
    // where x and y of the band fit them, else in the column's slots
    constexpr bool kRegs = RW <= 18;
    const float2* dcs = reinterpret_cast<const float2*>(cc + (size_t)A.Nh * 8);  // (delta, C) per column
    for (int k = threadIdx.x; k < A.Nh; k += blockDim.x) {
      const float2 dc = __ldg(dcs + k);
      float2 yc = cbuf[k], ya = cbuf[S::LDY + k];
      float2* col = buf + k;
      float2 x[RW], y[kRegs ? RW : 1];
#pragma unroll
      for (int r = 0; r < RW; ++r) x[r] = col[(size_t)r * S::LDY];
      if (k == 0) {
#pragma unroll
        for (int f = 0; f < S::F; ++f) col[(size_t)(2 * f) * S::LDY] = make_float2(x[2 * f].x, x[2 * f + 1].x);
        continue;
      }
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        if (r < nb) yc = tri_step(x[r], yc, dc.x);
        if constexpr (kRegs)
          y[r] = yc;
        else
          col[(size_t)r * S::LDY] = yc;
      }
      const bool edge = 2 * k == S::N;
#pragma unroll
      for (int f = S::F - 1; f >= 0; --f) {
        float2 u[2];
#pragma unroll
        for (int h = 1; h >= 0; --h) {
          const int r = 2 * f + h;
          u[h] = x[r];
          if (r < nb) {
            ya = tri_step(x[r], ya, dc.x);
            u[h] = cscale(csub(cadd(kRegs ? y[kRegs ? r : 0] : col[(size_t)r * S::LDY], ya), x[r]), dc.y);
          }
        }
        float2 lo, hi;
        tri_pack_pair<S>(u[0], u[1], edge, lo, hi);
        col[(size_t)(2 * f) * S::LDY] = lo;
        col[(size_t)(2 * f + 1) * S::LDY] = hi;
      }
    }
  } else {
    // thread t takes the column pair (2j, 2j + 1), 16-byte shared-memory accesses;
    // columns >= Nh are padding
    for (int j = threadIdx.x; 2 * j < A.Nh; j += blockDim.x) {
      const int k0 = 2 * j;
      // (delta, C) of both columns in one coalesced 16-byte load (the plan's compact table)
      const float4 dc = __ldg(reinterpret_cast<const float4*>(cc + (size_t)A.Nh * 8) + j);
      const float4 yc4 = reinterpret_cast<const float4*>(cbuf)[j];
      const float4 ya4 = reinterpret_cast<const float4*>(cbuf + S::LDY)[j];
      float2 yc0 = make_float2(yc4.x, yc4.y), yc1 = make_float2(yc4.z, yc4.w);
      float2 ya0 = make_float2(ya4.x, ya4.y), ya1 = make_float2(ya4.z, ya4.w);
      float4* col = reinterpret_cast<float4*>(buf) + j;
      float4 x[RW], y[RW];
#pragma unroll
      for (int r = 0; r < RW; ++r) x[r] = col[(size_t)r * (S::LDY / 2)];
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        if (r < nb) {
          yc0 = tri_step(make_float2(x[r].x, x[r].y), yc0, dc.x);
          yc1 = tri_step(make_float2(x[r].z, x[r].w), yc1, dc.z);
        }
        y[r] = make_float4(yc0.x, yc0.y, yc1.x, yc1.y);
      }
      const bool e0 = k0 == 0 || 2 * k0 == S::N, e1 = 2 * (k0 + 1) == S::N;
#pragma unroll
      for (int f = S::F - 1; f >= 0; --f) {
        float2 u0[2], u1[2];
#pragma unroll
        for (int h = 1; h >= 0; --h) {
          const int r = 2 * f + h;
          const float2 x0 = make_float2(x[r].x, x[r].y), x1 = make_float2(x[r].z, x[r].w);
          u0[h] = x0;
          u1[h] = x1;
          if (r < nb) {
            ya0 = tri_step(x0, ya0, dc.x);
            ya1 = tri_step(x1, ya1, dc.z);
            if (k0 > 0) u0[h] = cscale(csub(cadd(make_float2(y[r].x, y[r].y), ya0), x0), dc.y);
            u1[h] = cscale(csub(cadd(make_float2(y[r].z, y[r].w), ya1), x1), dc.w);
          }
        }
        float2 lo0, hi0, lo1, hi1;
        tri_pack_pair<S>(u0[0], u0[1], e0, lo0, hi0);
        tri_pack_pair<S>(u1[0], u1[1], e1, lo1, hi1);
        col[(size_t)(2 * f) * (S::LDY / 2)] = make_float4(lo0.x, lo0.y, lo1.x, lo1.y);
        col[(size_t)(2 * f + 1) * (S::LDY / 2)] = make_float4(hi0.x, hi0.y, hi1.x, hi1.y);
      }
    }
  }
}

// stage-1 inputs of transform f from the slots tri_solve_band left: input l of
// row 2f at l below N/2, of row 2f + 1 at N - l from N/2 on
template <class S>
__device__ __forceinline__ void tri_load_pair(float2 (&v)[S::R1], const float2* band, int f, int t) {
  constexpr int half = S::N / 2;
  const float2* lo_row = band + (size_t)(2 * f) * S::LDY;
  const float2* hi_row = lo_row + S::LDY + S::N;
#pragma unroll
  for (int r = 0; r < S::R1; ++r) {
    // l = t + R2 r with t < R2: whether l lies below or above N/2 is known at
    // compile time except for the one r whose range contains N/2
    const int l = t + S::R2 * r;
    const bool all_lo = S::R2 * r + S::R2 - 1 < half;
    const bool all_hi = S::R2 * r >= half;
    v[r] = all_lo ? lo_row[l] : (all_hi ? hi_row[-l] : *(l < half ? lo_row + l : hi_row - l));
  }
}

// Per-field statistics of the stored output (colour correction, Eq. 25): item
// g of a field writes (n, mean, sum of squared deviations) of its stored values in
// FP64 at partial (as doubles) + field * kMaxRowBlocks / 2 + kStatsOff + 3 g.

template <class S, typename T, bool TRI, bool STATS>
__global__ void __launch_bounds__(S::THREADS, S::MINB_INV) k_fast_rows_inv(const float2* __restrict__ Y,
                                                              float* __restrict__ partial, T* __restrict__ out,
                                                              const float2* __restrict__ twg, FastArgs A,
                                                              const float2* __restrict__ tri,
                                                              const float* __restrict__ cc) {
  extern __shared__ __align__(16) float2 sm[];
  float2* tw2 = sm;
  float2* buf = sm + S::R1 * S::R2;  // staged rows of Y (TRI: of S) [2F][ldY], then the stage-1 exchange
  float2* cbuf = sm + S::CBUF;        // TRI: the band's two carries [2][LDY]
  __shared__ float u00s[2];
  __shared__ __align__(8) uint64_t bar;
  constexpr int RW = 2 * S::F;       // rows of Y per item
  const int tid = threadIdx.x;
  const int f = tid / S::T, t = tid - f * S::T;
  const bool act = f < S::F;
  for (int i = tid; i < S::R1 * S::R2; i += blockDim.x) {
    const int j = i / S::R2, r = i - j * S::R2;
    tw2[i] = twg[r * j];
  }
  float2* mybuf = buf + (act ? f : 0) * S::NP;
  const int half = S::N / 2;
  const int items = A.nf * A.ngroups;
  // one thread: stage the rows of item w (prefetch: only start fetching them
  // into L2, for the copy one item later)
  auto issue = [&](int w, bool prefetch) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    const int r0 = g * RW, nr = (A.H - r0) < RW ? (A.H - r0) : RW;
    if constexpr (TRI) {  // the whole band of S (its rows past the image feed the recursions) and its carries
      const unsigned rb = (unsigned)(RW * A.ldY * sizeof(float2)), cb = (unsigned)(2 * A.ldY * sizeof(float2));
      const float2* ss = Y + ((size_t)field * A.srows + r0) * A.ldY;
      const float2* cs = tri + (size_t)field * A.tri_field + (size_t)g * 2 * A.ldY;
      if (prefetch) {
        l2_prefetch(ss, rb);
        l2_prefetch(cs, cb);
        return;
      }
      mbar_expect_tx(&bar, rb + cb);
      if (A.l2res)  // the band's last read
        bulk_copy_hint(buf, ss, rb, &bar, l2_policy_evict_first());
      else
        bulk_copy(buf, ss, rb, &bar);
      bulk_copy(cbuf, cs, cb, &bar);
    } else {
      const float2* ys = Y + ((size_t)field * A.H + r0) * A.ldY;
      const unsigned nb = (unsigned)(nr * A.ldY * sizeof(float2));
      if (prefetch)
        l2_prefetch(ys, nb);
      else
        bulk_load(buf, ys, nb, &bar);
    }
  };
  // warp 0 loads the u[0,0] partial sums of the next item while this one is
  // transformed (lane-strided, the same order as a plain loop over them); with
  // the recursive column solve the carry sweep has already combined them into
  // the field's u[0,0] (kTriU00), one value to load
  constexpr int KPF = TRI ? 1 : 5;
  double pf[KPF];
  auto prefetch = [&](int w) {
    if (tid < 32 && w < items) {
      const double* pp = reinterpret_cast<const double*>(partial) + (size_t)(w / A.ngroups) * (kMaxRowBlocks / 2);
      if constexpr (TRI) {
        pf[0] = tid == 0 ? pp[kTriU00] : 0.0;
      } else {
#pragma unroll
        for (int k = 0; k < KPF; ++k) pf[k] = (tid + 32 * k < A.nparts) ? pp[tid + 32 * k] : 0.0;
      }
    }
  };
  if (tid == 0) mbar_init(&bar, 1);
  __syncthreads();
  if constexpr (TRI) wait_for_predecessor();
  if (tid == 0 && (int)blockIdx.x < items) issue(blockIdx.x, false);
  if (tid == 0 && (int)(blockIdx.x + gridDim.x) < items) issue(blockIdx.x + gridDim.x, true);
  prefetch(blockIdx.x);
  int parity = 0;
  unsigned phase = 0;
#pragma unroll 1
  for (int w = blockIdx.x; w < items; w += gridDim.x, parity ^= 1, phase ^= 1u) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    if constexpr (TRI) {
      if (tid == 0) u00s[parity] = (float)pf[0];
    } else if (tid < 32) {
      // u[0,0] from the column blocks' FP64 partial sums: lane-strided, then a
      // fixed shuffle tree (the same order on every call)
      double s2 = 0.0;
      if (A.nparts <= 32 * KPF) {
#pragma unroll
        for (int k = 0; k < KPF; ++k) s2 += pf[k];
      } else {
        const double* pp = reinterpret_cast<const double*>(partial) + (size_t)field * (kMaxRowBlocks / 2);
        for (int i = tid; i < A.nparts; i += 32) s2 += pp[i];
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s2 += __shfl_down_sync(0xffffffffu, s2, o);
      if (tid == 0) u00s[parity] = (float)s2;
    }
    const bool landed = mbar_wait(&bar, phase);
    if (__syncthreads_or(!landed)) {  // the copy never completed: report, let it drain, stop
      if (tid == 0) atomicExch(A.err, kErrBulkWait);
      mbar_wait(&bar, phase);
      if (tid == 0) bulk_store_wait();
      return;
    }
    if constexpr (TRI) {
      if (A.l2res)  // the band's rows of S are in shared memory and dead in global memory: drop their L2 lines
        l2_discard_range(Y + ((size_t)field * A.srows + (size_t)g * RW) * A.ldY, (size_t)RW * A.ldY * sizeof(float2),
                         tid, blockDim.x);
      tri_solve_band<S>(buf, cbuf, cc, g, A);
      __syncthreads();
    }
    const int ia = g * 2 * S::F + 2 * f, ib = ia + 1;
    const bool va = act && ia < A.H, vb = act && ib < A.H;
    float2 v[S::R1];
    if constexpr (TRI) {
      tri_load_pair<S>(v, buf, act ? f : 0, t);
    } else {
    const float2* ya_row = buf + (size_t)(va ? 2 * f : 0) * A.ldY;
    const float2* yb_row = buf + (size_t)(vb ? 2 * f + 1 : 0) * A.ldY;
#pragma unroll
    for (int r = 0; r < S::R1; ++r) {
      // l = t + R2 r with t < R2: whether l lies below or above N/2 is known at
      // compile time except for the one r whose range contains N/2
      const int l = t + S::R2 * r;
      const bool all_lo = S::R2 * r + S::R2 - 1 < half;
      const bool all_hi = S::R2 * r > half;
      const bool lo = all_lo || (!all_hi && l < half);
      const int src = lo ? l : S::N - l;
      float2 ya = va ? ya_row[src] : make_float2(0.0f, 0.0f);
      float2 yb = vb ? yb_row[src] : make_float2(0.0f, 0.0f);
      // bins 0 and N/2 are real in a real transform: drop their imaginary parts
      const bool may_edge = (r == 0) || (!all_lo && !all_hi);
      if (may_edge && (src == 0 || src == half)) {
        ya.y = 0.0f;
        yb.y = 0.0f;
      }
      v[r] = lo ? make_float2(ya.x - yb.y, ya.y + yb.x) : make_float2(ya.x + yb.y, yb.x - ya.y);
    }
    }
    if (act) dft_reg<S::R1, +1>(v);
    __syncthreads();  // every staged row read: buf becomes the exchange buffer
    if (act) {
#pragma unroll
      for (int s2 = 0; s2 < S::R1; ++s2) mybuf[t * S::R1P + s2] = v[s2];
    }
    __syncthreads();
    const bool act2 = act && t < S::JSPAN;
    const float u00 = u00s[parity];
    T* o = out + (size_t)field * A.H * A.W;
    // one stage-2 butterfly per thread: once its inputs are in registers the
    // exchange buffer is free, and the item's output rows are staged there
    // ([2F][W], the output's own row pitch, at its remainder from a 16-byte
    // boundary) and leave by one bulk copy
    const bool stage = S::J2 == 1 && A.stage_out;
    const int r0s = g * 2 * S::F, nrs = (A.H - r0s) < 2 * S::F ? (A.H - r0s) : 2 * S::F;
    T* srows = reinterpret_cast<T*>(buf) + (reinterpret_cast<uintptr_t>(o + (size_t)r0s * A.W) & 15) / sizeof(T);
    // STATS: this thread's stored values as float sums about its first value
    float st_sh = 0.0f, st_s = 0.0f, st_q = 0.0f;
    int st_n = 0;
    auto st_add = [&](float x) {
      if (st_n == 0) st_sh = x;
      const float d = x - st_sh;
      st_s += d;
      st_q = fmaf(d, d, st_q);
      ++st_n;
    };
#pragma unroll
    for (int jj = 0; jj < S::J2; ++jj) {
      const int j = t + S::R2 * jj;
      float2 u[S::R2];
      if (act2) {
        u[0] = mybuf[j];
#pragma unroll
        for (int r = 1; r < S::R2; ++r) u[r] = cmul(mybuf[j + S::R1P * r], cconj(tw2[j * S::R2 + r]));
      }
      if (jj == S::J2 - 1) {
        if (stage) {
          __syncthreads();  // every stage-2 input read: buf takes the output rows
        } else {
          fence_proxy_async_smem();  // this thread's accesses of buf precede the next bulk copy into it
          __syncthreads();           // buf free
          if (tid == 0 && w + (int)gridDim.x < items) issue(w + gridDim.x, false);
          if (tid == 0 && w + 2 * (int)gridDim.x < items) issue(w + 2 * gridDim.x, true);
          prefetch(w + gridDim.x);
        }
      }
      if (act2) {
        dft_reg<S::R2, +1>(u);
#pragma unroll
        for (int s2 = 0; s2 < S::R2; ++s2) {
          const int jc = j + S::R1 * s2 - kP;
          // columns of this stage inside [0, WMIN) for every t need no crop test
          const bool sure = (S::R2 * jj + S::R1 * s2 >= kP) && (S::R2 * jj + S::JSPAN - 1 + S::R1 * s2 - kP < S::WMIN);
          if (sure || (jc >= 0 && jc < A.W)) {
            const T qa = f_from_f<T>(u[s2].x - u00), qb = f_from_f<T>(u[s2].y - u00);
            if (stage) {
              srows[(size_t)(2 * f) * A.W + jc] = qa;
              srows[(size_t)(2 * f + 1) * A.W + jc] = qb;
            } else {
              if (va) o[(size_t)ia * A.W + jc] = qa;
              if (vb) o[(size_t)ib * A.W + jc] = qb;
            }
            if constexpr (STATS) {
              if (va) st_add(f_to_f(qa));
              if (vb) st_add(f_to_f(qb));
            }
          }
        }
      }
    }
    if (stage) {
      fence_proxy_async_smem();  // the staged rows precede the bulk copy that reads them
      __syncthreads();
      if (tid < 32) store_run(o + (size_t)r0s * A.W, srows, (unsigned)(nrs * A.W), tid);
      if (tid == 0) {
        bulk_store_wait_read();  // buf read out: the next item may land in it
        if (w + (int)gridDim.x < items) issue(w + gridDim.x, false);
        if (w + 2 * (int)gridDim.x < items) issue(w + 2 * gridDim.x, true);
      }
      prefetch(w + gridDim.x);
    }
    if constexpr (STATS) {
      // (count, mean, M2) of the thread, combined pairwise (Chan et al.'s update,
      // stable in FP32) down a shuffle tree and across the warps in order; the
      // item's (count, mean, M2) go out in FP64
      float cn = (float)st_n, cm = st_n ? st_sh + st_s / cn : 0.0f, c2 = st_n ? st_q - st_s * (st_s / cn) : 0.0f;
      auto chan = [](float& n, float& m, float& m2, float nb, float mb, float m2b) {
        const float nt = n + nb;
        if (nt > 0.0f) {
          const float d = mb - m, fb = nb / nt;
          m = fmaf(d, fb, m);
          m2 = m2 + m2b + d * d * n * fb;
        }
        n = nt;
      };
#pragma unroll
      for (int o2 = 16; o2 > 0; o2 >>= 1) {
        const float nb = __shfl_xor_sync(0xffffffffu, cn, o2), mb = __shfl_xor_sync(0xffffffffu, cm, o2),
                    m2b = __shfl_xor_sync(0xffffffffu, c2, o2);
        chan(cn, cm, c2, nb, mb, m2b);
      }
      __shared__ float st_red[3 * (S::THREADS / 32)];
      if ((tid & 31) == 0) {
        st_red[3 * (tid >> 5)] = cn;
        st_red[3 * (tid >> 5) + 1] = cm;
        st_red[3 * (tid >> 5) + 2] = c2;
      }
      __syncthreads();
      if (tid == 0) {
        float n = 0.0f, m = 0.0f, m2 = 0.0f;
        for (int k = 0; k < S::THREADS / 32; ++k) chan(n, m, m2, st_red[3 * k], st_red[3 * k + 1], st_red[3 * k + 2]);
        double* dst = reinterpret_cast<double*>(partial) + (size_t)field * (kMaxRowBlocks / 2) + kStatsOff + 3 * g;
        dst[0] = (double)n;
        dst[1] = (double)m;
        dst[2] = (double)m2;
      }
      // st_red is rewritten only after the next item's barriers
    }
  }
  if (tid == 0) bulk_store_wait();  // the last staged rows are stored before the kernel ends
}

// Colour correction of Eq. 25 for fields whose statistics the inverse row pass
// took as it stored them. k_fast_color_finish: one warp per field combines the
// items' (count, mean, M2) in FP64 in a fixed order (lane-strided, then a
// shuffle tree) into the field's mean and population standard deviation and
// writes (mean, gain = ref_std / std or 0 when std = 0, ref_mean) at
// kColorCoef of the field's scratch. k_fast_color_apply maps
// x <- (x - mean) gain + ref_mean, 16 bytes per access where the field allows.
static __global__ void __launch_bounds__(256) k_fast_color_finish(float* __restrict__ partial, int nitems, int nf,
                                                                  const float* __restrict__ ref_mean,
                                                                  const float* __restrict__ ref_std) {
  const int field = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (field >= nf) return;
  const double* pp = reinterpret_cast<const double*>(partial) + (size_t)field * (kMaxRowBlocks / 2) + kStatsOff;
  // N = sum n_i, mean = sum n_i m_i / N, M2 = sum (M2_i + n_i (m_i - mean)^2): one
  // FP64 division a field (pairwise updates of (n, m, M2) take one a step, 2 us each
  // here: 19 us for 24 fields of 120 items, 10 us this way)
  double n = 0.0, s = 0.0, m2 = 0.0;
  for (int i = lane; i < nitems; i += 32) {
    n += pp[3 * i];
    s += pp[3 * i] * pp[3 * i + 1];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    n += __shfl_xor_sync(0xffffffffu, n, o);
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  const double m = n > 0.0 ? s / n : 0.0;
  for (int i = lane; i < nitems; i += 32) {
    const double d = pp[3 * i + 1] - m;
    m2 += pp[3 * i + 2] + pp[3 * i] * (d * d);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
  if (lane == 0) {
    const double sd = n > 0.0 ? sqrt(fmax(m2 / n, 0.0)) : 0.0;
    float* c = partial + (size_t)field * kMaxRowBlocks + kColorCoef;
    c[0] = (float)m;
    c[1] = sd > 0.0 ? (float)((double)ref_std[field] / sd) : 0.0f;
    c[2] = ref_mean[field];
  }
}

template <typename T, int V>
__global__ void __launch_bounds__(256) k_fast_color_apply(T* __restrict__ out, const float* __restrict__ partial,
                                                          long long n) {
  const int field = blockIdx.y;
  const float* c = partial + (size_t)field * kMaxRowBlocks + kColorCoef;
  const float mc = c[0], gsc = c[1], mi = c[2];
  T* x = out + (long long)field * n;
  const long long nv = n / V;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (long long)gridDim.x * blockDim.x) {
    if constexpr (V == 4) {
      float4 v = reinterpret_cast<float4*>(x)[i];
      v.x = fmaf(v.x - mc, gsc, mi);
      v.y = fmaf(v.y - mc, gsc, mi);
      v.z = fmaf(v.z - mc, gsc, mi);
      v.w = fmaf(v.w - mc, gsc, mi);
      reinterpret_cast<float4*>(x)[i] = v;
    } else {
      x[i] = f_from_f<T>(fmaf(f_to_f(x[i]) - mc, gsc, mi));
    }
  }
}

// ---------------------------------------------------------------------------
// adjoint pass C: w = inverse transform of the row-major spectrum Y (rows
// 0..H, torus rows p..p+H). The transpose of the divergence is formed in the
// row-frequency domain, one output row i per transform:
//   grad_gx[i] = F^-1((1 - exp(2 pi i l / N)) Y[i])     (w[i][j] - w[i][j+1])
//   grad_gy[i] = F^-1(Y[i] - Y[i+1])                   (w[i][j] - w[i+1][j])
// Both spectra are Hermitian, so one complex inverse transform of
// A + i B gives grad_gx in its real part and grad_gy in its imaginary part.
// ---------------------------------------------------------------------------
// Recursive column solve, the adjoint's inverse pass side: the F staged rows of
// half-band g of S (and row F, the next half-band's first row) become the inputs
// of the half-band's F inverse transforms, one column per thread. From the
// half-band's two carries: the causal recursion down the half-band, row F from the
// causal value above it and the anticausal carry (which is y' at row F), then the
// anticausal recursion up, U = C_l (y + y' - X); column 0 already holds its exact
// solution. With A_i = d_l U_i (d_l = 1 - exp(2 pi i l / N)) and B_i = U_i - U_(i+1)
// the thread writes A_i + i B_i at l and its Hermitian extension at N - l of
// transform i's buffer, so the transforms read one value per input and the staged
// rows are free for the next item. (Solved in place, they read U_i, U_(i+1) and d
// for every input: five passes over the data against two and a half.) Rows past
// the torus keep X, which is zero there: no output row needs them.
template <class S>
__device__ __forceinline__ void tri_solve_half(const float2* stg, const float2* cbuf, const float2* dtab, float2* buf,
                                               const float* __restrict__ cc, int g, const FastArgs& A) {
  constexpr int F = S::F;
  const int nb = min(F, A.M - A.p - g * F);
  const bool extra = nb == F && g * F + F < A.srows;
  const float2* dcs = reinterpret_cast<const float2*>(cc + (size_t)A.Nh * 8);  // (delta, C) per column
  for (int k = threadIdx.x; k < A.Nh; k += blockDim.x) {
    const float2 dc = __ldg(dcs + k), d = dtab[k];
    float2 yc = cbuf[k], ya = cbuf[S::LDY + k];
    const float2* col = stg + k;
    float2 x[F], y[F];
#pragma unroll
    for (int r = 0; r < F; ++r) x[r] = col[(size_t)r * S::LDY];
    const bool solve = k > 0, edge = k == 0 || 2 * k == S::N;
#pragma unroll
    for (int r = 0; r < F; ++r) {
      if (r < nb) yc = tri_step(x[r], yc, dc.x);
      y[r] = yc;
    }
    float2 un = make_float2(0.0f, 0.0f);  // U of the row below
    if (extra) {
      const float2 xf = col[(size_t)F * S::LDY];
      un = solve ? cscale(csub(cadd(tri_step(xf, yc, dc.x), ya), xf), dc.y) : xf;
    }
    float2* z = buf + k;
#pragma unroll
    for (int r = F - 1; r >= 0; --r) {
      float2 u = x[r];
      if (r < nb) {
        ya = tri_step(x[r], ya, dc.x);
        if (solve) u = cscale(csub(cadd(y[r], ya), x[r]), dc.y);
      }
      float2 p = u, q = un;
      if (edge) p.y = q.y = 0.0f;  // bins 0 and N/2 are real in a real transform
      const float2 a = cmul(p, d), b = csub(p, q);
      if (2 * k < S::N) z[r * S::NP] = make_float2(a.x - b.y, a.y + b.x);
      if (solve) z[r * S::NP + S::N - 2 * k] = make_float2(a.x + b.y, b.x - a.y);
      un = u;
    }
  }
}

// The same with the solved rows U left in place of the staged ones (column 0 kept),
// for transforms that read U_i and U_(i+1) themselves: see PACK_ADJ.
template <class S>
__device__ __forceinline__ void tri_solve_half_rows(float2* stg, const float2* cbuf, const float* __restrict__ cc, int g,
                                               const FastArgs& A) {
  constexpr int F = S::F;
  const int nb = min(F, A.M - A.p - g * F);
  const bool extra = nb == F && g * F + F < A.srows;
  const float2* dcs = reinterpret_cast<const float2*>(cc + (size_t)A.Nh * 8);  // (delta, C) per column
  for (int k = 1 + threadIdx.x; k < A.Nh; k += blockDim.x) {
    const float2 dc = __ldg(dcs + k);
    float2 yc = cbuf[k], ya = cbuf[S::LDY + k];
    float2* col = stg + k;
    float2 x[F + 1];
#pragma unroll
    for (int r = 0; r < F; ++r) x[r] = col[(size_t)r * S::LDY];
    x[F] = extra ? col[(size_t)F * S::LDY] : make_float2(0.0f, 0.0f);
#pragma unroll
    for (int r = 0; r < F; ++r)
      if (r < nb) {
        yc = tri_step(x[r], yc, dc.x);
        col[(size_t)r * S::LDY] = yc;
      }
    if (extra) col[(size_t)F * S::LDY] = cscale(csub(cadd(tri_step(x[F], yc, dc.x), ya), x[F]), dc.y);
#pragma unroll
    for (int r = F - 1; r >= 0; --r)
      if (r < nb) {
        ya = tri_step(x[r], ya, dc.x);
        col[(size_t)r * S::LDY] = cscale(csub(cadd(col[(size_t)r * S::LDY], ya), x[r]), dc.y);
      }
  }
}

// TRI: the recursive column solve's adjoint; Y is then the row-major spectrum
// S of Crop^T(grad_out) (srows rows per field), an item is half-band g (output
// rows gF .. gF + F - 1), whose F + 1 rows of S and two carries arrive by bulk
// copy and are solved before the output transforms, into their inputs
// (tri_solve_half) or in place (tri_solve_half_rows): see PACK_ADJ.
template <class S, typename T, bool TRI = false>
__global__ void __launch_bounds__(S::THREADS, S::MINB_ADJ) k_fast_rows_adj(const float2* __restrict__ Y, T* __restrict__ ggx,
                                                                 T* __restrict__ ggy, const float2* __restrict__ twg,
                                                                 FastArgs A, const float2* __restrict__ tri = nullptr,
                                                                 const float* __restrict__ cc = nullptr) {
  extern __shared__ __align__(16) float2 sm[];
  float2* tw2 = sm;                          // [R1][R2]: w_N^(r j)
  float2* buf = sm + S::R1 * S::R2;          // [F][NP] exchange
  float2* dtab = buf + S::F * S::NP;         // [N/2 + 1] 1 - exp(2 pi i l / N)
  float2* stg = reinterpret_cast<float2*>(reinterpret_cast<char*>(sm) + S::adj_stage_offset());  // [F + 1][ldY]
  float2* cbuf = stg + (size_t)(S::F + 1) * S::LDY;  // TRI: the half-band's carries [2][LDY]
  __shared__ __align__(8) uint64_t bar;
  const int tid = threadIdx.x;
  const int f = tid / S::T, t = tid - f * S::T;
  const bool act = f < S::F;
  const int half = S::N / 2;
  for (int i = tid; i < S::R1 * S::R2; i += blockDim.x) {
    const int j = i / S::R2, r = i - j * S::R2;
    tw2[i] = twg[r * j];
  }
  for (int l = tid; l <= half; l += blockDim.x) {
    // 1 - cos is formed as sin^2 / (1 + cos) where cos > 0, avoiding the
    // cancellation near DC; the imaginary part is -sin
    const float2 e = twg[l];
    const float cs = e.x, sn = -e.y;
    dtab[l] = make_float2((cs > 0.0f) ? __fdividef(sn * sn, 1.0f + cs) : 1.0f - cs, -sn);
  }
  float2* mybuf = buf + (act ? f : 0) * S::NP;
  const int items = A.nf * A.ngroups;
  // one thread: rows gF .. gF + F of Y (fewer at the end of a field); prefetch:
  // only start fetching them into L2, for the copy one item later
  auto issue = [&](int w, bool prefetch) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    const int r0 = g * S::F;
    if constexpr (TRI) {
      const int nr = (A.srows - r0) < S::F + 1 ? (A.srows - r0) : S::F + 1;
      const float2* ys = Y + ((size_t)field * A.srows + r0) * A.ldY;
      const float2* cs = tri + (size_t)field * A.tri_field + (size_t)g * 2 * A.ldY;
      const unsigned nb = (unsigned)(nr * A.ldY * sizeof(float2)), cb = (unsigned)(2 * A.ldY * sizeof(float2));
      if (prefetch) {
        l2_prefetch(ys, nb);
        l2_prefetch(cs, cb);
      } else {
        mbar_expect_tx(&bar, nb + cb);
        bulk_copy(stg, ys, nb, &bar);
        bulk_copy(cbuf, cs, cb, &bar);
      }
      return;
    }
    const int nr = (A.H + 1 - r0) < S::F + 1 ? (A.H + 1 - r0) : S::F + 1;
    const float2* ys = Y + ((size_t)field * (A.H + 1) + r0) * A.ldY;
    const unsigned nb = (unsigned)(nr * A.ldY * sizeof(float2));
    if (prefetch)
      l2_prefetch(ys, nb);
    else
      bulk_load(stg, ys, nb, &bar);
  };
  if (tid == 0) mbar_init(&bar, 1);
  __syncthreads();
  if (tid == 0 && (int)blockIdx.x < items) issue(blockIdx.x, false);
  if (tid == 0 && (int)(blockIdx.x + gridDim.x) < items) issue(blockIdx.x + gridDim.x, true);
  unsigned phase = 0;
#pragma unroll 1
  for (int w = blockIdx.x; w < items; w += gridDim.x, phase ^= 1u) {
    const int field = w / A.ngroups, g = w - field * A.ngroups;
    const int i = g * S::F + f;  // output row of this transform
    const bool vi = act && i < A.H;
    const bool landed = mbar_wait(&bar, phase);
    float2 v[S::R1];
    if constexpr (TRI && S::PACK_ADJ) {
      // (the barrier also ends the previous item's stage 2 with buf)
      if (__syncthreads_or(!landed)) {  // the copies never completed: report, let them drain, stop
        if (tid == 0) atomicExch(A.err, kErrBulkWait);
        mbar_wait(&bar, phase);
        return;
      }
      tri_solve_half<S>(stg, cbuf, dtab, buf, cc, g, A);
      fence_proxy_async_smem();  // this thread's reads of the staged rows precede the next bulk copy
      __syncthreads();           // the transforms' inputs visible; the staged rows read
      if (tid == 0 && w + (int)gridDim.x < items) issue(w + gridDim.x, false);
      if (tid == 0 && w + 2 * (int)gridDim.x < items) issue(w + 2 * gridDim.x, true);
#pragma unroll
      for (int r = 0; r < S::R1; ++r) v[r] = mybuf[t + S::R2 * r];
      __syncthreads();  // every input read: buf becomes the exchange buffer
    } else {
    if constexpr (TRI) {
      if (__syncthreads_or(!landed)) {  // the copies never completed: report, let them drain, stop
        if (tid == 0) atomicExch(A.err, kErrBulkWait);
        mbar_wait(&bar, phase);
        return;
      }
      tri_solve_half_rows<S>(stg, cbuf, cc, g, A);
      __syncthreads();
    }
    const float2* y0 = stg + (size_t)(vi ? f : 0) * A.ldY;
    const float2* y1 = y0 + A.ldY;  // row i + 1 (Y holds H + 1 rows)
#pragma unroll
    for (int r = 0; r < S::R1; ++r) {
      const int l = t + S::R2 * r;
      const bool all_lo = S::R2 * r + S::R2 - 1 < half;
      const bool all_hi = S::R2 * r > half;
      const bool lo = all_lo || (!all_hi && l < half);
      const int src = lo ? l : S::N - l;
      float2 ya = vi ? y0[src] : make_float2(0.0f, 0.0f);
      float2 yb = vi ? y1[src] : make_float2(0.0f, 0.0f);
      const bool may_edge = (r == 0) || (!all_lo && !all_hi);
      if (may_edge && (src == 0 || src == half)) {
        ya.y = 0.0f;
        yb.y = 0.0f;
      }
      const float2 a = cmul(ya, dtab[src]);
      const float2 b = csub(ya, yb);
      v[r] = lo ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, b.x - a.y);
    }
    fence_proxy_async_smem();  // this thread's reads of the staged rows precede the next bulk copy
    if (__syncthreads_or(!landed)) {  // the copy never completed: report, let it drain, stop
      if (tid == 0) atomicExch(A.err, kErrBulkWait);
      mbar_wait(&bar, phase);
      return;
    }
    // every staged row read, and the previous item's stage 2 done with buf
    if (tid == 0 && w + (int)gridDim.x < items) issue(w + gridDim.x, false);
    if (tid == 0 && w + 2 * (int)gridDim.x < items) issue(w + 2 * gridDim.x, true);
    }
    if (act) {
      dft_reg<S::R1, +1>(v);
#pragma unroll
      for (int s2 = 0; s2 < S::R1; ++s2) mybuf[t * S::R1P + s2] = v[s2];
    }
    __syncthreads();
    if (act && t < S::JSPAN && vi) {
      T* ox = ggx + (size_t)field * A.H * A.W + (size_t)i * A.W;
      T* oy = ggy + (size_t)field * A.H * A.W + (size_t)i * A.W;
#pragma unroll
      for (int jj = 0; jj < S::J2; ++jj) {
        const int j = t + S::R2 * jj;
        float2 u[S::R2];
        u[0] = mybuf[j];
#pragma unroll
        for (int r = 1; r < S::R2; ++r) u[r] = cmul(mybuf[j + S::R1P * r], cconj(tw2[j * S::R2 + r]));
        dft_reg<S::R2, +1>(u);
#pragma unroll
        for (int s2 = 0; s2 < S::R2; ++s2) {
          const int jc = j + S::R1 * s2 - kP;
          const bool sure = (S::R2 * jj + S::R1 * s2 >= kP) && (S::R2 * jj + S::JSPAN - 1 + S::R1 * s2 - kP < S::WMIN);
          if (sure || (jc >= 0 && jc < A.W)) {
            ox[jc] = f_from_f<T>(u[s2].x);
            oy[jc] = f_from_f<T>(u[s2].y);
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// host side: one size pair (row schedule RS, column schedule CS)
// ---------------------------------------------------------------------------

// Packed-row buffer elements per field: it holds pass L's packed rows and later
// pass B's row-major output (H + 1 rows for the adjoint).
template <class RS>
size_t fast_zbuf_elems_for(int H) {
  const size_t groups = (size_t)(((H + 2) / 2) + RS::F - 1) / RS::F;
  const size_t packed = groups * RS::F * ((RS::N + 3) & ~3);
  const size_t rows = (size_t)(H + 1) * (((RS::N / 2 + 1) + 3) & ~3);
  return packed > rows ? packed : rows;
}

// Bands of the recursive column solve for an H-row image (the gradient's
// row pairs grouped F at a time: pass A's items).
template <class RS>
int fast_tri_groups_for(int H) {
  return (((H + 2) / 2) + RS::F - 1) / RS::F;
}

// Set the kernel's shared-memory cap (each kernel here has one fixed size) and
// return how many blocks of it fit on the device at once.
template <typename K>
static cudaError_t fast_setup(K kernel, int threads, size_t smem, int* slots) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0, dev = 0, sms = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem)) != cudaSuccess) return e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  *slots = (per_sm > 0 ? per_sm : 1) * sms;
  return cudaSuccess;
}

// Launch a kernel that, with `overlap`, may start while the one ahead of it in the
// stream ends (its reads of that one's results come after wait_for_predecessor):
// the launch latency and the twiddle tables' loads overlap the predecessor's last
// blocks. Taken for short solves (overlap_launches): three fields of 801x1200 41.1
// -> 39.0 us, 48 Laplacians of 512x512 94.3 -> 89.1, 24 thresholded and corrected
// fields of 720x1080 235 -> 220. With it / without, over ten row lengths from 64 to
// 1960, solves and Laplacians in FP32 and BF16, geometric mean (least to most): 12
// million pixels 0.956 (0.90 to 1.005), 24 0.982 (0.94 to 1.028), 36 0.987 (0.97 to
// 1.034), 48 0.987 (0.97 to 1.006), 64 0.989 (0.975 to 1.006), 80 0.990, 100 0.993;
// the ones above 1.01 are N = 1250 at 24 and 36 million. Not for long ones, where it
// gives 1% at most lengths but blocks that start early beside the predecessor's can
// unbalance the persistent grids (100 fields of 801x1200 529 -> 609 us), nor for the
// adjoint (most lengths 3% faster, but 312x312 and 492x492 10 to 13% slower), nor where
// other streams could use the slots that waiting blocks hold (64 ragged images 1746 ->
// 1871).
constexpr double kOverlapMaxPixels = 48e6;
static int overlap_launches(const gfc_plan* P, int nf) {
  return !P->shares_gpu && P->nslots == 1 && (double)nf * P->H * P->W <= kOverlapMaxPixels;
}
template <typename... P, typename... Q>
static cudaError_t launch_after(int overlap, void (*kernel)(P...), dim3 grid, int threads, size_t smem,
                                cudaStream_t st, Q... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// The carry sweep of the chunk's fields over its A.G bands (tables for those bands;
// k_tri_carries' shared-memory cap already raised).
static cudaError_t launch_sweep(float2* spec, float2* tri, const float* cc, const float* powc, double* pd,
                                const FastArgs& A, int nkb, cudaStream_t st) {
  if (A.G <= kTriRegG) {
    const dim3 grid((A.nf * (nkb + 1) + kTriRegWarps - 1) / kTriRegWarps);
    auto k = A.G <= 8 ? k_tri_carries_reg<8> : (A.G <= 16 ? k_tri_carries_reg<16> : k_tri_carries_reg<kTriRegG>);
    return launch_after(A.overlap, k, grid, 32 * kTriRegWarps, 0, st, spec, tri, cc, pd, A, nkb);
  }
  const size_t tsm = A.G <= kTriTileMaxG ? (size_t)2 * A.G * kTriCols * sizeof(float2) : 0;
  return launch_after(A.overlap, k_tri_carries, dim3(nkb + 1, A.nf), 32 * kTriSeg, tsm, st, spec, tri, cc, powc, pd, A);
}

// The fused row pass stages its input rows in the exchange buffers, extended
// where the rows are longer than they are (16-byte spans of FP32 rows against 8
// bytes of each exchange element leave short row pairs a few hundred bytes
// over), as long as the MINB_FWD blocks an SM its registers are planned for
// still fit: fused_smem_cap is that limit (1.5 KB of a block left for its static
// shared memory, 1 KB reserved by the system). Measured on 24 fields of
// 720x1080 (threshold edit): staged 86 us, through packed rows in global memory
// 92 us.
constexpr int kSmemPerSM = 228 * 1024, kSmemBlockMax = 227 * 1024, kSmemBlockExtra = 2560;
template <class S>
constexpr size_t fused_smem_cap() {
  const size_t least = (size_t)S::R1 * S::R2 * sizeof(float2) + fused_exchange_bytes<S>();
  size_t cap = (size_t)(kSmemPerSM / S::MINB_FWD - kSmemBlockExtra) / 16 * 16;
  if (cap > (size_t)(kSmemBlockMax - kSmemBlockExtra)) cap = (size_t)(kSmemBlockMax - kSmemBlockExtra);
  return cap > least ? cap : least;
}
// the fused row pass's shared memory for rows of W, 0 where they are too wide
template <class S, typename T>
static size_t fused_smem(int W, int in) {
  const size_t st = fused_stage_bytes<S, T>(W, in), ex = fused_exchange_bytes<S>();
  const size_t n = (size_t)S::R1 * S::R2 * sizeof(float2) + (st > ex ? st : ex);
  return n <= fused_smem_cap<S>() ? n : 0;
}
// blocks of the fused row pass resident at once: `slots` at the exchange
// buffers' size, fewer where its staging is larger
template <class S>
static int fused_slots(int slots, size_t smem) {
  const size_t ex = (size_t)S::R1 * S::R2 * sizeof(float2) + fused_exchange_bytes<S>();
  if (smem <= ex) return slots;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    return slots;
  const int fit = (int)(kSmemPerSM / (smem + kSmemBlockExtra));
  const int lim = (fit < 1 ? 1 : fit) * sms;
  return lim < slots ? lim : slots;
}
// fast_setup for the fused row pass: occupancy at the exchange buffers' size,
// the shared-memory cap at its limit
template <class S, typename K>
static cudaError_t fused_setup(K kernel, int* slots) {
  const cudaError_t e = fast_setup(kernel, S::THREADS, S::smem_bytes_fwd(), slots);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem_cap<S>());
}

}  // namespace gfc

// the one-launch solve for small tori (thread-block clusters, spectrum kept in
// shared memory), tried first by plain gradient solves below
#include "fused_small.cuh"

namespace gfc {

// The adjoint on a plan with the recursive column solve (reading: the
// transpose of the solve, z = Crop^T(grad_out) - (sum grad_out) e_00 through
// the same Green operator, then the forward differences' transposes): the
// forward row pass packs grad_out into z's rows (row-pair sums for the e_00
// term) and stores S with half-band sums; the carry sweep runs over the
// half-bands with -sum at torus row 0, each of its blocks (warps) reducing the
// row pairs' sums for itself; the adjoint's inverse row pass solves each
// half-band in shared memory and writes grad_gx, grad_gy. Needs grad_out rows
// that fit the forward pass's staging and at most kAdjTotal row pairs; returns
// cudaErrorNotSupported otherwise.
template <class RS, typename T>
static cudaError_t run_fast_adj_tri(gfc_plan* P, const Bufs& bf, const T* gout, T* ggx, T* ggy, int nf,
                                    cudaStream_t st) {
  const size_t smem_a = fused_smem<RS, T>(P->W, kInAdj);
  if (smem_a == 0 || getenv("GFC_UNFUSED_DIV") != nullptr) return cudaErrorNotSupported;
  FastArgs A;
  A.stage_out = 0;
  A.invM = 1.0 / (double)P->M;
  A.invN = 1.0 / (double)P->N;
  A.adj = 1;
  A.l2res = 0;
  A.overlap = 0;
  A.H = P->H; A.W = P->W; A.p = P->pad; A.M = P->M; A.N = P->N; A.Nh = P->Nh; A.ldM = P->ldM;
  A.nrows = P->H;
  A.ncols = P->W;
  A.npairs = (A.nrows + 1) / 2;
  A.ldz = (RS::N + 3) & ~3;
  A.ngroups = P->triG;  // the forward pass's items: the bands of 2F rows
  A.zpairs = A.ngroups * RS::F;
  A.nparts = 0;
  A.nf = nf;
  A.ldY = (P->Nh + 3) & ~3;
  A.err = P->dev_err;
  A.srows = 2 * A.zpairs;
  A.G = P->triGh;       // the sweep's half-bands of F rows
  A.tri_field = P->tri_field;
  const int nkb = (P->Nh + kTriCols - 1) / kTriCols;
  // the row pairs' FP64 sums have kAdjTotal slots a field: taller images (above
  // 2030 to 2045 rows) run the generic adjoint
  if (A.zpairs > kAdjTotal) return cudaErrorNotSupported;
  if ((size_t)2 * RS::F * A.ldY > (size_t)RS::F * RS::NP || (size_t)A.srows * A.ldY > P->spec_field || nkb > kTriCnt)
    return cudaErrorInvalidConfiguration;
  static std::mutex mu;
  static int slots_a = 0, slots_c = 0;
  cudaError_t e;
  {
    std::lock_guard<std::mutex> lock(mu);
    static bool ready = false;
    if (!ready) {
      int unused = 0;
      if ((e = fused_setup<RS>(k_fast_rows_fwd_div<RS, T, kInAdj, true>, &slots_a)) != cudaSuccess) return e;
      if ((e = fast_setup(k_fast_rows_adj<RS, T, true>, RS::THREADS, RS::smem_bytes_adj_tri(), &slots_c)) !=
          cudaSuccess)
        return e;
      if ((e = fast_setup(k_tri_carries, 32 * kTriSeg, (size_t)2 * kTriTileMaxG * kTriCols * sizeof(float2),
                          &unused)) != cudaSuccess)
        return e;
      ready = true;
    }
  }
  const bool one = P->block_items;
  auto grid_for = [one](long items, int slots) { return (int)((one || items < slots) ? items : slots); };
  prof_begin(P, 0, st);
  k_fast_rows_fwd_div<RS, T, kInAdj, true>
      <<<grid_for((long)nf * A.ngroups, fused_slots<RS>(slots_a, smem_a)), RS::THREADS, smem_a, st>>>(
          gout, nullptr, bf.spec, P->twN, bf.partial, A, bf.tri, P->colcoef_h);
  prof_end(P, st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  prof_begin(P, 1, st);
  double* pd = reinterpret_cast<double*>(bf.partial);
  e = launch_sweep(bf.spec, bf.tri, P->colcoef_h, P->powc_h, pd, A, nkb, st);
  prof_end(P, st);
  if (e != cudaSuccess) return e;
  FastArgs C = A;
  C.ngroups = (P->H + RS::F - 1) / RS::F;  // half-bands holding output rows
  prof_begin(P, 2, st);
  k_fast_rows_adj<RS, T, true><<<grid_for((long)nf * C.ngroups, slots_c), RS::THREADS, RS::smem_bytes_adj_tri(),
                                 st>>>(bf.spec, ggx, ggy, P->twN, C, bf.tri, P->colcoef_h);
  prof_end(P, st);
  return cudaGetLastError();
}

// MODE 0: solve from gradient, 1: from Laplacian, 2: adjoint (in0 = grad_out,
// out0 = grad_gx, out1 = grad_gy). Solves (modes 0 and 1) on a plan with the
// recursive column solve run pass A, the carry sweep and pass C; otherwise
// pass A, the column transforms (pass B) and pass C.
template <class RS, class CS, typename T, int MODE>
static cudaError_t run_fast_mode(gfc_plan* P, const Bufs& bf, const T* in0, const T* in1, T* out0, T* out1, int nf,
                                 cudaStream_t st, const EditArgs* ed = nullptr) {
  constexpr bool kCols = !std::is_same_v<CS, NoCols>;  // column transforms compiled for this shape
  // the short lengths and 16-bit storage on the lengths compiled for their rows
  // only: edits go through pass L and there are no statistics (fast_rows_stats);
  // in 16 bits Laplacians go through pass L too and nothing is solved in one
  // launch (half the kernels of a length, of two types)
  constexpr bool kLean16 = !kCols && sizeof(T) == 2;
  constexpr bool kLean = !kCols && (sizeof(T) == 2 || RS::N <= kRowPolicyMin);
  static_assert(!kCols || RS::N <= 2048, "the adjoint packing pass covers a whole row in one block");
  if constexpr (MODE == 0 && !kLean16) {
    if (P->tri && ed == nullptr) {  // plain solves of fields whose spectrum fits a cluster's shared memory
      const cudaError_t ef = run_fused_small<RS, T>(P, in0, in1, out0, nf, st);
      if (ef != cudaErrorNotSupported) return ef;
    }
  }
  if constexpr (MODE == 2) {
    if (P->tri) {  // the adjoint by the recursive column solve where its staging fits
      const cudaError_t ea = run_fast_adj_tri<RS, T>(P, bf, in0, out0, out1, nf, st);
      if (ea != cudaErrorNotSupported || !kCols) return ea;
      if constexpr (kCols)
        if (P->M != CS::M) return ea;  // the row passes of this shape alone
    }
  }
  constexpr bool kTriMode = MODE != 2;
  const bool tri = kTriMode && P->tri;
  if (!kCols && !tri) return cudaErrorNotSupported;
  FastArgs A;
  A.stage_out = 0;
  A.invM = 1.0 / (double)P->M;
  A.invN = 1.0 / (double)P->N;
  A.adj = 0;
  A.l2res = (tri && P->l2res) ? 1 : 0;
  A.overlap = overlap_launches(P, nf);
  A.H = P->H; A.W = P->W; A.p = P->pad; A.M = P->M; A.N = P->N; A.Nh = P->Nh; A.ldM = P->ldM;
  A.nrows = (MODE == 0) ? P->H + 1 : P->H;
  A.ncols = (MODE == 0) ? P->W + 1 : P->W;
  A.npairs = (A.nrows + 1) / 2;
  A.ldz = (RS::N + 3) & ~3;
  A.ngroups = (A.npairs + RS::F - 1) / RS::F;
  if (tri) A.ngroups = P->triG;  // the bands of the column solve: every mode uses the gradient's
  A.zpairs = A.ngroups * RS::F;
  A.nparts = kCols ? (P->Nh + CS::C - 1) / CS::C : 0;
  A.nf = nf;
  A.ldY = (P->Nh + 3) & ~3;
  A.err = P->dev_err;
  A.srows = 2 * A.zpairs;
  A.G = P->triG;
  A.tri_field = P->tri_field;
  // the row passes stage their F packed rows / 2F rows of Y in the exchange buffer
  // (and the column-FFT adjoint sums grad_out per packed row, in kAdjTotal slots)
  if ((size_t)2 * RS::F * A.ldY > (size_t)RS::F * RS::NP || A.ldz > RS::NP || (MODE == 2 && A.zpairs > kAdjTotal))
    return cudaErrorInvalidConfiguration;
  if (tri && (size_t)A.srows * A.ldY > P->spec_field) return cudaErrorInvalidConfiguration;
  if (tri && (P->Nh + kTriCols - 1) / kTriCols > kTriCnt) return cudaErrorInvalidConfiguration;
  static std::mutex mu;
  static int slots_a = 0, slots_b = 0, slots_c = 0, slots_d = 0, slots_ta = 0, slots_tc = 0, slots_td = 0,
             slots_ts = 0, slots_tde = 0;
  cudaError_t e;
  {
    std::lock_guard<std::mutex> lock(mu);
    static bool ready = false;
    if (!ready) {
      int unused = 0;
      if ((e = fast_setup(k_fast_div<T, MODE>, 512, 0, &unused)) != cudaSuccess) return e;
      if constexpr (kCols) {
        if ((e = fast_setup(k_fast_cols<CS, MODE>, CS::THREADS, CS::smem_bytes(), &slots_b)) != cudaSuccess) return e;
        if constexpr (MODE == 2) {
          if ((e = fast_setup(k_fast_rows_adj<RS, T>, RS::THREADS, RS::smem_bytes_adj(), &slots_c)) != cudaSuccess)
            return e;
        } else {
          if ((e = fast_setup(k_fast_rows_inv<RS, T, false, false>, RS::THREADS, RS::smem_bytes(), &slots_c)) !=
              cudaSuccess)
            return e;
        }
        if ((e = fast_setup(k_fast_rows_fwd<RS, false>, RS::THREADS, RS::smem_bytes_fwd(), &slots_a)) != cudaSuccess)
          return e;
        if constexpr (MODE != 1)
          if ((e = fused_setup<RS>(k_fast_rows_fwd_div<RS, T, MODE, false>, &slots_d)) != cudaSuccess) return e;
      }
      if constexpr (MODE != 2) {
        int unused_k = 0;
        if ((e = fast_setup(k_tri_carries, 32 * kTriSeg, (size_t)2 * kTriTileMaxG * kTriCols * sizeof(float2),
                            &unused_k)) != cudaSuccess)
          return e;
        if ((e = fast_setup(k_fast_rows_inv<RS, T, true, false>, RS::THREADS, RS::smem_bytes_tri_inv(), &slots_tc)) !=
            cudaSuccess)
          return e;
        if ((e = fast_setup(k_fast_rows_fwd<RS, true>, RS::THREADS, RS::smem_bytes_fwd(), &slots_ta)) != cudaSuccess)
          return e;
        if constexpr (MODE == 0 || !kLean16)
          if ((e = fused_setup<RS>(k_fast_rows_fwd_div<RS, T, MODE, true>, &slots_td)) != cudaSuccess) return e;
      }
      if constexpr (MODE == 0 && !kLean) {
        if ((e = fast_setup(k_fast_rows_inv<RS, T, true, true>, RS::THREADS, RS::smem_bytes_tri_inv(), &slots_ts)) !=
            cudaSuccess)
          return e;
        if ((e = fused_setup<RS>(k_fast_rows_fwd_div<RS, T, kInGrad, true, kEditThreshold>, &slots_tde)) != cudaSuccess)
          return e;
      }
      ready = true;
    }
  }
  // persistent grids (as many blocks as fit, each looping over items), or one block per item
  const bool one = P->block_items;
  auto grid_for = [one](long items, int slots) { return (int)((one || items < slots) ? items : slots); };
  // Plain gradient solves, Laplacian solves and the adjoint fold pass L (the
  // adjoint: its packing of grad_out with the row-pair sums) into the row pass
  // when the staged rows fit its shared memory.
  const size_t smem_f = fused_smem<RS, T>(P->W, MODE);
  const int edit_kind = (MODE == 0 && ed) ? ed->kind : kEditNone;
  // the threshold edit is staged with the gradient (recursive column solve plans)
  const bool fused_edit = edit_kind == kEditThreshold && tri && !kLean;
  const bool fused_div = (MODE != 1 || (tri && !kLean16)) && (edit_kind == kEditNone || fused_edit) && smem_f != 0 &&
                         getenv("GFC_UNFUSED_DIV") == nullptr;
  const long a_items = (long)nf * A.ngroups;
  if (fused_div) {
    prof_begin(P, 0, st);
    if constexpr (MODE != 2) {
      if (fused_edit) {
        if constexpr (MODE == 0 && !kLean)
          k_fast_rows_fwd_div<RS, T, kInGrad, true, kEditThreshold>
              <<<grid_for(a_items, fused_slots<RS>(slots_tde, smem_f)), RS::THREADS, smem_f, st>>>(
                  in0, in1, bf.spec, P->twN, bf.partial, A, bf.tri, P->colcoef, ed->t2);
      } else if (tri) {
        if constexpr (MODE == 0 || !kLean16)
          k_fast_rows_fwd_div<RS, T, MODE, true>
              <<<grid_for(a_items, fused_slots<RS>(slots_td, smem_f)), RS::THREADS, smem_f, st>>>(
                  in0, in1, bf.spec, P->twN, bf.partial, A, bf.tri, P->colcoef);
      } else if constexpr (kCols && MODE == 0) {
        k_fast_rows_fwd_div<RS, T, kInGrad, false>
            <<<grid_for(a_items, fused_slots<RS>(slots_d, smem_f)), RS::THREADS, smem_f, st>>>(
                in0, in1, bf.spec, P->twN, bf.partial, A, nullptr, nullptr);
      }
    } else if constexpr (kCols) {
      k_fast_rows_fwd_div<RS, T, kInAdj, false>
          <<<grid_for(a_items, fused_slots<RS>(slots_d, smem_f)), RS::THREADS, smem_f, st>>>(
              in0, in1, bf.spec, P->twN, bf.partial, A, nullptr, nullptr);
    }
    prof_end(P, st);
  }
  if (!fused_div) prof_begin(P, 3, st);
  {
    const int nq = A.ldz / 4;
    const int bx = (MODE == 2) ? ((nq + 31) / 32) * 32 : (nq >= 256 ? 256 : ((nq + 31) / 32) * 32);
    const dim3 grid((nq + bx - 1) / bx, A.zpairs, nf);
    const int kind = fused_div ? kEditNone : edit_kind;  // a fused edit needs no pass L
    const int ex = ((nq + 31) / 32) * 32 <= 512 ? ((nq + 31) / 32) * 32 : 256;  // whole warps
    const dim3 egrid((nq + ex - 1) / ex, (A.zpairs + kEditPairs - 1) / kEditPairs, nf);
    if (kind == kEditThreshold)
      k_fast_div_edit<T, kEditThreshold><<<egrid, ex, 0, st>>>(in0, in1, nullptr, ed->t2, 0.0f, bf.zbuf, A);
    else if (kind == kEditMerge)
      k_fast_div_edit<T, kEditMerge><<<egrid, ex, 0, st>>>(in0, in1, static_cast<const T*>(ed->edges), nullptr,
                                                           ed->alpha, bf.zbuf, A);
    else if (!fused_div)
      k_fast_div<T, MODE><<<grid, bx, 0, st>>>(in0, in1, bf.zbuf, bf.partial, A);
  }
  if (!fused_div) {
    prof_end(P, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    prof_begin(P, 0, st);
    if (tri)
      k_fast_rows_fwd<RS, true><<<grid_for(a_items, slots_ta), RS::THREADS, RS::smem_bytes_fwd(), st>>>(
          bf.zbuf, bf.spec, P->twN, A, bf.tri, P->colcoef, bf.partial);
    else if constexpr (kCols)
      k_fast_rows_fwd<RS, false><<<grid_for(a_items, slots_a), RS::THREADS, RS::smem_bytes_fwd(), st>>>(
          bf.zbuf, bf.spec, P->twN, A, nullptr, nullptr);
    prof_end(P, st);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  prof_begin(P, 1, st);
  const int nkb = (P->Nh + kTriCols - 1) / kTriCols;  // column blocks of the sweep (u[0,0] partials)
  if (tri) {
    e = launch_sweep(bf.spec, bf.tri, P->colcoef, P->powc, reinterpret_cast<double*>(bf.partial), A, nkb, st);
  } else if constexpr (kCols) {
    if (MODE == 2) {
      k_adj_total<<<nf, 32, 0, st>>>(reinterpret_cast<double*>(bf.partial), A.zpairs);
      P->prof.launches[1] += 1;  // a second launch in this pass
    }
    k_fast_cols<CS, MODE><<<grid_for((long)nf * A.nparts, slots_b), CS::THREADS, CS::smem_bytes(), st>>>(
        bf.spec, bf.zbuf, P->GT, P->twM, bf.partial, A);
  }
  prof_end(P, st);
  if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
  FastArgs C = A;
  // the inverse row pass stages its output rows in its exchange buffer and
  // stores them by bulk copy
  C.stage_out = MODE != 2 && run_bytes<T>((size_t)2 * RS::F * P->W) <= (size_t)RS::F * RS::NP * sizeof(float2);
  prof_begin(P, 2, st);
  if constexpr (MODE == 2) {
    C.ngroups = (P->H + RS::F - 1) / RS::F;
    k_fast_rows_adj<RS, T><<<grid_for((long)nf * C.ngroups, slots_c), RS::THREADS, RS::smem_bytes_adj(), st>>>(
        bf.zbuf, out0, out1, P->twN, C);
  } else {
    (void)out1;
    C.ngroups = ((P->H + 1) / 2 + RS::F - 1) / RS::F;
    const bool stats = MODE == 0 && !kLean && tri && ed && ed->ref_mean;  // (fast_rows_stats)
    if (stats) {
      C.nparts = nkb;
      if constexpr (MODE == 0 && !kLean)
        e = launch_after(A.overlap, k_fast_rows_inv<RS, T, true, true>, dim3(grid_for((long)nf * C.ngroups, slots_ts)),
                         RS::THREADS, RS::smem_bytes_tri_inv(), st, bf.spec, bf.partial, out0, P->twN, C, bf.tri,
                         P->colcoef);
    } else if (tri) {
      C.nparts = nkb;
      e = launch_after(A.overlap, k_fast_rows_inv<RS, T, true, false>, dim3(grid_for((long)nf * C.ngroups, slots_tc)),
                       RS::THREADS, RS::smem_bytes_tri_inv(), st, bf.spec, bf.partial, out0, P->twN, C, bf.tri,
                       P->colcoef);
    } else if constexpr (kCols) {
      k_fast_rows_inv<RS, T, false, false>
          <<<grid_for((long)nf * C.ngroups, slots_c), RS::THREADS, RS::smem_bytes(), st>>>(
              bf.zbuf, bf.partial, out0, P->twN, C, nullptr, nullptr);
    }
    if (stats) {
      prof_end(P, st);
      if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
      prof_begin(P, 3, st);  // counted with the other non-transform pass
      const long long n = (long long)P->H * P->W;
      k_fast_color_finish<<<(nf + 7) / 8, 256, 0, st>>>(bf.partial, C.ngroups, nf, ed->ref_mean, ed->ref_std);
      const bool v4 = sizeof(T) == 4 && n % 4 == 0 && (reinterpret_cast<uintptr_t>(out0) & 15) == 0;
      const long long per = v4 ? n / 4 : n;
      int nblk = (int)((per + 256 * 8 - 1) / (256 * 8));
      if (nblk < 1) nblk = 1;
      if (v4)
        k_fast_color_apply<T, 4><<<dim3(nblk, nf), 256, 0, st>>>(out0, bf.partial, n);
      else
        k_fast_color_apply<T, 1><<<dim3(nblk, nf), 256, 0, st>>>(out0, bf.partial, n);
    }
  }
  prof_end(P, st);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Shapes compiled for their row length only (the recursive column solve needs
// no column kernels); the caller falls back to the generic passes for anything
// else (cudaErrorNotSupported).
template <class RS, typename T>
cudaError_t run_rows_shape(gfc_plan* P, const Bufs& bf, int mode, const void* in0, const void* in1, void* out0,
                           void* out1, int nf, cudaStream_t st, const EditArgs* ed) {
  if (!P->tri) return cudaErrorNotSupported;
  const T* a = static_cast<const T*>(in0);
  const T* b = static_cast<const T*>(in1);
  T* o0 = static_cast<T*>(out0);
  T* o1 = static_cast<T*>(out1);
  if (mode == 0) return run_fast_mode<RS, NoCols, T, 0>(P, bf, a, b, o0, o1, nf, st, ed);
  if (mode == 2) return run_fast_mode<RS, NoCols, T, 2>(P, bf, a, b, o0, o1, nf, st);
  return run_fast_mode<RS, NoCols, T, 1>(P, bf, a, b, o0, o1, nf, st);
}

template <class RS, class CS>
cudaError_t run_fast_shape(gfc_plan* P, const Bufs& bf, int mode, const void* in0, const void* in1, void* out0,
                           void* out1, int nf, cudaStream_t st, const EditArgs* ed) {
  auto go = [&](auto tag) -> cudaError_t {
    using T = decltype(tag);
    const T* a = static_cast<const T*>(in0);
    const T* b = static_cast<const T*>(in1);
    T* o0 = static_cast<T*>(out0);
    T* o1 = static_cast<T*>(out1);
    if (mode == 0) return run_fast_mode<RS, CS, T, 0>(P, bf, a, b, o0, o1, nf, st, ed);
    if (mode == 1) return run_fast_mode<RS, CS, T, 1>(P, bf, a, b, o0, o1, nf, st);
    return run_fast_mode<RS, CS, T, 2>(P, bf, a, b, o0, o1, nf, st);
  };
  switch (P->dtype) {
    case GFC_F32: return go(float{});
    case GFC_F16: return go(__half{});
    default: return go(__nv_bfloat16{});
  }
}

}  // namespace gfc
