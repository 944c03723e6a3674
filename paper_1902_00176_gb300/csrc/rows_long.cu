// rows_long.cu -- row passes for row lengths above the compiled ones (images wider
// than 2050 pixels), for solves with the recursive column solve: three kernels
// per chunk, as in fast_kernels.cuh, with the schedule of the length chosen at
// run time.
//
// A row length N = R1 R2 R3 (radices 7 .. 25, N / R <= kLongThreads: all but 3430
// and 4000 of the 46 lengths from 2060 to 4096) is
// transformed in shared memory by one block of kLongThreads threads, one
// butterfly per thread and stage, its R values in registers between the two
// barriers of a stage, so one buffer of N values serves a transform. An item is
// kLongF row pairs (a band of 4 rows): two buffers and the twiddle table (100 KB at
// N = 3888), two blocks per SM.
//
// What bounds it: shared memory (a transform's values cross it eight times) and
// the barriers between the stages. The generic passes these replace run a
// transform of 3888 in seven radix-2 .. 8 stages over two buffers and a table
// (93 KB a transform) and transform every column twice: 345 + 295 + 231 us for
// three fields of 2160x3840.
#include "fast_kernels.cuh"

namespace gfc {
namespace {

constexpr int kLongThreads = 384;
constexpr int kLongF = 2;          // row pairs per item
constexpr int kLongMin = 2058;     // the longest compiled row length
// column length from which these passes serve: thinner strips have few bands and
// errors (relative L2 against 64 bits) above the generic passes' there: 5x2051
// 5.1e-6 against 1.2e-6, 3x3912 5.5e-5 against 9.3e-6; 21x3064 1.5e-6 against
// 1.2e-5, 33x2736 1.6e-6 against 7.3e-6, 700x3840 7.7e-7 against 3.2e-6
constexpr int kLongMinM = 24;

struct LongPlan {
  int n, r1, r2, r3;
  int p1;   // stride of a first-stage butterfly's outputs: odd, so that they spread over the banks
  int len;  // elements of a transform's buffer
};

constexpr int kLongRadices[] = {7, 9, 10, 12, 14, 15, 16, 18, 20, 21, 25};

bool is_long_radix(int r) {
  for (int x : kLongRadices)
    if (x == r) return true;
  return false;
}

// the schedule of a length: the one whose smallest radix is largest (the fewest
// butterflies of the fullest stage), the widest stages last
bool long_plan(int n, LongPlan* out) {
  if (n <= kLongMin || n > kMaxFftLen || (n & 1)) return false;
  int best = 0;
  for (int a : kLongRadices)
    for (int b : kLongRadices) {
      if (n % (a * b) != 0) continue;
      const int c = n / (a * b);
      if (!is_long_radix(c) || a > b || b > c || n / a > kLongThreads || a <= best) continue;
      best = a;
      out->n = n;
      out->r1 = a;
      out->r2 = b;
      out->r3 = c;
      out->p1 = a | 1;
      out->len = ((n / a) * out->p1 + 1) & ~1;
    }
  return best > 0;
}

// The twiddle table in shared memory, one spare slot every 16 elements: stage
// strides of 8 and 16 would otherwise meet in one bank. Every power is read from
// the table: formed as products they double the transform's rounding error, which
// the near-DC bins of the solve amplify by up to (N / 2 pi)^2.
__host__ __device__ constexpr int tw_slot(int m) { return m + (m >> 4); }

// v[r] *= w^r, r < R, w = the DIR root of index t
template <int R, int DIR>
__device__ __forceinline__ void long_twiddle(float2 (&v)[R], const float2* tw, int t) {
#pragma unroll
  for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw_dir<DIR>(tw[tw_slot(r * t)]));
}

// One stage of the transform in buf (Stockham, natural order in and out; between
// the first two stages element m = g R1 + s lies at g p1 + s). Every thread
// enters; ends with a barrier.
template <int R, int DIR>
__device__ __forceinline__ void long_stage(float2* buf, int stage, const LongPlan& L, const float2* tw) {
  const int nb = L.n / R;
  const bool act = (int)threadIdx.x < nb;
  const int j = act ? (int)threadIdx.x : 0;  // (the idle threads read butterfly 0 and store nothing)
  const int g = stage == 1 ? j / L.r1 : 0, k = stage == 1 ? j - g * L.r1 : j;
  float2 v[R];
  const float2* src = buf + (stage == 1 ? g * L.p1 + k : j);
  const int rstep = stage == 1 ? L.r3 * L.p1 : nb;
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = src[r * rstep];
  if (stage) long_twiddle<R, DIR>(v, tw, stage == 1 ? k * L.r3 : k);
  dft_reg<R, DIR>(v);
  __syncthreads();  // every value read
  if (act) {
    float2* dst = buf + (stage == 0 ? j * L.p1 : (stage == 1 ? g * L.r1 * R + k : j));
    const int step = stage == 0 ? 1 : (stage == 1 ? L.r1 : nb);
#pragma unroll
    for (int s = 0; s < R; ++s) dst[s * step] = v[s];
  }
  __syncthreads();
}

template <int DIR>
__device__ __noinline__ void long_fft(float2* buf, LongPlan L, const float2* tw) {
#pragma unroll 1
  for (int stage = 0; stage < 3; ++stage) {
    const int R = stage == 0 ? L.r1 : (stage == 1 ? L.r2 : L.r3);
    switch (R) {
      case 7: long_stage<7, DIR>(buf, stage, L, tw); break;
      case 9: long_stage<9, DIR>(buf, stage, L, tw); break;
      case 10: long_stage<10, DIR>(buf, stage, L, tw); break;
      case 12: long_stage<12, DIR>(buf, stage, L, tw); break;
      case 14: long_stage<14, DIR>(buf, stage, L, tw); break;
      case 15: long_stage<15, DIR>(buf, stage, L, tw); break;
      case 16: long_stage<16, DIR>(buf, stage, L, tw); break;
      case 18: long_stage<18, DIR>(buf, stage, L, tw); break;
      case 20: long_stage<20, DIR>(buf, stage, L, tw); break;
      case 21: long_stage<21, DIR>(buf, stage, L, tw); break;
      default: long_stage<25, DIR>(buf, stage, L, tw); break;
    }
  }
}

// Forward: one block per band of 4 rows. The divergence (or the given
// Laplacian) is formed from global memory, the rows' spectra and the band's
// sums go out as tri_store_item writes them.
template <typename T, int IN>
__global__ void __launch_bounds__(kLongThreads, 2) k_long_fwd(const T* __restrict__ in0, const T* __restrict__ in1,
                                                              float2* __restrict__ spec,
                                                              const float2* __restrict__ twg,
                                                              double* __restrict__ partial, FastArgs A, LongPlan L,
                                                              float2* __restrict__ tri, const float* __restrict__ cc) {
  extern __shared__ __align__(16) float2 sm[];
  constexpr int RW = 2 * kLongF;
  const int tid = threadIdx.x;
  float2* tw = sm + kLongF * L.len;
  for (int m = tid; m < L.n; m += kLongThreads) tw[tw_slot(m)] = twg[m];
  const int field = blockIdx.x / A.ngroups, g = blockIdx.x - field * A.ngroups;
  const size_t fe = (size_t)A.H * A.W;
  const T* a = in0 + field * fe;
  const T* b = IN == kInGrad ? in1 + field * fe : nullptr;
  if (g == 0 && tid == 0)  // the sweep's count of finished blocks for this field starts at 0
    reinterpret_cast<unsigned*>(partial + (size_t)field * (kMaxRowBlocks / 2) + kTriCnt)[0] = 0u;
  // the band's rows r0 .. r0 + 3 (and gy of the row above), four columns' loads in flight
  const int r0 = g * RW;
  const T* x0 = a + (size_t)r0 * A.W;
  const T* y0 = IN == kInGrad ? b + (size_t)r0 * A.W : nullptr;
#pragma unroll 2
  for (int c = tid; c < L.n; c += kLongThreads) {
    const int j = c - kP;
    float l[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) l[r] = 0.0f;
    if (j >= 0 && j < A.W) {
      if constexpr (IN == kInGrad) {
        float x1[RW], xm[RW], y1[RW + 1];
        y1[0] = r0 >= 1 && r0 <= A.H ? f_to_f(y0[j - A.W]) : 0.0f;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
          const bool h = r0 + r < A.H;
          x1[r] = h ? f_to_f(x0[(size_t)r * A.W + j]) : 0.0f;
          xm[r] = h && j > 0 ? f_to_f(x0[(size_t)r * A.W + j - 1]) : 0.0f;
          y1[r + 1] = h ? f_to_f(y0[(size_t)r * A.W + j]) : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < RW; ++r) l[r] = (x1[r] - xm[r]) + (y1[r + 1] - y1[r]);
      } else {
#pragma unroll
        for (int r = 0; r < RW; ++r) l[r] = r0 + r < A.H ? f_to_f(x0[(size_t)r * A.W + j]) : 0.0f;
      }
    } else if (IN == kInGrad && j == A.W) {  // the column after the image: -gx of its last one
#pragma unroll
      for (int r = 0; r < RW; ++r) l[r] = r0 + r < A.H ? 0.0f - f_to_f(x0[(size_t)r * A.W + j - 1]) : 0.0f;
    }
#pragma unroll
    for (int f = 0; f < kLongF; ++f) sm[f * L.len + c] = make_float2(l[2 * f], l[2 * f + 1]);
  }
  __syncthreads();
#pragma unroll 1
  for (int f = 0; f < kLongF; ++f) long_fft<-1>(sm + f * L.len, L, tw);
  float2* Sr = spec + ((size_t)field * A.srows + (size_t)g * RW) * A.ldY;
  float2* sums = tri_sums(tri, field, A);
  const int nb = min(RW, A.M - A.p - g * RW);
  for (int k = tid; k < A.Nh; k += kLongThreads) {
    const int km = k == 0 ? 0 : L.n - k;
    float2 x[RW];
#pragma unroll
    for (int q = 0; q < kLongF; ++q) {
      const float2 zk = sm[q * L.len + k], zm = sm[q * L.len + km];
      const float2 zc = make_float2(zm.x, -zm.y);
      x[2 * q] = cscale(cadd(zk, zc), 0.5f);
      const float2 d = csub(zk, zc);
      x[2 * q + 1] = cscale(make_float2(d.y, -d.x), 0.5f);
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) Sr[(size_t)r * A.ldY + k] = x[r];
    if (k == 0) {
      float* c0 = tri_col0(tri, field, A) + (size_t)g * RW;
#pragma unroll
      for (int r = 0; r < RW; ++r) c0[r] = x[r].x;
    }
    const float dl = __ldg(cc + (size_t)k * 8);
    float2 e = make_float2(0.0f, 0.0f), ep = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int r = 0; r < RW; ++r)
      if (r < nb) e = tri_step(x[r], e, dl);
#pragma unroll
    for (int r = RW - 1; r >= 0; --r)
      if (r < nb) ep = tri_step(x[r], ep, dl);
    float2* te = sums + ((size_t)(k / kTriCols) * A.G + g) * 2 * kTriCols + (k % kTriCols);
    te[0] = e;
    te[kTriCols] = ep;
  }
}

// Inverse: the band's rows of S solved column by column in registers
// (tri_solve_band's recursions), the Hermitian extension of each row pair
// written straight into its transform's buffer, inverse transforms, offset,
// crop and cast.
template <typename T>
__global__ void __launch_bounds__(kLongThreads, 2) k_long_inv(const float2* S, const double* partial,
                                                              T* __restrict__ out, const float2* __restrict__ twg,
                                                              FastArgs A, LongPlan L, const float2* tri,
                                                              const float* __restrict__ cc) {
  extern __shared__ __align__(16) float2 sm[];
  constexpr int RW = 2 * kLongF;
  const int tid = threadIdx.x;
  float2* tw = sm + kLongF * L.len;
  for (int m = tid; m < L.n; m += kLongThreads) tw[tw_slot(m)] = twg[m];
  const int field = blockIdx.x / A.ngroups, g = blockIdx.x - field * A.ngroups;
  const float u00 = (float)__ldcg(partial + (size_t)field * (kMaxRowBlocks / 2) + kTriU00);
  const float2* Sr = S + ((size_t)field * A.srows + (size_t)g * RW) * A.ldY;
  const float2* car = tri + (size_t)field * A.tri_field + (size_t)g * 2 * A.ldY;
  const float2* dcs = reinterpret_cast<const float2*>(cc + (size_t)A.Nh * 8);  // (delta, C) per column
  const int nb = min(RW, A.M - A.p - g * RW);
  for (int k = tid; k < A.Nh; k += kLongThreads) {
    float2 x[RW], u[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) x[r] = __ldcg(Sr + (size_t)r * A.ldY + k);
    if (k == 0) {  // holds its exact solution
#pragma unroll
      for (int r = 0; r < RW; ++r) u[r] = x[r];
    } else {
      const float2 dc = __ldg(dcs + k);
      float2 yc = __ldcg(car + k), ya = __ldcg(car + A.ldY + k);
#pragma unroll
      for (int r = 0; r < RW; ++r) {
        if (r < nb) yc = tri_step(x[r], yc, dc.x);
        u[r] = yc;
      }
#pragma unroll
      for (int r = RW - 1; r >= 0; --r)
        if (r < nb) {
          ya = tri_step(x[r], ya, dc.x);
          u[r] = cscale(csub(cadd(u[r], ya), x[r]), dc.y);
        }
    }
    const bool edge = k == 0 || 2 * k == L.n;  // bins 0 and N/2 are real in a real transform
#pragma unroll
    for (int f = 0; f < kLongF; ++f) {
      float2 ya = u[2 * f], yb = u[2 * f + 1];
      if (edge) ya.y = yb.y = 0.0f;
      float2* z = sm + f * L.len;
      z[k] = make_float2(ya.x - yb.y, ya.y + yb.x);
      if (!edge) z[L.n - k] = make_float2(ya.x + yb.y, yb.x - ya.y);
    }
  }
  __syncthreads();
  T* o = out + (size_t)field * A.H * A.W;
#pragma unroll 1
  for (int f = 0; f < kLongF; ++f) {
    const int ia = g * RW + 2 * f, ib = ia + 1;
    if (ia >= A.H) break;  // (the same for every thread)
    const float2* z = sm + f * L.len;
    long_fft<+1>(sm + f * L.len, L, tw);
    for (int j = tid; j < A.W; j += kLongThreads) {
      const float2 v = z[j + kP];
      o[(size_t)ia * A.W + j] = f_from_f<T>(v.x - u00);
      if (ib < A.H) o[(size_t)ib * A.W + j] = f_from_f<T>(v.y - u00);
    }
  }
}

// Shared memory of a block, and the most that any length takes (N = 4096).
size_t long_smem(const LongPlan& L) { return ((size_t)kLongF * L.len + tw_slot(L.n)) * sizeof(float2); }
constexpr int kLongSmemMax = 104448;

// Raise the kernels' shared-memory limits, once per device and storage type, to
// what the longest rows need: the attribute is set, not raised, and the modes
// share the inverse kernel, so a limit set by length would lower another plan's.
template <typename T>
cudaError_t long_setup(int device) {
  constexpr int kDevices = 64;
  static std::mutex mu;
  static bool ready[kDevices] = {};
  std::lock_guard<std::mutex> lock(mu);
  const bool known = device >= 0 && device < kDevices;
  if (known && ready[device]) return cudaSuccess;
  auto raise = [](auto kernel, int bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  cudaError_t e = raise(k_long_fwd<T, 0>, kLongSmemMax);
  if (e == cudaSuccess) e = raise(k_long_fwd<T, 1>, kLongSmemMax);
  if (e == cudaSuccess) e = raise(k_long_inv<T>, kLongSmemMax);
  if (e == cudaSuccess) e = raise(k_tri_carries, (int)((size_t)2 * kTriTileMaxG * kTriCols * sizeof(float2)));
  if (e == cudaSuccess && known) ready[device] = true;
  return e;
}

template <typename T, int MODE>
cudaError_t run_long(gfc_plan* P, const Bufs& bf, const T* in0, const T* in1, T* out, int nf, cudaStream_t st) {
  LongPlan L;
  if (!long_plan(P->N, &L)) return cudaErrorNotSupported;
  FastArgs A;
  A.stage_out = 0;
  A.invM = 1.0 / (double)P->M;
  A.invN = 1.0 / (double)P->N;
  A.adj = 0;
  A.l2res = 0;
  A.overlap = 0;  // (one field of 2160x3840: 337 us without, 345 with)
  A.H = P->H; A.W = P->W; A.p = P->pad; A.M = P->M; A.N = P->N; A.Nh = P->Nh; A.ldM = P->ldM;
  A.nrows = (MODE == 0) ? P->H + 1 : P->H;
  A.ncols = (MODE == 0) ? P->W + 1 : P->W;
  A.npairs = (A.nrows + 1) / 2;
  A.ldz = 0;
  A.ngroups = A.G = P->triG;
  A.zpairs = A.G * kLongF;
  A.nparts = 0;
  A.nf = nf;
  A.ldY = (P->Nh + 3) & ~3;
  A.err = P->dev_err;
  A.srows = 2 * A.zpairs;
  A.tri_field = P->tri_field;
  const int nkb = (P->Nh + kTriCols - 1) / kTriCols;
  if ((size_t)A.srows * A.ldY > P->spec_field || nkb > kTriCnt) return cudaErrorInvalidConfiguration;
  const size_t smem = long_smem(L);
  if (smem > (size_t)kLongSmemMax) return cudaErrorInvalidConfiguration;
  double* pd = reinterpret_cast<double*>(bf.partial);
  cudaError_t e = long_setup<T>(P->device);
  if (e != cudaSuccess) return e;
  prof_begin(P, 0, st);
  k_long_fwd<T, MODE><<<(unsigned)((long)nf * A.G), kLongThreads, smem, st>>>(in0, in1, bf.spec, P->twN, pd, A, L,
                                                                              bf.tri, P->colcoef);
  prof_end(P, st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  prof_begin(P, 1, st);
  e = launch_sweep(bf.spec, bf.tri, P->colcoef, P->powc, pd, A, nkb, st);
  prof_end(P, st);
  if (e != cudaSuccess) return e;
  FastArgs C = A;
  C.ngroups = ((P->H + 1) / 2 + kLongF - 1) / kLongF;
  prof_begin(P, 2, st);
  k_long_inv<T><<<(unsigned)((long)nf * C.ngroups), kLongThreads, smem, st>>>(bf.spec, pd, out, P->twN, C, L, bf.tri,
                                                                              P->colcoef);
  prof_end(P, st);
  return cudaGetLastError();
}

}  // namespace

bool long_rows_supported(int M, int N) {
  LongPlan L;
  return M >= kLongMinM && long_plan(N, &L);
}

int long_rows_items() { return kLongF; }

// plain solves only; edits and the adjoint run the generic passes
cudaError_t run_long_rows(gfc_plan* P, const Bufs& bf, int mode, const void* in0, const void* in1, void* out0, int nf,
                          cudaStream_t st, const EditArgs* ed) {
  if (!P->tri || mode == 2 || ed != nullptr) return cudaErrorNotSupported;
  auto go = [&](auto tag) -> cudaError_t {
    using T = decltype(tag);
    const T* a = static_cast<const T*>(in0);
    if (mode == 1) return run_long<T, 1>(P, bf, a, nullptr, static_cast<T*>(out0), nf, st);
    return run_long<T, 0>(P, bf, a, static_cast<const T*>(in1), static_cast<T*>(out0), nf, st);
  };
  switch (P->dtype) {
    case GFC_F32: return go(float{});
    case GFC_F16: return go(__half{});
    default: return go(__nv_bfloat16{});
  }
}

}  // namespace gfc
