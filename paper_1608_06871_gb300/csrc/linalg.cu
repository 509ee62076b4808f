// Batched dense linear algebra kernels (see linalg.cuh).
//
// FP64 on this part runs at a small fraction of the FP32 rate, so these
// kernels are arithmetic-bound by construction; they are tiled for data reuse
// in shared memory and use every SM through the batch and tile dimensions.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include <cooperative_groups.h>

#include "linalg.cuh"

namespace cg = cooperative_groups;

namespace hs {

bool prof_active(int family);
void prof_begin(cudaStream_t s, cudaEvent_t* a);
void prof_end(cudaStream_t s, cudaEvent_t a, double flops);

namespace {
template <typename T> struct is_cplx { static constexpr bool v = false; };
template <> struct is_cplx<double2> { static constexpr bool v = true; };
template <> struct is_cplx<float2> { static constexpr bool v = true; };
template <typename T> struct is_fp64 { static constexpr bool v = false; };
template <> struct is_fp64<double> { static constexpr bool v = true; };
template <> struct is_fp64<double2> { static constexpr bool v = true; };
template <typename TA, typename TB> constexpr double flops_per_mac() {
  return (is_cplx<TA>::v && is_cplx<TB>::v) ? 8.0 : ((is_cplx<TA>::v || is_cplx<TB>::v) ? 4.0 : 2.0);
}
constexpr int BK = 16;                    // k-step of the small GEMM tiles
constexpr int NB = 32;                    // LU panel / TRSM block size
constexpr int NBB = 128;                  // LU super-panel: k of the trailing updates
constexpr int kMaxCluster = 8;            // portable thread-block cluster size (split-k)

__device__ __forceinline__ double shfl_xor(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ float shfl_xor(float v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ double2 shfl_xor(double2 v, int m) {
  return make_double2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
__device__ __forceinline__ float2 shfl_xor(float2 v, int m) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}

template <typename T> __device__ __forceinline__ T ld_op(const T* P, int ld, int op, int r, int c) {
  return op == OP_N ? P[(long long)r * ld + c] : P[(long long)c * ld + r];
}

// TM x TN tile, one 256-thread CTA, (TM TN / 256) outputs per thread, the next
// k-step prefetched into registers.  blockIdx.z = batch * splits + split:
// with splits > 1 the kernel is launched in clusters of `splits` CTAs along z,
// each CTA covers a slice of k, and the partial tiles are summed through
// distributed shared memory in split order (deterministic, no atomics): rank r
// reduces and writes its share of the tile's rows.
// FP64: bound by the pipe, which takes two thread-operations per SM and clock
// whatever the tile, so the tile only has to keep padding and idle SMs small:
// 16 x 16 as well as 32 x 32 (fp64_tile), both saturate it (one DFMA per warp
// and 64 cycles leaves room for the two shared-memory loads it needs).  With
// this, the dot products and k_trsm_blk below a far field of one incidence on
// 4 x 4 leaves went from 2.52 to 0.54 ms, a k = 5 Gauss-Newton step from 16.3
// to 7.8 ms, the k = 40 FP64 batch from 263 to 227 ms.
template <typename TA, typename TB, typename TC, int TM, int TN>
__global__ void __launch_bounds__(256) k_gemm(int opA, int opB, int m, int n, int k, TC alpha, const TA* __restrict__ A,
                                              int lda, long long sA, const TB* __restrict__ B, int ldb, long long sB,
                                              TC beta, TC* __restrict__ C, int ldc, long long sC, int splits) {
  constexpr int RM = TM / 16, RN = TN / 16;                      // outputs per thread
  constexpr int NA = TM * BK / 256, NBq = TN * BK / 256;         // staged elements per thread
  constexpr size_t A_BYTES = sizeof(TA) * BK * (TM + 1), B_BYTES = sizeof(TB) * BK * (TN + 1);
  constexpr size_t RED_BYTES = sizeof(TC) * TM * TN;
  __shared__ __align__(16) unsigned char raw[A_BYTES + B_BYTES > RED_BYTES ? A_BYTES + B_BYTES : RED_BYTES];
  TA(*As)[TM + 1] = reinterpret_cast<TA(*)[TM + 1]>(raw);
  TB(*Bs)[TN + 1] = reinterpret_cast<TB(*)[TN + 1]>(raw + A_BYTES);
  const int b = blockIdx.z / splits, sp = blockIdx.z % splits;
  A += b * sA;
  B += b * sB;
  C += b * sC;
  const int kc = ((k + splits - 1) / splits + BK - 1) / BK * BK;
  const int kbeg = sp * kc, kend = min(k, kbeg + kc);
  const int row0 = blockIdx.y * TM, col0 = blockIdx.x * TN;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  TC acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = el<TC>::zero();
  TA ra[NA];
  TB rb[NBq];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = threadIdx.x + 256 * q;
      int r, kk;
      if (opA == OP_N) { r = e / BK; kk = e % BK; } else { kk = e / TM; r = e % TM; }
      const int gr = row0 + r, gk = k0 + kk;
      ra[q] = (gr < m && gk < kend) ? ld_op(A, lda, opA, gr, gk) : el<TA>::zero();
    }
#pragma unroll
    for (int q = 0; q < NBq; ++q) {
      const int e = threadIdx.x + 256 * q;
      int kk, c;
      if (opB == OP_N) { kk = e / TN; c = e % TN; } else { c = e / BK; kk = e % BK; }
      const int gk = k0 + kk, gc = col0 + c;
      rb[q] = (gk < kend && gc < n) ? ld_op(B, ldb, opB, gk, gc) : el<TB>::zero();
    }
  };
  if (kbeg < kend) load(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = threadIdx.x + 256 * q;
      if (opA == OP_N) As[e % BK][e / BK] = ra[q]; else As[e / TM][e % TM] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < NBq; ++q) {
      const int e = threadIdx.x + 256 * q;
      if (opB == OP_N) Bs[e / TN][e % TN] = rb[q]; else Bs[e % BK][e / BK] = rb[q];
    }
    __syncthreads();
    if (k0 + BK < kend) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      TA a[RM];
      TB bb[RN];
#pragma unroll
      for (int i = 0; i < RM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < RN; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fmac(acc[i][j], a[i], bb[j]);
    }
    __syncthreads();
  }
  if (splits == 1) {
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        int r = row0 + ty + 16 * i, c = col0 + tx + 16 * j;
        if (r < m && c < n) {
          TC v = scal<TC, TC>(alpha, acc[i][j]);
          long long o = (long long)r * ldc + c;
          if (!is_zero(beta)) v = addv(v, scal<TC, TC>(beta, C[o]));
          C[o] = v;
        }
      }
    return;
  }
  TC* red = reinterpret_cast<TC*>(raw);  // the k loop ended with a barrier
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) red[(ty + 16 * i) * TN + tx + 16 * j] = acc[i][j];
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  const int rows_per = (TM + splits - 1) / splits;
  const int rb0 = sp * rows_per, re = min(TM, rb0 + rows_per);
  for (int e = rb0 * TN + threadIdx.x; e < re * TN; e += 256) {
    TC sum = el<TC>::zero();
    for (int q = 0; q < splits; ++q) sum = addv(sum, cl.map_shared_rank(red, q)[e]);
    const int r = row0 + e / TN, c = col0 + e % TN;
    if (r < m && c < n) {
      TC v = scal<TC, TC>(alpha, sum);
      long long o = (long long)r * ldc + c;
      if (!is_zero(beta)) v = addv(v, scal<TC, TC>(beta, C[o]));
      C[o] = v;
    }
  }
  cl.sync();  // keep this CTA's partial tile alive until every rank has read it
}

// Products with at most eight columns (or, with the roles of the operands
// swapped by the host, rows): a warp takes RW rows and NC columns, lanes along
// k.  Such a product is a few passes over one operand; a square tile pads the
// columns to its width, and FP64 pays for padding on the pipe (224 x 1 x 224
// complex: 200 us with a 32 x 32 tile).  The RW NC sums are reduced together,
// each exchange halving the number of sums a lane carries (RW NC + log steps
// instead of five per sum; in FP64 the additions are on the pipe).
// Element strides, so that both transposes and the swap are the same code:
// A(i, l) = A[i ai + l ak], B(l, j) = B[l bk + j bj], C(i, j) = C[i ci + j cj].
constexpr int DOT_WARPS = 4;
template <typename TA, typename TB, typename TC, int NC, int RW>
__global__ void __launch_bounds__(32 * DOT_WARPS)
    k_gemm_dot(int m, int n, int k, TC alpha, const TA* __restrict__ A, long long ai, long long ak, long long sA,
               const TB* __restrict__ B, long long bk, long long bj, long long sB, TC beta, TC* __restrict__ C,
               long long ci, long long cj, long long sC) {
  constexpr int NV = NC * RW;  // sums, a power of two up to 32
  const int lane = threadIdx.x & 31;
  const int i0 = (blockIdx.x * DOT_WARPS + (threadIdx.x >> 5)) * RW, j0 = blockIdx.y * NC;
  if (i0 >= m) return;  // whole warp
  A += blockIdx.z * sA + i0 * ai;
  B += blockIdx.z * sB + j0 * bj;
  TC acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = el<TC>::zero();
#pragma unroll 2
  for (int l = lane; l < k; l += 32) {
    TA a[RW];
    TB b[NC];
#pragma unroll
    for (int r = 0; r < RW; ++r) a[r] = i0 + r < m ? A[r * ai + l * ak] : el<TA>::zero();
#pragma unroll
    for (int j = 0; j < NC; ++j) b[j] = j0 + j < n ? B[l * bk + j * bj] : el<TB>::zero();
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
      for (int j = 0; j < NC; ++j) acc[r * NC + j] = fmac(acc[r * NC + j], a[r], b[j]);
  }
  int off = 16;
#pragma unroll
  for (int nv = NV; nv > 1; nv >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int v = 0; v < nv / 2; ++v) {
      const TC keep = up ? acc[v + nv / 2] : acc[v], send = up ? acc[v] : acc[v + nv / 2];
      acc[v] = addv(keep, shfl_xor(send, off));
    }
  }
  for (; off > 0; off >>= 1) acc[0] = addv(acc[0], shfl_xor(acc[0], off));
  const int v = lane / (32 / NV), i = i0 + v / NC, j = j0 + v % NC;
  if (lane % (32 / NV) == 0 && i < m && j < n) {
    TC* c = C + blockIdx.z * sC + i * ci + j * cj;
    TC x = scal<TC, TC>(alpha, acc[0]);
    if (!is_zero(beta)) x = addv(x, scal<TC, TC>(beta, *c));
    *c = x;
  }
}

// 64 x 64 tile, 4 x 4 outputs per thread (more arithmetic per shared-memory
// load), k-step 8 with the next tile prefetched into registers.  For shapes
// with enough tiles to fill the machine.
constexpr int GB = 64, GK = 8;
template <typename TA, typename TB, typename TC>
__global__ void __launch_bounds__(256, 2) k_gemm_big(int opA, int opB, int m, int n, int k, TC alpha,
                                                  const TA* __restrict__ A, int lda, long long sA,
                                                  const TB* __restrict__ B, int ldb, long long sB, TC beta,
                                                  TC* __restrict__ C, int ldc, long long sC) {
  __shared__ TA As[GK][GB];
  __shared__ TB Bs[GK][GB];
  const int b = blockIdx.z;
  A += b * sA;
  B += b * sB;
  C += b * sC;
  const int kbeg = 0, kend = k;
  const int row0 = blockIdx.y * GB, col0 = blockIdx.x * GB;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  TC acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = el<TC>::zero();
  // each thread stages 2 elements of A and 2 of B per k-step (64 x 8 each)
  TA ra[2];
  TB rb[2];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      int e = threadIdx.x + 256 * q;
      int r, kk;
      if (opA == OP_N) { r = e / GK; kk = e % GK; } else { kk = e / GB; r = e % GB; }
      int gr = row0 + r, gk = k0 + kk;
      ra[q] = (gr < m && gk < kend) ? ld_op(A, lda, opA, gr, gk) : el<TA>::zero();
      int kk2, c;
      if (opB == OP_N) { kk2 = e / GB; c = e % GB; } else { c = e / GK; kk2 = e % GK; }
      int gk2 = k0 + kk2, gc = col0 + c;
      rb[q] = (gk2 < kend && gc < n) ? ld_op(B, ldb, opB, gk2, gc) : el<TB>::zero();
    }
  };
  auto store = [&]() {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      int e = threadIdx.x + 256 * q;
      int r, kk;
      if (opA == OP_N) { r = e / GK; kk = e % GK; } else { kk = e / GB; r = e % GB; }
      As[kk][r] = ra[q];
      int kk2, c;
      if (opB == OP_N) { kk2 = e / GB; c = e % GB; } else { c = e / GK; kk2 = e % GK; }
      Bs[kk2][c] = rb[q];
    }
  };
  load(kbeg);
  for (int k0 = kbeg; k0 < kend; k0 += GK) {
    store();
    __syncthreads();
    if (k0 + GK < kend) load(k0 + GK);
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      TA a[4];
      TB bb[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmac(acc[i][j], a[i], bb[j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int r = row0 + ty + 16 * i, c = col0 + tx + 16 * j;
      if (r < m && c < n) {
        TC v = scal<TC, TC>(alpha, acc[i][j]);
        long long o = (long long)r * ldc + c;
        if (!is_zero(beta)) v = addv(v, scal<TC, TC>(beta, C[o]));
        C[o] = v;
      }
    }
}


__device__ __forceinline__ double shfl(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ float shfl(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ double2 shfl(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ float2 shfl(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// Triangular solve with a diagonal block of size nb <= NB for many right-hand
// sides: one warp per right-hand side, lane r holding x_r; each substitution
// step broadcasts the finished unknown with a shuffle.  mode: 0 = L (unit
// lower), 1 = U (upper), 2 = U^T (lower, non-unit), 3 = L^T (upper, unit).
constexpr int TRSM_WARPS = 4;
template <typename E>
__global__ void __launch_bounds__(32 * TRSM_WARPS) k_trsm_diag(const E* A, int lda, long long sA, int i0, int nb,
                                                              int mode, E* B, int ldb, long long sB, int nrhs) {
  __shared__ E T[NB][NB + 1];
  const int b = blockIdx.y;
  A += b * sA;
  B += b * sB;
  for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
    int r = e / nb, c = e % nb;
    bool tr = (mode >= 2);
    const E a = tr ? A[(long long)(i0 + c) * lda + i0 + r] : A[(long long)(i0 + r) * lda + i0 + c];
    T[r][c] = r == c && (mode == 1 || mode == 2) ? el<E>::div(el<E>::one(), a) : a;  // reciprocal diagonal
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int col = blockIdx.x * TRSM_WARPS + warp;
  if (col >= nrhs) return;  // whole warp leaves together
  E x = lane < nb ? B[(long long)(i0 + lane) * ldb + col] : el<E>::zero();
  const bool lower = (mode == 0 || mode == 2);
  const bool unit = (mode == 0 || mode == 3);
  if (lower) {
    for (int s = 0; s < nb; ++s) {
      if (!unit && lane == s) x = x * T[s][s];
      E xs = shfl(x, s);
      if (lane > s && lane < nb) x = fmsc(x, T[lane][s], xs);
    }
  } else {
    for (int s = nb - 1; s >= 0; --s) {
      if (!unit && lane == s) x = x * T[s][s];
      E xs = shfl(x, s);
      if (lane < s) x = fmsc(x, T[lane][s], xs);
    }
  }
  if (lane < nb) B[(long long)(i0 + lane) * ldb + col] = x;
}

// Same solve, one thread per right-hand side with the 32 unknowns in
// registers (fully unrolled): the better choice when there are many
// right-hand sides in the batch (leaf and merge systems).
template <typename E>
__global__ void __launch_bounds__(128) k_trsm_diag_col(const E* A, int lda, long long sA, int i0, int nb, int mode,
                                                       E* B, int ldb, long long sB, int nrhs) {
  __shared__ E T[NB][NB + 1];
  const int b = blockIdx.y;
  A += b * sA;
  B += b * sB;
  const bool tr = (mode >= 2);
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    int r = e / NB, c = e % NB;
    const E a = (r < nb && c < nb) ? (tr ? A[(long long)(i0 + c) * lda + i0 + r] : A[(long long)(i0 + r) * lda + i0 + c])
                                   : el<E>::zero();
    T[r][c] = r == c && r < nb && (mode == 1 || mode == 2) ? el<E>::div(el<E>::one(), a) : a;  // reciprocal diagonal
  }
  __syncthreads();
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= nrhs) return;
  E x[NB];
#pragma unroll
  for (int r = 0; r < NB; ++r) x[r] = r < nb ? B[(long long)(i0 + r) * ldb + col] : el<E>::zero();
  const bool lower = (mode == 0 || mode == 2);
  const bool unit = (mode == 0 || mode == 3);
  if (lower) {
#pragma unroll
    for (int r = 0; r < NB; ++r) {
      E v = x[r];
#pragma unroll
      for (int c = 0; c < r; ++c) v = fmsc(v, T[r][c], x[c]);
      x[r] = (unit || r >= nb) ? v : v * T[r][r];
    }
  } else {
#pragma unroll
    for (int r = NB - 1; r >= 0; --r) {
      E v = x[r];
#pragma unroll
      for (int c = r + 1; c < NB; ++c) v = fmsc(v, T[r][c], x[c]);
      x[r] = (unit || r >= nb) ? v : v * T[r][r];
    }
  }
#pragma unroll
  for (int r = 0; r < NB; ++r)
    if (r < nb) B[(long long)(i0 + r) * ldb + col] = x[r];
}

// Many columns overall: one thread per column; few: one warp per column.
template <typename E>
void trsm_diag(cudaStream_t s, const E* A, int lda, long long sA, int i0, int nb, int mode, E* B, int ldb,
               long long sB, int nrhs, int batch) {
  if ((long long)nrhs * batch >= 8192) {
    const int threads = nrhs >= 128 ? 128 : ((nrhs + 31) / 32) * 32;
    dim3 g((nrhs + threads - 1) / threads, batch);
    k_trsm_diag_col<E><<<g, threads, 0, s>>>(A, lda, sA, i0, nb, mode, B, ldb, sB, nrhs);
  } else {
    dim3 g((nrhs + TRSM_WARPS - 1) / TRSM_WARPS, batch);
    k_trsm_diag<E><<<g, 32 * TRSM_WARPS, 0, s>>>(A, lda, sA, i0, nb, mode, B, ldb, sB, nrhs);
  }
  HS_COUNT_LAUNCH();
}

// The solve with a whole diagonal block of up to NBB rows in one launch: rows
// [i0, i0 + nbs) of B (CW columns per CTA, held in shared memory) against the
// block's triangle; mode as k_trsm_diag's (0: L, 1: U, 2: U^T, 3: L^T; 0 and 2
// run top down, 1 and 3 bottom up).  Per sub-block of SB rows one warp per
// column substitutes with shuffles, then every thread updates the rows still
// to solve.  The sub-block's columns of the triangle are staged in shared
// memory by cp.async, the next sub-block's while this one is solved.
// What bounds it is the substitution's chain and, in FP64, the pipe (two
// thread-operations per SM and clock): complex sub-blocks of 16 rows put the
// real and the imaginary part of a row on two lanes, two dependent
// multiply-adds a step instead of four on a half-idle warp, and the host takes
// as few columns per CTA as spread them over the SMs (trsm_cw).  A 128-row
// block with one FP64 complex column: 274 us with eight columns per CTA, of
// which seven were padding.
template <typename E> struct tb_sb { static constexpr int v = sizeof(E) == 16 ? 16 : 32; };  // sub-block rows

// One warp: x (rows r0 .. r0 + nb of column c in Bs) <- solve with the nb x nb
// triangle whose (r, t) entry is T[r][t].  The diagonal's reciprocals are taken
// by all lanes at once before the chain, which then only multiplies (a complex
// FP64 division inside it would be some thirty operations of the pipe a step).
template <typename E, int SB, int CW>
__device__ __forceinline__ void tri_solve_warp(const E (*T)[SB + 1], E (*Bs)[CW + 1], int r0, int nb, int c, bool down,
                                               bool unit, int lane) {
  if constexpr (sizeof(E) == 16) {  // complex FP64: lane = 2 row + part
    const int r = lane >> 1, im = lane & 1;
    const bool live = r < nb;
    double x = live ? (im ? Bs[r0 + r][c].y : Bs[r0 + r][c].x) : 0.0;
    const E inv = (live && !unit) ? el<E>::div(el<E>::one(), T[r][r]) : el<E>::one();
    for (int q = 0; q < nb; ++q) {
      const int t = down ? q : nb - 1 - q;
      if (!unit) {
        const double o = __shfl_xor_sync(0xffffffffu, x, 1);
        if (r == t) x = im ? fma(x, inv.x, o * inv.y) : fma(x, inv.x, -o * inv.y);
      }
      const double xr = __shfl_sync(0xffffffffu, x, 2 * t), xi = __shfl_sync(0xffffffffu, x, 2 * t + 1);
      if (live && (down ? r > t : r < t)) {
        const E l = T[r][t];
        // re -= l.x xr - l.y xi,  im -= l.x xi + l.y xr
        x = im ? fma(-l.y, xr, fma(-l.x, xi, x)) : fma(l.y, xi, fma(-l.x, xr, x));
      }
    }
    if (live) (im ? Bs[r0 + r][c].y : Bs[r0 + r][c].x) = x;
  } else {
    E x = lane < nb ? Bs[r0 + lane][c] : el<E>::zero();
    const E inv = (lane < nb && !unit) ? el<E>::div(el<E>::one(), T[lane][lane]) : el<E>::one();
    for (int q = 0; q < nb; ++q) {
      const int t = down ? q : nb - 1 - q;
      if (!unit && lane == t) x = x * inv;
      const E xt = shfl(x, t);
      if (lane < nb && (down ? lane > t : lane < t)) x = fmsc(x, T[lane][t], xt);
    }
    if (lane < nb) Bs[r0 + lane][c] = x;
  }
}

template <typename E, int CW>
__global__ void __launch_bounds__(CW <= 4 ? 128 : 32 * CW)
    k_trsm_blk(const E* __restrict__ A, int lda, long long sA, int i0, int nbs, int mode, E* __restrict__ B, int ldb,
               long long sB, int nrhs) {
  constexpr int SB = tb_sb<E>::v, NT = CW <= 4 ? 128 : 32 * CW;
  extern __shared__ __align__(16) unsigned char trsm_smem[];
  E(*Bs)[CW + 1] = reinterpret_cast<E(*)[CW + 1]>(trsm_smem);
  E(*Lp)[NBB][SB + 1] = reinterpret_cast<E(*)[NBB][SB + 1]>(trsm_smem + sizeof(E) * NBB * (CW + 1));
  const int b = blockIdx.y, c0 = blockIdx.x * CW, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool down = mode == 0 || mode == 2, unit = mode == 0 || mode == 3, tr = mode >= 2;
  A += b * sA + (long long)i0 * lda + i0;
  B += b * sB + (long long)i0 * ldb + c0;
  const int nsub = (nbs + SB - 1) / SB;
  // rows still to solve at sub-block `sub`, itself included: [lo, hi)
  auto range = [&](int sub, int& r0, int& nb, int& lo, int& hi) {
    r0 = sub * SB;
    nb = min(SB, nbs - r0);
    lo = down ? r0 : 0;
    hi = down ? nbs : r0 + nb;
  };
  auto stage = [&](int q) {
    int r0, nb, lo, hi;
    range(down ? q : nsub - 1 - q, r0, nb, lo, hi);
    if (!tr) {  // (r, t) at A[r][r0 + t]: rows of nb contiguous entries
      for (int e = tid; e < (hi - lo) * nb; e += NT) {
        const int r = lo + e / nb, t = e % nb;
        cp_elem<sizeof(E)>(&Lp[q & 1][r][t], A + (long long)r * lda + r0 + t);
      }
    } else {  // (r, t) at A[r0 + t][r]: contiguous along r
      const int nr = hi - lo;
      for (int e = tid; e < nr * nb; e += NT) {
        const int t = e / nr, r = lo + e % nr;
        cp_elem<sizeof(E)>(&Lp[q & 1][r][t], A + (long long)(r0 + t) * lda + r);
      }
    }
    cp_commit();
  };
  stage(0);
  for (int e = tid; e < nbs * CW; e += NT) {
    const int r = e / CW, c = e % CW;
    Bs[r][c] = c0 + c < nrhs ? B[(long long)r * ldb + c] : el<E>::zero();
  }
  for (int q = 0; q < nsub; ++q) {
    int r0, nb, lo, hi;
    range(down ? q : nsub - 1 - q, r0, nb, lo, hi);
    cp_wait<0>();
    __syncthreads();  // the panel has landed; the previous update of Bs is done
    if (q + 1 < nsub) stage(q + 1);
    for (int c = warp; c < CW && c0 + c < nrhs; c += NT / 32)
      tri_solve_warp<E, SB, CW>(&Lp[q & 1][r0], Bs, r0, nb, c, down, unit, lane);
    __syncthreads();
    const int ra = down ? r0 + nb : 0, rb = down ? nbs : r0;
    for (int e = tid; e < (rb - ra) * CW; e += NT) {
      const int r = ra + e / CW, c = e % CW;
      E acc = Bs[r][c];
      if (nb == SB) {
#pragma unroll
        for (int t = 0; t < SB; ++t) acc = fmsc(acc, Lp[q & 1][r][t], Bs[r0 + t][c]);
      } else {
        for (int t = 0; t < nb; ++t) acc = fmsc(acc, Lp[q & 1][r][t], Bs[r0 + t][c]);
      }
      Bs[r][c] = acc;
    }
  }
  __syncthreads();
  for (int e = tid; e < nbs * CW; e += NT) {
    const int r = e / CW, c = e % CW;
    if (c0 + c < nrhs) B[(long long)r * ldb + c] = Bs[r][c];
  }
}

// Columns per CTA: the fewest columns on the busiest SM (its CTAs share the
// pipe), more per CTA where that costs at most a tenth (the triangle is staged
// once per CTA).
int trsm_cw(int nrhs, int batch) {
  int best = 1;
  double bt = 1e300;
  for (int cw : {8, 4, 2, 1}) {
    const double t = std::ceil((double)((nrhs + cw - 1) / cw) * batch / 152.0) * cw;
    if (t < 0.9 * bt) {
      bt = t;
      best = cw;
    }
  }
  return best;
}

template <typename E, int CW>
void launch_trsm_blk(cudaStream_t s, const E* A, int lda, long long sA, int i0, int nbs, int mode, E* B, int ldb,
                     long long sB, int nrhs, int batch) {
  constexpr int SB = tb_sb<E>::v, NT = CW <= 4 ? 128 : 32 * CW;
  constexpr int smem = (int)sizeof(E) * (NBB * (CW + 1) + 2 * NBB * (SB + 1));
  if constexpr (smem > 48 * 1024) {
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr[dev]) {
      cudaFuncSetAttribute(k_trsm_blk<E, CW>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (dev >= 0 && dev < 64) attr[dev] = true;
    }
  }
  dim3 g((nrhs + CW - 1) / CW, batch);
  k_trsm_blk<E, CW><<<g, NT, smem, s>>>(A, lda, sA, i0, nbs, mode, B, ldb, sB, nrhs);
  HS_COUNT_LAUNCH();
}

// Solve with the diagonal block rows [i0, i0 + nbs) of A: one launch of
// k_trsm_blk when there are few columns overall (the root system and the top
// merges, where the NB-blocked sequence is launch- and latency-bound); with
// many (batched leaf and merge systems) the NB-blocked sequence of
// one-thread-per-column solves and products keeps more threads busy.
template <typename E>
void trsm_blk(cudaStream_t s, const E* A, int lda, long long sA, int i0, int nbs, int mode, E* B, int ldb,
              long long sB, int nrhs, int batch) {
  if ((long long)nrhs * batch < 8192) {
    switch (trsm_cw(nrhs, batch)) {
      case 8: launch_trsm_blk<E, 8>(s, A, lda, sA, i0, nbs, mode, B, ldb, sB, nrhs, batch); return;
      case 4: launch_trsm_blk<E, 4>(s, A, lda, sA, i0, nbs, mode, B, ldb, sB, nrhs, batch); return;
      case 2: launch_trsm_blk<E, 2>(s, A, lda, sA, i0, nbs, mode, B, ldb, sB, nrhs, batch); return;
      default: launch_trsm_blk<E, 1>(s, A, lda, sA, i0, nbs, mode, B, ldb, sB, nrhs, batch); return;
    }
  }
  const E m1 = -el<E>::one(), one = el<E>::one();
  const int I1 = i0 + nbs;
  const bool tr = mode >= 2;
  if (mode == 0 || mode == 2) {
    for (int j = i0; j < I1; j += NB) {
      const int nb = std::min(NB, I1 - j);
      trsm_diag<E>(s, A, lda, sA, j, nb, mode, B, ldb, sB, nrhs, batch);
      if (I1 - j - nb > 0)
        gemm<E, E, E>(s, tr ? OP_T : OP_N, OP_N, I1 - j - nb, nrhs, nb, m1,
                      tr ? A + (long long)j * lda + j + nb : A + (long long)(j + nb) * lda + j, lda, sA,
                      B + (long long)j * ldb, ldb, sB, one, B + (long long)(j + nb) * ldb, ldb, sB, batch);
    }
  } else {
    for (int j = i0 + ((nbs - 1) / NB) * NB; j >= i0; j -= NB) {
      const int nb = std::min(NB, I1 - j);
      trsm_diag<E>(s, A, lda, sA, j, nb, mode, B, ldb, sB, nrhs, batch);
      if (j > i0)
        gemm<E, E, E>(s, tr ? OP_T : OP_N, OP_N, j - i0, nrhs, nb, m1,
                      tr ? A + (long long)j * lda + i0 : A + (long long)i0 * lda + j, lda, sA,
                      B + (long long)j * ldb, ldb, sB, one, B + (long long)i0 * ldb, ldb, sB, batch);
    }
  }
}

template <typename E>
__global__ void k_swaps(const int* piv, long long sP, int n, int reverse, E* B, int ldb, long long sB, int nrhs) {
  const int b = blockIdx.y;
  piv += b * sP;
  B += b * sB;
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= nrhs) return;
  if (!reverse) {
    for (int j = 0; j < n; ++j) {
      int p = piv[j];
      if (p != j) {
        E t = B[(long long)j * ldb + col];
        B[(long long)j * ldb + col] = B[(long long)p * ldb + col];
        B[(long long)p * ldb + col] = t;
      }
    }
  } else {
    for (int j = n - 1; j >= 0; --j) {
      int p = piv[j];
      if (p != j) {
        E t = B[(long long)j * ldb + col];
        B[(long long)j * ldb + col] = B[(long long)p * ldb + col];
        B[(long long)p * ldb + col] = t;
      }
    }
  }
}
}  // namespace

namespace {
// Launch a small-tile product, k split over a cluster when splits > 1.
template <typename TA, typename TB, typename TC, int TM, int TN>
void launch_gemm(cudaStream_t s, int opA, int opB, int m, int n, int k, TC alpha, const TA* A, int lda, long long sA,
                 const TB* B, int ldb, long long sB, TC beta, TC* C, int ldc, long long sC, int batch, int splits) {
  dim3 grid((n + TN - 1) / TN, (m + TM - 1) / TM, batch * splits);
  if (splits == 1) {
    k_gemm<TA, TB, TC, TM, TN><<<grid, 256, 0, s>>>(opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc,
                                                    sC, 1);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = splits;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_gemm<TA, TB, TC, TM, TN>, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C,
                       ldc, sC, splits);
  }
  HS_COUNT_LAUNCH();
}

template <typename TA, typename TB, typename TC>
void launch_dot(cudaStream_t s, int m, int n, int k, TC alpha, const TA* A, long long ai, long long ak, long long sA,
                const TB* B, long long bk, long long bj, long long sB, TC beta, TC* C, long long ci, long long cj,
                long long sC, int batch) {
  // columns of one pass over A; four rows per warp once that leaves enough warps
  const int nc = n > 4 ? 8 : n > 2 ? 4 : n;
  const int rw = (long long)m * batch < 152LL * 16 * 4 ? 1 : nc == 8 && sizeof(TC) == 16 ? 2 : 4;
  dim3 grid((m + DOT_WARPS * rw - 1) / (DOT_WARPS * rw), (n + nc - 1) / nc, batch);
  auto go = [&](auto kernel) {
    kernel<<<grid, 32 * DOT_WARPS, 0, s>>>(m, n, k, alpha, A, ai, ak, sA, B, bk, bj, sB, beta, C, ci, cj, sC);
  };
  constexpr int RW = sizeof(TC) == 16 ? 2 : 4;  // of eight columns (registers)
  if (rw == 1) {
    if (nc == 8) go(k_gemm_dot<TA, TB, TC, 8, 1>);
    else if (nc == 4) go(k_gemm_dot<TA, TB, TC, 4, 1>);
    else if (nc == 2) go(k_gemm_dot<TA, TB, TC, 2, 1>);
    else go(k_gemm_dot<TA, TB, TC, 1, 1>);
  } else {
    if (nc == 8) go(k_gemm_dot<TA, TB, TC, 8, RW>);
    else if (nc == 4) go(k_gemm_dot<TA, TB, TC, 4, 4>);
    else if (nc == 2) go(k_gemm_dot<TA, TB, TC, 2, 4>);
    else go(k_gemm_dot<TA, TB, TC, 1, 4>);
  }
  HS_COUNT_LAUNCH();
}

// FP64 tile edge and k splits: the pipe's time of the busiest SM (the SM's
// CTAs share it, two thread-operations per clock) plus a latency per CTA.
struct Fp64Tile { int t, splits; double cycles; };
Fp64Tile fp64_tile(int m, int n, int k, int batch, double fma) {
  Fp64Tile best{64, 1, 0.0};
  double bt = 1e300;
  for (int t : {64, 32, 16})
    for (int sp = 1; sp <= (t == 64 ? 1 : kMaxCluster); ++sp) {
      if (sp > 1 && (k / sp < 2 * BK || (long long)batch * sp > 65535)) break;
      const double ctas = (double)((m + t - 1) / t) * ((n + t - 1) / t) * batch * sp;
      const int kc = ((k + sp - 1) / sp + BK - 1) / BK * BK;
      // the 64-wide tile has no such padding of k and better reuse when it fills the chip
      const double one = (double)t * t * fma * (t == 64 ? (k + 7) / 8 * 8 : kc) / 2.0 + (sp > 1 ? 3000.0 : 1500.0);
      if ((m + t - 1) / t > 65535) continue;  // grid.y
      const double time = std::ceil(ctas / 152.0) * one * (t == 64 ? 1.0 : t == 32 ? 1.02 : 1.06);
      if (time < bt) {
        bt = time;
        best = Fp64Tile{t, sp, time};
      }
    }
  return best;
}

// SIMT product (FP64, or FP32 where the tensor-core path is not taken).
template <typename TA, typename TB, typename TC>
void gemm_simt(cudaStream_t s, int opA, int opB, int m, int n, int k, TC alpha, const TA* A, int lda, long long sA,
               const TB* B, int ldb, long long sB, TC beta, TC* C, int ldc, long long sC, int batch) {
  const bool prof = prof_active(is_fp64<TC>::v ? 1 : 2);
  cudaEvent_t ev = nullptr;
  if (prof) prof_begin(s, &ev);
  const double fl = flops_per_mac<TA, TB>() * (double)m * n * k * batch;
  // few columns or rows: dot products (grid limits: rows / 4 in x, batch in z)
  if (std::min(m, n) <= 8 && batch <= 65535) {
    const long long ai = opA == OP_N ? lda : 1, ak = opA == OP_N ? 1 : lda;
    const long long bk = opB == OP_N ? ldb : 1, bj = opB == OP_N ? 1 : ldb;
    if (n <= m)
      launch_dot<TA, TB, TC>(s, m, n, k, alpha, A, ai, ak, sA, B, bk, bj, sB, beta, C, ldc, 1, sC, batch);
    else
      launch_dot<TB, TA, TC>(s, n, m, k, alpha, B, bj, bk, sB, A, ak, ai, sA, beta, C, 1, ldc, sC, batch);
    if (prof) prof_end(s, ev, fl);
    return;
  }
  if constexpr (is_fp64<TC>::v) {
    const Fp64Tile t = fp64_tile(m, n, k, batch, flops_per_mac<TA, TB>() / 2.0);
    if (t.t != 64) {
      if (t.t == 32)
        launch_gemm<TA, TB, TC, 32, 32>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch,
                                        t.splits);
      else
        launch_gemm<TA, TB, TC, 16, 16>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch,
                                        t.splits);
      if (prof) prof_end(s, ev, fl);
      return;
    }
    dim3 grid((n + GB - 1) / GB, (m + GB - 1) / GB, batch);
    k_gemm_big<TA, TB, TC><<<grid, 256, 0, s>>>(opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC);
    HS_COUNT_LAUNCH();
    if (prof) prof_end(s, ev, fl);
    return;
  }
  if constexpr (!is_fp64<TC>::v) {
    gemm_fp32<TA, TB, TC>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
    if (prof) prof_end(s, ev, fl);
  }
}

inline double re_of(double x) { return x; }
inline double re_of(double2 x) { return x.x; }
inline double im_of(double) { return 0.0; }
inline double im_of(double2 x) { return x.y; }

// mr x nr x kr: the sizes of the real product behind m x n x k.
bool emulation_pays(int mr, int nr, int kr, int m, int n, int k, int batch, bool b_shared, double fma) {
  return std::min(m, n) > 8 && oz_cycles(mr, nr, kr, batch, b_shared) <= 0.8 * fp64_tile(m, n, k, batch, fma).cycles;
}

// FP64 products by the emulated product on the tensor cores (ozaki.cu) where
// its estimated time is clearly below the FP64 pipe's: 36 bf16 products are
// about a tenth of the pipe's time per multiply-add, but operands are sliced
// first (two more launches, 16 bytes written and read per entry) and tiles are
// 128 x 32, so small and thin products stay on the pipe (the two models' times
// are compared, with a fifth in favour of the pipe).  The products of the k = 40
// FP64 batch: 160 ms on the pipe, 27 ms sliced and multiplied; the batch 227 ->
// 98.5 ms, a k = 20 gradient 65.8 -> 44.3 ms.  Error against 64 bits of random
// complex products: 7e-17 .. 1.3e-16 of the result for k = 32 .. 1792, on the
// pipe 2.5e-16 .. 7e-16 (rows whose entries spread over 1e5: 4.5e-16 against
// 3e-16 at k = 128, 4.8e-16 against 1.9e-15 at 1792).  It grows with the grading inside
// rows and columns (the bound in ozaki.cu), so a caller with graded operands keeps them on the
// pipe (PipeScope; the leaf elimination); far fields, fields, Jacobians and steps at k = 3 .. 20 are
// as close to the dense solution as on the pipe, within 2%.
// Batches, then columns, then k, are cut to what the calling thread's scratch holds.
// Factors that are neither real nor (real x complex) imaginary, and calls without
// scratch, are refused.
template <typename TA, typename TB, typename TC>
bool gemm_emulated(cudaStream_t s, int opA, int opB, int m, int n, int k, TC alpha, const TA* A, int lda, long long sA,
                   const TB* B, int ldb, long long sB, TC beta, TC* C, int ldc, long long sC, int batch) {
  constexpr bool ca = is_cplx<TA>::v, cb = is_cplx<TB>::v;
  const OzScratch* sc = g_oz_scratch;
  if (!g_oz_enabled || !sc || !sc->p || k <= 0 || im_of(beta) != 0.0) return false;
  // an imaginary factor of a real x complex product goes into the right operand
  const bool turn = !ca && cb && re_of(alpha) == 0.0;
  if (im_of(alpha) != 0.0 && !turn) return false;
  const double factor = turn ? im_of(alpha) : re_of(alpha);
  const int mr = ca && !cb ? 2 * m : m, nr = cb ? 2 * n : n, kr = ca && cb ? 2 * k : k;
  const bool bsh = sB == 0 && batch > 1;
  if (!emulation_pays(mr, nr, kr, m, n, k, batch, bsh, flops_per_mac<TA, TB>() / 2.0)) return false;
  const long long ea = ca ? 2 : 1, eb = cb ? 2 : 1;
  OzSrc a{reinterpret_cast<const double*>(A), ea * sA, ea * (opA == OP_N ? lda : 1), ea * (opA == OP_N ? 1 : lda),
          ca ? (cb ? OZ_CLEFT : OZ_PAIR) : OZ_REAL};
  OzSrc b{reinterpret_cast<const double*>(B), eb * sB, eb * (opB == OP_N ? 1 : ldb), eb * (opB == OP_N ? ldb : 1),
          cb ? (ca ? OZ_CRIGHT : turn ? OZ_PAIR_I : OZ_PAIR) : OZ_REAL};
  constexpr bool cc = ca || cb;
  OzView c{reinterpret_cast<double*>(C), (cc ? 2 : 1) * sC, (cc ? 2LL : 1LL) * ldc, 0, 1, 1};
  if (ca && !cb) c = OzView{reinterpret_cast<double*>(C), 2 * sC, 2LL * ldc, 1, 2, 2};
  // the largest batch chunk, then the most columns, then the longest piece of k
  // that the scratch holds
  int nb = batch, nn = nr, kc = kr;
  auto fits = [&] { return ozaki_scratch_bytes(mr, nn, kc, nb, bsh) <= sc->bytes; };
  while (nb > 1 && !fits()) nb = (nb + 1) / 2;
  while (nn > 2048 && !fits()) nn = ((nn + 1) / 2 + 63) / 64 * 64;
  while (kc > 384 && !fits()) kc = ((kc + 1) / 2 + 383) / 384 * 384;
  if (!fits()) return false;
  // (what is left over for the last parts fits too; a launch that fails stays the last CUDA error)
  for (int b0 = 0; b0 < batch; b0 += nb)
    for (int n0 = 0; n0 < nr; n0 += nn)
      for (int k0 = 0; k0 < kr; k0 += kc) {
        OzSrc ai = a, bi = b;
        OzView ci = c;
        const long long l0 = ca && cb ? k0 / 2 : k0, j0 = cb ? n0 / 2 : n0;  // (kc and nn are even)
        ai.p += b0 * a.sb + l0 * a.sk;
        bi.p += b0 * b.sb + l0 * b.sk + j0 * b.sr;
        ci.p += b0 * c.sb + n0 * c.sk;
        ozaki_gemm(s, mr, std::min(nn, nr - n0), std::min(kc, kr - k0), std::min(nb, batch - b0), factor, ai, bi, bsh,
                   k0 == 0 ? re_of(beta) : 1.0, ci, sc->p, sc->bytes);
      }
  return true;
}

// Products the split-TF32 tensor-core path takes (t32_gemm modes): complex x
// complex (2), real x complex (1), real x real (0), FP32, no transposes.
template <typename TA, typename TB, typename TC> struct t32_mode { static constexpr int v = -1; };
template <> struct t32_mode<float2, float2, float2> { static constexpr int v = 2; };
template <> struct t32_mode<float, float2, float2> { static constexpr int v = 1; };
template <> struct t32_mode<float, float, float> { static constexpr int v = 0; };

inline float2 as_f2(float2 x) { return x; }
inline float2 as_f2(float x) { return make_float2(x, 0.f); }
template <typename T> constexpr long long fl() { return sizeof(T) / sizeof(float); }  // floats per element

// Products worth measuring: at least 512 rows and 512 of k in the real
// product, at least 64 columns, and 2^28 real multiply-adds.  Smaller ones
// (the batched leaf, merge and sweep products, the short-k trailing updates)
// never reached the required speed-up over SIMT in the measurements (at most
// 1.4x) and stay there without a measurement, which keeps a frequency sweep,
// whose sizes change from step to step, from paying for one per new shape.
bool t32_candidate(int mode, int m, int n, int k, int batch) {
  const long long np = mode ? 2LL * n : n, kp = mode == 2 ? 2LL * k : k;
  return m >= 512 && np >= 64 && kp >= 512 && (long long)m * np * kp * batch >= (1LL << 28);
}

// Per-shape choice between the tensor-core and the SIMT product, measured
// once per shape class (both variants on a scratch copy of C, CUDA events,
// best of two after a warm-up) outside stream capture; inside a capture a
// shape not yet measured takes the default.
// Shapes are keyed in half-octave classes (a frequency sweep changes its sizes
// in small steps; one measurement serves a class).
inline int size_class(long long x) { return x <= 1 ? 0 : (int)std::lround(2.0 * std::log2((double)x)); }
struct TuneKey {
  int mode, m, n, k, batch, bsh;
  bool operator<(const TuneKey& o) const {
    return std::tie(mode, m, n, k, batch, bsh) < std::tie(o.mode, o.m, o.n, o.k, o.batch, o.bsh);
  }
};

std::mutex g_tune_mu;
std::map<TuneKey, bool> g_tune;

}  // namespace

bool g_autotune = true;             // hs_set_autotune
// The tensor-core product's accumulation is coarser than SIMT FMA chains, which
// slows the refinement of the mixed solver; it is kept only where it takes
// less than half the SIMT time (hs_set_tc_margin).
float g_tc_margin = 0.5f;
int g_t32_mode = 1;                 // hs_set_tensor_cores: 0 off, 1 per-shape choice, 2 forced
thread_local bool g_prof_suspended = false;
thread_local int g_last_gemm_tc = 0;

size_t zgemm_scratch_bytes(int m, int n, int k, int batch) {
  return g_oz_enabled && emulation_pays(m, 2 * n, 2 * k, m, n, k, batch, false, 4.0)
             ? ozaki_scratch_bytes(m, 2 * n, 2 * k, batch, false)
             : 0;
}

template <typename TA, typename TB, typename TC>
void gemm(cudaStream_t s, int opA, int opB, int m, int n, int k, TC alpha, const TA* A, int lda, long long sA,
          const TB* B, int ldb, long long sB, TC beta, TC* C, int ldc, long long sC, int batch) {
  if (m <= 0 || n <= 0 || batch <= 0) return;
  g_last_gemm_tc = 0;
  constexpr int mode = t32_mode<TA, TB, TC>::v;
  if constexpr (mode >= 0) {
    const bool force = g_t32_mode == 2;
    if (opA == OP_N && opB == OP_N && k > 0 && g_t32_mode != 0 && (force || t32_candidate(mode, m, n, k, batch))) {
      auto run_tc = [&](TC* Cd) {
        return t32_gemm(s, mode, m, n, k, as_f2(alpha), reinterpret_cast<const float*>(A), fl<TA>() * lda,
                        fl<TA>() * sA, reinterpret_cast<const float*>(B), fl<TB>() * ldb, fl<TB>() * sB, as_f2(beta),
                        Cd, ldc, sC, batch);
      };
      bool use = true;  // forced, or a candidate not yet measured inside a capture
      const TuneKey key{mode, size_class(m), size_class(n), size_class(k), size_class(batch),
                        (sB == 0 && batch > 1) ? 1 : 0};
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      cudaStreamIsCapturing(s, &cs);
      bool known = false;
      {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        auto it = g_tune.find(key);
        if (it != g_tune.end() && !force) {
          use = it->second;
          known = true;
        }
      }
      if (!known && !force && g_autotune && cs == cudaStreamCaptureStatusNone) {
        // measure both on a copy of C (the real C is written once, below)
        const long long span = (long long)(batch - 1) * sC + (long long)(m - 1) * ldc + n;
        TC* tmp = nullptr;
        if (cudaMalloc(&tmp, sizeof(TC) * span) == cudaSuccess) {
          long long* counter = g_launch_counter;
          g_launch_counter = nullptr;
          g_prof_suspended = true;
          cudaEvent_t ev[3];
          for (auto& e : ev) cudaEventCreate(&e);
          float best_tc = 1e30f, best_simt = 1e30f;
          bool tc_ok = true;
          for (int rep = 0; rep < 3 && tc_ok; ++rep) {
            cudaMemcpyAsync(tmp, C, sizeof(TC) * span, cudaMemcpyDeviceToDevice, s);
            cudaEventRecord(ev[0], s);
            tc_ok = run_tc(tmp);
            cudaEventRecord(ev[1], s);
            gemm_simt<TA, TB, TC>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, tmp, ldc, sC, batch);
            cudaEventRecord(ev[2], s);
            cudaEventSynchronize(ev[2]);
            float t1 = 0.f, t2 = 0.f;
            cudaEventElapsedTime(&t1, ev[0], ev[1]);
            cudaEventElapsedTime(&t2, ev[1], ev[2]);
            if (rep > 0) {
              best_tc = std::min(best_tc, t1);
              best_simt = std::min(best_simt, t2);
            }
          }
          for (auto& e : ev) cudaEventDestroy(e);
          cudaFree(tmp);
          g_prof_suspended = false;
          g_launch_counter = counter;
          use = tc_ok && best_tc < g_tc_margin * best_simt;
          std::lock_guard<std::mutex> lock(g_tune_mu);
          g_tune[key] = use;
        } else {
          cudaGetLastError();
        }
      }
      if (use && run_tc(C)) {
        g_last_gemm_tc = 1;
        return;
      }
    }
  }
  if constexpr (is_fp64<TC>::v)
    if (gemm_emulated<TA, TB, TC>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch)) return;
  gemm_simt<TA, TB, TC>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
}

namespace {
template <typename E> __global__ void k_identity(E* A, int n, int lda, long long sA) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)n * n) return;
  const int r = (int)(e / n), c = (int)(e % n);
  A[blockIdx.y * sA + (long long)r * lda + c] = r == c ? el<E>::one() : el<E>::zero();
}

// D[b] (NBB wide, holding the identity) <- the inverse of the n x n triangle at A.
template <typename E>
void tri_inverse(cudaStream_t s, const E* A, int lda, long long sA, int n, int mode, E* D, long long sD, int batch) {
  switch (trsm_cw(n, batch)) {
    case 8: launch_trsm_blk<E, 8>(s, A, lda, sA, 0, n, mode, D, NBB, sD, n, batch); return;
    case 4: launch_trsm_blk<E, 4>(s, A, lda, sA, 0, n, mode, D, NBB, sD, n, batch); return;
    case 2: launch_trsm_blk<E, 2>(s, A, lda, sA, 0, n, mode, D, NBB, sD, n, batch); return;
    default: launch_trsm_blk<E, 1>(s, A, lda, sA, 0, n, mode, D, NBB, sD, n, batch); return;
  }
}
}  // namespace

template <typename E>
void lu_factor(cudaStream_t s, E* A, int lda, long long sA, int n, int* piv, long long sP, int* info, int batch,
               const LuInv<E>& inv) {
  const E m1 = -el<E>::one(), one = el<E>::one();
  if (inv.d)
    for (int b = 0; b < batch; ++b) {
      const int blocks = 2 * ((n + NBB - 1) / NBB);
      k_identity<E><<<dim3(NBB * NBB / 256, blocks), 256, 0, s>>>(inv.d + b * inv.sd, NBB, NBB, (long long)NBB * NBB);
      HS_COUNT_LAUNCH();
    }
  // Two-level right-looking blocking: super-panels of NBB columns, each
  // factored as NB-wide pivoted panels whose updates stay inside the
  // super-panel; then U12 = L11^-1 A12 for the super-panel's rows and one
  // trailing update with k = NBB (the product the tensor cores take).
  for (int J0 = 0; J0 < n; J0 += NBB) {
    const int nbs = std::min(NBB, n - J0), J1 = J0 + nbs;
    for (int j0 = J0; j0 < J1; j0 += NB) {
      const int nb = std::min(NB, J1 - j0);
      lu_panel<E>(s, A, lda, sA, n, j0, nb, piv, sP, info, batch);  // row moves cover every column
      const int rin = J1 - j0 - nb;  // columns of the super-panel right of this panel
      if (rin > 0) {
        trsm_diag<E>(s, A, lda, sA, j0, nb, 0, A + j0 + nb, lda, sA, rin, batch);
        gemm<E, E, E>(s, OP_N, OP_N, n - j0 - nb, rin, nb, m1, A + (long long)(j0 + nb) * lda + j0, lda, sA,
                      A + (long long)j0 * lda + j0 + nb, lda, sA, one, A + (long long)(j0 + nb) * lda + j0 + nb, lda,
                      sA, batch);
      }
    }
    const int rest = n - J1;
    E* Li = inv.d ? inv.d + (long long)(J0 / NBB) * 2 * NBB * NBB : nullptr;
    if (inv.d) tri_inverse<E>(s, A + (long long)J0 * (lda + 1), lda, sA, nbs, 0, Li, inv.sd, batch);
    if (rest > 0) {
      // U12 = L11^-1 A12: on the tensor cores with the inverse (its operand is sliced
      // before the result is written, so in place), or by substitution
      bool done = false;
      if constexpr (is_fp64<E>::v)
        done = Li && gemm_emulated<E, E, E>(s, OP_N, OP_N, nbs, rest, nbs, one, Li, NBB, inv.sd,
                                            A + (long long)J0 * lda + J1, lda, sA, el<E>::zero(),
                                            A + (long long)J0 * lda + J1, lda, sA, batch);
      if (!done) trsm_blk<E>(s, A, lda, sA, J0, nbs, 0, A + J1, lda, sA, rest, batch);
      gemm<E, E, E>(s, OP_N, OP_N, rest, rest, nbs, m1, A + (long long)J1 * lda + J0, lda, sA,
                    A + (long long)J0 * lda + J1, lda, sA, one, A + (long long)J1 * lda + J1, lda, sA, batch);
    }
  }
  if (inv.d) {  // the inverses of the upper triangles: one launch for all whole blocks
    const int full = n / NBB, tail = n - full * NBB;
    E* Ui = inv.d + NBB * NBB;
    if (batch == 1 && full > 0)
      tri_inverse<E>(s, A, lda, (long long)NBB * (lda + 1), NBB, 1, Ui, 2LL * NBB * NBB, full);
    else
      for (int q = 0; q < full; ++q)
        tri_inverse<E>(s, A + (long long)q * NBB * (lda + 1), lda, sA, NBB, 1, Ui + q * 2LL * NBB * NBB, inv.sd, batch);
    if (tail > 0)
      tri_inverse<E>(s, A + (long long)full * NBB * (lda + 1), lda, sA, tail, 1, Ui + full * 2LL * NBB * NBB, inv.sd,
                     batch);
  }
}

template <typename E>
void lu_inverse(cudaStream_t s, const E* A, int lda, long long sA, int n, const int* piv, long long sP, E* Inv,
                int ldi, long long sI, int batch) {
  dim3 g((unsigned)(((long long)n * n + 255) / 256), batch);
  k_identity<E><<<g, 256, 0, s>>>(Inv, n, ldi, sI);
  HS_COUNT_LAUNCH();
  lu_solve<E>(s, OP_N, A, lda, sA, n, piv, sP, Inv, ldi, sI, n, batch);
}

template <typename E>
void lu_solve(cudaStream_t s, int trans, const E* A, int lda, long long sA, int n, const int* piv, long long sP, E* B,
              int ldb, long long sB, int nrhs, int batch, const LuInv<E>& inv) {
  dim3 gs((nrhs + 127) / 128, batch);
  const E m1 = -el<E>::one(), one = el<E>::one();
  if (inv.d && inv.tmp) {
    // With the diagonal blocks' inverses every step is a product: the first sweep
    // leaves its solution in tmp, the second one in B.  (One FP64 complex column:
    // 7 us a product, 53 us a block's substitution.)
    if (trans == OP_N) {
      k_swaps<E><<<gs, 128, 0, s>>>(piv, sP, n, 0, B, ldb, sB, nrhs);
      HS_COUNT_LAUNCH();
    }
    const int opd = trans, first = trans == OP_N ? 0 : 1;  // L then U, or U^T then L^T
    for (int c0 = 0; c0 < nrhs; c0 += inv.cols) {
      const int nc = std::min(inv.cols, nrhs - c0), ldt = inv.cols;
      const long long sT = (long long)n * ldt;
      E* b = B + c0;
      auto block = [&](int I0, int tri) { return inv.d + ((long long)(I0 / NBB) * 2 + tri) * NBB * NBB; };
      for (int I0 = 0; I0 < n; I0 += NBB) {
        const int I1 = std::min(n, I0 + NBB);
        E* y = inv.tmp + (long long)I0 * ldt;
        gemm<E, E, E>(s, opd, OP_N, I1 - I0, nc, I1 - I0, one, block(I0, first), NBB, inv.sd, b + (long long)I0 * ldb,
                      ldb, sB, el<E>::zero(), y, ldt, sT, batch);
        if (n - I1 > 0)
          gemm<E, E, E>(s, opd, OP_N, n - I1, nc, I1 - I0, m1,
                        trans == OP_N ? A + (long long)I1 * lda + I0 : A + (long long)I0 * lda + I1, lda, sA, y, ldt,
                        sT, one, b + (long long)I1 * ldb, ldb, sB, batch);
      }
      for (int I0 = (n - 1) / NBB * NBB; I0 >= 0; I0 -= NBB) {
        const int I1 = std::min(n, I0 + NBB);
        E* x = b + (long long)I0 * ldb;
        gemm<E, E, E>(s, opd, OP_N, I1 - I0, nc, I1 - I0, one, block(I0, 1 - first), NBB, inv.sd,
                      inv.tmp + (long long)I0 * ldt, ldt, sT, el<E>::zero(), x, ldb, sB, batch);
        if (I0 > 0)
          gemm<E, E, E>(s, opd, OP_N, I0, nc, I1 - I0, m1, trans == OP_N ? A + I0 : A + (long long)I0 * lda, lda, sA, x,
                        ldb, sB, one, inv.tmp, ldt, sT, batch);
      }
    }
    if (trans != OP_N) {
      k_swaps<E><<<gs, 128, 0, s>>>(piv, sP, n, 1, B, ldb, sB, nrhs);
      HS_COUNT_LAUNCH();
    }
    return;
  }
  if (trans == OP_N) {
    k_swaps<E><<<gs, 128, 0, s>>>(piv, sP, n, 0, B, ldb, sB, nrhs);
    HS_COUNT_LAUNCH();
    // blocks of NBB rows (one launch solves a block's diagonal triangle),
    // then one update of the remaining rows with k = NBB
    for (int I0 = 0; I0 < n; I0 += NBB) {  // L y = b
      const int I1 = std::min(n, I0 + NBB);
      trsm_blk<E>(s, A, lda, sA, I0, I1 - I0, 0, B, ldb, sB, nrhs, batch);
      if (n - I1 > 0)
        gemm<E, E, E>(s, OP_N, OP_N, n - I1, nrhs, I1 - I0, m1, A + (long long)I1 * lda + I0, lda, sA,
                      B + (long long)I0 * ldb, ldb, sB, one, B + (long long)I1 * ldb, ldb, sB, batch);
    }
    const int lastB = ((n - 1) / NBB) * NBB;
    for (int I0 = lastB; I0 >= 0; I0 -= NBB) {  // U x = y
      const int I1 = std::min(n, I0 + NBB);
      trsm_blk<E>(s, A, lda, sA, I0, I1 - I0, 1, B, ldb, sB, nrhs, batch);
      if (I0 > 0)
        gemm<E, E, E>(s, OP_N, OP_N, I0, nrhs, I1 - I0, m1, A + I0, lda, sA, B + (long long)I0 * ldb, ldb, sB, one, B,
                      ldb, sB, batch);
    }
  } else {
    for (int I0 = 0; I0 < n; I0 += NBB) {  // U^T y = b
      const int I1 = std::min(n, I0 + NBB);
      trsm_blk<E>(s, A, lda, sA, I0, I1 - I0, 2, B, ldb, sB, nrhs, batch);
      if (n - I1 > 0)
        gemm<E, E, E>(s, OP_T, OP_N, n - I1, nrhs, I1 - I0, m1, A + (long long)I0 * lda + I1, lda, sA,
                      B + (long long)I0 * ldb, ldb, sB, one, B + (long long)I1 * ldb, ldb, sB, batch);
    }
    const int lastB = ((n - 1) / NBB) * NBB;
    for (int I0 = lastB; I0 >= 0; I0 -= NBB) {  // L^T w = y
      const int I1 = std::min(n, I0 + NBB);
      trsm_blk<E>(s, A, lda, sA, I0, I1 - I0, 3, B, ldb, sB, nrhs, batch);
      if (I0 > 0)
        gemm<E, E, E>(s, OP_T, OP_N, I0, nrhs, I1 - I0, m1, A + (long long)I0 * lda, lda, sA, B + (long long)I0 * ldb,
                      ldb, sB, one, B, ldb, sB, batch);
    }
    k_swaps<E><<<gs, 128, 0, s>>>(piv, sP, n, 1, B, ldb, sB, nrhs);
    HS_COUNT_LAUNCH();
  }
}

// explicit instantiations
template void gemm<double, double, double>(cudaStream_t, int, int, int, int, int, double, const double*, int,
                                           long long, const double*, int, long long, double, double*, int, long long,
                                           int);
template void gemm<double2, double2, double2>(cudaStream_t, int, int, int, int, int, double2, const double2*, int,
                                              long long, const double2*, int, long long, double2, double2*, int,
                                              long long, int);
template void gemm<double, double2, double2>(cudaStream_t, int, int, int, int, int, double2, const double*, int,
                                             long long, const double2*, int, long long, double2, double2*, int,
                                             long long, int);
template void gemm<double2, double, double2>(cudaStream_t, int, int, int, int, int, double2, const double2*, int,
                                             long long, const double*, int, long long, double2, double2*, int,
                                             long long, int);
template void lu_factor<double>(cudaStream_t, double*, int, long long, int, int*, long long, int*, int,
                             const LuInv<double>&);
template void lu_factor<double2>(cudaStream_t, double2*, int, long long, int, int*, long long, int*, int,
                             const LuInv<double2>&);
template void lu_solve<double>(cudaStream_t, int, const double*, int, long long, int, const int*, long long, double*,
                               int, long long, int, int,
                               const LuInv<double>&);
template void lu_solve<double2>(cudaStream_t, int, const double2*, int, long long, int, const int*, long long,
                                double2*, int, long long, int, int,
                               const LuInv<double2>&);

template void gemm<float, float, float>(cudaStream_t, int, int, int, int, int, float, const float*, int, long long,
                                        const float*, int, long long, float, float*, int, long long, int);
template void gemm<float2, float2, float2>(cudaStream_t, int, int, int, int, int, float2, const float2*, int,
                                           long long, const float2*, int, long long, float2, float2*, int, long long,
                                           int);
template void gemm<float, float2, float2>(cudaStream_t, int, int, int, int, int, float2, const float*, int, long long,
                                          const float2*, int, long long, float2, float2*, int, long long, int);
template void gemm<float2, float, float2>(cudaStream_t, int, int, int, int, int, float2, const float2*, int,
                                          long long, const float*, int, long long, float2, float2*, int, long long,
                                          int);
template void lu_factor<float>(cudaStream_t, float*, int, long long, int, int*, long long, int*, int,
                             const LuInv<float>&);
template void lu_factor<float2>(cudaStream_t, float2*, int, long long, int, int*, long long, int*, int,
                             const LuInv<float2>&);
template void lu_inverse<double>(cudaStream_t, const double*, int, long long, int, const int*, long long, double*, int,
                                 long long, int);
template void lu_inverse<float>(cudaStream_t, const float*, int, long long, int, const int*, long long, float*, int,
                                long long, int);
template void lu_inverse<float2>(cudaStream_t, const float2*, int, long long, int, const int*, long long, float2*, int,
                                 long long, int);
template void lu_solve<float>(cudaStream_t, int, const float*, int, long long, int, const int*, long long, float*, int,
                              long long, int, int, const LuInv<float>&);
template void lu_solve<float2>(cudaStream_t, int, const float2*, int, long long, int, const int*, long long, float2*,
                               int, long long, int, int,
                               const LuInv<float2>&);

}  // namespace hs
