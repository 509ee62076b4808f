// Batched dense linear algebra on the GPU (row-major, FP64 real or complex).
//
// These are the dense building blocks of the direct solver of Sec. 2: the leaf
// factorisations, the interface systems of the merges and the exterior
// coupling system are LU factorisations with partial pivoting; every other
// step is a (batched) matrix product.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace hs {

enum { OP_N = 0, OP_T = 1 };

// C[b] = alpha * op(A[b]) * op(B[b]) + beta * C[b] for b < batch, row-major,
// op = identity or plain transpose (no conjugation).  beta == 0 never reads C.
template <typename TA, typename TB, typename TC>
void gemm(cudaStream_t s, int opA, int opB, int m, int n, int k, TC alpha, const TA* A, int lda,
          long long sA, const TB* B, int ldb, long long sB, TC beta, TC* C, int ldc, long long sC,
          int batch);

// Scratch (OzScratch) with which gemm() takes such a complex FP64 product to the tensor
// cores in one go; 0 where it runs on the FP64 pipe.
size_t zgemm_scratch_bytes(int m, int n, int k, int batch);

// The FP32 kernels behind gemm() (gemm32.cu), for the four operand forms.
template <typename TA, typename TB, typename TC>
void gemm_fp32(cudaStream_t s, int opA, int opB, int m, int n, int k, TC alpha, const TA* A, int lda, long long sA,
               const TB* B, int ldb, long long sB, TC beta, TC* C, int ldc, long long sC, int batch);

template <>
void gemm_fp32<float2, float2, float2>(cudaStream_t, int, int, int, int, int, float2, const float2*, int, long long, const float2*, int, long long, float2, float2*,
                    int, long long, int);
template <>
void gemm_fp32<float, float2, float2>(cudaStream_t, int, int, int, int, int, float2, const float*, int, long long, const float2*, int, long long, float2, float2*,
                    int, long long, int);
template <>
void gemm_fp32<float2, float, float2>(cudaStream_t, int, int, int, int, int, float2, const float2*, int, long long, const float*, int, long long, float2, float2*,
                    int, long long, int);
template <>
void gemm_fp32<float, float, float>(cudaStream_t, int, int, int, int, int, float, const float*, int, long long, const float*, int, long long, float, float*,
                    int, long long, int);

// Inverses of the 128-row diagonal blocks of an LU (unit lower and upper
// triangle), kept with the factors where a system is solved with again and again:
// d[b sd + (2 block + (0: L, 1: U)) 128^2] (leading dimension 128), and room for a
// copy of `cols` right-hand sides, tmp[b n cols + row cols + column].  Every step of
// a solve is then a product.  The substitution of a 128-row block is a chain
// bound by FP64 latency on as many SMs as there are columns; the root solves and the
// few large merges at the top of an FP64 tree (at most four systems of more than 128 rows:
// below that the batched substitutions fill the chip) gain: solve for one incidence
// at k = 5 554 -> 372 us, k = 5 Gauss-Newton step 5.55 -> 5.34 ms, k = 20 gradient
// 27.7 -> 26.1, k = 40 FP64 batch 61.7 -> 58.9 ms; errors against 64 bits unchanged.
template <typename E> struct LuInv {
  E* d = nullptr;
  long long sd = 0;
  E* tmp = nullptr;
  int cols = 0;
};
inline size_t lu_inv_elems(int n) { return (size_t)((n + 127) / 128) * 2 * 128 * 128; }

// In-place LU with partial pivoting P A = L U of a batch of n x n matrices.
// piv[j] (0-based) is the row swapped with row j at step j.  info[b] is set to
// j+1 at the first exactly-zero pivot of matrix b (it must be zeroed first).
template <typename E>
void lu_factor(cudaStream_t s, E* A, int lda, long long sA, int n, int* piv, long long sP, int* info,
               int batch, const LuInv<E>& inv = {});

// Inv[b] = A[b]^{-1} (n x n, leading dimension ldi) from the factors of
// lu_factor (identity right-hand sides through lu_solve).
template <typename E>
void lu_inverse(cudaStream_t s, const E* A, int lda, long long sA, int n, const int* piv, long long sP, E* Inv,
                int ldi, long long sI, int batch);

// Factor the panel columns [j0, j0 + nb) (nb <= 32) of the batch with row
// pivoting and apply the row swaps to whole rows (panel.cu); piv[j0 .. j0+nb)
// receives the swaps, piv[j0+nb .. n) is used as scratch.
template <typename E>
void lu_panel(cudaStream_t s, E* A, int lda, long long sA, int n, int j0, int nb, int* piv, long long sP, int* info,
              int batch);

// Solve A X = B (trans = OP_N) or A^T X = B (trans = OP_T) in place in B
// (n x nrhs, leading dimension ldb) from the factors of lu_factor.
template <typename E>
void lu_solve(cudaStream_t s, int trans, const E* A, int lda, long long sA, int n, const int* piv,
              long long sP, E* B, int ldb, long long sB, int nrhs, int batch, const LuInv<E>& inv = {});


// FP32 products on the tensor cores by a two-term TF32 split (tc32.cu):
// C = alpha A B + beta C, row-major, no transposes; mode 2: complex A and B,
// mode 1: real A, complex B, mode 0: real A and B (alpha, beta real: .x).
// Leading dimensions and batch strides of A and B in floats, of C in
// elements.  Returns false (nothing launched) when the product cannot run
// there (switched off, or no scratch while the stream is being captured).
bool t32_gemm(cudaStream_t s, int mode, int m, int n, int k, float2 alpha, const float* A, long long lda,
              long long sA, const float* B, long long ldb, long long sB, float2 beta, void* C, int ldc, long long sC,
              int batch);
// gemm() measures, once per shape, the tensor-core and the SIMT product and
// keeps the faster (g_autotune; off: a fixed size rule); g_last_gemm_tc is 1
// when the calling thread's last gemm() ran on the tensor cores.
extern bool g_autotune;
extern float g_tc_margin;  // the tensor cores are kept where they take < g_tc_margin of the SIMT time

// Tensor-core use for FP32 products (hs_set_tensor_cores): 0 never; 1 (the
// default) where the per-shape measurement finds them clearly faster; 2 every
// supported product.
extern int g_t32_mode;
extern thread_local bool g_prof_suspended;
extern thread_local int g_last_gemm_tc;
// Synchronises s, then reads and clears this device's flags that a bounded
// tensor-core wait gave up (the split-TF32 product's, the emulated-FP64 one's,
// and the one the host raises in tests; tcgemm.cu).
bool tc_timed_out(cudaStream_t s);
// One kernel family's flag: enqueues a copy of it to *v or (clear) of *v, a zero, to it.
void oz_timeout_flag(cudaStream_t s, int* v, bool clear);
void t32_timeout_flag(cudaStream_t s, int* v, bool clear);
cudaError_t tc_raise_timeout_flag();
// The host raised a flag that no check has read yet.
bool tc_timeout_raised();
// Set by the tensor-core products that the calling thread launches, where it points
// somewhere: the owner of the work then reads the flags once it has waited for it.
extern thread_local bool* g_tc_pending;

// FP64 products on the tensor cores by exact BF16 slices (ozaki.cu).
// Output view: element (b, i, j) at p[b sb + (i / ig) si + (i % ig) sg + j sk]
// (ig = 2 writes real rows 2 r, 2 r + 1 as the parts of complex rows).
struct OzView {
  double* p;
  long long sb, si, sg, sk;
  int ig;
};
// Source of an operand's rows (A's rows, or B's columns): entry (b, i, k), strides in doubles.
//   OZ_REAL    p[i sr + k sk]
//   OZ_PAIR    rows 2 r + q are the parts q of complex rows r: p[r sr + k sk + q]
//   OZ_PAIR_I  the same of i times those rows: (-im, re)
//   OZ_CLEFT   k = 2 l + q runs over the parts of a complex row: p[i sr + l sk + q]
//   OZ_CRIGHT  the right operand to OZ_CLEFT: rows 2 j, 2 j + 1 are (re, -im), (im, re)
//              of complex column j along k = 2 l + q, p[j sr + l sk + ...]
enum { OZ_REAL = 0, OZ_PAIR = 1, OZ_CLEFT = 2, OZ_CRIGHT = 3, OZ_PAIR_I = 4 };
struct OzSrc {
  const double* p;
  long long sb, sr, sk;
  int kind;
};
extern bool g_oz_enabled;
// Scratch bytes of ozaki_gemm for these sizes; with the operands' bytes (oz_operand_bytes)
// alone it runs too, without planes.
size_t ozaki_scratch_bytes(int m, int n, int k, int batch, bool b_shared);
// C[b] = alpha A[b] B[b] + beta C[b] (m x n, k inner; beta = 0 never reads C), sizes of the
// real product; b_shared: one B for every batch; sym: only the 128 x 32 tiles that meet the
// lower triangle are computed.  Returns cudaErrorInvalidValue on bad sizes, or the error of a
// launch, which also stays the CUDA runtime's last error.
cudaError_t ozaki_gemm(cudaStream_t s, int m, int n, int k, int batch, double alpha, OzSrc A, OzSrc Bt, bool b_shared,
                       double beta, OzView C, void* scratch, size_t scratch_bytes, bool sym = false);
// The same in two steps, for an operand used by many products: oz_slice cuts
// an operand into oz_operand_bytes of slices, once; oz_multiply multiplies two
// sliced operands.  planes (oz_plane_bytes, may be NULL): with fewer tiles than
// SMs the pieces of k run as separate tiles into FP64 planes summed in order.
size_t oz_operand_bytes(int rows, int k, int batch, bool is_a);
size_t oz_plane_bytes(int m, int n, int k, int batch);
void oz_slice(cudaStream_t s, OzSrc v, int rows, int k, int batch, bool is_a, void* buf);
cudaError_t oz_multiply(cudaStream_t s, int m, int n, int k, int batch, double alpha, const void* Aop, const void* Bop,
                        bool b_shared, double beta, OzView C, void* planes = nullptr, bool sym = false);
// Device scratch for the emulated products behind gemm<FP64>: set for the
// calling thread by whoever owns the stream's work (a context for the length
// of a call); without it FP64 products stay on the FP64 pipe.
struct OzScratch {
  char* p = nullptr;
  size_t bytes = 0;
};
extern thread_local const OzScratch* g_oz_scratch;
// Keeps the FP64 products enqueued in its scope on the FP64 pipe.
struct PipeScope {
  const OzScratch* const held = g_oz_scratch;
  PipeScope() { g_oz_scratch = nullptr; }
  ~PipeScope() { g_oz_scratch = held; }
  PipeScope(const PipeScope&) = delete;
  PipeScope& operator=(const PipeScope&) = delete;
};
// Estimated clocks of an emulated product on the whole chip (sizes of the real product).
double oz_cycles(int m, int n, int k, int batch, bool b_shared);
// Fields on the interior grid ([field][gy][gx], nX x nX) in the fixed point of
// oz_slice_khatri_rao, in place; their row exponents to exps (oz_fix_bytes).
size_t oz_fix_bytes(int fields, int nX);
void oz_fix_fields(cudaStream_t s, double2* F, int fields, int nX, void* exps);
// The left operand of the Jacobian's x-projection for the pairs c0 .. c0 + nc - 1
// of d * P + p, sliced straight from the fixed-point fields: rows 2 (c nX + gy) + part of
// u_d z_p over gx (2 nc nX rows, k = nX; oz_operand_bytes(2 nc nX, nX, 1, true)).
void oz_slice_khatri_rao(cudaStream_t s, const double2* Ug, const double2* Zg, const void* eu, const void* ez, int P,
                         int nX, long long c0, int nc, void* buf);

}  // namespace hs
