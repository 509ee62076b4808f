// FP32 matrix products of the mixed-precision path (see linalg.cuh).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include <cooperative_groups.h>

#include "linalg.cuh"

namespace cg = cooperative_groups;

namespace hs {
namespace {

// FP32 products (real or complex operands): TM x TN tile, RM x RN outputs per
// thread, operands staged by cp.async into a three-stage ring of 16-wide k-steps
// (16-byte copies where the rows are aligned to them, one element each
// otherwise; zero-filled at the edges), transposed operands in their own layout.
// The arithmetic is packed: fma.rn.f32x2 does two multiply-adds in one issue
// slot of two, so the loads and address work of the other slots no longer
// compete with it (scalar FFMAs: one slot each, 40-55% of the rate).  The FP32
// products of the k = 40 mixed batch: 15.7 -> 13.7 ms (batch 34.3 -> 32.6 ms),
// of the 64 x 64 leaf one at k = 35: 76 -> 68 ms; 60 TFLOP/s of 78 on the tiles of
// the largest leaf product (256 x 192 x 196 for 196 x 140 x 196: the rest is padding).
//   complex x complex: P += (ar, ar)(br, bi), Q += (ai, ai)(br, bi), the product
//     is (P.x - Q.y, P.y + Q.x); real x complex and complex x real: one; real:
//     two columns at a time.
// splits > 1: k split over a cluster, partial tiles summed in split order
// through distributed shared memory.
using u64 = unsigned long long;
__device__ __forceinline__ u64 pk2(float x, float y) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 upk2(u64 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void fma2(u64& d, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }

template <typename TA, typename TB> struct acc32;  // RN outputs of one row per thread
template <> struct acc32<float2, float2> {
  using TC = float2;
  template <int RN> struct row {
    u64 p[RN], q[RN];
    __device__ void zero() {
#pragma unroll
      for (int j = 0; j < RN; ++j) p[j] = q[j] = 0ull;
    }
    __device__ void add(float2 a, const float2 (&b)[RN]) {
      const u64 ar = pk2(a.x, a.x), ai = pk2(a.y, a.y);
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        const u64 bb = pk2(b[j].x, b[j].y);
        fma2(p[j], ar, bb);
        fma2(q[j], ai, bb);
      }
    }
    __device__ float2 get(int j) const {
      const float2 x = upk2(p[j]), y = upk2(q[j]);
      return make_float2(x.x - y.y, x.y + y.x);
    }
  };
};
template <> struct acc32<float, float2> {
  using TC = float2;
  template <int RN> struct row {
    u64 p[RN];
    __device__ void zero() {
#pragma unroll
      for (int j = 0; j < RN; ++j) p[j] = 0ull;
    }
    __device__ void add(float a, const float2 (&b)[RN]) {
      const u64 aa = pk2(a, a);
#pragma unroll
      for (int j = 0; j < RN; ++j) fma2(p[j], aa, pk2(b[j].x, b[j].y));
    }
    __device__ float2 get(int j) const { return upk2(p[j]); }
  };
};
template <> struct acc32<float2, float> {
  using TC = float2;
  template <int RN> struct row {
    u64 p[RN];
    __device__ void zero() {
#pragma unroll
      for (int j = 0; j < RN; ++j) p[j] = 0ull;
    }
    __device__ void add(float2 a, const float (&b)[RN]) {
      const u64 aa = pk2(a.x, a.y);
#pragma unroll
      for (int j = 0; j < RN; ++j) fma2(p[j], aa, pk2(b[j], b[j]));
    }
    __device__ float2 get(int j) const { return upk2(p[j]); }
  };
};
template <> struct acc32<float, float> {
  using TC = float;
  template <int RN> struct row {
    u64 p[RN / 2];
    __device__ void zero() {
#pragma unroll
      for (int j = 0; j < RN / 2; ++j) p[j] = 0ull;
    }
    __device__ void add(float a, const float (&b)[RN]) {
      const u64 aa = pk2(a, a);
#pragma unroll
      for (int j = 0; j < RN / 2; ++j) fma2(p[j], aa, pk2(b[2 * j], b[2 * j + 1]));
    }
    __device__ float get(int j) const { return j & 1 ? upk2(p[j / 2]).y : upk2(p[j / 2]).x; }
  };
};

constexpr int PK = 16, PST = 3;  // k-step, stages
template <typename TA, typename TB, int TM, int TN, int OPA, int OPB>
struct Cfg32 {
  using TC = typename acc32<TA, TB>::TC;
  // k-major rows are padded (16 bytes) so that neighbouring rows start in other banks
  static constexpr int AP = OPA == OP_N ? PK + 16 / (int)sizeof(TA) : TM;
  static constexpr int BP = OPB == OP_N ? TN : PK + 16 / (int)sizeof(TB);
  static constexpr int A_ST = (OPA == OP_N ? TM : PK) * AP * (int)sizeof(TA);
  static constexpr int B_ST = (OPB == OP_N ? PK : TN) * BP * (int)sizeof(TB);
  static constexpr int RING = PST * (A_ST + B_ST), RED = TM * TN * (int)sizeof(TC);
  static constexpr int SMEM = RING > RED ? RING : RED;
};


// One k-step of an operand: `lines` contiguous runs of `len` elements (rows
// along k, or k lines along the rows / columns) into dst (pitch P).
template <typename T, int LINES, int LEN, int P, int NT>
__device__ __forceinline__ void stage32(T* dst, const T* src, long long ld, int line0, int nline, int e0, int nelem,
                                        bool wide, int tid) {
  constexpr int E = 16 / (int)sizeof(T);
  if (wide) {
#pragma unroll
    for (int q = tid; q < LINES * (LEN / E); q += NT) {
      const int l = q / (LEN / E), x = (q % (LEN / E)) * E;
      const int valid = line0 + l < nline ? max(0, min(E, nelem - e0 - x)) : 0;
      cp16(dst + l * P + x, valid ? src + (line0 + l) * ld + e0 + x : src, valid * (int)sizeof(T));
    }
  } else {
#pragma unroll 4
    for (int q = tid; q < LINES * LEN; q += NT) {
      const int l = q / LEN, x = q % LEN;
      const bool ok = line0 + l < nline && e0 + x < nelem;
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + l * P + x);
      const T* p = ok ? src + (line0 + l) * ld + e0 + x : src;
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(p), "n"((int)sizeof(T)),
                   "r"(ok ? (int)sizeof(T) : 0)
                   : "memory");
    }
  }
}

template <typename TA, typename TB, int TM, int TN, int RM, int RN, int OPA, int OPB>
__global__ void __launch_bounds__((TM / RM) * (TN / RN), (TM / RM) * (TN / RN) > 128 ? 2 : 4)
    k_gemm32(int m, int n, int k, typename acc32<TA, TB>::TC alpha, const TA* __restrict__ A, int lda, long long sA,
             const TB* __restrict__ B, int ldb, long long sB, typename acc32<TA, TB>::TC beta,
             typename acc32<TA, TB>::TC* __restrict__ C, int ldc, long long sC, int splits, int wideA, int wideB) {
  using Cf = Cfg32<TA, TB, TM, TN, OPA, OPB>;
  using TC = typename Cf::TC;
  constexpr int TX = TN / RN, TY = TM / RM, NT = TX * TY;
  extern __shared__ __align__(16) unsigned char pipe_smem[];
  const int b = blockIdx.z / splits, sp = blockIdx.z % splits;
  A += b * sA;
  B += b * sB;
  C += b * sC;
  const int kc = ((k + splits - 1) / splits + PK - 1) / PK * PK;
  const int kbeg = sp * kc, kend = min(k, kbeg + kc);
  const int nsteps = kend > kbeg ? (kend - kbeg + PK - 1) / PK : 0;
  const int row0 = blockIdx.y * TM, col0 = blockIdx.x * TN;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  auto As = [&](int st) { return reinterpret_cast<TA*>(pipe_smem + st * (Cf::A_ST + Cf::B_ST)); };
  auto Bs = [&](int st) { return reinterpret_cast<TB*>(pipe_smem + st * (Cf::A_ST + Cf::B_ST) + Cf::A_ST); };
  auto issue = [&](int step, int st) {
    const int k0 = kbeg + step * PK;
    if constexpr (OPA == OP_N)
      stage32<TA, TM, PK, Cf::AP, NT>(As(st), A, lda, row0, m, k0, kend, wideA, tid);
    else
      stage32<TA, PK, TM, Cf::AP, NT>(As(st), A, lda, k0, kend, row0, m, wideA, tid);
    if constexpr (OPB == OP_N)
      stage32<TB, PK, TN, Cf::BP, NT>(Bs(st), B, ldb, k0, kend, col0, n, wideB, tid);
    else
      stage32<TB, TN, PK, Cf::BP, NT>(Bs(st), B, ldb, col0, n, k0, kend, wideB, tid);
  };
  // the thread's rows ty + TY i and column pairs 2 tx + 2 TX (j / 2) + j % 2
  typename acc32<TA, TB>::template row<RN> acc[RM];
#pragma unroll
  for (int i = 0; i < RM; ++i) acc[i].zero();
#pragma unroll
  for (int st = 0; st < PST - 1; ++st) {
    if (st < nsteps) issue(st, st);
    cp_commit();
  }
  for (int step = 0; step < nsteps; ++step) {
    cp_wait<PST - 2>();
    __syncthreads();  // stage `step` landed for every thread; slot (step - 1) % PST is free
    if (step + PST - 1 < nsteps) issue(step + PST - 1, (step + PST - 1) % PST);
    cp_commit();
    const TA* as = As(step % PST);
    const TB* bs = Bs(step % PST);
#pragma unroll
    for (int kk = 0; kk < PK; ++kk) {
      TB bb[RN];
#pragma unroll
      for (int j = 0; j < RN; j += 2) {
        const int c = 2 * tx + TX * j;
        if constexpr (OPB == OP_N) {
          struct alignas(2 * sizeof(TB)) two { TB x, y; };
          const two v = *reinterpret_cast<const two*>(bs + kk * Cf::BP + c);
          bb[j] = v.x;
          bb[j + 1] = v.y;
        } else {
          bb[j] = bs[c * Cf::BP + kk];
          bb[j + 1] = bs[(c + 1) * Cf::BP + kk];
        }
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
        acc[i].add(OPA == OP_N ? as[(ty + TY * i) * Cf::AP + kk] : as[kk * Cf::AP + ty + TY * i], bb);
    }
  }
  cp_wait<0>();
  __syncthreads();
  auto put = [&](int r, int c, TC v) {
    v = scal<TC, TC>(alpha, v);
    const long long o = (long long)r * ldc + c;
    if (!is_zero(beta)) v = addv(v, scal<TC, TC>(beta, C[o]));
    C[o] = v;
  };
  if (splits > 1) {
    TC* red = reinterpret_cast<TC*>(pipe_smem);  // the ring is free now
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j) red[(ty + TY * i) * TN + 2 * tx + TX * (j & ~1) + (j & 1)] = acc[i].get(j);
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int rows_per = (TM + splits - 1) / splits;
    const int rb = sp * rows_per, re = min(TM, rb + rows_per);
    for (int e = rb * TN + tid; e < re * TN; e += NT) {
      TC sum = el<TC>::zero();
      for (int q = 0; q < splits; ++q) sum = addv(sum, cl.map_shared_rank(red, q)[e]);
      const int r = row0 + e / TN, c = col0 + e % TN;
      if (r < m && c < n) put(r, c, sum);
    }
    cl.sync();  // keep this CTA's partial tile alive until every rank has read it
    return;
  }
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const int r = row0 + ty + TY * i, c = col0 + 2 * tx + TX * (j & ~1) + (j & 1);
      if (r < m && c < n) put(r, c, acc[i].get(j));
    }
}

template <typename TA, typename TB, int TM, int TN, int RM, int RN, int OPA, int OPB, typename TC>
void launch_gemm32(cudaStream_t s, int m, int n, int k, TC alpha, const TA* A, int lda, long long sA, const TB* B,
                   int ldb, long long sB, TC beta, TC* C, int ldc, long long sC, int batch, int splits) {
  constexpr int smem = Cfg32<TA, TB, TM, TN, OPA, OPB>::SMEM, NT = (TM / RM) * (TN / RN);
  auto kernel = k_gemm32<TA, TB, TM, TN, RM, RN, OPA, OPB>;
  if constexpr (smem > 48 * 1024) {
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr[dev]) {
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (dev >= 0 && dev < 64) attr[dev] = true;
    }
  }
  constexpr int EA = 16 / (int)sizeof(TA), EB = 16 / (int)sizeof(TB);
  const int wideA = lda % EA == 0 && sA % EA == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const int wideB = ldb % EB == 0 && sB % EB == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((n + TN - 1) / TN, (m + TM - 1) / TM, batch * splits);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = splits;
  cfg.attrs = at;
  cfg.numAttrs = splits > 1 ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, splits, wideA, wideB);
  HS_COUNT_LAUNCH();
}

// FP32 tile and k splits by the busiest SM's estimated clocks: 128 multiply-adds
// a clock at 3/4 (4 x 4 outputs per thread) or half (4 x 2) of the rate, and a
// latency per CTA.  Real left operands (the leaves' 196 and 56 rows) also take 56
// rows and 48 columns where that pads less: 196 x 140 x 196 over 4096 leaves 224 x 144
// instead of 256 x 192, 2.63 -> 2.35 ms.  For complex ones those tiles were
// slower than their padding (the 64 x 64 leaf batch at k = 35: 48.3 against 45.6 ms).
template <typename TA, typename TB, typename TC>
void gemm32(cudaStream_t s, int opA, int opB, int m, int n, int k, TC alpha, const TA* A, int lda, long long sA,
            const TB* B, int ldb, long long sB, TC beta, TC* C, int ldc, long long sC, int batch) {
  constexpr double fma = (sizeof(TA) / 4) * (sizeof(TB) / 4);
  constexpr bool all_tiles = sizeof(TA) == 4;
  int tm = 64, tn = 64, splits = 1;
  double bt = 1e300;
  for (int tile = 0; tile < 5; ++tile) {
    const int cm = tile == 4 ? 32 : tile < 2 ? 64 : 56, cn = tile == 4 ? 32 : tile % 2 ? 48 : 64;
    if (tile > 0 && tile < 4 && (!all_tiles || opB != OP_N)) continue;
    for (int sp = 1; sp <= 8; ++sp) {
      if (sp > 1 && (k / sp < 64 || (long long)batch * sp > 65535)) break;
      if ((m + cm - 1) / cm > 65535) continue;  // grid.y
      const double ctas = (double)((m + cm - 1) / cm) * ((n + cn - 1) / cn) * batch * sp;
      const double kc = ((k + sp - 1) / sp + PK - 1) / PK * PK;
      const double one = cm * cn * fma * kc / 128.0 / (tile < 4 ? 0.75 : 0.5);
      const double time = std::ceil(ctas / 152.0) * one + 1500.0 * std::ceil(ctas / 608.0) + (sp > 1 ? 1500.0 : 0.0);
      if (time < bt) {
        bt = time;
        tm = cm;
        tn = cn;
        splits = sp;
      }
    }
  }
  auto go = [&](auto oa, auto ob) {
    constexpr int OA = decltype(oa)::value, OB = decltype(ob)::value;
    auto run = [&](auto launch) { launch(s, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, splits); };
    if constexpr (all_tiles && OB == OP_N) {
      if (tm == 64 && tn == 48) return run(launch_gemm32<TA, TB, 64, 48, 4, 4, OA, OB, TC>);
      if (tm == 56 && tn == 64) return run(launch_gemm32<TA, TB, 56, 64, 4, 4, OA, OB, TC>);
      if (tm == 56) return run(launch_gemm32<TA, TB, 56, 48, 4, 4, OA, OB, TC>);
    }
    if (tm == 64) run(launch_gemm32<TA, TB, 64, 64, 4, 4, OA, OB, TC>);
    else run(launch_gemm32<TA, TB, 32, 32, 4, 2, OA, OB, TC>);
  };
  using N = std::integral_constant<int, OP_N>;
  using T = std::integral_constant<int, OP_T>;
  if (opA == OP_N && opB == OP_N) go(N{}, N{});
  else if (opA == OP_T && opB == OP_N) go(T{}, N{});
  else if (opA == OP_N) go(N{}, T{});
  else go(T{}, T{});
}

}  // namespace

template <>
void gemm_fp32<float2, float2, float2>(cudaStream_t s, int opA, int opB, int m, int n, int k, float2 alpha, const float2* A, int lda,
                    long long sA, const float2* B, int ldb, long long sB, float2 beta, float2* C, int ldc, long long sC, int batch) {
  gemm32<float2, float2, float2>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
}
template <>
void gemm_fp32<float, float2, float2>(cudaStream_t s, int opA, int opB, int m, int n, int k, float2 alpha, const float* A, int lda,
                    long long sA, const float2* B, int ldb, long long sB, float2 beta, float2* C, int ldc, long long sC, int batch) {
  gemm32<float, float2, float2>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
}
template <>
void gemm_fp32<float2, float, float2>(cudaStream_t s, int opA, int opB, int m, int n, int k, float2 alpha, const float2* A, int lda,
                    long long sA, const float* B, int ldb, long long sB, float2 beta, float2* C, int ldc, long long sC, int batch) {
  gemm32<float2, float, float2>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
}
template <>
void gemm_fp32<float, float, float>(cudaStream_t s, int opA, int opB, int m, int n, int k, float alpha, const float* A, int lda,
                    long long sA, const float* B, int ldb, long long sB, float beta, float* C, int ldc, long long sC, int batch) {
  gemm32<float, float, float>(s, opA, opB, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch);
}

}  // namespace hs
