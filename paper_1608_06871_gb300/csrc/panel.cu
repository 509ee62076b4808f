// LU panel factorisation (columns [j0, j0 + nb) of a batch of n x n matrices)
// for the blocked right-looking LU of linalg.cu.
//
// Panels of up to 4096 rows are factored with partial pivoting by one
// thread-block cluster per matrix (k_panel_cluster).
//
// Taller panels (root systems above 64 leaves per side, normal matrices) use
// tournament pivoting: sets of up to 256 rows are factored independently with
// partial pivoting (one CTA each) and each keeps its nb pivot rows; the
// candidates of 8 sets form the next round's sets until one set remains, whose
// partial-pivoting order gives the panel's pivot rows.  Those rows are swapped
// to the top (LAPACK swap sequence in piv) with their factored nb x nb block
// from the final round (partial pivoting inside the pivot rows reproduces that
// order), and the multipliers below solve L21 U11 = A21.  The sets of a round are
// independent, so the per-column latency of the pivot search is paid on 256
// rows in shared memory instead of on the whole column in global memory.
//
// Scratch for the candidate lists lives in piv[j0 + nb .. n) of each matrix,
// which later panels overwrite: for m = n - j0 > 256 rows it needs
// ceil(m / 256) nb + ... + 1 + 4 nb ints, below m - nb for nb = 32.
#include <algorithm>
#include <climits>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "linalg.cuh"

namespace hs {
namespace {

constexpr int PR = 256;      // rows per shared-memory tile (one thread per row)
constexpr int PNB = 32;      // panel width of the blocked LU
constexpr int PT = 256;      // threads of the tile kernels
constexpr int APPLY_CH = 32;  // columns per CTA of the row-permutation kernel

// Magnitude used for pivot selection, in the panel's own precision.
template <typename E> struct pmag;
template <> struct pmag<double> { using T = double; __device__ static double of(double a) { return fabs(a); } };
template <> struct pmag<double2> { using T = double; __device__ static double of(double2 a) { return a.x * a.x + a.y * a.y; } };
template <> struct pmag<float> { using T = float; __device__ static float of(float a) { return fabsf(a); } };
template <> struct pmag<float2> { using T = float; __device__ static float of(float2 a) { return a.x * a.x + a.y * a.y; } };

// 1 / x with one correctly rounded reciprocal: real x directly; complex x as
// conj(x) / |x|^2, or, where |x|^2 could leave the normal range, x = 2^e (a + i b)
// with the power of two from the larger component's exponent (exact), then
// (a - i b) / (a^2 + b^2) 2^-e.  The multipliers are formed as x_i (1 / pivot),
// as LAPACK's unblocked LU does.
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip(double x) { return __drcp_rn(x); }
__device__ __forceinline__ float2 recip(float2 x) {
  const float n2 = fmaf(x.x, x.x, x.y * x.y);
  if (n2 > 1e-30f && n2 < 1e30f) {  // |x|^2 safely inside the normal range
    const float d = __frcp_rn(n2);
    return make_float2(x.x * d, -x.y * d);
  }
  const int e = ilogbf(fmaxf(fabsf(x.x), fabsf(x.y)));
  const float a = scalbnf(x.x, -e), b = scalbnf(x.y, -e);
  const float d = scalbnf(__frcp_rn(fmaf(a, a, b * b)), -e);
  return make_float2(a * d, -b * d);
}
__device__ __forceinline__ double2 recip(double2 x) {
  const double n2 = fma(x.x, x.x, x.y * x.y);
  if (n2 > 1e-290 && n2 < 1e290) {
    const double d = __drcp_rn(n2);
    return make_double2(x.x * d, -x.y * d);
  }
  const int e = ilogb(fmax(fabs(x.x), fabs(x.y)));
  const double a = scalbn(x.x, -e), b = scalbn(x.y, -e);
  const double d = scalbn(__drcp_rn(fma(a, a, b * b)), -e);
  return make_double2(a * d, -b * d);
}

// Factor the rows x nb tile T (row stride ld, shared memory) with partial
// pivoting, one thread per row (blockDim.x = PT >= rows).  The rows stay where
// they are: each thread tracks the logical position of its own row (mylg), a
// pivot step only relabels two rows, and the thread whose row became a pivot
// row stops updating it, so every other thread can read the pivot row in
// place.  Per column there is a single barrier, after the warps publish their
// candidates (magnitude, then lowest logical position, as LAPACK's first
// maximum; FP32 magnitudes are reduced with redux.sync on their bit
// patterns).  The column loop is not unrolled (a small instruction footprint:
// the per-column latency is the point here); the thread keeps its row in
// registers and mirrors every updated entry to the tile.
// On return, loc[r] is the tile row holding logical row r, rid[] is permuted
// into logical order, and *zc is lowered to the first column whose pivot is
// exactly zero (that column is then left unscaled).
template <typename E>
__device__ void tile_lu(E* T, int ld, int rows, int nb, int* rid, int* loc, int* zc) {
  using M = typename pmag<E>::T;
  constexpr int NW = PT / 32;
  __shared__ M wbest[2][NW];
  __shared__ int wkey[2][NW];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int steps = min(rows, nb);
  bool active = t < rows;
  int mylg = t;
  const int myid = active ? rid[t] : 0;
  E* row = T + t * ld;
  // the thread's row in registers (entries right of the current column are
  // the live ones); shared memory holds a mirror that the others read when
  // this row becomes the pivot row
  E r[PNB];
#pragma unroll
  for (int c = 0; c < PNB; ++c) r[c] = (active && c < nb) ? row[c] : el<E>::zero();
  for (int j = 0; j < steps; ++j) {
    const int pb = j & 1;
    M best = active ? pmag<E>::of(row[j]) : M(-1);
    int key = active ? (mylg << 8) | t : INT_MAX;  // logical position, then tile row
    if constexpr (sizeof(M) == 4) {
      // FP32 magnitudes: the warp maximum of their bit patterns (ordered for
      // non-negative floats; +1 keeps an active zero above an inactive row),
      // then the smallest key among the lanes holding it: two redux.sync
      unsigned mb = active ? __float_as_uint(best) + 1u : 0u;
      mb = __reduce_max_sync(0xffffffffu, mb);
      key = (int)__reduce_min_sync(0xffffffffu, (active && __float_as_uint(best) + 1u == mb) ? (unsigned)key
                                                                                            : 0xffffffffu);
      if (lane == 0) { wbest[pb][warp] = __uint_as_float(mb); wkey[pb][warp] = key; }
      __syncthreads();
      const unsigned wb = lane < NW ? __float_as_uint(wbest[pb][lane]) : 0u;
      const unsigned wk = lane < NW ? (unsigned)wkey[pb][lane] : 0xffffffffu;
      const unsigned bb = __reduce_max_sync(0xffffffffu, wb);
      key = (int)__reduce_min_sync(0xffffffffu, wb == bb ? wk : 0xffffffffu);
    } else {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const M ob = __shfl_down_sync(0xffffffffu, best, o);
        const int ok = __shfl_down_sync(0xffffffffu, key, o);
        if (ob > best || (ob == best && ok < key)) { best = ob; key = ok; }
      }
      if (lane == 0) { wbest[pb][warp] = best; wkey[pb][warp] = key; }
      __syncthreads();
      best = wbest[pb][0];
      key = wkey[pb][0];
#pragma unroll
      for (int w = 1; w < NW; ++w) {
        const M ob = wbest[pb][w];
        const int ok = wkey[pb][w];
        if (ob > best || (ob == best && ok < key)) { best = ob; key = ok; }
      }
    }
    const int p = key & 255, lp = key >> 8;
    if (t == p) {
      active = false;
      mylg = j;
    } else if (mylg == j) {
      mylg = lp;
    }
    const E* prow = T + p * ld;
    const E pv = prow[j];
    if (!(pmag<E>::of(pv) > M(0))) {
      if (t == 0) atomicMin(zc, j);
    } else if (active) {
      const E l = row[j] * recip(pv);
      row[j] = l;
      // rank-1 update in registers, in groups of eight columns (groups left of
      // the column are skipped, warp-uniformly); each group's pivot entries are
      // loaded before its mirror stores are issued
#pragma unroll
      for (int g = 0; g < PNB / 8; ++g) {
        if (8 * g + 7 > j) {
          E u[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) u[q] = 8 * g + q < nb ? prow[8 * g + q] : el<E>::zero();
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int c = 8 * g + q;
            if (c > j && c < nb) {
              r[c] = fmsc(r[c], l, u[q]);
              row[c] = r[c];
            }
          }
        }
      }
    }
  }
  __syncthreads();
  if (t < rows) {
    loc[mylg] = t;
    rid[mylg] = myid;
  }
  __syncthreads();
}

// Stage rows x nb elements into the tile T (row stride ld): tile row r is
// source row ids[r] of A (row stride lda).  One warp per row, lanes along the
// columns, eight rows in flight per warp.
template <typename E>
__device__ void load_rows(E* T, int ld, int rows, int nb, const E* A, int lda, const int* ids) {
  constexpr int NW = PT / 32, RF = 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r0 = warp * RF; r0 < rows; r0 += NW * RF) {
    E v[RF];
#pragma unroll
    for (int q = 0; q < RF; ++q) {
      const int r = r0 + q;
      v[q] = (r < rows && lane < nb) ? A[(long long)ids[r] * lda + lane] : el<E>::zero();
    }
#pragma unroll
    for (int q = 0; q < RF; ++q)
      if (r0 + q < rows && lane < nb) T[(r0 + q) * ld + lane] = v[q];
  }
}

// One tournament round: set blockIdx.x of matrix blockIdx.y.  Round 0 takes
// rows j0 + 256 s .. ; later rounds take up to 256 candidate rows from the
// previous round's list (entries < 0 are empty).  Writes the set's nb pivot
// rows (absolute row numbers, in pivot order) to out, or, in the final round
// (one set), the factored pivot block, the LAPACK swap sequence
// piv[j0 .. j0 + nb) and the list of rows to move.
template <typename E>
__global__ void __launch_bounds__(PT) k_tp_select(E* A, int lda, long long sA, int n, int j0, int nb, int* piv,
                                                  long long sP, int* info, int in_off, int nin, int out_off,
                                                  int final_round, int aff_off) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* T = reinterpret_cast<E*>(smem_raw);
  __shared__ int rid[PR], loc[PR];
  __shared__ int wsum[PT / 32];
  __shared__ int zc;
  __shared__ int kpos[2 * PNB], korig[2 * PNB];
  const int b = blockIdx.y, set = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  A += b * sA;
  piv += b * sP;
  int* W = piv + j0 + nb;  // scratch: rows of later panels' pivots
  int myrow = -1;
  if (in_off < 0) {
    const int r = j0 + set * PR + t;
    if (r < n) myrow = r;
  } else {
    const int e = set * PR + t;
    if (e < nin) myrow = W[in_off + e];
  }
  // compact the valid rows, in order (ballot prefix sums)
  const unsigned bal = __ballot_sync(0xffffffffu, myrow >= 0);
  if (lane == 0) wsum[warp] = __popc(bal);
  if (t == 0) zc = INT_MAX;
  __syncthreads();
  int off = 0, rows = 0;
  for (int w = 0; w < PT / 32; ++w) {
    if (w < warp) off += wsum[w];
    rows += wsum[w];
  }
  if (myrow >= 0) rid[off + __popc(bal & ((1u << lane) - 1u))] = myrow;
  __syncthreads();
  const int ld = nb + 1;
  load_rows<E>(T, ld, rows, nb, A + j0, lda, rid);
  __syncthreads();
  tile_lu<E>(T, ld, rows, nb, rid, loc, &zc);
  if (!final_round) {
    if (t < nb) W[out_off + set * nb + t] = t < rows ? rid[t] : -1;
    return;
  }
  // the top nb rows of T are the factored pivot block (L11 \ U11): store it
  // in the pivot rows' panel columns, which the row moves carry to j0 .. j0 + nb
  for (int e = t; e < nb * nb; e += PT) {
    const int r = e / nb, c = e % nb;
    A[(long long)rid[r] * lda + j0 + c] = T[loc[r] * ld + c];
  }
  if (t == 0) {
    if (zc != INT_MAX && info[b] == 0) info[b] = j0 + zc + 1;
    // LAPACK swap sequence bringing rid[0 .. nb) to rows j0 .. j0 + nb, and
    // the resulting moves (kpos[k] now holds original row korig[k])
    int np = 0;
    const int steps = min(rows, nb);
    for (int j = 0; j < steps; ++j) {
      const int target = j0 + j, pj = rid[j];
      int q = pj;
      for (int k = 0; k < np; ++k)
        if (korig[k] == pj) { q = kpos[k]; break; }
      piv[j0 + j] = q;
      if (q != target) {
        int it = -1, iq = -1, vt = target;
        for (int k = 0; k < np; ++k) {
          if (kpos[k] == target) { it = k; vt = korig[k]; }
          if (kpos[k] == q) iq = k;
        }
        if (it < 0) { kpos[np] = target; it = np++; }
        korig[it] = pj;
        if (iq < 0) { kpos[np] = q; iq = np++; }
        korig[iq] = vt;
      }
    }
    int k2 = 0;
    int* aff = W + aff_off;
    for (int k = 0; k < np; ++k)
      if (korig[k] != kpos[k]) {
        aff[1 + k2] = kpos[k];
        aff[1 + 2 * PNB + k2] = korig[k];
        ++k2;
      }
    aff[0] = k2;
  }
}

// Move the rows listed by the final round (all n columns), through shared memory.
template <typename E>
__global__ void __launch_bounds__(PT) k_tp_apply(E* A, int lda, long long sA, int n, const int* piv, long long sP,
                                                 int aff_at) {
  __shared__ E buf[2 * PNB * APPLY_CH];
  const int b = blockIdx.y, t = threadIdx.x, c0 = blockIdx.x * APPLY_CH;
  A += b * sA;
  const int* aff = piv + b * sP + aff_at;
  const int na = aff[0];
  for (int e = t; e < na * APPLY_CH; e += PT) {
    const int a = e / APPLY_CH, c = c0 + e % APPLY_CH;
    if (c < n) buf[e] = A[(long long)aff[1 + 2 * PNB + a] * lda + c];
  }
  __syncthreads();
  for (int e = t; e < na * APPLY_CH; e += PT) {
    const int a = e / APPLY_CH, c = c0 + e % APPLY_CH;
    if (c < n) A[(long long)aff[1 + a] * lda + c] = buf[e];
  }
}

// Solve L21 U11 = A21 for the rows below the (factored, moved) pivot block,
// one thread per row.
constexpr int FIN_T = 128;
template <typename E>
__global__ void __launch_bounds__(FIN_T) k_tp_finish(E* A, int lda, long long sA, int n, int j0) {
  __shared__ E U[PNB][PNB + 1];
  const int b = blockIdx.y, t = threadIdx.x;
  A += b * sA;
  for (int e = t; e < PNB * PNB; e += FIN_T) U[e / PNB][e % PNB] = A[(long long)(j0 + e / PNB) * lda + j0 + e % PNB];
  __syncthreads();
  const int r = j0 + PNB + blockIdx.x * FIN_T + t;
  if (r >= n) return;
  E* row = A + (long long)r * lda + j0;
  E x[PNB];
#pragma unroll
  for (int c = 0; c < PNB; ++c) x[c] = row[c];
#pragma unroll
  for (int c = 0; c < PNB; ++c) {
#pragma unroll
    for (int i = 0; i < c; ++i) x[c] = fmsc(x[c], x[i], U[i][c]);
    if (el<E>::mag2(U[c][c]) > 0.0) x[c] = el<E>::div(x[c], U[c][c]);
  }
#pragma unroll
  for (int c = 0; c < PNB; ++c) row[c] = x[c];
}

void set_smem_once(const void* f, size_t bytes, bool wide_cluster = false) {
  static std::mutex mu;
  static std::vector<std::pair<const void*, int>> done;  // (kernel, device)
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  for (auto& d : done)
    if (d.first == f && d.second == dev) return;
  cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (wide_cluster) cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  done.emplace_back(f, dev);
}

// ---- panels of up to 4096 rows: one thread-block cluster per matrix ---------
//
// The panel's rows are dealt to the CTAs of a cluster (RPC rows each) and stay
// there, one thread per row and group of PNB / G columns (RPC G = 256), its
// entries in registers with a mirror in shared memory.  Rows are relabelled
// instead of moved.  Per column: the owners of the column reduce their
// magnitudes (redux.sync on the leading 32 bits, then the lowest logical row),
// the CTA's candidate row, its key and the reciprocal of its pivot go to every
// CTA of the cluster through distributed shared memory, and after one cluster
// barrier each CTA picks the best candidate and updates its rows from its local
// copy.  Buffers alternate, so a column needs one CTA and one cluster barrier.
// This is partial pivoting over the whole column (up to 2^-20 of the
// magnitude), the multipliers come out with it, and the cluster also applies
// the exchanges to the columns outside the panel.
// What bounds it: in FP64 the pipe (two thread-operations per SM and clock, m
// nb^2 / 2 multiply-adds of the panel), hence the spread over up to 16 SMs and
// the reciprocal formed by one warp instead of by every row's thread; in FP32
// the two barriers.  It replaces a 256-row CTA per set (180 us for a complex
// FP64 panel of 256 rows, on one SM's pipe; 93 us now) and, above 256 rows, the
// tournament of such sets with a separate solve for the multipliers (620 us at
// 1792 rows; 210 us now).  The panels of the k = 40 FP64 batch: 50 -> 18.5 ms.
__device__ __forceinline__ uint32_t cl_map(const void* p, uint32_t rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_st(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_st(uint32_t a, float v) { cl_st(a, __float_as_uint(v)); }
__device__ __forceinline__ void cl_st(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_st(uint32_t a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cl_st(uint32_t a, double2 v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ uint32_t cl_ld(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Leading 32 bits of a magnitude, ordered as the magnitude is; + 1 so that an
// active zero ranks above no row.
__device__ __forceinline__ unsigned mag_bits(float m) { return __float_as_uint(m) + 1u; }
__device__ __forceinline__ unsigned mag_bits(double m) { return (unsigned)__double2hiint(m) + 1u; }

constexpr int PC_MAX = 16;    // CTAs per cluster
constexpr int PC_STAGE = 64;  // columns staged at a time when the exchanges are applied

template <typename E, int RPC> struct PcSmem {
  static constexpr int LD = PNB + 1;
  static constexpr size_t tile = sizeof(E) * (size_t)(RPC * LD > 2 * PNB * PC_STAGE ? RPC * LD : 2 * PNB * PC_STAGE);
  static constexpr size_t crow = sizeof(E) * 2 * PC_MAX * PNB;
  static constexpr size_t cinv = sizeof(E) * 2 * PC_MAX;
  static constexpr size_t bytes = tile + crow + cinv;
};

template <typename E, int RPC>
__global__ void __launch_bounds__(PT) k_panel_cluster(E* A, int lda, long long sA, int n, int j0, int nb, int* piv,
                                                      long long sP, int* info, int nc) {
  using S = PcSmem<E, RPC>;
  using M = typename pmag<E>::T;
  constexpr int G = PT / RPC, CG = PNB / G, LD = S::LD, NW = PT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* T = reinterpret_cast<E*>(smem_raw);
  E(*crow)[PC_MAX][PNB] = reinterpret_cast<E(*)[PC_MAX][PNB]>(smem_raw + S::tile);
  E(*cinv)[PC_MAX] = reinterpret_cast<E(*)[PC_MAX]>(smem_raw + S::tile + S::crow);
  __shared__ unsigned cmag[2][PC_MAX], ckey[2][PC_MAX];
  __shared__ unsigned wmag[2][NW], wkey[2][NW];
  __shared__ int sp[PNB], naff, aff_d[2 * PNB], aff_s[2 * PNB];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned rank = nc > 1 ? blockIdx.x % nc : 0;
  const int b = blockIdx.x / nc;
  A += b * sA;
  piv += b * sP;
  const int m = n - j0, row0 = (int)rank * RPC, rows = max(0, min(RPC, m - row0));
  const int tr = t % RPC, g = t / RPC;  // the thread's row, column group
  if (t == 0) naff = 0;
  for (int e = t; e < rows * nb; e += PT) {
    const int r = e / nb, c = e % nb;
    T[r * LD + c] = A[(long long)(j0 + row0 + r) * lda + j0 + c];
  }
  if (nc > 1) cl_sync(); else __syncthreads();  // (every CTA runs before another writes to its memory)
  bool active = tr < rows;
  const bool mine = active;
  int mylg = row0 + tr;
  E* row = T + tr * LD;
  E r[CG];
#pragma unroll
  for (int c = 0; c < CG; ++c) r[c] = (active && g * CG + c < nb) ? row[g * CG + c] : el<E>::zero();
  const int steps = min(m, nb);
  int zc = INT_MAX;
  for (int j = 0; j < steps; ++j) {
    const int pb = j & 1;
    unsigned mb = 0u, key = 0xffffffffu;
    if (g == j / CG) {  // (whole warps: RPC is a multiple of 32)
      const unsigned mm = active ? mag_bits(pmag<E>::of(row[j])) : 0u;
      mb = __reduce_max_sync(0xffffffffu, mm);
      key = __reduce_min_sync(0xffffffffu, active && mm == mb ? ((unsigned)mylg << 8) | (unsigned)tr : 0xffffffffu);
    }
    if (lane == 0) {
      wmag[pb][warp] = mb;
      wkey[pb][warp] = key;
    }
    __syncthreads();
    {
      const unsigned wb = lane < NW ? wmag[pb][lane] : 0u, wk = lane < NW ? wkey[pb][lane] : 0xffffffffu;
      mb = __reduce_max_sync(0xffffffffu, wb);
      key = __reduce_min_sync(0xffffffffu, wb == mb ? wk : 0xffffffffu);
    }
    // this CTA's candidate to every CTA: warp w serves CTAs w, w + 8; a CTA
    // without active rows sends magnitude 0
    const E* prow = T + (key & 255u) * LD;
    if (mb > 0u) {
      for (int d = warp; d < nc; d += NW)
        if (lane < nb) cl_st(cl_map(&crow[pb][rank][lane], d), prow[lane]);
      if (warp == NW - 1) {
        const E pv = prow[j];
        const E inv = pmag<E>::of(pv) > M(0) ? recip(pv) : el<E>::zero();
        if (lane < nc) cl_st(cl_map(&cinv[pb][rank], lane), inv);
      }
    }
    if (warp == 0 && lane < nc) {
      cl_st(cl_map(&cmag[pb][rank], lane), mb);
      cl_st(cl_map(&ckey[pb][rank], lane), key);
    }
    if (nc > 1) cl_sync(); else __syncthreads();
    const unsigned cb = lane < nc ? cmag[pb][lane] : 0u, ck = lane < nc ? ckey[pb][lane] : 0xffffffffu;
    const unsigned best = __reduce_max_sync(0xffffffffu, cb);
    const unsigned bkey = __reduce_min_sync(0xffffffffu, cb == best ? ck : 0xffffffffu);
    const int win = __ffs(__ballot_sync(0xffffffffu, cb == best && ck == bkey)) - 1;
    const int lp = (int)(bkey >> 8);
    if (t == 0) sp[j] = lp;
    if (win == (int)rank && tr == (int)(bkey & 255u)) {
      active = false;
      mylg = j;
    } else if (mylg == j) {
      mylg = lp;
    }
    const E* u = crow[pb][win];
    if (!(pmag<E>::of(u[j]) > M(0))) {
      zc = min(zc, j);  // the column is left unscaled
    } else if (active) {
      const E l = row[j] * cinv[pb][win];
#pragma unroll
      for (int c = 0; c < CG; ++c) {
        const int cc = g * CG + c;
        if (cc > j && cc < nb) {
          r[c] = fmsc(r[c], l, u[cc]);
          row[cc] = r[c];
        } else if (cc == j) {
          r[c] = l;  // (the mirror keeps the unscaled entry: the row's other threads read it)
        }
      }
    }
  }
  // rows to their places; the list of exchanged rows collects in CTA 0
  if (mine) {
    E* out = A + (long long)(j0 + mylg) * lda + j0;
#pragma unroll
    for (int c = 0; c < CG; ++c)
      if (g * CG + c < nb) out[g * CG + c] = r[c];
    if (g == 0 && mylg != row0 + tr) {
      uint32_t slot;
      asm volatile("atom.shared::cluster.add.u32 %0, [%1], 1;" : "=r"(slot) : "r"(cl_map(&naff, 0)) : "memory");
      cl_st(cl_map(&aff_d[slot], 0), (uint32_t)(j0 + mylg));
      cl_st(cl_map(&aff_s[slot], 0), (uint32_t)(j0 + row0 + tr));
    }
  }
  if (rank == 0 && t == 0 && zc != INT_MAX && info[b] == 0) info[b] = j0 + zc + 1;
  if (nc > 1) cl_sync(); else __syncthreads();
  if (rank == 0 && t < steps) piv[j0 + t] = j0 + sp[t];  // (thread 0 wrote sp, the last entry after the loop's barrier)
  const int na = (int)cl_ld(cl_map(&naff, 0));
  if (rank != 0 && t < na) {
    aff_d[t] = (int)cl_ld(cl_map(&aff_d[t], 0));
    aff_s[t] = (int)cl_ld(cl_map(&aff_s[t], 0));
  }
  if (nc > 1) cl_sync(); else __syncthreads();  // nobody reads another CTA's memory after this
  // the same exchanges on the columns outside the panel, staged through T
  const int out_cols = n - nb, chunks = (out_cols + PC_STAGE - 1) / PC_STAGE;
  for (int ch = (int)rank; ch < chunks && na > 0; ch += nc) {
    const int c0 = ch * PC_STAGE;
    for (int e = t; e < na * PC_STAGE; e += PT) {
      const int a = e / PC_STAGE, cc = c0 + e % PC_STAGE;
      if (cc < out_cols) T[e] = A[(long long)aff_s[a] * lda + (cc < j0 ? cc : cc + nb)];
    }
    __syncthreads();
    for (int e = t; e < na * PC_STAGE; e += PT) {
      const int a = e / PC_STAGE, cc = c0 + e % PC_STAGE;
      if (cc < out_cols) A[(long long)aff_d[a] * lda + (cc < j0 ? cc : cc + nb)] = T[e];
    }
    __syncthreads();
  }
}

template <typename E, int RPC>
void launch_cluster(cudaStream_t s, E* A, int lda, long long sA, int n, int j0, int nb, int* piv, long long sP,
                    int* info, int batch, int nc) {
  const size_t smem = PcSmem<E, RPC>::bytes;
  set_smem_once((const void*)k_panel_cluster<E, RPC>, smem, true);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(batch * nc));
  cfg.blockDim = dim3(PT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_panel_cluster<E, RPC>, A, lda, sA, n, j0, nb, piv, sP, info, nc);
  HS_COUNT_LAUNCH();
}

// Rows per CTA for a panel of m rows: the fewest (the widest spread) that keep
// the cluster within PC_MAX CTAs and the batch within one CTA per SM (more
// CTAs would only queue: 1024 leaf matrices of 196 rows take one CTA each, 413 us a
// panel against 670 before); 0 where the panel has more than PC_MAX * 256 rows.
int cluster_rows(int m, int batch) {
  for (int rpc : {32, 64, 128, 256}) {
    const int nc = (m + rpc - 1) / rpc;
    if (nc <= PC_MAX && ((long long)nc * batch <= 152 || rpc == 256)) return rpc;
  }
  return 0;
}

}  // namespace

template <typename E>
void lu_panel(cudaStream_t s, E* A, int lda, long long sA, int n, int j0, int nb, int* piv, long long sP, int* info,
              int batch) {
  const int m = n - j0;
  const size_t tile_bytes = (size_t)PR * (PNB + 1) * sizeof(E);
  if (const int rpc = cluster_rows(m, batch)) {
    int nc = 1;
    while (nc * rpc < m) nc *= 2;
    auto go = [&](auto r) {
      launch_cluster<E, decltype(r)::value>(s, A, lda, sA, n, j0, nb, piv, sP, info, batch, nc);
    };
    if (rpc == 32) go(std::integral_constant<int, 32>{});
    else if (rpc == 64) go(std::integral_constant<int, 64>{});
    else if (rpc == 128) go(std::integral_constant<int, 128>{});
    else go(std::integral_constant<int, 256>{});
    return;
  }
  // tournament (nb == PNB here: only the last panel is narrower, and it is short)
  set_smem_once((const void*)k_tp_select<E>, tile_bytes);
  int sets = (m + PR - 1) / PR, total = 0;
  for (int k = sets; k > 1; k = (k * nb + PR - 1) / PR) total += k * nb;  // lists of the non-final rounds
  const int aff_off = total;
  int in_off = -1, nin = 0, out_off = 0;
  for (;;) {
    const int fin = sets == 1;
    k_tp_select<E><<<dim3(sets, batch), PT, tile_bytes, s>>>(A, lda, sA, n, j0, nb, piv, sP, info, in_off, nin,
                                                             out_off, fin, aff_off);
    HS_COUNT_LAUNCH();
    if (fin) break;
    in_off = out_off;
    nin = sets * nb;
    out_off += nin;
    sets = (nin + PR - 1) / PR;
  }
  k_tp_apply<E><<<dim3((n + APPLY_CH - 1) / APPLY_CH, batch), PT, 0, s>>>(A, lda, sA, n, piv, sP,
                                                                          j0 + nb + aff_off);
  HS_COUNT_LAUNCH();
  k_tp_finish<E><<<dim3((m - PNB + FIN_T - 1) / FIN_T, batch), FIN_T, 0, s>>>(A, lda, sA, n, j0);
  HS_COUNT_LAUNCH();
}

template void lu_panel<double>(cudaStream_t, double*, int, long long, int, int, int, int*, long long, int*, int);
template void lu_panel<double2>(cudaStream_t, double2*, int, long long, int, int, int, int*, long long, int*, int);
template void lu_panel<float>(cudaStream_t, float*, int, long long, int, int, int, int*, long long, int*, int);
template void lu_panel<float2>(cudaStream_t, float2*, int, long long, int, int, int, int*, long long, int*, int);

}  // namespace hs
