// FP64 matrix products on the 5th-generation tensor cores by exact integer
// slices (error-free splitting in the manner of Ozaki, Ogita, Oishi and Rump,
// 2012, with row / column scaling as in Ozaki, Uchino and Imamura's later
// variants), for the FP64 contractions of the Jacobian, the exterior rows of the mixed
// solver and the larger products of the FP64 one (gemm_emulated).
//
// C = alpha A B (+ beta C), A m x k and B k x n real FP64.  Every row i of A
// is scaled by 2^-ea_i so that its largest entry lies in [1/2, 1), every
// column j of B by 2^-eb_j, and the scaled values are split exactly into
// S = 8 slices of beta = 7 bits:
//   x 2^-e = sum_s a_s 2^(-7 (s + 1)) + tail,  a_0 in [-128, 128], a_s in [-64, 64],
// each an integer, hence exact in BF16.  The product of two slices is then an
// exact integer matrix; summed in FP32 it stays exact while every partial sum
// is an integer below 2^24.  The anti-diagonal d = s + t of the slice pairs
// (s + t <= 7: 36 pairs) carries the weight 2^(-7 (d + 2)), so the pairs of one
// diagonal accumulate into one FP32 accumulator in tensor memory:
//   |partial sum| <= K 4096 (d + 3) < 2^24  for K <= 384,
// which bounds the k extent of one piece (longer products sum their pieces in
// FP64).  The epilogue recombines the 8 diagonal sums exactly in integers and
// rounds them once to the double, formed from its bits.  What an entry of C can be
// off by is set by the largest entries of its row and column: 2^-56 of each from the
// 56-bit fixed point, and the pairs with s + t >= 8 left out, at most 3.6 2^-55 a term:
//   below 1.25 k u max|A_i.| max|B_.j|   (u = 2^-53),
// besides one rounding per piece and those of the sum of the pieces.  An FP64 product's
// bound is k u |A_i.| |B_.j|: about the same where the entries of a row are of one size,
// far smaller where they are graded against the column's (there this product loses
// bits that FP64 keeps; the leaf elimination stays on the FP64 pipe for that reason).
// A complex product is one real product: rows of A as (re, im) pairs along k,
// columns of B as the pairs (re, -im) and (im, re).
//
// Kernel: one persistent CTA per SM, 128 x 32 output tiles; warp 0 copies the
// 32-wide k-steps of the tile's slices (stored by the slicing kernels in the
// MMA operand layout, 64 + 16 KB in one piece each) into a two-stage ring with
// cp.async.bulk, warp 1 issues the tcgen05 BF16 MMAs (M = 128, N = 32 to 256,
// K = 16; 16 per stage of 32 k) into the eight diagonal accumulators (two sets of
// 256 TMEM columns), sixteen warps read them back.  Every mbarrier wait is
// bounded; a timeout sets the library's tensor-core timeout flag.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "linalg.cuh"

namespace hs {

bool prof_active(int family);
void prof_begin(cudaStream_t s, cudaEvent_t* a);
void prof_end(cudaStream_t s, cudaEvent_t a, double flops);

// Set to 1 by an emulated-FP64 product whose bounded mbarrier wait gave up
// (read and cleared by tc_timed_out with the tensor-core GEMM's own flag).
__device__ int g_oz_timeout = 0;

namespace {

constexpr int OZ_S = 8;          // slices per operand
constexpr int OZ_ND = 8;         // anti-diagonals kept (s + t <= 7)
constexpr int OZ_TM = 128;       // rows per tile
constexpr int OZ_TN = 32;        // columns per tile
constexpr int OZ_ACC = OZ_ND * OZ_TN;  // TMEM columns of one set of diagonal accumulators (two sets)
constexpr int OZ_KS = 32;        // k per stage
constexpr int OZ_KMAX = 384;     // k per piece keeping every diagonal sum below 2^24 (a multiple of 32)
constexpr int OZ_EPI = 16;       // epilogue warps
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI;  // warp 0 TMA, warp 1 MMA, the others epilogue
constexpr int OZ_A_SL = OZ_TM * 2 * OZ_KS;  // one slice of the A tile: 128 rows x 64 bytes (8 KB)
constexpr int OZ_B_SL = OZ_TN * 2 * OZ_KS;  // same for B (2 KB)
constexpr int OZ_STAGE = OZ_S * (OZ_A_SL + OZ_B_SL);  // 80 KB
constexpr int OZ_SMEM = 2 * OZ_STAGE + 1024;
constexpr long long OZ_WAIT = 1LL << 26;
constexpr int OZ_SR = 16;        // rows per CTA of the slicing kernel
// instruction descriptor: D = F32, A = B = BF16, both K-major, M = 128, N = n
__host__ __device__ constexpr uint32_t oz_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_TM >> 4) << 24);
}

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// K-major, 64-byte swizzle: rows of 64 bytes (32 BF16),
// atoms of 8 rows (512 bytes, the 8-row group stride); the k offset inside the
// row is added to the start address.
__device__ __forceinline__ uint64_t oz_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

__device__ __forceinline__ bool oz_wait(uint32_t bar, uint32_t parity) {
  for (long long it = 0; it < OZ_WAIT; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void oz_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(bar)
      : "memory");
}

// Where the pair of entries (row r, k, k + 1) of slice 0 lies in a sliced operand,
// in 32-bit words; slice s follows at s OZ_ROW TR.  The operand is stored as
// the product reads it: blocks [row tile of TR rows][32-wide k-step][slice][row],
// rows of 64 bytes with the 64-byte swizzle of the MMA operand layout (16-byte
// chunk c of row r at c ^ ((r / 2) % 4)), so a stage is one contiguous copy.
constexpr int OZ_ROW = 16;  // words per row
template <int TR>
__device__ __forceinline__ long long oz_at(long long r, int k, int nst) {
  const int rr = (int)(r % TR), kk = k % OZ_KS;
  return ((r / TR * nst + k / OZ_KS) * OZ_S * TR + rr) * OZ_ROW + ((((kk >> 3) ^ (rr >> 1)) & 3) << 2) + ((kk & 7) >> 1);
}

__device__ __forceinline__ void oz_ld8(uint32_t ta, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(ta));
}

// The slices of two k-neighbours N0, N1 (56-bit fixed point, |N| < 2^56), one
// 32-bit store per slice: the 8 balanced base-128 digits a_s of N,
// sum_s a_s 2^(49 - 7 s) = N, |a_0| <= 128, the others in [-64, 63].  With
// B = sum_(s>0) 64 2^(49 - 7 s), the digits of N + B are its bit fields less 64
// (the top one as it is).  Both numbers' fields are taken at once: a byte
// permutation puts 16-bit windows of the two side by side, one shift and one
// logical operation leave both fields under the BF16 128 (0x4300, unit 1), and a
// packed subtraction of 192 gives the two exact BF16 digits.  The signed top digits get
// their floats from 1.5 2^23 added below them.  (Field by field, with an FP32
// subtraction each, the pair took 45 logical operations instead of 24, and the
// slicing kernels were bound by them.)
__device__ __forceinline__ void put2(long long N0, long long N1, uint32_t* o, int plane) {
  constexpr long long B = (64LL << 42) | (64LL << 35) | (64LL << 28) | (64LL << 21) | (64LL << 14) | (64LL << 7) | 64LL;
  static_assert(OZ_S == 8, "seven fields and the top digit");
  N0 += B;
  N1 += B;
  auto top = [](long long n) { return __float_as_uint(__int_as_float(0x4B400000 + (int)(n >> 49)) - 12582912.0f); };
  o[0] = __byte_perm(top(N0), top(N1), 0x7632);
  auto digits = [](uint32_t w, int off) {
    uint32_t d;
    asm("sub.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(((w >> off) & 0x007F007Fu) | 0x43004300u), "r"(0x43404340u));
    return d;
  };
  const uint32_t l0 = (uint32_t)N0, l1 = (uint32_t)N1, h0 = (uint32_t)((unsigned long long)N0 >> 28),
                 h1 = (uint32_t)((unsigned long long)N1 >> 28);
  const uint32_t h01 = __byte_perm(h0, h1, 0x5410), l01 = __byte_perm(l0, l1, 0x5410);
  o[1 * plane] = digits(__byte_perm(h0, h1, 0x6521), 6);
  o[2 * plane] = digits(h01, 7);
  o[3 * plane] = digits(h01, 0);
  o[4 * plane] = digits(__byte_perm(l0, l1, 0x7632), 5);
  o[5 * plane] = digits(__byte_perm(l0, l1, 0x6521), 6);
  o[6 * plane] = digits(l01, 7);
  o[7 * plane] = digits(l01, 0);
}

// Row i of an operand's real form: entries 2 j and 2 j + 1 lie at p[j step + a0] and
// p[j step + a1], negated where f0, f1 say so.
struct OzRowAt {
  const double* p;
  long long step, a0, a1;
  bool f0, f1;
};
__device__ __forceinline__ OzRowAt row_at(const OzSrc& v, long long b, int i) {
  const int odd = i & 1;
  const double* p = v.p + b * v.sb;
  switch (v.kind) {
    case OZ_REAL: return {p + i * v.sr, 2 * v.sk, 0, v.sk, false, false};
    case OZ_PAIR: return {p + (i >> 1) * v.sr + odd, 2 * v.sk, 0, v.sk, false, false};
    case OZ_PAIR_I: return {p + (i >> 1) * v.sr + 1 - odd, 2 * v.sk, 0, v.sk, !odd, !odd};  // i times it: (-im, re)
    case OZ_CLEFT: return {p + i * v.sr, v.sk, 0, 1, false, false};
    default: return {p + (i >> 1) * v.sr, v.sk, odd, 1 - odd, false, !odd};  // OZ_CRIGHT: [re, -im; im, re]
  }
}

struct OzSliced {  // an operand and where its slices go
  OzSrc v;
  int rows, rpad, k, pl, nst;
  long long total;  // padded rows of all batches
  uint32_t* out;
  int* e;
};

// The slices of 16 rows and one piece of k, two rows a warp.
template <int TR>
__device__ __forceinline__ void slice_rows(const OzSliced& o, int block, double* tile) {
  const int k0 = blockIdx.y * o.pl, kc = min(o.pl, o.k - k0), kp = (kc + OZ_KS - 1) / OZ_KS * OZ_KS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, pitch = o.pl + 1;
  const long long r0 = (long long)block * OZ_SR, b = r0 / o.rpad;  // (rpad is a multiple of the 16 rows)
  const int i0 = (int)(r0 - b * o.rpad);
  auto entry = [&](const OzRowAt& at, bool row, int kk) {
    if (!row || kk >= kc) return 0.0;
    const double x = at.p[(k0 + kk) / 2 * at.step + (kk & 1 ? at.a1 : at.a0)];
    return (kk & 1 ? at.f1 : at.f0) ? -x : x;
  };
  if (o.v.sk <= 2) {  // along k, each warp its own rows
#pragma unroll
    for (int r = warp; r < OZ_SR; r += 8) {
      const OzRowAt at = row_at(o.v, b, min(i0 + r, o.rows - 1));
#pragma unroll 4
      for (int kk = lane; kk < kp; kk += 32) tile[r * pitch + kk] = entry(at, i0 + r < o.rows, kk);
    }
    __syncwarp();
  } else {  // along the rows where those are the contiguous direction
    const int r = threadIdx.x % OZ_SR;
    const OzRowAt at = row_at(o.v, b, min(i0 + r, o.rows - 1));
#pragma unroll 4
    for (int kk = threadIdx.x / OZ_SR; kk < kp; kk += 256 / OZ_SR)
      tile[r * pitch + kk] = entry(at, i0 + r < o.rows, kk);
    __syncthreads();
  }
  for (int r = warp; r < OZ_SR; r += 8) {
    const double* x = tile + r * pitch;
    long long mx = 0;
    for (int kk = lane; kk < kp; kk += 32) mx = max(mx, abs_bits(x[kk]));
    for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const int ex = row_exp(mx);
    if (lane == 0) o.e[blockIdx.y * o.total + r0 + r] = ex;
    for (int kk = 2 * lane; kk < kp; kk += 64)
      put2(fixed56(x[kk], ex), fixed56(x[kk + 1], ex), o.out + oz_at<TR>(r0 + r, k0 + kk, o.nst), OZ_ROW * TR);
  }
}

// Slices of the rows of one or both operands of a product (A's rows, or B's
// columns), one CTA per 16 rows and piece of k (the first na CTAs: A),
// written in blocks (oz_at, row b * rpad + i; BF16, zero padded), the piece's row
// exponents to e[piece][b * rpad + i].  The block is read once through shared memory
// (along k, or along the rows where those are the contiguous direction), the row's largest magnitude
// fixes e with max 2^-e in [1/2, 1), and each entry becomes the 56-bit fixed-point integer
// N = round(x 2^(56 - e)), |N| < 2^56, whose balanced base-128 digits are the
// slices and represent N exactly.  Integer arithmetic throughout (the FP64 pipe
// is the scarce unit).  Padding rows get zero slices.
// Most launches are small (the products of one merge or panel update) and bound by
// latency: with two launches a product, 64-bit divisions per entry and
// a block barrier they took 15 to 17 us each.  One launch, one division a block, rows loaded
// and sliced by the same warp: 10.2 -> 6.2 ms for the 209 products of a k = 40 FP64 batch
// (58.3 -> 55.3 ms), k = 20 gradient 25.8 -> 23.8 ms, k = 5 Gauss-Newton step 5.3 -> 5.1.
// (Pairs of k-neighbours loaded straight into registers: faster for the small launches, but the
// strided loads cost the large ones more, 60.2 ms.)
__global__ void __launch_bounds__(256) k_oz_slice(const __grid_constant__ OzSliced A, const __grid_constant__ OzSliced B,
                                                  unsigned na) {
  extern __shared__ double tile[];
  if (blockIdx.x < na)
    slice_rows<OZ_TM>(A, blockIdx.x, tile);
  else
    slice_rows<OZ_TN>(B, blockIdx.x - na, tile);
}

// Fields in fixed point, in place: each row piece (gx in one piece of k) of a
// field is scaled by 2^-e so that its largest part lies in [1/2, 1) and every
// part becomes U = round(x 2^(55 - e)) = U1 2^28 + U0 with both halves signed
// (|U1|, |U0| <= 2^27): (re1, re0, im1, im0) takes the place of the double2.
// e[row npc + piece]; one warp per row piece.
__global__ void __launch_bounds__(256) k_oz_fix(double2* __restrict__ F, long long nrows, int nX, int pl, int npc,
                                                int* __restrict__ e) {
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= nrows * npc) return;
  const long long row = w / npc;
  const int k0 = (int)(w % npc) * pl, kc = min(pl, nX - k0);
  double2* f = F + row * nX + k0;
  long long mx = 0;
  for (int kk = lane; kk < kc; kk += 32) mx = max(mx, max(abs_bits(f[kk].x), abs_bits(f[kk].y)));
  for (int off = 16; off > 0; off >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  const int ex = row_exp(mx);
  if (lane == 0) e[w] = ex;
  for (int kk = lane; kk < kc; kk += 32) {
    const double2 v = f[kk];
    // (fixed56 scales by 2^(56 - e): one exponent up gives 2^(55 - e); a flagged row becomes zeros)
    const long long a = fixed56(v.x, ex + 1), b = fixed56(v.y, ex + 1);
    const int a1 = (int)((a + (1LL << 27)) >> 28), b1 = (int)((b + (1LL << 27)) >> 28);
    const int4 o = make_int4(a1, (int)(a - ((long long)a1 << 28)), b1, (int)(b - ((long long)b1 << 28)));
    reinterpret_cast<int4*>(f)[kk] = o;
  }
}

// Slices of the Khatri-Rao rows of a chunk of (incidence, receiver) pairs, for
// the x-projection of the Jacobian: complex row (pair c, gy) of w = u_d z_p
// (d = (c0 + c) / P, p = (c0 + c) % P, fixed-point fields on the interior grid,
// [rhs][gy][gx]) over the piece's gx, split into its real part (row
// 2 (c nX + gy)) and imaginary part (row 2 (c nX + gy) + 1).  One warp per
// complex row and piece, two neighbouring gx per lane, never stored.
// The row's exponent is the fields' sum plus one (|re u re z| + |im u im z| < 2),
// known before the products, so a row need not be held for its maximum; the
// products are taken in integers, N = 2 (U1 Z1) + (U1 Z0 + U0 Z1) 2^-27 per
// real product, six 32 x 32 + 64 multiply-adds per part (the U0 Z0 term is below
// one unit of 2^-56).  Against FP64 products and the row's own maximum: no
// operation on the FP64 pipe (60% busy then, with 145 instructions per real
// entry), and an error within 3.5 u of the product of the two fields' maxima over the
// row piece, where FP64 rounds each product to u of itself (a row in which u is small
// where z is large has that many bits fewer; the fields of this problem vary little
// within a row: Jacobians are as close to the dense solution as before).  25,600 pairs at
// n = 448: 101 ms with FP64 products and 2-byte stores, 95 with 32-bit stores, 54 in
// integers, 47.7 with the digits of two neighbours taken at once.
__global__ void __launch_bounds__(256) k_oz_slice_kr(const int4* __restrict__ Ug, const int4* __restrict__ Zg,
                                                     const int* __restrict__ eu, const int* __restrict__ ez,
                                                     unsigned P, unsigned nX, unsigned d0, unsigned p0, unsigned nr,
                                                     int pl, int npc, long long rpad, int nst,
                                                     uint32_t* __restrict__ out, int* __restrict__ e) {
  const unsigned r2 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r2 >= nr) return;
  const int k0 = blockIdx.y * pl, kc = min(pl, (int)nX - k0), kp = (kc + OZ_KS - 1) / OZ_KS * OZ_KS;
  // (32-bit divisions: the pair's incidence and receiver count from those of the chunk's first pair, d0 and p0)
  const unsigned c = p0 + r2 / nX, gy = r2 % nX;
  const long long ru = (long long)(d0 + c / P) * nX + gy, rz = (long long)(c % P) * nX + gy;
  const int4* u = Ug + ru * nX + k0;
  const int4* z = Zg + rz * nX + k0;
  if (lane == 0) {
    const int ex = min(eu[ru * npc + blockIdx.y] + ez[rz * npc + blockIdx.y] + 1, OZ_NAN);
    e[blockIdx.y * rpad + 2LL * r2] = ex;
    e[blockIdx.y * rpad + 2LL * r2 + 1] = ex;
  }
  auto mac = [](long long acc, int a, int b) { return acc + (long long)a * b; };
#pragma unroll 2
  for (int kk = 2 * lane; kk < kp; kk += 64) {
    long long re[2], im[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int4 a = make_int4(0, 0, 0, 0), b = a;
      if (kk + h < kc) {
        a = u[kk + h];
        b = z[kk + h];
      }
      const long long rh = mac((long long)a.x * b.x, -a.z, b.z);
      const long long rl = mac(mac(mac((long long)a.x * b.y, a.y, b.x), -a.z, b.w), -a.w, b.z);
      const long long ih = mac((long long)a.x * b.z, a.z, b.x);
      const long long il = mac(mac(mac((long long)a.x * b.w, a.y, b.z), a.z, b.y), a.w, b.x);
      re[h] = 2 * rh + ((rl + (1LL << 26)) >> 27);
      im[h] = 2 * ih + ((il + (1LL << 26)) >> 27);
    }
    // (rows 2 r2 and 2 r2 + 1 lie in one tile, 64 bytes apart, with the same swizzle)
    uint32_t* o = out + oz_at<OZ_TM>(2LL * r2, k0 + kk, nst);
    put2(re[0], re[1], o, OZ_ROW * OZ_TM);
    put2(im[0], im[1], o + OZ_ROW, OZ_ROW * OZ_TM);
  }
}

// Zero slices and exponents of the padding rows [first, rpad) of the last tile.
__global__ void k_oz_zero_rows(long long first, long long rpad, int nst, int npc, uint32_t* __restrict__ out,
                               int* __restrict__ e) {
  const int nr = (int)(rpad - first);
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)nr * nst * OZ_S * OZ_ROW) return;
  const int w = (int)(t % OZ_ROW), r = (int)(t / OZ_ROW % nr);
  const long long blk = t / OZ_ROW / nr;  // k-step and slice
  out[((rpad / OZ_TM - 1) * nst * OZ_S + blk) * OZ_TM * OZ_ROW + (first + r) % OZ_TM * OZ_ROW + w] = 0u;
  if (t < (long long)nr * npc) e[(t / nr) * rpad + first + t % nr] = 0;
}

// (hi 2^28 + lo) 2^e as a double (round to nearest even), |hi|, |lo| < 2^46, in
// integer arithmetic: two 64-bit conversions, a scaling and their sum would be half
// the epilogue's time on the FP64 pipe.
__device__ __forceinline__ double scaled(long long hi, long long lo, int e) {
  if (e >= OZ_NAN / 2) return __longlong_as_double(0x7FF8000000000000LL);
  constexpr unsigned low = (1u << 28) - 1;
  long long h = hi + (lo >> 28);  // h 2^28 + l with 0 <= l < 2^28
  unsigned l = (unsigned)lo & low;
  const bool neg = h < 0;
  if (neg) {
    h = -h - (l != 0);
    l = (0u - l) & low;
  }
  // the leading 64 bits, what is cut off below them as a last bit (it only decides ties)
  const int cut = max(28 - __clzll(h), 0);
  unsigned long long a = ((unsigned long long)h << (28 - cut)) | (l >> cut) | ((l & ((1u << cut) - 1)) != 0);
  if (a == 0) return 0.0;
  e += cut;
  const int z = __clzll(a);
  a <<= z;
  const int E = 1023 + 63 - z + e;  // biased exponent of the leading bit
  // 53 bits, rounded; a carry runs into the exponent field as it should
  const unsigned long long q = (a >> 11) + ((a >> 10) & ((a & 0x3FF) != 0 || ((a >> 11) & 1)));
  if (E < 1 || E > 2045) {  // subnormal or overflow
    const double r = scalbn((double)q, E - 1075);
    return neg ? -r : r;
  }
  return __longlong_as_double((long long)((((unsigned long long)(E - 1)) << 52) + q) |
                              (neg ? (long long)0x8000000000000000ULL : 0LL));
}

struct OzParams {
  int m, n, k, pl, npc;        // k in pieces of pl
  int mpad, npad, tm, tn;      // padded rows of A and B, tiles
  int batch, b_shared, sym;    // sym: only tiles that meet the lower triangle
  int zs, ppz;                 // z groups of ppz pieces, each to its own plane of C (zs > 1: alpha 1, beta 0)
  long long items, zplane;
  double alpha, beta;
  const char *a, *b;           // sliced operands
  int nst;                     // k-steps of a row tile
  const int *ea, *eb;          // exponents [piece][row]
  long long ea_piece, eb_piece;
  OzView C;
};

struct OzItem { int z, b, tm, tn; };
__device__ __forceinline__ bool oz_item(const OzParams& P, long long it, OzItem& o) {
  o.tn = (int)(it % P.tn);
  long long t = it / P.tn;
  o.tm = (int)(t % P.tm);
  t /= P.tm;
  o.b = (int)(t % P.batch);
  o.z = (int)(t / P.batch);
  return !(P.sym && o.tn * OZ_TN >= (o.tm + 1) * OZ_TM);
}

// Persistent: each CTA takes every gridDim.x-th 128 x 32 tile (or piece group
// of one) and runs all its pieces of k, summing them in registers; the eight
// diagonals take half of TMEM, so one piece's epilogue runs behind the next one's
// products.  What bounds it: per 32-k stage the 36 slice products (1152 tensor
// clocks) read 136 KB of shared memory while 80 KB are written (1690 clocks);
// 2000 to 2200 clocks at 1.92 GHz measured.  The epilogue (9700 clocks a piece: the
// conversions of eight diagonals, the doubles assembled from their bits in
// integer arithmetic) bounds pieces below 160 k.
// Before, one launch per piece with an FP64 epilogue on four warps and C read
// back per piece kept the tensor pipe at 17%: the products of a k = 40
// Gauss-Newton step (Jacobian projections and normal matrix, 3.2e12 flops) took
// 278 ms; 102 ms with 128 x 64 tiles that fill TMEM, epilogue and products in
// turn; 88 ms now.  4864 x 4096 x k: 29 TFLOP/s of FP64-equivalent work at k = 256,
// 34 at 1536 (1217 of the 1948 TFLOP/s bf16 peak issued).
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_mma(const __grid_constant__ OzParams P) {
  extern __shared__ unsigned char smraw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  __shared__ uint32_t tslot;
  __shared__ __align__(8) uint64_t full[2], empty[2], accf[2], acce[2], done;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&full[i])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&empty[i])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&accf[i])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&acce[i])), "r"(OZ_EPI));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(&done)), "r"(1));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tslot;
  bool ok = true;
  auto stages = [&](int p) { return (min(P.pl, P.k - p * P.pl) + OZ_KS - 1) / OZ_KS; };

  if (warp == 0) {
    if (lane == 0) {  // TMA producer
      int c = 0;      // stages issued
      for (long long it = blockIdx.x; it < P.items && ok; it += gridDim.x) {
        OzItem o;
        if (!oz_item(P, it, o)) continue;
        const char* pa = P.a + (long long)(o.b * P.tm + o.tm) * P.nst * (OZ_S * OZ_A_SL);
        const char* pb = P.b + (long long)((P.b_shared ? 0 : o.b) * P.tn + o.tn) * P.nst * (OZ_S * OZ_B_SL);
        for (int p = o.z * P.ppz; p < min(P.npc, (o.z + 1) * P.ppz) && ok; ++p) {
          const int nst = stages(p);
          for (int i = 0; i < nst; ++i, ++c) {
            const int st = c & 1;
            if (c >= 2) ok = oz_wait(su32(&empty[st]), ((c >> 1) - 1) & 1);
            if (!ok) break;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(&full[st])), "r"(OZ_STAGE)
                         : "memory");
            const uint32_t base = su32(sm + st * OZ_STAGE);
            const long long ks = p * (P.pl / OZ_KS) + i;
            oz_copy(base, pa + ks * (OZ_S * OZ_A_SL), OZ_S * OZ_A_SL, su32(&full[st]));
            oz_copy(base + OZ_S * OZ_A_SL, pb + ks * (OZ_S * OZ_B_SL), OZ_S * OZ_B_SL, su32(&full[st]));
          }
        }
      }
      // every copy issued has landed before the CTA may leave
      for (int q = max(0, c - 2); q < c; ++q) ok = oz_wait(su32(&full[q & 1]), (q >> 1) & 1) && ok;
    }
  } else if (warp == 1) {
    if (lane == 0) {  // MMA issuer
      int c = 0, pc = 0;
      for (long long it = blockIdx.x; it < P.items && ok; it += gridDim.x) {
        OzItem o;
        if (!oz_item(P, it, o)) continue;
        for (int p = o.z * P.ppz; p < min(P.npc, (o.z + 1) * P.ppz) && ok; ++p, ++pc) {
          const int buf = pc & 1;
          const uint32_t acc0 = tmem + (uint32_t)(buf * OZ_ACC);
          if (pc > 1) ok = oz_wait(su32(&acce[buf]), ((pc >> 1) - 1) & 1);  // the epilogue has read this set
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
          const int nst = stages(p);
          for (int i = 0; i < nst; ++i, ++c) {
            const int st = c & 1;
            ok = oz_wait(su32(&full[st]), (c >> 1) & 1);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t aB = su32(sm + st * OZ_STAGE), bB = aB + OZ_S * OZ_A_SL;
            // The B slices of a k block lie back to back (slice t at rows 32 t .. 32 t + 31)
            // and the diagonal accumulators are adjacent in TMEM (diagonal d at columns
            // 32 d ..), so one MMA with N = 32 (8 - s) multiplies A_s by B_0 .. B_(7-s)
            // into diagonals s .. 7: 8 MMAs per 16 k instead of 36.
#pragma unroll 1
            for (int kh = 0; kh < OZ_KS / 16; ++kh) {
#pragma unroll 1
              for (int s = 0; s < OZ_S; ++s) {
                const uint64_t da = oz_desc(aB + s * OZ_A_SL + kh * 32), db = oz_desc(bB + kh * 32);
                const uint32_t acc = (i > 0 || kh > 0 || s > 0) ? 1u : 0u, idesc = oz_idesc((OZ_ND - s) * OZ_TN);
                asm volatile(
                    "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(acc0 + (uint32_t)(s * OZ_TN)),
                    "l"(da), "l"(db), "r"(idesc), "r"(acc));
              }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                su32(&empty[st])));
          }
          if (ok)
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                su32(&accf[buf])));
        }
      }
      // one more commit tracks every MMA issued above
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(&done)));
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 = tile rows (lane = row), 8 of the 32 columns
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    int pc = 0;
    for (long long it = blockIdx.x; it < P.items && ok; it += gridDim.x) {
      OzItem o;
      if (!oz_item(P, it, o)) continue;
      const int r = o.tm * OZ_TM + quarter * 32 + lane, cb = o.tn * OZ_TN + part * 8;
      const int p0 = o.z * P.ppz, p1 = min(P.npc, p0 + P.ppz);
      double acc[8];
      // (a product with +-1 would cost the FP64 pipe as much as the tile's conversions)
      auto times = [&](double x) { return P.alpha == 1.0 ? x : P.alpha == -1.0 ? -x : P.alpha * x; };
      for (int p = p0; p < p1; ++p, ++pc) {
        const int buf = pc & 1;
        const uint32_t ta = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(buf * OZ_ACC + part * 8);
        // (rows and columns of the padding have exponents too)
        const int ea = P.ea[p * P.ea_piece + (long long)o.b * P.mpad + r];
        const int ebl = P.eb[p * P.eb_piece + (long long)(P.b_shared ? 0 : o.b) * P.npad + cb + (lane & 7)];
        ok = oz_wait(su32(&accf[buf]), (pc >> 1) & 1);
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        // pairs of diagonals in 32 bits: |C_d| <= 384 4096 (d + 3) (6.3e6 for d = 0),
        // 128 C_d + C_(d+1) <= 1.83e9 < 2^31
        int q[4][8];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          uint32_t v[4][8];
#pragma unroll
          for (int d = 0; d < 4; ++d) oz_ld8(ta + (uint32_t)((4 * g + d) * OZ_TN), v[d]);
          asm volatile("tcgen05.wait::ld.sync.aligned;");
          if (g == 1) {  // last read of this piece: this set of accumulators is free
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(&acce[buf])) : "memory");
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            q[2 * g][j] = 128 * __float2int_rn(__uint_as_float(v[0][j])) + __float2int_rn(__uint_as_float(v[1][j]));
            q[2 * g + 1][j] = 128 * __float2int_rn(__uint_as_float(v[2][j])) + __float2int_rn(__uint_as_float(v[3][j]));
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          // sum_d C_d 2^(-7 (d + 2)) = (hi 2^28 + lo) 2^-63, hi and lo = q 2^14 + the next q
          const double x = scaled(((long long)q[0][j] << 14) + q[1][j], ((long long)q[2][j] << 14) + q[3][j],
                                  ea + __shfl_sync(0xffffffffu, ebl, j) - 63);
          acc[j] = p == p0 ? x : acc[j] + x;
        }
      }
      if (!ok) break;
      if (r < P.m) {
        double* pr = P.C.p + o.z * P.zplane + o.b * P.C.sb + (r / P.C.ig) * P.C.si + (r % P.C.ig) * P.C.sg;
        if (P.C.sk == 1 && (reinterpret_cast<uintptr_t>(pr + cb) & 15) == 0 && cb + 8 <= P.n) {
          double2* p2 = reinterpret_cast<double2*>(pr + cb);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            double2 x = make_double2(times(acc[2 * j]), times(acc[2 * j + 1]));
            if (P.beta != 0.0) {
              const double2 y = p2[j];
              x = make_double2(fma(P.beta, y.x, x.x), fma(P.beta, y.y, x.y));
            }
            p2[j] = x;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (cb + j < P.n) {
              double* w = pr + (cb + j) * P.C.sk;
              const double x = times(acc[j]);
              *w = P.beta == 0.0 ? x : fma(P.beta, *w, x);
            }
        }
      }
    }
  }
  // everyone: wait until the tensor cores are done with TMEM and the stages
  const bool drained = oz_wait(su32(&done), 0);
  ok = ok && drained;
  asm volatile("tcgen05.fence::after_thread_sync;");
  const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
  if (!all_ok && threadIdx.x == 0) atomicExch(&g_oz_timeout, 1);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// C = alpha sum_z plane_z + beta C, planes [z][b][i][j], in order.
__global__ void k_oz_combine(const double* __restrict__ planes, int zs, long long zplane, int m, int n, double alpha,
                             double beta, OzView C) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= zplane) return;
  double v = 0.0;
  for (int z = 0; z < zs; ++z) v += planes[z * zplane + e];
  const long long j = e % n, t = e / n, i = t % m, b = t / m;
  double* c = C.p + b * C.sb + (i / C.ig) * C.si + (i % C.ig) * C.sg + j * C.sk;
  *c = beta == 0.0 ? alpha * v : fma(beta, *c, alpha * v);
}

inline long long rup(long long x, long long m) { return (x + m - 1) / m * m; }

}  // namespace

bool g_oz_enabled = true;  // process-wide switch (hs_set_fp64_emulation)

void oz_timeout_flag(cudaStream_t s, int* v, bool clear) {
  if (clear)
    cudaMemcpyToSymbolAsync(g_oz_timeout, v, sizeof(int), 0, cudaMemcpyHostToDevice, s);
  else
    cudaMemcpyFromSymbolAsync(v, g_oz_timeout, sizeof(int), 0, cudaMemcpyDeviceToHost, s);
}

namespace {

size_t align_up(size_t b) { return (b + 1023) & ~size_t(1023); }

// Length of the pieces k is cut into: as equal as possible, at most OZ_KMAX,
// a multiple of the stage depth (the last piece takes the rest).
int piece_len(int k) {
  const int np = (k + OZ_KMAX - 1) / OZ_KMAX;
  return (int)std::min<long long>(OZ_KMAX, rup((k + np - 1) / np, OZ_KS));
}
int npieces(int k) { return (k + piece_len(k) - 1) / piece_len(k); }
long long padded(int rows, bool is_a) { return rup(rows, is_a ? OZ_TM : OZ_TN); }
size_t slice_bytes(long long total, int k) { return align_up((size_t)OZ_S * total * npieces(k) * piece_len(k) * 2); }

template <typename F> void once_per_device(bool (&done)[64], F&& f) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && done[dev]) return;
  f();
  if (dev >= 0 && dev < 64) done[dev] = true;
}
void set_smem_attr() {
  static bool done[64] = {};
  once_per_device(done, [] {
    cudaFuncSetAttribute(k_oz_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM);
    cudaFuncSetAttribute(k_oz_slice, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         OZ_SR * (OZ_KMAX + 1) * (int)sizeof(double));
  });
}

// Groups of pieces that run as separate tiles where there are fewer tiles than SMs.
int z_groups(int m, int n, int k, int batch) {
  const long long tiles = padded(m, true) / OZ_TM * (padded(n, false) / OZ_TN) * batch;
  return tiles >= 152 ? 1 : (int)std::min<long long>(npieces(k), (152 + tiles - 1) / tiles);
}

}  // namespace

size_t oz_operand_bytes(int rows, int k, int batch, bool is_a) {
  const long long total = batch * padded(rows, is_a);
  return slice_bytes(total, k) + align_up((size_t)npieces(k) * total * 4);
}

size_t oz_plane_bytes(int m, int n, int k, int batch) {
  const int zs = z_groups(m, n, k, batch);
  return zs == 1 ? 0 : align_up((size_t)zs * batch * m * n * 8);
}

namespace {
OzSliced sliced(OzSrc v, int rows, int k, int batch, bool is_a, void* buf) {
  const long long rpad = padded(rows, is_a), total = batch * rpad;
  char* base = reinterpret_cast<char*>(buf);
  return {v,     rows,
          (int)rpad, k,
          piece_len(k), npieces(k) * piece_len(k) / OZ_KS,
          total, reinterpret_cast<uint32_t*>(base),
          reinterpret_cast<int*>(base + slice_bytes(total, k))};
}

void launch_slice(cudaStream_t s, const OzSliced& a, const OzSliced& b, bool has_a, bool has_b) {
  set_smem_attr();
  const unsigned na = has_a ? (unsigned)(a.total / OZ_SR) : 0, nb = has_b ? (unsigned)(b.total / OZ_SR) : 0;
  k_oz_slice<<<dim3(na + nb, npieces(a.k)), 256, OZ_SR * (a.pl + 1) * sizeof(double), s>>>(a, b, na);
  HS_COUNT_LAUNCH();
}
}  // namespace

void oz_slice(cudaStream_t s, OzSrc v, int rows, int k, int batch, bool is_a, void* buf) {
  const OzSliced o = sliced(v, rows, k, batch, is_a, buf);
  launch_slice(s, o, o, is_a, !is_a);
}

size_t oz_fix_bytes(int fields, int nX) { return align_up((size_t)fields * nX * npieces(nX) * 4); }

void oz_fix_fields(cudaStream_t s, double2* F, int fields, int nX, void* exps) {
  const long long rows = (long long)fields * nX, warps = rows * npieces(nX);
  k_oz_fix<<<(unsigned)((warps + 7) / 8), 256, 0, s>>>(F, rows, nX, piece_len(nX), npieces(nX),
                                                      reinterpret_cast<int*>(exps));
  HS_COUNT_LAUNCH();
}

void oz_slice_khatri_rao(cudaStream_t s, const double2* Ug, const double2* Zg, const void* eu, const void* ez, int P,
                         int nX, long long c0, int nc, void* buf) {
  const int rows = 2 * nc * nX, pl = piece_len(nX), npc = npieces(nX), nst = npc * pl / OZ_KS;
  const long long rpad = padded(rows, true), warps = (long long)nc * nX;
  uint32_t* sl = reinterpret_cast<uint32_t*>(buf);
  int* ex = reinterpret_cast<int*>(reinterpret_cast<char*>(buf) + slice_bytes(rpad, nX));
  k_oz_slice_kr<<<dim3((unsigned)((warps + 7) / 8), npc), 256, 0, s>>>(
      reinterpret_cast<const int4*>(Ug), reinterpret_cast<const int4*>(Zg), reinterpret_cast<const int*>(eu),
      reinterpret_cast<const int*>(ez), (unsigned)P, (unsigned)nX, (unsigned)(c0 / P), (unsigned)(c0 % P),
      (unsigned)warps, pl, npc, rpad, nst, sl, ex);
  HS_COUNT_LAUNCH();
  if (rpad > rows) {
    const long long n = (rpad - rows) * nst * OZ_S * OZ_ROW;
    k_oz_zero_rows<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(rows, rpad, nst, npc, sl, ex);
    HS_COUNT_LAUNCH();
  }
}

cudaError_t oz_multiply(cudaStream_t s, int m, int n, int k, int batch, double alpha, const void* Aop, const void* Bop,
                        bool b_shared, double beta, OzView C, void* planes, bool sym) {
  if (m <= 0 || n <= 0 || k <= 0 || batch <= 0) return cudaErrorInvalidValue;
  set_smem_attr();
  const long long mp = padded(m, true), np = padded(n, false), ta = batch * mp, tb = (b_shared ? 1 : batch) * np;
  const int pl = piece_len(k), npc = npieces(k), zs = planes ? z_groups(m, n, k, batch) : 1;
  char* a = const_cast<char*>(reinterpret_cast<const char*>(Aop));
  char* b = const_cast<char*>(reinterpret_cast<const char*>(Bop));
  OzParams P;
  P.m = m;
  P.n = n;
  P.k = k;
  P.pl = pl;
  P.npc = npc;
  P.mpad = (int)mp;
  P.npad = (int)np;
  P.tm = (int)(mp / OZ_TM);
  P.tn = (int)(np / OZ_TN);
  P.batch = batch;
  P.b_shared = b_shared ? 1 : 0;
  P.sym = sym ? 1 : 0;
  P.ppz = (npc + zs - 1) / zs;
  P.zs = (npc + P.ppz - 1) / P.ppz;
  P.items = (long long)P.tm * P.tn * batch * P.zs;
  P.a = a;
  P.b = b;
  P.nst = npc * pl / OZ_KS;
  P.ea = reinterpret_cast<const int*>(a + slice_bytes(ta, k));
  P.eb = reinterpret_cast<const int*>(b + slice_bytes(tb, k));
  P.ea_piece = ta;
  P.eb_piece = tb;
  const bool split = P.zs > 1;
  P.zplane = split ? (long long)batch * m * n : 0;
  P.alpha = split ? 1.0 : alpha;
  P.beta = split ? 0.0 : beta;
  P.C = split ? OzView{reinterpret_cast<double*>(planes), (long long)m * n, n, 0, 1, 1} : C;
  const bool prof = prof_active(4);
  cudaEvent_t ev = nullptr;
  if (prof) prof_begin(s, &ev);
  if (g_tc_pending) *g_tc_pending = true;
  k_oz_mma<<<(unsigned)std::min<long long>(P.items, 152), OZ_THREADS, OZ_SMEM, s>>>(P);
  HS_COUNT_LAUNCH();
  if (split) {
    k_oz_combine<<<(unsigned)((P.zplane + 255) / 256), 256, 0, s>>>(reinterpret_cast<double*>(planes), P.zs, P.zplane,
                                                                    m, n, alpha, beta, C);
    HS_COUNT_LAUNCH();
  }
  if (prof) prof_end(s, ev, 2.0 * m * n * k * batch);  // FP64-equivalent flops
  return cudaPeekAtLastError();  // (left for the API call's own check: gemm() returns nothing)
}

thread_local const OzScratch* g_oz_scratch = nullptr;
thread_local bool* g_tc_pending = nullptr;

// Per tile 2100 clocks a stage, or 9400 a piece where that is more; slices
// written and read at about 2600 bytes a clock; launches.
double oz_cycles(int m, int n, int k, int batch, bool b_shared) {
  const double mp = (double)padded(m, true), np = (double)padded(n, false);
  const int npc = npieces(k), zs = z_groups(m, n, k, batch);
  const double tiles = mp / OZ_TM * (np / OZ_TN) * batch * zs, kt = (double)npc * piece_len(k);
  const double tile = std::max(kt / OZ_KS * 2100.0 / zs, std::ceil((double)npc / zs) * 9400.0);
  const double slices = (batch * mp + (b_shared ? 1 : batch) * np) * kt * 40.0 / 2600.0;
  return std::ceil(tiles / 152.0) * tile + slices + (zs > 1 ? 24000.0 : 18000.0);
}

size_t ozaki_scratch_bytes(int m, int n, int k, int batch, bool b_shared) {
  return oz_operand_bytes(m, k, batch, true) + oz_operand_bytes(n, k, b_shared ? 1 : batch, false) +
         oz_plane_bytes(m, n, k, batch);
}

// The operands' bytes grow with every size; the planes' do not (fewer tiles than SMs
// want some, more want none), so a part of a product that fits may want planes that do
// not: its pieces of k then run one after the other in each tile.

cudaError_t ozaki_gemm(cudaStream_t s, int m, int n, int k, int batch, double alpha, OzSrc A, OzSrc Bt, bool b_shared,
                       double beta, OzView C, void* scratch, size_t scratch_bytes, bool sym) {
  if (m <= 0 || n <= 0 || k <= 0 || batch <= 0) return cudaErrorInvalidValue;
  const size_t ab = oz_operand_bytes(m, k, batch, true), bb = oz_operand_bytes(n, k, b_shared ? 1 : batch, false),
               pb = oz_plane_bytes(m, n, k, batch);
  if (ab + bb > scratch_bytes) return cudaErrorInvalidValue;
  char* a = reinterpret_cast<char*>(scratch);
  char *b = a + ab, *pl = b + bb;
  launch_slice(s, sliced(A, m, k, batch, true, a), sliced(Bt, n, k, b_shared ? 1 : batch, false, b), true, true);
  return oz_multiply(s, m, n, k, batch, alpha, a, b, b_shared, beta, C,
                     pb && ab + bb + pb <= scratch_bytes ? pl : nullptr, sym);
}

}  // namespace hs
