// Mixed-precision pieces: FP64 residuals of the discrete system and the FP32
// particular (body-load) solve at the leaves.
//
// The discrete system solved by the direct solver (Sec. 2) has three kinds of
// rows: the collocated PDE at interior leaf nodes, continuity of u and of the
// normal derivative at shared leaf edge nodes, and the exterior identity
// (D - I/2)(u - u_inc) = S (d_n u - d_n u_inc) at boundary nodes (Sec. 2,
// Remark).  With FP32 factors, the solution is refined in FP64: the residual
// of every row is computed here in FP64 from the current FP64 iterate (leaf
// layout [leaf][252][nrhs]) and fed to an FP32 solve for the correction.
#include "tree.cuh"

namespace hs {

namespace {

// Leaf-local unknown index of node (a, b) (never a corner).
__device__ __forceinline__ int lidx(int a, int b) {
  if (a >= 1 && a <= 14 && b >= 1 && b <= 14) return (a - 1) * 14 + (b - 1);
  if (b == 0) return NI + a - 1;
  if (a == 15) return NI + 14 + b - 1;
  if (b == 15) return NI + 28 + a - 1;
  return NI + 42 + b - 1;
}

__global__ void k_d2f(const double2* __restrict__ a, float2* __restrict__ b, long long n) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = make_float2((float)a[i].x, (float)a[i].y);
}

__global__ void k_f2d_add(const float2* __restrict__ a, double2* __restrict__ b, long long n) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = make_double2(b[i].x + (double)a[i].x, b[i].y + (double)a[i].y);
}

constexpr int RCH = 8;              // right-hand sides per block in the PDE residual
constexpr int RP_THREADS = 49 * RCH;  // one thread per (a, b) in 1..7 x 1..7 and right-hand side

// A 56-bit fixed-point number as two signed limbs, v = v1 2^28 + v0.
__device__ __forceinline__ int2 limbs(long long v) {
  const int hi = (int)((v + (1LL << 27)) >> 28);
  return make_int2(hi, (int)(v - ((long long)hi << 28)));
}
// Sum of products of limb pairs: h of the high products (unit 2^56), m of the
// mixed ones (unit 2^28); the low products are below h's unit.
struct FixSum {
  long long h = 0, m = 0;
  __device__ __forceinline__ void mac(int2 a, int x1, int x0) {
    h += (long long)a.x * x1;
    m += (long long)a.x * x0;
    m += (long long)a.y * x1;
  }
  // 2^-n of the value, rounded
  __device__ __forceinline__ long long down(int n) const {
    const long long v = h + ((m + (1LL << 27)) >> 28);
    return (v + (long long)((1ULL << n) >> 1)) >> n;
  }
  __device__ friend FixSum operator+(FixSum a, FixSum b) { return FixSum{a.h + b.h, a.m + b.m}; }
  __device__ friend FixSum operator-(FixSum a, FixSum b) { return FixSum{a.h - b.h, a.m - b.m}; }
};
__device__ __forceinline__ float fix_float(long long v, int e) {
  const float f = (float)v;
  return e >= -126 && e <= 127 ? f * __int_as_float((e + 127) << 23) : scalbnf(f, e);
}
__device__ __forceinline__ double fix_double(long long v, int e) {
  const double f = (double)v;
  return e >= -1022 && e <= 1023 ? f * __longlong_as_double((long long)(e + 1023) << 52) : scalbn(f, e);
}

// RP[leaf][r][j] = -(Lap_h u + k^2 (1 - q) u) at interior node r, for the FP64
// iterate X, and DN[leaf][e][j], the outward normal derivative of u at edge node e.
// The second-derivative matrix D2 = (2/h)^2 D1 D1 of the Chebyshev points is
// centro-symmetric (D2[15-a][15-c] = D2[a][c]), so along a grid line with
// s_c = u_c + u_(15-c), d_c = u_c - u_(15-c) (c < 8) and E[a][c], O[a][c] the
// half sums and differences of D2[a][c] and D2[a][15-c]:
//   (D2 u)_a = sum_c E[a][c] s_c + O[a][c] d_c,  (D2 u)_(15-a) = the same with -O,
// half the multiply-adds of the plain row products.  Each thread forms the four
// mirror nodes (a, b), (15-a, b), (a, 15-b), (15-a, 15-b) of one right-hand side
// from the s, d of the two columns and two rows through them.
// The sums are taken in fixed point: a leaf's u of one right-hand side scaled by
// its largest part, each matrix row by its own, both to 56 bits in two limbs,
// three 32 x 32 + 64 bit multiply-adds per product (a line's 16 stay below 2^61).
// FP64 multiply-adds (two thread-operations per SM and clock) bounded this
// kernel; the integer ones run seven times as fast: 2.49 -> 1.2 ms for 1024 leaves
// and 128 right-hand sides, the normal derivatives included that the interface
// residuals formed by FP64 sums of their own before (0.8 ms a pass).  Rounding of Lap_h u +
// k^2 (1 - q) u for plane waves (k = 17, 25, 40, h = 1/16; root mean square over the nodes,
// from the exact sums with the same coefficients): 3.0e-11, 2.9e-11 and 2.7e-11, of the FP64
// sums 7.1e-11, 8.1e-11 and 7.6e-11 (truncated shifts gave 3.8e-11, 4.0e-11 and 3.0e-11, half
// of it a bias).
__global__ void __launch_bounds__(RP_THREADS, 2) k_res_pde(const double2* __restrict__ X, const double* __restrict__ q,
                                                        const double* __restrict__ D1, double k, double h, int nrhs,
                                                        float2* __restrict__ RP, double2* __restrict__ DN) {
  __shared__ double Dx[16][16], D2r[8][16], Ed[8][8], Od[8][8];
  __shared__ int2 E[8][8], O[8][8], N0[16], N15[16], cq[NI];
  __shared__ unsigned mu[RCH], mrow[8], mq, mn;  // largest magnitudes (leading words)
  extern __shared__ double2 rp_dyn[];  // u[NL][RCH], then sx, dx, sy, dy [14][8][RCH]; as limbs (re1, re0, im1, im0)
  auto ud = reinterpret_cast<double2(*)[RCH]>(rp_dyn);
  auto u = reinterpret_cast<int4(*)[RCH]>(rp_dyn);
  auto sx = reinterpret_cast<int4(*)[8][RCH]>(rp_dyn + NL * RCH);
  auto dx = sx + 14, sy = sx + 28, dy = sx + 42;
  const int leaf = blockIdx.x, j0 = blockIdx.y * RCH, t = threadIdx.x, lane = t & 31;
  const int nj = min(RCH, nrhs - j0), j = t % RCH;
  const double sc = 2.0 / h, kk = k * k;
  const double* ql = q + (long long)leaf * 256;
  if (t < RCH) mu[t] = mrow[t] = 0;
  if (t == RCH) mq = 0;
  for (int e = t; e < 256; e += RP_THREADS) Dx[e / 16][e % 16] = D1[e] * sc;
  __syncthreads();
  auto mag = [](double x) { return (unsigned)__double2hiint(x) & 0x7FFFFFFFu; };
  const bool whole = t < RP_THREADS / 32 * 32;  // (the last warp is a partial one)
  unsigned mx = 0;  // (the thread's elements are all of right-hand side j)
  for (int e = t; e < NL * RCH; e += RP_THREADS) {
    const int r = e / RCH;
    const double2 v = j < nj ? X[((long long)leaf * NL + r) * nrhs + j0 + j] : make_double2(0.0, 0.0);
    ud[r][j] = v;
    mx = max(mx, max(mag(v.x), mag(v.y)));
  }
  if (whole)
    for (int off = RCH; off < 32; off <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  if (lane < RCH) atomicMax(&mu[j], mx);
  // rows 1..7 of D2, and the largest coefficients
  for (int e = t; e < 7 * 16; e += RP_THREADS) {
    const int a = e / 16 + 1, c = e % 16;
    double acc = 0.0;
    for (int m = 0; m < 16; ++m) acc = fma(Dx[a][m], Dx[m][c], acc);
    D2r[a][c] = acc;
  }
  if (whole) {
    const unsigned vq = __reduce_max_sync(
        0xffffffffu, t < NI ? mag(kk * (1.0 - ql[(t / 14 + 1) * 16 + t % 14 + 1])) : 0u);
    if (lane == 0) atomicMax(&mq, vq);
    if (t < 32) {
      const unsigned vn = __reduce_max_sync(0xffffffffu, mag(t < 16 ? Dx[0][t] : Dx[15][t - 16]));
      if (lane == 0) mn = vn;
    }
  }
  __syncthreads();
  if (t < 7 * 8) {
    const int a = t / 8 + 1, c = t % 8;
    Ed[a][c] = 0.5 * (D2r[a][c] + D2r[a][15 - c]);
    Od[a][c] = 0.5 * (D2r[a][c] - D2r[a][15 - c]);
    atomicMax(&mrow[a], max(mag(Ed[a][c]), mag(Od[a][c])));
  }
  const int ex = row_exp((long long)mu[j] << 32);
  for (int e = t; e < NL * RCH; e += RP_THREADS) {  // (each thread its own elements, in place)
    const int r = e / RCH;
    const double2 v = ud[r][j];
    const int2 re = limbs(fixed56(v.x, ex)), im = limbs(fixed56(v.y, ex));
    u[r][j] = make_int4(re.x, re.y, im.x, im.y);
  }
  __syncthreads();
  const int en = row_exp((long long)mn << 32), eq = row_exp((long long)mq << 32);
  for (int e = t; e < 7 * 8; e += RP_THREADS) {
    const int a = e / 8 + 1, c = e % 8;
    const int er = row_exp((long long)mrow[a] << 32);
    E[a][c] = limbs(fixed56(Ed[a][c], er));
    O[a][c] = limbs(fixed56(Od[a][c], er));
  }
  if (t < 16) N0[t] = limbs(fixed56(Dx[0][t], en));
  else if (t < 32) N15[t - 16] = limbs(fixed56(Dx[15][t - 16], en));
  if (t < NI) cq[t] = limbs(fixed56(kk * (1.0 - ql[(t / 14 + 1) * 16 + t % 14 + 1]), eq));
  // the line sums and differences (x lines: column b = l + 1; y lines: row a = l + 1)
  for (int e = t; e < 2 * 14 * 8 * RCH; e += RP_THREADS) {
    const int c = (e / RCH) % 8, l = (e / (8 * RCH)) % 14, dir = e / (14 * 8 * RCH);
    const int4 p = dir == 0 ? u[lidx(c, l + 1)][j] : u[lidx(l + 1, c)][j];
    const int4 m = dir == 0 ? u[lidx(15 - c, l + 1)][j] : u[lidx(l + 1, 15 - c)][j];
    // limbs add limb by limb: below 2^29 and 2^28
    (dir == 0 ? sx : sy)[l][c][j] = make_int4(p.x + m.x, p.y + m.y, p.z + m.z, p.w + m.w);
    (dir == 0 ? dx : dy)[l][c][j] = make_int4(p.x - m.x, p.y - m.y, p.z - m.z, p.w - m.w);
  }
  __syncthreads();
  if (j >= nj) return;
  const bool bad = ex >= OZ_NAN / 2 || eq >= OZ_NAN / 2;  // an infinity or a NaN in the field (or the contrast)
  const float nanf_ = __int_as_float(0x7FC00000);
  {
    const int pr = t / RCH, a = pr / 7 + 1, b = pr % 7 + 1;  // a, b in 1..7; mirrors 15 - a, 15 - b
    const int ea = row_exp((long long)mrow[a] << 32), eb = row_exp((long long)mrow[b] << 32);
    const int em = max(max(ea, eb), eq), sa = min(em - ea, 63), sb = min(em - eb, 63), sq = min(em - eq, 63);
    // one part at a time: half the sums alive, two CTAs per SM
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
      auto part = [&](const int4& v) { return reinterpret_cast<const int2*>(&v)[p]; };
      FixSum xe[2], xo[2], ye[2], yo[2];  // columns b, 15 - b (rows a, 15 - a)
#pragma unroll 2
      for (int c = 0; c < 8; ++c) {
        const int2 ca = E[a][c], oa = O[a][c], cb = E[b][c], ob = O[b][c];
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          const int2 s1 = part(sx[w ? 14 - b : b - 1][c][j]), d1 = part(dx[w ? 14 - b : b - 1][c][j]);
          const int2 s2 = part(sy[w ? 14 - a : a - 1][c][j]), d2 = part(dy[w ? 14 - a : a - 1][c][j]);
          xe[w].mac(ca, s1.x, s1.y);
          xo[w].mac(oa, d1.x, d1.y);
          ye[w].mac(cb, s2.x, s2.y);
          yo[w].mac(ob, d2.x, d2.y);
        }
      }
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const int ma = n & 1, mb = n >> 1;  // mirrored in a, in b
        const int A = ma ? 15 - a : a, B = mb ? 15 - b : b, r = (A - 1) * 14 + (B - 1);
        const int2 uv = part(u[r][j]);
        const FixSum fx = ma ? xe[mb] - xo[mb] : xe[mb] + xo[mb];
        const FixSum fy = mb ? ye[ma] - yo[ma] : ye[ma] + yo[ma];
        FixSum fq;
        fq.mac(cq[r], uv.x, uv.y);
        const float o = -fix_float(fx.down(sa) + fy.down(sb) + fq.down(sq), ex + em - 56);
        reinterpret_cast<float*>(RP + ((long long)leaf * NL + r) * nrhs + j0 + j)[p] = bad ? nanf_ : o;
      }
    }
  }
  for (int e = t; e < NE * RCH; e += RP_THREADS) {
    const int r = e / RCH, side = r / 14, i = r % 14 + 1;
    FixSum f[2];
#pragma unroll 4
    for (int c = 0; c < 16; ++c) {
      const int4 v = side == 0 || side == 2 ? u[lidx(i, c)][j] : u[lidx(c, i)][j];
      const int2 d = side == 1 || side == 2 ? N15[c] : N0[c];
      f[0].mac(d, v.x, v.y);
      f[1].mac(d, v.z, v.w);
    }
    const double sg = side == 1 || side == 2 ? 1.0 : -1.0;
    const double2 dn = make_double2(sg * fix_double(f[0].down(0), ex + en - 56), sg * fix_double(f[1].down(0), ex + en - 56));
    DN[((long long)leaf * NE + r) * nrhs + j0 + j] =
        bad ? make_double2((double)nanf_, (double)nanf_) : dn;
  }
}

// Outward normal derivative of leaf field U (leaf layout, FP64) at its edge
// node (a, b), right-hand side j.
__device__ double2 normal_deriv(const double2* __restrict__ U, int nrhs, int j, const double* __restrict__ D1,
                                double sc, int a, int b) {
  double2 acc = make_double2(0.0, 0.0);
  if (b == 0) {
    for (int c = 0; c < 16; ++c) acc = acc - (D1[c] * sc) * U[(long long)lidx(a, c) * nrhs + j];
  } else if (a == 15) {
    for (int c = 0; c < 16; ++c) acc = acc + (D1[15 * 16 + c] * sc) * U[(long long)lidx(c, b) * nrhs + j];
  } else if (b == 15) {
    for (int c = 0; c < 16; ++c) acc = acc + (D1[15 * 16 + c] * sc) * U[(long long)lidx(a, c) * nrhs + j];
  } else {
    for (int c = 0; c < 16; ++c) acc = acc - (D1[c] * sc) * U[(long long)lidx(c, b) * nrhs + j];
  }
  return acc;
}

// Interface residual terms of one merge level: for interface node t of parent
// b, with r_C = -(u_a - u_b) and r_F = -(d_n u_a + d_n u_b) (the normal derivatives
// from k_res_pde), S3[b][t] = r_F + i eta r_C (s_a) and S3[b][ni + t] = r_F - i eta r_C (s_b).
__global__ void k_res_iface(const double2* __restrict__ X, const double2* __restrict__ DN, int nL,
                            const double* __restrict__ kp, int horiz, int sx, int sy, int ni, int nbx_p, int nrhs,
                            float2* __restrict__ S3) {
  const int b = blockIdx.y;
  const double eta = *kp;
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)ni * nrhs) return;
  const int t = (int)(e / nrhs), j = (int)(e % nrhs);
  const int px = b % nbx_p, py = b / nbx_p, node = t % 14;
  int la, lb, ea, eb;  // leaves and edge nodes on the alpha / beta side
  if (horiz) {
    const int x0 = px * 2 * sx, ly = py * sy + t / 14;
    la = ly * nL + (x0 + sx - 1);
    lb = ly * nL + (x0 + sx);
    ea = 14 + node;  // alpha: east edge
    eb = 42 + node;  // beta: west edge
  } else {
    const int lx = px * sx + t / 14, y0 = py * 2 * sy;
    la = (y0 + sy - 1) * nL + lx;
    lb = (y0 + sy) * nL + lx;
    ea = 28 + node;  // alpha: north edge
    eb = node;       // beta: south edge
  }
  const double2 ua = X[((long long)la * NL + NI + ea) * nrhs + j], ub = X[((long long)lb * NL + NI + eb) * nrhs + j];
  const double2 na = DN[((long long)la * NE + ea) * nrhs + j], nb2 = DN[((long long)lb * NE + eb) * nrhs + j];
  const double2 rc = ub - ua;                 // -(u_a - u_b)
  const double2 rf = -(na + nb2);
  // i eta rc = (-eta rc.y, eta rc.x)
  const double2 sa = make_double2(rf.x - eta * rc.y, rf.y + eta * rc.x);
  const double2 sbv = make_double2(rf.x + eta * rc.y, rf.y - eta * rc.x);
  S3[((long long)b * 2 * ni + t) * nrhs + j] = make_float2((float)sa.x, (float)sa.y);
  S3[((long long)b * 2 * ni + ni + t) * nrhs + j] = make_float2((float)sbv.x, (float)sbv.y);
}

// u and d_n u at the boundary nodes (root order: S, E, N, W, each by
// increasing coordinate) from the leaf fields.
__global__ void k_boundary_gather(const double2* __restrict__ X, const double* __restrict__ D1, int nL, double h,
                                  int nrhs, double2* __restrict__ ub, double2* __restrict__ psib) {
  const int nb = 56 * nL;
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)nb * nrhs) return;
  const int jn = (int)(e / nrhs), j = (int)(e % nrhs);
  const int side = jn / (14 * nL), i = (jn % (14 * nL)) / 14, t = jn % 14 + 1;
  int leaf, a, b;
  switch (side) {
    case 0: leaf = i; a = t; b = 0; break;                       // S: leaf (i, 0)
    case 1: leaf = i * nL + (nL - 1); a = 15; b = t; break;      // E: leaf (nL-1, i)
    case 2: leaf = (nL - 1) * nL + i; a = t; b = 15; break;      // N: leaf (i, nL-1)
    default: leaf = i * nL; a = 0; b = t; break;                 // W: leaf (0, i)
  }
  const double2* U = X + (long long)leaf * NL * nrhs;
  ub[e] = U[(long long)lidx(a, b) * nrhs + j];
  psib[e] = normal_deriv(U, nrhs, j, D1, 2.0 / h, a, b);
}

// H = -2 i eta u_e^p (particular outgoing impedance) from the edge rows of Upart.
__global__ void k_leaf_h(const float2* __restrict__ Upart, int nleaf, const double* __restrict__ kp, int nrhs,
                         float2* __restrict__ H) {
  const double eta = *kp;
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)nleaf * NE * nrhs) return;
  const int j = (int)(e % nrhs);
  const long long t = e / nrhs;
  const int r = (int)(t % NE), leaf = (int)(t / NE);
  float2 v = Upart[((long long)leaf * NL + NI + r) * nrhs + j];
  const float te = (float)(2.0 * eta);
  H[e] = make_float2(te * v.y, -te * v.x);  // -2 i eta (x + i y)
}

__global__ void k_scattered(const double2* __restrict__ ub, const double2* __restrict__ psib,
                            const double2* __restrict__ ui, const double2* __restrict__ dni, long long n,
                            double2* __restrict__ PS) {
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  PS[e] = ub[e] - ui[e];
  PS[n + e] = psib[e] - dni[e];
}

// Scattered boundary data [u - u_inc; d_n u - d_n u_inc] (root order) of an
// FP32 leaf field, in FP32; without the incident terms when sub_inc == 0 (a
// correction field).  Feeds the FP32 far field of one refinement pass.
__global__ void k_scattered32(const float2* __restrict__ U32, const double* __restrict__ D1, int nL, double h,
                              int nrhs, const double2* __restrict__ ui, const double2* __restrict__ dni, int sub_inc,
                              float2* __restrict__ PS) {
  const int nb = 56 * nL;
  const long long n = (long long)nb * nrhs;
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int jn = (int)(e / nrhs), j = (int)(e % nrhs);
  const int side = jn / (14 * nL), i = (jn % (14 * nL)) / 14, t = jn % 14 + 1;
  int leaf, a, b;
  switch (side) {
    case 0: leaf = i; a = t; b = 0; break;
    case 1: leaf = i * nL + (nL - 1); a = 15; b = t; break;
    case 2: leaf = (nL - 1) * nL + i; a = t; b = 15; break;
    default: leaf = i * nL; a = 0; b = t; break;
  }
  const float2* U = U32 + (long long)leaf * NL * nrhs;
  const float sc = (float)(2.0 / h);
  const int cpos = (a == 15 || b == 15) ? 15 : 0;
  const float sg = cpos == 15 ? 1.f : -1.f;
  float2 d = make_float2(0.f, 0.f);
  for (int c = 0; c < 16; ++c) {
    const float w = sg * (float)D1[cpos * 16 + c] * sc;
    const float2 v = (b == 0 || b == 15) ? U[(long long)lidx(a, c) * nrhs + j] : U[(long long)lidx(c, b) * nrhs + j];
    d = make_float2(d.x + w * v.x, d.y + w * v.y);
  }
  float2 u = U[(long long)lidx(a, b) * nrhs + j];
  if (sub_inc) {
    u = make_float2(u.x - (float)ui[e].x, u.y - (float)ui[e].y);
    d = make_float2(d.x - (float)dni[e].x, d.y - (float)dni[e].y);
  }
  PS[e] = u;
  PS[n + e] = d;
}

// DS = [D - I/2, -S] (nb x 2 nb): the exterior rows act on [u; d_n u] with one
// product; FP64 and FP32 copies.
__global__ void k_stack_ext(const double2* __restrict__ Dm, const double2* __restrict__ S, int nb,
                            double2* __restrict__ DS, float2* __restrict__ DS32) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 2LL * nb * nb) return;
  const long long r = e / (2 * nb);
  const int c = (int)(e % (2 * nb));
  const double2 v = c < nb ? Dm[r * nb + c] : -S[r * nb + c - nb];
  DS[e] = v;
  DS32[e] = make_float2((float)v.x, (float)v.y);
}

// out[0] += sum |a|^2 (FP32 data, FP64 sums)
// out += sum |a|^2: a grid of a few blocks per SM strides over a, each block
// reduces its threads' FP64 partial sums and adds them with one atomic (an
// atomic per warp serialised on the one address for fields of 3e7 values).
constexpr int kNormBlocks = 4 * 152;
__global__ void __launch_bounds__(256) k_norm2_32(const float2* __restrict__ a, long long n, double* __restrict__ out) {
  __shared__ double red[8];
  double v = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float2 x = a[i];
    v += (double)x.x * x.x + (double)x.y * x.y;
  }
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) atomicAdd(out, v);
  }
}

// ---- adjoint refinement: transposed residual r = L - A^T Y -------------------
//
// Y holds the adjoint in the row space of the discrete system: Ypde at every
// interior leaf node (the PDE rows), per merge level the adjoints of the
// interface terms s_a = r_F + i eta r_C and s_b = r_F - i eta r_C (so that the
// continuity rows u_a - u_b and the flux rows d_n u_a + d_n u_b carry
// Y_C = i eta (Ys_a - Ys_b) and Y_F = Ys_a + Ys_b), and the exterior rows
// [D - I/2, -S] [u; d_n u] at the boundary nodes (through V = [D - I/2, -S]^T Yext).
// L is the receiver functional u_far(p) = A2[p] . [u; d_n u] at the boundary.
// Per leaf edge node the edge coefficients (Eu of the node's own u, En of its
// outward normal derivative) collect the interface and exterior terms; the
// kernel then applies the transposed leaf rows.

// The transposed rows are summed as k_res_pde sums the rows: in fixed point (y and
// the normal coefficients of one right-hand side scaled by their largest parts),
// from the sums and differences of mirrored nodes, D2^T y at i and 15 - i from
// seven coefficients each; the own coefficients Eu are added in FP64.  One thread
// per part, right-hand side and mirrored quadruple of nodes: 49 interior
// quadruples, then the 14 that lie on the edges.
// FP64 multiply-adds bounded the plain sums (66 complex by real ones a node):
// the three residuals of a k = 20 Jacobian (256 leaves, 80 receivers) 1.4 -> 0.67 ms, the
// Jacobian 20.4 -> 19.6; of a k = 40 Gauss-Newton step (1024 leaves, 160 receivers) 10.9 -> 4.4.
// Root mean square rounding for plane waves (k = 40, h = 1/16): 1.0e-10 inside, 3.0e-10 on
// the edges, 2.1e-10 and 2.9e-10 of the FP64 sums.
__global__ void __launch_bounds__(RP_THREADS, 2) k_adj_res(const double2* __restrict__ Ypde, const int4* __restrict__ desc,
                                                        const double2* __restrict__ Yif, const double2* __restrict__ A2,
                                                        const double2* __restrict__ V, const double* __restrict__ q,
                                                        const double* __restrict__ D1, double k, double h, double eta,
                                                        int nb, int nrhs, int first, float2* __restrict__ G) {
  __shared__ double Dx[16][16], D2c[8][16], Ed[8][8], Od[8][8];
  __shared__ int2 E[8][8], O[8][8], N0[16], N15[16], cq[NI];
  __shared__ unsigned my[RCH], mz[RCH], mrow[8], mq, mn;  // largest magnitudes (leading words)
  extern __shared__ double2 rp_dyn[];  // y[NI], en[NE], eu[NE][RCH], then sx, dx, sy, dy [14][7][RCH]
  auto yd = reinterpret_cast<double2(*)[RCH]>(rp_dyn);
  auto end = yd + NI, eu = end + NE;
  auto y = reinterpret_cast<int4(*)[RCH]>(rp_dyn);
  auto en = y + NI;
  auto sx = reinterpret_cast<int4(*)[7][RCH]>(rp_dyn + (NI + 2 * NE) * RCH);
  auto dx = sx + 14, sy = sx + 28, dy = sx + 42;
  const int leaf = blockIdx.x, j0 = blockIdx.y * RCH, t = threadIdx.x, lane = t & 31;
  const int nj = min(RCH, nrhs - j0), j = t % RCH;
  const double sc = 2.0 / h, kk = k * k;
  const double* ql = q + (long long)leaf * 256;
  if (t < RCH) my[t] = mz[t] = mrow[t] = 0;
  if (t == RCH) mq = 0;
  for (int e = t; e < 256; e += RP_THREADS) Dx[e / 16][e % 16] = D1[e] * sc;
  __syncthreads();
  auto mag = [](double x) { return (unsigned)__double2hiint(x) & 0x7FFFFFFFu; };
  const bool whole = t < RP_THREADS / 32 * 32;  // (the last warp is a partial one)
  auto note = [&](unsigned m, unsigned* to) {
    if (whole)
      for (int off = RCH; off < 32; off <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, off));
    if (lane < RCH) atomicMax(&to[j], m);
  };
  unsigned mx = 0;  // (the thread's elements are all of right-hand side j)
  for (int e = t; e < NI * RCH; e += RP_THREADS) {
    const int r = e / RCH;
    const double2 v = !first && j < nj ? Ypde[((long long)leaf * NI + r) * nrhs + j0 + j] : make_double2(0.0, 0.0);
    yd[r][j] = v;
    mx = max(mx, max(mag(v.x), mag(v.y)));
  }
  note(mx, my);
  mx = 0;
  for (int e = t; e < NE * RCH; e += RP_THREADS) {
    const int r = e / RCH;
    double2 u = make_double2(0.0, 0.0), n = make_double2(0.0, 0.0);
    if (j < nj) {
      const int4 d = desc[leaf * NE + r];
      const long long p = j0 + j;
      if (d.z == 2) {  // boundary node d.x: u_far row minus the exterior rows' transpose
        u = A2[p * 2 * nb + d.x];
        n = A2[p * 2 * nb + nb + d.x];
        if (V) {
          u = u - V[(long long)d.x * nrhs + p];
          n = n - V[(long long)(nb + d.x) * nrhs + p];
        }
      } else if (!first) {  // interface node: d.x = (offset of its s_a row) / nrhs, d.y = ni
        const double2 sa = Yif[(long long)d.x * nrhs + p], sb = Yif[((long long)d.x + d.y) * nrhs + p];
        const double2 dd = sa - sb;
        const double2 yc = make_double2(-eta * dd.y, eta * dd.x);  // i eta (Ys_a - Ys_b)
        u = d.z == 0 ? -yc : yc;                                  // row u_a - u_b
        n = -(sa + sb);                                           // row d_n u_a + d_n u_b
      }
    }
    eu[r][j] = u;
    end[r][j] = n;
    mx = max(mx, max(mag(n.x), mag(n.y)));
  }
  note(mx, mz);
  // columns 0..7 of D2, and the largest coefficients
  for (int e = t; e < 8 * 14; e += RP_THREADS) {
    const int i = e / 14, a = e % 14 + 1;
    double acc = 0.0;
    for (int m = 0; m < 16; ++m) acc = fma(Dx[a][m], Dx[m][i], acc);
    D2c[i][a] = acc;
  }
  if (whole) {
    const unsigned vq = __reduce_max_sync(
        0xffffffffu, t < NI ? mag(kk * (1.0 - ql[(t / 14 + 1) * 16 + t % 14 + 1])) : 0u);
    if (lane == 0) atomicMax(&mq, vq);
    if (t < 32) {
      const unsigned vn = __reduce_max_sync(0xffffffffu, mag(t < 16 ? Dx[0][t] : Dx[15][t - 16]));
      if (lane == 0) mn = vn;
    }
  }
  __syncthreads();
  if (t < 8 * 7) {
    const int i = t / 7, c = t % 7;
    Ed[i][c] = 0.5 * (D2c[i][c + 1] + D2c[i][14 - c]);
    Od[i][c] = 0.5 * (D2c[i][c + 1] - D2c[i][14 - c]);
    atomicMax(&mrow[i], max(mag(Ed[i][c]), mag(Od[i][c])));
  }
  const int ey = row_exp((long long)my[j] << 32), ez = row_exp((long long)mz[j] << 32);
  for (int e = t; e < (NI + NE) * RCH; e += RP_THREADS) {  // (each thread its own elements, in place)
    const int r = e / RCH, ex = r < NI ? ey : ez;
    const double2 v = yd[r][j];
    const int2 re = limbs(fixed56(v.x, ex)), im = limbs(fixed56(v.y, ex));
    y[r][j] = make_int4(re.x, re.y, im.x, im.y);
  }
  __syncthreads();
  const int ed = row_exp((long long)mn << 32), eq = row_exp((long long)mq << 32);
  if (t < 8 * 7) {
    const int i = t / 7, c = t % 7, er = row_exp((long long)mrow[i] << 32);
    E[i][c] = limbs(fixed56(Ed[i][c], er));
    O[i][c] = limbs(fixed56(Od[i][c], er));
  }
  if (t < 16) N0[t] = limbs(fixed56(-Dx[0][t], ed));
  else if (t < 32) N15[t - 16] = limbs(fixed56(Dx[15][t - 16], ed));
  if (t < NI) cq[t] = limbs(fixed56(kk * (1.0 - ql[(t / 14 + 1) * 16 + t % 14 + 1]), eq));
  // the line sums and differences (x lines: column b = l + 1; y lines: row a = l + 1)
  for (int e = first ? 2 * 14 * 7 * RCH : t; e < 2 * 14 * 7 * RCH; e += RP_THREADS) {  // (no y at first)
    const int c = (e / RCH) % 7, l = (e / (7 * RCH)) % 14, dir = e / (14 * 7 * RCH);
    const int4 p = dir == 0 ? y[c * 14 + l][j] : y[l * 14 + c][j];
    const int4 m = dir == 0 ? y[(13 - c) * 14 + l][j] : y[l * 14 + 13 - c][j];
    // limbs add limb by limb: below 2^29 and 2^28
    (dir == 0 ? sx : sy)[l][c][j] = make_int4(p.x + m.x, p.y + m.y, p.z + m.z, p.w + m.w);
    (dir == 0 ? dx : dy)[l][c][j] = make_int4(p.x - m.x, p.y - m.y, p.z - m.z, p.w - m.w);
  }
  __syncthreads();
  if (j >= nj) return;
  const bool bad = max(max(ey, ez), eq) >= OZ_NAN / 2;  // an infinity or a NaN in the adjoint (or the contrast)
#pragma unroll 1
  for (int round = 0; round < 3; ++round) {
    const int g = t / RCH;
    int a, b, p = round;  // mirrors 15 - a, 15 - b; the x lines of b and y lines of a exist for 1..7
    if (round < 2) {
      a = g / 7 + 1;
      b = g % 7 + 1;
    } else {
      if (g >= 28) break;
      p = g / 14;
      a = g % 14 < 7 ? 0 : g % 7 + 1;
      b = g % 14 < 7 ? g % 7 + 1 : 0;
    }
    auto part = [&](const int4& v) { return reinterpret_cast<const int2*>(&v)[p]; };
    const int ea = row_exp((long long)mrow[a] << 32), eb = row_exp((long long)mrow[b] << 32);
    const int em = max(max(ea, eb), eq), none = -1 << 16;  // (zeros have no exponent)
    const int top = max(max(my[j] ? ey + em : none, mz[j] ? ez + ed : none), -1200);
    auto shift = [&](int e) { return min(max(top - e, 0), 63); };
    const int sa = shift(ey + ea), sb = shift(ey + eb), sq = shift(ey + eq), sn = shift(ez + ed);
    FixSum xe[2], xo[2], ye[2], yo[2];  // columns b, 15 - b (rows a, 15 - a)
    if (b > 0 && !first)
#pragma unroll 2
      for (int c = 0; c < 7; ++c)
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          const int2 s1 = part(sx[w ? 14 - b : b - 1][c][j]), d1 = part(dx[w ? 14 - b : b - 1][c][j]);
          xe[w].mac(E[a][c], s1.x, s1.y);
          xo[w].mac(O[a][c], d1.x, d1.y);
        }
    if (a > 0 && !first)
#pragma unroll 2
      for (int c = 0; c < 7; ++c)
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          const int2 s2 = part(sy[w ? 14 - a : a - 1][c][j]), d2 = part(dy[w ? 14 - a : a - 1][c][j]);
          ye[w].mac(E[b][c], s2.x, s2.y);
          yo[w].mac(O[b][c], d2.x, d2.y);
        }
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const int ma = n & 1, mb = n >> 1;  // mirrored in a, in b
      const int A = ma ? 15 - a : a, B = mb ? 15 - b : b, r = lidx(A, B);
      const FixSum fx = ma ? xe[mb] - xo[mb] : xe[mb] + xo[mb];
      const FixSum fy = mb ? ye[ma] - yo[ma] : ye[ma] + yo[ma];
      FixSum fq, fn;
      if (r < NI) {
        const int2 v = part(y[r][j]);
        fq.mac(cq[r], v.x, v.y);
      }
      auto normal = [&](int2 d, int e) {
        const int2 v = part(en[e][j]);
        fn.mac(d, v.x, v.y);
      };
      if (a > 0) {  // normal derivatives at the S and N nodes of column A
        normal(N0[B], A - 1);
        normal(N15[B], 28 + A - 1);
      }
      if (b > 0) {  // at the W and E nodes of row B
        normal(N0[A], 42 + B - 1);
        normal(N15[A], 14 + B - 1);
      }
      // (rounded shifts: truncation nearly doubled the error where the normal terms' unit is the coarser one)
      const long long v = fn.down(sn) - fx.down(sa) - fy.down(sb) - fq.down(sq);
      float o = fix_float(v, top - 56);
      if (r >= NI) o = (float)(fix_double(v, top - 56) + reinterpret_cast<const double*>(&eu[r - NI][j])[p]);
      reinterpret_cast<float*>(G + ((long long)leaf * NL + r) * nrhs + j0 + j)[p] = bad ? __int_as_float(0x7FC00000) : o;
    }
  }
}

// Edge rows of the transposed leaf step: G_e += -2 i eta Hadj (the adjoint of
// the leaf's particular outgoing impedance h = -2 i eta u_e).
__global__ void k_leaf_hadj(const float2* __restrict__ H, int nleaf, double eta, int nrhs, float2* __restrict__ G) {
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)nleaf * NE * nrhs) return;
  const int j = (int)(e % nrhs);
  const long long t = e / nrhs;
  const int r = (int)(t % NE), leaf = (int)(t / NE);
  const float2 v = H[e];
  const float te = (float)(2.0 * eta);
  float2* g = G + ((long long)leaf * NL + NI + r) * nrhs + j;
  *g = make_float2(g->x + te * v.y, g->y - te * v.x);
}

// Yif += [MU top; -MU bottom] for one level ([nbox][2 ni][nrhs]): the adjoints of
// s_a and s_b are Wt and -la3 of the transposed sweep.
__global__ void k_iface_adj_add(const float2* __restrict__ MU, int ni, int nrhs, long long n, double2* __restrict__ Y) {
  long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int t = (int)((e / nrhs) % (2 * ni));
  const float2 m = MU[e];
  const double sg = t < ni ? 1.0 : -1.0;
  Y[e] = make_double2(Y[e].x + sg * m.x, Y[e].y + sg * m.y);
}

inline unsigned blocks(long long n) { return (unsigned)((n + 255) / 256); }

}  // namespace

void adjoint_residual(cudaStream_t s, const double2* Ypde, const int4* desc, const double2* Yif, const double2* A2,
                      const double2* V, const double* q, const double* D1, int nleaf, int nb, double k, double h,
                      double eta, int nrhs, bool first, float2* G) {
  dim3 g(nleaf, (nrhs + RCH - 1) / RCH);
  constexpr int bytes = (NI + 2 * NE + 4 * 14 * 7) * RCH * (int)sizeof(double2);
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !attr[dev]) {
    cudaFuncSetAttribute(k_adj_res, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (dev >= 0 && dev < 64) attr[dev] = true;
  }
  k_adj_res<<<g, RP_THREADS, bytes, s>>>(Ypde, desc, Yif, A2, V, q, D1, k, h, eta, nb, nrhs, first ? 1 : 0, G);
  HS_COUNT_LAUNCH();
}

void leaf_hadj(cudaStream_t s, const float2* H, int nleaf, double eta, int nrhs, float2* G) {
  long long n = (long long)nleaf * NE * nrhs;
  k_leaf_hadj<<<blocks(n), 256, 0, s>>>(H, nleaf, eta, nrhs, G);
  HS_COUNT_LAUNCH();
}

void iface_adj_add(cudaStream_t s, const float2* MU, int nbox, int ni, int nrhs, double2* Y) {
  long long n = (long long)nbox * 2 * ni * nrhs;
  k_iface_adj_add<<<blocks(n), 256, 0, s>>>(MU, ni, nrhs, n, Y);
  HS_COUNT_LAUNCH();
}

void convert_d2f(cudaStream_t s, const double2* a, float2* b, long long n) {
  k_d2f<<<blocks(n), 256, 0, s>>>(a, b, n);
  HS_COUNT_LAUNCH();
}

void convert_f2d_add(cudaStream_t s, const float2* a, double2* b, long long n) {
  k_f2d_add<<<blocks(n), 256, 0, s>>>(a, b, n);
  HS_COUNT_LAUNCH();
}

void residual_pde(cudaStream_t s, const double2* X, const double* q, const double* D1, int nleaf, double k, double h,
                  int nrhs, float2* RP, double2* DN) {
  dim3 g(nleaf, (nrhs + RCH - 1) / RCH);
  constexpr int bytes = (NL + 4 * 14 * 8) * RCH * (int)sizeof(double2);
  static bool attr[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !attr[dev]) {
    cudaFuncSetAttribute(k_res_pde, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (dev >= 0 && dev < 64) attr[dev] = true;
  }
  k_res_pde<<<g, RP_THREADS, bytes, s>>>(X, q, D1, k, h, nrhs, RP, DN);
  HS_COUNT_LAUNCH();
}

void residual_iface(cudaStream_t s, const LevelMaps& L, const double2* X, const double2* DN, int nL,
                    const double* d_k, int nrhs, float2* S3) {
  dim3 g(blocks((long long)L.ni * nrhs), L.nbox);
  k_res_iface<<<g, 256, 0, s>>>(X, DN, nL, d_k, L.horiz, L.sx, L.sy, L.ni, L.nbx_p, nrhs, S3);
  HS_COUNT_LAUNCH();
}

void boundary_gather(cudaStream_t s, const double2* X, const double* D1, int nL, double h, int nrhs, double2* ub,
                     double2* psib) {
  long long n = 56LL * nL * nrhs;
  k_boundary_gather<<<blocks(n), 256, 0, s>>>(X, D1, nL, h, nrhs, ub, psib);
  HS_COUNT_LAUNCH();
}

// Particular leaf solution for body loads b held in Upart rows 0..195 (FP32):
// w = Aii^{-1} b, u_e = -Kinv Ni w, u_i = w - X u_e, and h = -2 i eta u_e.
// With w.Ainv the first step is one GEMM into wtmp (NI x nrhs per leaf) and a
// copy back; otherwise triangular solves with the LU factors.
void leaf_particular(cudaStream_t s, const LeafScratchT<float>& w, int nleaf, const double* d_k, int nrhs, float2* Upart,
                     float2* H, float2* tmp, float2* wtmp) {
  const long long sU = (long long)NL * nrhs;
  const float2 one = make_float2(1.f, 0.f), mone = make_float2(-1.f, 0.f), zero = make_float2(0.f, 0.f);
  if (w.P) {  // impedance-form leaves: [u_i; u_e] = P b in one product (b staged in wtmp)
    cudaMemcpy2DAsync(wtmp, (size_t)NI * nrhs * sizeof(float2), Upart, sU * sizeof(float2),
                      (size_t)NI * nrhs * sizeof(float2), nleaf, cudaMemcpyDeviceToDevice, s);
    gemm<float2, float2, float2>(s, OP_N, OP_N, NL, nrhs, NI, one, w.P, NI, (long long)NL * NI, wtmp, nrhs,
                                 (long long)NI * nrhs, zero, Upart, nrhs, sU, nleaf);
    const long long n = (long long)nleaf * NE * nrhs;
    k_leaf_h<<<blocks(n), 256, 0, s>>>(Upart, nleaf, d_k, nrhs, H);
    HS_COUNT_LAUNCH();
    return;
  }
  if (w.Ainv && wtmp) {
    gemm<float, float2, float2>(s, OP_N, OP_N, NI, nrhs, NI, one, w.Ainv, NI, (long long)NI * NI, Upart, nrhs, sU,
                                zero, wtmp, nrhs, (long long)NI * nrhs, nleaf);
    cudaMemcpy2DAsync(Upart, sU * sizeof(float2), wtmp, (size_t)NI * nrhs * sizeof(float2),
                      (size_t)NI * nrhs * sizeof(float2), nleaf, cudaMemcpyDeviceToDevice, s);
  } else {
    // complex right-hand sides are solved as 2 nrhs real columns
    lu_solve<float>(s, OP_N, w.Aii, NI, (long long)NI * NI, NI, w.piv, NI, reinterpret_cast<float*>(Upart), 2 * nrhs,
                    2 * sU, 2 * nrhs, nleaf);
  }
  gemm<float, float2, float2>(s, OP_N, OP_N, NE, nrhs, NI, one, w.Ni, NI, (long long)NE * NI, Upart, nrhs, sU, zero,
                              tmp, nrhs, (long long)NE * nrhs, nleaf);
  gemm<float2, float2, float2>(s, OP_N, OP_N, NE, nrhs, NE, mone, w.Kinv, NE, (long long)NE * NE, tmp, nrhs,
                               (long long)NE * nrhs, zero, Upart + (long long)NI * nrhs, nrhs, sU, nleaf);
  gemm<float, float2, float2>(s, OP_N, OP_N, NI, nrhs, NE, mone, w.Aie, NE, (long long)NI * NE,
                              Upart + (long long)NI * nrhs, nrhs, sU, one, Upart, nrhs, sU, nleaf);
  long long n = (long long)nleaf * NE * nrhs;
  k_leaf_h<<<blocks(n), 256, 0, s>>>(Upart, nleaf, d_k, nrhs, H);
  HS_COUNT_LAUNCH();
}

void scattered32(cudaStream_t s, const float2* U32, const double* D1, int nL, double h, int nrhs, const double2* ui,
                 const double2* dni, bool sub_inc, float2* PS) {
  long long n = 56LL * nL * nrhs;
  k_scattered32<<<blocks(n), 256, 0, s>>>(U32, D1, nL, h, nrhs, ui, dni, sub_inc ? 1 : 0, PS);
  HS_COUNT_LAUNCH();
}

void stack_exterior(cudaStream_t s, const double2* Dm, const double2* S, int nb, double2* DS, float2* DS32) {
  k_stack_ext<<<blocks(2LL * nb * nb), 256, 0, s>>>(Dm, S, nb, DS, DS32);
  HS_COUNT_LAUNCH();
}

void norm2_32(cudaStream_t s, const float2* a, long long n, double* out) {
  if (n <= 0) return;
  k_norm2_32<<<(unsigned)std::min<long long>(kNormBlocks, (n + 255) / 256), 256, 0, s>>>(a, n, out);
  HS_COUNT_LAUNCH();
}

void scattered_data(cudaStream_t s, const double2* ub, const double2* psib, const double2* ui, const double2* dni,
                    long long n, double2* PS) {
  k_scattered<<<blocks(n), 256, 0, s>>>(ub, psib, ui, dni, n, PS);
  HS_COUNT_LAUNCH();
}

}  // namespace hs
