// npr.cu -- the one-colour-trace four-fermion contraction of the NPR workload
// (Sec. 4 of the paper, Eq. (ffop); FP64, its 97 % kernel):
//   O(z) = sum_{A,B,C,D} [chibar1(z_A) (g_S1 x x_F1)_AB chi2(z_B)]
//                        [chibar3(z_C) (g_S2 x x_F2)_CD chi4(z_D)]
//                        [U_AD(z)]_{c1 c4} [U_CB(z)]_{c3 c2}
// on every hypercube z (sites z_A = 2z + A, corners A in {0,1}^4), with
//   (g_S x x_F)_AB = (1/4) Tr(g_A^dag g_S g_B g_F^dag),  g_A = g_1^A1 ... g_4^A4,
//   U_AD(z) = the average over the shortest paths from z_A to z_D inside the
//   hypercube of the link products (U_mu for +mu, U_mu^dag for -mu).
// One block per hypercube, 256 threads:
//   * the path averages W(A, D) in shared memory, both orientations (W(D, A) =
//     W(A, D)^dag, so that no read conjugates), W(A, A) = 1: level n = 1 is
//     the hypercube's 32 internal links; levels n = |A xor D| = 2, 3, 4 (a
//     table of the pairs A < D per level), one thread per matrix element: a
//     path's last step is one of the differing directions mu, so
//     W(A, D) = (1/n) sum_mu W(A, D xor mu) W(D xor mu, D);
//   * the spin-taste entries from the Clifford algebra: g_X g_Y = e(X, Y)
//     g_{X xor Y} with e(X, Y) = (-1)^(sum_{mu > nu} X_mu Y_nu), g_A^dag =
//     (-1)^(n(n-1)/2) g_A (n set bits), so (g_S x x_F)_AB is nonzero only for
//     A xor S xor B xor F = 0, where it is the product of those signs;
//   * thread (A, C) evaluates its term (B = A xor S1 xor F1, D = C xor S2 xor
//     F2), the block sums the 256 terms in a fixed order.
#include <cuda_runtime.h>

#include "launch.h"
#include "su3_fixed.cuh"

namespace stag {

namespace {

constexpr int NPR_BT = 256;

__device__ __forceinline__ double2 zm(double2 x, double2 y) { return make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x); }
__device__ __forceinline__ double2 za(double2 x, double2 y) { return make_double2(x.x + y.x, x.y + y.y); }
// s + x y as two FMA chains per component (4 FP64 instructions for 8 flops)
__device__ __forceinline__ double2 zfma(double2 x, double2 y, double2 s) {
  return make_double2(__fma_rn(-x.y, y.y, __fma_rn(x.x, y.x, s.x)), __fma_rn(x.y, y.x, __fma_rn(x.x, y.y, s.y)));
}

// reversal sign of g_A^dag = (-1)^(n(n-1)/2) g_A
__device__ __forceinline__ int rev_sign(int A) {
  const int n = __popc(A);
  return ((n * (n - 1) / 2) & 1) ? -1 : 1;
}
// e(X, Y): g_X g_Y = e g_{X xor Y}
__device__ __forceinline__ int mul_sign(int X, int Y) {
  int cnt = 0;
#pragma unroll
  for (int nu = 0; nu < 4; ++nu)
    if ((Y >> nu) & 1) cnt += __popc(X >> (nu + 1));
  return (cnt & 1) ? -1 : 1;
}
// (g_S x x_F)_AB (real: 0 or +-1)
__device__ __forceinline__ double spin_taste(int S, int F, int A, int B) {
  if ((A ^ S ^ B ^ F) != 0) return 0.0;
  const int s = rev_sign(A) * rev_sign(F) * mul_sign(A, S) * mul_sign(A ^ S, B) * mul_sign(A ^ S ^ B, F);
  return (double)s;
}

// the 120 corner pairs A < D of a hypercube, ordered by n = |A xor D|
// (32, 48, 32, 8 pairs), and the offset of each level
struct PairTable {
  unsigned char a[120], d[120];
  int off[5];
};
constexpr int popc4(int x) { return (x & 1) + ((x >> 1) & 1) + ((x >> 2) & 1) + ((x >> 3) & 1); }
constexpr PairTable make_pairs() {
  PairTable p{};
  int k = 0;
  for (int n = 1; n <= 4; ++n) {
    p.off[n - 1] = k;
    for (int A = 0; A < 16; ++A)
      for (int D = A + 1; D < 16; ++D)
        if (popc4(A ^ D) == n) {
          p.a[k] = (unsigned char)A;
          p.d[k] = (unsigned char)D;
          ++k;
        }
  }
  p.off[4] = k;
  return p;
}
__constant__ PairTable c_pairs = make_pairs();

struct NprArgs {
  int L[4], H[4];
  long long V;
  const double2 *U;  // [4][V][9]
  const double2 *cb1, *c2, *cb3, *c4;  // [V][3]
  int S1, F1, S2, F2;
  double2 *out;      // [nhyp]
};

// this block's hypercube; W(A, D) at index A * 16 + D, both orientations; fld:
// chibar1, chi2, chibar3, chi4 at the corners; red: a value a warp
__device__ __forceinline__ void npr_fp64(const NprArgs &a, double2 (*W)[9], double2 (*fld)[16][3], double2 *red,
                                         unsigned char *pa, unsigned char *pd) {
  const long long h = blockIdx.x;
  int zc[4];
  {
    long long r = h;
    zc[0] = (int)(r % a.H[0]);
    r /= a.H[0];
    zc[1] = (int)(r % a.H[1]);
    r /= a.H[1];
    zc[2] = (int)(r % a.H[2]);
    zc[3] = (int)(r / a.H[2]);
  }
  auto site = [&](int A) -> long long {
    const int x0 = 2 * zc[0] + (A & 1), x1 = 2 * zc[1] + ((A >> 1) & 1), x2 = 2 * zc[2] + ((A >> 2) & 1),
              x3 = 2 * zc[3] + ((A >> 3) & 1);
    return x0 + (long long)a.L[0] * (x1 + (long long)a.L[1] * (x2 + (long long)a.L[2] * x3));
  };
  const int t = threadIdx.x;
  // level n = 1, the hypercube's 32 internal links: W(A, D) = U_mu(z_A) for
  // D = A + mu (A_mu = 0), W(D, A) its adjoint; level 0: W(A, A) = 1
  for (int k = t; k < 32 * 9; k += NPR_BT) {
    const int l = k / 9, e = k % 9, mu = l / 8, y = l % 8;
    const int A = ((y >> mu) << (mu + 1)) | (y & ((1 << mu) - 1)), D = A | (1 << mu);
    const double2 u = a.U[((long long)mu * a.V + site(A)) * 9 + e];
    W[A * 16 + D][e] = u;
    W[D * 16 + A][(e % 3) * 3 + e / 3] = make_double2(u.x, -u.y);
  }
  for (int k = t; k < 4 * 16 * 3; k += NPR_BT) {
    const int f = k / 48, A = (k / 3) % 16, c = k % 3;
    const double2 *src = f == 0 ? a.cb1 : f == 1 ? a.c2 : f == 2 ? a.cb3 : a.c4;
    fld[f][A][c] = src[site(A) * 3 + c];
  }
  for (int k = t; k < 16 * 9; k += NPR_BT) {
    const int Y = k / 9, e = k % 9;
    W[Y * 17][e] = make_double2((e % 4 == 0) ? 1.0 : 0.0, 0.0);
  }
  if (t < 120) {
    pa[t] = c_pairs.a[t];
    pd[t] = c_pairs.d[t];
  }
  __syncthreads();
  // levels n = 2, 3, 4, the pairs A < D from the table: the last step of a
  // path is one of the differing directions mu, from P = D xor mu, so
  // W(A, D) = (1/n) sum_mu W(A, P) W(P, D) (W(P, D): a link or its adjoint);
  // one thread per matrix element, which also writes the adjoint entry
  for (int n = 2; n <= 4; ++n) {
    const int p0 = c_pairs.off[n - 1], nitem = (c_pairs.off[n] - p0) * 9;
    for (int item = t; item < nitem; item += NPR_BT) {
      const int pr = p0 + item / 9, e = item % 9;
      const int A = pa[pr], D = pd[pr];
      const int i = e / 3, j = e % 3;
      double2 s = make_double2(0.0, 0.0);
      for (int mu = 0; mu < 4; ++mu) {
        if (!(((A ^ D) >> mu) & 1)) continue;
        const int P = D ^ (1 << mu);
        const double2 *wa = W[A * 16 + P], *wb = W[P * 16 + D];
#pragma unroll
        for (int k = 0; k < 3; ++k) s = zfma(wa[i * 3 + k], wb[k * 3 + j], s);
      }
      const double inv = n == 2 ? 0.5 : n == 3 ? 1.0 / 3.0 : 0.25;  // constants: no FP64 division
      s = make_double2(s.x * inv, s.y * inv);
      W[A * 16 + D][e] = s;
      W[D * 16 + A][j * 3 + i] = make_double2(s.x, -s.y);
    }
    __syncthreads();
  }
  // thread (A, C): its term
  const int A = t >> 4, C = t & 15;
  const int B = A ^ a.S1 ^ a.F1, Dd = C ^ a.S2 ^ a.F2;
  const double s = spin_taste(a.S1, a.F1, A, B) * spin_taste(a.S2, a.F2, C, Dd);
  double2 t1 = make_double2(0.0, 0.0), t2 = make_double2(0.0, 0.0);
  {
    auto wget = [&](int X, int Y, int i, int j) -> double2 { return W[X * 16 + Y][i * 3 + j]; };
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double2 v1 = make_double2(0.0, 0.0), v2 = make_double2(0.0, 0.0);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        v1 = zfma(wget(A, Dd, i, j), fld[3][Dd][j], v1);
        v2 = zfma(wget(C, B, i, j), fld[1][B][j], v2);
      }
      t1 = zfma(fld[0][A][i], v1, t1);
      t2 = zfma(fld[2][C][i], v2, t2);
    }
  }
  double2 term = zm(t1, t2);
  term.x *= s;
  term.y *= s;
  // fixed-order block sum
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    term.x += __shfl_xor_sync(0xffffffffu, term.x, o);
    term.y += __shfl_xor_sync(0xffffffffu, term.y, o);
  }
  if ((t & 31) == 0) red[t >> 5] = term;
  __syncthreads();
  if (t == 0) {
    double2 o = make_double2(0.0, 0.0);
    for (int w = 0; w < NPR_BT / 32; ++w) o = za(o, red[w]);
    a.out[h] = o;
  }
}

__global__ void __launch_bounds__(NPR_BT) k_npr(const NprArgs a) {
  __shared__ double2 W[256][9];
  __shared__ double2 fld[4][16][3];
  __shared__ double2 red[NPR_BT / 32];
  __shared__ unsigned char pa[120], pd[120];
  npr_fp64(a, W, fld, red, pa, pd);
}

// ---------------------------------------------------------------------------
// the same contraction on the integer pipe (fields that pass fx_field)
// ---------------------------------------------------------------------------
// k_npr keeps the FP64 pipe 95 % busy (12 000 complex multiply-adds a
// hypercube; 3.90 ms at 20^3 x 64, 1.30 ms here: issue slots 48 % and shared
// memory 50 % busy, the levels' barriers between).  Here they are fixed-point
// sums (fixed.cuh): links and path averages at 2^58, a field at 2^57 under one
// exponent a corner (its 3 colours).  FP64 is left for the product of the two
// bilinears and the sum of the 256 terms.
// Ranges, every link stretching a vector by at most 1.0015 (near_unitary): a path
// average W of up to 4 links by 1.006, so its elements have |h| < 2^29.1, W y of a
// y with components |.| <= 1 has components below 1.006 sqrt(6) 2^57, |h| < 2^29.4,
// and x . (W y) is below 6.1 2^56.  A sum of up to 4 x 3 complex products has |hh|
// <= 4 x 1.006 2^58 and, its limbs at most 2^29.1 and 2^28, |cr| <= 48 2^57.1 < 2^63.
// Errors are fractions of the corners' scales: a bilinear x W y errs by up to
// 45 x 2^-57 of their product.  What FP64 would keep beyond that stays in FP64:
//   * corners 0 or 1 step apart, where single elements of W decide: a bilinear
//     with a real or imaginary part whose terms' magnitudes sum to less than 2^-5
//     is formed in FP64 from the FP64 link; the others err by at most 90 x 2^-53 of those
//     magnitudes.  Three partial sums, each a lower bound, spare most the count: with Gaussian
//     fields 9 % of the warps take it, 1e-5 of the threads FP64.  (Two and more
//     steps average two and more paths of three terms each: no small W from mixing
//     links.)
//   * a hypercube with over an eighth of its links' real components below FX_SMALL,
//     as in a cold region of a rough field, or whose fields hold numbers far from 1,
//     infinities or NaNs at a corner: all of it, as k_npr does.

// v / n, n = 2, 3, 4
__device__ __forceinline__ long long fx_over(long long v, int n) {
  return n == 2 ? v >> 1 : n == 4 ? v >> 2 : fx_third(v);
}

constexpr int NPR_E0 = 600, NPR_E1 = 1400;  // exponent fields of the integer form
constexpr int NPR_LINE = 1 << 19;           // 2^-5 of the scales, in the high word of a bilinear (unit 2^-56)

// the whole hypercube in FP64 (out of line: the kernel's registers are the integer form's)
__device__ __noinline__ void npr_block_fp64(const NprArgs &a, double2 (*W)[9], double2 (*fld)[16][3], double2 *red,
                                            unsigned char *pa, unsigned char *pd) {
  npr_fp64(a, W, fld, red, pa, pd);
}

// whether the terms of x^T W y sum to less than 2^-5 in magnitude, in its real or in its imaginary part
__device__ __forceinline__ bool terms_small(const int4 *x, const int4 *w, const int4 *y) {
  float re = 0.f, im = 0.f;
  for (int i = 0; i < 3; ++i) {
    float vr = 0.f, vi = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float wr = fabsf((float)w[3 * i + j].x), wi = fabsf((float)w[3 * i + j].z);
      const float yr = fabsf((float)y[j].x), yi = fabsf((float)y[j].z);
      vr += wr * yr + wi * yi;
      vi += wr * yi + wi * yr;
    }
    const float xr = fabsf((float)x[i].x), xi = fabsf((float)x[i].z);
    re += xr * vr + xi * vi;
    im += xr * vi + xi * vr;
  }
  return fminf(re, im) < 0x1p80f;  // units of 2^-28, 2^-29 and 2^-28
}

// b, or, where its terms are small, x^T W y in FP64: W = 1 (u null), the link u or (dag) its adjoint;
// xs, ys the corners' colours, x, w, y the fixed-point ones
__device__ __noinline__ double2 bilinear_checked(double2 b, const int4 *x, const int4 *w, const int4 *y,
                                                 const double2 *xs, const double2 *ys, const double2 *u, bool dag) {
  if (!terms_small(x, w, y)) return b;
  double2 sum = make_double2(0.0, 0.0);
  double2 v[3], f[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    v[k] = __ldg(ys + k);
    f[k] = __ldg(xs + k);
  }
  for (int i = 0; i < 3; ++i) {
    double2 l = v[i];
    if (u != nullptr) {
      double2 s = make_double2(0.0, 0.0);
      for (int j = 0; j < 3; ++j) {
        l = __ldg(u + (dag ? 3 * j + i : 3 * i + j));
        if (dag) l.y = -l.y;
        s = zfma(l, v[j], s);
      }
      l = s;
    }
    sum = zfma(f[i], l, sum);
  }
  return sum;
}

__global__ void __launch_bounds__(NPR_BT, 4) k_npr_fx(const __grid_constant__ NprArgs a) {
  __shared__ int4 W[256][9];      // as npr_fp64, fixed-point
  __shared__ int4 fld[4][16][3];  // the fields at the corners, fixed-point
  __shared__ double2 term[NPR_BT];
  __shared__ int top[4][16];  // largest exponent bits of a field at a corner, 0 where it is zero
  __shared__ int nsmall;      // real components of the links below FX_SMALL
  __shared__ unsigned char pa[120], pd[120];
  const long long h = blockIdx.x;
  int zc[4];
  {
    long long r = h;
    zc[0] = (int)(r % a.H[0]);
    r /= a.H[0];
    zc[1] = (int)(r % a.H[1]);
    r /= a.H[1];
    zc[2] = (int)(r % a.H[2]);
    zc[3] = (int)(r / a.H[2]);
  }
  auto site = [&](int A) -> long long {
    const int x0 = 2 * zc[0] + (A & 1), x1 = 2 * zc[1] + ((A >> 1) & 1), x2 = 2 * zc[2] + ((A >> 2) & 1),
              x3 = 2 * zc[3] + ((A >> 3) & 1);
    return x0 + (long long)a.L[0] * (x1 + (long long)a.L[1] * (x2 + (long long)a.L[2] * x3));
  };
  const int t = threadIdx.x;
  const int ff = t / 48, fa = (t / 3) % 16, fc = t % 3;  // this thread's field, corner and colour (t < 192)
  const double2 *fsrc = ff == 0 ? a.cb1 : ff == 1 ? a.c2 : ff == 2 ? a.cb3 : a.c4;
  double2 fv = make_double2(0.0, 0.0);
  if (t < 192) fv = fsrc[site(fa) * 3 + fc];
  if (t < 64) (&top[0][0])[t] = 0;
  if (t == 64) nsmall = 0;
  int small = 0;
  for (int k = t; k < 32 * 9; k += NPR_BT) {
    const int l = k / 9, e = k % 9, mu = l / 8, y = l % 8;
    const int A = ((y >> mu) << (mu + 1)) | (y & ((1 << mu) - 1)), D = A | (1 << mu);
    const double2 u = a.U[((long long)mu * a.V + site(A)) * 9 + e];
    const Fx re = fx_link(__double2hiint(u.x), __double2loint(u.x));
    const Fx im = fx_link(__double2hiint(u.y), __double2loint(u.y));
    const int4 w = make_int4(re.h, re.l, im.h, im.l);
    small += (abs(re.h) < (int)(FX_SMALL * 0x1p29f)) + (abs(im.h) < (int)(FX_SMALL * 0x1p29f));
    W[A * 16 + D][e] = w;
    W[D * 16 + A][(e % 3) * 3 + e / 3] = fx_conj(w);
  }
  for (int k = t; k < 16 * 9; k += NPR_BT) {
    const int Y = k / 9, e = k % 9;
    W[Y * 17][e] = make_int4((e % 4 == 0) ? 1 << FX_LO : 0, 0, 0, 0);
  }
  if (t < 120) {
    pa[t] = c_pairs.a[t];
    pd[t] = c_pairs.d[t];
  }
  __syncthreads();
  small = __reduce_add_sync(0xffffffffu, small);
  if ((t & 31) == 0 && small > 0) atomicAdd(&nsmall, small);
  if (t < 192) {
    int hi = max(__double2hiint(fv.x) & 0x7fffffff, __double2hiint(fv.y) & 0x7fffffff);
    if (hi == 0 && (__double2loint(fv.x) | __double2loint(fv.y)) != 0) hi = 1;  // a denormal
    atomicMax(&top[ff][fa], hi);
  }
  bool off = false;  // uniform over the block after the last level
  // levels n = 2, 3: one thread a row of W(A, D) (each W(A, P) row serves three
  // elements); level 4, with only 8 pairs: one thread an element
#pragma unroll
  for (int n = 2; n <= 4; ++n) {
    const int p0 = c_pairs.off[n - 1], np = c_pairs.off[n] - p0;
    constexpr int COLS = 3;
    const int per = n < 4 ? 3 : 9;
    for (int item = t; item < np * per; item += NPR_BT) {
      const int pr = p0 + item / per, e = item % per;
      const int A = pa[pr], D = pd[pr];
      const int i = n < 4 ? e : e / 3, j0 = n < 4 ? 0 : e % 3;
      CAcc c[COLS];
#pragma unroll
      for (int j = 0; j < COLS; ++j) c[j] = cacc_zero();
      for (int mu = 0; mu < 4; ++mu) {
        if (!(((A ^ D) >> mu) & 1)) continue;
        const int Pm = D ^ (1 << mu);
        const int4 *wa = W[A * 16 + Pm], *wb = W[Pm * 16 + D];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const int4 x = wa[i * 3 + k];
          if (n < 4) {
#pragma unroll
            for (int j = 0; j < COLS; ++j) fx_cmac(c[j], x, wb[k * 3 + j]);
          } else {
            fx_cmac(c[0], x, wb[k * 3 + j0]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < COLS; ++j) {
        if (n == 4 && j > 0) break;
        const int4 w = fx_pair(fx_over(fx_sum(c[j].re), n), fx_over(fx_sum(c[j].im), n));
        W[A * 16 + D][i * 3 + j0 + j] = w;
        W[D * 16 + A][(j0 + j) * 3 + i] = fx_conj(w);
      }
    }
    if (n == 3 && t < 192) {  // top is complete since the last barrier
      const int hi = top[ff][fa], E = hi >> 20;
      off = hi != 0 && (E < NPR_E0 || E > NPR_E1);
      const Fx re = fx_vec(__double2hiint(fv.x), __double2loint(fv.x), off ? 2047 : E);
      const Fx im = fx_vec(__double2hiint(fv.y), __double2loint(fv.y), off ? 2047 : E);
      fld[ff][fa][fc] = make_int4(re.h, re.l, im.h, im.l);
    }
    if (n < 4) __syncthreads();
  }
  off = __syncthreads_or(off || nsmall > 32 * 18 / 8) != 0;
  if (off) {
    npr_block_fp64(a, reinterpret_cast<double2(*)[9]>(&W[0][0]), reinterpret_cast<double2(*)[16][3]>(&fld[0][0][0]),
                   term, pa, pd);
    return;
  }
  const int A = t >> 4, C = t & 15;
  const int B = A ^ a.S1 ^ a.F1, Dd = C ^ a.S2 ^ a.F2;
  const double s = spin_taste(a.S1, a.F1, A, B) * spin_taste(a.S2, a.F2, C, Dd);
  // the bilinear of fields f at corner X and g at corner Y: x^T W y with x, y at
  // 2^57, W at 2^58: W y at 2^57, the sum at 2^56
  auto bilinear = [&](int f, int X, int g, int Y, bool &check) {
    const int4 *x = fld[f][X], *w = W[X * 16 + Y], *y = fld[g][Y];
    CAcc sum = cacc_zero();
    int seen_re = 0, seen_im = 0;  // bits of the partial sums' magnitudes
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      CAcc v = cacc_zero();
#pragma unroll
      for (int j = 0; j < 3; ++j) fx_cmac(v, w[i * 3 + j], y[j]);
      fx_cmac(sum, x[i], fx_cval(v));
      const int hr = (int)(sum.re.hh >> 32), hi = (int)(sum.im.hh >> 32);
      seen_re |= hr ^ (hr >> 31);
      seen_im |= hi ^ (hi >> 31);
    }
    const int tx = top[f][X], ty = top[g][Y], step = X ^ Y;
    // units 2^(E - 1022) of each corner and 2^-56; 0 with a zero corner
    const bool zero = tx == 0 || ty == 0;
    check = !zero && min(seen_re, seen_im) < NPR_LINE && (step & (step - 1)) == 0;
    const double unit = zero ? 0.0 : __hiloint2double(((tx >> 20) + (ty >> 20) - 2 * 1022 - 56 + 1023) << 20, 0);
    return make_double2((double)fx_sum(sum.re) * unit, (double)fx_sum(sum.im) * unit);
  };
  bool check1, check2;
  double2 b1 = bilinear(0, A, 3, Dd, check1), b2 = bilinear(2, C, 1, B, check2);
  if (check1 || check2) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (!(q ? check2 : check1)) continue;
      const int X = q ? C : A, Y = q ? B : Dd, step = X ^ Y;
      const double2 *u = step ? a.U + ((long long)(__ffs(step) - 1) * a.V + site(X & Y)) * 9 : nullptr;
      double2 &b = q ? b2 : b1;
      b = bilinear_checked(b, fld[q ? 2 : 0][X], W[X * 16 + Y], fld[q ? 1 : 3][Y], (q ? a.cb3 : a.cb1) + site(X) * 3,
                           (q ? a.c2 : a.c4) + site(Y) * 3, u, X > Y);
    }
  }
  const double2 z = zm(b1, b2);
  term[t] = make_double2(s * z.x, s * z.y);
  __syncthreads();
  // fixed-order sum of the 256 terms by one warp
  if (t < 32) {
    double2 o = term[t];
#pragma unroll
    for (int k = 1; k < NPR_BT / 32; ++k) o = za(o, term[t + 32 * k]);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      o.x += __shfl_xor_sync(0xffffffffu, o.x, d);
      o.y += __shfl_xor_sync(0xffffffffu, o.y, d);
    }
    if (t == 0) a.out[h] = o;
  }
}

// out[0] = sum of the n values of in, fixed order (one block)
__global__ void __launch_bounds__(NPR_BT) k_npr_sum(const double2 *in, long long n, double2 *out) {
  __shared__ double2 red[NPR_BT / 32];
  double2 s = make_double2(0.0, 0.0);
  for (long long i = threadIdx.x; i < n; i += NPR_BT) s = za(s, in[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double2 o = make_double2(0.0, 0.0);
    for (int w = 0; w < NPR_BT / 32; ++w) o = za(o, red[w]);
    *out = o;
  }
}

}  // namespace

cudaError_t launch_npr(const int dims[4], const double2 *U, const int st[4], const double2 *cb1, const double2 *c2,
                       const double2 *cb3, const double2 *c4, double2 *out, double2 *sum, bool fx, cudaStream_t s) {
  NprArgs a;
  long long nh = 1;
  for (int k = 0; k < 4; ++k) {
    a.L[k] = dims[k];
    a.H[k] = dims[k] / 2;
    nh *= a.H[k];
  }
  a.V = 16 * nh;
  a.U = U;
  a.cb1 = cb1;
  a.c2 = c2;
  a.cb3 = cb3;
  a.c4 = c4;
  a.S1 = st[0];
  a.F1 = st[1];
  a.S2 = st[2];
  a.F2 = st[3];
  a.out = out;
  if (fx) k_npr_fx<<<(unsigned)nh, NPR_BT, 0, s>>>(a);
  else k_npr<<<(unsigned)nh, NPR_BT, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !sum) return e;
  k_npr_sum<<<1, NPR_BT, 0, s>>>(out, nh, sum);
  return cudaGetLastError();
}

}  // namespace stag
