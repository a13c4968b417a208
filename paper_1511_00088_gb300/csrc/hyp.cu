// hyp.cu -- HYP smearing of the gauge field on the GPU (FP64): the one-link
// field of the "HYP-smeared staggered quarks" whose CG Sec. 3 benchmarks.
//
// Three levels of decorated links, each a projection to SU(3) of the thin link
// plus a weighted staple sum over the level below, staples kept inside the
// hypercubes of the link (parameters (a1, a2, a3), Hasenfratz-Knechtli's
// (0.75, 0.6, 0.3) by default):
//   Vb(x,mu;e)  = P[(1-a3) U_mu(x) + a3/2 sum_{+-e} U_e U_mu U_e^dag]              (e != mu)
//   Vt(x,mu;nu) = P[(1-a2) U_mu(x) + a2/4 sum_{+-r, r != mu,nu} Vb(r;s) Vb(mu;s) Vb(r;s)^dag]
//                 (s = the direction outside {mu, nu, r})
//   V(x,mu)     = P[(1-a1) U_mu(x) + a1/6 sum_{+-nu != mu} Vt(nu;mu) Vt(mu;nu) Vt(nu;mu)^dag]
// A positive staple in direction d at x is W_d(x) W_mu(x+d) W_d(x+mu)^dag,
// a negative one W_d(x-d)^dag W_mu(x-d) W_d(x-d+mu).
// P(X) = the unitary polar factor of X with the phase of its determinant
// removed by the principal cube root.  Here the polar factor comes from
// Newton's iteration with determinant scaling (Y <- (g Y + (g Y)^-dag) / 2,
// g = |det Y|^(-1/3); Higham, "Computing the polar decomposition", 1986),
// which reaches the same unique factor in fewer steps than the plain one, and
// the determinant's phase from Newton's iteration for a complex cube root.
// Fields that pass fx_field run on the integer pipe instead (k_hyp*_fx below).
// One thread per (decorated link, site); links in the ABI layout
// [direction][site][3][3] complex (decorated: [12 (mu, decoration) slots][site][3][3]).
#include <cmath>
#include <cuda_runtime.h>

#include "launch.h"
#include "su3_fixed.cuh"

namespace stag {

namespace {

struct M3 {
  double2 a[9];
};

__device__ __forceinline__ double2 cm(double2 x, double2 y) { return make_double2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x); }
__device__ __forceinline__ double2 ccj(double2 x) { return make_double2(x.x, -x.y); }
// s + x y as two FMA chains per component (4 FP64 instructions for 8 flops)
__device__ __forceinline__ double2 cfma(double2 x, double2 y, double2 s) {
  return make_double2(__fma_rn(-x.y, y.y, __fma_rn(x.x, y.x, s.x)), __fma_rn(x.y, y.x, __fma_rn(x.x, y.y, s.y)));
}

// a b - c e as FMA chains (4 FP64 instructions per component)
__device__ __forceinline__ double2 cdet2(double2 a, double2 b, double2 c, double2 e) {
  return make_double2(__fma_rn(a.x, b.x, __fma_rn(-a.y, b.y, __fma_rn(-c.x, e.x, c.y * e.y))),
                      __fma_rn(a.x, b.y, __fma_rn(a.y, b.x, __fma_rn(-c.x, e.y, (-c.y) * e.x))));
}

__device__ __forceinline__ M3 ld(const double2 *p) {
  M3 m;
#pragma unroll
  for (int k = 0; k < 9; ++k) m.a[k] = p[k];
  return m;
}

// c += a b, with either factor optionally daggered
template <bool DA, bool DB>
__device__ __forceinline__ void mul_add(const M3 &a, const M3 &b, M3 &c) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double2 s = c.a[i * 3 + j];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double2 x = DA ? ccj(a.a[k * 3 + i]) : a.a[i * 3 + k];
        const double2 y = DB ? ccj(b.a[j * 3 + k]) : b.a[k * 3 + j];
        s = cfma(x, y, s);
      }
      c.a[i * 3 + j] = s;
    }
}

template <bool DA, bool DB>
__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b) {
  M3 c;
#pragma unroll
  for (int k = 0; k < 9; ++k) c.a[k] = make_double2(0.0, 0.0);
  mul_add<DA, DB>(a, b, c);
  return c;
}

__device__ __forceinline__ double2 det3(const M3 &m) {
  const double2 *a = m.a;
  const double2 t0 = cdet2(a[4], a[8], a[5], a[7]);
  const double2 t1 = cdet2(a[5], a[6], a[3], a[8]);
  const double2 t2 = cdet2(a[3], a[7], a[4], a[6]);
  return cfma(a[2], t2, cfma(a[1], t1, cm(a[0], t0)));
}

// P(X): scaled Newton polar iteration, then the determinant's phase removed.
// One step is N = (g Y + (g Y)^-dag) / 2 = h Y + conj(C e) with C the cofactor
// matrix of Y ((Y^-1)^dag = conj(C / det Y)), h = g / 2 and e = s conj(det Y),
// s = 1 / (2 g |det Y|^2).  For Y = Q H (polar form) any positive g and s give
// N = Q (g H + c H^-1) / 2, the same Q: the scaled steps take g ~ |det Y|^(-1/3)
// and s = g^5 / 2 from FP32 arithmetic; the unscaled steps (g = 1) need s to
// FP64 accuracy, since with c != 1 the iterates would converge to sqrt(c) Q.
// Scaling while a step still changes Y by more than 1 % (relative); the
// iteration stops after an unscaled step that changed it by less than 1e-8:
// near the fixed point such a step leaves an error of about half its square
// (~5e-17, FP64 rounding).  The singular values of every iterate are >= 1
// (those of (g H + c H^-1) / 2 are >= sqrt(g c), = 1 unscaled), so |N|_F^2 >= 3
// and testing the squared step against 3 x (relative bound)^2 is never looser.
__device__ M3 project_su3(const M3 &X) {
  M3 Y = X;
  bool scaled = true;
  for (int it = 0; it < 60; ++it) {
    double2 C[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int r0 = (i + 1) % 3, r1 = (i + 2) % 3, c0 = (j + 1) % 3, c1 = (j + 2) % 3;
        C[i * 3 + j] = cdet2(Y.a[r0 * 3 + c0], Y.a[r1 * 3 + c1], Y.a[r0 * 3 + c1], Y.a[r1 * 3 + c0]);
      }
    const double2 d = cfma(Y.a[2], C[2], cfma(Y.a[1], C[1], cm(Y.a[0], C[0])));
    const double dd = __fma_rn(d.x, d.x, d.y * d.y);
    double h, sc;
    if (scaled) {
      // g = |det Y|^(-1/3) = dd^(-1/6)
      const double g = (dd > 1e-30 && dd < 1e30) ? (double)sqrtf(rcbrtf((float)dd)) : sqrt(rcbrt(dd));
      const double g2 = g * g;
      h = 0.5 * g;
      sc = 0.5 * (g2 * g2 * g);
    } else {
      h = 0.5;
      sc = 0.5 / dd;
    }
    const double2 e = make_double2(sc * d.x, -sc * d.y);
    double diff = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double2 c = C[k], y = Y.a[k];
      const double2 n = make_double2(__fma_rn(c.x, e.x, __fma_rn(-c.y, e.y, h * y.x)),
                                     __fma_rn(-c.x, e.y, __fma_rn(-c.y, e.x, h * y.y)));
      const double ex = n.x - y.x, ey = n.y - y.y;
      diff = __fma_rn(ex, ex, __fma_rn(ey, ey, diff));
      Y.a[k] = n;
    }
    if (!scaled && diff <= 3e-16) break;
    if (diff <= 3e-4) scaled = false;
  }
  // z = exp(-i arg(det Y) / 3), principal branch: an FP32 estimate (the branch
  // follows the sign of Im det, kept by the conversion), then two Newton steps
  // on z^3 det Y = 1 in FP64, z <- z (4 - z^3 det Y) / 3 (the residual
  // w - 1 becomes -(2/3)(w - 1)^2 + O((w - 1)^3): 1e-7 -> 1e-14 -> rounding)
  const double2 d = det3(Y);
  float sf, cf;
  sincosf(atan2f((float)d.y, (float)d.x) / 3.0f, &sf, &cf);
  double2 z = make_double2((double)cf, -(double)sf);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double2 w = cm(cm(cm(z, z), z), d);
    z = cm(z, make_double2((4.0 - w.x) * (1.0 / 3.0), -w.y * (1.0 / 3.0)));
  }
  M3 W;
#pragma unroll
  for (int k = 0; k < 9; ++k) W.a[k] = cm(Y.a[k], z);
  return W;
}

struct Lat {
  int L[4];
  long long V;
};

__device__ __forceinline__ void coords(const Lat &g, long long i, int (&x)[4]) {
  x[0] = (int)(i % g.L[0]);
  i /= g.L[0];
  x[1] = (int)(i % g.L[1]);
  i /= g.L[1];
  x[2] = (int)(i % g.L[2]);
  x[3] = (int)(i / g.L[2]);
}

__device__ __forceinline__ long long lexs(const Lat &g, const int (&x)[4], int d, int s, int d2 = -1, int s2 = 0) {
  int y[4] = {x[0], x[1], x[2], x[3]};
  y[d] = (y[d] + s + g.L[d]) % g.L[d];
  if (d2 >= 0) y[d2] = (y[d2] + s2 + g.L[d2]) % g.L[d2];
  return y[0] + (long long)g.L[0] * (y[1] + (long long)g.L[1] * (y[2] + (long long)g.L[2] * y[3]));
}

// slot of the decorated link (dir, deco != dir) among the 12 stored: [dir][3]
__device__ __forceinline__ int dslot(int dir, int deco) { return dir * 3 + (deco < dir ? deco : deco - 1); }

// a field of links: thin (deco < 0: [dir][V]) or decorated ([12][V], slot dslot(dir, deco))
struct Fld {
  const double2 *p;
  long long V;
  __device__ __forceinline__ const double2 *at(int dir, int deco, long long site) const {
    return deco < 0 ? p + ((long long)dir * V + site) * 9 : p + ((long long)dslot(dir, deco) * V + site) * 9;
  }
};

// acc += the two staples in direction d of the link (x, mu): side links of
// field A with decoration da, middle link of field B with decoration db
__device__ __forceinline__ void staples(const Lat &g, const int (&x)[4], long long i, int mu, int d, const Fld &A,
                                        int da, const Fld &B, int db, M3 &acc) {
  // + d: A_d(x) B_mu(x+d) A_d(x+mu)^dag
  {
    const M3 a = ld(A.at(d, da, i));
    const M3 b = ld(B.at(mu, db, lexs(g, x, d, 1)));
    const M3 c = ld(A.at(d, da, lexs(g, x, mu, 1)));
    const M3 t = mul<false, false>(a, b);
    mul_add<false, true>(t, c, acc);
  }
  // - d: A_d(x-d)^dag B_mu(x-d) A_d(x-d+mu)
  {
    const long long xm = lexs(g, x, d, -1);
    const M3 a = ld(A.at(d, da, xm));
    const M3 b = ld(B.at(mu, db, xm));
    const M3 c = ld(A.at(d, da, lexs(g, x, d, -1, mu, 1)));
    const M3 t = mul<true, false>(a, b);
    mul_add<false, false>(t, c, acc);
  }
}

__device__ __forceinline__ void smear_store(const double2 *u, double a, double w, const M3 &acc, double2 *out) {
  M3 X;
#pragma unroll
  for (int k = 0; k < 9; ++k) X.a[k] = make_double2((1.0 - a) * u[k].x + w * acc.a[k].x, (1.0 - a) * u[k].y + w * acc.a[k].y);
  const M3 W = project_su3(X);
#pragma unroll
  for (int k = 0; k < 9; ++k) out[k] = W.a[k];
}

// The FP64 levels.  run != nullptr: only for a field that the fixed-point
// levels left alone.
// level 1: thread over (mu, e != mu, site); Vb stored [dslot(mu, e)][V]
__global__ void k_hyp1(Lat g, const FieldCheck *run, const double2 *U, double a3, double2 *Vb) {
  if (run != nullptr && fx_field(*run, 4 * g.V)) return;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 12 * g.V) return;
  const long long i = t % g.V;
  const int pr = (int)(t / g.V), mu = pr / 3, e = (pr % 3 >= mu) ? pr % 3 + 1 : pr % 3;
  int x[4];
  coords(g, i, x);
  const Fld thin{U, g.V};
  M3 acc;
#pragma unroll
  for (int k = 0; k < 9; ++k) acc.a[k] = make_double2(0.0, 0.0);
  staples(g, x, i, mu, e, thin, -1, thin, -1, acc);
  smear_store(thin.at(mu, -1, i), a3, a3 / 2.0, acc, Vb + ((long long)dslot(mu, e) * g.V + i) * 9);
}

// level 2: thread over (mu, nu != mu, site); Vt stored [dslot(mu, nu)][V]
__global__ void k_hyp2(Lat g, const FieldCheck *run, const double2 *U, const double2 *Vb, double a2, double2 *Vt) {
  if (run != nullptr && fx_field(*run, 4 * g.V)) return;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 12 * g.V) return;
  const long long i = t % g.V;
  const int pr = (int)(t / g.V), mu = pr / 3, nu = (pr % 3 >= mu) ? pr % 3 + 1 : pr % 3;
  int x[4];
  coords(g, i, x);
  const Fld vb{Vb, g.V};
  M3 acc;
#pragma unroll
  for (int k = 0; k < 9; ++k) acc.a[k] = make_double2(0.0, 0.0);
  for (int r = 0; r < 4; ++r) {
    if (r == mu || r == nu) continue;
    const int s = 6 - mu - nu - r;  // the direction outside {mu, nu, r}
    staples(g, x, i, mu, r, vb, s, vb, s, acc);
  }
  smear_store(U + ((long long)mu * g.V + i) * 9, a2, a2 / 4.0, acc, Vt + ((long long)dslot(mu, nu) * g.V + i) * 9);
}

// level 3: thread over (mu, site); out may alias U (each thread reads only its own thin link)
__global__ void k_hyp3(Lat g, const FieldCheck *run, const double2 *U, const double2 *Vt, double a1, double2 *out) {
  if (run != nullptr && fx_field(*run, 4 * g.V)) return;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * g.V) return;
  const long long i = t % g.V;
  const int mu = (int)(t / g.V);
  int x[4];
  coords(g, i, x);
  const Fld vt{Vt, g.V};
  M3 acc;
#pragma unroll
  for (int k = 0; k < 9; ++k) acc.a[k] = make_double2(0.0, 0.0);
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    // sides Vt(., nu; mu), middle Vt(., mu; nu)
    // + nu
    {
      const M3 a = ld(vt.at(nu, mu, i));
      const M3 b = ld(vt.at(mu, nu, lexs(g, x, nu, 1)));
      const M3 c = ld(vt.at(nu, mu, lexs(g, x, mu, 1)));
      mul_add<false, true>(mul<false, false>(a, b), c, acc);
    }
    // - nu
    {
      const long long xm = lexs(g, x, nu, -1);
      const M3 a = ld(vt.at(nu, mu, xm));
      const M3 b = ld(vt.at(mu, nu, xm));
      const M3 c = ld(vt.at(nu, mu, lexs(g, x, nu, -1, mu, 1)));
      mul_add<false, false>(mul<true, false>(a, b), c, acc);
    }
  }
  double2 u[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) u[k] = U[((long long)mu * g.V + i) * 9 + k];
  smear_store(u, a1, a1 / 6.0, acc, out + ((long long)mu * g.V + i) * 9);
}

// ---------------------------------------------------------------------------
// the same three levels on the integer pipe (fields that pass fx_field)
// ---------------------------------------------------------------------------
// The FP64 levels keep the FP64 pipe 95 % busy: per site 20 700 FMAs of staples
// and 33 600 of projections (44.8 ms at 20^3 x 64).  Here the staples are
// fixed-point products (fixed.cuh; decorated links are SU(3), the thin ones within
// 1e-3 of unitary, so products stay below 2) and the projection is
// project_su3_fx.  The sum to project is formed as c U + (staples) 2^-q with
// c = 2^-q (1 - a) / w and 2^q >= (1 - a) / w + number of staples: P ignores a
// positive scale.  Fields lie as [slot][element][site] int4, so that a warp's
// 32 sites are 512 contiguous bytes a load.  A thread whose projection does not
// converge (a sum near singular) projects in FP64; where that has no result
// either, levels 1 and 2 mark the field as bad, and the FP64 levels run, as on
// a field whose conversion did not pass fx_field (links that mix too little keep
// small elements, which fixed-point numbers hold to 2^-58 only).
struct FLat {
  Lat g;
  FastDiv d0, d1, d2;
};

__device__ __forceinline__ void coords_fx(const FLat &f, unsigned i, int (&x)[4]) {
  const unsigned q1 = fast_div(i, f.d0), q2 = fast_div(q1, f.d1), q3 = fast_div(q2, f.d2);
  x[0] = (int)(i - q1 * f.g.L[0]);
  x[1] = (int)(q1 - q2 * f.g.L[1]);
  x[2] = (int)(q2 - q3 * f.g.L[2]);
  x[3] = (int)q3;
}

// the site one step s = +-1 from site i (coordinate xd) in direction d
__device__ __forceinline__ unsigned step_fx(const FLat &f, unsigned i, int xd, int d, int s) {
  const unsigned str = d == 0 ? 1u : d == 1 ? (unsigned)f.g.L[0]
                                 : d == 2 ? (unsigned)(f.g.L[0] * f.g.L[1])
                                          : (unsigned)(f.g.L[0] * f.g.L[1] * f.g.L[2]);
  const int L = f.g.L[d];
  const int k = s > 0 ? (xd + 1 == L ? 1 - L : 1) : (xd == 0 ? L - 1 : -1);
  return i + (unsigned)(k * (int)str);
}

constexpr int HFX_BT = 128;

// two 64-bit integers in the four words of an int4
__device__ __forceinline__ long long lo64(const int4 &v) { return ((long long)v.y << 32) | (unsigned)v.x; }
__device__ __forceinline__ long long hi64(const int4 &v) { return ((long long)v.w << 32) | (unsigned)v.z; }
__device__ __forceinline__ int4 pack64(long long a, long long b) {
  return make_int4((int)a, (int)(a >> 32), (int)b, (int)(b >> 32));
}

// X (unit 2^-58, pairs of 64-bit sums, one column of shared memory a thread: element k at X[k HFX_BT])
// += a b c^dag (neg = 0) or a^dag b c (neg = 1); each factor at p + element V.
// One body serves both: the daggers are strides and signs.
__device__ __forceinline__ void staple_fx(const int4 *pa, const int4 *pb, const int4 *pc, int V, int neg, int4 *X) {
  int4 b[9], c[9], a[3], an[3];
  const int ra = neg ? V : 3 * V, ca = neg ? 3 * V : V;  // row i of (a or a^dag): i ra + k ca
  const int rc = neg ? 3 * V : V, cc = neg ? V : 3 * V;  // element (k, j) of (c^dag or c): k rc + j cc
  const int sa = neg ? -1 : 1, sc = -sa;
#pragma unroll
  for (int k = 0; k < 3; ++k) a[k] = __ldg(pa + k * ca);
#pragma unroll
  for (int k = 0; k < 9; ++k) b[k] = __ldg(pb + k * V);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    c[k] = __ldg(pc + (k / 3) * rc + (k % 3) * cc);
    c[k].z *= sc;
    c[k].w *= sc;
  }
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    const int nx = i < 2 ? (i + 1) * ra : 0;  // the next row, in flight while this one is computed
#pragma unroll
    for (int k = 0; k < 3; ++k) an[k] = __ldg(pa + nx + k * ca);
    int4 t[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[k].z *= sa;
      a[k].w *= sa;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      CAcc s = cacc_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmac(s, a[k], b[3 * k + j]);
      t[j] = fx_cval(s);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      CAcc s = cacc_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmac(s, t[k], c[3 * k + j]);
      const int4 x = X[(3 * i + j) * HFX_BT];
      X[(3 * i + j) * HFX_BT] = pack64(lo64(x) + fx_sum(s.re), hi64(x) + fx_sum(s.im));
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) a[k] = an[k];
  }
}

// P(X) in FP64 where the fixed-point projection gave up; false: no finite result
__device__ __noinline__ bool project_fallback(const int4 *X, int4 *W) {
  M3 x;
  for (int k = 0; k < 9; ++k) {
    const int4 v = X[k * HFX_BT];
    x.a[k] = make_double2((double)fx_join(v.x, v.y) * 0x1p-58, (double)fx_join(v.z, v.w) * 0x1p-58);
  }
  const M3 w = project_su3(x);
  bool ok = true;
  for (int k = 0; k < 9; ++k) {
    ok = ok && fabs(w.a[k].x) < 1.5 && fabs(w.a[k].y) < 1.5;
    W[k * HFX_BT] = fx_pair(__double2ll_rn(w.a[k].x * 0x1p58), __double2ll_rn(w.a[k].y * 0x1p58));
  }
  return ok;
}

struct HfxShared {
  int4 X[9][HFX_BT];   // the staple sums (64-bit), then the matrix to project
  int4 Q[9][HFX_BT];   // its projection
  float f[27][HFX_BT];
};

// a thin link's element in fixed point
__device__ __forceinline__ int4 thin_fx(const double2 &w) {
  const Fx a = fx_link(__double2hiint(w.x), __double2loint(w.x)), b = fx_link(__double2hiint(w.y), __double2loint(w.y));
  return make_int4(a.h, a.l, b.h, b.l);
}

// the mix of c U (U(k): its element k) and the staples in X, and its projection into Q; c = (h, l) limbs
template <class Thin>
__device__ __forceinline__ bool smear_fx(const Thin &U, Fx c, int q, int4 *X, int4 *Q, float *f) {
  const long long half = q > 0 ? 1ll << (q - 1) : 0ll;
#pragma unroll 3
  for (int k = 0; k < 9; ++k) {
    const int4 u = U(k);
    FxAcc re, im;
    re.hh = re.cr = im.hh = im.cr = 0;
    fx_mac(re, u.x, u.y, c.h, c.l);
    fx_mac(im, u.z, u.w, c.h, c.l);
    const int4 s = X[k * HFX_BT];
    X[k * HFX_BT] = fx_pair(fx_sum(re) + ((lo64(s) + half) >> q), fx_sum(im) + ((hi64(s) + half) >> q));
  }
  if (project_su3_fx<HFX_BT>(X, Q, f)) return true;
  return project_fallback(X, Q);
}

// canonical FP64 links -> [mu][9][V] fixed-point, and the check of the field
__global__ void __launch_bounds__(256) k_hyp_fix(long long V, const double2 *__restrict__ U, int4 *F, FieldCheck *check) {
  const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
  bool ok = true;
  int nsmall = 0;
  if (t < 4 * V) {
    const long long mu = t / V, i = t - mu * V;
    float2 u[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) {
      const double2 w = U[t * 9 + e];
      const int hx = __double2hiint(w.x), hy = __double2hiint(w.y);
      ok = ok && (hx & 0x7fffffff) < 0x40000000 && (hy & 0x7fffffff) < 0x40000000;
      const int4 v = thin_fx(w);
      F[(mu * 9 + e) * V + i] = v;
      u[e] = make_float2((float)v.x * 0x1p-29f, (float)v.z * 0x1p-29f);
    }
    ok = ok && near_unitary(u);
    nsmall = small_parts(u);
  }
  check_link(check, ok, nsmall);
}

struct HypFx {
  FLat f;
  long long V;
  const double2 *U;  // the thin links, canonical
  FieldCheck *check;
  Fx c;
  int q;
};

// whether a level leaves the field alone; other blocks of it may be marking the
// field, so the block's threads decide together (whole warps project together)
__device__ __forceinline__ bool hyp_off(const HypFx &h) {
  bool off = false;
  if (threadIdx.x == 0) {
    FieldCheck f;
    f.small = h.check->small;
    f.bad = *(volatile int *)&h.check->bad;
    off = !fx_field(f, 4 * h.V);
  }
  return __syncthreads_or(off) != 0;
}

// level 1 (LEVEL = 1: Vb from U) and level 2 (Vt from Vb); blockIdx.y = slot
template <int LEVEL>
__global__ void __launch_bounds__(HFX_BT, 3) k_hyp12_fx(const HypFx h, const int4 *__restrict__ src, int4 *dst) {
  if (hyp_off(h)) return;
  // threads past the last site repeat it (whole warps project together) and store nothing
  const unsigned i0 = blockIdx.x * HFX_BT + threadIdx.x, i = i0 < h.V ? i0 : (unsigned)h.V - 1;
  const int pr = blockIdx.y, mu = pr / 3, e = (pr % 3 >= mu) ? pr % 3 + 1 : pr % 3;
  const long long V = h.V;
  int x[4];
  coords_fx(h.f, i, x);
  const int xmu = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
  const unsigned imu = step_fx(h.f, i, xmu, mu, 1);
  extern __shared__ HfxShared hsh[];
  int4 *X = &hsh->X[0][threadIdx.x], *Q = &hsh->Q[0][threadIdx.x];
#pragma unroll
  for (int k = 0; k < 9; ++k) X[k * HFX_BT] = make_int4(0, 0, 0, 0);
#pragma unroll 1
  for (int d = 0; d < 4; ++d) {
    if (LEVEL == 1 ? d != e : (d == mu || d == e)) continue;
    const int s = 6 - mu - e - d;  // level 2: the direction outside {mu, nu, d}
    const int4 *A = src + (LEVEL == 1 ? d : dslot(d, s)) * 9 * V;
    const int4 *B = src + (LEVEL == 1 ? mu : dslot(mu, s)) * 9 * V;
    const int xd = d == 0 ? x[0] : d == 1 ? x[1] : d == 2 ? x[2] : x[3];
    const unsigned up = step_fx(h.f, i, xd, d, 1), dn = step_fx(h.f, i, xd, d, -1), dnmu = step_fx(h.f, imu, xd, d, -1);
#pragma unroll 1
    for (int neg = 0; neg < 2; ++neg)
      staple_fx(A + (neg ? dn : i), B + (neg ? dn : up), A + (neg ? dnmu : imu), (int)V, neg, X);
  }
  // level 1 reads the thin links in fixed point anyway (src)
  const int4 *pf = src + (long long)mu * 9 * V + i;
  const double2 *pu = h.U + ((long long)mu * V + i) * 9;
  auto thin = [&](int k) { return LEVEL == 1 ? __ldg(pf + k * V) : thin_fx(__ldg(pu + k)); };
  if (!smear_fx(thin, h.c, h.q, X, Q, &hsh->f[0][threadIdx.x])) h.check->bad = 1;
  if (i0 >= h.V) return;
#pragma unroll
  for (int k = 0; k < 9; ++k) dst[((long long)pr * 9 + k) * V + i] = Q[k * HFX_BT];
}

// level 3 (the smeared links, FP64 ABI layout; may be the buffer U came from); blockIdx.y = mu
__global__ void __launch_bounds__(HFX_BT, 3) k_hyp3_fx(const HypFx h, const int4 *__restrict__ Vt, double2 *out) {
  if (hyp_off(h)) return;
  const unsigned i0 = blockIdx.x * HFX_BT + threadIdx.x, i = i0 < h.V ? i0 : (unsigned)h.V - 1;
  const int mu = blockIdx.y;
  const long long V = h.V;
  int x[4];
  coords_fx(h.f, i, x);
  const int xmu = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
  const unsigned imu = step_fx(h.f, i, xmu, mu, 1);
  extern __shared__ HfxShared hsh[];
  int4 *X = &hsh->X[0][threadIdx.x], *Q = &hsh->Q[0][threadIdx.x];
#pragma unroll
  for (int k = 0; k < 9; ++k) X[k * HFX_BT] = make_int4(0, 0, 0, 0);
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    const int4 *A = Vt + dslot(nu, mu) * 9 * V, *B = Vt + dslot(mu, nu) * 9 * V;
    const int xn = nu == 0 ? x[0] : nu == 1 ? x[1] : nu == 2 ? x[2] : x[3];
    const unsigned up = step_fx(h.f, i, xn, nu, 1), dn = step_fx(h.f, i, xn, nu, -1), dnmu = step_fx(h.f, imu, xn, nu, -1);
#pragma unroll 1
    for (int neg = 0; neg < 2; ++neg)
      staple_fx(A + (neg ? dn : i), B + (neg ? dn : up), A + (neg ? dnmu : imu), (int)V, neg, X);
  }
  // out may be the thin links' buffer: each thread reads its own link before it
  // writes it, and those past the last site, whose link another thread writes, read none
  const double2 *pu = h.U + ((long long)mu * V + i) * 9;
  auto thin = [&](int k) { return i0 < V ? thin_fx(pu[k]) : make_int4(k % 4 == 0 ? 1 << FX_LO : 0, 0, 0, 0); };
  const bool ok = smear_fx(thin, h.c, h.q, X, Q, &hsh->f[0][threadIdx.x]);
  if (i0 >= h.V) return;
  const double one = ok ? 0x1p-58 : __longlong_as_double(0x7ff8000000000000ll);
  double2 *o = out + ((long long)mu * V + i) * 9;
#pragma unroll 3
  for (int k = 0; k < 9; ++k) {
    const int4 w = Q[k * HFX_BT];
    o[k] = make_double2((double)fx_join(w.x, w.y) * one, (double)fx_join(w.z, w.w) * one);
  }
}

// coefficient and shift of a level; false where the fixed-point mix does not hold it
bool mix_of(double a, double w, int staples, Fx *c, int *q) {
  if (!(a > 0.0) || !(a <= 1.0)) return false;
  const double r = (1.0 - a) / w;
  if (!(r <= 60.0)) return false;
  *q = 0;
  while ((double)(1 << *q) < r + staples) ++*q;
  const long long C = llrint(ldexp(r, 58 - *q));
  *c = fx_split(C);
  return true;
}

}  // namespace

cudaError_t launch_hyp(const int dims[4], const double2 *U, const double alpha[3], double2 *Vb, double2 *Vt,
                       double2 *out, FieldCheck *check, cudaStream_t st) {
  Lat g;
  for (int k = 0; k < 4; ++k) g.L[k] = dims[k];
  g.V = (long long)dims[0] * dims[1] * dims[2] * dims[3];
  const int bt = 128;
  Fx c[3];
  int q[3];
  cudaError_t e = cudaSuccess;
  const FieldCheck *run = nullptr;
  if (check != nullptr && g.V < (1ll << 27) && mix_of(alpha[2], alpha[2] / 2.0, 2, &c[0], &q[0]) &&
      mix_of(alpha[1], alpha[1] / 4.0, 4, &c[1], &q[1]) && mix_of(alpha[0], alpha[0] / 6.0, 6, &c[2], &q[2])) {
    for (const void *k : {(const void *)k_hyp12_fx<1>, (const void *)k_hyp12_fx<2>, (const void *)k_hyp3_fx}) {
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(HfxShared));
      if (e != cudaSuccess) return e;
    }
    e = cudaMemsetAsync(check, 0, sizeof(FieldCheck), st);
    if (e != cudaSuccess) return e;
    run = check;
    HypFx h;
    h.f.g = g;
    h.f.d0 = make_fastdiv((unsigned)dims[0]);
    h.f.d1 = make_fastdiv((unsigned)dims[1]);
    h.f.d2 = make_fastdiv((unsigned)dims[2]);
    h.V = g.V;
    h.U = U;
    int4 *fixU = reinterpret_cast<int4 *>(Vt);  // level 1's thin links, until level 2 writes Vt
    h.check = check;
    k_hyp_fix<<<(unsigned)((4 * g.V + 255) / 256), 256, 0, st>>>(g.V, U, fixU, check);
    const unsigned nb = (unsigned)((g.V + HFX_BT - 1) / HFX_BT);
    h.c = c[0];
    h.q = q[0];
    k_hyp12_fx<1><<<dim3(nb, 12), HFX_BT, sizeof(HfxShared), st>>>(h, fixU, reinterpret_cast<int4 *>(Vb));
    h.c = c[1];
    h.q = q[1];
    k_hyp12_fx<2><<<dim3(nb, 12), HFX_BT, sizeof(HfxShared), st>>>(h, reinterpret_cast<const int4 *>(Vb), reinterpret_cast<int4 *>(Vt));
    h.c = c[2];
    h.q = q[2];
    k_hyp3_fx<<<dim3(nb, 4), HFX_BT, sizeof(HfxShared), st>>>(h, reinterpret_cast<const int4 *>(Vt), out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  k_hyp1<<<(unsigned)((12 * g.V + bt - 1) / bt), bt, 0, st>>>(g, run, U, alpha[2], Vb);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_hyp2<<<(unsigned)((12 * g.V + bt - 1) / bt), bt, 0, st>>>(g, run, U, Vb, alpha[1], Vt);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_hyp3<<<(unsigned)((4 * g.V + bt - 1) / bt), bt, 0, st>>>(g, run, U, Vt, alpha[0], out);
  return cudaGetLastError();
}

}  // namespace stag
