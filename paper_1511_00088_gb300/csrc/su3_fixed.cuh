// su3_fixed.cuh -- the projection of a 3 x 3 matrix to SU(3) in fixed-point and
// FP32 arithmetic, to FP64 accuracy (used by hyp.cu).
//
//   1. the unitary polar factor Q by scaled Newton steps in FP32 (~1e-6);
//   2. corrections Q <- Q (1 + D) from residuals in fixed point: with M = Q^dag X,
//      E = Q^dag Q - 1, the exact factor has D = Ds + Da to first order,
//        Ds = -E / 2,   H Da + Da H = (M - M^dag) + Ds H - H Ds,   H = (M + M^dag) / 2,
//      solved in FP32 (each correction gains the factor that this is accurate to),
//      until a correction leaves too little to matter;
//   3. the phase of det Q: z = z0 (1 - e/3 + 2 e^2/9), z0 ~ det^(-1/3) from
//      FP32, e = z0^3 det - 1 in fixed point.
// Everything that decides the result's last bits is an integer sum (unit 2^-58),
// everything that only has to be near is FP32: none of it needs GB300's FP64
// pipe, which took 1200 FMAs a projection (19 000 clocks a warp).
#pragma once

#include "fixed.cuh"

namespace stag {

// Each correction leaves the fraction of itself that its FP32 solution is off by:
// 1e-6 for well-conditioned matrices, up to 1e-2 at condition numbers of some
// hundreds.  The fraction is seen in how much smaller a correction m is than the
// one before, so the last is the first with m (m / previous m) below FX_LEFT.  (A
// line for m alone, 2^-34, stopped after the second correction whatever the
// condition: at a condition number of 300 errors of 4e-13, where the FP64 form has 1e-14.)
// Measured on the CPU (elements against 113-bit arithmetic, 1500 matrices a condition
// number, median / largest; the FP64 form): 4: 6e-18 / 1e-17 (1e-16 / 3e-16),
// 30: 2e-17 / 3e-16 (2e-16 / 7e-16), 100: 4e-17 / 2e-15 (4e-16 / 3e-15), 300: 1e-16 / 8e-16
// (1e-15 / 1e-14), with the singular values spread evenly; from some hundreds on an
// increasing part does not converge in five corrections and is left to FP64.
// Two corrections, or three from condition numbers near 10 on.
constexpr float FX_LEFT = 0x1p-56f;

struct C3 {  // FP32 3 x 3
  float2 a[9];
};
// A fixed-point 3 x 3 matrix (unit 2^-58, int4 limbs of the real and imaginary
// parts) lies in memory as 9 elements a stride apart, one column of shared
// memory a thread, so that loops over its rows stay loops: unrolled, the code
// outgrew the instruction caches (half of all stalls waited for instructions).

FX_HD float2 c_mul(float2 x, float2 y) { return make_float2(x.x * y.x - x.y * y.y, x.x * y.y + x.y * y.x); }
FX_HD float2 c_fma(float2 x, float2 y, float2 s) {
  return make_float2(fmaf(-x.y, y.y, fmaf(x.x, y.x, s.x)), fmaf(x.y, y.x, fmaf(x.x, y.y, s.y)));
}
FX_HD float2 c_conj(float2 x) { return make_float2(x.x, -x.y); }
FX_HD C3 c3_mul(const C3 &x, const C3 &y) {
  C3 r;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      r.a[3 * i + j] = c_fma(x.a[3 * i + 2], y.a[6 + j], c_fma(x.a[3 * i + 1], y.a[3 + j], c_mul(x.a[3 * i], y.a[j])));
  return r;
}
// T (unit 2^-58) as FP32
FX_HD float fx_float(long long T) {
  const Fx f = fx_split(T);
  return fmaf((float)f.l, 0x1p-58f, (float)f.h * 0x1p-29f);
}
FX_HD int4 fx_pair(long long re, long long im) {
  const Fx a = fx_split(re), b = fx_split(im);
  return make_int4(a.h, a.l, b.h, b.l);
}
// v / 3, rounded down
FX_HD long long fx_third(long long v) {
#ifdef __CUDA_ARCH__
  return __mul64hi(v, 0x5555555555555556ll);
#else
  return (long long)(((__int128)v * 0x5555555555555556ll) >> 64);
#endif
}
FX_HD long long fx_join(int h, int l) { return ((long long)h << FX_LO) + l; }
FX_HD int4 fx_conj(const int4 &x) { return make_int4(x.x, x.y, -x.z, -x.w); }

struct CAcc {  // complex sum of products
  FxAcc re, im;
};
FX_HD CAcc cacc_zero() {
  CAcc s;
  s.re.hh = s.re.cr = s.im.hh = s.im.cr = 0;
  return s;
}
// s += x y
FX_HD void fx_cmac(CAcc &s, const int4 &x, const int4 &y) {
  fx_mac(s.re, x.x, x.y, y.x, y.y);
  fx_mac(s.re, x.z, x.w, -y.z, -y.w);
  fx_mac(s.im, x.x, x.y, y.z, y.w);
  fx_mac(s.im, x.z, x.w, y.x, y.y);
}
// s += conj(x) y
FX_HD void fx_cmac_c(CAcc &s, const int4 &x, const int4 &y) {
  fx_mac(s.re, x.x, x.y, y.x, y.y);
  fx_mac(s.re, x.z, x.w, y.z, y.w);
  fx_mac(s.im, x.x, x.y, y.z, y.w);
  fx_mac(s.im, x.z, x.w, -y.x, -y.y);
}
// s += x conj(y)
FX_HD void fx_cmac_d(CAcc &s, const int4 &x, const int4 &y) {
  fx_mac(s.re, x.x, x.y, y.x, y.y);
  fx_mac(s.re, x.z, x.w, y.z, y.w);
  fx_mac(s.im, x.x, x.y, -y.z, -y.w);
  fx_mac(s.im, x.z, x.w, y.x, y.y);
}
FX_HD int4 fx_cval(const CAcc &s) { return fx_pair(fx_sum(s.re), fx_sum(s.im)); }

// Unitary polar factor of x in FP32: Newton steps N = (g Y + (g Y)^-dag) / 2
// scaled by g ~ |det Y|^(-1/3) until Y is near unitary, then unscaled until a
// step changes it by less than 2e-5; false where the matrix is too singular.
// (A warp's 32 lanes call this and project_su3_fx together and leave every loop
// together, by a vote; a lane that is done takes harmless further steps.  Left to
// the lanes' own exits, the loops did not reconverge, and all that follows ran
// once a group of lanes: 7150 instead of 3860 clocks a warp.)
FX_HD bool any_lane(bool v) {
#ifdef __CUDA_ARCH__
  return __any_sync(0xffffffffu, v);
#else
  return v;
#endif
}
FX_HD bool polar32(C3 &y) {
  bool scaled = true, good = true, done = false;
#pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    float2 C[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int r0 = (i + 1) % 3, r1 = (i + 2) % 3, c0 = (j + 1) % 3, c1 = (j + 2) % 3;
        const float2 p = y.a[r0 * 3 + c0], q = y.a[r1 * 3 + c1], u = y.a[r0 * 3 + c1], v = y.a[r1 * 3 + c0];
        C[i * 3 + j] = c_fma(p, q, make_float2(u.y * v.y - u.x * v.x, -(u.x * v.y + u.y * v.x)));
      }
    const float2 d = c_fma(y.a[2], C[2], c_fma(y.a[1], C[1], c_mul(y.a[0], C[0])));
    const float dd = d.x * d.x + d.y * d.y;
    good = good && dd > 1e-16f && dd < 1e16f;
    float h = 0.5f, sc = 0.5f / dd;
    if (scaled) {
      const float g = exp2f(log2f(dd) * (-1.f / 6.f));
      h = 0.5f * g;
      sc /= g;
    }
    const float2 e = make_float2(sc * d.x, -sc * d.y);
    float diff = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const float2 n = make_float2(fmaf(C[k].x, e.x, fmaf(-C[k].y, e.y, h * y.a[k].x)),
                                   fmaf(-C[k].x, e.y, fmaf(-C[k].y, e.x, h * y.a[k].y)));
      const float dx = n.x - y.a[k].x, dy = n.y - y.a[k].y;
      diff = fmaf(dx, dx, fmaf(dy, dy, diff));
      y.a[k] = n;
    }
    done = done || (!scaled && diff <= 1e-9f);
    if (diff <= 3e-3f) scaled = false;
    if (!any_lane(good && !done)) break;
  }
  return good && done;
}

// X of H X + X H = R, H Hermitian positive, R anti-Hermitian, with D = 3 X / tr H
// returned for the H given (Hoger and Carlson, "On the derivative of the square
// root of a tensor and Guo's rate theorems", J. Elasticity 14, 1984): with
// A = 3 H / tr H and its invariants I1 = 3, I2, I3,
//   2 I3 (I1 I2 - I3) Y = I1 A^2 R A^2 - I1^2 (A^2 R A + A R A^2) + (I1 I2 - I3)(A^2 R + R A^2)
//     + (I1^3 + I3) A R A - I1^2 I2 (A R + R A) + (I1^2 I3 + (I1 I2 - I3) I2) R,
// X = Y 3 / tr H.  No difference of eigenvalues is divided by.  As R is
// anti-Hermitian, each pair is P - P^dag of its first product P.
FX_HD C3 sylvester32(const C3 &H, const C3 &R) {
  const float s = 3.f / (H.a[0].x + H.a[4].x + H.a[8].x);
  C3 A;
#pragma unroll
  for (int k = 0; k < 9; ++k) A.a[k] = make_float2(s * H.a[k].x, s * H.a[k].y);
  auto n2 = [](float2 v) { return v.x * v.x + v.y * v.y; };
  const float a = A.a[0].x, b = A.a[4].x, c = A.a[8].x;
  const float n01 = n2(A.a[1]), n02 = n2(A.a[2]), n12 = n2(A.a[5]);
  const float I1 = a + b + c, I2 = a * b + a * c + b * c - n01 - n02 - n12;
  const float2 t = c_mul(c_mul(A.a[1], A.a[5]), A.a[6]);
  const float I3 = a * b * c + 2.f * t.x - a * n12 - b * n02 - c * n01;
  const float J = I1 * I2 - I3;
  const C3 AR = c3_mul(A, R), AAR = c3_mul(A, AR);
  C3 Y;
  const float k0 = I1 * I1 * I3 + J * I2;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      // AR + R A = AR - (AR)^dag, A^2 R + R A^2 likewise
      const float2 p = AR.a[3 * i + j], q = AR.a[3 * j + i], u = AAR.a[3 * i + j], v = AAR.a[3 * j + i],
                   r = R.a[3 * i + j];
      const float c1 = -I1 * I1 * I2;
      Y.a[3 * i + j] = make_float2(k0 * r.x + c1 * (p.x - q.x) + J * (u.x - v.x),
                                   k0 * r.y + c1 * (p.y + q.y) + J * (u.y + v.y));
    }
  const C3 ARA = c3_mul(AR, A);
  const float k3 = I1 * I1 * I1 + I3;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    Y.a[k].x = fmaf(k3, ARA.a[k].x, Y.a[k].x);
    Y.a[k].y = fmaf(k3, ARA.a[k].y, Y.a[k].y);
  }
  const C3 AARA = c3_mul(AAR, A);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float2 p = AARA.a[3 * i + j], q = AARA.a[3 * j + i];
      Y.a[3 * i + j].x = fmaf(-I1 * I1, p.x - q.x, Y.a[3 * i + j].x);
      Y.a[3 * i + j].y = fmaf(-I1 * I1, p.y + q.y, Y.a[3 * i + j].y);
    }
  const C3 Z = c3_mul(AARA, A);
  const float f = s / (2.f * I3 * J);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    Y.a[k].x = f * fmaf(I1, Z.a[k].x, Y.a[k].x);
    Y.a[k].y = f * fmaf(I1, Z.a[k].y, Y.a[k].y);
  }
  return Y;
}

FX_HD int fx_round(float v) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(v);
#else
  return (int)rintf(v);
#endif
}

// Q (fixed) += Q D, D of size < m in FP32
template <int ST>
FX_HD void add_product(int4 *Q, const C3 &D, float m) {
  // Q D in units of 2^(sh - 58), below 2^30
  int e = 0;
#ifdef __CUDA_ARCH__
  e = ((__float_as_int(m) >> 23) & 0xff) - 126;  // m < 2^e
#else
  frexpf(m, &e);
#endif
  int sh = e + 58 + 3 - 30;
  sh = sh < 0 ? 0 : sh;
#ifdef __CUDA_ARCH__
  const float unit = __int_as_float((127 + 58 - sh) << 23);
#else
  const float unit = ldexpf(1.f, 58 - sh);
#endif
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    int4 o[3];
    float2 q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      o[k] = Q[(3 * i + k) * ST];
      q[k] = make_float2((float)o[k].x * 0x1p-29f, (float)o[k].z * 0x1p-29f);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float2 v = c_fma(q[2], D.a[6 + j], c_fma(q[1], D.a[3 + j], c_mul(q[0], D.a[j])));
      const int x = fx_round(v.x * unit), y = fx_round(v.y * unit);
      Q[(3 * i + j) * ST] = fx_pair(fx_join(o[j].x, o[j].y) + ((long long)x << sh), fx_join(o[j].z, o[j].w) + ((long long)y << sh));
    }
  }
}

// Q = P(X) for X of elements |.| <= 1 or little more (any positive scale of the
// matrix meant); false where the FP32 start or the corrections do not converge
// (X near singular): the caller then projects in FP64.  f: 27 floats of scratch.
// All 32 lanes of a warp call it together.
template <int ST>
FX_HD bool project_su3_fx(const int4 *X, int4 *Q, float *f) {
  bool good, done = false;
  float prev = 1.f;  // the correction before
  {
    C3 y;
#pragma unroll
    for (int k = 0; k < 9; ++k) y.a[k] = make_float2((float)X[k * ST].x * 0x1p-29f, (float)X[k * ST].z * 0x1p-29f);
    good = polar32(y);
#pragma unroll
    for (int k = 0; k < 9; ++k) Q[k * ST] = make_int4(fx_round(y.a[k].x * 0x1p29f), 0, fx_round(y.a[k].y * 0x1p29f), 0);
  }
#pragma unroll 1
  for (int it = 0; it < 5; ++it) {
    // E = Q^dag Q - 1 and M = Q^dag X, entry by entry on and above the diagonal:
    // f = Ds = -E / 2, the Hermitian part of M and twice its anti-Hermitian part
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
      const int i = p < 3 ? p : (p == 5 ? 1 : 0), j = p < 3 ? p : (p == 3 ? 1 : 2);
      CAcc e = cacc_zero(), m = cacc_zero(), n = cacc_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int4 qi = Q[(3 * k + i) * ST], qj = Q[(3 * k + j) * ST];
        fx_cmac_c(e, qi, qj);
        fx_cmac_c(m, qi, X[(3 * k + j) * ST]);
        fx_cmac_c(n, qj, X[(3 * k + i) * ST]);
      }
      const long long mr = fx_sum(m.re), mi = fx_sum(m.im), nr = fx_sum(n.re), ni = fx_sum(n.im);
      float *o = f + p * ST;  // re of Ds, H, R (p < 3: R imaginary), then (p >= 3) the imaginary parts
      o[0] = -0.5f * fx_float(fx_sum(e.re) - (p < 3 ? 1ll << 58 : 0ll));
      o[9 * ST] = 0.5f * (fx_float(mr) + fx_float(nr));
      if (p < 3) {
        o[18 * ST] = fx_float(mi + ni);
      } else {
        o[18 * ST] = fx_float(mr - nr);
        o[3 * ST] = -0.5f * fx_float(fx_sum(e.im));
        o[12 * ST] = 0.5f * (fx_float(mi) - fx_float(ni));
        o[21 * ST] = fx_float(mi + ni);
      }
    }
    C3 H, R, D;
#pragma unroll
    for (int p = 0; p < 6; ++p) {
      const int i = p < 3 ? p : (p == 5 ? 1 : 0), j = p < 3 ? p : (p == 3 ? 1 : 2);
      const float dr = f[p * ST], hr = f[(9 + p) * ST], rr = f[(18 + p) * ST];
      if (p < 3) {
        D.a[4 * i] = make_float2(dr, 0.f);
        H.a[4 * i] = make_float2(hr, 0.f);
        R.a[4 * i] = make_float2(0.f, rr);
      } else {
        const float di = f[(3 + p) * ST], hi = f[(12 + p) * ST], ri = f[(21 + p) * ST];
        D.a[3 * i + j] = make_float2(dr, di);
        D.a[3 * j + i] = make_float2(dr, -di);
        H.a[3 * i + j] = make_float2(hr, hi);
        H.a[3 * j + i] = make_float2(hr, -hi);
        R.a[3 * i + j] = make_float2(rr, ri);
        R.a[3 * j + i] = make_float2(-rr, ri);
      }
    }
    // R += Ds H - H Ds = P - P^dag, P = Ds H
    const C3 P = c3_mul(D, H);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        R.a[3 * i + j].x += P.a[3 * i + j].x - P.a[3 * j + i].x;
        R.a[3 * i + j].y += P.a[3 * i + j].y + P.a[3 * j + i].y;
      }
    const C3 Y = sylvester32(H, R);
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      D.a[k].x += Y.a[k].x;
      D.a[k].y += Y.a[k].y;
      m = fmaxf(m, fmaxf(fabsf(D.a[k].x), fabsf(D.a[k].y)));
    }
    good = good && m < 1e-2f;  // false for NaN
    add_product<ST>(Q, D, good ? m : 1e-2f);
    done = done || m * m < FX_LEFT * prev;
    prev = m;
    if (!any_lane(good && !done)) break;
  }
  // det Q = row 0 . (row 1 x row 2)
  CAcc det = cacc_zero();
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    const int j1 = j == 2 ? 0 : j + 1, j2 = j == 0 ? 2 : j - 1;
    CAcc s = cacc_zero();
    fx_cmac(s, Q[(3 + j1) * ST], Q[(6 + j2) * ST]);
    const int4 n = Q[(3 + j2) * ST];
    fx_cmac(s, make_int4(-n.x, -n.y, -n.z, -n.w), Q[(6 + j1) * ST]);
    fx_cmac(det, Q[j * ST], fx_cval(s));
  }
  const long long dr = fx_sum(det.re), di = fx_sum(det.im);
  // principal cube root: the branch follows the sign of Im det
  float sf, cf;
  const float th = atan2f(fx_float(di), fx_float(dr)) * (1.f / 3.f);
#ifdef __CUDA_ARCH__
  sincosf(th, &sf, &cf);
#else
  sf = sinf(th), cf = cosf(th);
#endif
  const int4 z0 = make_int4(fx_round(cf * 0x1p29f), 0, -fx_round(sf * 0x1p29f), 0);
  // e = z0^3 det - 1; z = z0 (1 - e/3 + 2 e^2/9)
  int4 z = fx_pair(dr, di);
#pragma unroll 1
  for (int k = 0; k < 3; ++k) {
    CAcc s = cacc_zero();
    fx_cmac(s, z, z0);
    z = fx_cval(s);
  }
  const long long er = fx_join(z.x, z.y) - (1ll << 58), ei = fx_join(z.z, z.w);
  const float fr = fx_float(er), fi = fx_float(ei);
  const long long qr = fx_round((2.f / 9.f) * (fr * fr - fi * fi) * 0x1p58f);
  const long long qi = fx_round((4.f / 9.f) * (fr * fi) * 0x1p58f);
  {
    CAcc s = cacc_zero();
    fx_cmac(s, z0, fx_pair((1ll << 58) - fx_third(er) + qr, qi - fx_third(ei)));
    z = fx_cval(s);
  }
#pragma unroll 1
  for (int k = 0; k < 9; ++k) {
    CAcc s = cacc_zero();
    fx_cmac(s, Q[k * ST], z);
    Q[k * ST] = fx_cval(s);
  }
  return good && done;
}

}  // namespace stag
