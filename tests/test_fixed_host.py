"""The fixed-point arithmetic (fixed.cuh, su3_fixed.cuh) compiled for the host: products, the field check and the
projection to SU(3) against exact and extended-precision arithmetic."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1511_00088_gb300 import build, synth

SOURCE = r"""
#include <cstring>
#include "su3_fixed.cuh"
using namespace stag;
static void bits(double v, int &hi, int &lo) { long long b; memcpy(&b, &v, 8); hi = (int)(b >> 32); lo = (int)b; }
extern "C" {
// T (6, unit 2^-57 of the scale 2^(E - 1022)) = u v, u 3 x 3 complex, v 3 complex; returns E
int host_product(const double *u, const double *v, long long *T) {
  int E = 0, hi, lo;
  for (int i = 0; i < 6; ++i) { bits(v[i], hi, lo); E = hi >> 20 & 0x7ff ? (E > (hi >> 20 & 0x7ff) ? E : hi >> 20 & 0x7ff) : E; }
  for (int i = 0; i < 3; ++i) {
    CAcc s = cacc_zero();
    for (int k = 0; k < 3; ++k) {
      int4 a, b;
      Fx f;
      bits(u[2 * (3 * i + k)], hi, lo); f = fx_link(hi, lo); a.x = f.h; a.y = f.l;
      bits(u[2 * (3 * i + k) + 1], hi, lo); f = fx_link(hi, lo); a.z = f.h; a.w = f.l;
      bits(v[2 * k], hi, lo); f = fx_vec(hi, lo, E); b.x = f.h; b.y = f.l;
      bits(v[2 * k + 1], hi, lo); f = fx_vec(hi, lo, E); b.z = f.h; b.w = f.l;
      fx_cmac(s, a, b);
    }
    T[2 * i] = fx_sum(s.re);
    T[2 * i + 1] = fx_sum(s.im);
  }
  return E;
}
int host_field(const float *u, long long n) {
  FieldCheck f = {0, 0};
  for (long long i = 0; i < n; ++i) {
    float2 m[9];
    memcpy(m, u + 18 * i, sizeof m);
    if (!near_unitary(m)) f.bad = 1;
    f.small += small_parts(m);
  }
  return fx_field(f, n);
}
// X, W: n matrices as units of 2^-58; ok[i] = 0 where the projection left it to FP64
void host_project(const long long *X, long long *W, int *ok, long long n) {
  for (long long i = 0; i < n; ++i) {
    int4 x[9], q[9];
    float f[27];
    for (int k = 0; k < 9; ++k) x[k] = fx_pair(X[18 * i + 2 * k], X[18 * i + 2 * k + 1]);
    ok[i] = project_su3_fx<1>(x, q, f);
    for (int k = 0; k < 9; ++k) {
      W[18 * i + 2 * k] = fx_join(q[k].x, q[k].y);
      W[18 * i + 2 * k + 1] = fx_join(q[k].z, q[k].w);
    }
  }
}
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("host")
    (d / "host.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, *build.ARCH, "-shared",
                    "-Xcompiler", "-fPIC", "-o", str(d / "host.so"), str(d / "host.cu")], check=True, capture_output=True)
    return ctypes.CDLL(str(d / "host.so"))


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("spread", [0, 6, 20])
def test_products(host, spread):
    """u v of three complex products a component: off by at most 6 units of 2^-57 of the scale (v truncated: 2.5 with
    rows of norm 1, u rounded: 1.5, l l' dropped: 1.5, rounding: 1/2)."""
    rng = np.random.default_rng(1501)
    U = synth.su3_matrices(rng, 200, 1.0)
    for u in U:
        v = (rng.standard_normal(3) + 1j * rng.standard_normal(3)) * 10.0 ** rng.uniform(-spread, 0, 3) * 2.0 ** rng.integers(-90, 90)
        T = np.zeros(6, np.int64)
        E = host.host_product(ptr(u), ptr(v), ptr(T))
        scale = Fraction(2) ** (E - 1022)
        assert scale / 2 <= max(np.abs(v.real).max(), np.abs(v.imag).max()) < scale
        for i in range(3):
            re = sum(Fraction(a.real) * Fraction(b.real) - Fraction(a.imag) * Fraction(b.imag) for a, b in zip(u[i], v))
            im = sum(Fraction(a.real) * Fraction(b.imag) + Fraction(a.imag) * Fraction(b.real) for a, b in zip(u[i], v))
            unit = scale / 2 ** 57
            assert abs(int(T[2 * i]) - re / unit) <= 6 and abs(int(T[2 * i + 1]) - im / unit) <= 6


def test_fields_that_are_taken(host):
    def taken(U):
        f = np.ascontiguousarray(U.reshape(-1, 9)).astype(np.complex64)
        return bool(host.host_field(ptr(f), ctypes.c_longlong(len(f))))
    rng = np.random.default_rng(1511)
    rough = synth.su3_matrices(rng, 1000, 0.4)
    assert taken(rough) and taken(synth.su3_matrices(rng, 1000, 0.1)) and taken(synth.su3_matrices(rng, 1000, 3.0))
    assert taken(rough * np.exp(0.7j))  # U(3)
    assert not taken(synth.su3_matrices(rng, 1000, 0.02))
    assert not taken(np.broadcast_to(np.eye(3), (10, 3, 3)) + 0j)
    for bad in (np.full((3, 3), 3 ** -0.5), 1.001 * rough[0], np.full((3, 3), np.nan), rough[0] * np.array([1, 1, 0])):
        U = rough.copy()
        U[500] = bad
        assert not taken(U)


def polar(X):
    """Unitary polar factor without the phase of its determinant, in numpy's long double (Newton's iteration)."""
    def inverse_dagger(y):
        r = [y[:, i] for i in range(3)]
        cof = np.stack([np.cross(r[1], r[2]), np.cross(r[2], r[0]), np.cross(r[0], r[1])], 1)
        det = (r[0] * cof[:, 0]).sum(-1)
        return np.conj(cof / det[:, None, None]), det
    y = X.astype(np.clongdouble)
    for k in range(40):
        z, det = inverse_dagger(y)
        g = np.abs(det)[:, None, None] ** np.longdouble(-1 / 3) if k < 20 else 1
        y = (g * y + z / g) / 2
    det = inverse_dagger(y)[1]
    t = np.exp(-1j * np.angle(det.astype(np.complex128)) / 3).astype(np.clongdouble)
    for _ in range(3):
        t = t * (4 - t * t * t * det) / 3
    return y * t[:, None, None]


@pytest.mark.parametrize("pair", [False, True])  # the singular values: spread evenly, or two small ones
@pytest.mark.parametrize("cond", [1.5, 4, 10, 30, 100, 300, 1000, 1e5])
def test_projection_as_accurate_as_fp64(host, cond, pair):
    """An FP64 Newton iteration errs like a change of X by some 4 x 2^-52 |X|, which moves the polar factor by up to
    2 / (s2 + s3) of it; the fixed-point one stays within that, or leaves the matrix to FP64."""
    n = 1500
    rng = np.random.default_rng(int(cond * 10) + pair)
    A, B = (synth.su3_matrices(rng, n, 3.0) for _ in range(2))
    s = np.array([1.0, 1 / cond if pair else cond ** -0.5, 1 / cond])
    X = 0.9 * np.einsum("nik,k,nkj->nij", A, s, B) * np.exp(1j * rng.uniform(-1, 1, (n, 1, 1)))
    fixed = np.rint(np.ascontiguousarray(X).view(np.float64) * 2.0 ** 58).astype(np.int64)
    W, ok = np.zeros_like(fixed), np.zeros(n, np.int32)
    host.host_project(ptr(fixed), ptr(W), ptr(ok), ctypes.c_longlong(n))
    ref = polar((fixed[..., 0::2] + 1j * fixed[..., 1::2].astype(np.clongdouble)) * np.longdouble(2.0) ** -58)
    got = (W[..., 0::2] + 1j * W[..., 1::2].astype(np.clongdouble)) * np.longdouble(2.0) ** -58
    err = np.abs(got - ref).max((1, 2))
    assert np.all(err[ok == 1] <= 8 * 2.0 ** -52 / (s[1] + s[2]))
    if cond <= 30:
        assert ok.all()
