// fixed.cuh -- FP64-grade products on the integer pipe.
//
// GB300 issues FP64 FMAs at 2 lanes a clock and SM, 32 x 32 + 64 bit integer
// multiply-adds (IMAD.WIDE) at 64 (both measured: 4.08 ms and 0.18 ms for the
// same 2.5e9 of them).  SU(3) links are bounded by 1 and a site's neighbour
// vectors can be scaled by one power of two, so their products need no
// floating point: a link element u becomes U = u 2^58, a vector element v of
// |v| <= 1 (after scaling) V = v 2^57, each split as
//   h 2^29 + l,  -2^28 <= l < 2^28,
// and a product is three multiply-adds into two 64-bit sums,
//   hh += h h'  (unit 2^-57),   cr += h l' + l h'  (unit 2^-86);
// l l' is dropped (below 2^-59 a product, either sign).  The sums are exact; the
// result hh + cr / 2^29 has an absolute error near 2^-57 of the largest factor,
// a tenth of an FP64 FMA chain's, and becomes FP64 with one rounding.  That error
// is absolute: where a sum's own products are all far below the largest factor
// (components of very different sizes that the links do not mix), it would lose
// bits that FP64 keeps.  So the operator and the NPR contraction test their sums
// and leave such ones to FP64, and HYP and NPR run on FP64 altogether on fields
// whose links mix too little (FX_SMALL below).
// Range, for a row of u of 2-norm^2 <= 2 (near_unitary: within 1e-3 of 1) on 6 components
// |v| <= 1, eight hops: by Cauchy-Schwarz |hh| <= 8 sqrt(12) 2^57 < 2^61.8 and
// |cr| <= 8 (sqrt(12) 2^57 + 6 2^56) < 2^62.7.
#pragma once

#include <cuda_runtime.h>

namespace stag {

#define FX_HD __host__ __device__ __forceinline__

constexpr int FX_LO = 29;    // bits of the low limb
constexpr int FX_VBITS = 57; // fraction bits of a vector element

struct Fx {
  int h, l;
};

// V as its two limbs
FX_HD Fx fx_split(long long V) {
  const long long t = V + (1ll << (FX_LO - 1));
  Fx f;
  f.h = (int)(t >> FX_LO);
  f.l = (int)((unsigned)t & ((1u << FX_LO) - 1u)) - (1 << (FX_LO - 1));
  return f;
}

// the FP64 number (hi, lo) as (mantissa << UP) >> (E - its exponent field),
// E >= that field; the bits shifted out are dropped, or rounded (magnitudes,
// halves up), and zeros and denormals become 0 where E >= 64
template <int UP, bool ROUND>
FX_HD Fx fx_from(int hi, int lo, int E) {
  int sh = E - ((hi >> 20) & 0x7ff);
  sh = sh < 63 ? sh : 63;
  unsigned long long m = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)lo;
  m <<= UP;
  if (ROUND) m += (1ull << sh) >> 1;
  m >>= sh;
  const Fx a = fx_split((long long)m);
  const int s = (hi >> 31) | 1;
  Fx f;
  f.h = a.h * s;
  f.l = a.l * s;
  return f;
}
// a link element, |u| < 2: u 2^58
FX_HD Fx fx_link(int hi, int lo) { return fx_from<6, true>(hi, lo, 1023); }
// a vector element scaled by 2^(1022 - E), E >= the exponent fields of its site: v 2^57
FX_HD Fx fx_vec(int hi, int lo, int E) { return fx_from<4, false>(hi, lo, E); }

// sums of products
struct FxAcc {
  long long hh, cr;
};
// s += a b, one IMAD.WIDE (written as PTX: from s + (long long)a * b the
// compiler may make a multiply and a two-instruction add)
FX_HD void fx_wide(long long &s, int a, int b) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s) : "r"(a), "r"(b));
#else
  s += (long long)a * b;
#endif
}
FX_HD void fx_mac(FxAcc &s, int ah, int al, int bh, int bl) {
  fx_wide(s.hh, ah, bh);
  fx_wide(s.cr, ah, bl);
  fx_wide(s.cr, al, bh);
}
// the sum at the unit of hh
FX_HD long long fx_sum(const FxAcc &s) {
  return s.hh + ((s.cr + (1ll << (FX_LO - 1))) >> FX_LO);
}

// Whether the rows of a 3 x 3 matrix are orthonormal to 1e-3, element by element
// of u u^dag (false for NaN): then |u v| <= 1.0015 |v| for any v, and so for
// products of such matrices.  Norms alone would not do: a matrix with all
// elements 3^-1/2 has rows and columns of norm 1 and stretches by sqrt(3), which
// took the limbs of the NPR contraction out of their 32 bits.
FX_HD bool near_unitary(const float2 (&u)[9]) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      float re = i == j ? -1.f : 0.f, im = 0.f;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float2 a = u[3 * i + k], b = u[3 * j + k];
        re += a.x * b.x + a.y * b.y;
        im += a.y * b.x - a.x * b.y;
      }
      ok = ok && fabsf(re) <= 1e-3f && fabsf(im) <= 1e-3f;
    }
  return ok;
}

// A field's links mix the colours, and real with imaginary parts, if few of
// their real components are small.  HYP smearing and the NPR contraction, whose
// products of links keep small elements only to 2^-58, run on FP64 where over an
// eighth are below 2^-6 (unit, diagonal, real or nearly such links).  Links
// exp(i c H): 3 % below at c = 0.4 and for Haar matrices, 11 % at c = 0.1.
// (The operator tests each of its sums, and takes every near-unitary field.)
constexpr float FX_SMALL = 0x1p-6f;
FX_HD int small_parts(const float2 (&u)[9]) {
  int n = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k) n += (fabsf(u[k].x) < FX_SMALL) + (fabsf(u[k].y) < FX_SMALL);
  return n;
}
// what a conversion found out about the nlinks links of its field
struct FieldCheck {
  unsigned long long small;  // real components below FX_SMALL
  int bad;                   // a link is not near unitary
};
FX_HD bool fx_field(const FieldCheck &f, long long nlinks) {
  return f.bad == 0 && 8 * f.small <= 18 * (unsigned long long)nlinks;
}

#ifdef __CUDACC__
// one thread's link (ok: it is near unitary) into the check, all threads of a block together
__device__ __forceinline__ void check_link(FieldCheck *f, bool ok, int nsmall) {
  if (!ok) f->bad = 1;
  const int n = __reduce_add_sync(0xffffffffu, nsmall);
  if ((threadIdx.x & 31) == 0 && n > 0) atomicAdd(&f->small, (unsigned long long)n);
}
#endif

}  // namespace stag
