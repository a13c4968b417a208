// dslash_fx.cu -- the FP64 half operator from fixed-point links (PFX): the
// FP64 CG, the reliable updates and the operator calls on near-unitary gauge
// fields.  The products run on the integer pipe (fixed.cuh).
//
// A block owns chunks of 32 output sites; warp mu holds direction mu of all of
// them, one lane a site, and each thread takes the forward and the backward
// hop: 6 vector and 18 link loads of 16 bytes, all of a warp's 32 lanes on
// consecutive sites, issued before any arithmetic (one memory round trip; with
// whole sites to a thread or two the links came in a second, register-bound
// one: 103 us at 20^3 x 64 where the bytes take 48).  Each thread scales its two
// neighbour vectors by their own largest exponent; its six sums meet the other
// directions' in shared memory as 64-bit integers, where 96 threads, one a
// (site, colour), bring them to a common exponent, add, round once to FP64 and
// run the epilogue: FP64 instructions are spent once a component, not once a
// lane, as they are the scarce ones (a warp's takes 16 clocks of an SM).
// Measured (M^dag M call on device buffers, 20^3 x 64; its two passes over the
// links take 96 us at the copy rate): 364 us on FP64 FMAs with packed copies of
// the vectors, 178 us in this form, 156 us with the caller's layout read and
// written directly (abi_in, abi_center, abi_out); FP64 CG iteration on 16^3 x 32:
// 115 us before, 51 us.
// The error of such a sum is absolute: up to 11.4 units of 2^-57 of a direction's
// scale 2^E, the power of two above its largest neighbour component (neighbours truncated
// 4.9, links rounded 3, l l' dropped 3, rounding 1/2), so up to 50 of the site's with the
// alignment.  A component made of products far below the scale alone (colours of
// very different sizes that these links do not mix) would lose bits that FP64
// keeps.  So one of its four direction sums or their forward halves, each a lower
// bound of m, the sum of its 48 products' magnitudes, has to reach 2^-5 of the scale:
// then it errs by at most 99 x 2^-53 m, where 48 FMAs may err by 48 x 2^-53 m (typically
// by five times as much as this).  Else the thread sums the component on FP64 FMAs
// from the FP64 links, as it does next to an infinity, a NaN or numbers near the
// ends of the exponent range.  That branch costs its block some 5 us.  On links exp(i c H),
// c = 0.1 ... 0.4, and Gaussian vectors less than 1e-6 of the components take it (a line
// at 2^-4: 5e-6; the direction sums alone, at 2^-5: 4e-5, which made the FP64 CG on
// 16^3 x 32 a quarter slower).  Unit and nearly unit links do not mix, but Gaussian
// vectors on them pass as well (M^dag M call 20^3 x 64: 150 us, FP64 form 357); vectors
// of one colour or of real numbers on them take the branch for most components (424 and 480 us).
#include "launch.h"

namespace stag {

namespace {

constexpr int FXB = 128;        // threads: 4 directions x 32 sites
constexpr int FX_ZERO = 0;        // exponent mark of a direction whose neighbours are zero
constexpr int FX_FP64 = 1 << 16;  // and of one that the integer form does not hold
constexpr int FX_E0 = 64;         // smallest exponent field of the integer form
constexpr int FX_E1 = 2030;       // the largest
constexpr int FX_LINE = 1 << 20;  // 2^-5 of the scale, in the high word of a sum

// row `col` of D in at site s of parity P on FP64 FMAs, `in` with strides is, ic
__device__ __noinline__ double2 row_fp64(const Geom &g, const double2 *canon, const double2 *in, long long is,
                                         long long ic, int P, int s, int col) {
  int x[4];
  site_coords(g, P, s, x);
  const long long V = 2ll * g.Ve;
  const long long lex = x[0] + (long long)g.L0 * (x[1] + (long long)g.L1 * (x[2] + (long long)g.L2 * x[3]));
  double2 acc = make_double2(0.0, 0.0);
  int eb = 0;
  long long str = 1;
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    const int L = mu == 0 ? g.L0 : mu == 1 ? g.L1 : mu == 2 ? g.L2 : g.L3;
    const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
    const int xp = (xm + 1 == L) ? 0 : xm + 1, xn = (xm == 0) ? L - 1 : xm - 1;
    const int sf = cb_of(g, mu == 0 ? xp : x[0], mu == 1 ? xp : x[1], mu == 2 ? xp : x[2], mu == 3 ? xp : x[3]);
    const int sb = cb_of(g, mu == 0 ? xn : x[0], mu == 1 ? xn : x[1], mu == 2 ? xn : x[2], mu == 3 ? xn : x[3]);
    const double2 *uf = canon + (mu * V + lex) * 9 + 3 * col;
    const double2 *ub = canon + (mu * V + lex + (xn - xm) * str) * 9 + col;
    double2 f[3], b[3], vf[3], vb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      f[k] = __ldg(uf + k);
      b[k] = __ldg(ub + 3 * k);
      vf[k] = __ldg(in + k * ic + sf * is);
      vb[k] = __ldg(in + k * ic + sb * is);
    }
    double gf = (eb & 1) ? -1.0 : 1.0, gb = -gf;  // backward hops enter with a minus
    if (mu == 3 && g.ap) {
      if (xm == g.L3 - 1) gf = -gf;
      if (xm == 0) gb = -gb;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double fr = gf * f[k].x, fi = gf * f[k].y, br = gb * b[k].x, bi = gb * b[k].y;
      acc.x = __fma_rn(-fi, vf[k].y, __fma_rn(fr, vf[k].x, acc.x));
      acc.y = __fma_rn(fi, vf[k].x, __fma_rn(fr, vf[k].y, acc.y));
      acc.x = __fma_rn(bi, vb[k].y, __fma_rn(br, vb[k].x, acc.x));
      acc.y = __fma_rn(-bi, vb[k].x, __fma_rn(br, vb[k].y, acc.y));
    }
    eb += xm;
    str *= L;
  }
  return acc;
}

// Blocks an SM: 4 (128 registers) for the plain operator, 3 (168) for the CG
// kernels and the residual, whose epilogue operands would spill (20^3 x 64: M^dag
// M call 151 us at 4, 167 at 3; FP64 CG on 16^3 x 32, 708 iterations: 41.2 and 36.0 ms).
template <int EPI, int OP>
__global__ void __launch_bounds__(FXB, (EPI == EPI_PLAIN || EPI == EPI_MDAGM) ? 4 : 3) k_dslash_fx(const DsArgs a) {
  typedef typename Tr<OP>::S2 OS2;
  typedef typename Tr<OP>::R OR;
  constexpr int NV = (EPI == EPI_CG_K2 || EPI == EPI_RESID) ? 2 : 1;
  constexpr bool REDUCES = EPI == EPI_CG_K1R || EPI == EPI_CG_K2 || EPI == EPI_RESID;
  __shared__ long long part_t[2][4][6][32];
  __shared__ int2 part_f[2][4][3][32];  // high words of the forward hop's sums
  __shared__ int part_e[2][4][32];
  const Geom g = a.g;
  const int Ve = g.Ve, P = a.par_out, G = a.ngroups;
  const int grp = blockIdx.x % G, bx0 = blockIdx.x / G, nbx = (int)gridDim.x / G;
  const int nchunk = (Ve + 31) / 32;
  const int lane = threadIdx.x & 31, mu = threadIdx.x >> 5;
  grid_dep_trigger();
  grid_dep_wait();
  __shared__ SysState sst[1];
  const SysState *S = (a.ctl.st != nullptr) ? a.ctl.st + grp : nullptr;
  if (a.fold != FIN_NONE) {
    fold_state<1, FXB>(a, grp, bx0, sst);
    S = sst;
  }
  const bool act = a.gate == GATE_NONE || S == nullptr || state_gate(*S, a.gate);
  const double m4 = S != nullptr ? S->m4 : a.m4_single;
  const double beta = S != nullptr ? S->beta : 0.0;
  const double alpha = S != nullptr ? S->alpha : 0.0;
  double part[1][NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) part[0][v] = 0.0;
  if (act) {
    const int4 *links = reinterpret_cast<const int4 *>(a.links);
    const long long sys = (long long)grp * a.in.sstr;
    const double2 *in = reinterpret_cast<const double2 *>(a.in.v) + sys;
    // strides of a vector's sites and colours, the ABI's or the device layout's
    const long long is = a.abi_in ? 3 : 1, ic = a.abi_in ? 1 : Ve;
    const int Lmu = mu == 0 ? g.L0 : mu == 1 ? g.L1 : mu == 2 ? g.L2 : g.L3;
    int buf = 0;
    for (int bx = bx0; bx < nchunk; bx += nbx, buf ^= 1) {
      const int s = bx * 32 + lane;
      // the epilogue's operands of (site lane, colour mu), in flight with the hops
      const bool epi = mu < 3 && s < Ve;
      const long long o = sys + (long long)mu * Ve + s, oa = 3ll * s + mu;
      double2 c0, c1, c2;
      if (epi) {
        if (EPI == EPI_CG_K2) {
          c0 = reinterpret_cast<const double2 *>(a.center.v)[o];
          c1 = reinterpret_cast<const double2 *>(a.aux.v)[o];
          c2 = reinterpret_cast<const double2 *>(a.xlo.v)[o];
        } else if (EPI == EPI_CG_K1R) {
          c0 = reinterpret_cast<const double2 *>(a.out.v)[o];
        } else if (EPI == EPI_MDAGM) {
          c0 = __ldg(reinterpret_cast<const double2 *>(a.center.v) + (a.abi_center ? oa : o));
        } else if (EPI == EPI_RESID) {
          c0 = __ldg(reinterpret_cast<const double2 *>(a.center.v) + o);
          c1 = __ldg(reinterpret_cast<const double2 *>(a.aux.v) + o);
          c2 = make_double2(0.0, 0.0);
          if (a.dir.v != nullptr) {
            const auto w = to_r2(ldg2(reinterpret_cast<const OS2 *>(a.dir.v) + o));
            c2 = make_double2((double)w.x, (double)w.y);
          }
        }
      }
      if (s < Ve) {
        int x[4];
        site_coords(g, P, s, x);
        int eb = 0;  // x_0 + ... + x_{mu-1}
        if (mu > 0) eb += x[0];
        if (mu > 1) eb += x[1];
        if (mu > 2) eb += x[2];
        const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
        const int xp = (xm + 1 == Lmu) ? 0 : xm + 1, xn = (xm == 0) ? Lmu - 1 : xm - 1;
        const int sf = cb_of(g, mu == 0 ? xp : x[0], mu == 1 ? xp : x[1], mu == 2 ? xp : x[2], mu == 3 ? xp : x[3]);
        const int sb = cb_of(g, mu == 0 ? xn : x[0], mu == 1 ? xn : x[1], mu == 2 ? xn : x[2], mu == 3 ? xn : x[3]);
        unsigned ff = (eb & 1) ? 0x80000000u : 0u, fb = ff ^ 0x80000000u;  // backward hops enter with a minus
        if (mu == 3 && g.ap) {
          if (xm == g.L3 - 1) ff ^= 0x80000000u;
          if (xm == 0) fb ^= 0x80000000u;
        }
        const int4 *uf = links + (long long)((P * 4 + mu) * 9) * Ve + s;
        const int4 *ub = links + (long long)(((1 - P) * 4 + mu) * 9) * Ve + sb;
        double2 wf[3], wb[3];
        int4 lf[9], lb[9];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          wf[c] = __ldg(in + c * ic + sf * is);
          wb[c] = __ldg(in + c * ic + sb * is);
        }
#pragma unroll
        for (int e = 0; e < 9; ++e) {
          lf[e] = __ldg(uf + (long long)e * Ve);
          lb[e] = __ldg(ub + (long long)e * Ve);
        }
        int top = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          top = max(top, max(__double2hiint(wf[c].x) & 0x7fffffff, __double2hiint(wf[c].y) & 0x7fffffff));
          top = max(top, max(__double2hiint(wb[c].x) & 0x7fffffff, __double2hiint(wb[c].y) & 0x7fffffff));
        }
        int E = top >> 20;
        long long T[6];
        bool zero = false;
        if (E < FX_E0 && top == 0) {
          int any = 0;
#pragma unroll
          for (int c = 0; c < 3; ++c)
            any |= __double2loint(wf[c].x) | __double2loint(wf[c].y) | __double2loint(wb[c].x) | __double2loint(wb[c].y);
          zero = any == 0;
        }
        if (zero || E < FX_E0 || E > FX_E1) {
          E = zero ? FX_ZERO : FX_FP64;
#pragma unroll
          for (int i = 0; i < 6; ++i) T[i] = 0;
        } else {
          FxAcc sum[6];
#pragma unroll
          for (int i = 0; i < 6; ++i) sum[i].hh = sum[i].cr = 0;
#pragma unroll
          for (int b = 0; b < 3; ++b) {  // (ur + i ui)(r + i m)
            const Fx r = fx_vec(__double2hiint(wf[b].x) ^ (int)ff, __double2loint(wf[b].x), E);
            const Fx m = fx_vec(__double2hiint(wf[b].y) ^ (int)ff, __double2loint(wf[b].y), E);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const int4 u = lf[3 * k + b];
              fx_mac(sum[2 * k], u.x, u.y, r.h, r.l);
              fx_mac(sum[2 * k], u.z, u.w, -m.h, -m.l);
              fx_mac(sum[2 * k + 1], u.x, u.y, m.h, m.l);
              fx_mac(sum[2 * k + 1], u.z, u.w, r.h, r.l);
            }
          }
#pragma unroll
          for (int k = 0; k < 3; ++k)
            part_f[buf][mu][k][lane] = make_int2((int)(sum[2 * k].hh >> 32), (int)(sum[2 * k + 1].hh >> 32));
#pragma unroll
          for (int b = 0; b < 3; ++b) {  // (ur - i ui)(r + i m)
            const Fx r = fx_vec(__double2hiint(wb[b].x) ^ (int)fb, __double2loint(wb[b].x), E);
            const Fx m = fx_vec(__double2hiint(wb[b].y) ^ (int)fb, __double2loint(wb[b].y), E);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const int4 u = lb[3 * b + k];
              fx_mac(sum[2 * k], u.x, u.y, r.h, r.l);
              fx_mac(sum[2 * k], u.z, u.w, m.h, m.l);
              fx_mac(sum[2 * k + 1], u.x, u.y, m.h, m.l);
              fx_mac(sum[2 * k + 1], u.z, u.w, -r.h, -r.l);
            }
          }
#pragma unroll
          for (int i = 0; i < 6; ++i) T[i] = fx_sum(sum[i]);
        }
        part_e[buf][mu][lane] = E;
#pragma unroll
        for (int i = 0; i < 6; ++i) part_t[buf][mu][i][lane] = T[i];
      }
      // one barrier a chunk: the next chunk writes the other buffer, and its
      // barrier follows every read of this one
      __syncthreads();
      if (epi) {
        int E = FX_ZERO;
#pragma unroll
        for (int d = 0; d < 4; ++d) E = max(E, part_e[buf][d][lane]);
        double2 v = make_double2(0.0, 0.0);
        if (E != FX_ZERO) {
          long long re = 0, im = 0;
          int seen_re = 0, seen_im = 0;  // bits of the direction sums' magnitudes
#pragma unroll
          for (int d = 0; d < 4; ++d) {
            const int sh = min(E - part_e[buf][d][lane], 63);
            const long long a_re = part_t[buf][d][2 * mu][lane] >> sh, a_im = part_t[buf][d][2 * mu + 1][lane] >> sh;
            const int h_re = (int)(a_re >> 32), h_im = (int)(a_im >> 32);
            seen_re |= h_re ^ (h_re >> 31);
            seen_im |= h_im ^ (h_im >> 31);
            re += a_re;
            im += a_im;
          }
          bool f64 = E == FX_FP64;
          if (seen_re < FX_LINE || seen_im < FX_LINE) {  // then those of their forward halves
#pragma unroll 1
            for (int d = 0; d < 4; ++d) {
              const int2 f = part_f[buf][d][mu][lane];  // (unset where the direction is zero: shifted out)
              const int sh = min(E - part_e[buf][d][lane], 31), f_re = f.x >> sh, f_im = f.y >> sh;
              seen_re |= f_re ^ (f_re >> 31);
              seen_im |= f_im ^ (f_im >> 31);
            }
            f64 |= seen_re < FX_LINE || seen_im < FX_LINE;
          }
          if (f64) {
            v = row_fp64(g, a.canon, in, is, ic, P, s, mu);
          } else {
            // unit 2^(E - 1022 - 57): its exponent field stays in 1 .. 2046
            const double unit = __hiloint2double((E - 1022 - FX_VBITS + 1023) << 20, 0);
            v = make_double2((double)re * unit, (double)im * unit);
          }
        }
        if (EPI == EPI_CG_K2) {
          // p = r + beta p_old; Ap = 4 m^2 p - D_eo t; r -= alpha Ap; x += alpha p
          c0.x = __fma_rn(beta, c0.x, c1.x);
          c0.y = __fma_rn(beta, c0.y, c1.y);
          c1.x = __fma_rn(-alpha, __fma_rn(m4, c0.x, -v.x), c1.x);
          c1.y = __fma_rn(-alpha, __fma_rn(m4, c0.y, -v.y), c1.y);
          c2.x = __fma_rn(alpha, c0.x, c2.x);
          c2.y = __fma_rn(alpha, c0.y, c2.y);
          reinterpret_cast<double2 *>(a.center.v)[o] = c0;
          reinterpret_cast<double2 *>(a.aux.v)[o] = c1;
          reinterpret_cast<double2 *>(a.xlo.v)[o] = c2;
          part[0][0] = __fma_rn(c1.x, c1.x, __fma_rn(c1.y, c1.y, part[0][0]));
          part[0][NV - 1] = __fma_rn(c1.x, c0.x, __fma_rn(c1.y, c0.y, part[0][NV - 1]));
        } else if (EPI == EPI_CG_K1R) {
          // t = D_oe r + beta t_old
          v.x = __fma_rn(beta, c0.x, v.x);
          v.y = __fma_rn(beta, c0.y, v.y);
          reinterpret_cast<double2 *>(a.out.v)[o] = v;
          part[0][0] = __fma_rn(v.x, v.x, __fma_rn(v.y, v.y, part[0][0]));
        } else if (EPI == EPI_RESID) {
          // r = b - (4 m^2 x - D in), stored at OP; |r|^2, and Re<r, p> of the stored r
          v.x = c1.x - __fma_rn(m4, c0.x, -v.x);
          v.y = c1.y - __fma_rn(m4, c0.y, -v.y);
          const OR rx = (OR)v.x, ry = (OR)v.y;
          reinterpret_cast<OS2 *>(a.out.v)[o] = from_r<OP>(rx, ry);
          part[0][0] = __fma_rn(v.x, v.x, __fma_rn(v.y, v.y, part[0][0]));
          part[0][NV - 1] = __fma_rn((double)rx, c2.x, __fma_rn((double)ry, c2.y, part[0][NV - 1]));
        } else {
          if (EPI == EPI_MDAGM) {
            v.x = __fma_rn(m4, c0.x, -v.x);
            v.y = __fma_rn(m4, c0.y, -v.y);
            if (a.out_scale != 0.0) {
              v.x *= a.out_scale;
              v.y *= a.out_scale;
            }
          }
          reinterpret_cast<double2 *>(a.out.v)[a.abi_out ? oa : o] = v;
        }
      }
    }
  }
  if (REDUCES) {
    if (a.ctl.st != nullptr) block_partials<1, NV>(a.ctl, part, grp, a.nsys, bx0);
  }
}

template <int EPI, int OP>
cudaError_t fx_one(int nblocks, cudaStream_t st, const DsArgs &a, const void **kptr) {
  auto k = k_dslash_fx<EPI, OP>;
  if (kptr) {
    *kptr = (const void *)k;
    return cudaSuccess;
  }
  return launch_ex_full(k, nblocks, FXB, 0u, st, a.pdl != 0, a.l2_base, a.l2_bytes, a.l2_hit, a);
}

}  // namespace

cudaError_t launch_dslash_fx(int recon, int VP, int OP, int NS, int EPI, int lanes, int nblocks, cudaStream_t st,
                             const DsArgs &a, const void **kptr) {
  if (recon != 0 || VP != P64 || NS != 1 || lanes != FX_LANES) return cudaErrorNotSupported;
#define STAG_FX_CASE(EPI_, OP_) \
  if (EPI == EPI_ && OP == OP_) return fx_one<EPI_, OP_>(nblocks, st, a, kptr);
  STAG_FX_CASE(EPI_PLAIN, P64) STAG_FX_CASE(EPI_MDAGM, P64) STAG_FX_CASE(EPI_CG_K1R, P64)
  STAG_FX_CASE(EPI_CG_K2, P64) STAG_FX_CASE(EPI_RESID, P64) STAG_FX_CASE(EPI_RESID, P32)
#undef STAG_FX_CASE
  return cudaErrorNotSupported;
}

}  // namespace stag
