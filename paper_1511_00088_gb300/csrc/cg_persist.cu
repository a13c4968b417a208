// cg_persist.cu -- the CG iterations between two reliable updates as one
// cooperative kernel (FP32 links and vectors; one system, or a few on a small
// lattice).
//
// Launched as two kernels an iteration, a small lattice's iteration is all
// latency: launch, prologue, the predecessor's sums read and finished by every
// block.  Here 152 / nsys blocks own a system from one reliable update to the
// next, and each half iteration costs its own work and one exchange between the
// blocks.
//   * A block has 15 compute warps and one scalar warp.  When the compute warps
//     are done with a half iteration, the scalar warp adds their sums, posts them,
//     makes the block's writes visible (fence) and counts the block's arrival; when
//     all blocks have arrived, what they wrote is visible: one exchange, 1.2 us
//     for 152 blocks.
//   * The compute warps then gather and apply the hops at once; the scalars (every
//     block reads all sums and adds them alike) are needed only in the epilogue
//     and hide behind the hops.
//   * A warp takes chunks of 32 / LANES sites, LANES lanes a site, 8 / LANES hops a
//     lane (more lanes on smaller lattices, so that the SMs have work).  The block's
//     first chunks keep their links in shared memory for the whole launch (all of
//     them up to 43 000 sites a parity with reconstruct-12), the others read theirs
//     with the gather.  A half iteration's first chunk has its indices and its own
//     vector elements before the exchange is over.
//   * k_cg_persist_sm (lattices with work for one thread a site): the links of the
//     next chunk ahead in shared memory.
// Measured (us per iteration of a whole solve, reliable updates included; two kernels
// an iteration / this): 8^4 12.4 / 7.1, 12^3 x 24 17.9 / 8.4, 16^3 x 32 22.6 / 13.9 (full
// links); 20^3 x 64 with reconstruct-12 49.2 / 39.4.  There an iteration's algorithmic
// bytes are 258 MB; 120 MB of them cross DRAM (0.4 of the copy rate, the rest is
// served by L2, where 85 MB of the 98 MB of links persist), 390 MB cross L2 at 8.4 TB/s,
// and a third of the issue slots are used: bound by the gathers' way through L2.
// Every wait is bounded; a block that gives up sets the error flag and ends, and
// so do the others, their waits running out.  The host then runs the solve again
// with two kernels an iteration.
#include "launch.h"

namespace stag {

namespace {

constexpr int PS_CW = 15;                // compute warps (with a 17th warp a thread has 96 registers, not 128)
constexpr int PS_BT = 32 * (PS_CW + 1);  // threads of a block
constexpr unsigned PS_SMEM = 226u * 1024u;  // dynamic shared memory a block may ask for
constexpr unsigned PS_POLLS = 1u << 21;
constexpr int BAR_DATA = 1, BAR_SCAL = 2, BAR_DONE = 3;

__device__ __forceinline__ void bar_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(PS_BT) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(PS_BT) : "memory"); }

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// The scalar warp's side of the exchange.  post: this block's sums (w0, w1) into
// its word, then, everything the block wrote before being visible, one arrival.
// wait: until `target` arrivals have been counted; false after two seconds and
// 2^21 polls (over a second of the block's own time: time in which the GPU ran
// something else does not count).
// One word is polled, by one lane a block: with every block polling the words of
// all, the posts queued behind the polls (152 blocks: 4 us from the last post to
// the first block that saw it).
__device__ __forceinline__ void post(const PsArgs &a, int half, int grp, int blk, float w0, float w1) {
  unsigned long long *slot = a.slots + ((long long)grp * 2 + half) * PS_MAXB + blk;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(slot),
               "l"(((unsigned long long)__float_as_uint(w1) << 32) | __float_as_uint(w0))
               : "memory");
  fence_gpu();
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(a.arrived + grp * PS_ASTRIDE) : "memory");
}
__device__ __forceinline__ bool wait_for(const PsArgs &a, int grp, unsigned target) {
  const unsigned *p = a.arrived + grp * PS_ASTRIDE;
  if (a.giveup) return false;
  const unsigned long long t0 = global_ns();
  for (unsigned poll = 0;; ++poll) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if ((int)(v - target) >= 0) return true;
    if (poll >= PS_POLLS && (poll & 63) == 63 && global_ns() - t0 > 2000000000ull) return false;
  }
}
// all blocks' words (every lane of the warp; after the wait)
__device__ __forceinline__ void read_slots(const PsArgs &a, int half, int grp, int nbg, unsigned (&x0)[PS_PER],
                                           unsigned (&x1)[PS_PER]) {
  const unsigned long long *s = a.slots + ((long long)grp * 2 + half) * PS_MAXB;
#pragma unroll
  for (int u = 0; u < PS_PER; ++u) {
    const int i = (int)(threadIdx.x & 31) + 32 * u;
    unsigned long long w = 0ull;
    if (i < nbg) asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(s + i) : "memory");
    x0[u] = (unsigned)w;
    x1[u] = (unsigned)(w >> 32);
  }
}

// Sum of a warp's FP32 values (bit patterns) x 2^up, the same whatever their
// order: each at 20 bits below the largest one's last place, added as integers
// (what lies below, 2^-44 of the largest value, is dropped: the values are FP32
// sums, good to 2^-24 of themselves).  Denormals count: a source of 1e-12 has
// nothing else once its residual is 1e-10 of it.  FP64 additions, 67 clocks each
// in a chain of ten, took three times as long, and every block waits for this.
__device__ __forceinline__ double fixed_sum(const unsigned (&x)[PS_PER], int up) {
  unsigned top = 0;
#pragma unroll
  for (int u = 0; u < PS_PER; ++u) top = max(top, x[u] & 0x7fffffffu);
  top = __reduce_max_sync(0xffffffffu, top);
  const int E = max((int)(top >> 23), 1);
  if (E == 255) return __longlong_as_double(0x7ff8000000000000ll);
  long long t = 0;
#pragma unroll
  for (int u = 0; u < PS_PER; ++u) {
    const int e = (int)(x[u] >> 23) & 0xff;
    const unsigned long long m = (unsigned long long)((x[u] & 0x7fffffu) | (e ? 0x800000u : 0u)) << 20;
    const long long v = (long long)(m >> min(E - max(e, 1), 63));
    t += (int)x[u] < 0 ? -v : v;
  }
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)t & 0xffffffu);
  const int hi = __reduce_add_sync(0xffffffffu, (int)(t >> 24));
  const double d = (double)(((long long)hi << 24) + (long long)lo);
  return d * __hiloint2double((E + up - 127 - 23 - 20 + 1023) << 20, 0);  // exact: E - 170 is in FP64's range
}

// a / b as FP32, from an FP32 quotient of the significands and its residual in
// FP64 (within 2^-45 before the rounding); a, b finite and positive
__device__ __forceinline__ float ratio_f(double a, double b) {
  const int ea = __double2hiint(a) >> 20, eb = __double2hiint(b) >> 20;
  const double ma = __hiloint2double((__double2hiint(a) & 0xfffff) | 0x3ff00000, __double2loint(a));
  const double mb = __hiloint2double((__double2hiint(b) & 0xfffff) | 0x3ff00000, __double2loint(b));
  const float fb = (float)mb, q = (float)ma / fb;
  const float r = (float)__fma_rn(-(double)q, mb, ma);
  return ldexpf(q + r / fb, ea - eb);
}

// hop h of site x (parity P): neighbour and sign (minus for the backward hops);
// mu = h >> 1, backward for odd h
__device__ __forceinline__ void hop_of(const Geom &g, const int (&x)[4], int h, int &nb, float &sg) {
  const int mu = h >> 1;
  const int xm = mu == 0 ? x[0] : mu == 1 ? x[1] : mu == 2 ? x[2] : x[3];
  const int L = mu == 0 ? g.L0 : mu == 1 ? g.L1 : mu == 2 ? g.L2 : g.L3;
  int eb = 0;
  if (mu > 0) eb += x[0];
  if (mu > 1) eb += x[1];
  if (mu > 2) eb += x[2];
  const int xn = (h & 1) ? (xm == 0 ? L - 1 : xm - 1) : (xm + 1 == L ? 0 : xm + 1);
  nb = cb_of(g, mu == 0 ? xn : x[0], mu == 1 ? xn : x[1], mu == 2 ? xn : x[2], mu == 3 ? xn : x[3]);
  bool neg = ((eb ^ h) & 1) != 0;
  if (mu == 3 && g.ap && xm == ((h & 1) ? 0 : L - 1)) neg = !neg;
  sg = neg ? -1.f : 1.f;
}

__device__ __forceinline__ float2 ld2(const VecArg &f, int j, int c, int s, int Ve) {
  return reinterpret_cast<const float2 *>(f.v)[(long long)j * f.sstr + (long long)c * Ve + s];
}
__device__ __forceinline__ void st2(const VecArg &f, int j, int c, int s, int Ve, float2 v) {
  reinterpret_cast<float2 *>(f.v)[(long long)j * f.sstr + (long long)c * Ve + s] = v;
}

struct PsShared {
  SysState st;
  float red[2][PS_CW];
  float alpha, beta;
  volatile int stop;
};

// The scalar warp of a block that runs.  What the compute warps wait for (alpha,
// beta, stop) is published first; the state's own FP64 update (finalize_system)
// follows while they go on.
__device__ __forceinline__ void scalar_warp(const PsArgs &a, PsShared &sh, int grp, int blk, int nbg,
                                            unsigned &arrivals) {
  SysState &st = sh.st;
  const int lane = threadIdx.x & 31;
  bool ok = true;
  if (lane == 0) sh.beta = (float)st.beta;
  __syncwarp();
  bar_arrive(BAR_DATA);
  bar_arrive(BAR_SCAL);
  const double tol2 = st.tol * st.tol * st.bnorm2;
  for (;;) {
    // half iteration 1: |t|^2
    const double m4p2 = st.m4 * (st.rho + st.beta * (2.0 * st.rp + st.beta * st.pnorm2));
    const double rho = st.rho, low = st.delta * st.delta * st.rmax2;
    const bool last = st.iter + 1 >= st.maxiter;
    // a block adds its warps' sums in FP32: scaled down where the sum of 15 might
    // overflow (|t|^2 <= 64 |p|^2; all blocks hold the same state)
    const int up = fmax(st.rho, st.pnorm2) > 0x1p90 ? 4 : 0;
    const float down = up ? 0x1p-4f : 1.f;
    unsigned x0[PS_PER], x1[PS_PER];
    bar_sync(BAR_DONE);
    {
      const float w = warp_sum(lane < PS_CW ? down * sh.red[0][lane] : 0.f);
      arrivals += nbg;
      if (lane == 0) {
        post(a, 0, grp, blk, w, 0.f);
        ok = wait_for(a, grp, arrivals);
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
    }
    bar_arrive(BAR_DATA);
    {
      read_slots(a, 0, grp, nbg, x0, x1);
      const double sum[2] = {fixed_sum(x0, up), 0.0};
      const double pAp = m4p2 + sum[0];
      const bool stop = !(pAp > 0.0) || !isfinite(pAp) || !ok;
      if (lane == 0) {
        if (!stop) sh.alpha = ratio_f(rho, pAp);
        if (stop) sh.stop = 1;
      }
      __syncwarp();
      bar_arrive(BAR_SCAL);
      if (lane == 0) finalize_system(st, FIN_ALPHA_R, sum);
      __syncwarp();
      if (stop) break;
    }
    // half iteration 2: |r|^2, Re<r, p>.  A block posts here only after it has
    // read half iteration 1's words, and the other way round: but the others
    // may not have, so the two halves use different words.
    bar_sync(BAR_DONE);
    {
      const float w0 = warp_sum(lane < PS_CW ? down * sh.red[0][lane] : 0.f);
      const float w1 = warp_sum(lane < PS_CW ? down * sh.red[1][lane] : 0.f);
      arrivals += nbg;
      if (lane == 0) {
        post(a, 1, grp, blk, w0, w1);
        ok = wait_for(a, grp, arrivals);
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
    }
    bar_arrive(BAR_DATA);
    {
      read_slots(a, 1, grp, nbg, x0, x1);
      const double rr = fixed_sum(x0, up);
      // finalize_system's conditions for FIN_NORM
      const bool stop = !isfinite(rr) || rr <= tol2 || last || rr < low || !ok;
      if (lane == 0) {
        if (!stop) sh.beta = ratio_f(rr, rho);
        if (stop) sh.stop = 1;
      }
      __syncwarp();
      bar_arrive(BAR_SCAL);
      const double sum[2] = {rr, fixed_sum(x1, up)};
      if (lane == 0) finalize_system(st, FIN_NORM, sum);
      __syncwarp();
      if (stop) break;
    }
  }
  if (lane == 0 && !ok) atomicExch(a.ctl.flags + 4, 1);
}

// The end of a pass, by one thread of each group: the state stored, and by the
// last group the loop's flags and graph conditions.
__device__ __forceinline__ void end_of_pass(const PsArgs &a, const SysState &st, int grp, int nact, bool run,
                                            unsigned arrivals) {
  if (run) {
    a.ctl.st[grp] = st;
    a.counted[grp] = arrivals;
  }
  int running = 0, upd = 0;
  __threadfence();
  if (nact > 1) {
    if (atomicAdd(a.ctl.all_ticket, 1u) != (unsigned)(nact - 1)) return;
    *a.ctl.all_ticket = 0u;
    __threadfence();
  }
  for (int q = 0; q < a.nsys; ++q) {
    const int done = __ldcg(&a.ctl.st[q].done);
    if (done == 0 || done == 3) {
      running = 1;
      if (__ldcg(&a.ctl.st[q].update)) upd = 1;
    }
  }
  const int passes = a.ctl.flags[2] + 1;
  a.ctl.flags[2] = passes;
  if (passes > a.ctl.flags[3]) running = 0;
  if (*(volatile int *)(a.ctl.flags + 4) != 0) running = upd = 0;
  a.ctl.flags[0] = running;
  a.ctl.flags[1] = upd;
  if (a.ctl.use_graph_cond) {
    cudaGraphSetConditional(a.ctl.h_update, (unsigned)upd);
    cudaGraphSetConditional(a.ctl.h_loop, (unsigned)running);
  }
}

template <int RECON, int LANES>
__global__ void __launch_bounds__(PS_BT, 1) k_cg_persist(const PsArgs a) {
  constexpr int HPL = 8 / LANES, SPW = 32 / LANES, NE = RECON ? 6 : 9;
  constexpr int NC = LANES == 2 ? 2 : 1;              // colours a lane stores: q LANES + l
  extern __shared__ __align__(16) float2 resident[];       // [entry][hop of the lane][element][lane]
  __shared__ PsShared sh;
  const Geom g = a.g;
  const int Ve = g.Ve;
  const int nact = a.map[0], nbg = a.map[1];
  if ((int)blockIdx.x >= nact * nbg) return;
  const int grp = a.map[2 + blockIdx.x / nbg], blk = blockIdx.x % nbg;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    sh.st = a.ctl.st[grp];
    sh.stop = *(volatile int *)(a.ctl.flags + 4) != 0;  // an earlier kernel's wait gave up
  }
  __syncthreads();
  const bool run = sh.st.done == 0 && !sh.stop;
  unsigned arrivals = a.counted[grp];
  const float m4 = (float)sh.st.m4;
  __syncthreads();  // the state read by all before the scalar warp changes it
  if (run && warp == PS_CW) {
    scalar_warp(a, sh, grp, blk, nbg, arrivals);
  } else if (run) {
    const int l = lane % LANES;
    // this block's chunks, an even share of the lattice in one piece; its warps take them in turn
    const int nall = (Ve + SPW - 1) / SPW;
    const int first = (int)((long long)nall * blk / nbg), c1 = (int)((long long)nall * (blk + 1) / nbg);
    const int c0 = first + warp, nown = c1 - first;
    int s = 0, nb[HPL];
    unsigned neg = 0;  // bit k: hop k of this lane enters with a minus
    bool valid = false;
    float2 o0[NC], o1[NC], o2[NC];  // this lane's colours of the epilogue's vectors
    const float2 *link[HPL];
    auto colour = [&](int q) { return LANES == 4 ? l : q * LANES + l; };
    // chunk c on parity P: site, hops, and the epilogue's operands on their way
    auto prep = [&](int P, int c) {
      s = c * SPW + lane / LANES;
      valid = s < Ve;
      if (!valid) s = Ve - 1;
      int x[4];
      site_coords(g, P, s, x);
      neg = 0;
#pragma unroll
      for (int k = 0; k < HPL; ++k) {
        const int h = l * HPL + k;
        float sg;
        hop_of(g, x, h, nb[k], sg);
        if (sg < 0.f) neg |= 1u << k;
        link[k] = reinterpret_cast<const float2 *>(a.links) +
                  (long long)((((h & 1) ? 1 - P : P) * 4 + (h >> 1)) * NE) * Ve + ((h & 1) ? nb[k] : s);
      }
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const int cc = colour(q);
        if (cc >= 3) continue;
        if (P == 1) {
          o0[q] = ld2(a.t, grp, cc, s, Ve);
        } else {
          o0[q] = ld2(a.p, grp, cc, s, Ve);
          o1[q] = ld2(a.r, grp, cc, s, Ve);
          o2[q] = ld2(a.x, grp, cc, s, Ve);
        }
      }
    };
    // entry of chunk c on parity P among the resident ones (odd output first)
    auto entry = [&](int P, int c) { return (P == 1 ? 0 : nown) + c - first; };
    auto hops = [&](int P, int c, const VecArg &in, float (&acc)[6]) {
      float v[HPL][6];
#pragma unroll
      for (int k = 0; k < HPL; ++k) load_vec_rw<P32>(in, grp, nb[k], Ve, v[k]);
#pragma unroll
      for (int i = 0; i < 6; ++i) acc[i] = 0.f;
      const int e = entry(P, c);
      auto apply = [&](int k, const float (&u)[18]) {
        const float sg = (neg >> k & 1) ? -1.f : 1.f;
        if (k & 1) mvdag_acc(u, v[k], sg, acc);
        else mv_acc(u, v[k], sg, acc);
      };
      if (e < a.nres) {
#pragma unroll
        for (int k = 0; k < HPL; ++k) {
          float u[18];
          load_link_at<P32, RECON, true>(resident + ((long long)e * HPL + k) * (NE * 32) + lane, 32, u);
          apply(k, u);
        }
      } else {
#pragma unroll
        for (int k = 0; k < HPL; ++k) {
          float u[18];
          load_link_at<P32, RECON, false>(link[k], Ve, u);
          apply(k, u);
        }
      }
#pragma unroll
      for (int o = 1; o < LANES; o <<= 1)
#pragma unroll
        for (int i = 0; i < 6; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
    };
    auto pick = [&](const float (&acc)[6], int c) {
      return c == 0 ? make_float2(acc[0], acc[1]) : c == 1 ? make_float2(acc[2], acc[3]) : make_float2(acc[4], acc[5]);
    };
    // the resident links: each lane its own hops', read by that lane alone
#pragma unroll 1
    for (int P = 1; P >= 0; --P)
#pragma unroll 1
      for (int c = c0; c < c1 && entry(P, c) < a.nres; c += PS_CW) {
        prep(P, c);
#pragma unroll
        for (int k = 0; k < HPL; ++k)
#pragma unroll
          for (int i = 0; i < NE; ++i)
            resident[((long long)entry(P, c) * HPL + k) * (NE * 32) + i * 32 + lane] = __ldg(link[k] + (long long)i * Ve);
      }
    for (;;) {
      // ---- half iteration 1: t = D_oe r + beta t (odd sites), |t|^2
      float part = 0.f, part2 = 0.f;
      bool scal = false;
      if (c0 < c1) prep(1, c0);
      bar_sync(BAR_DATA);
      for (int c = c0; c < c1; c += PS_CW) {
        if (c > c0) prep(1, c);
        float acc[6];
        hops(1, c, a.r, acc);
        if (!scal) {
          bar_sync(BAR_SCAL);
          scal = true;
          if (sh.stop) break;
        }
        const float beta = sh.beta;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          const int cc = colour(q);
          if (!valid || cc >= 3) continue;
          const float2 d = pick(acc, cc);
          const float2 t = make_float2(fmaf(beta, o0[q].x, d.x), fmaf(beta, o0[q].y, d.y));
          st2(a.t, grp, cc, s, Ve, t);
          part += t.x * t.x + t.y * t.y;
        }
      }
      if (!scal) bar_sync(BAR_SCAL);
      if (sh.stop) break;
      part = warp_sum(part);
      if (lane == 0) sh.red[0][warp] = part;
      bar_arrive(BAR_DONE);
      // ---- half iteration 2: p = r + beta p; A p = 4 m^2 p - D_eo t; r -= alpha A p; x += alpha p (even sites)
      const float beta = sh.beta;
      part = 0.f;
      scal = false;
      if (c0 < c1) prep(0, c0);
      bar_sync(BAR_DATA);
      for (int c = c0; c < c1; c += PS_CW) {
        if (c > c0) prep(0, c);
        float acc[6];
        hops(0, c, a.t, acc);
        if (!scal) {
          bar_sync(BAR_SCAL);
          scal = true;
          if (sh.stop) break;
        }
        const float alpha = sh.alpha;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
          const int cc = colour(q);
          if (!valid || cc >= 3) continue;
          const float2 d = pick(acc, cc);
          const float2 p = make_float2(fmaf(beta, o0[q].x, o1[q].x), fmaf(beta, o0[q].y, o1[q].y));
          const float2 r = make_float2(fmaf(-alpha, fmaf(m4, p.x, -d.x), o1[q].x),
                                       fmaf(-alpha, fmaf(m4, p.y, -d.y), o1[q].y));
          st2(a.p, grp, cc, s, Ve, p);
          st2(a.r, grp, cc, s, Ve, r);
          st2(a.x, grp, cc, s, Ve, make_float2(fmaf(alpha, p.x, o2[q].x), fmaf(alpha, p.y, o2[q].y)));
          part += r.x * r.x + r.y * r.y;
          part2 += r.x * p.x + r.y * p.y;
        }
      }
      if (!scal) bar_sync(BAR_SCAL);
      if (sh.stop) break;
      part = warp_sum(part);
      part2 = warp_sum(part2);
      if (lane == 0) {
        sh.red[0][warp] = part;
        sh.red[1][warp] = part2;
      }
      bar_arrive(BAR_DONE);
    }
  }
  __syncthreads();
  if (blk == 0 && threadIdx.x == 32 * PS_CW) end_of_pass(a, sh.st, grp, nact, run, arrivals);
}

// One thread a site, the links of the next chunk (a half iteration's first one
// too, across the exchange between the blocks) copied ahead into shared memory:
// 8 bytes at a time, each thread its own site's, so that no barrier is needed
// and the registers are left to the gathered vectors.  Full links: six of the
// eight fit 15 warps' shares, the last two come with the gather.
constexpr int ps_staged_links(int recon) { return recon ? 8 : 6; }  // k_cg_persist_sm: links of a site in shared memory

template <int RECON>
__global__ void __launch_bounds__(PS_BT, 1) k_cg_persist_sm(const PsArgs a) {
  constexpr int NE = RECON ? 6 : 9, NST = ps_staged_links(RECON);
  extern __shared__ __align__(16) float2 stage_links[];  // [warp][staged link][element][lane]
  __shared__ PsShared sh;
  const Geom g = a.g;
  const int Ve = g.Ve;
  const int nact = a.map[0], nbg = a.map[1];
  if ((int)blockIdx.x >= nact * nbg) return;
  const int grp = a.map[2 + blockIdx.x / nbg], blk = blockIdx.x % nbg;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    sh.st = a.ctl.st[grp];
    sh.stop = *(volatile int *)(a.ctl.flags + 4) != 0;  // an earlier kernel's wait gave up
  }
  __syncthreads();
  const bool run = sh.st.done == 0 && !sh.stop;
  unsigned arrivals = a.counted[grp];
  const float m4 = (float)sh.st.m4;
  __syncthreads();  // the state read by all before the scalar warp changes it
  if (run && warp == PS_CW) {
    scalar_warp(a, sh, grp, blk, nbg, arrivals);
  } else if (run) {
    const int nall = (Ve + 31) / 32;
    const int c1 = (int)((long long)nall * (blk + 1) / nbg);
    const int c0 = (int)((long long)nall * blk / nbg) + warp;
    float2 *mine = stage_links + warp * (NST * NE * 32) + lane;
    const float2 *links = reinterpret_cast<const float2 *>(a.links);
    int nb[8];
    unsigned neg = 0;  // bit h: hop h enters with a minus
    int s = 0;
    bool valid = false;
    // indices and signs of chunk c's site of parity P, and its links on their way
    auto stage = [&](int P, int c) {
      s = c * 32 + lane;
      valid = s < Ve;
      if (!valid) s = Ve - 1;
      int x[4];
      site_coords(g, P, s, x);
      neg = 0;
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        float sg;
        hop_of(g, x, h, nb[h], sg);
        if (sg < 0.f) neg |= 1u << h;
        if (h < NST) {
          const float2 *src = links + (long long)((((h & 1) ? 1 - P : P) * 4 + (h >> 1)) * NE) * Ve + ((h & 1) ? nb[h] : s);
#pragma unroll
          for (int e = 0; e < NE; ++e)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(mine + (h * NE + e) * 32)),
                         "l"(src + (long long)e * Ve)
                         : "memory");
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto hops = [&](int P, const VecArg &in, float (&acc)[6]) {
      float v[8][6];
#pragma unroll
      for (int h = 0; h < 8; ++h) load_vec_rw<P32>(in, grp, nb[h], Ve, v[h]);
#pragma unroll
      for (int i = 0; i < 6; ++i) acc[i] = 0.f;
      asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        float u[18];
        if (h < NST) {
          load_link_at<P32, RECON, true>(mine + h * NE * 32, 32, u);
        } else {
          load_link<P32, RECON>(a.links, Ve, (h & 1) ? 1 - P : P, h >> 1, (h & 1) ? nb[h] : s, u);
        }
        const float sg = (neg >> h & 1) ? -1.f : 1.f;
        if (h & 1) mvdag_acc(u, v[h], sg, acc);
        else mv_acc(u, v[h], sg, acc);
      }
    };
    if (c0 < c1) stage(1, c0);
    for (;;) {
      // ---- half iteration 1: t = D_oe r + beta t (odd sites), |t|^2
      float part = 0.f, part2 = 0.f;
      bool scal = false;
      bar_sync(BAR_DATA);
      for (int c = c0; c < c1; c += PS_CW) {
        const int sc = s;
        const bool on = valid;
        float2 tv[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) tv[q] = ld2(a.t, grp, q, sc, Ve);
        float acc[6];
        hops(1, a.r, acc);
        if (c + PS_CW < c1) stage(1, c + PS_CW);
        else stage(0, c0);
        if (!scal) {
          bar_sync(BAR_SCAL);
          scal = true;
          if (sh.stop) break;
        }
        if (on) {
          const float beta = sh.beta;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float2 tn = make_float2(fmaf(beta, tv[q].x, acc[2 * q]), fmaf(beta, tv[q].y, acc[2 * q + 1]));
            st2(a.t, grp, q, sc, Ve, tn);
            part += tn.x * tn.x + tn.y * tn.y;
          }
        }
      }
      if (!scal) bar_sync(BAR_SCAL);
      if (sh.stop) break;
      part = warp_sum(part);
      if (lane == 0) sh.red[0][warp] = part;
      bar_arrive(BAR_DONE);
      // ---- half iteration 2: p = r + beta p; A p = 4 m^2 p - D_eo t; r -= alpha A p; x += alpha p (even sites)
      const float beta = sh.beta;
      part = 0.f;
      scal = false;
      bar_sync(BAR_DATA);
      for (int c = c0; c < c1; c += PS_CW) {
        const int sc = s;
        const bool on = valid;
        float2 pv[3], rv[3], xv[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          pv[q] = ld2(a.p, grp, q, sc, Ve);
          rv[q] = ld2(a.r, grp, q, sc, Ve);
          xv[q] = ld2(a.x, grp, q, sc, Ve);
        }
        float acc[6];
        hops(0, a.t, acc);
        if (c + PS_CW < c1) stage(0, c + PS_CW);
        else stage(1, c0);
        if (!scal) {
          bar_sync(BAR_SCAL);
          scal = true;
          if (sh.stop) break;
        }
        if (on) {
          const float alpha = sh.alpha;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float2 p = make_float2(fmaf(beta, pv[q].x, rv[q].x), fmaf(beta, pv[q].y, rv[q].y));
            const float2 r = make_float2(fmaf(-alpha, fmaf(m4, p.x, -acc[2 * q]), rv[q].x),
                                         fmaf(-alpha, fmaf(m4, p.y, -acc[2 * q + 1]), rv[q].y));
            st2(a.p, grp, q, sc, Ve, p);
            st2(a.r, grp, q, sc, Ve, r);
            st2(a.x, grp, q, sc, Ve, make_float2(fmaf(alpha, p.x, xv[q].x), fmaf(alpha, p.y, xv[q].y)));
            part += r.x * r.x + r.y * r.y;
            part2 += r.x * p.x + r.y * p.y;
          }
        }
      }
      if (!scal) bar_sync(BAR_SCAL);
      if (sh.stop) break;
      part = warp_sum(part);
      part2 = warp_sum(part2);
      if (lane == 0) {
        sh.red[0][warp] = part;
        sh.red[1][warp] = part2;
      }
      bar_arrive(BAR_DONE);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");  // none outstanding at exit
  }
  __syncthreads();
  if (blk == 0 && threadIdx.x == 32 * PS_CW) end_of_pass(a, sh.st, grp, nact, run, arrivals);
}

// The systems that run and the blocks each gets in the next launch: those that
// have converged leave theirs to the others.  (A kernel of its own: a group may
// end, and change its state, before another block of the launch has started.)
__global__ void k_ps_map(const PsArgs a, int nblocks, int full) {
  const int lane = threadIdx.x;
  int n = 0;
  for (int base = 0; base < a.nsys; base += 32) {
    const int j = base + lane;
    const bool on = j < a.nsys && a.ctl.st[j].done == 0;
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (on) a.map[2 + n + __popc(m & ((1u << lane) - 1u))] = j;
    n += __popc(m);
  }
  if (lane == 0) {
    int nb = n > 0 ? nblocks / n : 0;
    nb = nb < PS_MAXB ? nb : PS_MAXB;
    a.map[0] = n;
    a.map[1] = nb < full ? nb : full;
    if (n == 0) {  // nothing runs: the loop ends
      a.ctl.flags[0] = a.ctl.flags[1] = 0;
      if (a.ctl.use_graph_cond) {
        cudaGraphSetConditional(a.ctl.h_update, 0u);
        cudaGraphSetConditional(a.ctl.h_loop, 0u);
      }
    }
  }
}

// A kernel and the most dynamic shared memory that any launch of it asks for.
// That limit belongs to the process, not to the launch: it is always set to
// `most`, as another thread's context may be between its own setting and its launch.
struct PsKernel {
  void (*k)(PsArgs) = nullptr;
  unsigned most = 0;
};
constexpr unsigned ps_link_bytes(int recon) { return (recon ? 6u : 9u) * 32u * 8u; }  // one link of 32 lanes
// of a chunk (32 / lanes sites)
constexpr unsigned ps_chunk_bytes(int recon, int lanes) { return (unsigned)(8 / lanes) * ps_link_bytes(recon); }
PsKernel ps_kernel(int recon, int lanes) {
  PsKernel p;
  if (lanes == 1) {
    p.k = recon ? k_cg_persist_sm<1> : k_cg_persist_sm<0>;
    p.most = PS_CW * (unsigned)ps_staged_links(recon) * ps_link_bytes(recon);
  } else if (lanes == 2 || lanes == 4) {
    p.k = lanes == 2 ? (recon ? k_cg_persist<1, 2> : k_cg_persist<0, 2>) : (recon ? k_cg_persist<1, 4> : k_cg_persist<0, 4>);
    p.most = PS_SMEM / ps_chunk_bytes(recon, lanes) * ps_chunk_bytes(recon, lanes);
  }
  return p;
}

cudaError_t ps_launch(const PsKernel &p, unsigned smem, int nblocks, cudaStream_t st, const PsArgs &a) {
  const cudaError_t e = cudaFuncSetAttribute(p.k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.most);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.dynamicSmemBytes = smem;
  cfg.gridDim = dim3((unsigned)nblocks);
  cfg.blockDim = dim3(PS_BT);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  unsigned n = 0;
  at[n].id = cudaLaunchAttributeCooperative;  // its blocks wait for one another
  at[n++].val.cooperative = 1;
  if (a.l2_bytes > 0) {
    at[n].id = cudaLaunchAttributeAccessPolicyWindow;
    at[n].val.accessPolicyWindow.base_ptr = const_cast<void *>(a.l2_base);
    at[n].val.accessPolicyWindow.num_bytes = a.l2_bytes;
    at[n].val.accessPolicyWindow.hitRatio = a.l2_hit;
    at[n].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    at[n].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    ++n;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, p.k, a);
}

}  // namespace

int cg_persist_sites(int lanes) { return 32 * PS_CW / lanes; }

cudaError_t cg_persist_fit(int recon, int lanes, int *blocks_per_sm) {
  *blocks_per_sm = 0;
  const PsKernel p = ps_kernel(recon, lanes);
  if (p.k == nullptr) return cudaErrorNotSupported;
  const cudaError_t e = cudaFuncSetAttribute(p.k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.most);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, p.k, PS_BT, p.most);
}

cudaError_t launch_cg_persist(int recon, int lanes, int nblocks, cudaStream_t st, PsArgs a) {
  const PsKernel p = ps_kernel(recon, lanes);
  if (p.k == nullptr) return cudaErrorNotSupported;
  k_ps_map<<<1, 32, 0, st>>>(a, nblocks, (a.g.Ve + cg_persist_sites(lanes) - 1) / cg_persist_sites(lanes));
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (lanes == 1) return ps_launch(p, p.most, nblocks, st, a);
  // shared memory for the links of as many chunks as fit, at most all of a block's
  const int sites = 32 / lanes, nall = (a.g.Ve + sites - 1) / sites;
  const unsigned bytes = ps_chunk_bytes(recon, lanes);
  const int nbg = a.nsys > 0 && nblocks >= a.nsys ? nblocks / a.nsys : 1;  // while all systems run
  const int most = 2 * ((nall + nbg - 1) / nbg);
  a.nres = (int)(p.most / bytes);
  if (a.nres > most) a.nres = most;
  return ps_launch(p, (unsigned)a.nres * bytes, nblocks, st, a);
}

}  // namespace stag
