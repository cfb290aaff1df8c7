// Wilson operator on FP64 fields in 64-bit fixed point (the operator of Sec. 3
// kernel 1 at FP64 accuracy, used by every FP64 application, the FP64 CG and
// the true residuals of the mixed-precision solves).
//
// Why integers.  This part issues 2 FP64 operations per clock and SM but 64
// 32 x 32 + 64 bit integer multiply-adds, so an FP64 stencil (906 FP64
// instructions per site) is bound by the FP64 pipe at 450 clocks per site
// while its bytes need 44.  A link element is at most 1 in magnitude and the
// spinors a site reads are summed anyway, so both are integers with a scale
// and the hopping term is summed exactly:
//   link     u = round(u 2^61)            = uh 2^31 + ul   (|ul| <= 2^30)
//   spinor   P = p 2^(1080 - E) truncated  = ph 2^31 + pl   (0 <= pl < 2^31)
// with E the largest biased exponent among the eight neighbour sites (written per site with
// the field, ExpRange).  A product is three multiply-adds, uh ph 2^62 + (uh pl + ul ph) 2^31;
// the dropped ul pl has mean zero and is at most a quarter of the last place kept.  A row is
// rounded once, the eight hops add exactly, the result is converted to FP64 once, and kappa
// and the centre enter in FP64.  Against a computation in extended precision the result is
// 1.6 times closer than that of FP64 arithmetic (2-norm 5.4e-17 against 9.1e-17 at 8^4).
//
// Range: |P| < 2^58, a projected component < 2^59, a row of a unitary link at most
// sqrt(6) 2^59 / 2, eight hops below 2^62.4; the middle products sum to at most
// sqrt(6) 2^61 + 6 2^58.
//
// What does not fit goes, site by site, through the same stencil in FP64
// arithmetic: sites with a neighbour marked kFixSlow, and every site when
// some link is not unitary to 1e-3 (a flag set when the links are converted).
//
// Two threads per site, as in lq_dfsplit.cuh: lane 0 of a pair computes what
// comes from the first projected colour vector of each hop, lane 1 from the
// second; each accumulates its upper spin, the lower spin it keeps ("keep":
// z, t hops) and the one it hands over at the end ("give": x, y hops).
#pragma once
#include <algorithm>

#include "lq_internal.h"

namespace lq {

constexpr int kFixBlock = 256;

// round(x 2^61) of |x| < 2 as limbs (integer operations: FP64 conversions issue at 2 per clock
// and SM; 24^3 x 32 links 166 us with them); larger or non-finite x gives some other value
__device__ __forceinline__ int2 fix_element(double x) {
  const int hi = __double2hiint(x);
  const unsigned d = 1023u - ((unsigned)hi << 1 >> 21);
  const unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(x)) << 10;
  unsigned long long v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(d));           // shifts beyond 63 give 0
  v = (v >> 1) + (v & 1);
  const long long s = hi >> 31, w = ((long long)v ^ s) - s;
  const int lo = (int)((unsigned)w << 1) >> 1;                     // low 31 bits, signed
  return make_int2((int)((w - lo) >> 31), lo);
}
__device__ __forceinline__ int4 fix_link(double2 u) {
  const int2 a = fix_element(u.x), b = fix_element(u.y);
  return make_int4(a.x, a.y, b.x, b.y);
}

// Running sums of one lane: the upper spin, the lower spin handed to the partner and the
// one kept, [colour][re, im].
struct FixAcc {
  long long up[3][2], give[3][2], keep[3][2];
};

// 32 x 32 + 64 bits, signed.  Written out: the compiler proves the low limbs non-negative, zero-extends
// them and would multiply in full 64 bits (13,058 instead of 8988 instructions per site).
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// |x| 2^(1080 - E) without its fraction (e2 = E << 21 | 0x1fffff, E >= the exponent of x), and
// the sign of x as 0 or -1.
struct FixTerm {
  unsigned long long v;
  int s;
};
__device__ __forceinline__ FixTerm fix_of(double x, unsigned e2) {
  const int hi = __double2hiint(x);
  const unsigned d = (e2 - (unsigned)hi - (unsigned)hi) >> 21;     // E - exponent(x); the sign bit shifts out
  const unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(x)) << 5;
  FixTerm t;
  asm("shr.u64 %0, %1, %2;" : "=l"(t.v) : "l"(m), "r"(d));         // shifts beyond 63 give 0
  t.s = hi >> 31;
  return t;
}
// a + b, each negated where its mask is -1: complements, and the ones they lack in one small term
__device__ __forceinline__ long long fix_add(FixTerm a, int ma, FixTerm b, int mb) {
  const int sa = a.s ^ ma, sb = b.s ^ mb;
  return (long long)(a.v ^ (unsigned long long)(long long)sa) + (long long)(b.v ^ (unsigned long long)(long long)sb) +
         (long long)(unsigned)(-sa - sb);
}

// acc += a b in the two columns: (hi, lo) limbs of a and b
__device__ __forceinline__ void fix_mac(long long& hh, long long& mm, int ah, int al, int2 b) {
  hh = mad_wide(ah, b.x, hh);
  mm = mad_wide(ah, b.y, mm);
  mm = mad_wide(al, b.x, mm);
}
__device__ __forceinline__ int2 fix_limbs(long long h) { return make_int2((int)(h >> 31), (int)h & 0x7fffffff); }

// One hop of lane `half` (ls = 0 for lane 0, -1 for lane 1) in direction MU with projector
// sign S: the link U_mu(link) (FWD) or its adjoint times the projected spinor of site n.
// flip: 0, or -1 when the hop crosses the antiperiodic time boundary.
template <int MU, int S, bool FWD>
__device__ __forceinline__ void fix_hop(const double2* psi, int sstride, const int4* U, int V, int n, int link,
                                        int half, int ls, int flip, unsigned e2, FixAcc& a) {
  const int b = (MU <= 1) ? 3 - half : 2 + half;
  const double2* pa = psi + (size_t)(3 * half) * sstride + n;
  const double2* pb = psi + (size_t)(3 * b) * sstride + n;
  // h = pa + sigma q, q = i pb (x, z) or pb (y, t); sigma = S for x, t; -S, S for y; S, -S for z (lanes 0, 1)
  constexpr int pos = S > 0 ? 0 : -1;
  const int sg = MU == 1 ? ~(pos ^ ls) : MU == 2 ? pos ^ ls : pos;          // 0: +, -1: -
  int2 hr[3], hi[3];                                                        // (hi, lo) limbs
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 x = __ldg(pa + (size_t)c * sstride), y = __ldg(pb + (size_t)c * sstride);
    const FixTerm xr = fix_of(x.x, e2), xi = fix_of(x.y, e2), yr = fix_of(y.x, e2), yi = fix_of(y.y, e2);
    if constexpr (MU == 0 || MU == 2) {
      hr[c] = fix_limbs(fix_add(xr, flip, yi, flip ^ ~sg));
      hi[c] = fix_limbs(fix_add(xi, flip, yr, flip ^ sg));
    } else {
      hr[c] = fix_limbs(fix_add(xr, flip, yr, flip ^ sg));
      hi[c] = fix_limbs(fix_add(xi, flip, yi, flip ^ sg));
    }
  }
  const int4* u0 = U + (size_t)MU * 9 * V + link;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    long long rh = 0, rm = 1 << 30, ih = 0, im = 1 << 30;                   // middle column rounded to nearest
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int4 u = __ldg(u0 + (size_t)(FWD ? 3 * i + j : 3 * j + i) * V);
      fix_mac(rh, rm, u.x, u.y, hr[j]);
      fix_mac(ih, im, u.x, u.y, hi[j]);
      fix_mac(rh, rm, FWD ? -u.z : u.z, FWD ? -u.w : u.w, hi[j]);
      fix_mac(ih, im, FWD ? u.z : -u.z, FWD ? u.w : -u.w, hr[j]);
    }
    const long long wr = rh + (rm >> 31), wi = ih + (im >> 31);
    a.up[i][0] += wr;
    a.up[i][1] += wi;
    // lower spins: x: -S i w; y: -S w, S w; z: -S i w, S i w; t: S w (lanes 0, 1).  The lane-dependent
    // sign is a bitwise complement; the missing +1 is in the start value of the sums (fix_clear).
    const long long m = (long long)(~pos ^ ls);
    if constexpr (MU == 0) {
      if (S > 0) { a.give[i][0] += wi; a.give[i][1] -= wr; }
      else       { a.give[i][0] -= wi; a.give[i][1] += wr; }
    } else if constexpr (MU == 1) {
      a.give[i][0] += wr ^ m;
      a.give[i][1] += wi ^ m;
    } else if constexpr (MU == 2) {
      a.keep[i][0] -= wi ^ m;
      a.keep[i][1] += wr ^ m;
    } else {
      if (S > 0) { a.keep[i][0] += wr; a.keep[i][1] += wi; }
      else       { a.keep[i][0] -= wr; a.keep[i][1] -= wi; }
    }
  }
}

// Start of a site's sums: zero, plus one for each sum that gets one complemented term (each
// lane: one of the two y hops, one of the two z hops).
__device__ __forceinline__ void fix_clear(FixAcc& a) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    a.up[i][0] = a.up[i][1] = 0;
    a.give[i][0] = a.give[i][1] = 1;
    a.keep[i][0] = -1;
    a.keep[i][1] = 1;
  }
}

// ------------------------------------------------------------ the FP64 path of a site
template <int MU, int S, bool FWD>
__device__ __forceinline__ void split_hop64(const double2* psi, int sstride, const double2* U, int V, int n, int link,
                                            int half, bool flip, double (&up)[3][2], double (&give)[3][2],
                                            double (&keep)[3][2]) {
  const int b = (MU <= 1) ? 3 - half : 2 + half;
  cplx<double> h[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 x = __ldg(psi + (size_t)(3 * half + c) * sstride + n), y = __ldg(psi + (size_t)(3 * b + c) * sstride + n);
    const cplx<double> p{x.x, x.y}, q{y.x, y.y};
    cplx<double> t;
    if constexpr (MU == 0) t = times_i(q);
    else if constexpr (MU == 1) t = (half == 0) ? -q : q;
    else if constexpr (MU == 2) t = (half == 0) ? times_i(q) : -times_i(q);
    else t = q;
    h[c] = (S > 0) ? p + t : p - t;
    if (flip) h[c] = -h[c];
  }
  const double2* u0 = U + (size_t)MU * 9 * V + link;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cplx<double> w{0.0, 0.0};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double2 e = __ldg(u0 + (size_t)(FWD ? 3 * i + j : 3 * j + i) * V);
      w = FWD ? cmadd(w, cplx<double>{e.x, e.y}, h[j]) : cjmadd(w, cplx<double>{e.x, e.y}, h[j]);
    }
    up[i][0] += w.re;
    up[i][1] += w.im;
    const double sg = ((MU == 1) == (half == 0)) ? (S > 0 ? -1.0 : 1.0) : (S > 0 ? 1.0 : -1.0);   // y: -S, S; z: S, -S
    if constexpr (MU == 0) { give[i][0] += (S > 0) ? w.im : -w.im; give[i][1] += (S > 0) ? -w.re : w.re; }
    else if constexpr (MU == 1) { give[i][0] += sg * w.re; give[i][1] += sg * w.im; }
    else if constexpr (MU == 2) { keep[i][0] += sg * w.im; keep[i][1] -= sg * w.re; }
    else { keep[i][0] += (S > 0) ? w.re : -w.re; keep[i][1] += (S > 0) ? w.im : -w.im; }
  }
}

// The lane's sums of site s in FP64 arithmetic, as bit patterns (out: up, give, keep).
template <bool DAG>
__device__ __noinline__ void split_site64(Geom geo, const double2* psi, int sstride, const double2* U, int s, int half,
                                          FixAcc* out) {
  constexpr int SF = DAG ? +1 : -1;
  int c[4];
  site_coords(geo, s, c);
  double up[3][2] = {}, give[3][2] = {}, keep[3][2] = {};
  int n;
  n = nbr_fwd(geo, s, c, 0); split_hop64<0, SF, true>(psi, sstride, U, geo.V, n, s, half, false, up, give, keep);
  n = nbr_bwd(geo, s, c, 0); split_hop64<0, -SF, false>(psi, sstride, U, geo.V, n, n, half, false, up, give, keep);
  n = nbr_fwd(geo, s, c, 1); split_hop64<1, SF, true>(psi, sstride, U, geo.V, n, s, half, false, up, give, keep);
  n = nbr_bwd(geo, s, c, 1); split_hop64<1, -SF, false>(psi, sstride, U, geo.V, n, n, half, false, up, give, keep);
  n = nbr_fwd(geo, s, c, 2); split_hop64<2, SF, true>(psi, sstride, U, geo.V, n, s, half, false, up, give, keep);
  n = nbr_bwd(geo, s, c, 2); split_hop64<2, -SF, false>(psi, sstride, U, geo.V, n, n, half, false, up, give, keep);
  n = nbr_fwd(geo, s, c, 3);
  split_hop64<3, SF, true>(psi, sstride, U, geo.V, n, s, half, geo.antiperiodic && c[3] == geo.L[3] - 1, up, give, keep);
  n = nbr_bwd(geo, s, c, 3);
  split_hop64<3, -SF, false>(psi, sstride, U, geo.V, n, n, half, geo.antiperiodic && c[3] == 0, up, give, keep);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      out->up[i][q] = __double_as_longlong(up[i][q]);
      out->give[i][q] = __double_as_longlong(give[i][q]);
      out->keep[i][q] = __double_as_longlong(keep[i][q]);
    }
}

// ------------------------------------------------------------ the operator
// Component of element k of a lane's six (spin half, then spin half + 2, colour fastest).
__device__ __forceinline__ int fix_comp(int half, int k) { return k < 3 ? 3 * half + k : 3 * (half + 2) + (k - 3); }

// Applies M (or M^dag) at the sites of pair `first`, first + stride, ... of one lattice.
// Spinor fields are [chunk][element] with chunk stride `sstride` (V for a single lattice, the
// batch's element count for one column of a batch) and the lattice's sites at elements
// off .. off + V - 1; `in.norm` holds the sites' exponent words.  The epilogue gets the
// element index.
template <bool DAG, class Epi>
__device__ __forceinline__ void fix_sites(const Geom& geo, const FixGauge& U, const SpinorRef& in, int sstride, int off,
                                          double kappa, const Epi& epi, int first, int stride, double (&red)[1]) {
  constexpr int SF = DAG ? +1 : -1;
  const double2* psi = static_cast<const double2*>(in.p) + off;
  const int* word = reinterpret_cast<const int*>(in.norm) + off;
  const bool bad = __ldg(U.bad) != 0;
  const int half = threadIdx.x & 1, ls = -half;
  const int Vr = (geo.V + 15) & ~15;                     // whole warps iterate together
  for (int s0 = first; s0 < Vr; s0 += stride) {
    const bool active = s0 < geo.V;
    const int s = active ? s0 : 0;
    int c[4];
    site_coords(geo, s, c);
    int f[4], b[4], E = kFixMinExp, any = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      f[m] = nbr_fwd(geo, s, c, m);
      b[m] = nbr_bwd(geo, s, c, m);
      const int wf = __ldg(word + f[m]), wb = __ldg(word + b[m]);
      any |= wf | wb;
      E = max(E, max(wf & 0x7ff, wb & 0x7ff));
    }
    const bool slow = bad || (any & kFixSlow);
    FixAcc a;
    if (!slow) {
      const unsigned e2 = (unsigned)E << 21 | 0x1fffffu;
      const int ff = (geo.antiperiodic && c[3] == geo.L[3] - 1) ? -1 : 0, fb = (geo.antiperiodic && c[3] == 0) ? -1 : 0;
      fix_clear(a);
      fix_hop<0, SF, true>(psi, sstride, U.fix, geo.V, f[0], s, half, ls, 0, e2, a);
      fix_hop<0, -SF, false>(psi, sstride, U.fix, geo.V, b[0], b[0], half, ls, 0, e2, a);
      fix_hop<1, SF, true>(psi, sstride, U.fix, geo.V, f[1], s, half, ls, 0, e2, a);
      fix_hop<1, -SF, false>(psi, sstride, U.fix, geo.V, b[1], b[1], half, ls, 0, e2, a);
      fix_hop<2, SF, true>(psi, sstride, U.fix, geo.V, f[2], s, half, ls, 0, e2, a);
      fix_hop<2, -SF, false>(psi, sstride, U.fix, geo.V, b[2], b[2], half, ls, 0, e2, a);
      fix_hop<3, SF, true>(psi, sstride, U.fix, geo.V, f[3], s, half, ls, ff, e2, a);
      fix_hop<3, -SF, false>(psi, sstride, U.fix, geo.V, b[3], b[3], half, ls, fb, e2, a);
    } else {
      FixAcc t64;
      split_site64<DAG>(geo, psi, sstride, U.f64, s, half, &t64);
      a = t64;
    }
    // each lane completes the lower spin it keeps with the partner's sums (both lanes of a
    // pair took the same path)
    cplx<double> v[6];
    const double ks = slow ? -kappa : -kappa * __hiloint2double((E - 56) << 20, 0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double2 c0 = __ldg(psi + (size_t)fix_comp(half, i) * sstride + s);
      const double2 c1 = __ldg(psi + (size_t)fix_comp(half, 3 + i) * sstride + s);
      double lo[2], hi[2];
#pragma unroll
      for (int q2 = 0; q2 < 2; ++q2) {
        const long long got = __shfl_xor_sync(0xffffffffu, a.give[i][q2], 1);
        hi[q2] = slow ? __longlong_as_double(a.up[i][q2]) : (double)a.up[i][q2];
        lo[q2] = slow ? __longlong_as_double(a.keep[i][q2]) + __longlong_as_double(got) : (double)(a.keep[i][q2] + got);
      }
      v[i] = {fma(ks, hi[0], c0.x), fma(ks, hi[1], c0.y)};
      v[3 + i] = {fma(ks, lo[0], c1.x), fma(ks, lo[1], c1.y)};
    }
    epi.apply(sstride, off + s, half, active, v, red);
  }
}

// MINB: resident blocks per SM asked for (register cap).
template <bool DAG, class Epi, int MINB>
__global__ void __launch_bounds__(kFixBlock, MINB)
    dslash_fix_kernel(Geom geo, FixGauge U, SpinorRef in, double kappa, Epi epi, ReduceScratch rs) {
  if (epi.halted()) return;
  double red[1] = {0.0};
  fix_sites<DAG, Epi>(geo, U, in, geo.V, 0, kappa, epi, (blockIdx.x * blockDim.x + threadIdx.x) >> 1,
                      (gridDim.x * blockDim.x) >> 1, red);
  if constexpr (Epi::REDUCE) {
    double tot[1];
    if (grid_sum<1>(red, rs, tot)) epi.finalize(tot);
  }
}

// ------------------------------------------------------------ epilogues (one lane's six components)
__device__ __forceinline__ void load6(const SpinorRef& f, int V, int e, int half, cplx<double> v[6]) {
  const double2* p = static_cast<const double2*>(f.p);
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double2 w = p[(size_t)fix_comp(half, k) * V + e];
    v[k] = {w.x, w.y};
  }
}
// v, and where the field has them the site's exponent word (every lane of the warp calls)
__device__ __forceinline__ void store6(const SpinorRef& f, int V, int e, int half, bool active,
                                       const cplx<double> v[6]) {
  double2* p = static_cast<double2*>(f.p);
  if (active) {
#pragma unroll
    for (int k = 0; k < 6; ++k) p[(size_t)fix_comp(half, k) * V + e] = make_double2(v[k].re, v[k].im);
  }
  if (f.norm) {
    ExpRange r;
    r.spin(v);
    r.spin(v + 3);
    r.mx = max(r.mx, __shfl_xor_sync(0xffffffffu, r.mx, 1));
    r.mn = min(r.mn, __shfl_xor_sync(0xffffffffu, r.mn, 1));
    r.lo |= __shfl_xor_sync(0xffffffffu, r.lo, 1);
    if (active && half == 0) reinterpret_cast<int*>(f.norm)[e] = r.word();
  }
}
__device__ __forceinline__ double norm6(const cplx<double> v[6]) {
  double a = 0.0;
#pragma unroll
  for (int k = 0; k < 6; ++k) { a = fma(v[k].re, v[k].re, a); a = fma(v[k].im, v[k].im, a); }
  return a;
}

struct FixEpiStore {                    // out = M psi
  static constexpr bool REDUCE = false;
  SpinorRef out;
  __device__ bool halted() const { return false; }
  __device__ void apply(int V, int e, int half, bool active, const cplx<double> v[6], double (&)[1]) const {
    store6(out, V, e, half, active, v);
  }
  __device__ void finalize(double (&)[1]) const {}
};

// CG step 1 and 2 (EpiCG1, EpiCG2 of lq_dslash.cuh hold the scalar updates)
struct FixEpiCG1 {
  static constexpr bool REDUCE = true;
  EpiCG1<SStore::F64> base;
  __device__ bool halted() const { return base.halted(); }
  __device__ void apply(int V, int e, int half, bool active, const cplx<double> v[6], double (&red)[1]) const {
    store6(base.t, V, e, half, active, v);
    if (active) red[0] += norm6(v);
  }
  __device__ void finalize(double (&tot)[1]) const { base.finalize(tot); }
};

struct FixEpiCG2 {
  static constexpr bool REDUCE = true;
  EpiCG2<SStore::F64, SStore::F64, SStore::F64> base;
  __device__ bool halted() const { return base.halted(); }
  __device__ void apply(int V, int e, int half, bool active, const cplx<double> v[6], double (&red)[1]) const {
    const double alpha = base.st->alpha;
    cplx<double> r[6], x[6], p[6];
    load6(base.r, V, e, half, r);
    load6(base.x, V, e, half, x);
    load6(base.p, V, e, half, p);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      r[k] = {fma(-alpha, v[k].re, r[k].re), fma(-alpha, v[k].im, r[k].im)};
      x[k] = {fma(alpha, p[k].re, x[k].re), fma(alpha, p[k].im, x[k].im)};
    }
    store6(base.r, V, e, half, active, r);
    store6(base.x, V, e, half, active, x);
    if (active) red[0] += norm6(r);
  }
  __device__ void finalize(double (&tot)[1]) const { base.finalize(tot); }
};

// |r|^2 of a single solve goes to its state
struct FinSolver {
  SolverState* st;
  __device__ void operator()(double rr) const { st->rr_true = rr; }
};

// True residual: v = M^dag (M x) -> r = phi - v, |r|^2 to the finaliser; STORE_LO: r also in
// the inner format (reliable update); STORE_R: r itself
template <SStore SLO, bool STORE_LO, class Fin = FinSolver, bool STORE_R = true>
struct FixEpiResidual {
  static constexpr bool REDUCE = true;
  SpinorRef phi, r, r_lo;
  Fin fin;
  __device__ bool halted() const { return false; }
  __device__ void apply(int V, int e, int half, bool active, const cplx<double> v[6], double (&red)[1]) const {
    cplx<double> ph[6], rv[6];
    load6(phi, V, e, half, ph);
#pragma unroll
    for (int k = 0; k < 6; ++k) rv[k] = ph[k] - v[k];
    if constexpr (STORE_R) store6(r, V, e, half, active, rv);
    if constexpr (STORE_LO) {
      // the inner-format copy needs all 12 components of the site (per-site norm): lane 0 gathers
      cplx<float> full[12];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const cplx<float> mine = {(float)rv[k].re, (float)rv[k].im};
        const cplx<float> o = {__shfl_xor_sync(0xffffffffu, mine.re, 1), __shfl_xor_sync(0xffffffffu, mine.im, 1)};
        full[fix_comp(0, k)] = mine;
        full[fix_comp(1, k)] = o;
      }
      if (active && half == 0) store_spinor<SLO, float>(r_lo, V, e, full);
    }
    if (active) red[0] += norm6(rv);
  }
  __device__ void finalize(double (&tot)[1]) const { fin(tot[0]); }
};

// Blocks of 256
// threads (128 sites), two per SM; measured slower: 64-site blocks at the same occupancy (286
// against 241 us at 24^3 x 32: fewer of the x and y neighbours are in the block's own lines),
// three blocks of 80 registers (344, spills), blocks of 4 x 4 x 4 x 2 sites (304: shorter runs per
// load).  A lattice that leaves SMs without a block takes smaller blocks, and without the register
// cap (its warps are alone on their schedulers: 8^4 14.4 -> 10.3 us).
template <bool DAG, class Epi>
inline void launch_dslash_fix(const Geom& geo, const FixGauge& U, SpinorRef in, double kappa, const Epi& epi,
                              const ReduceScratch& rs, cudaStream_t stream) {
  static const int sms = sm_count();
  const int blocks = grid_for(2 * geo.V, kFixBlock);
  if (blocks <= sms) {
    int bs = kFixBlock;
    while (bs > 32 && grid_for(2 * geo.V, bs) < sms) bs >>= 1;
    dslash_fix_kernel<DAG, Epi, 1><<<grid_for(2 * geo.V, bs), bs, 0, stream>>>(geo, U, in, kappa, epi, rs);
    return;
  }
  static const int wave = resident_grid(reinterpret_cast<const void*>(&dslash_fix_kernel<DAG, Epi, 2>), kFixBlock);
  dslash_fix_kernel<DAG, Epi, 2><<<std::min(blocks, wave), kFixBlock, 0, stream>>>(geo, U, in, kappa, epi, rs);
}

}  // namespace lq
