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
// the dropped ul pl has mean zero and is at most half of the last place kept.  A row is
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
// A warp whose sites all go there skips the integer hops.
//
// Two threads per site, as in lq_dfsplit.cuh: lane 0 of a pair computes what
// comes from the first projected colour vector of each hop, lane 1 from the
// second; each accumulates its upper spin, the lower spin it keeps ("keep":
// z, t hops) and the one it hands over at the end ("give": x, y hops).
#pragma once
#include <algorithm>
#include <atomic>

#include "lq_internal.h"

namespace lq {

constexpr int kFixBlock = 256;

// Whether a row or column of squared length n is that of a unitary link to 1e-3; false for NaN.  Longer
// ones leave the range of the fixed-point sums.  Shorter ones lose digits to the fixed unit: in products
// of links (plaquettes of links 1e-4 long 9% off), and where a link is zero, as on an open boundary,
// because the site behind it still sets the common exponent.
__device__ __forceinline__ bool unit_length(float n) { return n >= 0.999f && n <= 1.001f; }

// How far element k of a link is from that of a real diagonal matrix, in units of 2^-30; all elements of a
// "smooth" link are below kFixSmooth (k_gauge.cu).
constexpr int kFixSmooth = 1 << 25;
__device__ __forceinline__ int fix_far(int4 u, int k) { return k % 4 ? max(abs(u.x), abs(u.z)) : abs(u.z); }

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
// a + b + BIAS, a and b negated where their masks are -1: complements, and the ones they lack in one small term
template <int BIAS = 0>
__device__ __forceinline__ long long fix_add(FixTerm a, int ma, FixTerm b, int mb) {
  const int sa = a.s ^ ma, sb = b.s ^ mb;
  return (long long)(a.v ^ (unsigned long long)(long long)sa) + (long long)(b.v ^ (unsigned long long)(long long)sb) +
         (long long)(unsigned)(BIAS - sa - sb);
}

// acc += a b in the two columns: (hi, lo) limbs of a and b
__device__ __forceinline__ void fix_mac(long long& hh, long long& mm, int ah, int al, int2 b) {
  hh = mad_wide(ah, b.x, hh);
  mm = mad_wide(ah, b.y, mm);
  mm = mad_wide(al, b.x, mm);
}
__device__ __forceinline__ int2 fix_limbs(long long h) { return make_int2((int)(h >> 31), (int)h & 0x7fffffff); }
// The limbs of h - kLimbBias with a signed low one, as the links have: a product of two numbers that both
// come from fix_limbs drops low limbs of one sign, up to a last place each.
constexpr int kLimbBias = 1 << 30;
__device__ __forceinline__ int2 fix_limbs_signed(long long h) {
  return make_int2((int)(h >> 31), ((int)h & 0x7fffffff) - kLimbBias);
}

// Where the operator reads: [chunk][element] fields with fixed-point links (V: the lattice's
// volume, sstride: the chunk stride of the spinor field, psi its first element).
struct SoaAccess {
  const double2* psi;
  int sstride;
  const int4* fix;
  const double2* f64;
  int V;
  // component `comp` of site n and the k-th after it; the link (mu, s) and its element e
  __device__ __forceinline__ const double2* site(int comp, int n) const { return psi + (size_t)comp * sstride + n; }
  __device__ __forceinline__ double2 spin(const double2* p, int k) const { return p[(size_t)k * sstride]; }
  __device__ __forceinline__ const int4* link(int mu, int s) const { return fix + (size_t)mu * 9 * V + s; }
  __device__ __forceinline__ int4 element(const int4* p, int e) const { return __ldg(p + (size_t)e * V); }
  __device__ __forceinline__ double2 element64(int mu, int e, int s) const {
    return __ldg(f64 + ((size_t)mu * 9 + e) * V + s);
  }
};

// The lane's two spins (half and its partner in the projection of direction MU) of site n, as read.
struct FixRaw {
  double2 x[3], y[3];
};
template <int MU, class Acc>
__device__ __forceinline__ void fix_load(const Acc& in, int n, int half, FixRaw& r) {
  const int b = (MU <= 1) ? 3 - half : 2 + half;
  const double2 *pa = in.site(3 * half, n), *pb = in.site(3 * b, n);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    r.x[c] = in.spin(pa, c);
    r.y[c] = in.spin(pb, c);
  }
}

// Projected spinor of lane `half` (ls = 0 for lane 0, -1 for lane 1) in direction MU with projector
// sign S as limbs.  flip: 0, or -1 when the hop crosses the antiperiodic time boundary.
template <int MU, int S>
__device__ __forceinline__ void fix_half(const FixRaw& r, int ls, int flip, unsigned e2, int2 (&hr)[3], int2 (&hi)[3]) {
  // h = x + sigma q, q = i y (x, z) or y (y, t); sigma = S for x, t; -S, S for y; S, -S for z (lanes 0, 1)
  constexpr int pos = S > 0 ? 0 : -1;
  const int sg = MU == 1 ? ~(pos ^ ls) : MU == 2 ? pos ^ ls : pos;          // 0: +, -1: -
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const FixTerm xr = fix_of(r.x[c].x, e2), xi = fix_of(r.x[c].y, e2), yr = fix_of(r.y[c].x, e2), yi = fix_of(r.y[c].y, e2);
    if constexpr (MU == 0 || MU == 2) {
      hr[c] = fix_limbs(fix_add(xr, flip, yi, flip ^ ~sg));
      hi[c] = fix_limbs(fix_add(xi, flip, yr, flip ^ sg));
    } else {
      hr[c] = fix_limbs(fix_add(xr, flip, yr, flip ^ sg));
      hi[c] = fix_limbs(fix_add(xi, flip, yi, flip ^ sg));
    }
  }
}

// U h (FWD) or U^dag h added to the lane's sums; link(e): element e of the link as limbs.
template <int MU, int S, bool FWD, class Link>
__device__ __forceinline__ void fix_rows(const Link& link, const int2 (&hr)[3], const int2 (&hi)[3], int ls, FixAcc& a) {
  constexpr int pos = S > 0 ? 0 : -1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    long long rh = 0, rm = 1 << 30, ih = 0, im = 1 << 30;                   // middle column rounded to nearest
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int4 u = link(FWD ? 3 * i + j : 3 * j + i);
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

// One hop: the link U_mu(link) (FWD) or its adjoint times the projected spinor of site n.
template <int MU, int S, bool FWD, class Acc>
__device__ __forceinline__ void fix_hop(const Acc& in, int n, int link, int half, int ls, int flip, unsigned e2,
                                        FixAcc& a) {
  FixRaw r;
  fix_load<MU>(in, n, half, r);
  int2 hr[3], hi[3];
  fix_half<MU, S>(r, ls, flip, e2, hr, hi);
  const auto u0 = in.link(MU, link);
  fix_rows<MU, S, FWD>([&](int e) { return in.element(u0, e); }, hr, hi, ls, a);
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
__device__ __forceinline__ double sign_xor(double v, int bit) {
  return __hiloint2double(__double2hiint(v) ^ bit, __double2loint(v));
}
__device__ __forceinline__ cplx<double> sign_xor(cplx<double> v, int bit) { return {sign_xor(v.re, bit), sign_xor(v.im, bit)}; }

template <int MU, int S, bool FWD, class Acc>
__device__ __forceinline__ void split_hop64(const Acc& in, int n, int link, int half, bool flip, double (&up)[3][2], double (&give)[3][2],
                                            double (&keep)[3][2]) {
  const int b = (MU <= 1) ? 3 - half : 2 + half;
  cplx<double> h[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double2 x = in.spin(in.site(3 * half, n), c), y = in.spin(in.site(3 * b, n), c);
    const cplx<double> p{x.x, x.y}, q{y.x, y.y};
    // signs that depend on the lane or the boundary: integer operations, the FP64 pipe is the bound
    const int sl = (half == 0) == (MU == 1) ? (int)0x80000000 : 0;
    cplx<double> t;
    if constexpr (MU == 0) t = times_i(q);
    else if constexpr (MU == 1) t = sign_xor(q, sl);
    else if constexpr (MU == 2) t = times_i(sign_xor(q, sl));
    else t = q;
    h[c] = (S > 0) ? p + t : p - t;
    if constexpr (MU == 3) h[c] = sign_xor(h[c], flip ? (int)0x80000000 : 0);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cplx<double> w{0.0, 0.0};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double2 e = in.element64(MU, FWD ? 3 * i + j : 3 * j + i, link);
      w = FWD ? cmadd(w, cplx<double>{e.x, e.y}, h[j]) : cjmadd(w, cplx<double>{e.x, e.y}, h[j]);
    }
    // the first contribution to a sum sets it
    constexpr bool SET = MU == 0 && FWD, SETK = MU == 2 && FWD;
    auto add = [](double& a, double x, bool set) { a = set ? x : a + x; };
    add(up[i][0], w.re, SET);
    add(up[i][1], w.im, SET);
    const double sg = ((MU == 1) == (half == 0)) ? (S > 0 ? -1.0 : 1.0) : (S > 0 ? 1.0 : -1.0);   // y: -S, S; z: S, -S
    if constexpr (MU == 0) { add(give[i][0], (S > 0) ? w.im : -w.im, SET); add(give[i][1], (S > 0) ? -w.re : w.re, SET); }
    else if constexpr (MU == 1) { give[i][0] += sg * w.re; give[i][1] += sg * w.im; }
    else if constexpr (MU == 2) { keep[i][0] = SETK ? sg * w.im : fma(sg, w.im, keep[i][0]); keep[i][1] = SETK ? -sg * w.re : fma(-sg, w.re, keep[i][1]); }
    else { keep[i][0] += (S > 0) ? w.re : -w.re; keep[i][1] += (S > 0) ? w.im : -w.im; }
  }
}

// The lane's sums of site s in FP64 arithmetic, as bit patterns (out: up, give, keep).
// Bound by the FP64 pipe, so signs are integer operations and no sum starts with an addition to zero:
// links that are not unitary, M at 24^3 x 32, 789 -> 703 us.
template <bool DAG, class Acc>
__device__ __noinline__ void split_site64(Geom geo, Acc in, int s, int half, FixAcc* out) {
  constexpr int SF = DAG ? +1 : -1;
  int c[4];
  site_coords(geo, s, c);
  double up[3][2], give[3][2], keep[3][2];
  int n;
  n = nbr_fwd(geo, s, c, 0); split_hop64<0, SF, true>(in, n, s, half, false, up, give, keep);
  n = nbr_bwd(geo, s, c, 0); split_hop64<0, -SF, false>(in, n, n, half, false, up, give, keep);
  n = nbr_fwd(geo, s, c, 1); split_hop64<1, SF, true>(in, n, s, half, false, up, give, keep);
  n = nbr_bwd(geo, s, c, 1); split_hop64<1, -SF, false>(in, n, n, half, false, up, give, keep);
  n = nbr_fwd(geo, s, c, 2); split_hop64<2, SF, true>(in, n, s, half, false, up, give, keep);
  n = nbr_bwd(geo, s, c, 2); split_hop64<2, -SF, false>(in, n, n, half, false, up, give, keep);
  n = nbr_fwd(geo, s, c, 3);
  split_hop64<3, SF, true>(in, n, s, half, geo.antiperiodic && c[3] == geo.L[3] - 1, up, give, keep);
  n = nbr_bwd(geo, s, c, 3);
  split_hop64<3, -SF, false>(in, n, n, half, geo.antiperiodic && c[3] == 0, up, give, keep);
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

// The eight hops of site s (coordinates c, neighbours f, b) with common exponent E.
template <bool DAG, class Acc>
__device__ __forceinline__ void fix_hops(const Geom& geo, const Acc& in, int s, const int c[4], const int f[4],
                                         const int b[4], int half, int E, FixAcc& a) {
  constexpr int SF = DAG ? +1 : -1;
  const int ls = -half;
  const unsigned e2 = (unsigned)E << 21 | 0x1fffffu;
  const int ff = (geo.antiperiodic && c[3] == geo.L[3] - 1) ? -1 : 0, fb = (geo.antiperiodic && c[3] == 0) ? -1 : 0;
  fix_hop<0, SF, true>(in, f[0], s, half, ls, 0, e2, a);
  fix_hop<0, -SF, false>(in, b[0], b[0], half, ls, 0, e2, a);
  fix_hop<1, SF, true>(in, f[1], s, half, ls, 0, e2, a);
  fix_hop<1, -SF, false>(in, b[1], b[1], half, ls, 0, e2, a);
  fix_hop<2, SF, true>(in, f[2], s, half, ls, 0, e2, a);
  fix_hop<2, -SF, false>(in, b[2], b[2], half, ls, 0, e2, a);
  fix_hop<3, SF, true>(in, f[3], s, half, ls, ff, e2, a);
  fix_hop<3, -SF, false>(in, b[3], b[3], half, ls, fb, e2, a);
}

// The same with the operands of the next hop copied to shared memory (cp.async) while a hop
// computes: the stencil is bound by the latency of its loads at the 16 warps per SM its registers
// allow, and the copies need none.  Per stage a block holds 21 rows of 16 bytes per site: the 9 link
// elements (copied by both lanes of a pair, 5 and 4), then each lane's 6 spinor components; two
// stages.  `stage` points at the pair's column of stage 0.
constexpr int kFixRows = 21;
constexpr size_t fix_smem(int block) { return (size_t)2 * kFixRows * (block / 2) * sizeof(int4); }

__device__ __forceinline__ void fix_copy16(int4* smem, const void* gmem) {
  const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(gmem) : "memory");
}
template <int H, int BS>
__device__ __forceinline__ void fix_issue(const SoaAccess& in, const int f[4], const int b[4], int s, int half,
                                          int4* stage) {
  constexpr int MU = H >> 1;
  constexpr bool FWD = (H & 1) == 0;
  constexpr int P = BS / 2;
  const int n = FWD ? f[MU] : b[MU];
  int4* st = stage + (H & 1) * (kFixRows * P);
  const int4* u = in.link(MU, FWD ? s : n) + (size_t)(5 * half) * in.V;
#pragma unroll
  for (int e = 0; e < 4; ++e) fix_copy16(st + (5 * half + e) * P, u + (size_t)e * in.V);
  if (half == 0) fix_copy16(st + 4 * P, u + (size_t)4 * in.V);
  const int q = (MU <= 1) ? 3 - half : 2 + half;
  const double2 *pa = in.site(3 * half, n), *pb = in.site(3 * q, n);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    fix_copy16(st + (9 + 6 * half + c) * P, pa + (size_t)c * in.sstride);
    fix_copy16(st + (12 + 6 * half + c) * P, pb + (size_t)c * in.sstride);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int H, bool DAG, int BS>
__device__ __forceinline__ void fix_step(const SoaAccess& in, const int f[4], const int b[4], int s, int half, int flip,
                                         unsigned e2, int4* stage, FixAcc& a) {
  constexpr int MU = H >> 1, P = BS / 2;
  constexpr bool FWD = (H & 1) == 0;
  constexpr int S = (DAG ? +1 : -1) * (FWD ? 1 : -1);
  if constexpr (H < 7) {
    fix_issue<H + 1, BS>(in, f, b, s, half, stage);
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
  } else {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  }
  __syncwarp();                                       // the partner's copies of the link
  const int4* st = stage + (H & 1) * (kFixRows * P);
  FixRaw r;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    r.x[c] = *reinterpret_cast<const double2*>(st + (9 + 6 * half + c) * P);
    r.y[c] = *reinterpret_cast<const double2*>(st + (12 + 6 * half + c) * P);
  }
  int2 hr[3], hi[3];
  fix_half<MU, S>(r, -half, flip, e2, hr, hi);
  fix_rows<MU, S, FWD>([&](int e) { return st[e * P]; }, hr, hi, -half, a);
  __syncwarp();                                       // the stage may be refilled
}
template <bool DAG, int BS>
__device__ __forceinline__ void fix_hops_async(const Geom& geo, const SoaAccess& in, int s, const int c[4],
                                               const int f[4], const int b[4], int half, int E, int4* stage, FixAcc& a) {
  const unsigned e2 = (unsigned)E << 21 | 0x1fffffu;
  const int ff = (geo.antiperiodic && c[3] == geo.L[3] - 1) ? -1 : 0, fb = (geo.antiperiodic && c[3] == 0) ? -1 : 0;
  fix_step<0, DAG, BS>(in, f, b, s, half, 0, e2, stage, a);
  fix_step<1, DAG, BS>(in, f, b, s, half, 0, e2, stage, a);
  fix_step<2, DAG, BS>(in, f, b, s, half, 0, e2, stage, a);
  fix_step<3, DAG, BS>(in, f, b, s, half, 0, e2, stage, a);
  fix_step<4, DAG, BS>(in, f, b, s, half, 0, e2, stage, a);
  fix_step<5, DAG, BS>(in, f, b, s, half, 0, e2, stage, a);
  fix_step<6, DAG, BS>(in, f, b, s, half, ff, e2, stage, a);
  fix_step<7, DAG, BS>(in, f, b, s, half, fb, e2, stage, a);
}

// The lane's two spins of M psi at site s: centre + ks * hopping sums.  Each lane completes the
// lower spin it keeps with the partner's sums (both lanes of a pair took the same path; every lane
// of the warp calls).  slow: the sums are FP64 bit patterns.  One branch around the twelve values, not one
// around each: those became selections, and the conversions of the integer side took 24 of 902 places on
// the FP64 pipe that bounds slow sites (24^3 x 32 705 -> 684 us, 16^4 125 -> 121).
template <class Acc>
__device__ __forceinline__ void fix_finish(const Acc& in, const FixAcc& a, int s, int half, bool slow, double ks,
                                           cplx<double> v[6]) {
  long long got[3][2];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int q = 0; q < 2; ++q) got[i][q] = __shfl_xor_sync(0xffffffffu, a.give[i][q], 1);
  double up[3][2], lo[3][2];
  if (slow) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        up[i][q] = __longlong_as_double(a.up[i][q]);
        lo[i][q] = __longlong_as_double(a.keep[i][q]) + __longlong_as_double(got[i][q]);
      }
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        up[i][q] = (double)a.up[i][q];
        lo[i][q] = (double)(a.keep[i][q] + got[i][q]);
      }
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double2 c0 = in.spin(in.site(3 * half, s), i), c1 = in.spin(in.site(3 * (half + 2), s), i);
    v[i] = {fma(ks, up[i][0], c0.x), fma(ks, up[i][1], c0.y)};
    v[3 + i] = {fma(ks, lo[i][0], c1.x), fma(ks, lo[i][1], c1.y)};
  }
}

// Applies M (or M^dag) at the sites of pair `first`, first + stride, ... of one lattice.
// Spinor fields are [chunk][element] with chunk stride `sstride` (V for a single lattice, the
// batch's element count for one column of a batch) and the lattice's sites at elements
// off .. off + V - 1; `in.norm` holds the sites' exponent words.  The epilogue gets the
// element index.  ASYNC: threads per block of the copying variant, 0: loads at their use.
template <bool DAG, int ASYNC, class Epi>
__device__ __forceinline__ void fix_sites(const Geom& geo, const FixGauge& U, const SpinorRef& in, int sstride, int off,
                                          double kappa, const Epi& epi, int first, int stride, double (&red)[1]) {
  const SoaAccess acc{static_cast<const double2*>(in.p) + off, sstride, U.fix, U.f64, geo.V};
  const int* word = reinterpret_cast<const int*>(in.norm) + off;
  const bool bad = __ldg(U.flags + kFixBad) != 0;
  const int half = threadIdx.x & 1;
  extern __shared__ int4 fix_stages[];
  int4* stage = fix_stages + (threadIdx.x >> 1);
  const int Vr = (geo.V + 15) & ~15;                     // whole warps iterate together
  // A warp whose sites all took FP64 arithmetic looks at the next sites' words before it copies anything; the
  // others copy first (a vote before the hops would make those wait for the words: 2 to 4% of M).
  bool look = bad;
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
    }
    if constexpr (ASYNC) {
      if (!look) fix_issue<0, ASYNC>(acc, f, b, s, half, stage);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int wf = word[f[m]], wb = word[b[m]];
      any |= wf | wb;
      E = max(E, max(wf & 0x7ff, wb & 0x7ff));
    }
    const bool slow = bad || (any & kFixSlow);
    FixAcc a;
    fix_clear(a);
    if constexpr (ASYNC) {
      if (look && !bad && !__all_sync(0xffffffffu, slow)) {
        fix_issue<0, ASYNC>(acc, f, b, s, half, stage);
        look = false;
      }
      if (!look) fix_hops_async<DAG, ASYNC>(geo, acc, s, c, f, b, half, E, stage, a);   // every lane: warp barriers
    } else if (!slow) {
      fix_hops<DAG>(geo, acc, s, c, f, b, half, E, a);
    }
    if (slow) {
      FixAcc t64;
      split_site64<DAG>(geo, acc, s, half, &t64);
      a = t64;
    }
    if constexpr (ASYNC) look = bad || __all_sync(0xffffffffu, slow);
    cplx<double> v[6];
    fix_finish(acc, a, s, half, slow, slow ? -kappa : -kappa * __hiloint2double((E - 56) << 20, 0), v);
    epi.apply(sstride, off + s, half, active, v, red);
  }
}

template <bool DAG, class Epi, int BS>
__global__ void __launch_bounds__(BS, 512 / BS)
    dslash_fix_kernel(Geom geo, FixGauge U, SpinorRef in, double kappa, Epi epi, ReduceScratch rs) {
  pdl_wait();
  if (epi.halted()) return;
  double red[1] = {0.0};
  fix_sites<DAG, BS, Epi>(geo, U, in, geo.V, 0, kappa, epi, (blockIdx.x * blockDim.x + threadIdx.x) >> 1,
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

// The lane's two spins of M psi, split by direction: four warps (dir) share 16 sites (32 lanes), the first
// adds the integer sums (in any order the same) and finishes the sites; v is valid in its lanes.
// Every thread of the block calls.
template <bool DAG, class Acc>
__device__ __forceinline__ void fix_dir_site(const Geom& geo, const Acc& acc, int s, const int c[4], const int f[4],
                                             const int b[4], int E, bool slow, int lane, int dir, double kappa,
                                             long long (&part)[3][12][32], cplx<double> v[6]) {
  constexpr int SF = DAG ? +1 : -1;
  const int half = lane & 1, ls = -half;
  const unsigned e2 = (unsigned)E << 21 | 0x1fffffu;
  FixAcc a;
  fix_clear(a);
  if (__all_sync(0xffffffffu, slow)) {
    // the four warps hold the same 16 sites, so all of them skip the hops
  } else if (dir == 0) {
    fix_hop<0, SF, true>(acc, f[0], s, half, ls, 0, e2, a);
    fix_hop<0, -SF, false>(acc, b[0], b[0], half, ls, 0, e2, a);
  } else if (dir == 1) {
    fix_hop<1, SF, true>(acc, f[1], s, half, ls, 0, e2, a);
    fix_hop<1, -SF, false>(acc, b[1], b[1], half, ls, 0, e2, a);
  } else if (dir == 2) {
    fix_hop<2, SF, true>(acc, f[2], s, half, ls, 0, e2, a);
    fix_hop<2, -SF, false>(acc, b[2], b[2], half, ls, 0, e2, a);
  } else {
    const int ff = (geo.antiperiodic && c[3] == geo.L[3] - 1) ? -1 : 0, fb = (geo.antiperiodic && c[3] == 0) ? -1 : 0;
    fix_hop<3, SF, true>(acc, f[3], s, half, ls, ff, e2, a);
    fix_hop<3, -SF, false>(acc, b[3], b[3], half, ls, fb, e2, a);
  }
  // x, y add to "give", z, t to "keep"; the start values of fix_clear (give 1; keep -1, 1) are
  // counted once each, those of the warps of y and z
  if (dir > 0) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        part[dir - 1][2 * i + q][lane] = a.up[i][q];
        part[dir - 1][6 + 2 * i + q][lane] =
            dir == 1 ? a.give[i][q] : dir == 2 ? a.keep[i][q] : a.keep[i][q] - (q ? 1 : -1);
      }
  }
  __syncthreads();
  if (dir > 0) return;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      a.up[i][q] += part[0][2 * i + q][lane] + part[1][2 * i + q][lane] + part[2][2 * i + q][lane];
      a.give[i][q] += part[0][6 + 2 * i + q][lane] - 1;
      a.keep[i][q] = part[1][6 + 2 * i + q][lane] + part[2][6 + 2 * i + q][lane];
    }
  if (slow) {
    FixAcc t64;
    split_site64<DAG>(geo, acc, s, half, &t64);
    a = t64;
  }
  fix_finish(acc, a, s, half, slow, slow ? -kappa : -kappa * __hiloint2double((E - 56) << 20, 0), v);
}

// Small lattices leave most of the chip idle, and a pass takes as long as one thread needs for its
// eight hops: split by direction.  Split against two threads per site, us: M 4^4 5.2 / 9.7, 8^4 8.6 / 9.9,
// 8^3 x 16 9.1 / 10.1, 8^2 x 12^2 9.2 / 10.2, 8 x 12^3 16.3 / 13.3; static M^dag M 4^4 22.8 / 51.8, 8^4 34.9 / 51.3,
// 8^3 x 16 34.9 / 52.0, 8^2 x 12^2 34.9 / 51.9, 8 x 12^3 58.9 / 53.3; an FP64 CG iteration, whose reductions want
// few blocks, 4^4 24.0 / 32.6, 8^4 31.6 / 32.4, 8^3 x 12 33.7 / 33.5, 8^3 x 16 34.3 / 32.9.  One line for all
// three, at a size where it costs the iteration 4% and saves the others 10 and 33%.
constexpr int kFixDirSites = 8192;
template <bool DAG, class Epi>
__global__ void __launch_bounds__(128, 4)
    dslash_fix_dir_kernel(Geom geo, FixGauge U, SpinorRef in, double kappa, Epi epi, ReduceScratch rs) {
  __shared__ long long part[3][12][32];
  pdl_wait();
  if (epi.halted()) return;
  const SoaAccess acc{static_cast<const double2*>(in.p), geo.V, U.fix, U.f64, geo.V};
  const int* word = reinterpret_cast<const int*>(in.norm);
  const bool bad = __ldg(U.flags + kFixBad) != 0;
  const int lane = threadIdx.x & 31, dir = threadIdx.x >> 5;
  double red[1] = {0.0};
  for (int base = blockIdx.x * 16; base < geo.V; base += gridDim.x * 16) {
    const bool active = base + (lane >> 1) < geo.V;
    const int s = active ? base + (lane >> 1) : 0;
    int c[4];
    site_coords(geo, s, c);
    int f[4], b[4], E = kFixMinExp, any = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      f[m] = nbr_fwd(geo, s, c, m);
      b[m] = nbr_bwd(geo, s, c, m);
      const int wf = word[f[m]], wb = word[b[m]];
      any |= wf | wb;
      E = max(E, max(wf & 0x7ff, wb & 0x7ff));
    }
    const bool slow = bad || (any & kFixSlow);
    cplx<double> v[6];
    fix_dir_site<DAG>(geo, acc, s, c, f, b, E, slow, lane, dir, kappa, part, v);
    if (dir == 0) epi.apply(geo.V, s, lane & 1, active, v, red);
    __syncthreads();
  }
  if constexpr (Epi::REDUCE) {
    double tot[1];
    if (grid_sum<1>(red, rs, tot)) epi.finalize(tot);
  }
}

// Opts a kernel in to the shared memory of the copying stencil, once per device; its resident
// blocks there.  `cache`: one slot per device, kept with the kernel's launcher.
constexpr int kFixDevices = 64;
inline int fix_wave(const void* kernel, int block, std::atomic<int> (&cache)[kFixDevices]) {
  int dev = 0;
  cudaGetDevice(&dev);
  std::atomic<int>& slot = cache[dev & (kFixDevices - 1)];
  int wave = slot.load(std::memory_order_acquire);
  if (wave == 0) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fix_smem(block));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, fix_smem(block));
    wave = sm_count() * std::max(1, per_sm);
    slot.store(wave, std::memory_order_release);
  }
  return wave;
}

// Blocks of 256 threads (128 sites), two per SM; measured slower: 64-site blocks at the same occupancy (286
// against 241 us at 24^3 x 32: fewer of the x and y neighbours are in the block's own lines),
// three blocks of 80 registers (344, spills), blocks of 4 x 4 x 4 x 2 sites (304: shorter runs per
// load).  Operands copied ahead (fix_hops_async): 254 instead of 300 us for CG pass 1 there, 290 instead of
// 342 for pass 2, M^dag M at 32^3 x 64 2.68 instead of 3.6 ms.
// Internal linkage: every translation unit launches its own instance of the kernel and has to opt
// that instance in (a count cached across units would leave the others at the default shared memory).
template <bool DAG, class Epi, int BS>
static void launch_fix_async(const Geom& geo, const FixGauge& U, SpinorRef in, double kappa, const Epi& epi,
                             const ReduceScratch& rs, cudaStream_t stream) {
  static std::atomic<int> waves[kFixDevices];
  const int wave = fix_wave(reinterpret_cast<const void*>(&dslash_fix_kernel<DAG, Epi, BS>), BS, waves);
  launch_pdl(&dslash_fix_kernel<DAG, Epi, BS>, std::min(grid_for(2 * geo.V, BS), wave), BS, fix_smem(BS), stream, geo, U, in,
             kappa, epi, rs);
}

// Threads per block for V sites: the SM with most work has ceil(blocks / SMs) of them, which at a few
// blocks per SM is well above the average; blocks of 128 where that SM then has at least 5% less to
// do (12^4: 3 of 128 instead of 2 of 256, FP64 CG iteration 58 -> 50 us; 16^4: 7 instead of 4, pass 1
// 47 -> 44 us; blocks of 64 were no better: 51 us at 12^4).
inline int fix_block(int V) {
  static const int sms = sm_count();
  constexpr int half = kFixBlock / 2;
  const long long full = 2ll * grid_for(grid_for(2 * V, kFixBlock), sms), small = grid_for(grid_for(2 * V, half), sms);
  return 20 * small < 19 * full ? half : kFixBlock;
}

template <bool DAG, class Epi>
static void launch_dslash_fix(const Geom& geo, const FixGauge& U, SpinorRef in, double kappa, const Epi& epi,
                              const ReduceScratch& rs, cudaStream_t stream) {
  if (geo.V <= kFixDirSites) {
    static const int dir_wave = resident_grid(reinterpret_cast<const void*>(&dslash_fix_dir_kernel<DAG, Epi>), 128);
    launch_pdl(&dslash_fix_dir_kernel<DAG, Epi>, std::min(grid_for(geo.V, 16), dir_wave), 128, 0, stream, geo, U, in,
               kappa, epi, rs);
    return;
  }
  switch (fix_block(geo.V)) {
    case 128: launch_fix_async<DAG, Epi, 128>(geo, U, in, kappa, epi, rs, stream); break;
    default: launch_fix_async<DAG, Epi, 256>(geo, U, in, kappa, epi, rs, stream); break;
  }
}

}  // namespace lq
