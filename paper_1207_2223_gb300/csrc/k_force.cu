// Fermion force (paper Sec. 3, kernel 3: the driving force of the fermion
// fields, fused with the momentum evolution; fixed point, lq_fix64.cuh), and the pseudofermion-action
// difference used in Delta H (Eq. 5).  FP64.
//
// With X = (M^dag M)^{-1} phi and Y = M X, the derivative of
// S_f = phi^dag (M^dag M)^{-1} phi under U_mu(x) -> exp(i w t_a) U_mu(x) is
//   F_a(x, mu) = 2 kappa s Im tr(t_a Q),
//   Q = sum_spin [ X(x) (U (1 + g_mu) Y(x+mu))^dag - U X(x+mu) ((1 - g_mu) Y(x))^dag ],
// s the sign of the hop x -> x+mu.  (1 -+ g_mu) has rank 2, so each spin sum
// reduces to two colour outer products of projected half spinors
// (sum_spin conj(((1+S g) a)_s) b_s = conj(h(a)_0) h(b)_0 + conj(h(a)_1) h(b)_1,
// h = the two independent components of the projection), which is the
// paper's observation that the gamma algebra leaves few non-zero terms.
#include "lq_internal.h"
#include "lq_su3.cuh"
#include "lq_fixsu3.cuh"

namespace lq {

static constexpr int kBS = 256;

template <int MU>
__device__ __forceinline__ M3 force_matrix(const cplx<double> Xx[12], const cplx<double> Yx[12],
                                           const cplx<double> Xf[12], const cplx<double> Yf[12], const M3& U) {
  cplx<double> a0[3], a1[3], b0[3], b1[3];
  M3 Q;
#pragma unroll
  for (int k = 0; k < 9; ++k) Q.m[k] = {0.0, 0.0};
  // A = sum_k (U h(X(x+mu))_k) h(Y(x))_k^dag with (1 - g_mu)
  project<MU, -1>(Xf, a0, a1);
  project<MU, -1>(Yx, b0, b1);
  cplx<double> u0[3], u1[3];
  su3_mul(U.m, a0, u0);
  su3_mul(U.m, a1, u1);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cplx<double> t = cjmul(b0[j], u0[i]);       // u0_i conj(b0_j)
      t = cjmadd(t, b1[j], u1[i]);
      Q.m[3 * i + j] = Q.m[3 * i + j] - t;
    }
  // B = sum_k h(X(x))_k (U h(Y(x+mu))_k)^dag with (1 + g_mu)
  project<MU, +1>(Xx, a0, a1);
  project<MU, +1>(Yf, b0, b1);
  su3_mul(U.m, b0, u0);
  su3_mul(U.m, b1, u1);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cplx<double> t = cjmul(u0[j], a0[i]);       // a0_i conj((U b0)_j)
      t = cjmadd(t, u1[j], a1[i]);
      Q.m[3 * i + j] = Q.m[3 * i + j] + t;
    }
  return Q;
}

// The FP64 path of a link: f_a of force_matrix.
static __device__ __noinline__ void force_link64(Geom geo, const double2* g, SpinorRef X, SpinorRef Y, int mu, int s,
                                                 int xf, double* fa) {
  cplx<double> Xx[12], Yx[12], Xf[12], Yf[12];
  load_spinor<SStore::F64, double>(X, geo.V, s, Xx);
  load_spinor<SStore::F64, double>(Y, geo.V, s, Yx);
  load_spinor<SStore::F64, double>(X, geo.V, xf, Xf);
  load_spinor<SStore::F64, double>(Y, geo.V, xf, Yf);
  const M3 U = load_m3(g, geo.V, mu, s);
  M3 Q;
  switch (mu) {
    case 0: Q = force_matrix<0>(Xx, Yx, Xf, Yf, U); break;
    case 1: Q = force_matrix<1>(Xx, Yx, Xf, Yf, U); break;
    case 2: Q = force_matrix<2>(Xx, Yx, Xf, Yf, U); break;
    default: Q = force_matrix<3>(Xx, Yx, Xf, Yf, U); break;
  }
  im_tr_ta(Q, fa);
}

// Projection (1 + S g_mu) of the spinor of site n in fixed point with exponent word e2 (project), signed limbs.
template <int MU, int S>
__device__ __forceinline__ void fix_project(const double2* f, int V, int n, unsigned e2, FixRow& h0, FixRow& h1) {
  constexpr int P = S > 0 ? 0 : -1, N = ~P;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    FixTerm re[4], im[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double2 w = __ldg(f + (size_t)(3 * k + c) * V + n);
      re[k] = fix_of(w.x, e2);
      im[k] = fix_of(w.y, e2);
    }
    if constexpr (MU == 0) {           // p0 + S i p3, p1 + S i p2
      h0.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[0], 0, im[3], N));
      h0.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[0], 0, re[3], P));
      h1.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[1], 0, im[2], N));
      h1.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[1], 0, re[2], P));
    } else if constexpr (MU == 1) {    // p0 - S p3, p1 + S p2
      h0.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[0], 0, re[3], N));
      h0.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[0], 0, im[3], N));
      h1.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[1], 0, re[2], P));
      h1.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[1], 0, im[2], P));
    } else if constexpr (MU == 2) {    // p0 + S i p2, p1 - S i p3
      h0.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[0], 0, im[2], N));
      h0.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[0], 0, re[2], P));
      h1.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[1], 0, im[3], P));
      h1.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[1], 0, re[3], N));
    } else {                           // p0 + S p2, p1 + S p3
      h0.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[0], 0, re[2], P));
      h0.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[0], 0, im[2], P));
      h1.re[c] = fix_limbs_signed(fix_add<kLimbBias>(re[1], 0, re[3], P));
      h1.im[c] = fix_limbs_signed(fix_add<kLimbBias>(im[1], 0, im[3], P));
    }
  }
}

// The sums Im tr(t_a Q) is made of: Im(Q_ij + Q_ji), Re(Q_ij - Q_ji) for (01), (02), (12), then Im Q_ii.
struct ForceSums {
  long long pair[3][2], diag[3];
};
// + a b^dag, in units of 2^60 of the product of the operands' units: two bits finer than the first
// column, so that the four roundings of a sum are a quarter of what FP64 products cost
__device__ __forceinline__ long long force_join(long long h, long long m) { return (h << 2) + (m >> 29); }
__device__ __forceinline__ void force_outer(const FixRow& a, const FixRow& b, ForceSums& f) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
    long long h = 0, m = 1 << 28;       // Im T_ij + Im T_ji, T_ij = a_i conj(b_j)
    fix_mac(h, m, a.im[i].x, a.im[i].y, b.re[j]);
    fix_mac(h, m, -a.re[i].x, -a.re[i].y, b.im[j]);
    fix_mac(h, m, a.im[j].x, a.im[j].y, b.re[i]);
    fix_mac(h, m, -a.re[j].x, -a.re[j].y, b.im[i]);
    f.pair[q][0] += force_join(h, m);
    h = 0;
    m = 1 << 28;                        // Re T_ij - Re T_ji
    fix_mac(h, m, a.re[i].x, a.re[i].y, b.re[j]);
    fix_mac(h, m, a.im[i].x, a.im[i].y, b.im[j]);
    fix_mac(h, m, -a.re[j].x, -a.re[j].y, b.re[i]);
    fix_mac(h, m, -a.im[j].x, -a.im[j].y, b.im[i]);
    f.pair[q][1] += force_join(h, m);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    long long h = 0, m = 1 << 28;
    fix_mac(h, m, a.im[i].x, a.im[i].y, b.re[i]);
    fix_mac(h, m, -a.re[i].x, -a.re[i].y, b.im[i]);
    f.diag[i] += force_join(h, m);
  }
}
// U h in half the unit of h, NEG: - U h
template <bool NEG>
__device__ __forceinline__ FixRow fix_matvec(const Fix3& u, const FixRow& h) {
  FixRow r;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    long long rh = kLimbBias, rm = 1 << 30, ih = kLimbBias, im = 1 << 30;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int4 e = u.m[3 * i + j];
      fix_mac(rh, rm, e.x, e.y, h.re[j]);
      fix_mac(rh, rm, -e.z, -e.w, h.im[j]);
      fix_mac(ih, im, e.x, e.y, h.im[j]);
      fix_mac(ih, im, e.z, e.w, h.re[j]);
    }
    r.re[i] = fix_limbs_signed(rh + (rm >> 31));
    r.im[i] = fix_limbs_signed(ih + (im >> 31));
    if constexpr (NEG) {
      r.re[i] = neg2(r.re[i]);
      r.im[i] = neg2(r.im[i]);
    }
  }
  return r;
}

template <int MU>
__device__ __forceinline__ void force_sums(const double2* X, const double2* Y, const int4* g, int V, int s, int xf,
                                           unsigned ex, unsigned exf, unsigned ey, unsigned eyf, ForceSums& f) {
  const Fix3 U = load_fix3(g, V, MU, s);
  FixRow a0, a1, b0, b1;
  // - (U h(X(x+mu))) h(Y(x))^dag with (1 - g_mu)
  fix_project<MU, -1>(X, V, xf, exf, a0, a1);
  a0 = fix_matvec<true>(U, a0);
  a1 = fix_matvec<true>(U, a1);
  fix_project<MU, -1>(Y, V, s, ey, b0, b1);
  force_outer(a0, b0, f);
  force_outer(a1, b1, f);
  // + h(X(x)) (U h(Y(x+mu)))^dag with (1 + g_mu)
  fix_project<MU, +1>(Y, V, xf, eyf, b0, b1);
  b0 = fix_matvec<false>(U, b0);
  b1 = fix_matvec<false>(U, b1);
  fix_project<MU, +1>(X, V, s, ex, a0, a1);
  force_outer(a0, b0, f);
  force_outer(a1, b1, f);
}

// One thread per link, fixed point (lq_fix64.cuh) with an exponent for each of its four spinors.  The two
// terms X(x+mu) Y(x) and X(x) Y(x+mu) need a common unit: the one with the smaller exponent sum takes
// its X in a larger unit, which drops only bits below the other term's last.  (One exponent for both X
// and one for both Y lost the square of the ratio where a field falls from site to site: 1.7e-15 at an
// eighth.)  Links whose spinors or matrix do not fit take FP64 arithmetic.  Only the sums the generators
// ask for are formed (30 of the 36 real products of an outer product).
// |h| < 2^60.3 and |U h| < 2^59.3 as vectors: a sum of four products is below 2^57.6 in the first column,
// the four of them 2^61.6 in units of 2^60; 2^61.3 in the middle column.
// FP64 arithmetic took 212 clocks per link and SM (24^3 x 32: 1.27 ms); 0.54 ms here.  Error against extended
// precision (2-norm of a link): 0.9e-16, FP64 arithmetic 1.8e-16, at any fall from site to site.
template <bool UPDATE>
__global__ void __launch_bounds__(128, 2) fermion_force_kernel(Geom geo, FixGauge G, SpinorRef X, SpinorRef Y, double* f,
                                                               double kappa, double eps) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4 * geo.V) return;
  const int mu = idx / geo.V, s = idx - mu * geo.V;
  int c[4];
  site_coords(geo, s, c);
  const int xf = nbr_fwd(geo, s, c, mu);
  const double sign = (mu == 3 && geo.antiperiodic && c[3] == geo.L[3] - 1) ? -1.0 : 1.0;
  const int *wx = reinterpret_cast<const int*>(X.norm), *wy = reinterpret_cast<const int*>(Y.norm);
  const int x0 = __ldg(wx + s), x1 = __ldg(wx + xf), y0 = __ldg(wy + s), y1 = __ldg(wy + xf);
  double fa[8];
  if (__ldg(G.flags + kFixBad) || ((x0 | x1 | y0 | y1) & kFixSlow)) {
    force_link64(geo, G.f64, X, Y, mu, s, xf, fa);
  } else {
    // exponents of X(x+mu), Y(x) and X(x), Y(x+mu); 60 places up nothing of a term is left.  A word holds
    // exponents to 2047: what X cannot take goes to Y.
    int e[4] = {max(kFixMinExp, x1), max(kFixMinExp, y0), max(kFixMinExp, x0), max(kFixMinExp, y1)};
    const int d = e[0] + e[1] - e[2] - e[3], up = min(abs(d), 60);
    const int EX = d > 0 ? e[0] : e[2], EY = d > 0 ? e[1] : e[3];
    const int dx = min(up, 2047 - (d > 0 ? e[2] : e[0]));
    if (d > 0) { e[2] += dx; e[3] += up - dx; }
    else { e[0] += dx; e[1] += up - dx; }
    auto word = [](int E) { return (unsigned)E << 21 | 0x1fffffu; };
    const unsigned exf = word(e[0]), ey = word(e[1]), ex = word(e[2]), eyf = word(e[3]);
    const double2 *px = static_cast<const double2*>(X.p), *py = static_cast<const double2*>(Y.p);
    ForceSums q{};
    switch (mu) {
      case 0: force_sums<0>(px, py, G.fix, geo.V, s, xf, ex, exf, ey, eyf, q); break;
      case 1: force_sums<1>(px, py, G.fix, geo.V, s, xf, ex, exf, ey, eyf, q); break;
      case 2: force_sums<2>(px, py, G.fix, geo.V, s, xf, ex, exf, ey, eyf, q); break;
      default: force_sums<3>(px, py, G.fix, geo.V, s, xf, ex, exf, ey, eyf, q); break;
    }
    // unit of the sums: 2^60 * 2 * 2^(EX - 1080) * 2^(EY - 1080), in two factors that do not underflow
    const double ux = __hiloint2double((EX - 26) << 20, 0), uy = __hiloint2double((EY - 27) << 20, 0);
    const double r2 = 0.70710678118654752440 * ux, r6 = 0.40824829046386301637 * ux;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int t = 0; t < 2; ++t) fa[(p == 0 ? 0 : p == 1 ? 3 : 5) + t] = r2 * (double)q.pair[p][t] * uy;
    fa[2] = r2 * (double)(q.diag[0] - q.diag[1]) * uy;
    fa[7] = r6 * ((double)(q.diag[0] - q.diag[2]) + (double)(q.diag[1] - q.diag[2])) * uy;
  }
  const double sc = 2.0 * kappa * sign;
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    double* q = f + ((size_t)mu * 8 + a) * geo.V + s;
    if (UPDATE) *q -= eps * sc * fa[a];
    else *q = sc * fa[a];
  }
}

// out[0] = sum_x [ Re phi(x)^dag X(x) - |chi(x)|^2 ]
__global__ void __launch_bounds__(kBS) fermion_action_diff_kernel(int V, SpinorRef phi, SpinorRef X, SpinorRef chi,
                                                                  ReduceScratch rs, double* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  double red[1] = {0.0};
  if (s < V) {
    cplx<double> a[12], b[12], c[12];
    load_spinor<SStore::F64, double>(phi, V, s, a);
    load_spinor<SStore::F64, double>(X, V, s, b);
    load_spinor<SStore::F64, double>(chi, V, s, c);
#pragma unroll
    for (int k = 0; k < 12; ++k) red[0] += (a[k].re * b[k].re + a[k].im * b[k].im) - norm2(c[k]);
  }
  double tot[1];
  if (grid_sum<1>(red, rs, tot)) out[0] = tot[0];
}

// Complex gradient of S_f with respect to the entries of U_mu(x) in the
// convention dS = Re sum conj(G) dU (that of torch.autograd):
//   G = conj(2 kappa s C),  C_ij = sum_spin conj(((1 - g_mu) Y(x))_i) X(x+mu)_j
//                                + sum_spin conj(X(x)_i) ((1 + g_mu) Y(x+mu))_j,
// each spin sum again over the two half-spinor components.  G is written in
// the canonical layout [V][4][3][3] complex.
template <int MU>
__device__ __forceinline__ M3 grad_matrix(const cplx<double> Xx[12], const cplx<double> Yx[12],
                                          const cplx<double> Xf[12], const cplx<double> Yf[12]) {
  cplx<double> a0[3], a1[3], b0[3], b1[3];
  M3 C;
  project<MU, -1>(Yx, a0, a1);
  project<MU, -1>(Xf, b0, b1);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cplx<double> t = cjmul(a0[i], b0[j]);
      C.m[3 * i + j] = cjmadd(t, a1[i], b1[j]);
    }
  project<MU, +1>(Xx, a0, a1);
  project<MU, +1>(Yf, b0, b1);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cplx<double> t = cjmadd(C.m[3 * i + j], a0[i], b0[j]);
      C.m[3 * i + j] = cjmadd(t, a1[i], b1[j]);
    }
  return C;
}

__global__ void __launch_bounds__(kBS) fermion_grad_kernel(Geom geo, SpinorRef X, SpinorRef Y, double2* G,
                                                           double kappa) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4 * geo.V) return;
  const int mu = idx / geo.V, s = idx - mu * geo.V;
  int c[4];
  site_coords(geo, s, c);
  const int xf = nbr_fwd(geo, s, c, mu);
  const double sign = (mu == 3 && geo.antiperiodic && c[3] == geo.L[3] - 1) ? -1.0 : 1.0;
  cplx<double> Xx[12], Yx[12], Xf[12], Yf[12];
  load_spinor<SStore::F64, double>(X, geo.V, s, Xx);
  load_spinor<SStore::F64, double>(Y, geo.V, s, Yx);
  load_spinor<SStore::F64, double>(X, geo.V, xf, Xf);
  load_spinor<SStore::F64, double>(Y, geo.V, xf, Yf);
  M3 C;
  switch (mu) {
    case 0: C = grad_matrix<0>(Xx, Yx, Xf, Yf); break;
    case 1: C = grad_matrix<1>(Xx, Yx, Xf, Yf); break;
    case 2: C = grad_matrix<2>(Xx, Yx, Xf, Yf); break;
    default: C = grad_matrix<3>(Xx, Yx, Xf, Yf); break;
  }
  const double sc = 2.0 * kappa * sign;
  double2* out = G + ((size_t)s * 4 + mu) * 9;
#pragma unroll
  for (int k = 0; k < 9; ++k) out[k] = make_double2(sc * C.m[k].re, -sc * C.m[k].im);
}

// out[0] = sum_x Re phi(x)^dag X(x)
__global__ void __launch_bounds__(kBS) dot_re_kernel(int V, SpinorRef a, SpinorRef b, ReduceScratch rs,
                                                     double* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  double red[1] = {0.0};
  if (s < V) {
    cplx<double> u[12], v[12];
    load_spinor<SStore::F64, double>(a, V, s, u);
    load_spinor<SStore::F64, double>(b, V, s, v);
#pragma unroll
    for (int k = 0; k < 12; ++k) red[0] += u[k].re * v[k].re + u[k].im * v[k].im;
  }
  double tot[1];
  if (grid_sum<1>(red, rs, tot)) out[0] = tot[0];
}

void launch_fermion_grad(const Geom& g, SpinorRef X, SpinorRef Y, double* G, double kappa, cudaStream_t st) {
  fermion_grad_kernel<<<grid_for(4 * g.V, kBS), kBS, 0, st>>>(g, X, Y, reinterpret_cast<double2*>(G), kappa);
}
void launch_dot_re(const Geom& g, SpinorRef a, SpinorRef b, const ReduceScratch& rs, double* out, cudaStream_t st) {
  dot_re_kernel<<<grid_for(g.V, kBS), kBS, 0, st>>>(g.V, a, b, rs, out);
}

void launch_fermion_force(const Geom& g, const FixGauge& U, SpinorRef X, SpinorRef Y, double* f, double kappa,
                          double eps, bool update, cudaStream_t st) {
  const int grid = grid_for(4 * g.V, 128);
  if (update) fermion_force_kernel<true><<<grid, 128, 0, st>>>(g, U, X, Y, f, kappa, eps);
  else fermion_force_kernel<false><<<grid, 128, 0, st>>>(g, U, X, Y, f, kappa, eps);
}
void launch_fermion_action_diff(const Geom& g, SpinorRef phi, SpinorRef X, SpinorRef chi, const ReduceScratch& rs,
                                double* out, cudaStream_t st) {
  fermion_action_diff_kernel<<<grid_for(g.V, kBS), kBS, 0, st>>>(g.V, phi, X, chi, rs, out);
}

}  // namespace lq
