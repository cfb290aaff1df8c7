// Gauge-side kernels of the molecular dynamics (paper Sec. 3, kernels 2 and 4;
// Eq. 5): plaquettes and the Wilson gauge action, the gauge force fused with
// the momentum update, the link update U <- exp(i eps p) U with
// reunitarisation, and the kinetic-energy difference.  All FP64; plaquettes and
// staples multiply links in fixed point (lq_fixsu3.cuh), and in FP64 arithmetic
// when some link is not unitary (staples also where the field is smooth).
//
// Momenta and forces are stored site-major as double [32][V], entry
// (4 mu + ... ) -> index (8 mu + a) * V + site, for su(3) coefficient a.
#include "lq_internal.h"
#include "lq_su3.cuh"
#include "lq_fixsu3.cuh"

namespace lq {

static constexpr int kBS = 256;

__device__ __forceinline__ double site_plaquettes(const double2* g, const Geom& geo, int s, const int c[4]) {
  double sum = 0.0;
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    const int xm = nbr_fwd(geo, s, c, mu);
    const M3 Umu = load_m3(g, geo.V, mu, s);
#pragma unroll 1
    for (int nu = mu + 1; nu < 4; ++nu) {
      const int xn = nbr_fwd(geo, s, c, nu);
      // Re tr(U_mu(x) U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag) = Re tr[(U_mu(x) U_nu(x+mu)) (U_nu(x) U_mu(x+nu))^dag]
      const M3 a = mul(Umu, load_m3(g, geo.V, nu, xm));
      const M3 b = mul(load_m3(g, geo.V, nu, s), load_m3(g, geo.V, mu, xn));
      sum += re_tr_mul_dag(a, b);
    }
  }
  return sum;
}

static __device__ __noinline__ double site_plaquettes64(const double2* g, Geom geo, int s) {
  int c[4];
  site_coords(geo, s, c);
  return site_plaquettes(g, geo, s, c);
}

// out[0] = sum_x sum_{mu<nu} Re tr U_P with fixed-point links: per site the two-link products of
// both paths row by row and their scalar product, summed exactly in units of 2^-58; links that are not unitary
// in FP64 arithmetic.  24^3 x 32: 1.19 ms in FP64 arithmetic (1400 multiply-adds per site at 2 per clock and
// SM), 0.31 ms in fixed point.
__global__ void __launch_bounds__(kFixBlock, 2) plaquette_kernel(Geom geo, FixGauge U, ReduceScratch rs,
                                                                     double* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  const int4* __restrict__ g = U.fix;
  double red[1] = {0.0};
  if (__ldg(U.flags + kFixBad)) {
    if (s < geo.V) red[0] = site_plaquettes64(U.f64, geo, s);
  } else if (s < geo.V) {
    int c[4];
    site_coords(geo, s, c);
    long long sum = 0;
#pragma unroll 1
    for (int mu = 0; mu < 3; ++mu) {
      const int xm = nbr_fwd(geo, s, c, mu);
#pragma unroll 1
      for (int nu = mu + 1; nu < 4; ++nu) {
        const int xn = nbr_fwd(geo, s, c, nu);
        const Fix3 p = load_fix3(g, geo.V, nu, xm), q = load_fix3(g, geo.V, mu, xn);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          long long a[3][2], b[3][2];
          fix_vecmat<false>(fix_row(g, geo.V, mu, s, i), p, a);
          fix_vecmat<false>(fix_row(g, geo.V, nu, s, i), q, b);
          const FixRow x = fix_split_signed(a), y = fix_split(b);
          long long h = 0, m = 1 << 30;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            fix_mac(h, m, x.re[k].x, x.re[k].y, y.re[k]);
            fix_mac(h, m, x.im[k].x, x.im[k].y, y.im[k]);
          }
          sum += h + (m >> 31);
        }
      }
    }
    red[0] = (double)sum * 0x1p-58;
  }
  double tot[1];
  if (grid_sum<1>(red, rs, tot)) out[0] = tot[0];
}

// out[0] = sum_x sum_{mu<nu} Re tr U_P (gauge a), out[1] = the same minus that of gauge b, site by site; FP64.
__global__ void __launch_bounds__(kBS) plaquette_diff_kernel(Geom geo, const double2* ga, const double2* gb,
                                                             ReduceScratch rs, double* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  double red[2] = {0.0, 0.0};
  if (s < geo.V) {
    int c[4];
    site_coords(geo, s, c);
    const double pa = site_plaquettes(ga, geo, s, c);
    red[0] = pa;
    red[1] = pa - site_plaquettes(gb, geo, s, c);
  }
  double tot[2];
  if (grid_sum<2>(red, rs, tot)) { out[0] = tot[0]; out[1] = tot[1]; }
}

// Im tr(t_a U_mu(x) Sigma_mu(x)) in FP64 arithmetic, Sigma the six staples.
static __device__ __noinline__ void gauge_link64(Geom geo, const double2* g, int mu, int s, double* fa) {
  int c[4];
  site_coords(geo, s, c);
  const int xm = nbr_fwd(geo, s, c, mu);
  int cm[4] = {c[0], c[1], c[2], c[3]};
  cm[mu] = (c[mu] + 1) % geo.L[mu];
  M3 S;
#pragma unroll
  for (int k = 0; k < 9; ++k) S.m[k] = {0.0, 0.0};
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    const int xn = nbr_fwd(geo, s, c, nu);
    const int xmn = nbr_bwd(geo, s, c, nu);          // x - nu
    const int xpm_mn = nbr_bwd(geo, xm, cm, nu);     // x + mu - nu
    // upper: U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
    M3 up = mul_dag(load_m3(g, geo.V, nu, xm), load_m3(g, geo.V, mu, xn));
    up = mul_dag(up, load_m3(g, geo.V, nu, s));
    add_to(S, up);
    // lower: U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu) = (U_mu(x-nu) U_nu(x+mu-nu))^dag U_nu(x-nu)
    M3 lo = mul(load_m3(g, geo.V, mu, xmn), load_m3(g, geo.V, nu, xpm_mn));
    lo = dag_mul(lo, load_m3(g, geo.V, nu, xmn));
    add_to(S, lo);
  }
  im_tr_ta(mul(load_m3(g, geo.V, mu, s), S), fa);
}

// The same in fixed point, q_a 2^-57 without the generators' norms.  The rows of a staple are independent
// chains of two row-vector products, so one plane needs two links in registers (72) and one row at a time
// of the third; the staple sum is 18 64-bit integers.  Units: staples 2^-59, their sum 2^-58 after a
// shift, W = U Sigma 2^-57; |Sigma| <= 6 keeps every sum in 63 bits.
__device__ __forceinline__ void gauge_link_fix(const Geom& geo, const int4* __restrict__ g, int mu, int s,
                                               long long (&q)[8]) {
  int c[4];
  site_coords(geo, s, c);
  const int xm = nbr_fwd(geo, s, c, mu);
  int cm[4] = {c[0], c[1], c[2], c[3]};
  cm[mu] = (c[mu] + 1) % geo.L[mu];
  long long S[3][3][2] = {};
#pragma unroll 1
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    {
      // upper: U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
      const Fix3 b = load_fix3(g, geo.V, mu, nbr_fwd(geo, s, c, nu)), d = load_fix3(g, geo.V, nu, s);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        long long w[3][2], v[3][2];
        fix_vecmat<true>(fix_row(g, geo.V, nu, xm, i), b, w);
        fix_vecmat<true>(fix_split(w), d, v);
#pragma unroll
        for (int j = 0; j < 3; ++j) { S[i][j][0] += v[j][0]; S[i][j][1] += v[j][1]; }
      }
    }
    {
      // lower: U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
      const int xmn = nbr_bwd(geo, s, c, nu), xpm = nbr_bwd(geo, xm, cm, nu);
      const Fix3 b = load_fix3(g, geo.V, mu, xmn), d = load_fix3(g, geo.V, nu, xmn);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        long long w[3][2], v[3][2];
        fix_vecmat<true>(fix_row_dag(g, geo.V, nu, xpm, i), b, w);
        fix_vecmat<false>(fix_split(w), d, v);
#pragma unroll
        for (int j = 0; j < 3; ++j) { S[i][j][0] += v[j][0]; S[i][j][1] += v[j][1]; }
      }
    }
  }
  // W = U Sigma
  FixRow R[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      R[k].re[j] = fix_limbs(S[k][j][0] >> 1);
      R[k].im[j] = fix_limbs(S[k][j][1] >> 1);
    }
  long long W[3][3][2];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const FixRow u = fix_row(g, geo.V, mu, s, i);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      long long rh = 0, rm = 1 << 30, ih = 0, im = 1 << 30;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        fix_mac(rh, rm, u.re[k].x, u.re[k].y, R[k].re[j]);
        fix_mac(rh, rm, -u.im[k].x, -u.im[k].y, R[k].im[j]);
        fix_mac(ih, im, u.re[k].x, u.re[k].y, R[k].im[j]);
        fix_mac(ih, im, u.im[k].x, u.im[k].y, R[k].re[j]);
      }
      W[i][j][0] = rh + (rm >> 31);
      W[i][j][1] = ih + (im >> 31);
    }
  }
  // Im tr(t_a W) (im_tr_ta), the sums of matrix elements exact
  q[0] = W[0][1][1] + W[1][0][1];
  q[1] = W[0][1][0] - W[1][0][0];
  q[2] = W[0][0][1] - W[1][1][1];
  q[3] = W[0][2][1] + W[2][0][1];
  q[4] = W[0][2][0] - W[2][0][0];
  q[5] = W[1][2][1] + W[2][1][1];
  q[6] = W[1][2][0] - W[2][1][0];
  q[7] = W[0][0][1] + W[1][1][1] - 2 * W[2][2][1];
}

// F_a(x, mu) = (beta/3) Im tr(t_a U_mu(x) Sigma_mu(x)).  UPDATE: p -= eps F, otherwise F is stored.
//
// One thread per link, in fixed point: 1404 real products per link took 770 clocks per link and SM on the
// FP64 pipe (24^3 x 32: 4.65 ms); 1.28 ms here, now bound by load latency at 8 warps per SM
// (168 registers for 12 warps spill: 1.36 ms; 128: 1.51 ms).
//
// FP64 arithmetic where fixed point would know less than it.  Links that are not unitary (kFixBad).  Links of a
// smooth field: an absolute error of 4e-18 in each q is 1.5e-16 of the force, as much as FP64 products
// leave, where the largest q is 2^-3, and only near real diagonal links do FP64 products get better than
// that, because their small imaginary parts keep their own digits.  So a link goes to FP64 arithmetic
// with q below 2^-3 and its matrix within 2^-5 of real diagonal, and without trying fixed point
// when every link of the lattice is that close (no kFixRough).  Error against extended precision, fixed / FP64:
// roughness 0.3 2.9e-18 / 1.7e-16, 0.01 4.5e-17 / 1.5e-16, 0.003 1.5e-16 / 1.5e-16, 1e-4 4.5e-15 /
// 1.5e-16.  The check of q costs nothing measurable; one of the matrix before the staples cost 26%.
template <bool UPDATE>
__global__ void __launch_bounds__(128, 2) gauge_force_kernel(Geom geo, FixGauge U, double* f, double beta, double eps) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4 * geo.V) return;
  const int mu = idx / geo.V, s = idx - mu * geo.V;
  double fa[8];
  bool fp64 = __ldg(U.flags + kFixBad) || !__ldg(U.flags + kFixRough);
  if (!fp64) {
    long long q[8], top = 0;
    gauge_link_fix(geo, U.fix, mu, s, q);
#pragma unroll
    for (int a = 0; a < 8; ++a) top = max(top, llabs(q[a]));
    const double r2 = 0.70710678118654752440 * 0x1p-57, r6 = 0.40824829046386301637 * 0x1p-57;
#pragma unroll
    for (int a = 0; a < 8; ++a) fa[a] = (a == 7 ? r6 : r2) * (double)q[a];
    if (top < 1ll << 54) {
      int far = 0;
#pragma unroll
      for (int k = 0; k < 9; ++k) far = max(far, fix_far(__ldg(U.fix + ((size_t)mu * 9 + k) * geo.V + s), k));
      fp64 = far < kFixSmooth;
    }
  }
  if (fp64) gauge_link64(geo, U.f64, mu, s, fa);
  const double sc = beta / 3.0;
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    double* q = f + ((size_t)mu * 8 + a) * geo.V + s;
    if (UPDATE) *q -= eps * sc * fa[a];
    else *q = sc * fa[a];
  }
}

// U_mu(x) <- reunitarise(exp(i eps P) U_mu(x)), P = sum_a p_a t_a (lq_su3.cuh).  Bound by the
// FP64 pipe (2 operations per clock and SM): 24^3 x 32 2.07 ms with the closed form of the
// exponential for every link (~700 operations), 1.16 ms with the series and two of three rows.
__global__ void __launch_bounds__(kBS) link_update_kernel(Geom geo, double2* g, const double* p, double eps) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4 * geo.V) return;
  const int mu = idx / geo.V, s = idx - mu * geo.V;
  double pa[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) pa[a] = p[((size_t)mu * 8 + a) * geo.V + s];
  const double r2 = 0.70710678118654752440 * eps, r6 = 0.40824829046386301637 * eps;
  const double x = r2 * pa[2], y = r6 * pa[7];
  const H3 q{{y + x, y - x, -2.0 * y}, {r2 * pa[0], -r2 * pa[1]}, {r2 * pa[3], -r2 * pa[4]}, {r2 * pa[5], -r2 * pa[6]}};
  // Q^2, c1 = tr(Q^2) / 2, c0 = det Q = tr(Q^3) / 3
  const double n01 = norm2(q.u01), n02 = norm2(q.u02), n12 = norm2(q.u12);
  H3 q2;
  q2.d[0] = fma(q.d[0], q.d[0], n01 + n02);
  q2.d[1] = fma(q.d[1], q.d[1], n01 + n12);
  q2.d[2] = fma(q.d[2], q.d[2], n02 + n12);
  // (Q^2)_01 = Q01 (Q00 + Q11) + Q02 conj(Q12) = -Q22 Q01 + ..., the trace being zero
  const cplx<double> t01 = cjmul(q.u12, q.u02), t02 = cmul(q.u01, q.u12), t12 = cjmul(q.u01, q.u02);
  q2.u01 = {fma(-q.d[2], q.u01.re, t01.re), fma(-q.d[2], q.u01.im, t01.im)};
  q2.u02 = {fma(-q.d[1], q.u02.re, t02.re), fma(-q.d[1], q.u02.im, t02.im)};
  q2.u12 = {fma(-q.d[0], q.u12.re, t12.re), fma(-q.d[0], q.u12.im, t12.im)};
  const double c1 = 0.5 * (q2.d[0] + q2.d[1] + q2.d[2]);
  M3 U = load_m3_rw(g, geo.V, mu, s);
  if (c1 <= 0.75) {
    const double c0 = q.d[0] * fma(q.d[1], q.d[2], -n12) - q.d[1] * n02 - q.d[2] * n01 +
                      2.0 * (t02.re * q.u02.re + t02.im * q.u02.im);
    cplx<double> r0[3], r1[3];
    expi_rows(q, c1, c0, c1 <= 0.046875 ? 12 : 18, U.m, r0, r1, q2);
#pragma unroll
    for (int j = 0; j < 3; ++j) { U.m[j] = r0[j]; U.m[3 + j] = r1[j]; }
  } else {
    U = mul(expi_hermitian(eps_algebra(pa, eps)), U);
  }
  reunitarise(U);
  store_m3(g, geo.V, mu, s, U);
}

// canonical [V][32] <-> [32][V] through shared memory (a row of 32 padded to 33), both sides in
// contiguous runs.  One thread per site, 256 bytes apart, took 153 us (unpack) and 71 us (pack) at
// 24^3 x 32, where the bytes need 34; here 43 and 34 us.
constexpr int kMomTile = 64;
__global__ void __launch_bounds__(kBS) pack_mom_kernel(int V, const double* __restrict__ canon, double* __restrict__ soa) {
  __shared__ double sh[kMomTile * 33];
  const int s0 = blockIdx.x * kMomTile, n = min(kMomTile, V - s0);
  for (int i = threadIdx.x; i < n * 32; i += kBS) sh[(i >> 5) * 33 + (i & 31)] = canon[(size_t)s0 * 32 + i];
  __syncthreads();
  for (int i = threadIdx.x; i < kMomTile * 32; i += kBS) {
    const int sl = i & (kMomTile - 1), k = i / kMomTile;
    if (sl < n) soa[(size_t)k * V + s0 + sl] = sh[sl * 33 + k];
  }
}
__global__ void __launch_bounds__(kBS) unpack_mom_kernel(int V, const double* __restrict__ soa, double* __restrict__ canon) {
  __shared__ double sh[kMomTile * 33];
  const int s0 = blockIdx.x * kMomTile, n = min(kMomTile, V - s0);
  for (int i = threadIdx.x; i < kMomTile * 32; i += kBS) {
    const int sl = i & (kMomTile - 1), k = i / kMomTile;
    if (sl < n) sh[sl * 33 + k] = soa[(size_t)k * V + s0 + sl];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n * 32; i += kBS) canon[(size_t)s0 * 32 + i] = sh[(i >> 5) * 33 + (i & 31)];
}

// out[0] = (1/2) sum (p^2 - p0^2), per element, then summed
__global__ void __launch_bounds__(kBS) kinetic_diff_kernel(int V, const double* p, const double* p0,
                                                           ReduceScratch rs, double* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  double red[1] = {0.0};
  if (s < V) {
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      const double a = p[(size_t)k * V + s], b = p0[(size_t)k * V + s];
      red[0] += 0.5 * (a - b) * (a + b);
    }
  }
  double tot[1];
  if (grid_sum<1>(red, rs, tot)) out[0] = tot[0];
}

void launch_plaquette_diff(const Geom& g, const void* ga, const void* gb, const ReduceScratch& rs, double* out,
                           cudaStream_t st) {
  plaquette_diff_kernel<<<grid_for(g.V, kBS), kBS, 0, st>>>(g, static_cast<const double2*>(ga),
                                                            static_cast<const double2*>(gb), rs, out);
}
void launch_plaquette(const Geom& g, const FixGauge& U, const ReduceScratch& rs, double* out, cudaStream_t st) {
  plaquette_kernel<<<grid_for(g.V, kFixBlock), kFixBlock, 0, st>>>(g, U, rs, out);
}
void launch_gauge_force(const Geom& g, const FixGauge& U, double* f, double beta, double eps, bool update,
                        cudaStream_t st) {
  const int grid = grid_for(4 * g.V, 128);
  if (update) gauge_force_kernel<true><<<grid, 128, 0, st>>>(g, U, f, beta, eps);
  else gauge_force_kernel<false><<<grid, 128, 0, st>>>(g, U, f, beta, eps);
}
void launch_link_update(const Geom& g, void* gauge, const double* p, double eps, cudaStream_t st) {
  link_update_kernel<<<grid_for(4 * g.V, kBS), kBS, 0, st>>>(g, static_cast<double2*>(gauge), p, eps);
}
void launch_pack_mom(const Geom& g, const double* canon, double* soa, cudaStream_t st) {
  pack_mom_kernel<<<grid_for(g.V, kMomTile), kBS, 0, st>>>(g.V, canon, soa);
}
void launch_unpack_mom(const Geom& g, const double* soa, double* canon, cudaStream_t st) {
  unpack_mom_kernel<<<grid_for(g.V, kMomTile), kBS, 0, st>>>(g.V, soa, canon);
}
void launch_kinetic_diff(const Geom& g, const double* p, const double* p0, const ReduceScratch& rs, double* out,
                         cudaStream_t st) {
  kinetic_diff_kernel<<<grid_for(g.V, kBS), kBS, 0, st>>>(g.V, p, p0, rs, out);
}

}  // namespace lq
