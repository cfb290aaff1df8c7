// Products of SU(3) links in fixed point: the links of lq_fix64.cuh (2^61 u in
// two limbs of 31 bits) multiplied row by row with 32 x 32 + 64 bit integer
// multiply-adds, 32 times the rate of the FP64 pipe.  A row-vector times a link
// keeps its unit: with the vector's unit 2^-q the product is exact in units of
// 2^-(q - 1) up to the dropped product of the low limbs (mean zero, as one of the
// two has signed low limbs, and at most half a last place) and one rounding.  Elements of products of unitary matrices
// are at most 1, so a chain of two products starting from a link stays at 59
// fractional bits, 2^-6 of the last place of FP64.
#pragma once
#include "lq_fix64.cuh"

namespace lq {

struct Fix3 {
  int4 m[9];        // row-major, (re.hi, re.lo, im.hi, im.lo)
};
__device__ __forceinline__ Fix3 load_fix3(const int4* __restrict__ g, int V, int mu, int s) {
  Fix3 r;
  const int4* p = g + (size_t)mu * 9 * V + s;
#pragma unroll
  for (int c = 0; c < 9; ++c) r.m[c] = __ldg(p + (size_t)c * V);
  return r;
}

// A row vector of three complex numbers as limbs.
struct FixRow {
  int2 re[3], im[3];
};
// row i of a link, and row i of its adjoint (column i conjugated)
__device__ __forceinline__ FixRow fix_row(const int4* __restrict__ g, int V, int mu, int s, int i) {
  FixRow r;
  const int4* p = g + ((size_t)mu * 9 + 3 * i) * V + s;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 u = __ldg(p + (size_t)k * V);
    r.re[k] = make_int2(u.x, u.y);
    r.im[k] = make_int2(u.z, u.w);
  }
  return r;
}
__device__ __forceinline__ FixRow fix_row_dag(const int4* __restrict__ g, int V, int mu, int s, int i) {
  FixRow r;
  const int4* p = g + ((size_t)mu * 9 + i) * V + s;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 u = __ldg(p + (size_t)(3 * k) * V);
    r.re[k] = make_int2(u.x, u.y);
    r.im[k] = make_int2(-u.z, -u.w);
  }
  return r;
}
__device__ __forceinline__ int2 neg2(int2 a) { return make_int2(-a.x, -a.y); }

// w = r m (DAG: r m^dag), [column][re, im], in half the unit of r
template <bool DAG>
__device__ __forceinline__ void fix_vecmat(const FixRow& r, const Fix3& m, long long (&w)[3][2]) {
  int2 n[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) n[k] = neg2(DAG ? r.re[k] : r.im[k]);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    long long rh = 0, rm = 1 << 30, ih = 0, im = 1 << 30;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int4 u = DAG ? m.m[3 * j + k] : m.m[3 * k + j];
      fix_mac(rh, rm, u.x, u.y, r.re[k]);
      fix_mac(ih, im, u.x, u.y, r.im[k]);
      fix_mac(rh, rm, u.z, u.w, DAG ? r.im[k] : n[k]);
      fix_mac(ih, im, u.z, u.w, DAG ? n[k] : r.re[k]);
    }
    w[j][0] = rh + (rm >> 31);
    w[j][1] = ih + (im >> 31);
  }
}
__device__ __forceinline__ FixRow fix_split(const long long (&w)[3][2]) {
  FixRow r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.re[k] = fix_limbs(w[k][0]);
    r.im[k] = fix_limbs(w[k][1]);
  }
  return r;
}

// the same with signed low limbs, for an operand whose partner comes from fix_split
__device__ __forceinline__ FixRow fix_split_signed(const long long (&w)[3][2]) {
  FixRow r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.re[k] = fix_limbs_signed(w[k][0] + kLimbBias);
    r.im[k] = fix_limbs_signed(w[k][1] + kLimbBias);
  }
  return r;
}

}  // namespace lq
