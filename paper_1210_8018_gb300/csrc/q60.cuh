// q60.cuh -- products of SU(3) matrices in 60-bit fixed point on the integer pipe (the large-step double
// update, the plaquette, the gauge functional and its gradient).
#pragma once
#include "su3.cuh"

namespace lgf {

// A number of magnitude below 2 as (h 2^30 + l) 2^-60 in two 32-bit limbs. A dot product of complex vectors
// gathers the products of the high limbs in one 64-bit sum and the two cross products in another, so that a
// real multiply-add is three 32 x 32 + 64-bit multiply-adds and nothing else; the sums are joined and
// split into limbs again once per element. This GPU does two FP64 multiply-adds per SM and clock, and about
// 32 of these multiply-adds.
//
// Range: with rows a and columns b of unit length (six real entries, sum |a_k| <= 6^(1/2)) the cross sum
// stays below 2 * 2.45 * 2^60 < 2^63, and that holds up to sum |a_k| + sum |b_k| = 8. Callers send entries
// of magnitude 2 and above, infinities and NaN (lq_in_range), and matrices whose rows or columns are longer, to
// the FP64 form.
// Error: the dropped products of the low limbs are below 2^-60 each and the splits truncate by less than
// 2^-60, so an element is off by less than 2^-57 before its one rounding to double.
struct lq {
  int h, l;
};
struct clq {
  lq r, i;
};
// `top` collects the largest high word of the magnitudes converted.
__device__ __forceinline__ lq to_lq(double x, unsigned &top) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  top = max(top, hi & 0x7FFFFFFFu);
  // |x| 2^60 with the leading one at bit 60 for |x| in [1, 2), shifted right by 1023 - exponent field
  const unsigned long long m =
      ((unsigned long long)((__funnelshift_l(lo, hi, 8) & 0x0FFFFFFFu) | 0x10000000u) << 32) | (lo << 8);
  const unsigned long long q = m >> min(1023u - ((hi >> 20) & 0x7FFu), 63u);
  const int h = (int)(q >> 30), l = (int)((unsigned)q & 0x3FFFFFFFu), sg = (int)hi >> 31;
  return {(h ^ sg) - sg, (l ^ sg) - sg};
}
__device__ __forceinline__ bool lq_in_range(unsigned top) { return top < 0x40000000u; }  // every |x| < 2
__device__ __forceinline__ clq to_clq(cx<double> v, unsigned &top) { return {to_lq(v.r, top), to_lq(v.i, top)}; }
__device__ __forceinline__ lq lq_neg(lq a) { return {-a.h, -a.l}; }

struct lacc {
  long long hh, c;
};
__device__ __forceinline__ void lmac(lacc &s, lq a, lq b) {
  s.hh += (long long)a.h * b.h;
  s.c += (long long)a.h * b.l;
  s.c += (long long)a.l * b.h;
}
__device__ __forceinline__ long long lacc_value(lacc s) { return s.hh + (s.c >> 30); }  // times 2^-60
// of two sums whose cross sums may not fit in 64 bits together (their mean does)
__device__ __forceinline__ long long lacc_value(lacc s, lacc w) {
  return s.hh + w.hh + (((s.c & w.c) + ((s.c ^ w.c) >> 1)) >> 29);
}
__device__ __forceinline__ lq lq_split(long long v) { return {(int)(v >> 30), (int)((unsigned)v & 0x3FFFFFFFu)}; }
__device__ __forceinline__ long long lq_join(lq a) { return ((long long)a.h << 30) + a.l; }
// v 2^-60 rounded to nearest
__device__ __forceinline__ double q60_double(long long v) { return __ll2double_rn(v) * 0x1p-60; }

// Limb planes: one complex number in 16 bytes.
__device__ __forceinline__ clq ldg_q(const int4 *p, int64_t idx) {
  const int4 v = __ldg(p + idx);
  return {{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ int4 to_int4(clq a) { return make_int4(a.r.h, a.r.l, a.i.h, a.i.l); }
__device__ __forceinline__ double lq_double(lq a) { return q60_double(lq_join(a)); }

// Rows and columns of about unit length: at most (to 1.5%), so that the products of such matrices, and their sums,
// stay in range whatever the entries are, and at least a quarter, because FP64 products of shorter ones would err by
// less than 2^-57. Gathered one element at a time (|x| < 2 each: 14-bit squares, 31-bit sums).
struct unit_check {
  int row[3] = {0, 0, 0}, col[3] = {0, 0, 0};
  __device__ static __forceinline__ int square(clq a) {
    const int x = a.r.h >> 17, y = a.i.h >> 17;
    return x * x + y * y;
  }
  __device__ __forceinline__ void add(int i, int j, clq a) {
    const int n = square(a);
    row[i] += n;
    col[j] += n;
  }
  __device__ __forceinline__ bool ok(unsigned top) const {
    constexpr int most = 69000000, least = 1 << 22;  // 2^26 is a unit vector
    return lq_in_range(top) &&
           max(max(max(row[0], row[1]), row[2]), max(max(col[0], col[1]), col[2])) <= most &&
           min(min(min(row[0], row[1]), row[2]), min(min(col[0], col[1]), col[2])) >= least;
  }
};

// The elements by their part in an anti-Hermitian matrix, over all the matrices that enter a sum: the three pairs
// beside the diagonal and the three imaginary parts on it. Where the elements of one of them are all small, as those
// of fields close to unity are, its 2^-60 would be more than the rounding of FP64. The line, 2^-6: the rms errors of the
// two gradients of random fields around unity meet at parts of 2^-7.8, the largest of a site's then lying about there
// (2^-59.3 against 2^-59.7 at half of that, 2^-58.9 against 2^-58.8 at twice).
struct part_check {
  int pair[3] = {0, 0, 0}, diag[3] = {0, 0, 0};
  __device__ __forceinline__ void add(int i, int j, clq a) {
    if (i == j) diag[i] |= (a.i.h >> 17) * (a.i.h >> 17);
    else pair[i + j - 1] |= unit_check::square(a);
  }
  __device__ __forceinline__ bool small() const {  // all below 2^-6
    return min(min(min(pair[0], pair[1]), pair[2]), min(min(diag[0], diag[1]), diag[2])) < (1 << 14);
  }
};

// acc += a b, += a conj(b)
struct clacc {
  lacc re, im;
};
__device__ __forceinline__ void clmac(clacc &s, clq a, clq b) {
  lmac(s.re, a.r, b.r);
  lmac(s.re, a.i, lq_neg(b.i));
  lmac(s.im, a.r, b.i);
  lmac(s.im, a.i, b.r);
}
__device__ __forceinline__ void clmac_cj(clacc &s, clq a, clq b) {
  lmac(s.re, a.r, b.r);
  lmac(s.re, a.i, b.i);
  lmac(s.im, a.i, b.r);
  lmac(s.im, a.r, lq_neg(b.i));
}
__device__ __forceinline__ clq clacc_split(const clacc &s) { return {lq_split(lacc_value(s.re)), lq_split(lacc_value(s.im))}; }

// The words of a complex double (x: re lo, y: re hi, z: im lo, w: im hi) as limbs, for callers who have checked
// the range. The sign is exact: a complement alone would save two operations of sixteen, but lengthens every
// negative number by 2^-60, and the links with it, a little in each update.
__device__ __forceinline__ lq words_lq(unsigned hi, unsigned lo) {
  const unsigned long long m =
      ((unsigned long long)((__funnelshift_l(lo, hi, 8) & 0x0FFFFFFFu) | 0x10000000u) << 32) | (lo << 8);
  const long long q = (long long)(m >> min((0x3FFFFFFFu - (hi & 0x7FFFFFFFu)) >> 20, 63u));
  const long long v = (int)hi < 0 ? -q : q;
  return {(int)(v >> 30), (int)((unsigned)v & 0x3FFFFFFFu)};
}
__device__ __forceinline__ clq words_clq(int4 v) {
  return {words_lq((unsigned)v.y, (unsigned)v.x), words_lq((unsigned)v.w, (unsigned)v.z)};
}
__device__ __forceinline__ cx<double> words_double(int4 v) {
  return {__hiloint2double(v.y, v.x), __hiloint2double(v.w, v.z)};
}
__device__ __forceinline__ clq limbs_of(int4 v) { return {{v.x, v.y}, {v.z, v.w}}; }

// The link g(x) U g^+(x + mu) in FP64: rows 0 and 1 by products, row 2 = conj(row0 x row1). gx_of, u_of and
// g_of give the elements of g(x) (rows 0-1 are used), U and g(x + mu); out(e, value) takes the nine elements.
template <typename XOf, typename UOf, typename GOf, typename Out>
__device__ __forceinline__ void link_product_fp64(XOf gx_of, UOf u_of, GOf g_of, Out out) {
  m3<double> t, o;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    cx<double> gi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) gi[k] = gx_of(3 * i + k);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cx<double> acc = gi[0] * u_of(j);
      acc = cmac(acc, gi[1], u_of(3 + j));
      acc = cmac(acc, gi[2], u_of(6 + j));
      t.e[3 * i + j] = acc;
    }
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const cx<double> h0 = g_of(3 * j), h1 = g_of(3 * j + 1), h2 = g_of(3 * j + 2);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      cx<double> acc = {0, 0};
      acc = cmac_cj(acc, t.e[3 * i], h0);
      acc = cmac_cj(acc, t.e[3 * i + 1], h1);
      acc = cmac_cj(acc, t.e[3 * i + 2], h2);
      o.e[3 * i + j] = acc;
    }
  }
  complete_row2(o);
#pragma unroll
  for (int e = 0; e < 9; ++e) out(e, o.e[e]);
}

}  // namespace lgf
