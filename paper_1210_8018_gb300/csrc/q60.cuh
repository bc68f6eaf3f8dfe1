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
// of magnitude 2 and above, infinities and NaN (lq_in_range) to the FP64 form.
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

// Rows and columns of at most unit length (to 1.5%): the products of such matrices, and their sums, stay in
// range whatever the entries are. Gathered one element at a time (|x| < 2 each: 14-bit squares, 31-bit sums).
struct unit_check {
  int row[3] = {0, 0, 0}, col[3] = {0, 0, 0};
  __device__ __forceinline__ void add(int i, int j, clq a) {
    const int x = a.r.h >> 17, y = a.i.h >> 17, n = x * x + y * y;
    row[i] += n;
    col[j] += n;
  }
  __device__ __forceinline__ bool ok(unsigned top) const {
    constexpr int limit = 69000000;  // 2^26 is a unit vector
    return lq_in_range(top) &&
           max(max(max(row[0], row[1]), row[2]), max(max(col[0], col[1]), col[2])) <= limit;
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

// The link g(x) U g^+(x + mu): rows 0 and 1 by products, row 2 = conj(row0 x row1). gx_of, u_of and g_of give
// the elements of g(x) (rows 0-1 are used), U and g(x + mu); out(e, value) is called for the nine elements,
// unless some lane of the warp has an entry out of range: then nothing is written and the answer is false.
// The lanes that are active in a warp call it together.
template <typename XOf, typename UOf, typename GOf, typename Out>
__device__ __forceinline__ bool link_product_q60(XOf gx_of, UOf u_of, GOf g_of, Out out) {
  unsigned top = 0;
  clq gx[6];
#pragma unroll
  for (int e = 0; e < 6; ++e) gx[e] = to_clq(gx_of(e), top);
  clq t[6];  // rows 0-1 of g(x) U, one column of U at a time
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    lacc re[2] = {}, im[2] = {};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const clq u = to_clq(u_of(3 * k + j), top);
      const lq ni = lq_neg(u.i);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        lmac(re[i], gx[3 * i + k].r, u.r);
        lmac(re[i], gx[3 * i + k].i, ni);
        lmac(im[i], gx[3 * i + k].r, u.i);
        lmac(im[i], gx[3 * i + k].i, u.r);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) t[3 * i + j] = {lq_split(lacc_value(re[i])), lq_split(lacc_value(im[i]))};
  }
  clq o[6];  // rows 0-1 of the result
#pragma unroll
  for (int j = 0; j < 3; ++j) {  // one row of g(x + mu) at a time
    lacc re[2] = {}, im[2] = {};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const clq g = to_clq(g_of(3 * j + k), top);
      const lq ni = lq_neg(g.i);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        lmac(re[i], t[3 * i + k].r, g.r);
        lmac(re[i], t[3 * i + k].i, g.i);
        lmac(im[i], t[3 * i + k].i, g.r);
        lmac(im[i], t[3 * i + k].r, ni);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
      o[3 * i + j] = {lq_split(lacc_value(re[i])), lq_split(lacc_value(im[i]))};
  }
  if (__any_sync(__activemask(), !lq_in_range(top))) return false;
#pragma unroll
  for (int e = 0; e < 6; ++e) out(e, cx<double>{q60_double(lq_join(o[e].r)), q60_double(lq_join(o[e].i))});
#pragma unroll
  for (int e = 6; e < 9; ++e) {  // conj(a b - c d)
    const clq a = o[e == 6 ? 1 : e == 7 ? 2 : 0], b = o[e == 6 ? 5 : e == 7 ? 3 : 4];
    const clq c = o[e == 6 ? 2 : e == 7 ? 0 : 1], d = o[e == 6 ? 4 : e == 7 ? 5 : 3];
    lacc re = {}, im = {};
    lmac(re, a.r, b.r);
    lmac(re, a.i, lq_neg(b.i));
    lmac(re, c.r, lq_neg(d.r));
    lmac(re, c.i, d.i);
    lmac(im, a.r, lq_neg(b.i));
    lmac(im, a.i, lq_neg(b.r));
    lmac(im, c.r, d.i);
    lmac(im, c.i, d.r);
    out(e, cx<double>{q60_double(lacc_value(re)), q60_double(lacc_value(im))});
  }
  return true;
}

// The same in FP64, for entries of any size.
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
