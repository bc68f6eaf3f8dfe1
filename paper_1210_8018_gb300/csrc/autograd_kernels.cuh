// autograd_kernels.cuh -- the gauge functional as a differentiable function of a Lie-algebra field:
//   F(omega) = F_U[g] with g(x) = exp(i omega(x)), omega(x) = sum_a omega^a(x) T^a, T^a = lambda^a / 2
// (Eq. 1 of the paper evaluated at g = exp(i omega)), and its gradient dF/d omega^a(x), the
// steepest-ascent direction that the Fourier-accelerated method preconditions.
//
// Gradient: g(x) enters F through S = Re Tr[g(x) K(x)] with the staple
//   K(x) = sum_mu [ U_mu(x) g^+(x+mu) + U_mu^+(x-mu) g^+(x-mu) ].
// The derivative of the exponential, dg = i (phi(i ad_H) dH) g with H = omega, ad_H X = [H, X] and
// phi(z) = (e^z - 1)/z, and ad_H being self-adjoint under the trace give
//   dF/d omega^a = -(1/(12 V)) Tr[ T^a phi(-i ad_H) A ],   A = (M - M^+)/(2i), M = g K,
// where phi(-i ad_H) A = sum_n D^n A / (n+1)!, D A = -i [H, A], is a sum of Hermitian matrices (44 multiply-adds
// a term). At omega = 0 it reduces to -(i/(24 V)) Tr[T^a Delta(x)] with Delta of Eq. 5.
//
// The exponential itself is the Taylor series with the powers of H reduced by Cayley-Hamilton,
// H^3 = c1 H + c0 (c1 = Tr H^2 / 2, c0 = det H): g = f0 + f1 H + f2 H^2, five multiply-adds a term on real
// numbers. Both series run on H / 2^m of Frobenius norm below 1/2 and are doubled back m times,
//   exp(2iH): f -> f f reduced by the same relation,   phi(2z) = phi(z) (e^z + 1)/2: Y <- (Y + g^+ Y g)/2.
// Above a norm of 3, and for omega that is not finite, the eigenvectors W of omega serve (omega = W diag(l)
// W^+, Daleckii-Krein: W (Phi o (W^+ K W)) W^+ with Phi_jk = exp(i (l_j + l_k)/2) sinc((l_j - l_k)/2)).
//
// Products with O(1) matrices (g U, the staple) run in 60-bit fixed point (q60.cuh); a site that meets a link
// which is not near SU(3) forms them in FP64, and so does the staple of a site around which all matrices have the
// same elements close to zero (part_check), the gradient of which may be as small.
#pragma once
#include "site_kernels.cuh"

namespace lgf {

// Hermitian matrix H = sum_a w^a lambda^a / 2.
__device__ __forceinline__ void algebra_matrix(const double w[8], m3<double> &H) {
  const double s3 = 0.57735026918962576451;  // 1/sqrt(3)
  H.e[0] = {0.5 * (w[2] + s3 * w[7]), 0};
  H.e[4] = {0.5 * (-w[2] + s3 * w[7]), 0};
  H.e[8] = {-s3 * w[7], 0};
  H.e[1] = {0.5 * w[0], -0.5 * w[1]};
  H.e[3] = {0.5 * w[0], 0.5 * w[1]};
  H.e[2] = {0.5 * w[3], -0.5 * w[4]};
  H.e[6] = {0.5 * w[3], 0.5 * w[4]};
  H.e[5] = {0.5 * w[5], -0.5 * w[6]};
  H.e[7] = {0.5 * w[5], 0.5 * w[6]};
}

// Cyclic Jacobi eigen-decomposition of a Hermitian 3x3 matrix: H = W diag(l) W^+ (W unitary).
// Each rotation first makes H_pq real with a phase on column q, then applies the real Jacobi rotation.
// At most 12 sweeps (quadratic convergence; 4-5 are used in practice).
__device__ __forceinline__ void jacobi_eigh(m3<double> H, m3<double> &W, double l[3]) {
  for (int e = 0; e < 9; ++e) W.e[e] = {(e % 4 == 0) ? 1.0 : 0.0, 0.0};
  const double scale = sqrt(norm2(H.e[0]) + norm2(H.e[4]) + norm2(H.e[8]) +
                            2.0 * (norm2(H.e[1]) + norm2(H.e[2]) + norm2(H.e[5]))) + 1e-300;
  for (int sweep = 0; sweep < 12; ++sweep) {
    const double off = norm2(H.e[1]) + norm2(H.e[2]) + norm2(H.e[5]);
    if (off <= 1e-34 * scale * scale) break;
    for (int pq = 0; pq < 3; ++pq) {
      const int p = pq == 2 ? 1 : 0, q = pq == 0 ? 1 : 2;
      const cx<double> h = H.e[3 * p + q];
      const double r = sqrt(norm2(h));
      if (r <= 1e-300) continue;
      // phase: column q times d = conj(h)/r, row q times conj(d) -> H_pq becomes r (real)
      const cx<double> d = {h.r / r, -h.i / r};
      for (int k = 0; k < 3; ++k) {
        H.e[3 * k + q] = H.e[3 * k + q] * d;
        W.e[3 * k + q] = W.e[3 * k + q] * d;
      }
      for (int k = 0; k < 3; ++k) H.e[3 * q + k] = H.e[3 * q + k] * conjg(d);
      // real rotation on (p, q)
      const double app = H.e[3 * p + p].r, aqq = H.e[3 * q + q].r;
      const double tau = (aqq - app) / (2.0 * r);
      const double t = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
      const double c = 1.0 / sqrt(1.0 + t * t), s = t * c;
      // columns: H <- H R, W <- W R with R = [[c, s], [-s, c]] on (p, q)
      for (int k = 0; k < 3; ++k) {
        const cx<double> hp = H.e[3 * k + p], hq = H.e[3 * k + q];
        H.e[3 * k + p] = {c * hp.r - s * hq.r, c * hp.i - s * hq.i};
        H.e[3 * k + q] = {s * hp.r + c * hq.r, s * hp.i + c * hq.i};
        const cx<double> wp = W.e[3 * k + p], wq = W.e[3 * k + q];
        W.e[3 * k + p] = {c * wp.r - s * wq.r, c * wp.i - s * wq.i};
        W.e[3 * k + q] = {s * wp.r + c * wq.r, s * wp.i + c * wq.i};
      }
      // rows: H <- R^T H
      for (int k = 0; k < 3; ++k) {
        const cx<double> hp = H.e[3 * p + k], hq = H.e[3 * q + k];
        H.e[3 * p + k] = {c * hp.r - s * hq.r, c * hp.i - s * hq.i};
        H.e[3 * q + k] = {s * hp.r + c * hq.r, s * hp.i + c * hq.i};
      }
      H.e[3 * p + q] = {0, 0};
      H.e[3 * q + p] = {0, 0};
    }
  }
  l[0] = H.e[0].r;
  l[1] = H.e[4].r;
  l[2] = H.e[8].r;
}

// g = W diag(exp(i l)) W^+
__device__ __forceinline__ void expi_from_eig(const m3<double> &W, const double l[3], m3<double> &g) {
  cx<double> ph[3];
  for (int k = 0; k < 3; ++k) {
    double sn, cs;
    sincos(l[k], &sn, &cs);
    ph[k] = {cs, sn};
  }
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      cx<double> acc = {0, 0};
      for (int k = 0; k < 3; ++k) acc = cmac_cj(acc, W.e[3 * i + k] * ph[k], W.e[3 * j + k]);
      g.e[3 * i + j] = acc;
    }
}

// Hermitian matrix with diagonal d and upper elements 01, 02, 12.
struct herm {
  double d[3];
  cx<double> a, b, c;
};
__device__ __forceinline__ herm algebra_herm(const double w[8], double scale) {
  const double s3 = 0.57735026918962576451, h = 0.5 * scale;  // 1/sqrt(3)
  return {{h * fma(s3, w[7], w[2]), h * fma(s3, w[7], -w[2]), -2.0 * h * s3 * w[7]},
          {h * w[0], -h * w[1]},
          {h * w[3], -h * w[4]},
          {h * w[5], -h * w[6]}};
}
// Squared Frobenius norm of omega, and the m for which omega / 2^m has a norm below 1/2.
__device__ __forceinline__ double algebra_norm2(const double w[8]) {
  double t = 0;
#pragma unroll
  for (int a = 0; a < 8; ++a) t = fma(w[a], w[a], t);
  return 0.5 * t;
}
// Norm 3 (m <= 3): below it the gradient's error is smaller than by eigenvectors (rms 2.2e-16 of the gradient against
// 1.0e-15 at |omega| = 0.1, 8.7e-16 against 1.2e-15 at 2), at a norm of 10 the doublings have made it larger.
constexpr double kSeriesNorm2 = 9.0;
__device__ __forceinline__ int halvings(double norm2) {
  return max(0, (((__double2hiint(norm2) >> 20) & 0x7FF) - 1023 + 4) >> 1);
}
// exp(i H) = f0 + f1 H + f2 H^2
struct exp_poly {
  cx<double> f0, f1, f2;
  double c0, c1;
};
// 1/n! with the sign of i^n (real parts for even n, imaginary for odd)
__constant__ double kExpCoef[20] = {1.0,
                                    1.0,
                                    -1.0 / 2,
                                    -1.0 / 6,
                                    1.0 / 24,
                                    1.0 / 120,
                                    -1.0 / 720,
                                    -1.0 / 5040,
                                    1.0 / 40320,
                                    1.0 / 362880,
                                    -1.0 / 3628800,
                                    -1.0 / 39916800,
                                    1.0 / 479001600,
                                    1.0 / 6227020800.0,
                                    -1.0 / 87178291200.0,
                                    -1.0 / 1307674368000.0,
                                    1.0 / 20922789888000.0,
                                    1.0 / 355687428096000.0,
                                    -1.0 / 6402373705728000.0,
                                    -1.0 / 121645100408832000.0};
__device__ __forceinline__ exp_poly exp_series(const herm &h, float norm) {
  exp_poly p;
  p.c1 = fma(0.5, fma(h.d[0], h.d[0], fma(h.d[1], h.d[1], h.d[2] * h.d[2])), norm2(h.a) + norm2(h.b) + norm2(h.c));
  const cx<double> ac = h.a * h.c;
  const double acb = fma(ac.r, h.b.r, ac.i * h.b.i);  // Re a c conj(b)
  p.c0 = fma(2.0, acb, h.d[0] * h.d[1] * h.d[2]) - h.d[0] * norm2(h.c) - h.d[1] * norm2(h.b) - h.d[2] * norm2(h.a);
  // H^n = a + b H + d H^2
  double a = 0, b = 0, d = 1;
  p.f0 = {1.0, 0.0};
  p.f1 = {0.0, 1.0};
  p.f2 = {-0.5, 0.0};
  float term = 0.5f * norm * norm;
#pragma unroll 1
  for (int n = 3; n < 19; n += 2) {  // an odd and an even power
    auto next = [&]() {
      const double t = d * p.c0;
      d = fma(d, p.c1, a);  // (the new b)
      a = t;
      const double nb = d;
      d = b;
      b = nb;
    };
    next();
    p.f0.i = fma(kExpCoef[n], a, p.f0.i);
    p.f1.i = fma(kExpCoef[n], b, p.f1.i);
    p.f2.i = fma(kExpCoef[n], d, p.f2.i);
    next();
    p.f0.r = fma(kExpCoef[n + 1], a, p.f0.r);
    p.f1.r = fma(kExpCoef[n + 1], b, p.f1.r);
    p.f2.r = fma(kExpCoef[n + 1], d, p.f2.r);
    term *= norm * norm / (float)(n * (n + 1));  // norm^(n+1) / (n+1)!
    if (term < 1e-18f) break;
  }
  return p;
}
// exp(2iH) from exp(iH), still as a polynomial in H
__device__ __forceinline__ void exp_double(exp_poly &p) {
  const cx<double> q = p.f1 * p.f2, s = p.f2 * p.f2, f00 = p.f0 * p.f0, f01 = p.f0 * p.f1, f02 = p.f0 * p.f2,
                   f11 = p.f1 * p.f1;
  const double c0 = p.c0, c1 = p.c1;
  p.f0 = {fma(2.0 * c0, q.r, f00.r), fma(2.0 * c0, q.i, f00.i)};
  p.f1 = {2.0 * fma(c1, q.r, f01.r) + c0 * s.r, 2.0 * fma(c1, q.i, f01.i) + c0 * s.i};
  p.f2 = {fma(2.0, f02.r, f11.r) + c1 * s.r, fma(2.0, f02.i, f11.i) + c1 * s.i};
}
__device__ __forceinline__ void exp_matrix(const exp_poly &p, const herm &h, m3<double> &g) {
  const double na = norm2(h.a), nb = norm2(h.b), nc = norm2(h.c);
  const double s[3] = {fma(h.d[0], h.d[0], na + nb), fma(h.d[1], h.d[1], na + nc), fma(h.d[2], h.d[2], nb + nc)};
#pragma unroll
  for (int i = 0; i < 3; ++i)
    g.e[4 * i] = {fma(p.f2.r, s[i], fma(p.f1.r, h.d[i], p.f0.r)), fma(p.f2.i, s[i], fma(p.f1.i, h.d[i], p.f0.i))};
  const cx<double> bc = h.b * conjg(h.c), ac = h.a * h.c, ab = conjg(h.a) * h.b;
  const double t0 = h.d[0] + h.d[1], t1 = h.d[0] + h.d[2], t2 = h.d[1] + h.d[2];
  auto put = [&](int up, int lo, cx<double> x, cx<double> x2) {
    g.e[up] = cmac(p.f1 * x, p.f2, x2);
    g.e[lo] = cmac(p.f1 * conjg(x), p.f2, conjg(x2));
  };
  put(1, 3, h.a, {fma(t0, h.a.r, bc.r), fma(t0, h.a.i, bc.i)});
  put(2, 6, h.b, {fma(t1, h.b.r, ac.r), fma(t1, h.b.i, ac.i)});
  put(5, 7, h.c, {fma(t2, h.c.r, ab.r), fma(t2, h.c.i, ab.i)});
}
__device__ __noinline__ void expi_by_eigenvectors(const double *w, m3<double> *g) {
  m3<double> H, W;
  double l[3];
  algebra_matrix(w, H);
  jacobi_eigh(H, W, l);
  expi_from_eig(W, l, *g);
}

// omega (V x 8, site-major) -> g in limb planes, and where asked in planes of doubles.
// A g that is not finite is marked by kNoLimb, which the readers turn into NaN.
// Bound by the FP64 pipe (92% busy, about 180 operations a site at |omega| = 0.1): 0.113 ms at 24^4, where the
// eigenvectors by Jacobi sweeps are thousands of operations.
constexpr int kNoLimb = (int)0x80000000;
template <int NT>
__global__ void __launch_bounds__(NT) k_expi(const double *__restrict__ omega, int4 *__restrict__ Gq,
                                            double *__restrict__ G, int64_t V) {
  const int64_t s = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (s >= V) return;
  double w[8];
#pragma unroll
  for (int a = 0; a < 8; a += 2) {
    const double2 v = reinterpret_cast<const double2 *>(omega)[s * 4 + a / 2];
    w[a] = v.x;
    w[a + 1] = v.y;
  }
  m3<double> g;
  const double n2 = algebra_norm2(w);
  if (n2 <= kSeriesNorm2) {
    const int m = halvings(n2);
    const double sc = __hiloint2double((1023 - m) << 20, 0);
    const herm h = algebra_herm(w, sc);
    exp_poly p = exp_series(h, (float)(sqrt((float)n2) * (float)sc));
    for (int k = 0; k < m; ++k) exp_double(p);
    exp_matrix(p, h, g);
  } else {
    m3<double> t;
    expi_by_eigenvectors(w, &t);
    g = t;
  }
  unsigned top = 0;
  clq q[9];
#pragma unroll
  for (int e = 0; e < 9; ++e) q[e] = to_clq(g.e[e], top);
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    Gq[(int64_t)e * V + s] = lq_in_range(top) ? to_int4(q[e]) : make_int4(kNoLimb, 0, 0, 0);
    if (G) st(G, (int64_t)e * V + s, g.e[e]);
  }
}
__device__ __forceinline__ cx<double> g_element(const int4 *Gq, int64_t idx) {
  const clq q = ldg_q(Gq, idx);
  if (q.r.h == kNoLimb) return {__longlong_as_double(0x7FF8000000000000ll), __longlong_as_double(0x7FF8000000000000ll)};
  return {lq_double(q.r), lq_double(q.i)};
}

// Re Tr[g(x) U g^+(y)] in FP64, for links out of the fixed-point range.
__device__ __noinline__ double link_trace_fp64(const double2 *u, const int4 *Gq, int64_t V, int64_t s, int64_t sf) {
  double f = 0;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      cx<double> t = {0, 0};
      for (int k = 0; k < 3; ++k)
        t = cmac(t, g_element(Gq, (int64_t)(3 * i + k) * V + s), from_vec<double>(u[3 * k + j]));
      const cx<double> gy = g_element(Gq, (int64_t)(3 * i + j) * V + sf);
      f += t.r * gy.r + t.i * gy.i;
    }
  return f;
}

// F partials: sum_mu Re Tr[g(x) U_mu(x) g^+(x+mu)] per site, reduced in FP64. U: the caller's links, read once;
// g in limb planes. At 24^4 0.12 ms (the integer multiplies and the conversions of U share the time).
template <int NT>
__global__ void __launch_bounds__(NT, 2) k_functional_g(const double *__restrict__ U, const int4 *__restrict__ Gq,
                                                       double *partials, Ctrl *ctrl, Lattice L, int spt) {
  const int64_t V = L.V;
  double f = 0.0;
#pragma unroll 1
  for (int n = 0; n < spt; ++n) {
    const int64_t s = ((int64_t)blockIdx.x * spt + n) * NT + threadIdx.x;
    if (s >= V) break;
    int c[4];
    site_coords(L, s, c);
    clq gx[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) gx[e] = ldg_q(Gq, (int64_t)e * V + s);
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      const int64_t sf = site_fwd(L, s, mu, c[mu]);
      const double2 *u = reinterpret_cast<const double2 *>(U) + ((int64_t)mu * V + s) * 9;
      unsigned top = 0;
      unit_check unit;
      long long sum = 0;
      bool bad = gx[0].r.h == kNoLimb;
#pragma unroll
      for (int j = 0; j < 3; ++j) {  // column j of g(x) U against column j of g(x + mu)
        clacc t[3] = {};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const clq x = to_clq(from_vec<double>(__ldg(u + 3 * k + j)), top);
          unit.add(k, j, x);
#pragma unroll
          for (int i = 0; i < 3; ++i) clmac(t[i], gx[3 * i + k], x);
        }
        lacc dot = {};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const clq y = ldg_q(Gq, (int64_t)(3 * i + j) * V + sf), z = clacc_split(t[i]);
          bad |= y.r.h == kNoLimb;
          lmac(dot, z.r, y.r);
          lmac(dot, z.i, y.i);
        }
        sum += lacc_value(dot);
      }
      f += bad || !unit.ok(top) ? link_trace_fp64(u, Gq, V, s, sf) : q60_double(sum);
    }
  }
  double th = 0.0;
  reduce_and_finalize<NT>(th, f, partials, ctrl, V, 0);
}

__device__ __forceinline__ double sinc_half(double x) {  // sin(x)/x
  const double ax = fabs(x);
  if (ax < 1e-4) {
    const double x2 = x * x;
    return 1.0 - x2 / 6.0 + x2 * x2 / 120.0;
  }
  return sin(x) / x;
}

// The staple K(x) in FP64, for fields that are not for the fixed point. g in planes.
__device__ __noinline__ void staple_fp64(const double2 *U, const double *G, const Lattice *L, int64_t s, const int *c,
                                         m3<double> *K) {
  const int64_t V = L->V;
  for (int e = 0; e < 9; ++e) K->e[e] = {0, 0};
  for (int mu = 0; mu < 4; ++mu) {
    const int64_t sf = site_fwd(*L, s, mu, c[mu]), sb = site_back(*L, s, mu, c[mu]);
    const double2 *u = U + ((int64_t)mu * V + s) * 9, *ub = U + ((int64_t)mu * V + sb) * 9;
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        cx<double> t = K->e[3 * i + j], b = {0, 0};
        for (int k = 0; k < 3; ++k) {
          t = cmac_cj(t, from_vec<double>(u[3 * i + k]), ldg(G, (int64_t)(3 * j + k) * V + sf));
          b = cmac(b, ldg(G, (int64_t)(3 * j + k) * V + sb), from_vec<double>(ub[3 * k + i]));
        }
        K->e[3 * i + j] = t + conjg(b);
      }
  }
}

// Tr[T^a Q'] of the derivative by eigenvectors, Q' = W (Phi o (W^+ K W)) W^+ (imaginary parts).
__device__ __noinline__ void gradient_by_eigenvectors(const double *w, const m3<double> *K, double *gr) {
  m3<double> H, W, M, Q, T1, Wd;
  double l[3];
  algebra_matrix(w, H);
  jacobi_eigh(H, W, l);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) Wd.e[3 * i + j] = conjg(W.e[3 * j + i]);
  mul(Wd, *K, T1);
  mul(T1, W, M);
  for (int j = 0; j < 3; ++j)
    for (int k = 0; k < 3; ++k) {
      double sn, cs;
      sincos(0.5 * (l[j] + l[k]), &sn, &cs);
      const double sc = sinc_half(0.5 * (l[j] - l[k]));
      M.e[3 * j + k] = M.e[3 * j + k] * cx<double>{cs * sc, sn * sc};
    }
  mul(W, M, T1);
  mul_adj(T1, W, Q);
  const double s3 = 0.57735026918962576451;
  gr[0] = 0.5 * (Q.e[3].i + Q.e[1].i);                       // lambda1: Q10 + Q01
  gr[1] = 0.5 * (-Q.e[3].r + Q.e[1].r);                      // lambda2: -i Q10 + i Q01
  gr[2] = 0.5 * (Q.e[0].i - Q.e[4].i);                       // lambda3
  gr[3] = 0.5 * (Q.e[6].i + Q.e[2].i);                       // lambda4: Q20 + Q02
  gr[4] = 0.5 * (-Q.e[6].r + Q.e[2].r);                      // lambda5
  gr[5] = 0.5 * (Q.e[7].i + Q.e[5].i);                       // lambda6: Q21 + Q12
  gr[6] = 0.5 * (-Q.e[7].r + Q.e[5].r);                      // lambda7
  gr[7] = 0.5 * s3 * (Q.e[0].i + Q.e[4].i - 2.0 * Q.e[8].i);  // lambda8
}

// D A = -i [H, A]
__device__ __forceinline__ herm commutator(const herm &h, const herm &x) {
  auto minus_i = [](cx<double> v) { return cx<double>{v.i, -v.r}; };
  auto off = [&](cx<double> z, double dh, double dx, cx<double> hz) {  // dh z - hz dx
    return cx<double>{fma(dh, z.r, -dx * hz.r), fma(dh, z.i, -dx * hz.i)};
  };
  herm y;
  cx<double> t = off(x.a, h.d[0] - h.d[1], x.d[0] - x.d[1], h.a);
  t = cmac_cj(t, h.b, x.c);
  y.a = minus_i(cmac_cj(t, cx<double>{-x.b.r, -x.b.i}, h.c));
  t = off(x.b, h.d[0] - h.d[2], x.d[0] - x.d[2], h.b);
  t = cmac(t, h.a, x.c);
  y.b = minus_i(cmac(t, cx<double>{-h.c.r, -h.c.i}, x.a));
  t = off(x.c, h.d[1] - h.d[2], x.d[1] - x.d[2], h.c);
  t = cmac_cj(t, x.b, h.a);
  y.c = minus_i(cmac_cj(t, cx<double>{-h.b.r, -h.b.i}, x.a));
  // 2 Im of the diagonal of H A
  const double ia = fma(h.a.i, x.a.r, -h.a.r * x.a.i), ib = fma(h.b.i, x.b.r, -h.b.r * x.b.i);
  const double ic = fma(h.c.i, x.c.r, -h.c.r * x.c.i);
  y.d[0] = 2 * (ia + ib);
  y.d[1] = 2 * (ic - ia);
  y.d[2] = -2 * (ib + ic);
  return y;
}
__device__ __forceinline__ void herm_axpy(herm &y, double s, const herm &x) {
#pragma unroll
  for (int i = 0; i < 3; ++i) y.d[i] = fma(s, x.d[i], y.d[i]);
  y.a = {fma(s, x.a.r, y.a.r), fma(s, x.a.i, y.a.i)};
  y.b = {fma(s, x.b.r, y.b.r), fma(s, x.b.i, y.b.i)};
  y.c = {fma(s, x.c.r, y.c.r), fma(s, x.c.i, y.c.i)};
}
// Y <- (Y + g^+ Y g) / 2
__device__ __noinline__ void conjugate_average(herm *y, const m3<double> *g) {
  m3<double> Y, T, R;
  Y.e[0] = {y->d[0], 0};
  Y.e[4] = {y->d[1], 0};
  Y.e[8] = {y->d[2], 0};
  Y.e[1] = y->a;
  Y.e[2] = y->b;
  Y.e[5] = y->c;
  Y.e[3] = conjg(y->a);
  Y.e[6] = conjg(y->b);
  Y.e[7] = conjg(y->c);
  mul(Y, *g, T);
  for (int i = 0; i < 3; ++i)
    for (int j = i; j < 3; ++j) {
      cx<double> acc = {0, 0};
      for (int k = 0; k < 3; ++k) acc = cmac(acc, conjg(g->e[3 * k + i]), T.e[3 * k + j]);
      R.e[3 * i + j] = acc;
    }
  for (int i = 0; i < 3; ++i) y->d[i] = 0.5 * (y->d[i] + R.e[4 * i].r);
  y->a = scale(y->a + R.e[1], 0.5);
  y->b = scale(y->b + R.e[2], 0.5);
  y->c = scale(y->c + R.e[5], 0.5);
}

// dF/d omega^a(x), a = 0..7, written site-major (V x 8), scaled by `scale` (the incoming gradient). U: the
// caller's links; g in limb planes and in planes of doubles. The staple is summed in 59 fractional bits (its elements reach 8).
// Bound by the FP64 pipe (87% busy, 570 of 900 operations in the eleven terms of the series at |omega| = 0.1): 0.61 ms
// at 24^4. A step of gradient-based fixing (F, gradient, Fourier filter) took 5.40 ms with Jacobi eigenvectors and FP64
// products in both calls, and takes 1.57 ms (1.55 without part_check). (The terms below 2^-34 of the sum in float would make it 1.44, with
// those of links beyond 1e38 infinite.)
template <int NT>
__global__ void __launch_bounds__(NT, 3) k_functional_grad(const double *__restrict__ U, const int4 *__restrict__ Gq,
                                                       const double *__restrict__ G, const double *omega, double *grad, Lattice L, double scale) {
  const int64_t V = L.V;
  const int64_t s = (int64_t)blockIdx.x * NT + threadIdx.x;
  if (s >= V) return;
  int c[4];
  site_coords(L, s, c);
  const double2 *U2 = reinterpret_cast<const double2 *>(U);
  m3<double> K;
  {
    long long kr[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, ki[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    bool bad = false;
    part_check parts;
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      const int64_t sf = site_fwd(L, s, mu, c[mu]), sb = site_back(L, s, mu, c[mu]);
      {  // U_mu(x) g^+(x+mu)
        const double2 *u = U2 + ((int64_t)mu * V + s) * 9;
        unsigned top = 0;
        unit_check unit;
        clq g[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) g[e] = ldg_q(Gq, (int64_t)e * V + sf);
        bad |= g[0].r.h == kNoLimb;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          clacc t[3] = {};
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const clq x = to_clq(from_vec<double>(__ldg(u + 3 * i + k)), top);
            unit.add(i, k, x);
            parts.add(i, k, x);
#pragma unroll
            for (int j = 0; j < 3; ++j) clmac_cj(t[j], x, g[3 * j + k]);
          }
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            kr[3 * i + j] += lacc_value(t[j].re) >> 1;
            ki[3 * i + j] += lacc_value(t[j].im) >> 1;
          }
        }
        bad |= !unit.ok(top);
      }
      {  // U_mu^+(x-mu) g^+(x-mu) = (g(x-mu) U_mu(x-mu))^+
        const double2 *u = U2 + ((int64_t)mu * V + sb) * 9;
        unsigned top = 0;
        unit_check unit;
        clq g[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) g[e] = ldg_q(Gq, (int64_t)e * V + sb);
        bad |= g[0].r.h == kNoLimb;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          clacc t[3] = {};
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const clq x = to_clq(from_vec<double>(__ldg(u + 3 * k + i)), top);
            unit.add(k, i, x);
            parts.add(k, i, x);
#pragma unroll
            for (int j = 0; j < 3; ++j) clmac(t[j], g[3 * j + k], x);
          }
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            kr[3 * i + j] += lacc_value(t[j].re) >> 1;
            ki[3 * i + j] -= lacc_value(t[j].im) >> 1;
          }
        }
        bad |= !unit.ok(top);
      }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) parts.add(e / 3, e % 3, ldg_q(Gq, (int64_t)e * V + s));
    if (bad || parts.small()) {
      m3<double> t;
      const Lattice Lc = L;
      staple_fp64(U2, G, &Lc, s, c, &t);
      K = t;
    } else {
#pragma unroll
      for (int e = 0; e < 9; ++e) K.e[e] = {__ll2double_rn(kr[e]) * 0x1p-59, __ll2double_rn(ki[e]) * 0x1p-59};
    }
  }
  double w[8];
#pragma unroll
  for (int a = 0; a < 8; a += 2) {
    const double2 v = reinterpret_cast<const double2 *>(omega)[s * 4 + a / 2];
    w[a] = v.x;
    w[a + 1] = v.y;
  }
  const double f = -scale / (12.0 * (double)V);  // times Tr[T^a Y], T^a = lambda^a / 2
  const double n2 = algebra_norm2(w);
  double gr[8];
  if (n2 <= kSeriesNorm2) {
    herm x;  // A = (M - M^+)/(2i), M = g K (its trace part drops out)
    {
      cx<double> M[9];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) M[3 * i + j] = {0, 0};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const cx<double> g = ldg(G, (int64_t)(3 * i + k) * V + s);
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            if (i != j) M[3 * i + j] = cmac(M[3 * i + j], g, K.e[3 * k + j]);
            else M[3 * i + j].i = fma(g.r, K.e[3 * k + j].i, fma(g.i, K.e[3 * k + j].r, M[3 * i + j].i));
          }
        }
      }
      auto off = [](cx<double> u, cx<double> l) { return cx<double>{0.5 * (u.i + l.i), 0.5 * (l.r - u.r)}; };
      x = {{M[0].i, M[4].i, M[8].i}, off(M[1], M[3]), off(M[2], M[6]), off(M[5], M[7])};
    }
    const int m = halvings(n2);
    const double sc = __hiloint2double((1023 - m) << 20, 0);
    const herm h = algebra_herm(w, sc);
    const float norm = sqrt((float)n2) * (float)sc;
    herm y = x;
    const float z = 1.41422f * norm;  // bounds |ad_H|: its eigenvalues are differences of those of H
    float term = 1.f;
#pragma unroll 1
    for (int n = 1; n < 19; ++n) {  // z < 0.71: the 18th term is below 1e-18 of the sum
      x = commutator(h, x);
      herm_axpy(y, fabs(kExpCoef[n + 1]), x);
      term *= z / (float)(n + 1);  // z^n / (n+1)!
      if (term < 1e-17f) break;
    }
    if (m > 0) {
      exp_poly p = exp_series(h, norm);
      for (int k = 0; k < m; ++k) {
        m3<double> g;
        exp_matrix(p, h, g);
        conjugate_average(&y, &g);
        exp_double(p);
      }
    }
    const double is3 = 0.28867513459481288225;  // 1/(2 sqrt(3))
    gr[0] = y.a.r;
    gr[1] = -y.a.i;
    gr[2] = 0.5 * (y.d[0] - y.d[1]);
    gr[3] = y.b.r;
    gr[4] = -y.b.i;
    gr[5] = y.c.r;
    gr[6] = -y.c.i;
    gr[7] = is3 * (y.d[0] + y.d[1] - 2.0 * y.d[2]);
  } else {
    m3<double> Kc = K;
    double wc[8], gc[8];
    for (int a = 0; a < 8; ++a) wc[a] = w[a];
    gradient_by_eigenvectors(wc, &Kc, gc);
    for (int a = 0; a < 8; ++a) gr[a] = gc[a];
  }
#pragma unroll
  for (int a = 0; a < 8; a += 2)
    reinterpret_cast<double2 *>(grad)[s * 4 + a / 2] = make_double2(f * gr[a], f * gr[a + 1]);
}

}  // namespace lgf
