// gf_autograd.cuh -- F_U[g] and theta as functions of the Lie-algebra parameters of g,
// and their gradient (the backward of an autograd function), FP64.
//
// g(x) = exp(i X(x)), X = sum_a c_a(x) lambda_a (Gell-Mann); W_mu(x) = g(x) U_mu(x)
// g(x+mu)^+ (Eq. (1)'s transformed links); F(c) = Eq. (1), theta(c) = Eqs. (2)-(3) of W.
//
// Everything here is bound by the FP64 pipe (two lanes per SM), so the passes are laid out
// to form each quantity once and to do it in few FP64 instructions:
//   k_ad_exp       g, one site per thread;
//   k_ad_links     W, once per link (and F), kept for the next passes: 216 instructions a
//                  link.  A pass that rebuilt the links it reads would form each twice
//                  (Delta) or three times (the gradient);
//   k_ad_delta     Delta from the anti-Hermitian parts of W (and theta), kept as its 8 reals;
//   k_ad_backward  the gradient from W and Delta.
// 32^4 at c ~ N(0, 0.3^2), forward and backward: 52.9 ms with links rebuilt per
// pass and exp by matrix Taylor series, 7.4 ms so.
//
// exp.  X is Hermitian and traceless, so X^3 = c1 X + c0 with c1 = Tr X^2 / 2, c0 = det X
// (Cayley-Hamilton; C. Morningstar and M. Peardon, Phys. Rev. D 69, 054501 (2004), use the
// same reduction with closed forms for the coefficients), and every power series in X is
// a polynomial f0 + f1 X + f2 X^2.  Its coefficients come from the scalar recurrence of the
// powers, X^{n+1} = d_n c0 + (a_n + d_n c1) X + b_n X^2, in place of matrix products: five
// instructions a term.  Arguments with a spectral radius above 1 are halved s times first and the
// polynomial is squared modulo X^3 - c1 X - c0 afterwards, up to kPolySquarings times: its
// coefficients grow with the square of the radius where eigenvalues (nearly) coincide, df/dc0
// faster (gradient off by 1.4e-11 at radius 200).  Above that exp and its derivative are
// squared as matrices, L -> exp L + L exp, whose errors grow with the radius only.
//
// Gradient.  With S = sum_mu W_mu(x) (wF + wT B_mu(x)) + W_mu(x-mu)^+ (wF - wT B_mu(x-mu)),
// wF = F_bar / (nd Nc V), wT = -4 theta_bar / (Nc V) and B_nu(y) = Delta(y+nu) - Delta(y)
// (the adjoint of link W_nu(y) in theta), dL = Re Tr[S dg g^+]; dg g^+ is anti-Hermitian and
// traceless, so only that part P of S counts, and the wF terms of P are -wF Delta(x) / 2.
// With E = g^+ P, dL = Re Tr[E dg] and, dg being the derivative of f0 + f1 X + f2 X^2,
//   dL/dc_a = Re Tr[lambda_a (f1 E + f2 (E X + X E) + alpha X^2 + beta X)],
//   alpha = sum_j df_j/dc0 Tr[E X^j],  beta = sum_j df_j/dc1 Tr[E X^j].
// The recurrence gives h = df/dc0 alongside f.  With X^n = q_n p + r_n for p = X^3 - c1 X -
// c0 and r_n its remainder, dr_n/dc0 = q_n mod p and dr_n/dc1 = X q_n mod p: df/dc1 is X h.
// The backward recomputes g, W and Delta from c and U (nothing is kept from the forward).
#pragma once

#include "gf_kernels.cuh"

namespace gf {

// Hermitian traceless X = sum_a c_a lambda_a: real diagonal and upper triangle
struct Herm {
  double d0, d1, d2;
  c64 x01, x02, x12;
};

__device__ __forceinline__ Herm lie_to_X(const double* __restrict__ c) {
  const double s3 = 0.57735026918962576451;  // 1/sqrt(3)
  const double2* p = reinterpret_cast<const double2*>(c);
  const bool wide = (reinterpret_cast<uintptr_t>(c) & 15) == 0;  // c is 8-byte aligned
  double v[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (wide) {
      const double2 w = p[k];
      v[2 * k] = w.x;
      v[2 * k + 1] = w.y;
    } else {
      v[2 * k] = c[2 * k];
      v[2 * k + 1] = c[2 * k + 1];
    }
  }
  const double e = s3 * v[7];
  return {v[2] + e, e - v[2], -2.0 * e, {v[0], -v[1]}, {v[3], -v[4]}, {v[5], -v[6]}};
}

// X^2 (Hermitian, its trace kept)
__device__ __forceinline__ Herm herm_square(const Herm& x) {
  Herm q;
  const double n01 = cnorm2(x.x01), n02 = cnorm2(x.x02), n12 = cnorm2(x.x12);
  q.d0 = gf_fma(x.d0, x.d0, n01 + n02);
  q.d1 = gf_fma(x.d1, x.d1, n01 + n12);
  q.d2 = gf_fma(x.d2, x.d2, n02 + n12);
  // (01) = x01 (d0 + d1) + x02 conj(x12); d0 + d1 = -d2, and so on
  q.x01 = cmul_conj_fma(x.x02, x.x12);
  q.x01 = {gf_fma(-x.d2, x.x01.re, q.x01.re), gf_fma(-x.d2, x.x01.im, q.x01.im)};
  q.x02 = cmul_fma(x.x01, x.x12);
  q.x02 = {gf_fma(-x.d1, x.x02.re, q.x02.re), gf_fma(-x.d1, x.x02.im, q.x02.im)};
  q.x12 = cmul_conj_fma(x.x02, x.x01);
  q.x12 = {gf_fma(-x.d0, x.x12.re, q.x12.re), gf_fma(-x.d0, x.x12.im, q.x12.im)};
  return q;
}

// a b modulo p = X^3 - c1 X - c0, for polynomials of degree 2 with complex coefficients
__device__ __forceinline__ void poly_mul(const c64 (&a)[3], const c64 (&b)[3], double c0, double c1,
                                         c64 (&out)[3]) {
  c64 p3 = cmul_fma(a[1], b[2]);
  cmac(p3, a[2], b[1]);
  const c64 p4 = cmul_fma(a[2], b[2]);
  c64 p0 = cmul_fma(a[0], b[0]), p1 = cmul_fma(a[0], b[1]), p2 = cmul_fma(a[0], b[2]);
  cmac(p1, a[1], b[0]);
  cmac(p2, a[1], b[1]);
  cmac(p2, a[2], b[0]);
  out[0] = {gf_fma(c0, p3.re, p0.re), gf_fma(c0, p3.im, p0.im)};
  out[1] = {gf_fma(c0, p4.re, gf_fma(c1, p3.re, p1.re)), gf_fma(c0, p4.im, gf_fma(c1, p3.im, p1.im))};
  out[2] = {gf_fma(c1, p4.re, p2.re), gf_fma(c1, p4.im, p2.im)};
}

// Tr X^2 / 2
__device__ __forceinline__ double herm_c1(const Herm& x) {
  return 0.5 * gf_fma(x.d0, x.d0, gf_fma(x.d1, x.d1, x.d2 * x.d2)) + (cnorm2(x.x01) + cnorm2(x.x02) + cnorm2(x.x12));
}

constexpr int kPolySquarings = 3;  // radius 8
// whether exp_coefficients halves x more often than that
__device__ __forceinline__ bool exp_is_large(const Herm& x) { return herm_c1(x) * (4.0 / 3.0) > 64.0; }

// exp(i 2^k x) = f0 + f1 x + f2 x^2, k = min(s, kPolySquarings), for the scaled x (x := 2^-s X on
// return, s the returned value) and, with DERIV, h = df/dc0 at fixed c1 (c0, c1 of the scaled x).
template <bool DERIV>
__device__ __forceinline__ int exp_coefficients(Herm& x, c64 (&f)[3], c64 (&h)[3], double& c0, double& c1) {
  c1 = herm_c1(x);
  // the largest eigenvalue is at most 2 sqrt(c1 / 3)
  int s = 0;
  double r2 = c1 * (4.0 / 3.0);
  while (r2 > 1.0 && s < 60) {
    r2 *= 0.25;
    ++s;
  }
  if (s) {
    const double sc = __hiloint2double((1023 - s) << 20, 0);  // 2^-s
    x.d0 *= sc; x.d1 *= sc; x.d2 *= sc;
    x.x01 = cscale(x.x01, sc);
    x.x02 = cscale(x.x02, sc);
    x.x12 = cscale(x.x12, sc);
    c1 *= sc * sc;
  }
  // det: d0 d1 d2 + 2 Re(x01 x12 conj(x02)) - d0 |x12|^2 - d1 |x02|^2 - d2 |x01|^2
  const c64 t = cmul_fma(x.x01, x.x12);
  c0 = 2.0 * gf_fma(t.re, x.x02.re, t.im * x.x02.im);
  c0 = gf_fma(x.d0, gf_fma(x.d1, x.d2, -cnorm2(x.x12)), c0);
  c0 = gf_fma(-x.d1, cnorm2(x.x02), c0);
  c0 = gf_fma(-x.d2, cnorm2(x.x01), c0);
  // X^n = a + b X + d X^2 (from n = 2 on), da = d/dc0 and so on; terms i^n / n! up to n = 20
  // (1 / 21! = 2e-20)
  constexpr double inv_fact[21] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040,
                                   1.0 / 40320, 1.0 / 362880, 1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600,
                                   1.0 / 6227020800.0, 1.0 / 87178291200.0, 1.0 / 1307674368000.0,
                                   1.0 / 20922789888000.0, 1.0 / 355687428096000.0, 1.0 / 6402373705728000.0,
                                   1.0 / 121645100408832000.0, 1.0 / 2432902008176640000.0};
  double a = 0.0, b = 0.0, d = 1.0, da = 0.0, db = 0.0, dd = 0.0;
  f[0] = {1.0, 0.0};
  f[1] = {0.0, 1.0};
  f[2] = {-0.5, 0.0};
#pragma unroll
  for (int j = 0; j < 3; ++j) h[j] = {0.0, 0.0};
#pragma unroll
  for (int n = 3; n <= 20; ++n) {
    if (DERIV) {
      const double na = gf_fma(c0, dd, d), nb = gf_fma(c1, dd, da), nd = db;
      da = na;
      db = nb;
      dd = nd;
    }
    const double na = d * c0, nb = gf_fma(d, c1, a), nd = b;
    a = na;
    b = nb;
    d = nd;
    const double w = (n & 2) ? -inv_fact[n] : inv_fact[n];  // i^n = 1, i, -1, -i
    if (n & 1) {
      f[0].im = gf_fma(w, a, f[0].im);
      f[1].im = gf_fma(w, b, f[1].im);
      f[2].im = gf_fma(w, d, f[2].im);
      if (DERIV) {
        h[0].im = gf_fma(w, da, h[0].im);
        h[1].im = gf_fma(w, db, h[1].im);
        h[2].im = gf_fma(w, dd, h[2].im);
      }
    } else {
      f[0].re = gf_fma(w, a, f[0].re);
      f[1].re = gf_fma(w, b, f[1].re);
      f[2].re = gf_fma(w, d, f[2].re);
      if (DERIV) {
        h[0].re = gf_fma(w, da, h[0].re);
        h[1].re = gf_fma(w, db, h[1].re);
        h[2].re = gf_fma(w, dd, h[2].re);
      }
    }
  }
#pragma unroll 1
  for (int k = 0; k < (s < kPolySquarings ? s : kPolySquarings); ++k) {
    c64 sq[3];
    poly_mul(f, f, c0, c1, sq);
    if (DERIV) {
      // f^2 = q p + sq with q = 2 f1 f2 + f2^2 X, so d sq/dc0 = 2 f h mod p + q
      c64 fh[3];
      poly_mul(f, h, c0, c1, fh);
      const c64 q0 = cmul_fma(f[1], f[2]), q1 = cmul_fma(f[2], f[2]);
      h[0] = cscale(cadd(fh[0], q0), 2.0);
      h[1] = {gf_fma(2.0, fh[1].re, q1.re), gf_fma(2.0, fh[1].im, q1.im)};
      h[2] = cscale(fh[2], 2.0);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) f[j] = sq[j];
  }
  return s;
}

__device__ __forceinline__ void m3_mul(const c64* a, const c64* b, c64* out) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      c64 v = cmul_fma(a[3 * i], b[j]);
      cmac(v, a[3 * i + 1], b[3 + j]);
      cmac(v, a[3 * i + 2], b[6 + j]);
      out[3 * i + j] = v;
    }
}
// g -> g^(2^n), and with it the derivative z -> that of the power: the rare sites of large
// parameters, kept out of the callers' registers
__device__ __noinline__ void m3_squarings(c64* g, c64* z, int n) {
#pragma unroll 1
  for (int k = 0; k < n; ++k) {
    c64 t[9], u[9];
    if (z) {
      m3_mul(g, z, t);
      m3_mul(z, g, u);
      for (int e = 0; e < 9; ++e) z[e] = cadd(t[e], u[e]);
    }
    m3_mul(g, g, t);
    for (int e = 0; e < 9; ++e) g[e] = t[e];
  }
}

// acc + s a for a real s
__device__ __forceinline__ void rmac(c64& acc, double s, c64 a) {
  acc.re = gf_fma(s, a.re, acc.re);
  acc.im = gf_fma(s, a.im, acc.im);
}
// acc + i s a
__device__ __forceinline__ void imac(c64& acc, double s, c64 a) {
  acc.re = gf_fma(-s, a.im, acc.re);
  acc.im = gf_fma(s, a.re, acc.im);
}

// f0 + f1 X + f2 X^2, Q = X^2
__device__ __forceinline__ void poly_matrix(const c64 (&f)[3], const Herm& X, const Herm& Q, c64* g) {
  g[0] = f[0]; rmac(g[0], X.d0, f[1]); rmac(g[0], Q.d0, f[2]);
  g[4] = f[0]; rmac(g[4], X.d1, f[1]); rmac(g[4], Q.d1, f[2]);
  g[8] = f[0]; rmac(g[8], X.d2, f[1]); rmac(g[8], Q.d2, f[2]);
  g[1] = cmul_fma(f[1], X.x01); cmac(g[1], f[2], Q.x01);
  g[2] = cmul_fma(f[1], X.x02); cmac(g[2], f[2], Q.x02);
  g[5] = cmul_fma(f[1], X.x12); cmac(g[5], f[2], Q.x12);
  g[3] = cmul_conj_fma(f[1], X.x01); cmac_conj(g[3], f[2], Q.x01);
  g[6] = cmul_conj_fma(f[1], X.x02); cmac_conj(g[6], f[2], Q.x02);
  g[7] = cmul_conj_fma(f[1], X.x12); cmac_conj(g[7], f[2], Q.x12);
}

// ------------------------------------------------------------------------- site and buffers
// A thread's site from its number i within the time slices t0, t0 + 1, ... of a launch.
struct AdSite {
  unsigned s3;       // lexicographic index within the slice
  int x, y, z, t;
};
__device__ __forceinline__ AdSite ad_site(const LatDev& lat, unsigned i, int t0) {
  const unsigned V3 = 2u * (unsigned)lat.V3h;
  const unsigned k = i / V3;
  AdSite s;
  s.s3 = i - k * V3;
  int t = t0 + (int)k;
  if (t >= lat.L[3]) t -= lat.L[3];
  s.t = t;
  const unsigned q1 = __umulhi(s.s3, lat.mx), q2 = __umulhi(q1, lat.my);
  s.x = (int)(s.s3 - q1 * (unsigned)lat.L[0]);
  s.y = (int)(q1 - q2 * (unsigned)lat.L[1]);
  s.z = (int)q2;
  return s;
}
// the neighbour in direction mu (dir = +1 or -1), periodic
__device__ __forceinline__ AdSite ad_step(const LatDev& lat, AdSite s, int mu, int dir) {
  const int L = lat.L[mu];
  const int c = mu == 0 ? s.x : mu == 1 ? s.y : mu == 2 ? s.z : s.t;
  const int n = dir > 0 ? (c == L - 1 ? 0 : c + 1) : (c == 0 ? L - 1 : c - 1);
  if (mu == 3) {
    s.t = n;
    return s;
  }
  const int stride = mu == 0 ? 1 : mu == 1 ? lat.L[0] : lat.L[0] * lat.L[1];
  s.s3 = (unsigned)((int)s.s3 + (n - c) * stride);
  if (mu == 0) s.x = n;
  else if (mu == 1) s.y = n;
  else s.z = n;
  return s;
}
__device__ __forceinline__ long long ad_lexi(const LatDev& lat, const AdSite& s) {
  return (long long)s.t * (2LL * lat.V3h) + s.s3;
}
// place in the W buffer, which holds the slices w_t0, w_t0 + 1, ... (periodic)
__device__ __forceinline__ long long ad_wplace(const AdArgs& a, const AdSite& s) {
  int tl = s.t - a.w_t0;
  if (tl < 0) tl += a.lat.L[3];
  return (long long)tl * (2LL * a.lat.V3h) + s.s3;
}

// planes of 16-byte words, one entry per site
__device__ __forceinline__ void ad_load9(const c64* __restrict__ base, long long n, long long at, c64 (&m)[9]) {
  const double2* p = reinterpret_cast<const double2*>(base) + at;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const double2 v = p[e * n];
    m[e] = {v.x, v.y};
  }
}
__device__ __forceinline__ void ad_store9(c64* base, long long n, long long at, const c64 (&m)[9]) {
  double2* p = reinterpret_cast<double2*>(base) + at;
#pragma unroll
  for (int e = 0; e < 9; ++e) p[e * n] = make_double2(m[e].re, m[e].im);
}

__device__ __forceinline__ int ad_storage_idx(const LatDev& lat, const AdSite& s) {
  return ((s.x + s.y + s.z + s.t) & 1) * lat.Vh + (int)(ad_lexi(lat, s) >> 1);
}
// W_mu(s) from the buffer, or formed (BUF false)
template <bool BUF>
__device__ __forceinline__ void ad_link(const AdArgs& a, const AdSite& s, int mu, c64 (&u)[9]) {
  if constexpr (BUF) {
    ad_load9(a.w + 9 * mu * a.w_n, a.w_n, ad_wplace(a, s), u);
  } else {
    c64 g[9];
    Store<GF_FP64_18>::load(a.links + a.lat.off_bytes, a.lat.V, mu, ad_storage_idx(a.lat, s), u);
    ad_load9(a.g, a.lat.V, ad_lexi(a.lat, s), g);
    left_mul(g, u);
    ad_load9(a.g, a.lat.V, ad_lexi(a.lat, ad_step(a.lat, s, mu, +1)), g);
    right_mul_dag(u, g);
  }
}

// anti-Hermitian traceless matrix: upper triangle and the imaginary diagonal
struct AntiH {
  c64 b01, b02, b12;
  double d0, d1, d2;
};
__device__ __forceinline__ AntiH ad_load_delta(const AdArgs& a, long long at) {
  const double2* p = reinterpret_cast<const double2*>(a.delta) + at;
  const double2 u = p[0], v = p[a.lat.V], w = p[2 * a.lat.V], d = p[3 * a.lat.V];
  return {{u.x, u.y}, {v.x, v.y}, {w.x, w.y}, d.x, d.y, -(d.x + d.y)};
}
__device__ __forceinline__ AntiH antih_sub(const AntiH& x, const AntiH& y) {
  return {csub(x.b01, y.b01), csub(x.b02, y.b02), csub(x.b12, y.b12), x.d0 - y.d0, x.d1 - y.d1, x.d2 - y.d2};
}

// R += C - C^+ for C = M B, M = W or W^+ (DAG): the three upper elements and the imaginary
// diagonal (75 instructions)
template <bool DAG>
__device__ __forceinline__ c64 ad_el(const c64 (&W)[9], int i, int j) {
  return DAG ? cconj(W[3 * j + i]) : W[3 * i + j];
}
template <bool DAG>
__device__ __forceinline__ void add_antih_product(AntiH& R, const c64 (&W)[9], const AntiH& B) {
  const c64 n10 = cneg(cconj(B.b01)), n20 = cneg(cconj(B.b02)), n21 = cneg(cconj(B.b12));
#define M_(i, j) ad_el<DAG>(W, i, j)
  // C01 - conj(C10); conj(C10) = conj(M10 i d0 + M11 n10 + M12 n20)
  cmac(R.b01, M_(0, 0), B.b01);
  imac(R.b01, B.d1, M_(0, 1));
  cmac(R.b01, M_(0, 2), n21);
  imac(R.b01, B.d0, cconj(M_(1, 0)));  // - conj(i d0 M) = i d0 conj(M)
  cmac(R.b01, cconj(M_(1, 1)), B.b01); // - conj(M n10) = conj(M) b01
  cmac(R.b01, cconj(M_(1, 2)), B.b02);
  // C02 - conj(C20)
  cmac(R.b02, M_(0, 0), B.b02);
  cmac(R.b02, M_(0, 1), B.b12);
  imac(R.b02, B.d2, M_(0, 2));
  imac(R.b02, B.d0, cconj(M_(2, 0)));
  cmac(R.b02, cconj(M_(2, 1)), B.b01);
  cmac(R.b02, cconj(M_(2, 2)), B.b02);
  // C12 - conj(C21); - conj(M20 b01) = conj(M20) n10
  cmac(R.b12, M_(1, 0), B.b02);
  cmac(R.b12, M_(1, 1), B.b12);
  imac(R.b12, B.d2, M_(1, 2));
  cmac(R.b12, cconj(M_(2, 0)), n10);
  imac(R.b12, B.d1, cconj(M_(2, 1)));
  cmac(R.b12, cconj(M_(2, 2)), B.b12);
  // Im C_kk (half of C - C^+ there; doubled by the caller)
  const c64 m00 = M_(0, 0), m01 = M_(0, 1), m02 = M_(0, 2), m10 = M_(1, 0), m11 = M_(1, 1), m12 = M_(1, 2);
  const c64 m20 = M_(2, 0), m21 = M_(2, 1), m22 = M_(2, 2);
#undef M_
  R.d0 = gf_fma(m00.re, B.d0, R.d0);
  R.d0 = gf_fma(m01.re, n10.im, gf_fma(m01.im, n10.re, R.d0));
  R.d0 = gf_fma(m02.re, n20.im, gf_fma(m02.im, n20.re, R.d0));
  R.d1 = gf_fma(m10.re, B.b01.im, gf_fma(m10.im, B.b01.re, R.d1));
  R.d1 = gf_fma(m11.re, B.d1, R.d1);
  R.d1 = gf_fma(m12.re, n21.im, gf_fma(m12.im, n21.re, R.d1));
  R.d2 = gf_fma(m20.re, B.b02.im, gf_fma(m20.im, B.b02.re, R.d2));
  R.d2 = gf_fma(m21.re, B.b12.im, gf_fma(m21.im, B.b12.re, R.d2));
  R.d2 = gf_fma(m22.re, B.d2, R.d2);
}

}  // namespace gf
