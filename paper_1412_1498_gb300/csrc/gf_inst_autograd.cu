// gf_inst_autograd.cu -- forward and backward of F(c), theta(c) (FP64-18 storage).
#include "gf_autograd.cuh"

namespace gf {

namespace {
constexpr int kT = 128;
}

__global__ void __launch_bounds__(kT) k_ad_exp(AdArgs a) {
  const long long x = blockIdx.x * (long long)kT + threadIdx.x;
  if (x >= a.lat.V) return;
  Herm X = lie_to_X(a.c + 8 * x);
  c64 f[3], h[3];
  double c0, c1;
  const int s = exp_coefficients<false>(X, f, h, c0, c1);
  c64 g[9];
  poly_matrix(f, X, herm_square(X), g);
  if (s > kPolySquarings) {
    c64 t[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) t[e] = g[e];
    m3_squarings(t, nullptr, s - kPolySquarings);
#pragma unroll
    for (int e = 0; e < 9; ++e) g[e] = t[e];
  }
  ad_store9(a.g, a.lat.V, x, g);
}

// W_mu(x) = g(x) U_mu(x) g(x+mu)^+ for the sites of `n_t` slices from a.w_t0 on, and Re Tr
// of those whose slice is one of the n_f from f_t0 on (a slab's halo slice belongs to
// another slab's F).  Without a buffer (BUF false): the whole lattice, for F alone.
template <bool BUF>
__global__ void __launch_bounds__(kT) k_ad_links(AdArgs a, int n_t, int f_t0, int n_f, int part0) {
  __shared__ double red[32];
  const unsigned i = blockIdx.x * (unsigned)kT + threadIdx.x;
  const unsigned n = 2u * (unsigned)a.lat.V3h * (unsigned)n_t;
  double v[1] = {0.0};
  if (i < n) {
    const AdSite s = ad_site(a.lat, i, a.w_t0);
    const long long lexi = ad_lexi(a.lat, s), place = BUF ? ad_wplace(a, s) : 0;
    const int idx = ad_storage_idx(a.lat, s);
    int tf = s.t - f_t0;
    if (tf < 0) tf += a.lat.L[3];
    c64 g[9];
    ad_load9(a.g, a.lat.V, lexi, g);
    double f = 0.0;
#pragma unroll 1
    for (int mu = 0; mu < a.nd; ++mu) {
      cx<double> u[9];
      Store<GF_FP64_18>::load(a.links + a.lat.off_bytes, a.lat.V, mu, idx, u);
      c64 gn[9];
      ad_load9(a.g, a.lat.V, ad_lexi(a.lat, ad_step(a.lat, s, mu, +1)), gn);
      left_mul(g, u);
      right_mul_dag(u, gn);
      f += u[0].re + u[4].re + u[8].re;
      if constexpr (BUF) ad_store9(a.w + 9 * mu * a.w_n, a.w_n, place, u);
    }
    if (tf < n_f) v[0] = f;
  }
  block_sum<1>(v, red);
  if (threadIdx.x == 0) a.part[2 * (part0 + blockIdx.x)] = v[0];
}

// Delta(x) (Eq. (3)) of the slices t0 .. t0 + n_t - 1 and Tr[Delta Delta^+].  The last block
// of the last slab's launch adds the partials of all `n_parts` blocks in a fixed order.
template <bool BUF>
__global__ void __launch_bounds__(kT) k_ad_delta(AdArgs a, int t0, int n_t, int part0, int n_links_parts,
                                                 int n_parts) {
  __shared__ double red[64];
  __shared__ int s_last;
  const unsigned i = blockIdx.x * (unsigned)kT + threadIdx.x;
  const unsigned n = 2u * (unsigned)a.lat.V3h * (unsigned)n_t;
  double v[1] = {0.0};
  if (i < n) {
    const AdSite s = ad_site(a.lat, i, t0);
    // D = A - A^+, A = sum_nu W_nu(x - nu) - W_nu(x): upper elements, imaginary diagonal
    c64 d01 = {0.0, 0.0}, d02 = d01, d12 = d01;
    double e0 = 0.0, e1 = 0.0, e2 = 0.0;
#pragma unroll 1
    for (int nu = 0; nu < a.nd; ++nu) {
      c64 f[9], b[9];
      ad_link<BUF>(a, s, nu, f);
      ad_link<BUF>(a, ad_step(a.lat, s, nu, -1), nu, b);
      d01 = cadd(d01, csub(csub(b[1], f[1]), cconj(csub(b[3], f[3]))));
      d02 = cadd(d02, csub(csub(b[2], f[2]), cconj(csub(b[6], f[6]))));
      d12 = cadd(d12, csub(csub(b[5], f[5]), cconj(csub(b[7], f[7]))));
      e0 += b[0].im - f[0].im;
      e1 += b[4].im - f[4].im;
      e2 += b[8].im - f[8].im;
    }
    const double tr = (e0 + e1 + e2) * (1.0 / 3.0);
    e0 = 2.0 * (e0 - tr);
    e1 = 2.0 * (e1 - tr);
    e2 = 2.0 * (e2 - tr);
    const long long x = ad_lexi(a.lat, s);
    double2* p = reinterpret_cast<double2*>(a.delta) + x;
    p[0] = make_double2(d01.re, d01.im);
    p[a.lat.V] = make_double2(d02.re, d02.im);
    p[2 * a.lat.V] = make_double2(d12.re, d12.im);
    p[3 * a.lat.V] = make_double2(e0, e1);
    v[0] = 2.0 * (cnorm2(d01) + cnorm2(d02) + cnorm2(d12)) + gf_fma(e0, e0, gf_fma(e1, e1, e2 * e2));
  }
  if (a.out == nullptr) return;  // the backward's Delta: no sums
  block_sum<1>(v, red);
  if (threadIdx.x == 0) {
    a.part[2 * (part0 + blockIdx.x) + 1] = v[0];
    __threadfence();
    s_last = atomicAdd(a.ticket, 1u) == (unsigned)n_parts - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double w[2] = {0.0, 0.0};
  for (int k = threadIdx.x; k < n_links_parts; k += kT) w[0] += __ldcg(a.part + 2 * k);
  for (int k = threadIdx.x; k < n_parts; k += kT) w[1] += __ldcg(a.part + 2 * k + 1);
  __syncthreads();  // block_sum's shared words are free again
  block_sum<2>(w, red);
  if (threadIdx.x == 0) {
    a.out[0] = w[0] / ((double)a.nd * 3.0 * (double)a.lat.V);
    a.out[1] = w[1] / (3.0 * (double)a.lat.V);
    *a.ticket = 0u;
  }
}

// M = E X + X E and the factors of X^2 and X in the derivative in the direction E (gf_autograd.cuh)
__device__ __forceinline__ void frechet_terms(const c64 (&E)[9], const Herm& X, const c64 (&h)[3], double c0, double c1,
                                              c64 (&M)[9], c64& alpha, c64& beta) {
  const c64 trE = cadd(cadd(E[0], E[4]), E[8]);
  c64 trEX, trEX2;
  {
    const c64 c01 = cconj(X.x01), c02 = cconj(X.x02), c12 = cconj(X.x12);
    c64 EX[9];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const c64 e0 = E[3 * r], e1 = E[3 * r + 1], e2 = E[3 * r + 2];
      EX[3 * r] = cmul_fma(e1, c01);
      cmac(EX[3 * r], e2, c02);
      rmac(EX[3 * r], X.d0, e0);
      EX[3 * r + 1] = cmul_fma(e0, X.x01);
      cmac(EX[3 * r + 1], e2, c12);
      rmac(EX[3 * r + 1], X.d1, e1);
      EX[3 * r + 2] = cmul_fma(e0, X.x02);
      cmac(EX[3 * r + 2], e1, X.x12);
      rmac(EX[3 * r + 2], X.d2, e2);
    }
    trEX = cadd(cadd(EX[0], EX[4]), EX[8]);
    trEX2 = cmul_fma(EX[1], c01);
    cmac(trEX2, EX[2], c02);
    cmac(trEX2, EX[5], c12);
    cmac(trEX2, EX[3], X.x01);
    cmac(trEX2, EX[6], X.x02);
    cmac(trEX2, EX[7], X.x12);
    rmac(trEX2, X.d0, EX[0]);
    rmac(trEX2, X.d1, EX[4]);
    rmac(trEX2, X.d2, EX[8]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const c64 e0 = E[c], e1 = E[3 + c], e2 = E[6 + c];
      M[c] = EX[c];
      rmac(M[c], X.d0, e0);
      cmac(M[c], X.x01, e1);
      cmac(M[c], X.x02, e2);
      M[3 + c] = EX[3 + c];
      cmac(M[3 + c], c01, e0);
      rmac(M[3 + c], X.d1, e1);
      cmac(M[3 + c], X.x12, e2);
      M[6 + c] = EX[6 + c];
      cmac(M[6 + c], c02, e0);
      cmac(M[6 + c], c12, e1);
      rmac(M[6 + c], X.d2, e2);
    }
  }
  alpha = cmul_fma(h[0], trE);
  beta = cmul_fma(cscale(h[2], c0), trE);
  cmac(alpha, h[1], trEX);
  cmac(alpha, h[2], trEX2);
  cmac(beta, c64{gf_fma(c1, h[2].re, h[0].re), gf_fma(c1, h[2].im, h[0].im)}, trEX);
  cmac(beta, h[1], trEX2);
}

// The gradient of a site whose exponential is squared as a matrix: Z, the derivative of exp(i 2^k x)
// in the direction E, as a whole matrix.  The polynomial's terms leave its multiple of 1 open
// (they assume a traceless dx), which Tr Z = i 2^k Tr[E exp(i 2^k x)] fixes.  Not inlined: the
// other sites' registers stay free of it.
__device__ __noinline__ void ad_gradient_large(const c64* Ep, const double* c, double* out) {
  c64 E[9], M[9], f[3], h[3], alpha, beta;
#pragma unroll
  for (int e = 0; e < 9; ++e) E[e] = Ep[e];
  Herm X = lie_to_X(c);
  double c0, c1;
  const int sh = exp_coefficients<true>(X, f, h, c0, c1);
  frechet_terms(E, X, h, c0, c1, M, alpha, beta);
  const Herm Q = herm_square(X);
  c64 g[9], z[9];
  poly_matrix(f, X, Q, g);
  const c64 fz[3] = {{0.0, 0.0}, beta, alpha};
  poly_matrix(fz, X, Q, z);
  c64 trEg = {0.0, 0.0}, tr = {0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      cmac(z[3 * i + j], f[1], E[3 * i + j]);
      cmac(z[3 * i + j], f[2], M[3 * i + j]);
      cmac(trEg, E[3 * i + j], g[3 * j + i]);
    }
  tr = cadd(cadd(z[0], z[4]), z[8]);
  constexpr double p = 1 << kPolySquarings;
  const c64 one = {(-p * trEg.im - tr.re) / 3.0, (p * trEg.re - tr.im) / 3.0};
  z[0] = cadd(z[0], one);
  z[4] = cadd(z[4], one);
  z[8] = cadd(z[8], one);
  m3_squarings(g, z, sh - kPolySquarings);
  const double s3 = 0.57735026918962576451;
  const double sc = __hiloint2double((1023 - sh) << 20, 0);  // 2^-s: dx = 2^-s dX
  // Re Tr[lambda_a Z]
  out[0] = sc * (z[1].re + z[3].re);
  out[1] = sc * (z[3].im - z[1].im);
  out[2] = sc * (z[0].re - z[4].re);
  out[3] = sc * (z[2].re + z[6].re);
  out[4] = sc * (z[6].im - z[2].im);
  out[5] = sc * (z[5].re + z[7].re);
  out[6] = sc * (z[7].im - z[5].im);
  out[7] = sc * (s3 * (z[0].re + z[4].re - 2.0 * z[8].re));
}

template <bool BUF>
__global__ void __launch_bounds__(kT, 4) k_ad_backward(AdArgs a, int t0, int n_t) {
  const unsigned i = blockIdx.x * (unsigned)kT + threadIdx.x;
  if (i >= 2u * (unsigned)a.lat.V3h * (unsigned)n_t) return;
  const AdSite s = ad_site(a.lat, i, t0);
  const long long x = ad_lexi(a.lat, s);
  const double V = (double)a.lat.V;
  const double wF = a.upstream[0] / ((double)a.nd * 3.0 * V);
  const double wT = -a.upstream[1] * 4.0 / (3.0 * V);
  // R = S - S^+ without the weights: sum_mu W_mu(x) B_mu(x) - W_mu(x-mu)^+ B_mu(x-mu)
  const AntiH D = ad_load_delta(a, x);
  AntiH R = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}, 0.0, 0.0, 0.0};
#pragma unroll 1
  for (int mu = 0; mu < a.nd; ++mu) {
    const AdSite sp = ad_step(a.lat, s, mu, +1), sm = ad_step(a.lat, s, mu, -1);
    c64 u[9];
    ad_link<BUF>(a, s, mu, u);
    add_antih_product<false>(R, u, antih_sub(ad_load_delta(a, ad_lexi(a.lat, sp)), D));
    ad_link<BUF>(a, sm, mu, u);
    // -B_mu(x-mu) = Delta(x-mu) - Delta(x)
    add_antih_product<true>(R, u, antih_sub(ad_load_delta(a, ad_lexi(a.lat, sm)), D));
  }
  // P = R / 2, traceless, with the wF part -wF Delta(x) / 2
  const double hT = 0.5 * wT, hF = -0.5 * wF;
  AntiH P;
  P.b01 = {gf_fma(hF, D.b01.re, hT * R.b01.re), gf_fma(hF, D.b01.im, hT * R.b01.im)};
  P.b02 = {gf_fma(hF, D.b02.re, hT * R.b02.re), gf_fma(hF, D.b02.im, hT * R.b02.im)};
  P.b12 = {gf_fma(hF, D.b12.re, hT * R.b12.re), gf_fma(hF, D.b12.im, hT * R.b12.im)};
  const double tr = (R.d0 + R.d1 + R.d2) * (1.0 / 3.0);
  P.d0 = gf_fma(hF, D.d0, wT * (R.d0 - tr));
  P.d1 = gf_fma(hF, D.d1, wT * (R.d1 - tr));
  P.d2 = gf_fma(hF, D.d2, wT * (R.d2 - tr));
  // E = g^+ P
  c64 E[9];
  {
    c64 g[9];
    ad_load9(a.g, a.lat.V, x, g);
    const c64 n10 = cneg(cconj(P.b01)), n20 = cneg(cconj(P.b02)), n21 = cneg(cconj(P.b12));
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const c64 g0 = cconj(g[r]), g1 = cconj(g[3 + r]), g2 = cconj(g[6 + r]);
      E[3 * r] = cmul_fma(g1, n10);
      cmac(E[3 * r], g2, n20);
      imac(E[3 * r], P.d0, g0);
      E[3 * r + 1] = cmul_fma(g0, P.b01);
      cmac(E[3 * r + 1], g2, n21);
      imac(E[3 * r + 1], P.d1, g1);
      E[3 * r + 2] = cmul_fma(g0, P.b02);
      cmac(E[3 * r + 2], g1, P.b12);
      imac(E[3 * r + 2], P.d2, g2);
    }
  }
  Herm X = lie_to_X(a.c + 8 * x);
  if (exp_is_large(X)) {
    c64 t[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) t[e] = E[e];
    ad_gradient_large(t, a.c + 8 * x, a.grad + 8 * x);
    return;
  }
  c64 f[3], h[3];
  double c0, c1;
  const int sh = exp_coefficients<true>(X, f, h, c0, c1);
  c64 M[9], alpha, beta;
  frechet_terms(E, X, h, c0, c1, M, alpha, beta);
  // Z = f1 E + f2 M + alpha X^2 + beta X; only its Hermitian part counts.  The X terms have
  // a Hermitian part Re(alpha) X^2 + Re(beta) X.
  const Herm Q = herm_square(X);
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    c64 z = cmul_fma(f[1], E[e]);
    cmac(z, f[2], M[e]);
    E[e] = z;
  }
  const double ar = alpha.re, br = beta.re;
  const c64 z01 = {gf_fma(ar, Q.x01.re, br * X.x01.re), gf_fma(ar, Q.x01.im, br * X.x01.im)};
  const c64 z02 = {gf_fma(ar, Q.x02.re, br * X.x02.re), gf_fma(ar, Q.x02.im, br * X.x02.im)};
  const c64 z12 = {gf_fma(ar, Q.x12.re, br * X.x12.re), gf_fma(ar, Q.x12.im, br * X.x12.im)};
  const double z0 = gf_fma(ar, Q.d0, gf_fma(br, X.d0, E[0].re));
  const double z1 = gf_fma(ar, Q.d1, gf_fma(br, X.d1, E[4].re));
  const double z2 = gf_fma(ar, Q.d2, gf_fma(br, X.d2, E[8].re));
  const double s3 = 0.57735026918962576451;
  const double sc = __hiloint2double((1023 - sh) << 20, 0);  // 2^-s: dx = 2^-s dX
  double gr[8];
  gr[0] = sc * gf_fma(2.0, z01.re, E[1].re + E[3].re);
  gr[1] = sc * gf_fma(-2.0, z01.im, E[3].im - E[1].im);
  gr[2] = sc * (z0 - z1);
  gr[3] = sc * gf_fma(2.0, z02.re, E[2].re + E[6].re);
  gr[4] = sc * gf_fma(-2.0, z02.im, E[6].im - E[2].im);
  gr[5] = sc * gf_fma(2.0, z12.re, E[5].re + E[7].re);
  gr[6] = sc * gf_fma(-2.0, z12.im, E[7].im - E[5].im);
  gr[7] = sc * (s3 * gf_fma(-2.0, z2, z0 + z1));
  double* out = a.grad + 8 * x;
#pragma unroll
  for (int k = 0; k < 8; ++k) out[k] = gr[k];
}

static unsigned int blocks(long long n) { return (unsigned int)((n + kT - 1) / kT); }

// Time slices of sites that one pass over the W buffer serves: all of them when the buffer
// holds the lattice, else as many as it holds besides the slice before them (whose time
// links they need).  Without a buffer (w_slices = 0) one pass serves the lattice.
static int slab_slices(int w_slices, int Lt) { return w_slices == 0 || w_slices >= Lt ? Lt : w_slices - 1; }
static int slab_slices(const AdArgs& a) { return slab_slices(a.w_slices, a.lat.L[3]); }

// Slices of W the workspace keeps: the whole lattice up to kWBytes (15 million sites), else
// what kWBytes hold (at least two slices); larger lattices are served in slabs, which
// form the links twice in the backward.  With few and very large time slices two of them
// can cost far more than the lattice's other buffers (32 x 32 x 65536 sites: 77 GB); a lattice on which the
// buffer would take more than kWBytes above the 80 bytes a site that it saves in g and Delta
// keeps none (0), and its passes form the links they need (twice as many products).
int ad_w_slices(const int* L) {
  constexpr size_t kWBytes = (size_t)8 << 30;
  const size_t sites = (size_t)L[0] * L[1] * L[2], slice = sites * 4 * 9 * 16;
  const size_t k = kWBytes / slice;
  if (k >= (size_t)L[3]) return L[3];
  if (k >= 2) return (int)k;
  return 2 * slice <= kWBytes + 80 * sites * L[3] ? 2 : 0;
}

size_t ad_partial_doubles(const int* L) {
  // one pair per block, slabs of at least one slice each with one halo slice
  const long long V3 = (long long)L[0] * L[1] * L[2];
  const int w = ad_w_slices(L), n = slab_slices(w, L[3]);
  const int slabs = (L[3] + n - 1) / n;
  return 2 * (size_t)slabs * (size_t)((V3 * (w == 0 ? L[3] : w) + kT - 1) / kT);
}

// Runs `use(t0, n, part)` for each slab with its links in the W buffer.
template <class F>
static void for_slabs(AdArgs& a, cudaStream_t s, int* link_parts, F use) {
  const long long V3 = 2LL * a.lat.V3h;
  const int Lt = a.lat.L[3], n = slab_slices(a);
  int lp = 0;
  for (int t0 = 0; t0 < Lt; t0 += n) {
    const int m = t0 + n <= Lt ? n : Lt - t0;
    const int nt = m == Lt ? Lt : m + 1;
    a.w_t0 = nt == Lt ? 0 : (t0 + Lt - 1) % Lt;
    const unsigned nb = blocks(V3 * nt);
    if (a.w_slices) k_ad_links<true><<<nb, kT, 0, s>>>(a, nt, t0, m, lp);
    else k_ad_links<false><<<nb, kT, 0, s>>>(a, nt, t0, m, lp);
    lp += (int)nb;
    use(t0, m);
  }
  *link_parts = lp;
}

static void delta_pass(AdArgs& a, cudaStream_t s) {
  const long long V3 = 2LL * a.lat.V3h;
  const int Lt = a.lat.L[3], n = slab_slices(a);
  // blocks of all links and Delta launches, known before the first
  int n_lp = 0, n_dp = 0;
  for (int t0 = 0; t0 < Lt; t0 += n) {
    const int m = t0 + n <= Lt ? n : Lt - t0;
    n_lp += (int)blocks(V3 * (m == Lt ? Lt : m + 1));
    n_dp += (int)blocks(V3 * m);
  }
  int lp = 0, dp = 0;
  for_slabs(a, s, &lp, [&](int t0, int m) {
    const unsigned nb = blocks(V3 * m);
    if (a.w_slices) k_ad_delta<true><<<nb, kT, 0, s>>>(a, t0, m, dp, n_lp, n_dp);
    else k_ad_delta<false><<<nb, kT, 0, s>>>(a, t0, m, dp, n_lp, n_dp);
    dp += (int)nb;
  });
}

void launch_ad_forward(const AdArgs& args, cudaStream_t s) {
  AdArgs a = args;
  k_ad_exp<<<blocks(a.lat.V), kT, 0, s>>>(a);
  delta_pass(a, s);
}

void launch_ad_backward(const AdArgs& args, cudaStream_t s) {
  AdArgs a = args;
  k_ad_exp<<<blocks(a.lat.V), kT, 0, s>>>(a);
  delta_pass(a, s);
  const long long V3 = 2LL * a.lat.V3h;
  const int Lt = a.lat.L[3];
  if (a.w_slices == 0) {
    k_ad_backward<false><<<blocks(V3 * Lt), kT, 0, s>>>(a, 0, Lt);
    return;
  }
  if (slab_slices(a) >= Lt) {  // W of the whole lattice is still there
    k_ad_backward<true><<<blocks(V3 * Lt), kT, 0, s>>>(a, 0, Lt);
    return;
  }
  int lp = 0;
  for_slabs(a, s, &lp, [&](int t0, int m) { k_ad_backward<true><<<blocks(V3 * m), kT, 0, s>>>(a, t0, m); });
}

}  // namespace gf
