// HMC step kernels (Section 2 of the paper):
//   T[eps]: U -> exp(i eps P) U,   S[eps]: P -> P - eps F,   H = sum tr P^2 + S,
// and the Gaussian draws of momenta (P ~ exp(-sum tr P^2)) and of the heat
// bath noise chi (exp(-chi^dag chi)).
//
// exp(iQ) for Hermitian traceless Q = eps P follows the Cayley-Hamilton
// closed form of Morningstar and Peardon (Phys. Rev. D 69 (2004) 054501,
// Section III): exp(iQ) = f0 + f1 Q + f2 Q^2 with the f_j from
// c0 = det Q, c1 = tr Q^2 / 2; negative c0 is mapped to positive c0 by the
// symmetry f_j(-c0) = (-1)^j conj(f_j(c0)), which keeps the denominator
// 9u^2 - w^2 away from zero.  The product is reunitarised (Gram-Schmidt on
// rows 0 and 1, row 2 = (r0 x r1)^*) and written to the FP64 links and to
// both FP32 link copies in the same pass.  Row 2 of the reunitarised product
// comes from the other two, so row 2 of exp(iQ) and of the product is never formed.
// Bound by the FP64 pipe: 472 bytes a link would take 0.58 ms at 32^3 x 64, about 400
// FP64 instructions a link (33 ns each on 608 schedulers, 32 links) 5.3 ms.
// Measured 7.55 ms with whole matrices, divisions and square roots; 5.62 ms with two
// rows and Newton steps from FP32 seeds; 5.36 ms with the FP32 copies rounded by
// integer operations; 5.44 ms with the square root and the quotient of the
// exponential corrected by their residuals.
//
// Random numbers: Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11) with key
// (seed, 0) and counter (j, stream, 0, 0); the four words of block j give
// u_k = ((x_k >> 11) + 1/2) 2^-53 and two Box-Muller pairs, which are the
// Gaussian reals 4j..4j+3 of the field in its lexicographic real order.
#include <cmath>

#include "dslash_impl.cuh"

namespace wd {

constexpr int H_THREADS = 128;

// cos x and sin(x)/x from y = -x^2 by their Taylor series through x^14; for
// |x| <= 0.5 the first omitted terms are below 1e-18.
__device__ __forceinline__ double cos_series(double y) {
  double t = 1.0 / 87178291200.0;              // 1/14!
  t = fma(t, y, 1.0 / 479001600.0);            // 1/12!
  t = fma(t, y, 1.0 / 3628800.0);
  t = fma(t, y, 1.0 / 40320.0);
  t = fma(t, y, 1.0 / 720.0);
  t = fma(t, y, 1.0 / 24.0);
  t = fma(t, y, 0.5);
  return fma(t, y, 1.0);
}
__device__ __forceinline__ double sinc_series(double y) {
  double t = 1.0 / 1307674368000.0;            // 1/15!
  t = fma(t, y, 1.0 / 6227020800.0);           // 1/13!
  t = fma(t, y, 1.0 / 39916800.0);
  t = fma(t, y, 1.0 / 362880.0);
  t = fma(t, y, 1.0 / 5040.0);
  t = fma(t, y, 1.0 / 120.0);
  t = fma(t, y, 1.0 / 6.0);
  return fma(t, y, 1.0);
}

// 1/sqrt(x) and 1/x for x > 0 within FP32's range: an FP32 seed (relative error
// about 1e-7) and two Newton steps, each squaring the error.  The last step adds a
// correction to the iterate, so that the result carries its own rounding and little of the step's.
// GB300 runs FP64 at 1/64 of the FP32 rate; the division and square root of the
// language cost several times as many FP64 instructions.
__device__ __forceinline__ bool beyond_seed(double x) { return __double2hiint(x) >= 0x46000000; }   // x > 1e29, inf, NaN
__device__ __forceinline__ double rsqrt_newton(double x) {
  if (beyond_seed(x)) return 1.0 / sqrt(x);
  double y = (double)rsqrtf((float)x);
  const double hx = 0.5 * x;
#pragma unroll
  for (int it = 0; it < 2; ++it) y = fma(y, fma(-hx * y, y, 0.5), y);
  return y;
}
__device__ __forceinline__ double rcp_newton(double x) {
  if (beyond_seed(x)) return 1.0 / x;
  double y = (double)(1.0f / (float)x);
#pragma unroll
  for (int it = 0; it < 2; ++it) y = fma(y, fma(-x, y, 1.0), y);
  return y;
}

// Rows 0 and 1 of exp(iQ), Q Hermitian and traceless with diagonal q00, q11, q22
// and upper triangle q01, q02, q12.  Row 2 follows from them (SU(3)).
__device__ __forceinline__ void cayley_hamilton_rows(double q00, double q11, double q22, cpx<double> q01,
                                                     cpx<double> q02, cpx<double> q12, cpx<double> (&E)[6]) {
  const double n01 = fma(q01.r, q01.r, q01.i * q01.i), n02 = fma(q02.r, q02.r, q02.i * q02.i),
               n12 = fma(q12.r, q12.r, q12.i * q12.i);
  // Q^2, with q00 + q11 = -q22 and its permutations
  const cpx<double> m = cmul(q01, q12);
  const double s00 = fma(q00, q00, n01 + n02), s11 = fma(q11, q11, n01 + n12);
  const double c1 = 0.5 * (s00 + s11 + fma(q22, q22, n02 + n12));
  cpx<double> s01 = cfma_c(q12, q02, mk(-q22 * q01.r, -q22 * q01.i));
  cpx<double> s02 = mk(fma(-q11, q02.r, m.r), fma(-q11, q02.i, m.i));
  cpx<double> s12 = cfma_c(q01, q02, mk(-q00 * q12.r, -q00 * q12.i));
  // c0 = det Q = q00 q11 q22 + 2 Re(q01 q12 q02^*) - q00 |q12|^2 - q11 |q02|^2 - q22 |q01|^2
  double c0 = 2.0 * fma(m.r, q02.r, m.i * q02.i);
  c0 = fma(q22, fma(q00, q11, -n01), fma(-q11, n02, fma(-q00, n12, c0)));
  cpx<double> f0, f1, f2;
  if (c1 < 1e-24) {
    f0 = mk(1.0, 0.0);
    f1 = mk(0.0, 1.0);
    f2 = mk(-0.5, 0.0);
  } else {
    const bool neg = c0 < 0;
    const double t3 = c1 * (1.0 / 3.0);
    const double y = rsqrt_newton(t3);             // 1 / sqrt(c1 / 3)
    double st3 = t3 * y;                           // sqrt(c1 / 3), corrected by its residual
    st3 = fma(fma(-st3, st3, t3), 0.5 * y, st3);
    // r = |c0| / (2 (c1/3)^{3/2}), the quotient corrected the same way.  Links after a step of
    // eps against 128-bit arithmetic, rms, with square root and divisions / uncorrected / this:
    // eps 0.1 9.3e-17 / 7.3e-17 / 7.3e-17, 2 2.38e-16 / 2.89e-16 / 2.31e-16, 3 3.44e-16 / 4.20e-16 / 3.44e-16
    const double y3 = y * y * y, q0 = 0.5 * fabs(c0);
    double r = q0 * y3;
    r = fma(fma(-t3 * st3, r, q0), y3, r);
    r = r > 1.0 ? 1.0 : r;
    // cs = cos(th/3), th = acos(r) in [0, pi/2]: the root of 4 cs^3 - 3 cs = r
    // in [cos(pi/6), 1], where the derivative 12 cs^2 - 3 lies in [6, 9]; an
    // FP32 seed and two Newton steps whose FP64 residual is scaled by the FP32
    // derivative: the error shrinks by 1e-7 a step
    const float csf = cosf(acosf((float)r) * (1.0f / 3.0f));
    const double inv = (double)(1.0f / (12.0f * csf * csf - 3.0f));
    double cs = (double)csf;
#pragma unroll
    for (int it = 0; it < 2; ++it) cs = fma(-inv, fma(cs, fma(4.0 * cs, cs, -3.0), -r), cs);
    const double u = st3 * cs;
    const double u2 = u * u;
    const double w2 = c1 * (1.0 - cs) * (1.0 + cs);  // w = sqrt(c1) sin(th/3)
    double cw, xi0, cu, su;
    if (w2 <= 0.25) {
      cw = cos_series(-w2);
      xi0 = sinc_series(-w2);
    } else {
      const double w = sqrt(w2);
      double sw;
      sincos(w, &sw, &cw);
      xi0 = sw / w;
    }
    if (u2 <= 0.25) {
      cu = cos_series(-u2);
      su = u * sinc_series(-u2);
    } else {
      sincos(u, &su, &cu);
    }
    const cpx<double> e2 = mk(fma(cu, cu, -su * su), 2.0 * su * cu);   // exp(2iu)
    const cpx<double> em = mk(cu, -su);                                  // exp(-iu)
    const double den = rcp_newton(fma(9.0, u2, -w2));
    const double tu = 2.0 * u;
    const cpx<double> k0 = mk(8.0 * u2 * cw, tu * fma(3.0, u2, w2) * xi0);
    const cpx<double> k1 = mk(-tu * cw, fma(3.0, u2, -w2) * xi0);
    const cpx<double> k2 = mk(-cw, -3.0 * u * xi0);
    const double d0 = u2 - w2;
    f0 = cfma(em, k0, mk(d0 * e2.r, d0 * e2.i));
    f1 = cfma(em, k1, mk(tu * e2.r, tu * e2.i));
    f2 = cfma(em, k2, e2);
    f0 = mk(den * f0.r, den * f0.i);
    f1 = mk(den * f1.r, den * f1.i);
    f2 = mk(den * f2.r, den * f2.i);
    if (neg) {
      f0 = conj(f0);
      f1 = mk(-f1.r, f1.i);
      f2 = conj(f2);
    }
  }
  E[0] = mk(fma(f2.r, s00, fma(f1.r, q00, f0.r)), fma(f2.i, s00, fma(f1.i, q00, f0.i)));
  E[1] = cfma(f2, s01, cmul(f1, q01));
  E[2] = cfma(f2, s02, cmul(f1, q02));
  E[3] = cfma(f2, conj(s01), cmul(f1, conj(q01)));
  E[4] = mk(fma(f2.r, s11, fma(f1.r, q11, f0.r)), fma(f2.i, s11, fma(f1.i, q11, f0.i)));
  E[5] = cfma(f2, s12, cmul(f1, q12));
}

// 1/sqrt(n) of a squared row norm.  The rows come from a product of unitary
// matrices, so n = 1 + d with d a few 1e-16: 1 - d/2 + 3 d^2/8 - 5 d^3/16 (next
// term below 3e-21 for |d| < 1e-5) replaces the square root; links loaded less
// accurately than that take it.
__device__ __forceinline__ double inv_norm(double n) {
  const double d = n - 1.0;
  if (fabs(d) < 1e-5) return fma(d, fma(d, fma(d, -0.3125, 0.375), -0.5), 1.0);
  return 1.0 / sqrt(n);
}

// Gram-Schmidt on rows 0 and 1, row 2 = (r0 x r1)^*
__device__ __forceinline__ void reunitarize(cpx<double> (&U)[9]) {
  double n0 = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) n0 = fma(U[j].r, U[j].r, fma(U[j].i, U[j].i, n0));
  n0 = inv_norm(n0);
#pragma unroll
  for (int j = 0; j < 3; ++j) U[j] = mk(n0 * U[j].r, n0 * U[j].i);
  const cpx<double> d = cfma_c(U[2], U[5], cfma_c(U[1], U[4], cmul_c(U[0], U[3])));
  const cpx<double> md = mk(-d.r, -d.i);
#pragma unroll
  for (int j = 0; j < 3; ++j) U[3 + j] = cfma(md, U[j], U[3 + j]);
  double n1 = 0;
#pragma unroll
  for (int j = 3; j < 6; ++j) n1 = fma(U[j].r, U[j].r, fma(U[j].i, U[j].i, n1));
  n1 = inv_norm(n1);
#pragma unroll
  for (int j = 3; j < 6; ++j) U[j] = mk(n1 * U[j].r, n1 * U[j].i);
  third_row(U);
}

__global__ void __launch_bounds__(H_THREADS) k_step_T(Geom g, const double* P, double eps, double2* U64,
                                                      float2* U32, float4* U12, float4* Udd) {
  const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= 8 * g.Vh) return;
  const int mp = (int)(tid / g.Vh);   // mu * 2 + parity
  const long cb = tid - mp * g.Vh;
  double p[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) p[a] = P[((long)mp * 8 + a) * g.Vh + cb];
  double2* u = U64 + (long)mp * 9 * g.Vh + cb;
  cpx<double> E[6], U[9], V[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) { double2 v = u[j * g.Vh]; U[j] = mk(v.x, v.y); }
  // Q = eps sum_a p_a lambda_a / 2
  const double h = 0.5 * eps, d3 = h * p[2], d8 = (h * 0.57735026918962576451) * p[7];
  cayley_hamilton_rows(d8 + d3, d8 - d3, -2.0 * d8, mk(h * p[0], -h * p[1]), mk(h * p[3], -h * p[4]),
                       mk(h * p[5], -h * p[6]), E);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) V[3 * i + j] = cfma(E[3 * i + 2], U[6 + j], cfma(E[3 * i + 1], U[3 + j], cmul(E[3 * i], U[j])));
  reunitarize(V);
#pragma unroll
  for (int j = 0; j < 9; ++j) u[j * g.Vh] = make_double2(V[j].r, V[j].i);
  float2* v32 = U32 + (long)mp * 9 * g.Vh + cb;
  float2 f[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) v32[j * g.Vh] = f[j] = make_float2(f32_of(V[j].r), f32_of(V[j].i));
  float4* v12 = U12 + (long)mp * 3 * g.Vh + cb;
#pragma unroll
  for (int j = 0; j < 3; ++j) v12[j * g.Vh] = make_float4(f[2 * j].x, f[2 * j].y, f[2 * j + 1].x, f[2 * j + 1].y);
  if (Udd != nullptr) {
    float4* vd = Udd + (long)mp * 9 * g.Vh + cb;
#pragma unroll
    for (int j = 0; j < 9; ++j)
      vd[j * g.Vh] = make_float4(f[j].x, f32_of(V[j].r - f64_of(f[j].x)), f[j].y, f32_of(V[j].i - f64_of(f[j].y)));
  }
}

int step_T_k(wd_ctx* c, const double* P, double eps) {
  const long n = 8 * c->g.Vh;
  links_written(c);
  k_step_T<<<nblocks(n, H_THREADS), H_THREADS, 0, c->stream>>>(c->g, P, eps, c->gauge64, c->gauge32,
                                                                c->gauge32r12, c->gauge_dd);
  WD_CHECK_LAUNCH();
  return WD_OK;
}

__global__ void k_axpy_alg(long n, double a, const double* x, double* y) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] += a * x[i];
}

int step_S_k(wd_ctx* c, double* P, const double* F, double eps) {
  const long n = 64 * c->g.Vh;   // 4 mu x 2 parities x 8 coordinates
  k_axpy_alg<<<nblocks(n, 256), 256, 0, c->stream>>>(n, -eps, F, P);
  WD_CHECK_LAUNCH();
  return WD_OK;
}

__global__ void __launch_bounds__(256) k_sumsq(long n, const double* x, Reduce red) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  double v[1] = {0.0};
  // 8 consecutive values per thread keeps the block count small
  for (int q = 0; q < 8; ++q) {
    const long k = i * 8 + q;
    if (k < n) v[0] += x[k] * x[k];
  }
  double tot[1];
  grid_sum<1>(red, v, tot);
}

int kinetic_k(wd_ctx* c, const double* P, double* out) {
  const long n = 64 * c->g.Vh;
  const int nb = nblocks((n + 7) / 8, 256);
  if (nb > RED_MAX_BLOCKS) return fail(WD_ERR_ARG, "kinetic: lattice too large");
  k_sumsq<<<nb, 256, 0, c->stream>>>(n, P, reducer_host(c));
  WD_CHECK_LAUNCH();
  double s;
  WD_TRY(fetch_host(c, 1, &s));
  *out = 0.5 * s;
  return WD_OK;
}

// ----------------------------------------------------------------------------
// Philox4x64-10
__device__ __forceinline__ void philox4x64(uint64_t (&x)[4], uint64_t k0, uint64_t k1) {
  const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
  const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) { k0 += W0; k1 += W1; }
    const uint64_t hi0 = __umul64hi(M0, x[0]), lo0 = M0 * x[0];
    const uint64_t hi1 = __umul64hi(M1, x[2]), lo1 = M1 * x[2];
    const uint64_t n0 = hi1 ^ x[1] ^ k0, n2 = hi0 ^ x[3] ^ k1;
    x[0] = n0; x[1] = lo1; x[2] = n2; x[3] = lo0;
  }
}

__device__ __forceinline__ void gauss4(uint64_t j, uint64_t seed, uint64_t stream, double (&g)[4]) {
  uint64_t x[4] = {j, stream, 0ull, 0ull};
  philox4x64(x, seed, 0ull);
  double u[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) u[k] = ((double)(x[k] >> 11) + 0.5) * 0x1.0p-53;
  const double r0 = sqrt(-2.0 * log(u[0])), r2 = sqrt(-2.0 * log(u[2]));
  const double two_pi = 6.283185307179586232;
  g[0] = r0 * cos(two_pi * u[1]);
  g[1] = r0 * sin(two_pi * u[1]);
  g[2] = r2 * cos(two_pi * u[3]);
  g[3] = r2 * sin(two_pi * u[3]);
}

// spinor: lexicographic reals e = (lex * 12 + comp) * 2 + re/im; a block holds
// reals 4j..4j+3 = complex components 2q, 2q+1 of one site (q = j mod 6)
__global__ void k_draw_spinor(Geom g, int parity, uint64_t seed, uint64_t stream, double2* out) {
  const long j = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= 6 * g.V) return;
  const long lex = j / 6;
  const int q = (int)(j % 6);
  const int x = (int)(lex % g.L[0]);
  long r = lex / g.L[0];
  const int y = (int)(r % g.L[1]); r /= g.L[1];
  const int z = (int)(r % g.L[2]);
  const int t = (int)(r / g.L[2]);
  if (((x + y + z + t) & 1) != parity) return;
  double v[4];
  gauss4((uint64_t)j, seed, stream, v);
  const long cb = lex >> 1;
  out[(2 * q) * g.Vh + cb] = make_double2(v[0], v[1]);
  out[(2 * q + 1) * g.Vh + cb] = make_double2(v[2], v[3]);
}

// algebra: lexicographic reals e = (lex * 4 + mu) * 8 + a; block j covers
// coordinates 4h..4h+3 (h = j mod 2) of link (lex, mu)
__global__ void k_draw_alg(Geom g, uint64_t seed, uint64_t stream, double* out) {
  const long j = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= 8 * g.V) return;
  const int h = (int)(j & 1);
  const long lm = j >> 1;
  const int mu = (int)(lm & 3);
  const long lex = lm >> 2;
  const int x = (int)(lex % g.L[0]);
  long r = lex / g.L[0];
  const int y = (int)(r % g.L[1]); r /= g.L[1];
  const int z = (int)(r % g.L[2]);
  const int t = (int)(r / g.L[2]);
  const int par = (x + y + z + t) & 1;
  const long cb = lex >> 1;
  double v[4];
  gauss4((uint64_t)j, seed, stream, v);
#pragma unroll
  for (int k = 0; k < 4; ++k) out[((long)(mu * 2 + par) * 8 + 4 * h + k) * g.Vh + cb] = v[k];
}

int gaussian_draw_k(wd_ctx* c, int what, int parity, uint64_t seed, uint64_t stream, double* out) {
  if (what == 0) {
    const long n = 6 * c->g.V;
    k_draw_spinor<<<nblocks(n, 256), 256, 0, c->stream>>>(c->g, parity, seed, stream, (double2*)out);
  } else {
    const long n = 8 * c->g.V;
    k_draw_alg<<<nblocks(n, 256), 256, 0, c->stream>>>(c->g, seed, stream, out);
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

}  // namespace wd
