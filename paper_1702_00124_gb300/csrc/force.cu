// Force kernels.
//
// Fermion force (Section 2 of the paper: dS_F/dU = -phi^dag K^-1 (dK/dU) K^-1 phi).
// Convention: F_a(x,mu) = dS/dw for U_mu(x) -> exp(i w T_a) U_mu(x), stored as
// algebra coordinates [mu][parity][a][cb].  For full-lattice fields Y, X the
// per-link derivative of Re(Y^dag D X) is
//     Re(i tr(T_a W)) = -1/2 Im tr(lambda_a W),  W = U A1 - A2 U^dag,
//     A1 = sum_s [(1 - g_mu) X(x+mu)]_s Y_s(x)^dag,
//     A2 = sum_s [(1 + g_mu) X(x)]_s Y_s(x+mu)^dag,
// with the fermion sign on links across the time boundary.  Because the
// projector (1 + s g) has rank 2, sum_s [(1+s g)X]_s Y_s^dag equals
// sum_{a=0,1} h_a(X) h_a(Y)^dag with h the half spinor of the same projector,
// so each A is two 3x3 outer products.  The kernel adds coef times this to F.
//
// Gauge force: S_G = beta sum_{x, mu<nu} (1 - Re tr U_munu / 3) (the workload's
// Wilson plaquette action; the paper names S_G only), whose derivative is
// -(beta/3) Re(i tr(T_a U_mu(x) A_mu(x))) with A the sum of the six staples.
#include "dslash_impl.cuh"

namespace wd {

constexpr int F_THREADS = 128;

template <class T>
__device__ __forceinline__ void proj_ta(const cpx<T> (&W)[9], T (&f)[8]) {
  // f_a = -1/2 Im tr(lambda_a W); W[3*i+j] = W_ij
  const T h = (T)0.5;
  f[0] = -h * (W[3].i + W[1].i);
  f[1] = -h * (W[1].r - W[3].r);
  f[2] = -h * (W[0].i - W[4].i);
  f[3] = -h * (W[6].i + W[2].i);
  f[4] = -h * (W[2].r - W[6].r);
  f[5] = -h * (W[7].i + W[5].i);
  f[6] = -h * (W[5].r - W[7].r);
  f[7] = -h * (W[0].i + W[4].i - (T)2 * W[8].i) * (T)0.57735026918962576451;
}

// 3 x 3 products.  FP32: two chains of three per component, which keep the rounding of the
// separately rounded products before them (against FP64, 16^3 x 32: gauge force 7.17e-8, one
// chain of six 7.47e-8, two of three 7.19e-8; Hasenbusch force 1.026e-6, 1.088e-6, 1.035e-6).  FP64: one chain
// of six, the fewest operations on the pipe that bounds it.
template <class T>
__device__ __forceinline__ void mat_mul(const cpx<T> (&A)[9], const cpx<T> (&B)[9], cpx<T> (&C)[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if constexpr (sizeof(T) == 4) C[3 * i + j] = dot3(A[3 * i], B[j], A[3 * i + 1], B[3 + j], A[3 * i + 2], B[6 + j]);
      else C[3 * i + j] = cfma(A[3 * i + 2], B[6 + j], cfma(A[3 * i + 1], B[3 + j], cmul(A[3 * i], B[j])));
    }
}
// C = A B^dag
template <class T>
__device__ __forceinline__ void mat_mul_nd(const cpx<T> (&A)[9], const cpx<T> (&B)[9], cpx<T> (&C)[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if constexpr (sizeof(T) == 4)
        C[3 * i + j] = dot3_c(B[3 * j], A[3 * i], B[3 * j + 1], A[3 * i + 1], B[3 * j + 2], A[3 * i + 2]);
      else C[3 * i + j] = cfma_c(B[3 * j + 2], A[3 * i + 2], cfma_c(B[3 * j + 1], A[3 * i + 1], cmul_c(B[3 * j], A[3 * i])));
    }
}
// C = A^dag B
template <class T>
__device__ __forceinline__ void mat_mul_dn(const cpx<T> (&A)[9], const cpx<T> (&B)[9], cpx<T> (&C)[9]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if constexpr (sizeof(T) == 4) C[3 * i + j] = dot3_c(A[i], B[j], A[3 + i], B[3 + j], A[6 + i], B[6 + j]);
      else C[3 * i + j] = cfma_c(A[6 + i], B[6 + j], cfma_c(A[3 + i], B[3 + j], cmul_c(A[i], B[j])));
    }
}

// h_a(X) for the projector (1 + SG g_mu): 2 x 3 complex
template <int MU, int SG, class T>
__device__ __forceinline__ void half_of(const cpx<T> (&s)[12], cpx<T> (&h)[6]) {
  spin_project<MU, SG>(s, h);
}

// A += sum_a h_a k_a^dag
template <class T>
__device__ __forceinline__ void outer_acc(cpx<T> (&A)[9], const cpx<T> (&h)[6], const cpx<T> (&k)[6]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) A[3 * i + j] = cfma_c(k[3 + j], h[3 + i], cfma_c(k[j], h[i], A[3 * i + j]));
}

// A += sum_a h_a k_a^dag with the sum formed by itself, so that A1 and A2^dag round apart
template <class T>
__device__ __forceinline__ void outer_apart(cpx<T> (&A)[9], const cpx<T> (&h)[6], const cpx<T> (&k)[6]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) A[3 * i + j] = A[3 * i + j] + cfma_c(k[3 + j], h[3 + i], cmul_c(k[j], h[i]));
}

// F += coef sum_i dRe(Y_i^dag D X_i) over n groups of NP (Y, X) pairs.
//
// Re(i tr(T_a M)) is the same for -M and M^dag, so -A2 U^dag counts as U A2^dag: with
// A = A1 + A2^dag the link's derivative is that of W = U A, one matrix product
// for all pairs of a group.  A is summed over a group's pairs in the arithmetic of the fields,
// the groups' derivatives in FP64, and F is read and written once for all of
// them.  Summing a group's two pairs in FP32 does not round more than a product and a projection for
// each and an FP64 sum: polynomial force of degree 16, 16^3 x 32, against FP64 9.36e-7 and 9.42e-7
// (two pairs apart 9.82e-7 in the kernel before); degree 24, 8^3 x 16 5.05e-6, 5.07e-6, 5.14e-6.  A polynomial term has one group of two pairs per root; its segment of
// roots goes out in one launch.
//
// Block: 32 sites of one parity x 4 directions, one warp a direction, so that
// a site's own spinors are read once from L2 and three times from L1.  One FP32 pair
// on all but small lattices: k_force_site below.
//
// Measured at 16^3 x 32 (FP32): the kernel before it (one thread per site, two products
// per pair, F updated for every pair of pairs) 94 us per root, 16 roots 1.51 ms; the
// whole polynomial force of degree 16 3.02 -> 2.39 ms (2.02 ms today).
constexpr int F_MAXP = 2 * FORCE_ROOTS;   // pairs per launch
template <class S, class G>
struct ForceArgs {
  Geom g;
  S Ye[F_MAXP], Yo[F_MAXP], Xe[F_MAXP], Xo[F_MAXP];
  G gauge;
  double coef;
  int n;                     // groups
  double* F;                 // [4][2][8][Vh]
};

template <int MU, int NP, class T, class S, class G>
__device__ __forceinline__ void force_dir(const ForceArgs<S, G>& a, int par, long cb, const int (&c)[4], bool ok) {
  const Geom& g = a.g;
  const long nb = g.template nbr<2 * MU>((unsigned)cb, c);
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int i = 0; i < a.n; ++i) {
    cpx<T> A[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) A[j] = mk<T>(0, 0);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const int p = i * NP + q;
      cpx<T> s[12], h[6], k[6];
      (par ? a.Xe[p] : a.Xo[p]).loadT(nb, s);      // A1: (1 - g) X(x+mu) with (1 - g) Y(x)
      half_of<MU, -1>(s, h);
      (par ? a.Yo[p] : a.Ye[p]).loadT(cb, s);
      half_of<MU, -1>(s, k);
      outer_acc(A, h, k);
      (par ? a.Ye[p] : a.Yo[p]).loadT(nb, s);      // A2^dag: (1 + g) Y(x+mu) with (1 + g) X(x)
      half_of<MU, +1>(s, h);
      (par ? a.Xo[p] : a.Xe[p]).loadT(cb, s);
      half_of<MU, +1>(s, k);
      if constexpr (NP == 1 && sizeof(T) == 4) outer_apart(A, h, k);
      else outer_acc(A, h, k);
    }
    cpx<T> U[9], W[9];
    a.gauge.load(MU, par, cb, U);
    mat_mul(U, A, W);
    T f[8];
    proj_ta(W, f);
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] += to_f64(f[q]);
  }
  // links across the time boundary carry the fermion sign
  const double k = (MU == 3 && c[3] == g.L[3] - 1) ? -a.coef : a.coef;
  double* F = a.F + ((long)(MU * 2 + par) * 8) * g.Vh + cb;
  if (ok) {
#pragma unroll
    for (int q = 0; q < 8; ++q) F[q * g.Vh] = fma(k, acc[q], F[q * g.Vh]);
  }
}

// Two FP32 pairs: latency of the spinor reads, so five blocks per SM (96 registers, 14
// words spilled).  16 roots at 16^3 x 32, whole force: link kept over the groups, 138
// registers 2.10 ms; link read again per group (L1), 110 registers 2.05 ms; this 2.00 ms.
// One FP32 pair, on small lattices, takes 154 registers; FP64 is bound by its arithmetic.
template <class T, int NP> constexpr int force_blocks() { return sizeof(T) == 4 && NP == 2 ? 5 : 1; }
template <class T, int NP, class S, class G>
__global__ void __launch_bounds__(F_THREADS, force_blocks<T, NP>()) k_force(ForceArgs<S, G> a) {
  const int lane = threadIdx.x & 31, mu = threadIdx.x >> 5;
  const int par = blockIdx.y;
  const long site = (long)blockIdx.x * 32 + lane;
  const bool ok = site < a.g.Vh;
  const long cb = ok ? site : 0;               // a lane without a site repeats site 0 and stores nothing
  int c[4];
  a.g.coords(cb, par, c);
  switch (mu) {
    case 0: force_dir<0, NP, T>(a, par, cb, c, ok); break;
    case 1: force_dir<1, NP, T>(a, par, cb, c, ok); break;
    case 2: force_dir<2, NP, T>(a, par, cb, c, ok); break;
    default: force_dir<3, NP, T>(a, par, cb, c, ok); break;
  }
}

// One FP32 pair: one thread per site, the directions in turn.  Its own X and Y stay in
// registers (the warps per direction above read them four times) and 128 sites share
// their neighbours through L1; four blocks per SM (128 registers).  Derivative, sums and
// results are bit for bit those of k_force.  Latency of the spinor reads bounds it on small
// lattices, HBM on large ones: links, X, Y and F move 2.1 GB at 32^3 x 64, 0.31 ms.
// One call of the force from given X and Y (two conversions, two hops, this), k_force -> this:
// 12^3 x 24 33 -> 25 us, 16^3 x 32 94 -> 66, 24^4 243 -> 180, 24^3 x 48 467 -> 331, 32^3 x 64
// 1413 -> 958 (five blocks per SM 1003, no bound 1087).  From one block per SM on (156 blocks
// 24.0 -> 21.2 us); 8^3 x 16, 64 blocks, 17.1 -> 18.8.
template <int MU, class S, class G>
__device__ __forceinline__ void force_site_dir(const ForceArgs<S, G>& a, int par, long cb, const int (&c)[4],
                                               const cpx<float> (&Xs)[12], const cpx<float> (&Ys)[12]) {
  const Geom& g = a.g;
  const long nb = g.template nbr<2 * MU>((unsigned)cb, c);
  cpx<float> A[9], s[12], h[6], k[6];
#pragma unroll
  for (int j = 0; j < 9; ++j) A[j] = mk<float>(0, 0);
  (par ? a.Xe[0] : a.Xo[0]).loadT(nb, s);
  half_of<MU, -1>(s, h);
  half_of<MU, -1>(Ys, k);
  outer_acc(A, h, k);
  (par ? a.Ye[0] : a.Yo[0]).loadT(nb, s);
  half_of<MU, +1>(s, h);
  half_of<MU, +1>(Xs, k);
  outer_apart(A, h, k);
  cpx<float> U[9], W[9];
  a.gauge.load(MU, par, cb, U);
  mat_mul(U, A, W);
  float f[8];
  proj_ta(W, f);
  const double coef = (MU == 3 && c[3] == g.L[3] - 1) ? -a.coef : a.coef;
  double* F = a.F + ((long)(MU * 2 + par) * 8) * g.Vh + cb;
#pragma unroll
  for (int q = 0; q < 8; ++q) F[q * g.Vh] = fma(coef, to_f64(f[q]), F[q * g.Vh]);
}
template <class S, class G>
__global__ void __launch_bounds__(F_THREADS, 4) k_force_site(ForceArgs<S, G> a) {
  const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= 2 * a.g.Vh) return;
  const int par = (int)(tid / a.g.Vh);
  const long cb = tid - par * a.g.Vh;
  int c[4];
  a.g.coords(cb, par, c);
  cpx<float> Xs[12], Ys[12];
  (par ? a.Xo[0] : a.Xe[0]).loadT(cb, Xs);
  (par ? a.Yo[0] : a.Ye[0]).loadT(cb, Ys);
  force_site_dir<0>(a, par, cb, c, Xs, Ys);
  force_site_dir<1>(a, par, cb, c, Xs, Ys);
  force_site_dir<2>(a, par, cb, c, Xs, Ys);
  force_site_dir<3>(a, par, cb, c, Xs, Ys);
}

template <class T, int NP, class S, class G>
static void force_launch(wd_ctx* c, const G& gauge, double coef, int n, const Field* Ye, const Field* Yo,
                         const Field* Xe, const Field* Xo, double* F) {
  using P = decltype(S::p);
  const long Vh = c->g.Vh;
  for (int i0 = 0; i0 < n; i0 += F_MAXP / NP) {
    ForceArgs<S, G> a{};
    a.g = c->g;
    a.gauge = gauge;
    a.coef = coef;
    a.F = F;
    a.n = n - i0 < F_MAXP / NP ? n - i0 : F_MAXP / NP;
    for (int p = 0; p < a.n * NP; ++p) {
      const int s = i0 * NP + p;
      a.Ye[p] = S{(P)Ye[s].data, Vh};
      a.Yo[p] = S{(P)Yo[s].data, Vh};
      a.Xe[p] = S{(P)Xe[s].data, Vh};
      a.Xo[p] = S{(P)Xo[s].data, Vh};
    }
    c->launches += 1;
    if constexpr (NP == 1 && sizeof(T) == 4) {
      const int nb = nblocks(2 * Vh, F_THREADS);
      if (a.n == 1 && nb >= c->nsm) {          // a block for every SM
        k_force_site<<<nb, F_THREADS, 0, c->stream>>>(a);
        continue;
      }
    }
    k_force<T, NP><<<dim3(nblocks(Vh, 32), 2), F_THREADS, 0, c->stream>>>(a);
  }
}

static int force_groups(wd_ctx* c, double coef, int n, int np, const Field* Ye, const Field* Yo, const Field* Xe,
                        const Field* Xo, double* F) {
  const int f = Ye[0].fmt;
  for (int p = 0; p < n * np; ++p)
    if (Ye[p].fmt != f || Yo[p].fmt != f || Xe[p].fmt != f || Xo[p].fmt != f)
      return fail(WD_ERR_ARG, "force: formats differ");
  const long Vh = c->g.Vh;
  if (f == WD_F64) {
    const GF64 G{c->gauge64, Vh};
    if (np == 1) force_launch<double, 1, SpF64>(c, G, coef, n, Ye, Yo, Xe, Xo, F);
    else force_launch<double, 2, SpF64>(c, G, coef, n, Ye, Yo, Xe, Xo, F);
  } else if (f == WD_F32) {
    const GF32 G{c->gauge32, Vh};
    if (np == 1) force_launch<float, 1, SpF32>(c, G, coef, n, Ye, Yo, Xe, Xo, F);
    else force_launch<float, 2, SpF32>(c, G, coef, n, Ye, Yo, Xe, Xo, F);
  } else {
    return fail(WD_ERR_ARG, "force: fields must be FP64 or FP32");
  }
  WD_CUDA(cudaGetLastError());
  return WD_OK;
}

int force_outer(wd_ctx* c, double coef, const Field& Ye, const Field& Yo, const Field& Xe,
                const Field& Xo, double* F, int prec) {
  if (Ye.fmt == WD_F64 && prec != WD_F64) return fail(WD_ERR_ARG, "force: fields must be FP64 (prec FP64) or FP32");
  return force_groups(c, coef, 1, 1, &Ye, &Yo, &Xe, &Xo, F);
}

// n groups of two pairs: entries 2 i and 2 i + 1 of the arrays
int force_pairs(wd_ctx* c, double coef, int n, const Field* Ye, const Field* Yo, const Field* Xe, const Field* Xo,
                double* F) {
  return force_groups(c, coef, n, 2, Ye, Yo, Xe, Xo, F);
}

// ----------------------------------------------------------------------------
// gauge action and force
template <class T, class G>
__device__ __forceinline__ void link_at(const Geom& g, const G& gauge, int mu, const int (&c)[4], cpx<T> (&U)[9]) {
  const int par = (c[0] + c[1] + c[2] + c[3]) & 1;
  gauge.load(mu, par, g.cb_of(c[0], c[1], c[2], c[3]), U);
}

__device__ __forceinline__ void step(const Geom& g, int (&c)[4], int mu, int d) {
  int v = c[mu] + d;
  c[mu] = v < 0 ? v + g.L[mu] : (v >= g.L[mu] ? v - g.L[mu] : v);
}

// One thread per site, every direction in turn, FP32 at four blocks per SM (128 registers).
// Measured at 32^3 x 64 (FP32): 1.58 ms, 1.26 ms with the products as chains of six, 1.33 ms with two
// chains of three (1.55 ms without the register bound: 136, three blocks).  One warp per direction
// with the planes unrolled took 1.39 ms (links of 18 reals: three at a time fill the registers).
template <class T, class G>
__global__ void __launch_bounds__(F_THREADS, sizeof(T) == 4 ? 4 : 1) k_gauge_force(Geom g, G gauge, double coef, double* F) {
  const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= 2 * g.Vh) return;
  const int par = (int)(tid / g.Vh);
  const long cb = tid - par * g.Vh;
  int c[4];
  g.coords(cb, par, c);
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    cpx<T> A[9], t1[9], t2[9], t3[9], Ua[9], Ub[9], Uc[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) A[j] = mk<T>(0, 0);
#pragma unroll 1
    for (int nu = 0; nu < 4; ++nu) {
      if (nu == mu) continue;
      // upper staple U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
      int p[4] = {c[0], c[1], c[2], c[3]};
      step(g, p, mu, +1);
      link_at<T>(g, gauge, nu, p, Ua);
      int q[4] = {c[0], c[1], c[2], c[3]};
      step(g, q, nu, +1);
      link_at<T>(g, gauge, mu, q, Ub);
      link_at<T>(g, gauge, nu, c, Uc);
      mat_mul_nd(Ua, Ub, t1);
      mat_mul_nd(t1, Uc, t2);
#pragma unroll
      for (int j = 0; j < 9; ++j) A[j] = A[j] + t2[j];
      // lower staple U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
      int r[4] = {c[0], c[1], c[2], c[3]};
      step(g, r, nu, -1);
      int s[4] = {r[0], r[1], r[2], r[3]};
      step(g, s, mu, +1);
      link_at<T>(g, gauge, nu, s, Ua);
      link_at<T>(g, gauge, mu, r, Ub);
      link_at<T>(g, gauge, nu, r, Uc);
      mat_mul(Ub, Ua, t1);              // U_mu(x-nu) U_nu(x+mu-nu)
      mat_mul_dn(t1, Uc, t3);           // (U_mu U_nu')^dag U_nu(x-nu)
#pragma unroll
      for (int j = 0; j < 9; ++j) A[j] = A[j] + t3[j];
    }
    cpx<T> U[9], W[9];
    gauge.load(mu, par, cb, U);
    mat_mul(U, A, W);
    T f[8];
    proj_ta(W, f);
    double* Fp = F + ((long)(mu * 2 + par) * 8) * g.Vh + cb;
#pragma unroll
    for (int a = 0; a < 8; ++a) Fp[a * g.Vh] = fma(coef, (double)f[a], Fp[a * g.Vh]);
  }
}

int gauge_force_k(wd_ctx* c, double beta, int prec, double coef, double* F) {
  const int nb = nblocks(2 * c->g.Vh, F_THREADS);
  const double k = -coef * beta / 3.0;
  if (prec == WD_F64) k_gauge_force<double><<<nb, F_THREADS, 0, c->stream>>>(c->g, GF64{c->gauge64, c->g.Vh}, k, F);
  else k_gauge_force<float><<<nb, F_THREADS, 0, c->stream>>>(c->g, GF32{c->gauge32, c->g.Vh}, k, F);
  WD_CHECK_LAUNCH();
  return WD_OK;
}

template <class G>
__global__ void __launch_bounds__(F_THREADS) k_gauge_action(Geom g, G gauge, Reduce red) {
  const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  double v[1] = {0.0};
  if (tid < 2 * g.Vh) {
    const int par = (int)(tid / g.Vh);
    const long cb = tid - par * g.Vh;
    int c[4];
    g.coords(cb, par, c);
    for (int mu = 0; mu < 4; ++mu) {
      for (int nu = mu + 1; nu < 4; ++nu) {
        cpx<double> Um[9], Un[9], Umn[9], Unm[9], t1[9], t2[9];
        link_at<double>(g, gauge, mu, c, Um);
        int p[4] = {c[0], c[1], c[2], c[3]};
        step(g, p, mu, +1);
        link_at<double>(g, gauge, nu, p, Un);      // U_nu(x+mu)
        int q[4] = {c[0], c[1], c[2], c[3]};
        step(g, q, nu, +1);
        link_at<double>(g, gauge, mu, q, Umn);     // U_mu(x+nu)
        link_at<double>(g, gauge, nu, c, Unm);     // U_nu(x)
        mat_mul(Um, Un, t1);
        mat_mul_nd(t1, Umn, t2);
        // Re tr(t2 Unm^dag)
        double tr = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = 0; j < 3; ++j) tr += t2[3 * i + j].r * Unm[3 * i + j].r + t2[3 * i + j].i * Unm[3 * i + j].i;
        v[0] += 1.0 - tr / 3.0;
      }
    }
  }
  double tot[1];
  grid_sum<1>(red, v, tot);
}

int gauge_action_k(wd_ctx* c, double* S) {
  const int nb = nblocks(2 * c->g.Vh, F_THREADS);
  if (nb > RED_MAX_BLOCKS) return fail(WD_ERR_ARG, "gauge action: lattice too large");
  k_gauge_action<<<nb, F_THREADS, 0, c->stream>>>(c->g, GF64{c->gauge64, c->g.Vh}, reducer_host(c));
  WD_CHECK_LAUNCH();
  return fetch_host(c, 1, S);
}

}  // namespace wd
