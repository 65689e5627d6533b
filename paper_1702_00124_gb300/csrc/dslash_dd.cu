// Double-float instantiation of the hopping stencil: spinors and links in
// double-float storage (16 bytes per complex, like FP64), arithmetic by
// error-free transformations on the FP32 pipes (about 44-48 significant bits).
//
// Arithmetic: the SU(3) x half-spinor products use the compensated dot
// product of Ogita, Rump and Oishi (2005, "Dot2") instead of one normalised
// double-float operation per step: each real component of U h is a sum of
// six products, each product is split exactly by an FMA (two-product, with
// the cross terms of the low words), the high words are summed exactly
// (two-sum) and every rounding error is added into one FP32 word.  The site's
// sum over directions keeps that unnormalised form, folded once half way and
// normalised before the store.
//
// Eight threads per site, one per neighbour direction, as dslash_split.cuh: a block
// is 32 sites, warp w forms U h (U^dag h) of direction w, the products meet in
// shared memory and the block's warps share the components of the sum.  The
// product is one piece of code for every direction (rows or conjugated columns by
// stride and sign), the projection one per mu, so the kernel stays inside the
// instruction cache; all eight directions unrolled in one thread did not (1.24 ms per hop at
// 32^3 x 64), which had split the hop into two launches with a partial sum in
// between.  FP32 issue bounds it (72 % of the slots taken, 54 to 58 % of them by the FMA pipe) with
// memory 44 % busy: about 9,000 FP32 instructions a site would take 230 us per hop at 32^3 x 64 and its
// 1.6 GB 240 us, the hop takes about 430 us.
// K_hat in a chain (conversions included), two launches -> this: 32^3 x 64 2349 -> 1992 us,
// 24^4 501 -> 338, 16^3 x 32 201 -> 143, 8^3 x 16 113 -> 30, 4^4 115 -> 19; without the
// links' way through shared memory 2126, 365, 157, 29, 27.  Error against FP64
// 3.26e-15 at every size, as before (3.52e-15 without the fold half way).
#include "dslash_staged.cuh"

namespace wd {

// value s + c with c the collected rounding errors (not normalised)
struct lz {
  float s, c;
};
struct lzc {
  lz r, i;
};

// a += p + e for FP32 p and e: two-sum of the high words, e and the sum's
// error go to the low word
__device__ __forceinline__ void lz_add(lz& a, float p, float e) {
  const float t = a.s + p;
  const float z = t - a.s;
  a.c += ((a.s - (t - z)) + (p - z)) + e;
  a.s = t;
}
// exact product split of x y: p + e, e including the low-word cross terms
__device__ __forceinline__ void two_prod(dd x, dd y, float& p, float& e) {
  p = x.hi * y.hi;
  e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
}
__device__ __forceinline__ void lz_fma(lz& a, dd x, dd y) {
  float p, e;
  two_prod(x, y, p, e);
  lz_add(a, p, e);
}
__device__ __forceinline__ lz lz_first(dd x, dd y) {
  lz a;
  two_prod(x, y, a.s, a.c);
  return a;
}
__device__ __forceinline__ dd neg(dd x) { return dd(-x.hi, -x.lo); }
__device__ __forceinline__ dd lz_norm(const lz& a) { return dd_2sum(a.s, a.c); }
__device__ __forceinline__ lz lz_fold(const lz& a) {
  const dd n = lz_norm(a);
  return {n.hi, n.lo};
}

// a += i^K u
template <int K>
__device__ __forceinline__ void lz_add_ipow(lzc& a, const lzc& u) {
  constexpr int k = ((K % 4) + 4) % 4;
  if constexpr (k == 0) {
    lz_add(a.r, u.r.s, u.r.c);
    lz_add(a.i, u.i.s, u.i.c);
  } else if constexpr (k == 1) {
    lz_add(a.r, -u.i.s, -u.i.c);
    lz_add(a.i, u.r.s, u.r.c);
  } else if constexpr (k == 2) {
    lz_add(a.r, -u.r.s, -u.r.c);
    lz_add(a.i, -u.i.s, -u.i.c);
  } else {
    lz_add(a.r, u.i.s, u.i.c);
    lz_add(a.i, -u.r.s, -u.r.c);
  }
}

// sum_k u_k h_k of one colour vector h: re = ur vr - ui vi, im = ur vi + ui vr
__device__ __forceinline__ lzc row_lz(const cpx<dd> (&u)[3], const cpx<dd>* h) {
  lz re, im;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const cpx<dd> v = h[k];
    if (k == 0) {
      re = lz_first(u[k].r, v.r);
      im = lz_first(u[k].r, v.i);
    } else {
      lz_fma(re, u[k].r, v.r);
      lz_fma(im, u[k].r, v.i);
    }
    lz_fma(re, neg(u[k].i), v.i);
    lz_fma(im, u[k].i, v.r);
  }
  return {re, im};
}

__device__ __forceinline__ dd flip(dd x, unsigned m) {   // m = 0 or the sign bit
  return dd(__uint_as_float(__float_as_uint(x.hi) ^ m), __uint_as_float(__float_as_uint(x.lo) ^ m));
}

// h = psi_a + sg i^k psi_PERM(a) of the neighbour spinor, sg = +1 (m = 0) or -1 (m = the sign bit)
template <int MU>
__device__ __forceinline__ void project_dd(const SpDD& in, long i, unsigned m, cpx<dd> (&h)[6]) {
  using Gm = Gam<MU>;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int cc = c < 3 ? c : c - 3;
    const int q = 3 * (c < 3 ? Gm::p0 : Gm::p1) + cc;
    const float4 a = in.p[c * in.stride + i], b = in.p[q * in.stride + i];
    cpx<dd> v = {dd(b.x, b.y), dd(b.z, b.w)};
    v = c < 3 ? ipow<Gm::k0>(v) : ipow<Gm::k1>(v);
    h[c] = {dd(a.x, a.y) + flip(v.r, m), dd(a.z, a.w) + flip(v.i, m)};
  }
}

// component of sum_D (1 + SG g_mu) (x) u_D: of the upper spins (LOW = 0, j = 3 spin + colour)
// or of spin LOW = 2, 3 (j = colour); u = shared [8][6][32] + lane
template <int LOW, int D, bool DAG>
__device__ __forceinline__ void sum_term(const float4* u, int j, lzc& acc) {
  constexpr int MU = D >> 1;
  constexpr int SG = ((D & 1) == 0) == DAG ? +1 : -1;
  using Gm = Gam<MU>;
  constexpr bool first = LOW == Gm::p0;
  constexpr int q = LOW == 0 ? 0 : (SG > 0 ? 0 : 2) - (first ? Gm::k0 : Gm::k1);
  const int k = LOW == 0 ? j : (first ? j : 3 + j);
  const float4 v = u[(D * 6 + k) * 32];
  lz_add_ipow<q>(acc, lzc{{v.x, v.y}, {v.z, v.w}});
}
template <int LOW, bool DAG> __device__ __forceinline__ lzc sum_dirs(const float4* u, int j) {
  lzc acc = {{0.f, 0.f}, {0.f, 0.f}};
  sum_term<LOW, 0, DAG>(u, j, acc);
  sum_term<LOW, 1, DAG>(u, j, acc);
  sum_term<LOW, 2, DAG>(u, j, acc);
  sum_term<LOW, 3, DAG>(u, j, acc);
  // half way the error word is folded in: the later errors add to a smaller word
  acc = {lz_fold(acc.r), lz_fold(acc.i)};
  sum_term<LOW, 4, DAG>(u, j, acc);
  sum_term<LOW, 5, DAG>(u, j, acc);
  sum_term<LOW, 6, DAG>(u, j, acc);
  sum_term<LOW, 7, DAG>(u, j, acc);
  return acc;
}

template <bool DAG, bool XPAY>
__global__ void __launch_bounds__(256, 3) k_hop_dd(HopArgs<SpDD, SpDD, SpDD, GDD> a) {
  extern __shared__ float4 sh[];              // [8][6][32] products, [9][256] links
  pdl_trigger();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long site = (long)blockIdx.x * 32 + lane;
  const bool ok = site < a.g.Vh;
  const unsigned cb = ok ? (unsigned)site : 0u;   // a lane without a site repeats site 0 and stores nothing
  int c[4];
  a.g.coords(cb, a.out_par, c);
  const bool fwd = (w & 1) == 0;
  const int mu = w >> 1;
  unsigned nb;
  switch (w) {
    case 0: nb = a.g.nbr<0>(cb, c); break;
    case 1: nb = a.g.nbr<1>(cb, c); break;
    case 2: nb = a.g.nbr<2>(cb, c); break;
    case 3: nb = a.g.nbr<3>(cb, c); break;
    case 4: nb = a.g.nbr<4>(cb, c); break;
    case 5: nb = a.g.nbr<5>(cb, c); break;
    case 6: nb = a.g.nbr<6>(cb, c); break;
    default: nb = a.g.nbr<7>(cb, c); break;
  }
  // the nine link entries come through shared memory (cp.async, each thread its own):
  // in flight from the start without holding registers, and before the wait, for
  // they do not depend on the kernels before.  Rows of U_mu(x), or columns of
  // U_mu(x - mu) for the conjugate
  const long gs = a.gauge.stride;
  const float4* q = a.gauge.p + (long)(mu * 2 + (fwd ? a.out_par : 1 - a.out_par)) * 9 * gs + (fwd ? cb : nb);
  const long row = fwd ? 3 * gs : gs, col = fwd ? gs : 3 * gs;
  float4* lk = sh + 8 * 6 * 32 + threadIdx.x;
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int l = 0; l < 3; ++l) cpa16(lk + (3 * k + l) * 256, q + k * row + l * col);
  cpa_commit();
  pdl_wait();
  const unsigned m = fwd == DAG ? 0u : 0x80000000u;   // projector 1 + SG g_mu
  cpx<dd> h[6];
  switch (mu) {
    case 0: project_dd<0>(a.in, nb, m, h); break;
    case 1: project_dd<1>(a.in, nb, m, h); break;
    case 2: project_dd<2>(a.in, nb, m, h); break;
    default: project_dd<3>(a.in, nb, m, h); break;
  }
  // the antiperiodic sign goes into the link
  const bool wrap = mu == 3 && (fwd ? c[3] == a.g.L[3] - 1 : c[3] == 0);
  const unsigned mr = wrap ? 0x80000000u : 0u, mi = mr ^ (fwd ? 0u : 0x80000000u);
  cpa_wait<0>();
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cpx<dd> u[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      const float4 v = lk[(3 * k + l) * 256];
      u[l] = {flip(dd(v.x, v.y), mr), flip(dd(v.z, v.w), mi)};
    }
    const lzc o0 = row_lz(u, h), o1 = row_lz(u, h + 3);
    sh[(w * 6 + k) * 32 + lane] = make_float4(o0.r.s, o0.r.c, o0.i.s, o0.i.c);
    sh[(w * 6 + 3 + k) * 32 + lane] = make_float4(o1.r.s, o1.r.c, o1.i.s, o1.i.c);
  }
  __syncthreads();
  // component w, for warps 0 to 3 also component 8 + w (three for every scheduler)
  const float4* us = sh + lane;
  const dd al(a.alpha);
  for (int j = w; j < 12; j += 8) {
    const lzc t = j < 6 ? sum_dirs<0, DAG>(us, j) : (j < 9 ? sum_dirs<2, DAG>(us, j - 6) : sum_dirs<3, DAG>(us, j - 9));
    cpx<dd> r = {lz_norm(t.r), lz_norm(t.i)};
    if constexpr (XPAY) {
      const float4 v = a.y.p[j * a.y.stride + cb];
      r = cpx<dd>{dd(v.x, v.y), dd(v.z, v.w)} + al * r;
    }
    if (ok) a.out.p[j * a.out.stride + cb] = make_float4(r.r.hi, r.r.lo, r.i.hi, r.i.lo);
  }
}

template <bool DAG, bool XPAY>
static int hop_dd_launch(wd_ctx* c, const HopArgs<SpDD, SpDD, SpDD, GDD>& a) {
  constexpr int sm = (8 * 6 * 32 + 9 * 256) * (int)sizeof(float4);   // 61 KB: three blocks per SM
  const int nb = nblocks(c->g.Vh, 32);
  WD_CUDA(cudaFuncSetAttribute(k_hop_dd<DAG, XPAY>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
  pdl_launch_if(c, early_gains_dd(nb, c->nsm), k_hop_dd<DAG, XPAY>, nb, 256, sm, a);
  WD_CHECK_LAUNCH();
  return WD_OK;
}

int hop_dd(wd_ctx* c, int out_par, bool dag, const Field& in, const Field& out, const Field* y,
           double alpha, bool norm_cg, bool in_cg) {
  if (in.fmt != WD_DD || out.fmt != WD_DD || (y && y->fmt != WD_DD))
    return fail(WD_ERR_ARG, "hop_dd: field formats must all be double-float");
  if (c->gauge_dd == nullptr) return fail(WD_ERR_STATE, "hop_dd: no double-float link copy");
  if (norm_cg || in_cg) return fail(WD_ERR_ARG, "hop_dd: not used inside queued CG iterations");
  if (out.data == in.data || (y && out.data == y->data))
    return fail(WD_ERR_ARG, "hop_dd: the output may not alias an input");
  SpDD I = spdd(in), O = spdd(out), Y = y ? spdd(*y) : O;
  HopArgs<SpDD, SpDD, SpDD, GDD> a{c->g, out_par, I, O, Y, GDD{c->gauge_dd, c->g.Vh}, alpha,
                                    Reduce{nullptr, nullptr, nullptr}, nullptr};
  if (!dag) return y ? hop_dd_launch<false, true>(c, a) : hop_dd_launch<false, false>(c, a);
  return y ? hop_dd_launch<true, true>(c, a) : hop_dd_launch<true, false>(c, a);
}

}  // namespace wd
