// Hopping stencil with eight threads per site, one per neighbour direction
// (Section 3.1 of the paper: Wilson fermions, even-odd preconditioning).
//
// A block works on 32 sites: warp w forms u = U h (or U^dag h) of direction w for
// all of them, the eight u's meet in shared memory, and the block's warps share
// the 12 components of the sum, the epilogue and the store.
//
// FP64, up to SPLIT_MAX_VH_F64 sites per parity: GB300 has half an FP64 lane per
// scheduler and clock, so a warp instruction holds its scheduler's pipe for 33 ns
// and the ~900 of a site take 30 us in one thread.  Spread over eight warps they
// fill all four schedulers of an SM from 32 sites on; small lattices use eight
// times the SMs and larger ones end with a shorter last wave.  Per hop, one
// thread per site against eight: 8^3 x 16 36 -> 15 us, 12^3 x 24 66 -> 43,
// 16^3 x 32 127 -> 111 (floor 93: 840 instructions x 33 ns on 608 schedulers),
// 24^3 x 48 540 -> 518; from 32^4 on both take the same (808 and 810 us).
//
// FP32 and 16-bit, up to SPLIT_MAX_VH and SPLIT_MAX_VH_16: there a hop takes as long as
// one thread's eight neighbour reads; here all eight are in flight at once.  K_hat in
// a chain, the staged pipeline against this: FP32 (last hop with the Chebyshev
// step) 4^4 12.5 -> 8.8 us, 8^3 x 16 14.4 -> 13.5, 12^4 16.8 -> 15.2, with
// 18-real links 25.1 -> 15.1, 12^3 x 24 17.6 and 27.0; BF16 4^4 18.0 -> 14.7, 8^3 x 16 22.0 -> 21.4,
// 8^2 x 12 x 16 22.5 and 27.3.
#pragma once
#include "dslash_staged.cuh"

namespace wd {

constexpr int SPL_SITES = 32;
constexpr int SPL_THREADS = 8 * SPL_SITES;

// u = (U or U^dag) (projected neighbour spinor) of direction D; waits for the
// preceding kernels between the link's loads and the spinor's; false if the solver
// has stopped
template <int D, bool DAG, class T, class A>
__device__ __forceinline__ bool split_dir(const A& a, unsigned cb, const int (&c)[4], cpx<T> (&u)[6]) {
  constexpr int MU = D >> 1;
  constexpr bool FWD = (D & 1) == 0;
  constexpr int SG = FWD == DAG ? +1 : -1;
  const unsigned nb = a.g.template nbr<D>(cb, c);
  cpx<T> s[12], h[6], U[9];
  if constexpr (FWD) a.gauge.load(MU, a.out_par, cb, U);
  else a.gauge.load(MU, 1 - a.out_par, nb, U);
  pdl_wait();
  if (a.st != nullptr && a.st->flag != 0) return false;
  a.in.template loadT<false>(nb, s);
  spin_project<MU, SG>(s, h);
  if (MU == 3 && (FWD ? c[3] == a.g.L[3] - 1 : c[3] == 0)) {
#pragma unroll
    for (int j = 0; j < 6; ++j) h[j] = mk<T>(-h[j].r, -h[j].i);
  }
  if constexpr (FWD) su3_mul(U, h, u);
  else su3_dag_mul(U, h, u);
  return true;
}

// component J = 3 spin + colour of sum_D (1 + SG g_mu) (x) u_D; u = shared [8][6][32] + lane
template <int J, int D, bool DAG, class T>
__device__ __forceinline__ cpx<T> split_term(const cpx<T>* u) {
  constexpr int MU = D >> 1;
  constexpr int SG = ((D & 1) == 0) == DAG ? +1 : -1;
  using Gm = Gam<MU>;
  constexpr int spin = J / 3, col = J % 3;
  if constexpr (spin < 2) return u[(D * 6 + J) * SPL_SITES];
  else {
    constexpr int q = (SG > 0 ? 0 : 2) - (spin == Gm::p0 ? Gm::k0 : Gm::k1);
    constexpr int k = spin == Gm::p0 ? col : 3 + col;
    return ipow<q>(u[(D * 6 + k) * SPL_SITES]);
  }
}
// a direction's two neighbours first: partial sums of two, four, six and eight terms round
// less than those of two to eight (K_hat FP32 against FP64 at 8^3 x 16: 5.59e-8 -> 5.41e-8)
template <int J, int MU, bool DAG, class T> __device__ __forceinline__ cpx<T> split_pair(const cpx<T>* u) {
  return split_term<J, 2 * MU, DAG>(u) + split_term<J, 2 * MU + 1, DAG>(u);
}
template <int J, bool DAG, class T> __device__ __forceinline__ cpx<T> split_sum(const cpx<T>* u) {
  cpx<T> v = split_pair<J, 0, DAG>(u);
  v = v + split_pair<J, 1, DAG>(u);
  v = v + split_pair<J, 2, DAG>(u);
  return v + split_pair<J, 3, DAG>(u);
}
// the same with J known at run time (uniform in a warp)
template <bool DAG, class T> __device__ __forceinline__ cpx<T> split_sum_at(int j, const cpx<T>* u) {
  switch (j) {
    case 0: return split_sum<0, DAG>(u);
    case 1: return split_sum<1, DAG>(u);
    case 2: return split_sum<2, DAG>(u);
    case 3: return split_sum<3, DAG>(u);
    case 4: return split_sum<4, DAG>(u);
    case 5: return split_sum<5, DAG>(u);
    case 6: return split_sum<6, DAG>(u);
    case 7: return split_sum<7, DAG>(u);
    case 8: return split_sum<8, DAG>(u);
    case 9: return split_sum<9, DAG>(u);
    case 10: return split_sum<10, DAG>(u);
    default: return split_sum<11, DAG>(u);
  }
}

// EPI 0: out = D in; 1: out = y + alpha D in; 2 and 3: HopPoly on that (FP32)
template <class T, bool DAG, int EPI, bool NORM, class In, class Out, class Y, class G>
__global__ void __launch_bounds__(SPL_THREADS) k_hop_split(HopArgs<In, Out, Y, G> a, HopPoly pe) {
  constexpr bool F64 = std::is_same<T, double>::value;
  constexpr bool OUT64 = std::is_same<Out, SpF64>::value;   // FP64 fields, or an FP32 result widened
  constexpr bool WORDS = F64 || ((OUT64 || std::is_same<Out, SpF32>::value) && std::is_same<Y, SpF32>::value);
  static_assert(EPI < 2 || (WORDS && !F64), "the fused polynomial epilogues are FP32");
  __shared__ cpx<T> sh[8 * 6 * SPL_SITES];
  pdl_trigger();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long site = (long)blockIdx.x * SPL_SITES + lane;
  const bool ok = site < a.g.Vh;
  const unsigned cb = ok ? (unsigned)site : 0u;   // a lane without a site repeats site 0 and stores nothing
  int c[4];
  a.g.coords(cb, a.out_par, c);
  cpx<T> u[6];
  bool run;
  switch (w) {
    case 0: run = split_dir<0, DAG>(a, cb, c, u); break;
    case 1: run = split_dir<1, DAG>(a, cb, c, u); break;
    case 2: run = split_dir<2, DAG>(a, cb, c, u); break;
    case 3: run = split_dir<3, DAG>(a, cb, c, u); break;
    case 4: run = split_dir<4, DAG>(a, cb, c, u); break;
    case 5: run = split_dir<5, DAG>(a, cb, c, u); break;
    case 6: run = split_dir<6, DAG>(a, cb, c, u); break;
    default: run = split_dir<7, DAG>(a, cb, c, u); break;
  }
  if (!run) return;
  // the epilogue's operands are requested before the products meet
  double2 y0, y1;
  float4 yv, vv, sv, pv;
  if constexpr (EPI >= 1 && WORDS) {
    if constexpr (F64) {
      y0 = a.y.p[w * a.y.stride + cb];
      if (w < 4) y1 = a.y.p[(8 + w) * a.y.stride + cb];
    } else if (w < 6) {
      yv = a.y.p[w * a.y.stride + cb];
      if constexpr (EPI >= 2) vv = pe.v.p[w * pe.v.stride + cb];
      if constexpr (EPI == 2) {
        sv = pe.s.p[w * pe.s.stride + cb];
        pv = pe.sp.p[w * pe.sp.stride + cb];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) sh[(w * 6 + k) * SPL_SITES + lane] = u[k];
  __syncthreads();
  const cpx<T>* q = sh + lane;
  const T al = (T)a.alpha;
  double part[1] = {0.0};
  if constexpr (F64) {
    // warp w: component w, warps 0 to 3 also component 8 + w (three for every scheduler)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (k == 1 && w >= 4) break;
      const int j = k * 8 + w;
      cpx<T> r = split_sum_at<DAG>(j, q);
      if constexpr (EPI == 1) {
        const double2 y = k ? y1 : y0;
        r = mk<T>(fma(al, r.r, y.x), fma(al, r.i, y.y));
      }
      if (ok) {
        a.out.p[j * a.out.stride + cb] = make_double2(r.r, r.i);
        if constexpr (NORM) part[0] += r.r * r.r + r.i * r.i;
      }
    }
  } else if constexpr (WORDS) {
    // warps 0 to 5: one 16-byte word (two components) each
    if (w < 6) {
      const cpx<T> r0 = split_sum_at<DAG>(2 * w, q), r1 = split_sum_at<DAG>(2 * w + 1, q);
      float4 o = make_float4(r0.r, r0.i, r1.r, r1.i);
      if constexpr (EPI >= 1)
        o = make_float4(fmaf(al, o.x, yv.x), fmaf(al, o.y, yv.y), fmaf(al, o.z, yv.z), fmaf(al, o.w, yv.w));
      if constexpr (EPI == 2) {
        o.x = pe.ca * (vv.x + pe.cmu * sv.x - o.x) - pe.cb * pv.x;
        o.y = pe.ca * (vv.y + pe.cmu * sv.y - o.y) - pe.cb * pv.y;
        o.z = pe.ca * (vv.z + pe.cmu * sv.z - o.z) - pe.cb * pv.z;
        o.w = pe.ca * (vv.w + pe.cmu * sv.w - o.w) - pe.cb * pv.w;
      }
      if constexpr (EPI == 3) {
        const cpx<float> z = mk(pe.ca, pe.cb), e0 = cfma(z, mk(vv.x, vv.y), mk(o.x, o.y)),
                         e1 = cfma(z, mk(vv.z, vv.w), mk(o.z, o.w));
        o = make_float4(e0.r, e0.i, e1.r, e1.i);
      }
      if (ok) {
        if constexpr (OUT64) {
          a.out.p[2 * w * a.out.stride + cb] = make_double2(f64_of(o.x), f64_of(o.y));
          a.out.p[(2 * w + 1) * a.out.stride + cb] = make_double2(f64_of(o.z), f64_of(o.w));
        } else {
          a.out.p[w * a.out.stride + cb] = o;
        }
        if constexpr (NORM) part[0] = (double)fmaf(o.x, o.x, fmaf(o.y, o.y, fmaf(o.z, o.z, o.w * o.w)));
      }
    }
  } else {
    // a 16-bit field is scaled by its site's largest component: the components
    // come together again and warp 0 finishes the sites
    __shared__ cpx<T> sh2[12 * SPL_SITES];
    if (w < 6) {
      sh2[2 * w * SPL_SITES + lane] = split_sum_at<DAG>(2 * w, q);
      sh2[(2 * w + 1) * SPL_SITES + lane] = split_sum_at<DAG>(2 * w + 1, q);
    }
    __syncthreads();
    if (w == 0) {
      cpx<T> acc[12];
#pragma unroll
      for (int j = 0; j < 12; ++j) acc[j] = sh2[j * SPL_SITES + lane];
      if constexpr (EPI == 1) {
        cpx<T> y[12];
        a.y.template loadT<false>(cb, y);
#pragma unroll
        for (int j = 0; j < 12; ++j) acc[j] = y[j] + al * acc[j];
      }
      if (ok) {
        a.out.store(cb, acc);
        if constexpr (NORM) part[0] = site_norm2(acc);
      }
    }
  }
  if constexpr (NORM) {
    // the warps' values meet in warp 0 first: one FP64 tree in a block, not eight
    __shared__ double shn[SPL_THREADS];
    shn[threadIdx.x] = part[0];
    __syncthreads();
    part[0] = 0.0;
    if (w == 0) {
#pragma unroll
      for (int k = 0; k < 8; ++k) part[0] += shn[k * 32 + lane];
    }
    double tot[1];
    if (grid_sum<1, true>(a.red, part, tot)) {
      CGState* st = a.st;
      if (st != nullptr) {
        st->pAp = tot[0];
        if (!(tot[0] > 0.0) || !isfinite(tot[0])) st->flag |= FLAG_NAN;
        else st->alpha = st->rr / tot[0];
      }
    }
  }
}

// the lines lie between the last size that gains and the first that does not (above)
constexpr long SPLIT_MAX_VH_F64 = 500000;
constexpr long SPLIT_MAX_VH = 12288;
constexpr long SPLIT_MAX_VH_16 = 4096;   // a 16-bit output is finished by one warp of the eight
static_assert(SPLIT_MAX_VH_F64 / SPL_SITES < RED_MAX_BLOCKS, "a slot per block in the grid sum");

inline bool split_eligible(const wd_ctx* c, int fmt) {   // fmt of the input spinors
  return c->g.Vh <= (fmt == WD_F64 ? SPLIT_MAX_VH_F64 : fmt == WD_F32 ? SPLIT_MAX_VH : SPLIT_MAX_VH_16);
}

template <class T, class In, class Out, class Y, class G>
int hop_split(wd_ctx* c, bool dag, bool xpay, bool norm, const HopArgs<In, Out, Y, G>& a) {
  if (norm && (dag || !xpay)) return fail(WD_ERR_ARG, "hop: the |out|^2 epilogue exists for M_hat only");
  const int nb = nblocks(c->g.Vh, SPL_SITES);
  const HopPoly pe{};
  const bool early = !std::is_same<T, double>::value || early_gains_f64(nb, c->nsm);
  if (!dag) {
    if (!xpay) pdl_launch_if(c, early, k_hop_split<T, false, 0, false, In, Out, Y, G>, nb, SPL_THREADS, 0, a, pe);
    else if (!norm) pdl_launch_if(c, early, k_hop_split<T, false, 1, false, In, Out, Y, G>, nb, SPL_THREADS, 0, a, pe);
    else pdl_launch_if(c, early, k_hop_split<T, false, 1, true, In, Out, Y, G>, nb, SPL_THREADS, 0, a, pe);
  } else {
    if (!xpay) pdl_launch_if(c, early, k_hop_split<T, true, 0, false, In, Out, Y, G>, nb, SPL_THREADS, 0, a, pe);
    else pdl_launch_if(c, early, k_hop_split<T, true, 1, false, In, Out, Y, G>, nb, SPL_THREADS, 0, a, pe);
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

// FP32 arithmetic on the context's 12-real or 18-real links: eight threads per
// site on small lattices, else the staged pipeline
template <class In, class Out, class Y, class G>
int hop_fp32(wd_ctx* c, int out_par, bool dag, const In& I, const Out& O, const Y& Yv, const G& gauge, bool xpay,
             double alpha, bool norm_cg, bool in_cg) {
  const HopArgs<In, Out, Y, G> a{c->g, out_par, I, O, Yv, gauge, alpha, reducer(c), (norm_cg || in_cg) ? c->cgs : nullptr};
  if (split_eligible(c, In::fmt)) return hop_split<float>(c, dag, xpay, norm_cg, a);
  return hop_staged(c, dag, xpay, norm_cg, a);
}
template <class In, class Out, class Y>
int hop_links(wd_ctx* c, int out_par, bool dag, const In& I, const Out& O, const Y& Yv, bool xpay, double alpha,
              bool norm_cg, bool in_cg) {
  if (c->recon == WD_RECON_12)
    return hop_fp32(c, out_par, dag, I, O, Yv, GF32R12{c->gauge32r12, c->g.Vh}, xpay, alpha, norm_cg, in_cg);
  return hop_fp32(c, out_par, dag, I, O, Yv, GF32{c->gauge32, c->g.Vh}, xpay, alpha, norm_cg, in_cg);
}

}  // namespace wd
