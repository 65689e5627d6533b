// Staged hopping stencil for FP32 links (Section 3.1 of the paper: Wilson
// fermions, even-odd preconditioning), any spinor storage format.
//
// One thread per site.  A register-only kernel holds a direction's neighbour
// loads in registers, so at the register count that fills an SM too few bytes are in
// flight (long-scoreboard stalls dominate).  Here every thread runs its own
// software pipeline over the eight neighbour directions: the link of direction
// D + NST is copied global -> shared with cp.async while direction D is computed, so
// NST directions' links are in flight without holding registers, and the neighbour
// spinors of the next SA directions are in registers.  A thread reads only the
// shared words it copied itself, so no block barrier is needed; NST + 1 buffers
// make the buffer being refilled one whose values were consumed in the previous
// step.  Neighbour spinors are read through L1 (each is read by eight sites, several
// of them in the same block).
//
// How deep (hop_depth): a lattice of many waves of blocks is bound by HBM and wants
// resident blocks; one that fits the SMs at once is bound by the chain of
// eight neighbour reads, and registers that no second block would use hold more of them
// in flight.  K_hat in a chain on 152 SMs, its conversion from FP64 included (products in one chain), us, by depth
// (NST, SA, blocks per SM), FP32 spinors:
//                       12 reals                           18 reals
//                 blocks (2,1,5) (4,2,4) (6,3,3) (6,5,2)   (2,1,5) (4,2,4) (4,3,3) (5,5,2)
//   12^3 x 24        162   32.5    27.5    25.7    21.5      42.4    32.3    28.5    21.3
//   16^4             256   32.7    27.0    26.2    22.6      41.7    30.7    28.7    21.9
//   16^3 x 24        384   34.0    30.2    26.0    29.2      44.3    34.6    29.0    33.5
//   16^3 x 32        512   36.1    31.9    35.4    34.7      47.5    37.7    42.0    37.8
//   18x22x20x26      805   55.9    53.2    52.6    53.5      85.5    77.4    72.2    73.2
//   20x22x24x26     1073   69.9    67.1    72.6    76.2     107.4   100.3   100.8   105.4
//   24^4            1296   83.5    92.7    90.1    98.1     118.4   124.4   115.0   123.2
//   24^3 x 48       2592    171     176     178     193       229     225     215     225
//   32^3 x 64       8192    485     485     497     555       644     639     611     660
// so: two blocks per SM if all fit, three if all fit; with 12 reals four while that takes
// no more waves than the full occupancy; with 18 reals (9 KB a buffer) four if all fit, else three.
// 16-bit spinors, (2,1,6) (4,3,4) (6,4,3) on 12 reals: 12^3 x 24 34.2, 32.7, 29.2; 16^3 x 32
// 43.2, 35.6, 37.6; 24^4 80.3, 83.3, 83.7; 32^3 x 64 445, 464, 481; (2,1,5) (4,3,4) on 18 reals:
// 12^3 x 24 37.2, 36.4; 16^3 x 32 43.7, 37.3; 24^4 107, 115; 32^3 x 64 569, 577.
#pragma once
#include <atomic>

#include "dslash_impl.cuh"

namespace wd {

constexpr int HOP_ST_THREADS = 128;

__device__ __forceinline__ void cpa16(float4* sdst, const float4* gsrc) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gsrc) : "memory");
}

__device__ __forceinline__ void cpa8(float2* sdst, const float2* gsrc) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cpa_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// a thread's link in a buffer [words][threads]: 12 reals as three 16-byte words,
// 18 reals as nine 8-byte words
template <class G> struct LinkBuf;
template <> struct LinkBuf<GF32R12> {
  using W = float4;
  static constexpr int N = 3, NU = 6;
  __device__ __forceinline__ static void copy(W* s, int nt, const W* g, long stride) {
#pragma unroll
    for (int j = 0; j < 3; ++j) cpa16(s + j * nt, g + j * stride);
  }
  __device__ __forceinline__ static void read(const W* s, int nt, cpx<float> (&U)[6]) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float4 v = s[j * nt];
      U[2 * j] = {v.x, v.y};
      U[2 * j + 1] = {v.z, v.w};
    }
  }
  template <bool TWO>
  __device__ __forceinline__ static void mul(const cpx<float> (&U)[6], const cpx<float> (&h)[6], cpx<float> (&o)[6]) {
    if constexpr (TWO) su3_mul_r12_2c(U, h, o);
    else su3_mul_r12(U, h, o);
  }
  template <bool TWO>
  __device__ __forceinline__ static void dag_mul(const cpx<float> (&U)[6], const cpx<float> (&h)[6], cpx<float> (&o)[6]) {
    if constexpr (TWO) su3_dag_mul_r12_2c(U, h, o);
    else su3_dag_mul_r12(U, h, o);
  }
};
template <> struct LinkBuf<GF32> {
  using W = float2;
  static constexpr int N = 9, NU = 9;
  __device__ __forceinline__ static void copy(W* s, int nt, const W* g, long stride) {
#pragma unroll
    for (int j = 0; j < 9; ++j) cpa8(s + j * nt, g + j * stride);
  }
  __device__ __forceinline__ static void read(const W* s, int nt, cpx<float> (&U)[9]) {
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      const float2 v = s[j * nt];
      U[j] = {v.x, v.y};
    }
  }
  template <bool TWO>
  __device__ __forceinline__ static void mul(const cpx<float> (&U)[9], const cpx<float> (&h)[6], cpx<float> (&o)[6]) {
    if constexpr (TWO) su3_mul_2c(U, h, o);
    else su3_mul(U, h, o);
  }
  template <bool TWO>
  __device__ __forceinline__ static void dag_mul(const cpx<float> (&U)[9], const cpx<float> (&h)[6], cpx<float> (&o)[6]) {
    if constexpr (TWO) su3_dag_mul_2c(U, h, o);
    else su3_dag_mul(U, h, o);
  }
};
template <class G> constexpr size_t hop_smem(int nst) {
  return (size_t)(nst + 1) * LinkBuf<G>::N * HOP_ST_THREADS * sizeof(typename LinkBuf<G>::W);
}

// TWO: the products in two chains of three (dot3), for FP32 spinors from four blocks per SM on
// (18 reals: three), where other warps hide the longer issue: K_hat against FP64 keeps the
// rounding of separately rounded products (16^3 x 32, 18 / 12 reals: 5.46e-8 / 5.54e-8; one
// chain of six 5.57e-8 / 5.70e-8; two of three 5.46e-8 / 5.59e-8, 5.58e-8 with row 2 in products apart,
// which costs 1 % more time) and takes 0.5 to 1 % less time at 24^4 and above, 1 to 2 % more at 16^3 x 32.  With two or three blocks of 12 reals per SM, one wave, two chains
// cost 3 to 6 % and stay out (2 % more rounding); 16-bit spinors round far more by their format.
template <int NST, int SA, bool DAG, class A, bool TWO = false>
struct Staged {
  using G = typename std::remove_cv<decltype(A::gauge)>::type;
  using LB = LinkBuf<G>;
  static constexpr int NB = NST + 1;          // buffers
  static_assert(NST >= 1 && NST <= 7 && SA >= 0 && SA <= 7, "one to seven directions in flight");
  const A& a;
  long cb;
  int c[4];
  float4* buf;                                // [NB][LB::N][threads]
  int tid, nt;

  __device__ __forceinline__ typename LB::W* slot(int b) const {
    return reinterpret_cast<typename LB::W*>(buf) + b * LB::N * nt + tid;
  }

  template <int D> __device__ __forceinline__ long nbr() const { return a.g.template nbr<D>((unsigned)cb, c); }

  template <int D> __device__ __forceinline__ void issue() const {
    if constexpr (D < 8) {
      constexpr int MU = D >> 1;
      const int lpar = (D & 1) == 0 ? a.out_par : 1 - a.out_par;
      const long li = (D & 1) == 0 ? cb : nbr<D>();
      LB::copy(slot(D % NB), nt, a.gauge.p + ((long)(MU * 2 + lpar) * LB::N) * a.gauge.stride + li, a.gauge.stride);
    }
    cpa_commit();                              // possibly empty: keeps one group per step
  }

  template <int D> __device__ __forceinline__ void step(cpx<float> (&acc)[12]) const {
    cpx<float> s[12];
    a.in.template loadT<false>(nbr<D>(), s);
    compute<D>(acc, s);
  }

  // the same with SA directions' spinors in flight: direction D + SA is requested, D used
  template <int D, class R> __device__ __forceinline__ void first(R& r) const {
    if constexpr (D < SA) {
      a.in.loadRaw(nbr<D>(), r[D]);
      first<D + 1>(r);
    }
  }
  template <int D, class R> __device__ __forceinline__ void ahead(cpx<float> (&acc)[12], R& r) const {
    if constexpr (D < 8) {
      if constexpr (D + SA < 8) a.in.loadRaw(nbr<D + SA>(), r[(D + SA) % (SA + 1)]);
      cpx<float> s[12];
      a.in.unpack(r[D % (SA + 1)], s);
      compute<D>(acc, s);
      ahead<D + 1>(acc, r);
    }
  }

  template <int D> __device__ __forceinline__ void compute(cpx<float> (&acc)[12], const cpx<float> (&s)[12]) const {
    constexpr int MU = D >> 1;
    constexpr bool FWD = (D & 1) == 0;
    cpa_wait<NST - 1>();                       // direction D has landed
    cpx<float> U[LB::NU], h[6], u[6];
    LB::read(slot(D % NB), nt, U);
    issue<D + NST>();                          // refills the buffer of direction D - 1
    constexpr int SF = DAG ? +1 : -1;
    constexpr int SG = FWD ? SF : -SF;
    spin_project<MU, SG>(s, h);
    if (MU == 3 && (FWD ? c[3] == a.g.L[3] - 1 : c[3] == 0)) {
#pragma unroll
      for (int j = 0; j < 6; ++j) h[j] = mk<float>(-h[j].r, -h[j].i);
    }
    if constexpr (FWD) LB::template mul<TWO>(U, h, u);
    else LB::template dag_mul<TWO>(U, h, u);
    spin_accum<MU, SG, D == 0>(acc, u);        // direction 0 writes acc
  }

  // directions 0 .. NST - 1 go out before the first step
  template <int D> __device__ __forceinline__ void prologue() const {
    if constexpr (D < NST) {
      issue<D>();
      prologue<D + 1>();
    }
  }

  __device__ __forceinline__ void run_after_prologue(cpx<float> (&acc)[12]) const {
    if constexpr (SA > 0) {
      using In = typename std::remove_cv<decltype(a.in)>::type;
      typename In::Raw r[SA + 1];
      first<0>(r);
      ahead<0>(acc, r);
    } else {
      step<0>(acc);
      step<1>(acc);
      step<2>(acc);
      step<3>(acc);
      step<4>(acc);
      step<5>(acc);
      step<6>(acc);
      step<7>(acc);
    }
  }
};

// Operands fused into the last hop of K_hat (FP32):
//   EPI 2, the Chebyshev step out = ca (v + cmu s - (y + alpha D in)) - cb sp: saves
//          the K s vector and a five-vector pass
//   EPI 3, a factor of a root product out = y + alpha D in + (ca + i cb) v: saves a
//          four-vector pass
struct HopPoly {
  SpF32 v, s, sp;
  float ca, cmu, cb;
};

// EPI 0: out = D in; 1: out = y + alpha D in; 2 and 3: as above
template <bool DAG, int EPI, bool NORM, int NST, int SA, int MINB, class In, class Out, class Y, class G>
__global__ void __launch_bounds__(HOP_ST_THREADS, MINB) k_hop_st(HopArgs<In, Out, Y, G> a, HopPoly pe) {
  extern __shared__ float4 sbuf[];
  pdl_trigger();
  const long site = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool ok = site < a.g.Vh;
  const long cb = ok ? site : 0;               // a thread without a site repeats site 0 and stores nothing
  constexpr bool TWO = std::is_same<In, SpF32>::value && MINB >= (std::is_same<G, GF32>::value ? 3 : 4);
  Staged<NST, SA, DAG, HopArgs<In, Out, Y, G>, TWO> S{a, cb, {0, 0, 0, 0}, sbuf, (int)threadIdx.x, (int)blockDim.x};
  a.g.coords(cb, a.out_par, S.c);
  S.template prologue<0>();                    // the links do not depend on the kernels before
  pdl_wait();
  if (a.st != nullptr && a.st->flag != 0) {
    cpa_wait<0>();
    return;
  }
  cpx<float> acc[12];
  S.run_after_prologue(acc);
  if constexpr (EPI >= 1) {
    cpx<float> yv[12];
    a.y.template loadT<false>(cb, yv);
    const float al = (float)a.alpha;
#pragma unroll
    for (int j = 0; j < 12; ++j) acc[j] = yv[j] + al * acc[j];
  }
  if constexpr (EPI == 2) {
    cpx<float> x[12], q[12];
    pe.v.template loadT<false>(cb, x);
    pe.s.template loadT<false>(cb, q);
#pragma unroll
    for (int j = 0; j < 12; ++j) acc[j] = x[j] + pe.cmu * q[j] - acc[j];
    pe.sp.template loadT<false>(cb, q);
#pragma unroll
    for (int j = 0; j < 12; ++j) acc[j] = pe.ca * acc[j] - pe.cb * q[j];
  }
  if constexpr (EPI == 3) {
    cpx<float> x[12];
    pe.v.template loadT<false>(cb, x);
    const cpx<float> z = mk(pe.ca, pe.cb);
#pragma unroll
    for (int j = 0; j < 12; ++j) acc[j] = cfma(z, x[j], acc[j]);
  }
  double part[1] = {0.0};
  if constexpr (NORM) { if (ok) part[0] = site_norm2(acc); }
  if (ok) a.out.store(cb, acc);
  if constexpr (NORM) {
    double tot[1];
    if (grid_sum<1>(a.red, part, tot)) {
      CGState* st = a.st;
      if (st != nullptr) {
        st->pAp = tot[0];
        if (!(tot[0] > 0.0) || !isfinite(tot[0])) st->flag |= FLAG_NAN;
        else st->alpha = st->rr / tot[0];
      }
    }
  }
}

// Resident blocks per SM that the pipeline's depth is chosen for (table at the top):
// 2, 3, 4 or the full occupancy; full = 0: not beyond one wave of four, else three
inline int hop_depth(const wd_ctx* c, int full) {
  const int nb = nblocks(c->g.Vh, HOP_ST_THREADS), n = c->nsm > 0 ? c->nsm : 1;
  if (nb <= 2 * n) return 2;
  if (nb <= 3 * n) return 3;
  if (full == 0) return nb <= 4 * n ? 4 : 3;
  return (nb + 4 * n - 1) / (4 * n) <= (nb + full * n - 1) / (full * n) ? 4 : full;
}

template <bool DAG, int EPI, bool NORM, int NST, int SA, int MINB, class In, class Out, class Y, class G>
void hop_st_go(wd_ctx* c, const HopArgs<In, Out, Y, G>& a, const HopPoly& pe) {
  auto k = k_hop_st<DAG, EPI, NORM, NST, SA, MINB, In, Out, Y, G>;
  constexpr size_t sm = hop_smem<G>(NST);
  if constexpr (sm > 47 * 1024) {              // above 48 KB (with the grid sum's) a kernel has to ask, once per device
    static std::atomic<unsigned long long> asked{0};
    const unsigned long long bit = 1ull << (c->device & 63);
    if ((asked.load() & bit) == 0 || c->device >= 64) {
      (void)cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);   // a failure shows at the launch
      asked.fetch_or(bit);
    }
  }
  pdl_launch(c, k, nblocks(c->g.Vh, HOP_ST_THREADS), HOP_ST_THREADS, sm, a, pe);
}
template <bool DAG, int EPI, bool NORM, class In, class Out, class Y, class G>
void hop_st_depth(wd_ctx* c, const HopArgs<In, Out, Y, G>& a, const HopPoly& pe) {
  if constexpr (std::is_same<G, GF32>::value) {
    // 55 KB a block at NST = 5
    if constexpr (std::is_same<In, SpF32>::value) {
      switch (hop_depth(c, 0)) {
        case 2: hop_st_go<DAG, EPI, NORM, 5, 5, 2>(c, a, pe); break;
        case 4: hop_st_go<DAG, EPI, NORM, 4, 2, 4>(c, a, pe); break;
        default: hop_st_go<DAG, EPI, NORM, 4, 3, 3>(c, a, pe);
      }
    } else {
      if (hop_depth(c, 5) <= 4) hop_st_go<DAG, EPI, NORM, 4, 3, 4>(c, a, pe);
      else hop_st_go<DAG, EPI, NORM, 2, 1, 5>(c, a, pe);
    }
  } else if constexpr (std::is_same<In, SpF32>::value) {
    switch (hop_depth(c, 5)) {
      case 2: hop_st_go<DAG, EPI, NORM, 6, 5, 2>(c, a, pe); break;
      case 3: hop_st_go<DAG, EPI, NORM, 6, 3, 3>(c, a, pe); break;
      case 4: hop_st_go<DAG, EPI, NORM, 4, 2, 4>(c, a, pe); break;
      default: hop_st_go<DAG, EPI, NORM, 2, 1, 5>(c, a, pe);
    }
  } else {
    switch (hop_depth(c, 6)) {
      case 2:
      case 3: hop_st_go<DAG, EPI, NORM, 6, 4, 3>(c, a, pe); break;
      case 4: hop_st_go<DAG, EPI, NORM, 4, 3, 4>(c, a, pe); break;
      default: hop_st_go<DAG, EPI, NORM, 2, 1, 6>(c, a, pe);
    }
  }
}

// Launch of the staged stencil on the links G of the context
template <class In, class Out, class Y, class G>
int hop_staged(wd_ctx* c, bool dag, bool xpay, bool norm_cg, const HopArgs<In, Out, Y, G>& a) {
  if (norm_cg && nblocks(c->g.Vh, 64) > RED_MAX_BLOCKS) return fail(WD_ERR_ARG, "lattice too large for one reduction grid");
  if (norm_cg && (dag || !xpay)) return fail(WD_ERR_ARG, "hop: the |out|^2 epilogue exists for M_hat only");
  const HopPoly pe{};
  if (!dag) {
    if (!xpay) hop_st_depth<false, 0, false>(c, a, pe);
    else if (!norm_cg) hop_st_depth<false, 1, false>(c, a, pe);
    else hop_st_depth<false, 1, true>(c, a, pe);
  } else {
    if (!xpay) hop_st_depth<true, 0, false>(c, a, pe);
    else hop_st_depth<true, 1, false>(c, a, pe);
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

}  // namespace wd
