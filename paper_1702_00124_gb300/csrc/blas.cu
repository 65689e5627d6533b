// Vector kernels on half-lattice spinor fields: precision conversion, linear
// combinations, FP64 inner products (deterministic grid sums), and the fused
// conjugate-gradient updates whose scalars stay on the device.
//
// Arithmetic: FP64 when every field is FP64, FP32 otherwise; inner products
// and norms always accumulate in FP64.
//
// Work split: fields are structures of arrays, so all but the 16-bit stores
// (whose scale needs the whole site) work word by word, one 16-byte word of one
// component or component pair per thread, instead of site by site.  That is
// 6 to 12 times the threads: on a small lattice the FP64 operations spread
// over 6 to 12 times the schedulers (at 33 ns per warp instruction a complex FP64
// axpby of a whole site took 10 us in one thread), and every load of a thread is
// independent.  Sums run over a grid of at most SUM_BLOCKS blocks with a stride loop, so
// that the FP64 block trees and the last block's pass stay small.
// Measured on whole solves, site by site -> word by word: FP64 CG at 4^4 2.45 -> 2.14 ms,
// mixed FP32 CG at 8^3 x 16 3.36 -> 3.21 ms, BF16 CG at 12^3 x 24 8.00 -> 7.32 ms.
#include "dslash_impl.cuh"

namespace wd {

constexpr int BL_THREADS = 256;
// plain load (not the read-only path: see pdl_wait)
template <class W> __device__ __forceinline__ W ldw(const W* p) { return *p; }

// Eight blocks per SM, a full GB300.  FP64 CG at 16^3 x 32 with 152 / 304 / 608 / 1216 /
// 2432 blocks: 43.1 / 42.5 / 42.1 / 41.8 / 42.2 ms; BF16 CG at 12^3 x 24: 5.09 / 5.07 /
// 5.01 / 5.03 / 5.11 ms (fewer leave each thread a longer chain, more lengthen the last pass)
constexpr int SUM_BLOCKS = 8 * 152;


size_t field_bytes(int fmt, long Vh) {
  switch (fmt) {
    case WD_F64:
    case WD_DD: return (size_t)Vh * 24 * 8;
    case WD_F32: return (size_t)Vh * 24 * 4;
    default: return (size_t)Vh * 24 * 2;   // the norm array is separate
  }
}

template <class Fn>
static int with_fmt(const Field& f, Fn&& fn) {
  switch (f.fmt) {
    case WD_F64: return fn(sp64(f));
    case WD_F32: return fn(sp32(f));
    case WD_F16: return fn(sp16<__half>(f));
    case WD_BF16: return fn(sp16<__nv_bfloat16>(f));
    case WD_DD: return fn(spdd(f));
  }
  return fail(WD_ERR_ARG, "unknown field format");
}

// arithmetic of a kernel on two formats: FP64 when both are FP64, double-float
// when both are double-float, FP64 for conversions between the two, else FP32
template <class A, class B> struct Pick { using T = float; };
template <> struct Pick<SpF64, SpF64> { using T = double; };
template <> struct Pick<SpDD, SpDD> { using T = dd; };
template <> struct Pick<SpF64, SpDD> { using T = double; };
template <> struct Pick<SpDD, SpF64> { using T = double; };

// ---------------------------------------------------------------------------
// Words of a field: one component (double2; double-float float4) or a pair (FP32 float4)
template <class F> struct Words;
template <> struct Words<SpF64> {
  using W = double2;
  using T = double;
  static constexpr int N = 12, NC = 1;
  __device__ __forceinline__ static void get(const W& w, cpx<T> (&c)[NC]) { c[0] = {w.x, w.y}; }
  __device__ __forceinline__ static W put(const cpx<T> (&c)[NC]) { return make_double2(c[0].r, c[0].i); }
};
template <> struct Words<SpF32> {
  using W = float4;
  using T = float;
  static constexpr int N = 6, NC = 2;
  __device__ __forceinline__ static void get(const W& w, cpx<T> (&c)[NC]) {
    c[0] = {w.x, w.y};
    c[1] = {w.z, w.w};
  }
  __device__ __forceinline__ static W put(const cpx<T> (&c)[NC]) { return make_float4(c[0].r, c[0].i, c[1].r, c[1].i); }
};
template <> struct Words<SpDD> {
  using W = float4;
  using T = dd;
  static constexpr int N = 12, NC = 1;
  __device__ __forceinline__ static void get(const W& w, cpx<T> (&c)[NC]) { c[0] = {dd(w.x, w.y), dd(w.z, w.w)}; }
  __device__ __forceinline__ static W put(const cpx<T> (&c)[NC]) { return make_float4(c[0].r.hi, c[0].r.lo, c[0].i.hi, c[0].i.lo); }
};
// every field's stride is Vh: its words are one contiguous array
template <class F> inline long nwords(long Vh) { return (long)Words<F>::N * Vh; }
inline int sum_blocks(long n) { return (int)std::min<long>(SUM_BLOCKS, (n + BL_THREADS - 1) / BL_THREADS); }

// ---------------------------------------------------------------------------
// conversions site by site (a 16-bit side)
template <class T, class In, class Out>
__global__ void k_convert(long n, In in, Out out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  cpx<T> s[12];
  in.template loadT<false>(i, s);
  out.store(i, s);
}
// the same word by word; blockIdx.y = word of the format with fewer words
__global__ void k_f64_to_f32(long n, const double2* in, float4* out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= n) return;
  const double2 a = ldw(in + 2 * j * n + i), b = ldw(in + (2 * j + 1) * n + i);
  out[j * n + i] = make_float4(f32_of(a.x), f32_of(a.y), f32_of(b.x), f32_of(b.y));
}
__global__ void k_f32_to_f64(long n, const float4* in, double2* out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= n) return;
  const float4 v = ldw(in + j * n + i);
  out[2 * j * n + i] = make_double2(f64_of(v.x), f64_of(v.y));
  out[(2 * j + 1) * n + i] = make_double2(f64_of(v.z), f64_of(v.w));
}
__global__ void k_f64_to_dd(long n, const double2* in, float4* out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 v = ldw(in + i);
  const dd r(v.x), m(v.y);
  out[i] = make_float4(r.hi, r.lo, m.hi, m.lo);
}
__global__ void k_dd_to_f64(long n, const float4* in, double2* out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 v = ldw(in + i);
  out[i] = make_double2((double)dd(v.x, v.y), (double)dd(v.z, v.w));
}
// 16 bits to FP64: a word's four components (only the way back needs the site's largest).
// Site by site, with an early start, a hop between FP64 fields at 16^3 x 32 took 23 to 29 us, the
// blocks of this launch piling up on some SMs (plain launches of both conversions 19 us, but K_hat
// 5 % longer); word by word 20 us.
template <class S>
__global__ void k_16_to_f64(long n, S in, double2* out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= n) return;
  cpx<float> v[4];
  in.word(i, (int)j, v);
#pragma unroll
  for (int q = 0; q < 4; ++q) out[(4 * j + q) * n + i] = make_double2(f64_of(v[q].r), f64_of(v[q].i));
}
template <class W>
__global__ void k_copy(long n, const W* in, W* out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = ldw(in + i);
}

int convert(wd_ctx* c, const Field& in, const Field& out) {
  const long n = c->g.Vh;
  const int n12 = nblocks(12 * n, BL_THREADS);
  const dim3 g6(nblocks(n, BL_THREADS), 6);
  const int fi = in.fmt, fo = out.fmt;
  if (fi == WD_F64 && fo == WD_F64) {
    pdl_launch(c, k_copy<double2>, n12, BL_THREADS, 0, 12 * n, (const double2*)in.data, (double2*)out.data);
  } else if (fi == WD_DD && fo == WD_DD) {
    pdl_launch(c, k_copy<float4>, n12, BL_THREADS, 0, 12 * n, (const float4*)in.data, (float4*)out.data);
  } else if (fi == WD_F32 && fo == WD_F32) {
    pdl_launch(c, k_copy<float4>, nblocks(6 * n, BL_THREADS), BL_THREADS, 0, 6 * n, (const float4*)in.data,
               (float4*)out.data);
  } else if (fi == WD_F64 && fo == WD_F32) {
    pdl_launch(c, k_f64_to_f32, g6, BL_THREADS, 0, n, (const double2*)in.data, (float4*)out.data);
  } else if (fi == WD_F32 && fo == WD_F64) {
    pdl_launch(c, k_f32_to_f64, g6, BL_THREADS, 0, n, (const float4*)in.data, (double2*)out.data);
  } else if (fi == WD_F16 && fo == WD_F64) {
    pdl_launch(c, k_16_to_f64<Sp16<__half>>, dim3(nblocks(n, BL_THREADS), 3), BL_THREADS, 0, n, sp16<__half>(in), (double2*)out.data);
  } else if (fi == WD_BF16 && fo == WD_F64) {
    pdl_launch(c, k_16_to_f64<Sp16<__nv_bfloat16>>, dim3(nblocks(n, BL_THREADS), 3), BL_THREADS, 0, n, sp16<__nv_bfloat16>(in),
               (double2*)out.data);
  } else if (fi == WD_F64 && fo == WD_DD) {
    pdl_launch(c, k_f64_to_dd, n12, BL_THREADS, 0, 12 * n, (const double2*)in.data, (float4*)out.data);
  } else if (fi == WD_DD && fo == WD_F64) {
    pdl_launch(c, k_dd_to_f64, n12, BL_THREADS, 0, 12 * n, (const float4*)in.data, (double2*)out.data);
  } else {
    return with_fmt(in, [&](auto I) {
      return with_fmt(out, [&](auto O) {
        using T = typename Pick<decltype(I), decltype(O)>::T;
        pdl_launch(c, k_convert<T, decltype(I), decltype(O)>, nblocks(n, BL_THREADS), BL_THREADS, 0, n, I, O);
        WD_CHECK_LAUNCH();
        return (int)WD_OK;
      });
    });
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

// out = (ar + i ai) x + (br + i bi) y, all fields of one format, word by word.
// REAL: ai = bi = 0 (half the operations).
template <class F, bool REAL>
__global__ void k_axpby(long n, typename Words<F>::T ar, typename Words<F>::T ai, const typename Words<F>::W* x,
                        typename Words<F>::T br, typename Words<F>::T bi, const typename Words<F>::W* y,
                        typename Words<F>::W* out) {
  pdl_enter();
  using Q = Words<F>;
  using T = typename Q::T;
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  cpx<T> a[Q::NC], b[Q::NC];
  Q::get(ldw(x + i), a);
  Q::get(ldw(y + i), b);
#pragma unroll
  for (int j = 0; j < Q::NC; ++j) {
    if constexpr (REAL) a[j] = ar * a[j] + br * b[j];
    else a[j] = mk(ar, ai) * a[j] + mk(br, bi) * b[j];
  }
  out[i] = Q::put(a);
}
// the same for 16-bit fields, site by site
template <class T, class F>
__global__ void k_caxpby(long n, T ar, T ai, F x, T br, T bi, F y, F out) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  cpx<T> a[12], b[12];
  x.template loadT<false>(i, a);
  y.template loadT<false>(i, b);
  const cpx<T> ca = mk(ar, ai), cb = mk(br, bi);
#pragma unroll
  for (int j = 0; j < 12; ++j) a[j] = ca * a[j] + cb * b[j];
  out.store(i, a);
}

template <class F>
static void axpby_words(wd_ctx* c, double ar, double ai, const Field& x, double br, double bi, const Field& y,
                        const Field& out) {
  using T = typename Words<F>::T;
  using W = typename Words<F>::W;
  const long m = nwords<F>(c->g.Vh);
  const int nb = nblocks(m, BL_THREADS);
  if (ai == 0.0 && bi == 0.0)
    pdl_launch(c, k_axpby<F, true>, nb, BL_THREADS, 0, m, T(ar), T(ai), (const W*)x.data, T(br), T(bi),
                                                       (const W*)y.data, (W*)out.data);
  else
    pdl_launch(c, k_axpby<F, false>, nb, BL_THREADS, 0, m, T(ar), T(ai), (const W*)x.data, T(br), T(bi),
                                                        (const W*)y.data, (W*)out.data);
}
template <class H>
static void axpby_16(wd_ctx* c, double ar, double ai, const Field& x, double br, double bi, const Field& y,
                     const Field& out) {
  const long n = c->g.Vh;
  pdl_launch(c, k_caxpby<float, Sp16<H>>, nblocks(n, BL_THREADS), BL_THREADS, 0, n, (float)ar, (float)ai, sp16<H>(x), (float)br,
               (float)bi, sp16<H>(y), sp16<H>(out));
}

int caxpby(wd_ctx* c, double ar, double ai, const Field& x, double br, double bi, const Field& y,
           const Field& out) {
  if (x.fmt != y.fmt || x.fmt != out.fmt) return fail(WD_ERR_ARG, "caxpby: formats differ");
  switch (x.fmt) {
    case WD_F64: axpby_words<SpF64>(c, ar, ai, x, br, bi, y, out); break;
    case WD_F32: axpby_words<SpF32>(c, ar, ai, x, br, bi, y, out); break;
    case WD_DD: axpby_words<SpDD>(c, ar, ai, x, br, bi, y, out); break;
    case WD_F16: axpby_16<__half>(c, ar, ai, x, br, bi, y, out); break;
    case WD_BF16: axpby_16<__nv_bfloat16>(c, ar, ai, x, br, bi, y, out); break;
    default: return fail(WD_ERR_ARG, "unknown field format");
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

int axpby(wd_ctx* c, double a, const Field& x, double b, const Field& y, const Field& out) {
  return caxpby(c, a, 0.0, x, b, 0.0, y, out);
}

int zero(wd_ctx* c, const Field& f) {
  WD_CUDA(cudaMemsetAsync(f.data, 0, field_bytes(f.fmt, c->g.Vh), c->stream));
  if (f.norm) WD_CUDA(cudaMemsetAsync(f.norm, 0, sizeof(float) * c->g.Vh, c->stream));
  return WD_OK;
}

// ---------------------------------------------------------------------------
// inner products of FP64 fields, word by word: <a, b>, and |a|^2
__global__ void __launch_bounds__(BL_THREADS) k_dot64(long n, const double2* a, const double2* b, Reduce red) {
  pdl_enter();
  double v[2] = {0.0, 0.0};
  for (long i = (long)blockIdx.x * BL_THREADS + threadIdx.x; i < n; i += (long)gridDim.x * BL_THREADS) {
    const double2 x = ldw(a + i), y = ldw(b + i);
    v[0] = fma(x.y, y.y, fma(x.x, y.x, v[0]));
    v[1] = fma(-x.y, y.x, fma(x.x, y.y, v[1]));
  }
  grid_sum_hl<2>(red, v);
}
__global__ void __launch_bounds__(BL_THREADS) k_norm64(long n, const double2* a, Reduce red) {
  pdl_enter();
  double v[1] = {0.0};
  for (long i = (long)blockIdx.x * BL_THREADS + threadIdx.x; i < n; i += (long)gridDim.x * BL_THREADS) {
    const double2 x = ldw(a + i);
    v[0] = fma(x.y, x.y, fma(x.x, x.x, v[0]));
  }
  grid_sum_hl<1>(red, v);
}

int fetch_host(wd_ctx* c, int nv, double* out) {
  WD_CUDA(cudaStreamSynchronize(c->stream));
  for (int k = 0; k < nv; ++k) out[k] = c->host_scalar[k];
  return WD_OK;
}

static int check_sum(wd_ctx* c) {
  return nblocks(c->g.Vh, BL_THREADS) > RED_MAX_BLOCKS ? fail(WD_ERR_ARG, "dot: lattice too large") : (int)WD_OK;
}

int dot(wd_ctx* c, const Field& a, const Field& b, double* re, double* im) {
  if (a.fmt != WD_F64 || b.fmt != WD_F64) return fail(WD_ERR_ARG, "dot: FP64 fields");
  WD_TRY(check_sum(c));
  const long n = 12 * c->g.Vh;
  pdl_launch(c, k_dot64, sum_blocks(n), BL_THREADS, 0, n, (const double2*)a.data, (const double2*)b.data, reducer_host(c));
  WD_CHECK_LAUNCH();
  double v[2];
  WD_TRY(fetch_host(c, 2, v));
  if (re) *re = v[0];
  if (im) *im = v[1];
  return WD_OK;
}

int dot_hl(wd_ctx* c, const Field& a, const Field& b, double re[2]) {
  if (a.fmt != WD_F64 || b.fmt != WD_F64) return fail(WD_ERR_ARG, "dot_hl: FP64 fields");
  WD_TRY(check_sum(c));
  const long n = 12 * c->g.Vh;
  if (a.data == b.data) {
    pdl_launch(c, k_norm64, sum_blocks(n), BL_THREADS, 0, n, (const double2*)a.data, reducer_host(c));
    WD_CHECK_LAUNCH();
    return fetch_host(c, 2, re);
  }
  pdl_launch(c, k_dot64, sum_blocks(n), BL_THREADS, 0, n, (const double2*)a.data, (const double2*)b.data, reducer_host(c));
  WD_CHECK_LAUNCH();
  double v[4];
  WD_TRY(fetch_host(c, 4, v));
  re[0] = v[0];
  re[1] = v[2];
  return WD_OK;
}

// |b|^2 and whether x has an entry that is not zero, in one pass
__global__ void __launch_bounds__(BL_THREADS) k_norm_any(long n, const double2* b, const double2* x, Reduce red) {
  pdl_enter();
  double v[2] = {0.0, 0.0};
  bool any = false;
  for (long i = (long)blockIdx.x * BL_THREADS + threadIdx.x; i < n; i += (long)gridDim.x * BL_THREADS) {
    const double2 w = ldw(b + i), z = ldw(x + i);
    v[0] = fma(w.y, w.y, fma(w.x, w.x, v[0]));
    any = any || z.x != 0.0 || z.y != 0.0;     // true for NaN
  }
  v[1] = any ? 1.0 : 0.0;
  grid_sum_hl<2>(red, v);
}
int norm2_any(wd_ctx* c, const Field& b, const Field& x, double* bb, bool* nonzero) {
  if (b.fmt != WD_F64 || x.fmt != WD_F64) return fail(WD_ERR_ARG, "norm2_any: FP64 fields");
  WD_TRY(check_sum(c));
  const long n = 12 * c->g.Vh;
  pdl_launch(c, k_norm_any, sum_blocks(n), BL_THREADS, 0, n, (const double2*)b.data, (const double2*)x.data,
             reducer_host(c));
  WD_CHECK_LAUNCH();
  double v[4];
  WD_TRY(fetch_host(c, 4, v));
  *bb = v[0];
  *nonzero = v[1] != 0.0;
  return WD_OK;
}

int norm2(wd_ctx* c, const Field& a, double* out) {
  if (a.fmt != WD_F64) return fail(WD_ERR_ARG, "norm2: FP64 fields");
  WD_TRY(check_sum(c));
  const long n = 12 * c->g.Vh;
  pdl_launch(c, k_norm64, sum_blocks(n), BL_THREADS, 0, n, (const double2*)a.data, reducer_host(c));
  WD_CHECK_LAUNCH();
  return fetch_host(c, 1, out);
}

// r = b - t and |r|^2 in one pass; t FP64 or double-float
template <class F>
__global__ void __launch_bounds__(BL_THREADS) k_resid(long n, const double2* b, const typename Words<F>::W* t, double2* r,
                                                      Reduce red) {
  pdl_enter();
  double v[1] = {0.0};
  for (long i = (long)blockIdx.x * BL_THREADS + threadIdx.x; i < n; i += (long)gridDim.x * BL_THREADS) {
    const double2 x = ldw(b + i);
    double2 y;
    if constexpr (std::is_same<F, SpDD>::value) {
      const float4 w = ldw(t + i);
      y = make_double2((double)dd(w.x, w.y), (double)dd(w.z, w.w));
    } else {
      y = ldw(t + i);
    }
    const double2 d = make_double2(x.x - y.x, x.y - y.y);
    r[i] = d;
    v[0] = fma(d.y, d.y, fma(d.x, d.x, v[0]));
  }
  double tot[1];
  grid_sum<1>(red, v, tot);
}
int residual(wd_ctx* c, const Field& b, const Field& t, const Field& r, double* rr) {
  if (b.fmt != WD_F64 || r.fmt != WD_F64 || (t.fmt != WD_F64 && t.fmt != WD_DD))
    return fail(WD_ERR_ARG, "residual: b and r FP64, A x FP64 or double-float");
  WD_TRY(check_sum(c));
  const long n = 12 * c->g.Vh;
  if (t.fmt == WD_F64)
    pdl_launch(c, k_resid<SpF64>, sum_blocks(n), BL_THREADS, 0, n, (const double2*)b.data, (const double2*)t.data,
               (double2*)r.data, reducer_host(c));
  else
    pdl_launch(c, k_resid<SpDD>, sum_blocks(n), BL_THREADS, 0, n, (const double2*)b.data, (const float4*)t.data,
               (double2*)r.data, reducer_host(c));
  WD_CHECK_LAUNCH();
  return fetch_host(c, 1, rr);
}

// x += s, x FP64 and s FP32 or FP64 (a solver's increment); s is left zero
__global__ void k_fold32(long n, float4* s, double2* x) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= n) return;
  const float4 v = s[j * n + i];
  double2 a = x[2 * j * n + i], b = x[(2 * j + 1) * n + i];
  a.x += (double)v.x;
  a.y += (double)v.y;
  b.x += (double)v.z;
  b.y += (double)v.w;
  x[2 * j * n + i] = a;
  x[(2 * j + 1) * n + i] = b;
  s[j * n + i] = make_float4(0.f, 0.f, 0.f, 0.f);
}
__global__ void k_fold64(long n, double2* s, double2* x) {
  pdl_enter();
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 v = s[i], a = x[i];
  x[i] = make_double2(a.x + v.x, a.y + v.y);
  s[i] = make_double2(0.0, 0.0);
}
int fold(wd_ctx* c, const Field& s, const Field& x) {
  const long n = c->g.Vh;
  if (x.fmt != WD_F64 || (s.fmt != WD_F64 && s.fmt != WD_F32)) return fail(WD_ERR_ARG, "fold: x FP64, s FP32 or FP64");
  if (s.fmt == WD_F32)
    pdl_launch(c, k_fold32, dim3(nblocks(n, BL_THREADS), 6), BL_THREADS, 0, n, (float4*)s.data, (double2*)x.data);
  else
    pdl_launch(c, k_fold64, nblocks(12 * n, BL_THREADS), BL_THREADS, 0, 12 * n, (double2*)s.data, (double2*)x.data);
  WD_CHECK_LAUNCH();
  return WD_OK;
}

// ---------------------------------------------------------------------------
// CG: x += alpha p; r -= alpha Ap; rr = |r|^2 and the scalar logic in the
// last block (beta, stop and reliable-update flags).
__device__ __forceinline__ void cg_update_scalars(CGState* st, double rr) {
  if (!isfinite(rr)) { st->flag |= FLAG_NAN; return; }
  st->rr_old = st->rr;
  st->beta = rr / st->rr;
  st->rr = rr;
  st->iter += 1;
  if (rr <= st->upd_rr) st->flag |= FLAG_UPDATE;
  if (st->iter >= st->maxiter) st->flag |= FLAG_MAXITER;
}
// F: one format for all four fields, word by word; FP32 squares are summed per word
// in FP32, beyond the word in FP64
template <class F>
__global__ void __launch_bounds__(BL_THREADS) k_cg_update(long n, typename Words<F>::W* x, const typename Words<F>::W* p,
                                                          typename Words<F>::W* r, const typename Words<F>::W* ap,
                                                          CGState* st, Reduce red) {
  pdl_enter();
  using Q = Words<F>;
  using T = typename Q::T;
  if (st->flag != 0) return;
  const T al = (T)st->alpha;
  double v[1] = {0.0};
  for (long i = (long)blockIdx.x * BL_THREADS + threadIdx.x; i < n; i += (long)gridDim.x * BL_THREADS) {
    cpx<T> xv[Q::NC], pv[Q::NC], rv[Q::NC], av[Q::NC];
    Q::get(x[i], xv);
    Q::get(ldw(p + i), pv);
    Q::get(r[i], rv);
    Q::get(ldw(ap + i), av);
    T q = 0;
#pragma unroll
    for (int j = 0; j < Q::NC; ++j) {
      xv[j] = mk(fma_t(al, pv[j].r, xv[j].r), fma_t(al, pv[j].i, xv[j].i));
      rv[j] = mk(fma_t(-al, av[j].r, rv[j].r), fma_t(-al, av[j].i, rv[j].i));
      q = fma_t(rv[j].r, rv[j].r, fma_t(rv[j].i, rv[j].i, q));
    }
    x[i] = Q::put(xv);
    r[i] = Q::put(rv);
    v[0] += (double)q;
  }
  double tot[1];
  if (grid_sum<1>(red, v, tot)) cg_update_scalars(st, tot[0]);
}
// 16-bit p (scaled per site) with FP32 x, r, Ap: one 16-byte word of p, two of the others
template <class P>
__global__ void __launch_bounds__(BL_THREADS) k_cg_update16(long Vh, float4* x, P p, float4* r, const float4* ap,
               CGState* st, Reduce red) {
  pdl_enter();
  if (st->flag != 0) return;
  const float al = (float)st->alpha;
  double v[1] = {0.0};
  for (long k = (long)blockIdx.x * BL_THREADS + threadIdx.x; k < 3 * Vh; k += (long)gridDim.x * BL_THREADS) {
    const long j = k >= 2 * Vh ? 2 : (k >= Vh ? 1 : 0), i = k - j * Vh;
    cpx<float> pv[4];
    p.word(i, (int)j, pv);
    float q = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const long e = (2 * j + h) * Vh + i;
      float4 xv = x[e], rv = r[e];
      const float4 av = ldw(ap + e);
      const cpx<float> a = pv[2 * h], b = pv[2 * h + 1];
      xv = make_float4(fmaf(al, a.r, xv.x), fmaf(al, a.i, xv.y), fmaf(al, b.r, xv.z), fmaf(al, b.i, xv.w));
      rv = make_float4(fmaf(-al, av.x, rv.x), fmaf(-al, av.y, rv.y), fmaf(-al, av.z, rv.z), fmaf(-al, av.w, rv.w));
      q = fmaf(rv.x, rv.x, fmaf(rv.y, rv.y, fmaf(rv.z, rv.z, fmaf(rv.w, rv.w, q))));
      x[e] = xv;
      r[e] = rv;
    }
    v[0] += (double)q;
  }
  double tot[1];
  if (grid_sum<1>(red, v, tot)) cg_update_scalars(st, tot[0]);
}

// p = r + beta p, word by word
template <class F>
__global__ void k_cg_pupdate_w(long n, const typename Words<F>::W* r, typename Words<F>::W* p, CGState* st) {
  pdl_enter();
  using Q = Words<F>;
  using T = typename Q::T;
  if (st->flag != 0) return;
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T be = (T)st->beta;
  cpx<T> rv[Q::NC], pv[Q::NC];
  Q::get(ldw(r + i), rv);
  Q::get(p[i], pv);
#pragma unroll
  for (int j = 0; j < Q::NC; ++j) pv[j] = mk(fma_t(be, pv[j].r, rv[j].r), fma_t(be, pv[j].i, rv[j].i));
  p[i] = Q::put(pv);
}
// 16-bit p: the scale of a site is its largest component
template <class T, class R, class P>
__global__ void k_cg_pupdate(long n, R r, P p, CGState* st) {
  pdl_enter();
  if (st->flag != 0) return;
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T be = (T)st->beta;
  cpx<T> rv[12], pv[12];
  r.template loadT<false>(i, rv);
  p.template loadT<false>(i, pv);
#pragma unroll
  for (int j = 0; j < 12; ++j) pv[j] = rv[j] + be * pv[j];
  p.store(i, pv);
}

template <class F>
__global__ void __launch_bounds__(BL_THREADS) k_cg_dot_pap(long n, const typename Words<F>::W* p,
                                                           const typename Words<F>::W* ap, CGState* st, Reduce red) {
  pdl_enter();
  using Q = Words<F>;
  using T = typename Q::T;
  if (st->flag != 0) return;
  double v[1] = {0.0};
  for (long i = (long)blockIdx.x * BL_THREADS + threadIdx.x; i < n; i += (long)gridDim.x * BL_THREADS) {
    cpx<T> pv[Q::NC], av[Q::NC];
    Q::get(ldw(p + i), pv);
    Q::get(ldw(ap + i), av);
    T q = 0;
#pragma unroll
    for (int j = 0; j < Q::NC; ++j) q = fma_t(pv[j].r, av[j].r, fma_t(pv[j].i, av[j].i, q));
    v[0] += (double)q;
  }
  double tot[1];
  if (grid_sum<1>(red, v, tot)) {
    st->pAp = tot[0];
    if (!(tot[0] > 0.0) || !isfinite(tot[0])) st->flag |= FLAG_NAN;
    else st->alpha = st->rr / tot[0];
  }
}

int cg_update(wd_ctx* c, const Field& x, const Field& r, const Field& p, const Field& Ap) {
  const long n = c->g.Vh;
  if (x.fmt != r.fmt || x.fmt != Ap.fmt || (x.fmt != WD_F64 && x.fmt != WD_F32))
    return fail(WD_ERR_ARG, "cg_update: x, r, Ap must share FP64 or FP32");
  if (x.fmt == WD_F64 && p.fmt == WD_F64) {
    const long m = nwords<SpF64>(n);
    pdl_launch(c, k_cg_update<SpF64>, sum_blocks(m), BL_THREADS, 0, m, (double2*)x.data, (const double2*)p.data,
               (double2*)r.data, (const double2*)Ap.data, c->cgs,
               reducer(c));
  } else if (x.fmt == WD_F32 && p.fmt == WD_F32) {
    const long m = nwords<SpF32>(n);
    pdl_launch(c, k_cg_update<SpF32>, sum_blocks(m), BL_THREADS, 0, m, (float4*)x.data, (const float4*)p.data,
               (float4*)r.data, (const float4*)Ap.data, c->cgs,
               reducer(c));
  } else if (x.fmt == WD_F32 && p.fmt == WD_F16) {
    pdl_launch(c, k_cg_update16<Sp16<__half>>, sum_blocks(3 * n), BL_THREADS, 0, n, (float4*)x.data, sp16<__half>(p), (float4*)r.data,
               (const float4*)Ap.data, c->cgs, reducer(c));
  } else if (x.fmt == WD_F32 && p.fmt == WD_BF16) {
    pdl_launch(c, k_cg_update16<Sp16<__nv_bfloat16>>, sum_blocks(3 * n), BL_THREADS, 0, n, (float4*)x.data, sp16<__nv_bfloat16>(p),
               (float4*)r.data, (const float4*)Ap.data, c->cgs,
               reducer(c));
  } else {
    return fail(WD_ERR_ARG, "cg_update: p must be FP64 with FP64 fields, else FP32 or 16-bit");
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

int cg_pupdate(wd_ctx* c, const Field& r, const Field& p) {
  const long n = c->g.Vh;
  if (r.fmt == WD_F64 && p.fmt == WD_F64) {
    const long m = nwords<SpF64>(n);
    pdl_launch(c, k_cg_pupdate_w<SpF64>, nblocks(m, BL_THREADS), BL_THREADS, 0, m, (const double2*)r.data,
               (double2*)p.data, c->cgs);
  } else if (r.fmt == WD_F32 && p.fmt == WD_F32) {
    const long m = nwords<SpF32>(n);
    pdl_launch(c, k_cg_pupdate_w<SpF32>, nblocks(m, BL_THREADS), BL_THREADS, 0, m, (const float4*)r.data,
               (float4*)p.data, c->cgs);
  } else if (r.fmt == WD_F32 && p.fmt == WD_F16) {
    pdl_launch(c, k_cg_pupdate<float, SpF32, Sp16<__half>>, nblocks(n, 128), 128, 0, n, sp32(r), sp16<__half>(p), c->cgs);
  } else if (r.fmt == WD_F32 && p.fmt == WD_BF16) {
    pdl_launch(c, k_cg_pupdate<float, SpF32, Sp16<__nv_bfloat16>>, nblocks(n, 128), 128, 0, n, sp32(r), sp16<__nv_bfloat16>(p), c->cgs);
  } else {
    return fail(WD_ERR_ARG, "cg_pupdate: r must be FP64 or FP32, p of its format or 16-bit");
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

int cg_dot_pap(wd_ctx* c, const Field& p, const Field& Ap) {
  if (p.fmt != Ap.fmt || (p.fmt != WD_F64 && p.fmt != WD_F32))
    return fail(WD_ERR_ARG, "cg_dot_pap: p and Ap must share FP64 or FP32");
  if (p.fmt == WD_F64) {
    const long m = nwords<SpF64>(c->g.Vh);
    pdl_launch(c, k_cg_dot_pap<SpF64>, sum_blocks(m), BL_THREADS, 0, m, (const double2*)p.data, (const double2*)Ap.data,
               c->cgs, reducer(c));
  } else {
    const long m = nwords<SpF32>(c->g.Vh);
    pdl_launch(c, k_cg_dot_pap<SpF32>, sum_blocks(m), BL_THREADS, 0, m, (const float4*)p.data, (const float4*)Ap.data,
               c->cgs, reducer(c));
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

// ---------------------------------------------------------------------------
// Chebyshev recurrence step: out = a (v + mu s - Ks) - b sprev, word by word
template <class F>
__global__ void k_poly_step(long n, typename Words<F>::T a, typename Words<F>::T mu, typename Words<F>::T b,
                            const typename Words<F>::W* v, const typename Words<F>::W* s,
                            const typename Words<F>::W* ks, const typename Words<F>::W* sp, typename Words<F>::W* out) {
  pdl_enter();
  using Q = Words<F>;
  using T = typename Q::T;
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  cpx<T> vv[Q::NC], sv[Q::NC], kv[Q::NC], pv[Q::NC];
  Q::get(ldw(v + i), vv);
  Q::get(ldw(s + i), sv);
  Q::get(ldw(ks + i), kv);
  Q::get(ldw(sp + i), pv);
#pragma unroll
  for (int j = 0; j < Q::NC; ++j) vv[j] = a * (vv[j] + mu * sv[j] - kv[j]) - b * pv[j];
  out[i] = Q::put(vv);
}

template <class F>
static void poly_step_words(wd_ctx* c, double a, double mu, double b, const Field& v, const Field& s, const Field& Ks,
                            const Field& sprev, const Field& out) {
  using T = typename Words<F>::T;
  using W = typename Words<F>::W;
  const long m = nwords<F>(c->g.Vh);
  pdl_launch(c, k_poly_step<F>, nblocks(m, BL_THREADS), BL_THREADS, 0, m, T(a), T(mu), T(b), (const W*)v.data,
               (const W*)s.data, (const W*)Ks.data,
               (const W*)sprev.data, (W*)out.data);
}
int poly_step(wd_ctx* c, double a, double mu, double b, const Field& v, const Field& s,
              const Field& Ks, const Field& sprev, const Field& out) {
  switch (v.fmt) {
    case WD_F64: poly_step_words<SpF64>(c, a, mu, b, v, s, Ks, sprev, out); break;
    case WD_F32: poly_step_words<SpF32>(c, a, mu, b, v, s, Ks, sprev, out); break;
    case WD_DD: poly_step_words<SpDD>(c, a, mu, b, v, s, Ks, sprev, out); break;
    default: return fail(WD_ERR_ARG, "poly_step: FP64, FP32 or double-float fields only");
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

}  // namespace wd
