// Layout kernels: lexicographic host-order fields <-> even-odd structure-of-
// arrays device fields, and the FP32 link copies derived from the FP64 links.
#include "dslash_impl.cuh"

namespace wd {

// Lexicographic field: W elements of C doubles per site, W = nouter x nchunk
// (outer index = mu or nothing).  EO field: [outer][parity][nchunk][Vh] elements
// when parity < 0 (both parities), or [nchunk][Vh] for one parity.
//
// A block moves PACK_S consecutive lexicographic sites through shared memory: the
// lexicographic side is then one contiguous run, the EO side runs of PACK_S / 2
// elements (sites 2k and 2k + 1 share checkerboard index k), so both are
// coalesced.  One site per thread left the lexicographic side at a stride of a
// whole site (576 bytes for links).  Links at 32^3 x 64: pack 0.69 -> 0.46 ms, unpack
// 1.97 -> 0.44 ms (2.4 GB, 0.36 ms at the copy peak).
// The lexicographic side needs 8-byte alignment only; VEC: elements of the EO side
// move as 16-byte words.
// The shapes are compile-time constants: with run-time divisors the index arithmetic of
// algebra fields, whose elements are one double, cost more than the old strides at
// some sizes.  Algebra pack / unpack in us, one site per thread, run-time shapes, constants: 16^3 x 32
// 23.1 / 23.1, 24.9 / 25.7, 13.2 / 14.8; 18 x 22 x 20 x 26 34.7 / 36.5, 37.2 / 39.6, 23.2 / 25.1;
// 24^3 x 48 138 / 240, 107 / 112, 66 / 70.  Links 16^3 x 32 with the FP32 copies 62.0, 59.7, 51.9.
constexpr int PACK_S = 64, PACK_THREADS = 256;
constexpr int pack_pitch(int d, int c) { return d + (c == 2 ? 2 : 1 - (d & 1)); }   // doubles of a site in shared memory

template <int C, int NOUTER, int NCHUNK, bool VEC, bool UNPACK>
__global__ void __launch_bounds__(PACK_THREADS) k_pack(Geom g, int parity, const double* src, double* dst) {
  extern __shared__ double2 pack_sh[];
  double* sh = reinterpret_cast<double*>(pack_sh);   // [PACK_S][P]
  constexpr int W = NOUTER * NCHUNK, D = W * C, P = pack_pitch(D, C);
  const long lex0 = (long)blockIdx.x * PACK_S;
  const int n = (int)(g.V - lex0 < PACK_S ? g.V - lex0 : PACK_S), half = n / 2;   // V is even
  const int npar = parity >= 0 ? 1 : 2;
  // which of the sites 2k, 2k + 1 of this block has the parity
  auto site_of = [&](int k, int par) -> int {
    const unsigned r = (unsigned)((lex0 >> 1) + k);
    const unsigned r0 = g.dx.div(r), r1 = g.dy.div(r0), r2 = g.dz.div(r1);
    const int p0 = (int)((r0 - r1 * g.dy.d) + (r1 - r2 * g.dz.d) + r2) & 1;   // parity of the site with even x
    return 2 * k + (p0 != par ? 1 : 0);
  };
  if constexpr (!UNPACK) {
    for (int e = threadIdx.x; e < n * D; e += PACK_THREADS) {
      const int s = e / D;
      sh[s * P + (e - s * D)] = src[lex0 * D + e];
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < npar * W * half; e += PACK_THREADS) {
    const int q = half == PACK_S / 2 ? e / (PACK_S / 2) : e / half, k = e - q * half;
    const int p = q / W, w = q - p * W;
    const int par = parity >= 0 ? parity : p;
    const int o = w / NCHUNK, j = w - o * NCHUNK;
    const long base = parity >= 0 ? w : (long)(o * 2 + par) * NCHUNK + j;
    const long eo = (base * g.Vh + (lex0 >> 1) + k) * C;
    double* at = sh + site_of(k, par) * P + w * C;
    if constexpr (VEC) {
      if constexpr (UNPACK) *reinterpret_cast<double2*>(at) = *reinterpret_cast<const double2*>(src + eo);
      else *reinterpret_cast<double2*>(dst + eo) = *reinterpret_cast<const double2*>(at);
    } else {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if constexpr (UNPACK) at[c] = src[eo + c];
        else dst[eo + c] = at[c];
      }
    }
  }
  if constexpr (UNPACK) {
    __syncthreads();
    if (parity < 0) {
      for (int e = threadIdx.x; e < n * D; e += PACK_THREADS) {
        const int s = e / D;
        dst[lex0 * D + e] = sh[s * P + (e - s * D)];
      }
    } else {   // sites of the other parity are left as they are
      for (int e = threadIdx.x; e < half * D; e += PACK_THREADS) {
        const int k = e / D, s = site_of(k, parity);
        dst[(lex0 + s) * D + (e - k * D)] = sh[s * P + (e - k * D)];
      }
    }
  }
}

template <int C, int NOUTER, int NCHUNK, bool VEC>
static void pack_launch(wd_ctx* c, bool unpack, int parity, const double* src, double* dst) {
  constexpr size_t sm = sizeof(double) * PACK_S * pack_pitch(NOUTER * NCHUNK * C, C);   // links: 37.9 KB
  const int nb = (int)((c->g.V + PACK_S - 1) / PACK_S);
  if (unpack) k_pack<C, NOUTER, NCHUNK, VEC, true><<<nb, PACK_THREADS, sm, c->stream>>>(c->g, parity, src, dst);
  else k_pack<C, NOUTER, NCHUNK, VEC, false><<<nb, PACK_THREADS, sm, c->stream>>>(c->g, parity, src, dst);
}

int pack_k(wd_ctx* c, bool unpack, int nouter, int nchunk, int chunk, int parity, const double* src,
           double* dst) {
  const bool aligned = ((uintptr_t)(unpack ? src : dst) & 15) == 0;   // the EO side
  if (nouter == 4 && nchunk == 9 && chunk == 2) {            // links
    if (aligned) pack_launch<2, 4, 9, true>(c, unpack, parity, src, dst);
    else pack_launch<2, 4, 9, false>(c, unpack, parity, src, dst);
  } else if (nouter == 1 && nchunk == 12 && chunk == 2) {    // spinors
    if (aligned) pack_launch<2, 1, 12, true>(c, unpack, parity, src, dst);
    else pack_launch<2, 1, 12, false>(c, unpack, parity, src, dst);
  } else if (nouter == 4 && nchunk == 8 && chunk == 1) {     // algebra fields
    pack_launch<1, 4, 8, false>(c, unpack, parity, src, dst);
  } else {
    return fail(WD_ERR_ARG, "pack: unknown field shape");
  }
  WD_CHECK_LAUNCH();
  return WD_OK;
}

__global__ void k_gauge_lowprec(long n9, long Vh, const double2* U64, float2* U32, float4* U12, float4* Udd) {
  // one thread per link (mu, parity, cb): n = 8 Vh
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n9) return;
  const long mp = i / Vh, cb = i % Vh;
  const double2* u = U64 + mp * 9 * Vh + cb;
  double2 v[9];
#pragma unroll
  for (int j = 0; j < 9; ++j) v[j] = u[j * Vh];
  if (Udd != nullptr) {
    float4* o = Udd + mp * 9 * Vh + cb;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      const dd r(v[j].x), m(v[j].y);
      o[j * Vh] = make_float4(r.hi, r.lo, m.hi, m.lo);
    }
  }
  float2* o = U32 + mp * 9 * Vh + cb;
#pragma unroll
  for (int j = 0; j < 9; ++j) o[j * Vh] = make_float2((float)v[j].x, (float)v[j].y);
  float4* q = U12 + mp * 3 * Vh + cb;
#pragma unroll
  for (int j = 0; j < 3; ++j)
    q[j * Vh] = make_float4((float)v[2 * j].x, (float)v[2 * j].y, (float)v[2 * j + 1].x, (float)v[2 * j + 1].y);
}

int gauge_lowprec_k(wd_ctx* c) {
  const long n = 8 * c->g.Vh;
  links_written(c);
  k_gauge_lowprec<<<nblocks(n, 128), 128, 0, c->stream>>>(n, c->g.Vh, c->gauge64, c->gauge32, c->gauge32r12,
                                                          c->gauge_dd);
  WD_CHECK_LAUNCH();
  return WD_OK;
}

}  // namespace wd
