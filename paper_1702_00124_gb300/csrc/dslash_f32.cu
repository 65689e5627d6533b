// FP32 instantiations of the hopping stencil (float storage and arithmetic,
// FP32 links with 18 or 12 stored reals).
#include "dslash_tt.cuh"

namespace wd {

// whether hop_f32 can store FP64 (the tile-staged option cannot)
bool hop_widens(wd_ctx* c) { return !(c->recon == WD_RECON_12 && tt_eligible(c)); }

int hop_f32(wd_ctx* c, int out_par, bool dag, const Field& in, const Field& out, const Field* y,
            double alpha, bool norm_cg, bool in_cg) {
  if (in.fmt != WD_F32 || (out.fmt != WD_F32 && out.fmt != WD_F64) || (y && y->fmt != WD_F32))
    return fail(WD_ERR_ARG, "hop_f32: input and y must be FP32, the output FP32 or FP64");
  SpF32 I = sp32(in), Y = y ? sp32(*y) : I;
  if (out.fmt == WD_F64) {   // the FP32 result widened as it is stored: the last hop of an operator call
    if (!hop_widens(c) || norm_cg) return fail(WD_ERR_ARG, "hop_f32: no FP64 output on this path");
    return hop_links(c, out_par, dag, I, sp64(out), Y, y != nullptr, alpha, norm_cg, in_cg);
  }
  SpF32 O = sp32(out);
  if (c->recon == WD_RECON_12 && tt_eligible(c))
    return hop_tt(c, out_par, dag, I, O, Y, y != nullptr, alpha, norm_cg, in_cg);
  return hop_links(c, out_par, dag, I, O, Y, y != nullptr, alpha, norm_cg, in_cg);
}

// Self-test of the bounded barrier wait: thread 0 waits on a freshly
// initialised mbarrier that nothing arrives at; the wait expires after ns and
// the kernel records it in the device error word and returns.
__global__ void k_wait_selftest(unsigned* kerr, long long ns) {
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait_ns(&bar, 0u, ns)) atomicOr(kerr, 1u);
}

int wait_selftest(wd_ctx* c, long long ns) {
  if (c->kerr == nullptr) return fail(WD_ERR_STATE, "no device error word");
  k_wait_selftest<<<1, 32, 0, c->stream>>>(c->kerr, ns);
  WD_CHECK_LAUNCH();
  return WD_OK;
}

template <int EPI, class G>
static void hop_poly(wd_ctx* c, const G& gauge, double alpha, const Field& in, const Field& y, const Field& out,
                     const HopPoly& pe) {
  const HopArgs<SpF32, SpF32, SpF32, G> a{c->g, 0, sp32(in), sp32(out), sp32(y), gauge, alpha, reducer(c), nullptr};
  if (split_eligible(c, WD_F32))
    pdl_launch(c, k_hop_split<float, true, EPI, false, SpF32, SpF32, SpF32, G>, nblocks(c->g.Vh, SPL_SITES), SPL_THREADS,
               0, a, pe);
  else
    hop_st_depth<true, EPI, false>(c, a, pe);
}
template <int EPI>
static int hop_poly_links(wd_ctx* c, double alpha, const Field& in, const Field& y, const Field& out, const HopPoly& pe) {
  if (c->recon == WD_RECON_12) hop_poly<EPI>(c, GF32R12{c->gauge32r12, c->g.Vh}, alpha, in, y, out, pe);
  else hop_poly<EPI>(c, GF32{c->gauge32, c->g.Vh}, alpha, in, y, out, pe);
  WD_CHECK_LAUNCH();
  c->prof.all[WD_F32] += 1;
  return WD_OK;
}

// whether hop_shift is one launch on fields of the format (it takes a vector of its own if not)
bool hop_shift_fused(wd_ctx* c, int fmt) { return fmt == WD_F32 && hop_widens(c); }   // not the tile-staged option

// out = y + alpha D^dag_eo in + z v, the last hop of a factor (K_hat + z) v; out may be v
int hop_shift(wd_ctx* c, const Field& in, const Field& y, double alpha, double zr, double zi, const Field& v,
              const Field& out) {
  if (hop_shift_fused(c, in.fmt)) {
    const Field* fields[] = {&y, &v, &out};
    for (const Field* f : fields)
      if (f->fmt != WD_F32) return fail(WD_ERR_ARG, "hop_shift: formats differ");
    cudaEvent_t e0 = nullptr;
    prof_begin(c, &e0);
    WD_TRY(hop_poly_links<3>(c, alpha, in, y, out, HopPoly{sp32(v), sp32(v), sp32(v), (float)zr, 0.f, (float)zi}));
    // the hop's bytes and v
    const double v_bytes = 96.0 * (double)c->g.Vh;
    prof_end(c, e0, hop_bytes(WD_F32, WD_F32, true, c->recon == WD_RECON_12 ? 48 : 72, c->g.Vh) + v_bytes, WD_F32);
    return WD_OK;
  }
  WsGuard w(c);
  Field k;
  WD_TRY(w.get(in.fmt, &k));
  WD_TRY(hop(c, 0, true, in, k, &y, alpha, false, false));
  return caxpby(c, 1.0, 0.0, k, zr, zi, v, out);
}

// out = ca (v + cmu s - K_hat s) - cb sprev for FP32 fields (t1, t2 scratch)
int khat_poly_step_f32(wd_ctx* c, double kappa, const Field& s, Field& t1, Field& t2, const Field& v,
                       const Field& sprev, double ca, double cmu, double cb, const Field& out) {
  const Field* fields[] = {&s, &t1, &t2, &v, &sprev, &out};
  for (const Field* f : fields)
    if (f->fmt != WD_F32) return fail(WD_ERR_ARG, "khat_poly_step_f32: FP32 fields only");
  const double a2 = -kappa * kappa;
  WD_TRY(hop(c, 1, false, s, t1, nullptr, 0.0, false, false));
  WD_TRY(hop(c, 0, false, t1, t2, &s, a2, false, false));
  WD_TRY(hop(c, 1, true, t2, t1, nullptr, 0.0, false, false));
  const HopPoly hp{sp32(v), sp32(s), sp32(sprev), (float)ca, (float)cmu, (float)cb};
  if (c->recon == WD_RECON_12 && tt_eligible(c)) {
    HopArgs<SpF32, SpF32, SpF32, GF32R12> a{c->g, 0, sp32(t1), sp32(out), sp32(t2), GF32R12{c->gauge32r12, c->g.Vh},
                                            a2, reducer(c), nullptr};
    const TTPoly pe{sp32(v), sp32(s), sp32(sprev), (float)ca, (float)cmu, (float)cb};
    const Field* chk[] = {&t1, &t2, &v, &s, &sprev};
    for (const Field* f : chk)
      if (((uintptr_t)f->data & 15) != 0) return fail(WD_ERR_ARG, "khat_poly_step_f32: fields must be 16-byte aligned");
    WD_TRY((tt_launch<true, 2, false>(c, a, pe)));
    c->prof.all[WD_F32] += 1;
  } else {
    WD_TRY(hop_poly_links<2>(c, a2, t1, t2, out, hp));
  }
  c->nmat += 1;
  return WD_OK;
}

}  // namespace wd
