// FP64 instantiations of the hopping stencil (double storage, double arithmetic):
// eight threads per site (dslash_split.cuh), on large lattices one.
#include "dslash_split.cuh"

namespace wd {

int hop_f64(wd_ctx* c, int out_par, bool dag, const Field& in, const Field& out, const Field* y,
            double alpha, bool norm_cg, bool in_cg) {
  if (in.fmt != WD_F64 || out.fmt != WD_F64 || (y && y->fmt != WD_F64))
    return fail(WD_ERR_ARG, "hop_f64: field formats must all be FP64");
  SpF64 I = sp64(in), O = sp64(out), Y = y ? sp64(*y) : O;
  if (split_eligible(c, true)) {
    HopArgs<SpF64, SpF64, SpF64, GF64> a{c->g, out_par, I, O, Y, GF64{c->gauge64, c->g.Vh}, alpha, reducer(c),
                                         (norm_cg || in_cg) ? c->cgs : nullptr};
    return hop_split<double>(c, dag, y != nullptr, norm_cg, a);
  }
  return hop_with_gauge<double>(c, out_par, dag, I, O, Y, y != nullptr, alpha, norm_cg, in_cg, true);
}

}  // namespace wd
