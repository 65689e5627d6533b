// FP64 instantiations of the hopping stencil (double storage, double arithmetic):
// eight threads per site (dslash_split.cuh), on large lattices one.
#include "dslash_split.cuh"

namespace wd {

int hop_f64(wd_ctx* c, int out_par, bool dag, const Field& in, const Field& out, const Field* y,
            double alpha, bool norm_cg, bool in_cg) {
  if (in.fmt != WD_F64 || out.fmt != WD_F64 || (y && y->fmt != WD_F64))
    return fail(WD_ERR_ARG, "hop_f64: field formats must all be FP64");
  SpF64 I = sp64(in), O = sp64(out), Y = y ? sp64(*y) : O;
  HopArgs<SpF64, SpF64, SpF64, GF64> a{c->g, out_par, I, O, Y, GF64{c->gauge64, c->g.Vh}, alpha, reducer(c),
                                       (norm_cg || in_cg) ? c->cgs : nullptr};
  if (split_eligible(c, WD_F64)) return hop_split<double>(c, dag, y != nullptr, norm_cg, a);
  // tuning key: formats of in / out / y and the link storage (0: FP64)
  const long long key = (((long long)WD_F64 * 8 + WD_F64) * 8 + (y ? WD_F64 : 7)) * 4;
  return launch_hop<double>(c, dag, y != nullptr, norm_cg, key, !in_cg, a);
}

}  // namespace wd
