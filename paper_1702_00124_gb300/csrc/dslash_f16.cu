// FP16 spinors: see dslash_h16.cuh
#include "dslash_h16.cuh"

namespace wd {

int hop_f16(wd_ctx* c, int out_par, bool dag, const Field& in, const Field& out, const Field* y,
            double alpha, bool norm_cg, bool in_cg) {
  return hop_h<__half>(c, out_par, dag, in, out, y, alpha, norm_cg, in_cg);
}

}  // namespace wd
