// BF16 spinors: see dslash_h16.cuh
#include "dslash_h16.cuh"

namespace wd {

int hop_bf16(wd_ctx* c, int out_par, bool dag, const Field& in, const Field& out, const Field* y,
             double alpha, bool norm_cg, bool in_cg) {
  return hop_h<__nv_bfloat16>(c, out_par, dag, in, out, y, alpha, norm_cg, in_cg);
}

}  // namespace wd
