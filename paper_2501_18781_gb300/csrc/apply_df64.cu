// df64 instantiation of the apply kernels.
#include "apply_kernels.cuh"

namespace mf {

mf_status launch_scalar_apply_df64(mf_ctx* ctx, const mf_dofmap* m, int kind, int mode, bool beta, bool tr,
                                   const ScalarArgs<double>& a) {
  return dispatch_scalar<df64>(ctx, m, kind, mode, beta, tr, a);
}

}  // namespace mf
