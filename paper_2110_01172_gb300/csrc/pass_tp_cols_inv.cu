// pass_tp_cols_inv.cu - inverse column pass of the two-pass family.
#include "tp_cols_launch.cuh"

namespace gbdct {

cudaError_t run_tp_cols_inv(int lg1, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  return col_run<true, false>(lg1, a, PoissonArgs{}, batch, s, prepare);
}

}  // namespace gbdct
