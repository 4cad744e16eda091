// pass_tp_cols_fwd.cu - forward column pass of the two-pass family (half-length column
// FFTs of the even and odd reordered rows).
#include "tp_cols_launch.cuh"

namespace gbdct {

cudaError_t run_tp_cols_fwd(int lg1, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  return col_run<false, false>(lg1, a, PoissonArgs{}, batch, s, prepare);
}

}  // namespace gbdct
