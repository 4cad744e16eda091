// pass_tp_cols_poisson.cu - column pass of a Poisson solve's three inverses.
#include "tp_cols_launch.cuh"

namespace gbdct {

cudaError_t run_tp_cols_poisson(int lg1, const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  return col_run<true, true>(lg1, a, ps, 3, s, prepare);
}

}  // namespace gbdct
