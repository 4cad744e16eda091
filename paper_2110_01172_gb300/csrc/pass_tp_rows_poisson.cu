// pass_tp_rows_poisson.cu - inverse row pass of a Poisson solve: the three
// inverses of one spectrum as one batch.
#include "tp_rows_poisson_launch.cuh"

namespace gbdct {
namespace {

template <int L>
cudaError_t launch(const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  return launch_e<L, false>(a, ps, s, prepare);
}

}  // namespace

cudaError_t run_tp_rows_poisson(int lg2, const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  if (a.exact) return run_tp_rows_poisson_exact(lg2, a, ps, s, prepare);
  GBDCT_TP_ROWS_SWITCH(lg2, launch, a, ps, s, prepare);
}

}  // namespace gbdct
