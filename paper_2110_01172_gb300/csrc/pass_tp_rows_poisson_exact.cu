// pass_tp_rows_poisson_exact.cu - inverse row pass of a Poisson solve: the three
// inverses of one spectrum as one batch:
// its exact kernels (Dct2dArgs::exact).
#include "tp_rows_poisson_launch.cuh"

namespace gbdct {
namespace {

template <int L>
cudaError_t launch(const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  return launch_e<L, true>(a, ps, s, prepare);
}

}  // namespace

cudaError_t run_tp_rows_poisson_exact(int lg2, const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  GBDCT_TP_ROWS_SWITCH(lg2, launch, a, ps, s, prepare);
}

}  // namespace gbdct
