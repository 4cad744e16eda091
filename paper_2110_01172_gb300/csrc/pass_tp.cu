// pass_tp.cu - whole transforms of the two-pass family (forward: column pass, row
// pass; inverse: row pass, column pass).
#include "dct2d_launch.cuh"

namespace gbdct {

cudaError_t run_tp(int lg1, int lg2, bool inverse, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  if (prepare) {
    cudaError_t e = run_tp_rows_fwd(lg2, a, batch, s, true);
    if (e == cudaSuccess) e = run_tp_rows_inv(lg2, a, batch, s, true);
    if (e == cudaSuccess) e = run_tp_cols_fwd(lg1, a, batch, s, true);
    if (e == cudaSuccess) e = run_tp_cols_inv(lg1, a, batch, s, true);
    return e;
  }
  const int f = a.step_filter;
  cudaError_t e = cudaSuccess;
  if (!inverse) {
    if (f < 0 || f == 0) e = run_tp_cols_fwd(lg1, a, batch, s, false);
    if (e == cudaSuccess && (f < 0 || f == 1)) e = run_tp_rows_fwd(lg2, a, batch, s, false);
  } else {
    if (f < 0 || f == 0) e = run_tp_rows_inv(lg2, a, batch, s, false);
    if (e == cudaSuccess && (f < 0 || f == 1)) e = run_tp_cols_inv(lg1, a, batch, s, false);
  }
  return e;
}

cudaError_t run_tp_poisson(int lg1, int lg2, const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  cudaError_t e = run_tp_rows_poisson(lg2, a, ps, s, prepare);
  if (e == cudaSuccess) e = run_tp_cols_poisson(lg1, a, ps, s, prepare);
  return e;
}

}  // namespace gbdct
