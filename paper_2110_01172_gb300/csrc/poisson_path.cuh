// poisson_path.cuh - the fused Poisson solve of the two-pass family (used by
// gbdct_poisson.cu): the forward transform, then the three inverses as one
// batch that reads the one spectrum and scales it on the way in.
#pragma once

#include <cuda_runtime.h>

#include "../../include/gbdct.h"

namespace gbdct {

// A DCT-II plan whose workspace holds the three inverses; UNSUPPORTED where the
// two-pass family does not apply (sides outside 64..8192, or another family
// forced).  Released with gbdct_plan_destroy.
gbdct_status poisson_plan_create(gbdct_plan_t* out, const int64_t* dims);

// rho -> out = {psi, xi0, xi1}; w: wu[n1], wv[n2]; inv: 1 / (wu^2 + wv^2).
gbdct_status poisson_plan_solve(gbdct_plan_t p, const void* rho, void* const* out, const float* w, const float* inv,
                                cudaStream_t s);

}  // namespace gbdct
