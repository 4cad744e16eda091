// gemm_path.cuh - the split-BF16 DFT-GEMM precision mode of a 2D plan.
//
// The separable definition X = C1 x C2^T (Eq. 2d-dct-definition; C[k, j] =
// cos(pi k (2j+1) / 2N)) and its inverse x = D1 X D2^T (D = (2/N) C^T diag(w),
// w_0 = 1/2) evaluated as dense products on the tensor cores.  Because C[k, N-1-j]
// = (-1)^k C[k, j], an axis of length N needs two products of half its size
// instead of one: the even frequencies from the sums x_j + x_{N-1-j}, the odd
// ones from the differences (the inverse: the sum and difference of the two
// products).  Over both axes a transform is four quadrants (parity p1, p2) and
// half of the operations and operand bytes of the full products.  What bounds the
// products at 1024^2 is latency: 128 tiles for 152 SMs, eight blocks of K each, the
// epilogue behind the last of them (11.4 us a product by ncu; tensor pipe 22 % of a
// busy SM's cycles, L2 throughput 9 %, warps waiting for tensor memory and stores).
//
// Every operand v is split into bf16 parts hi = bf16(v), lo = bf16(v - hi), and
// each product A B is accumulated in FP32 as hi_A hi_B + hi_A lo_B + lo_A hi_B +
// lo_A lo_B.  The matrices are generated in FP64 from integer-reduced angles and
// split once.  Launches of a call: the input quadrants (sums or entries by
// parity) split into bf16, the product along axis 1 (its epilogue stores the
// intermediate split and transposed as the second product's operand), the
// product along axis 0, and for the inverse the mirror sums; consecutive
// launches overlap through programmatic dependent launch (launch_dep.cuh).
// Both products run in the hand-written tcgen05 kernel of tc_gemm.cuh.  The
// error is that of the split (about 5e-6 relative in L2), stated per result by
// the tests rather than held to the FP32 tolerance.
//
// Measured against full-size products with three of the four terms, forward /
// inverse: 1024^2 33.7 / 33.6 -> 21.1 / 23.2 us, 2048^2 128 / 128 -> 74.5 / 77.6,
// 64 x 256^2 38.5 / 38.3 -> 26.3 / 28.8; forward error against the FP32 path
// 128^2 5.3e-6 -> 4.6e-6, 1024^2 8.1e-6 -> 6.2e-6, 2048^2 1.36e-5 -> 9.6e-6.  The fourth
// term costs 1.4 us at 1024^2; without it the split of the sums is 4 % less
// exact than that of the values themselves.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/gbdct.h"

namespace gbdct {

struct GemmPath;

// kGemmMinSide <= n1, n2 <= kGemmMaxSide (powers of two); batch transforms
// stored back to back.  `err` is the plan's device error word (bounded waits
// that gave up set it).
constexpr int kGemmMinSide = 128;
constexpr int kGemmMaxSide = 2048;
GemmPath* gemm_create(int n1, int n2, int batch, int* err, gbdct_status* st);
// Bound (polls) of every device-side wait of the kernels; 0 restores the default.
void gemm_set_wait_polls(GemmPath* g, uint32_t polls);
gbdct_status gemm_exec(GemmPath* g, bool inverse, const float* in, float* out, cudaStream_t s);
size_t gemm_workspace_bytes(const GemmPath* g);
void gemm_destroy(GemmPath* g);

}  // namespace gbdct
