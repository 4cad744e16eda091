// tp_rows_launch.cuh - launch rules of the two-pass family's row passes, shared
// by the translation units of the forward, the inverse and the Poisson row pass.
#pragma once

#include "dct2d_launch.cuh"
#include "dct2d_tp_kernels.cuh"

namespace gbdct {

// Narrow (64-thread) CTAs when wide ones would give fewer than two CTAs per SM.
template <int L>
bool tp_rows_narrow(const Dct2dArgs& a, int batch) {
  const long long wide_ctas = (long long)(a.n1 / 4 / TpRows<L, false>::NP) * batch;
  return wide_ctas < 2LL * (a.nsm > 0 ? a.nsm : 1) && (a.n1 / 4) % TpRows<L, true>::NP == 0;
}

// Raises a kernel's dynamic shared-memory limit where it needs more than the default.
inline cudaError_t tp_smem_limit(const void* kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// FN<L>(args...) for L = 2^lg2, 64 .. 8192.
#define GBDCT_TP_ROWS_SWITCH(lg2, FN, ...)  \
  switch (lg2) {                            \
    case 6: return FN<64>(__VA_ARGS__);     \
    case 7: return FN<128>(__VA_ARGS__);    \
    case 8: return FN<256>(__VA_ARGS__);    \
    case 9: return FN<512>(__VA_ARGS__);    \
    case 10: return FN<1024>(__VA_ARGS__);  \
    case 11: return FN<2048>(__VA_ARGS__);  \
    case 12: return FN<4096>(__VA_ARGS__);  \
    case 13: return FN<8192>(__VA_ARGS__);  \
  }                                         \
  return cudaErrorInvalidValue

}  // namespace gbdct
