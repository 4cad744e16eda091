// pass_small_inv.cu - inverse small transforms, one CTA and one launch each.
#include "dct2d_launch.cuh"
#include "dct2d_small.cuh"

namespace gbdct {
namespace {

template <int LG1, int LG2>
cudaError_t launch(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  if constexpr (LG1 + LG2 > kSmallMaxLog2) {
    return cudaErrorInvalidValue;
  } else {
    using G = SmallGeom<LG1, LG2>;
    const auto k = k_small<LG1, LG2, true>;
    if (prepare && G::SMEM <= 48 * 1024) return cudaSuccess;  // within the default limit
    if (prepare)
      return cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)G::SMEM);
    return pdl::launch(k, dim3((batch + G::NT - 1) / G::NT), dim3(G::THREADS), G::SMEM, s, a, batch);
  }
}

template <int LG1>
cudaError_t launch_rows(int lg2, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  switch (lg2) {
    case 5: return launch<LG1, 5>(a, batch, s, prepare);
    case 6: return launch<LG1, 6>(a, batch, s, prepare);
    case 7: return launch<LG1, 7>(a, batch, s, prepare);
    case 8: return launch<LG1, 8>(a, batch, s, prepare);
    case 9: return launch<LG1, 9>(a, batch, s, prepare);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t run_small_inv(int lg1, int lg2, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  switch (lg1) {
    case 5: return launch_rows<5>(lg2, a, batch, s, prepare);
    case 6: return launch_rows<6>(lg2, a, batch, s, prepare);
    case 7: return launch_rows<7>(lg2, a, batch, s, prepare);
    case 8: return launch_rows<8>(lg2, a, batch, s, prepare);
    case 9: return launch_rows<9>(lg2, a, batch, s, prepare);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbdct
