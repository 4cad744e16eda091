// tp_cols_launch.cuh - launches of the two-pass family's column passes, shared by
// the translation units of the forward, the inverse and the Poisson column pass.
#pragma once

#include "dct2d_launch.cuh"
#include "dct2d_tp_kernels.cuh"

namespace gbdct {

// Tensor maps of the bulk-copy column pass: mx over the input (forward) or
// output (inverse) viewed as (x, row % 4, row / 4, batch), mw over the
// workspace (x, row, batch); boxes of 4 NP floats x ZB rows.
// N = 3 (the inverses of a Poisson solve): one map per output array.
template <int N>
bool encode_maps(const Dct2dArgs& a, const PoissonArgs& ps, int batch, bool inverse, int np, int zb, ColMaps<N>* maps) {
  const PFN_cuTensorMapEncodeTiled_v12000 fn = tma::encoder();
  if (!fn) return false;
  const cuuint64_t n1 = (cuuint64_t)a.n1, n2 = (cuuint64_t)a.n2;
  const cuuint64_t dx[4] = {n2, 4, n1 / 4, N == 3 ? 1 : (cuuint64_t)batch};
  const cuuint64_t sx[3] = {n2 * 4, 16 * n2, (cuuint64_t)(inverse ? a.out_bstride : a.in_bstride) * 4};
  const cuuint32_t bx[4] = {(cuuint32_t)(4 * np), 1, (cuuint32_t)zb, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  for (int i = 0; i < N; ++i) {
    void* xp = N == 3 ? ps.out[i] : inverse ? static_cast<void*>(a.out) : const_cast<float*>(a.in);
    if (fn(&maps->x[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, xp, dx, sx, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
           CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return false;
  }
  const cuuint64_t dw[3] = {n2, n1, (cuuint64_t)batch};
  const cuuint64_t sw[2] = {n2 * 4, (cuuint64_t)a.work_bstride * 8};
  const cuuint32_t bw[3] = {(cuuint32_t)(4 * np), (cuuint32_t)zb, 1};
  return fn(&maps->w, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, a.work, dw, sw, bw, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

template <int M, int NP, bool INV, bool POIS, bool EXACT>
cudaError_t col_launch_k(const Dct2dArgs& a, const PoissonArgs& ps, int batch, cudaStream_t s, bool prepare) {
  using G = TpColGeom<M, NP>;
  if (prepare) {
    if (G::SMEM_TMA <= 48 * 1024) return cudaSuccess;  // within the default limit
    cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k_tp_cols<M, NP, INV, POIS, EXACT>),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k_tp_cols_tma<M, NP, INV, POIS, EXACT>),
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM_TMA);
    return e;
  }
  const dim3 grid(a.n2 / 4 / NP, 2, batch);
  const bool overlap = INV || pdl::gains_from_overlap(2LL * grid.x * batch, a.nsm);
  // bulk tensor copies for device buffers; per-thread loads / stores for
  // host-mapped or managed buffers
  ColMaps<POIS ? 3 : 1> maps;
  if (a.io_dev && encode_maps(a, ps, batch, INV, NP, G::ZB, &maps))
    return pdl::launch_if(overlap, k_tp_cols_tma<M, NP, INV, POIS, EXACT>, grid, dim3(G::THREADS), G::SMEM_TMA, s, a, maps);
  return pdl::launch_if(overlap, k_tp_cols<M, NP, INV, POIS, EXACT>, grid, dim3(G::THREADS), G::SMEM, s, a, ps);
}

// The strip width: the plan's choice, else the default for M, halved (down
// to two column pairs and 64 threads) while the grid would give fewer than
// two CTAs per SM (a single transform with few columns, e.g. 1024^2), and
// never wider than the array.
template <int M>
int strip_np(const Dct2dArgs& a, int batch) {
  if (a.tpNP) return a.tpNP;
  int np = tp_default_np(M);
  while (np > a.n2 / 4) np /= 2;
  const long long nsm = a.nsm > 0 ? a.nsm : 1;
  while (np > 2 && (np / 2) * fft_tps(M) >= 64 && (long long)(a.n2 / 4 / np) * 2 * batch < 2 * nsm) np /= 2;
  return np;
}

// One width of one direction; the widths not built for M are INVALID_VALUE.
template <int M, int NP, bool INV, bool POIS>
cudaError_t col_width(const Dct2dArgs& a, const PoissonArgs& ps, int batch, cudaStream_t s, bool prepare) {
  using G = TpColGeom<M, NP>;
  if constexpr (POIS ? !G::POISSON : !G::VALID) {
    return cudaErrorInvalidValue;
  } else {
    if (!prepare && (a.n2 / 4) % NP) return cudaErrorInvalidValue;
    // exact plans with M > 32 have N2 = 64 (a stage of radix 2, M = 32, is exact anyway)
    if constexpr (M > 32 && NP <= 16 && G::POISSON)
      if (a.exact) return col_launch_k<M, NP, INV, POIS, true>(a, ps, batch, s, prepare);
    return a.exact && M > 32 ? cudaErrorInvalidValue : col_launch_k<M, NP, INV, POIS, false>(a, ps, batch, s, prepare);
  }
}

template <int M, bool INV, bool POIS>
cudaError_t col_np(const Dct2dArgs& a, const PoissonArgs& ps, int batch, cudaStream_t s, bool prepare) {
  auto width = [&](int np) {
    switch (np) {
      case 1: return col_width<M, 1, INV, POIS>(a, ps, batch, s, prepare);
      case 2: return col_width<M, 2, INV, POIS>(a, ps, batch, s, prepare);
      case 4: return col_width<M, 4, INV, POIS>(a, ps, batch, s, prepare);
      case 8: return col_width<M, 8, INV, POIS>(a, ps, batch, s, prepare);
      case 16: return col_width<M, 16, INV, POIS>(a, ps, batch, s, prepare);
      case 32: return col_width<M, 32, INV, POIS>(a, ps, batch, s, prepare);
      case 64: return col_width<M, 64, INV, POIS>(a, ps, batch, s, prepare);
    }
    return cudaErrorInvalidValue;
  };
  return width(strip_np<M>(a, batch));  // prepare: the width that a call with this batch runs
}

// N1 = 2 M.
template <bool INV, bool POIS>
cudaError_t col_run(int lg1, const Dct2dArgs& a, const PoissonArgs& ps, int batch, cudaStream_t s, bool prepare) {
  switch (lg1) {
    case 6: return col_np<32, INV, POIS>(a, ps, batch, s, prepare);
    case 7: return col_np<64, INV, POIS>(a, ps, batch, s, prepare);
    case 8: return col_np<128, INV, POIS>(a, ps, batch, s, prepare);
    case 9: return col_np<256, INV, POIS>(a, ps, batch, s, prepare);
    case 10: return col_np<512, INV, POIS>(a, ps, batch, s, prepare);
    case 11: return col_np<1024, INV, POIS>(a, ps, batch, s, prepare);
    case 12: return col_np<2048, INV, POIS>(a, ps, batch, s, prepare);
    case 13: return col_np<4096, INV, POIS>(a, ps, batch, s, prepare);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbdct
