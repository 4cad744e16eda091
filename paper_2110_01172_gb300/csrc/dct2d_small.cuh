// dct2d_small.cuh - a whole small 2D transform in one CTA and one launch.
//
// The two passes of the two-pass family (dct2d_tp_kernels.cuh: half-length
// column FFTs of the even and odd reordered rows, then row passes with the
// radix-2 column step folded in) run back to back on one transform of N1 x N2
// <= 16384 values held in shared memory, so nothing between the input and the
// output touches global memory.  Such transforms are bound by launches and
// latency when single, and by the extra pass over the workspace in batches;
// larger ones do not fit the registers of one CTA (64 values per thread, 256
// threads at 128 registers).  Measured, pair family -> one launch, forward /
// inverse: 64^2 8.2 / 10.6 -> 3.9 / 4.5 us, 203 x 64^2 12.3 / 15.9 -> 5.9 / 6.8,
// 2048 x 64^2 74 / 96 -> 18.3 / 19.2, 2048 x (64 x 256) 117 / 143 -> 78 / 80;
// two-pass family -> one launch: 2048 x 128^2 102 / 98 -> 72 / 76.  All but 128 x 128
// run exact (Dct2dArgs::exact), which costs 0.5 us of 203 x 64^2 forward.
//
// Shared memory of one transform is used in turn as the column FFTs' points
// (padded, the N2/4 float4 columns interleaved), the workspace rows E, O (E', O'),
// the row FFTs' points and the rows of the output (input), so global memory is
// only accessed as whole rows of float4.  The row strides WS and XS keep the
// groups of a warp, which work on consecutive rows, on distinct banks.
#pragma once

#include "dct2d_tp_kernels.cuh"

namespace gbdct {

template <int LG1, int LG2>
struct SmallGeom {
  static constexpr int N1 = 1 << LG1, L = 1 << LG2, M = N1 / 2;
  static constexpr int ST = L / 4;              // float4 per row
  static constexpr int TPM = M / 16;            // threads per column pair
  static constexpr int TPL = L / 16;            // threads per row group
  static constexpr int T = 2 * ST * TPM;        // threads per transform: 64 values each
  static constexpr int NT = T < 64 ? 64 / T : 1;  // transforms per CTA
  static constexpr int THREADS = T * NT;
  static constexpr int WS = ST + (TPL >= 16 ? 0 : TPL / 2);                          // workspace row stride (float4)
  static constexpr int XS = ST + (TPL >= 32 ? 0 : TPL >= 8 ? TPL / 4 : 1);           // input / output row stride
  static constexpr int LPM = M + M / 16;        // padded points per column pair
  static constexpr int max2(int a, int b) { return a > b ? a : b; }
  static constexpr int BUF = max2(max2(2 * ST * LPM, N1 * WS), max2(N1 * XS, (N1 / 4) * (L + L / 16)));
  static constexpr size_t SMEM = (size_t)NT * BUF * sizeof(float4);
  static constexpr int MINB = 512 / THREADS;    // up to 128 registers
  static constexpr bool EXACT = side_exact(LG1, LG2);
  // the radix-2 twiddles' rest: at N1 = 64 alone the other measures do not make up for the step
  static constexpr bool REST = EXACT && LG1 == 6;
  static_assert(LG1 >= 5 && LG2 >= 5 && LG1 + LG2 <= 14, "sides from 32, at most 16384 values");
};

// FFT of length M of the thread's column pair from registers (points g + TPM j);
// afterwards v holds output points, thread g's output i at small_col_out<M>(g, i).
// Called after a barrier that ends the last reads of s.
template <int M>
__device__ __forceinline__ int small_col_out(int g, int i) {
  constexpr int R = M / 16, TPM = M / 16;  // radix of the second stage (none for M = 16)
  if constexpr (M == 16) return i;
  else return g + (i / R) * TPM + 16 * (i % R);
}
template <int M, int ST, bool INV, bool EXACT>
__device__ __forceinline__ void small_col_fft(soa::C2* v, float4* __restrict__ s, int g,
                                              const float4* __restrict__ tw) {
  if constexpr (M == 16) {
    soa::dft<16, INV>(v);
  } else {
    constexpr int R = M / 16, NB = 16 / R, TPM = M / 16;
    soa::first_stage<M, INV, ST>(v, s, g);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NB; ++q) soa::load_butterfly<M, 16, ST>(v + q * R, s, g + q * TPM);
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      soa::Tw<R> w;
      const float4* twp = tw + tw_offset(M, 16) + g + q * TPM;
      w.load(twp, 16);
      soa::twiddle<R, INV, EXACT>(v + q * R, w, twp, 16);
      soa::dft<R, INV>(v + q * R);
    }
  }
}

template <int LG1, int LG2, bool INV>
__global__ void __launch_bounds__(SmallGeom<LG1, LG2>::THREADS, SmallGeom<LG1, LG2>::MINB)
    k_small(Dct2dArgs a, int batch) {
  using G = SmallGeom<LG1, LG2>;
  constexpr int N1 = G::N1, L = G::L, M = G::M, ST = G::ST, TPM = G::TPM, TPL = G::TPL;
  extern __shared__ float4 ssm[];
  const int tid = threadIdx.x % G::T;
  float4* s = ssm + (threadIdx.x / G::T) * G::BUF;
  const int b = blockIdx.x * G::NT + threadIdx.x / G::T;
  const bool live = G::NT == 1 || b < batch;  // the last CTA's spare threads compute the last transform, unstored
  const long long base = (long long)(live ? b : batch - 1) * (N1 * L);
  const float4* xin = reinterpret_cast<const float4*>(a.in + base);
  float4* xout = reinterpret_cast<float4*>(a.out + base);
  // column phase: column pair pi, rank g, parity par of the reordered row
  const int pi = tid % ST, g = tid / ST % TPM, par = tid / (ST * TPM);
  float4* cs = s + par * ST * G::LPM + pi;
  // row phase: group c, rank gr
  const int c = tid / TPL, gr = tid % TPL;
  const bool first = c == 0;
  const int kb = tp_item_b(c, M);
  float4* rs = s + c * (L + L / 16);
  const uint64_t pol = l2::evict_first();
  soa::C2 v[16];
  pdl::wait_prior_grid();
  if constexpr (!INV) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int row = reorder_src(2 * (g + TPM * j) + par, N1);
      float4 q = l2::ld(xin + row * ST + pi, pol);
      if (a.vkind == 1) {  // DST-II: (-1)^(n1 + n2)
        const float sr = (row & 1) ? -1.f : 1.f;
        q = vsign(q, sr, -sr);
      }
      v[j] = aos_to_soa(q);
    }
    small_col_fft<M, ST, false, G::EXACT>(v, cs, g, a.tw1x);
    __syncthreads();  // the workspace rows overlay the points
#pragma unroll
    for (int i = 0; i < 16; ++i) s[(par * M + small_col_out<M>(g, i)) * G::WS + pi] = soa::pack_aos(v[i]);
    __syncthreads();
    const float2* Zw = reinterpret_cast<const float2*>(s);
    const float2 *e1r = Zw + c * (2 * G::WS), *o1r = Zw + (M + c) * (2 * G::WS);
    const float2 *e2r = Zw + kb * (2 * G::WS), *o2r = Zw + (M + kb) * (2 * G::WS);
    const R2<false, G::REST> w(a, c, first);
    const int t = rowp::rev_lane_butterfly<TPL>(gr);
    if (rowp::warp_has_first<TPL>(first))
      tp_fwd_load<L, true, true, G::REST>(e1r, o1r, e2r, o2r, w, first, t, v);
    else
      tp_fwd_load<L, false, true, G::REST>(e1r, o1r, e2r, o2r, w, false, t, v);
    __syncthreads();
    soa::first_stage<L, false>(v, rs, t);
    rowp::stages_to_regs<L, 16, false, true, G::EXACT>(rs, gr, c, a.tw2x, v);
    pdl::launch_dependents();
    __syncthreads();
    fwd_post_x2<L, true, true, G::EXACT>(v, a, reinterpret_cast<float*>(s), 4 * G::XS, c, kb, first, gr);
    __syncthreads();
    if (live) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int f = tid + G::T * i;
        l2::st(xout + f, s[(f / ST) * G::XS + f % ST], pol);
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int f = tid + G::T * i;
      s[(f / ST) * G::XS + f % ST] = l2::ld(xin + f, pol);
    }
    __syncthreads();
    const float* C = reinterpret_cast<const float*>(s);
    const RowReads<true> A{inv_rows_of(a, C, c, 4 * G::XS, a.vkind), 0}, B{inv_rows_of(a, C, kb, 4 * G::XS, a.vkind), 0};
    int t;
    if (rowp::warp_has_first<TPL>(first))
      t = inv_pre_x2<L, true, true, G::EXACT>(a, A, B, a.vkind, c, kb, first, gr, v);
    else
      t = inv_pre_x2<L, true, false, G::EXACT>(a, A, B, a.vkind, c, kb, false, gr, v);
    __syncthreads();
    soa::first_stage<L, true>(v, rs, t);
    rowp::stages_to_regs<L, 16, true, false, G::EXACT>(rs, gr, c, a.tw2x, v);
    __syncthreads();
    float2* Zw = reinterpret_cast<float2*>(s);
    if (rowp::warp_has_first<TPL>(first))
      tp_inv_pair<L, true, G::REST>(v, a, Zw, 2 * G::WS, c, kb, first, gr);
    else
      tp_inv_pair<L, true, G::REST>(v, a, Zw, 2 * G::WS, c, kb, false, gr);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = aos_to_soa(s[(par * M + g + TPM * j) * G::WS + pi]);
    __syncthreads();
    small_col_fft<M, ST, true, G::EXACT>(v, cs, g, a.tw1x);
    pdl::launch_dependents();
    if (live) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int row = reorder_src(2 * small_col_out<M>(g, i) + par, N1);
        float4 y = soa_to_aos(v[i]);
        if (a.vkind) {  // output signs: (-1)^(n1+n2) DST-II, (-1)^n2 IDCT_IDXST, (-1)^n1 IDXST_IDCT
          const float sr = (a.vkind != 2 && (row & 1)) ? -1.f : 1.f;
          const float sc = (a.vkind != 3) ? -sr : sr;
          y = vsign(y, sr, sc);
        }
        l2::st(xout + row * ST + pi, y, pol);
      }
    }
  }
}

}  // namespace gbdct
