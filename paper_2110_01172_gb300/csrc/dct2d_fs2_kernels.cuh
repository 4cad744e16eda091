// dct2d_fs2_kernels.cuh - four-step column FFTs + row passes, occupancy-first.
//
// Method: arXiv 2110.01172, Algorithm 2 with the fused pre/postprocess of Section
// III; the column FFT of length N1 = A*B is split the four-step way so that every
// global access is a contiguous row segment.  Kernels shaped for occupancy:
//
//  * column steps: a CTA owns a slab of S rows (S = A or B) x a block of
//    complex columns; Q threads share a column group and each holds T = S/Q
//    points of it, so a DFT_S is a DFT_T in registers, a twiddle W_S^{q m},
//    an exchange through shared memory and DFT_Qs
//    (W_S^{(q+Qj)(m+Tp)} = W_S^{qm} W_Q^{qp} W_T^{jm}).  A thread has two adjacent
//    columns (16-byte accesses; Q = 4 or 8), one at S = 128;
//  * row passes: two items per thread group on the two-lane engine of fft_soa.cuh
//    (N2 <= 8192), or one sequence per group (float2, the radix-16 Stockham engine
//    of fft_core.cuh, ~64 registers per thread) at N2 = 16384.
//
// Workspace: N1 rows of N2/2 complex, row k1 of the column spectrum at physical row
// (k1 % B) * A + k1 / B.
// Launches overlap through programmatic dependent launch (8192 x 4096 forward /
// inverse 153.8 / 148.6 -> 147.0 / 142.6 us).
// Supported: N1 in {256, ..., 8192}, N2 in {256, ..., 16384}.
//
// The other kinds are index/sign maps around the DCT-II (Section V-B, Eq.
// idxst; DST-II per axis), folded into the first loads and last stores
// (a.vkind):
//   DST-II forward   x(n1,n2) (-1)^(n1+n2) in C1's loads; output (k1,k2) stored
//                    at (N1-1-k1, N2-1-k2) by the row pass
//   DST-II inverse   input read at (N1-1-k1, N2-1-k2) by the row pass's staging;
//                    (-1)^(n1+n2) in C1''s stores
//   IDCT_IDXST       input column k2 taken from column N2-k2 (column 0 zero):
//                    the preprocess swaps its reads k2 <-> N2-k2; (-1)^n2 in C1'
//   IDXST_IDCT       input row k1 taken from row N1-k1 (row 0 zero): the row
//                    pass swaps its two rows; (-1)^n1 in C1''s stores
#pragma once

#include "dct2d_kernels.cuh"
#include "fft_soa.cuh"
#include "l2_hint.cuh"
#include "launch_dep.cuh"
#include "row_pairs.cuh"
#include "tma_util.cuh"

#include <type_traits>

namespace gbdct {

// Calls f(integral_constant<int, I>) for I = B .. E-1 (compile-time loop).
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}

// Four-step split N1 = A * B of the column FFT (a tile parameter: the slabs of
// the column steps are A or B rows); both factors in {16, 32, 64, 128}.
template <int N1, int A_>
struct Fs2Geom {
  static constexpr int A = A_;
  static constexpr int B = N1 / A_;
  static_assert(A >= 16 && A <= 128 && B >= 16 && B <= 128, "four-step factors out of range");
};

// Physical workspace row of column-spectrum row k1 (A, B powers of two).
__device__ __forceinline__ int fs2_prow(int k1, int A, int B) { return (k1 & (B - 1)) * A + k1 / B; }

// ----------------------------------------------------------------------------
// Column steps, vector form (k_fs2_colv): each thread owns CPT adjacent complex
// columns (CPT = 2: 16-byte loads and stores) and T = S/Q points of each; Q
// threads share a column group.  DFT_S = DFT_T in registers, twiddle
// W_S^{q m}, one exchange through shared memory, then DFT_Q across the Q
// threads (S = Q T: W_S^{(q + Q j)(m + T p)} = W_S^{q m} W_Q^{q p} W_T^{j m}).
//   S = 16: Q 4, CPT 2;  S = 32: Q 4, CPT 2;  S = 64: Q 8, CPT 2;
//   S = 128: Q 8, CPT 1 (N1 = 8192).
// ----------------------------------------------------------------------------

// cos(2 pi k / 128), k = 0..127 (float roundings of the exact values)
__host__ __device__ constexpr float cos128(int k) {
  constexpr float t[128] = {
    1.000000000e+00f,
    9.987954562e-01f,
    9.951847267e-01f,
    9.891765100e-01f,
    9.807852804e-01f,
    9.700312532e-01f,
    9.569403357e-01f,
    9.415440652e-01f,
    9.238795325e-01f,
    9.039892931e-01f,
    8.819212643e-01f,
    8.577286100e-01f,
    8.314696123e-01f,
    8.032075315e-01f,
    7.730104534e-01f,
    7.409511254e-01f,
    7.071067812e-01f,
    6.715589548e-01f,
    6.343932842e-01f,
    5.956993045e-01f,
    5.555702330e-01f,
    5.141027442e-01f,
    4.713967368e-01f,
    4.275550934e-01f,
    3.826834324e-01f,
    3.368898534e-01f,
    2.902846773e-01f,
    2.429801799e-01f,
    1.950903220e-01f,
    1.467304745e-01f,
    9.801714033e-02f,
    4.906767433e-02f,
    6.123233996e-17f,
    -4.906767433e-02f,
    -9.801714033e-02f,
    -1.467304745e-01f,
    -1.950903220e-01f,
    -2.429801799e-01f,
    -2.902846773e-01f,
    -3.368898534e-01f,
    -3.826834324e-01f,
    -4.275550934e-01f,
    -4.713967368e-01f,
    -5.141027442e-01f,
    -5.555702330e-01f,
    -5.956993045e-01f,
    -6.343932842e-01f,
    -6.715589548e-01f,
    -7.071067812e-01f,
    -7.409511254e-01f,
    -7.730104534e-01f,
    -8.032075315e-01f,
    -8.314696123e-01f,
    -8.577286100e-01f,
    -8.819212643e-01f,
    -9.039892931e-01f,
    -9.238795325e-01f,
    -9.415440652e-01f,
    -9.569403357e-01f,
    -9.700312532e-01f,
    -9.807852804e-01f,
    -9.891765100e-01f,
    -9.951847267e-01f,
    -9.987954562e-01f,
    -1.000000000e+00f,
    -9.987954562e-01f,
    -9.951847267e-01f,
    -9.891765100e-01f,
    -9.807852804e-01f,
    -9.700312532e-01f,
    -9.569403357e-01f,
    -9.415440652e-01f,
    -9.238795325e-01f,
    -9.039892931e-01f,
    -8.819212643e-01f,
    -8.577286100e-01f,
    -8.314696123e-01f,
    -8.032075315e-01f,
    -7.730104534e-01f,
    -7.409511254e-01f,
    -7.071067812e-01f,
    -6.715589548e-01f,
    -6.343932842e-01f,
    -5.956993045e-01f,
    -5.555702330e-01f,
    -5.141027442e-01f,
    -4.713967368e-01f,
    -4.275550934e-01f,
    -3.826834324e-01f,
    -3.368898534e-01f,
    -2.902846773e-01f,
    -2.429801799e-01f,
    -1.950903220e-01f,
    -1.467304745e-01f,
    -9.801714033e-02f,
    -4.906767433e-02f,
    -1.836970199e-16f,
    4.906767433e-02f,
    9.801714033e-02f,
    1.467304745e-01f,
    1.950903220e-01f,
    2.429801799e-01f,
    2.902846773e-01f,
    3.368898534e-01f,
    3.826834324e-01f,
    4.275550934e-01f,
    4.713967368e-01f,
    5.141027442e-01f,
    5.555702330e-01f,
    5.956993045e-01f,
    6.343932842e-01f,
    6.715589548e-01f,
    7.071067812e-01f,
    7.409511254e-01f,
    7.730104534e-01f,
    8.032075315e-01f,
    8.314696123e-01f,
    8.577286100e-01f,
    8.819212643e-01f,
    9.039892931e-01f,
    9.238795325e-01f,
    9.415440652e-01f,
    9.569403357e-01f,
    9.700312532e-01f,
    9.807852804e-01f,
    9.891765100e-01f,
    9.951847267e-01f,
    9.987954562e-01f

  };
  return t[k & 127];
}

// a * W_R^E for R dividing 128, W_R = exp(-2 pi i / R) (forward) or exp(+2 pi i / R).
template <int R, int E, bool INV, typename T>
__device__ __forceinline__ T mul_w128(T a) {
  constexpr int e = ((E * (128 / R)) % 128 + 128) % 128;
  constexpr float c = cos128(e);
  constexpr float s = cos128((160 - e) % 128);  // sin(2 pi e / 128) = cos(2 pi (32 - e) / 128)
  if constexpr (e == 0) {
    return a;
  } else if constexpr (e == 32) {
    return mul_mj<INV>(a);
  } else if constexpr (e == 64) {
    return cneg(a);
  } else if constexpr (e == 96) {
    return mul_mj<!INV>(a);
  } else if constexpr (e % 32 == 16) {
    return cmul_diag(a, c, (INV ? s : -s) / c);
  } else {
    return cmulk(a, c, INV ? s : -s);
  }
}

template <int S>
struct ColCfg {
  static constexpr int Q = S >= 64 ? 8 : 4;           // threads per column group
  static constexpr int CPT = S >= 128 ? 1 : 2;        // complex columns per thread
  static constexpr int T = S / Q;                     // points per column per thread
  static constexpr int COLS = S >= 128 ? 64 : 128;    // complex columns per CTA
  static constexpr int NG = COLS / CPT;               // column groups per CTA
  static constexpr int THREADS = NG * Q;
  static constexpr size_t SMEM = (size_t)S * COLS * sizeof(float2);
  using V = typename std::conditional<CPT == 2, float4, float2>::type;
};

// x[m] *= W_S^{q m} (m < T) for the thread's warp-uniform q < Q.
template <int S, int Q, int T, bool INV, typename V>
__device__ __forceinline__ void colv_twiddle(V* x, int q) {
  static_for<1, Q>([&](auto qc) {
    constexpr int qq = decltype(qc)::value;
    if (q == qq) {
      static_for<1, T>([&](auto mc) {
        constexpr int m = decltype(mc)::value;
        x[m] = mul_w128<S, qq * m, INV>(x[m]);
      });
    }
  });
}

// DFT_S along the slab rows: on entry x[j] = slab row q + Q j (j < T); on return
// x[i Q + p] = output row (q T/Q + i) + T p  (i < T/Q, p < Q).
template <int S, bool INV, typename V>
__device__ __forceinline__ void colv_dft(V* x, int q, int c, V* ex) {
  using C = ColCfg<S>;
  constexpr int Q = C::Q, T = C::T, NG = C::NG, TQ = T / Q;
  dft<T, INV>(x);
  colv_twiddle<S, Q, T, INV>(x, q);
#pragma unroll
  for (int m = 0; m < T; ++m) ex[(q * T + m) * NG + c] = x[m];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TQ; ++i) {
    const int m = q * TQ + i;
    V y[Q];
#pragma unroll
    for (int p = 0; p < Q; ++p) y[p] = ex[(p * T + m) * NG + c];
    dft<Q, INV>(y);
#pragma unroll
    for (int p = 0; p < Q; ++p) x[i * Q + p] = y[p];
  }
  __syncthreads();
}

__device__ __forceinline__ float2 vsign(float2 v, float sr, float sc) { return make_float2(sr * v.x, sc * v.y); }
__device__ __forceinline__ float4 vsign(float4 v, float sr, float sc) {
  return make_float4(sr * v.x, sc * v.y, sr * v.z, sc * v.w);
}

template <int N1, int A, int KIND>
__global__ void __launch_bounds__(ColCfg<(KIND == 0 || KIND == 3) ? N1 / A : A>::THREADS,
                                  1024 / ColCfg<(KIND == 0 || KIND == 3) ? N1 / A : A>::THREADS)
k_fs2_colv(Dct2dArgs a) {
  using G = Fs2Geom<N1, A>;
  constexpr bool INV = KIND >= 2;
  constexpr int S = (KIND == 0 || KIND == 3) ? G::B : G::A;
  using C = ColCfg<S>;
  using V = typename C::V;
  constexpr int T = C::T, Q = C::Q, TQ = T / Q;
  extern __shared__ float4 scv[];
  V* ex = reinterpret_cast<V*>(scv);
  const int c = threadIdx.x % C::NG, q = threadIdx.x / C::NG;
  const int r = blockIdx.x;
  const int N2 = a.n2;
  const long long hv = N2 / 2 / C::CPT;  // V elements per workspace row
  const int colv = blockIdx.y * C::NG + c;  // V index within a row
  V* W = reinterpret_cast<V*>(a.work + (long long)blockIdx.z * a.work_bstride);

  // L2 policies: the streamed input / output evict first, the workspace
  // (read again by the next launch of the transform) evicts last
  const uint64_t pol_stream = l2::evict_first(), pol_keep = l2::evict_last();
  pdl::wait_prior_grid();
  V x[T];
#pragma unroll
  for (int j = 0; j < T; ++j) {
    const int i = q + Q * j;  // slab row of this input
    if constexpr (KIND == 0) {
      const float* xin = a.in + (long long)blockIdx.z * a.in_bstride;
      const int row = reorder_src(r + G::A * i, N1);
      x[j] = l2::ld_once(reinterpret_cast<const V*>(xin + (long long)row * N2) + colv, pol_stream);
      if (a.vkind == 1) {  // DST-II: (-1)^(n1 + n2); real columns alternate in parity
        const float sr = (row & 1) ? -1.f : 1.f;
        x[j] = vsign(x[j], sr, -sr);
      }
    } else if constexpr (KIND == 3) {
      x[j] = l2::ld_once(W + (long long)(i * G::A + r) * hv + colv, pol_stream);  // last use of the workspace
    } else {
      x[j] = l2::ld_once(W + (long long)(r * G::A + i) * hv + colv, pol_keep);
    }
  }
  colv_dft<S, INV>(x, q, c, ex);
  pdl::launch_dependents();
#pragma unroll
  for (int i = 0; i < TQ; ++i)
#pragma unroll
    for (int p = 0; p < Q; ++p) {
      const int o = q * TQ + i + T * p;  // k1b (KIND 0), k1a (1), n1a (2), n1b (3)
      V y = x[i * Q + p];
      if constexpr (KIND == 0) {
        y = cmul(y, __ldg(a.fstw + r * G::B + o));
        l2::st(W + (long long)(o * G::A + r) * hv + colv, y, pol_keep);
      } else if constexpr (KIND == 2) {
        y = cmulc(y, __ldg(a.fstw + o * G::B + r));
        l2::st(W + (long long)(r * G::A + o) * hv + colv, y, pol_keep);
      } else if constexpr (KIND == 1) {
        l2::st(W + (long long)(r * G::A + o) * hv + colv, y, pol_keep);
      } else {
        float* xo = a.out + (long long)blockIdx.z * a.out_bstride;
        const int row = reorder_src(r + G::A * o, N1);
        if (a.vkind) {  // output signs: (-1)^(n1+n2) DST-II, (-1)^n2 IDCT_IDXST, (-1)^n1 IDXST_IDCT
          const float sr = (a.vkind != 2 && (row & 1)) ? -1.f : 1.f;
          const float sc = (a.vkind != 3) ? -sr : sr;
          y = vsign(y, sr, sc);
        }
        l2::st(reinterpret_cast<V*>(xo + (long long)row * N2) + colv, y, pol_stream);
      }
    }
}

// ----------------------------------------------------------------------------
// Row passes (L = N2).  Item k1 in [0, N1/2) owns the row pair (k1, N1-k1);
// item 0 the packed pair (0, N1/2).  Forward: Hermitian split of the two
// column-spectrum rows, row FFT, symmetric-pair postprocess (Section III-B,
// Eqs. four-elements, s-t) -> output rows k1 and N1-k1.  Inverse: four-read
// preprocess (Eq. 2d_idct_pre, conjugated twiddle, 1/(N1 N2) in the a-table),
// row IFFT, column pairing Z_p(k1) = U(k1,p) + i U(k1,L-1-p) -> workspace.
// One item group per CTA with the rows staged by the threads (k_fs2_rows);
// used for N2 = 16384, where the two-item form below does not fit.
// ----------------------------------------------------------------------------
template <int L>
struct RowGeom {
  static constexpr int TPS = fft_tps(L);
  static constexpr int NI = (256 / TPS) > 0 ? 256 / TPS : 1;  // items per CTA
  static constexpr int THREADS = NI * TPS;
  static constexpr int LP = pad_len<float2>(L);
  static constexpr size_t SMEM = (size_t)NI * LP * sizeof(float2);
  static constexpr int MINB = 1024 / THREADS;  // caps registers at 64 per thread
};

__device__ __forceinline__ int row_mirror(int k1, int N1) { return k1 ? N1 - k1 : N1 / 2; }

// The two source rows (L floats each) of item k1 of batch entry b.  Forward:
// column-spectrum rows k1 and its mirror in the workspace (four-step physical
// order).  Inverse: input rows with the kind's row map folded in: DST-II reads
// rows N1-1-k1 and N1-1-kmir (columns reversed by inv_pre); IDXST_IDCT takes
// row k1 from row N1-k1, so the two rows trade places and the packed item's
// row 0 is zero (*ra = nullptr).
template <int L, bool INV>
__device__ __forceinline__ void row_sources(const Dct2dArgs& a, int b, int k1, const float** ra, const float** rb) {
  const int N1 = a.n1;
  const int kmir = row_mirror(k1, N1);
  if constexpr (!INV) {
    const float2* Zw = a.work + (long long)b * a.work_bstride;
    *ra = reinterpret_cast<const float*>(Zw + (long long)fs2_prow(k1, a.fsA, a.fsB) * (L / 2));
    *rb = reinterpret_cast<const float*>(Zw + (long long)fs2_prow(kmir, a.fsA, a.fsB) * (L / 2));
  } else {
    const float* C = a.in + (long long)b * a.in_bstride;
    int r0 = k1, r1 = kmir;
    if (a.vkind == 1) {
      r0 = N1 - 1 - k1;
      r1 = N1 - 1 - kmir;
    }
    *ra = C + (long long)r0 * L;
    *rb = C + (long long)r1 * L;
    if (a.vkind == 3) {
      if (k1) {
        const float* t = *ra;
        *ra = *rb;
        *rb = t;
      } else {
        *ra = nullptr;
      }
    }
  }
}

// Copies two rows of L floats (row0 -> sf[0, L), row1 -> sf[L, 2L)) into shared
// memory with 16-byte loads (TPS threads); a null row0 is left unwritten.
template <int L, int TPS>
__device__ __forceinline__ void stage_two_rows(float* sf, const float* row0, const float* row1, int g) {
  const float4* a4 = reinterpret_cast<const float4*>(row0);
  const float4* b4 = reinterpret_cast<const float4*>(row1);
  float4* s4 = reinterpret_cast<float4*>(sf);
  constexpr int Q = L / 4;  // float4 per row
  float4 t[2 * Q / TPS];
#pragma unroll
  for (int j = 0; j < Q / TPS; ++j) {
    if (a4) t[j] = a4[g + j * TPS];
    t[Q / TPS + j] = b4[g + j * TPS];
  }
#pragma unroll
  for (int j = 0; j < Q / TPS; ++j) {
    if (a4) s4[g + j * TPS] = t[j];
    s4[Q + g + j * TPS] = t[Q / TPS + j];
  }
}

// Forward split: st holds rows za (L/2 complex) and zb (L/2 complex); returns
// the thread's 16 points n2 = g + j TPS of the row to transform.
template <int L, int TPS>
__device__ __forceinline__ void fwd_split(const float2* st, bool packed, int g, float2* v) {
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int n2 = g + j * TPS;
    const bool lowhalf = n2 < L / 2;
    const int p = lowhalf ? n2 : L - 1 - n2;
    const float2 za = st[p];
    const float2 zb = st[L / 2 + p];
    if (packed) {
      v[j] = lowhalf ? make_float2(za.x, zb.x) : make_float2(za.y, zb.y);
    } else {
      v[j] = lowhalf ? make_float2(0.5f * (za.x + zb.x), 0.5f * (za.y - zb.y))
                     : make_float2(0.5f * (za.y + zb.y), 0.5f * (zb.x - za.x));
    }
  }
}

// Forward postprocess from the row spectrum in s (padded layout) to output
// rows k1 and kmir of y (DST-II: rows and columns reversed).
template <int L, int TPS>
__device__ __forceinline__ void fwd_post(const float2* s, const Dct2dArgs& a, float* y, int k1, int kmir,
                                         bool packed, int g) {
  const int N1 = a.n1;
  const float2 av = __ldg(a.fa + k1);
  const bool rev = a.vkind == 1;  // DST-II: output (k1, k2) goes to (N1-1-k1, N2-1-k2)
  float* row0 = y + (long long)(rev ? N1 - 1 - k1 : k1) * L;
  float* row1 = y + (long long)(rev ? N1 - 1 - kmir : kmir) * L;
  constexpr float RH = 0.70710678118654752f;
  for (int i = g; i < L / 8; i += TPS) {
    const int c = 4 * i;
    float2 Yq[5], Ym[5];
#pragma unroll
    for (int d = 0; d < 5; ++d) {
      Yq[d] = s[pidx<float2>(c + d)];
      Ym[d] = s[pidx<float2>((L - c - d) & (L - 1))];
    }
    float q0[4], q1[4], r0[4], r1[4];
#pragma unroll
    for (int d = 1; d <= 3; ++d) {
      const float2 bt = __ldg(a.fb + c + d);
      const float2 P = Yq[d], M = Ym[d];
      if (packed) {
        const float2 s0 = cmul(bt, make_float2(P.x + M.x, P.y - M.y));
        const float2 sh = cmul(bt, make_float2(RH * (P.y + M.y), RH * (M.x - P.x)));
        q0[d] = s0.x;
        q1[d] = sh.x;
        r0[4 - d] = -s0.y;
        r1[4 - d] = -sh.y;
      } else {
        const float2 aP = cmul(P, av);
        const float2 aM = cmul(M, av);
        const float2 sv = cmul(bt, make_float2(aP.x + aM.x, aP.y - aM.y));
        const float2 tv = cmul(bt, make_float2(aP.x - aM.x, aP.y + aM.y));
        q0[d] = sv.x;
        q1[d] = -tv.y;
        r0[4 - d] = -sv.y;
        r1[4 - d] = -tv.x;
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int col = e ? (L - c - 4) : c;
      const float2 P = e ? Ym[4] : Yq[0];
      const float2 M = e ? Yq[4] : Ym[0];
      const float2 bt = __ldg(a.fb + col);
      float o0, o1;
      if (packed) {
        const float2 s0 = cmul(bt, make_float2(P.x + M.x, P.y - M.y));
        const float2 sh = cmul(bt, make_float2(RH * (P.y + M.y), RH * (M.x - P.x)));
        o0 = s0.x;
        o1 = sh.x;
      } else {
        const float2 aP = cmul(P, av);
        const float2 aM = cmul(M, av);
        const float2 u = make_float2(aP.x + aM.x, aP.y - aM.y);
        const float2 w = make_float2(aP.x - aM.x, aP.y + aM.y);
        o0 = bt.x * u.x - bt.y * u.y;
        o1 = -(bt.x * w.y + bt.y * w.x);
      }
      if (e) {
        r0[0] = o0;
        r1[0] = o1;
      } else {
        q0[0] = o0;
        q1[0] = o1;
      }
    }
    if (!rev) {
      *reinterpret_cast<float4*>(row0 + c) = make_float4(q0[0], q0[1], q0[2], q0[3]);
      *reinterpret_cast<float4*>(row1 + c) = make_float4(q1[0], q1[1], q1[2], q1[3]);
      *reinterpret_cast<float4*>(row0 + L - c - 4) = make_float4(r0[0], r0[1], r0[2], r0[3]);
      *reinterpret_cast<float4*>(row1 + L - c - 4) = make_float4(r1[0], r1[1], r1[2], r1[3]);
    } else {
      *reinterpret_cast<float4*>(row0 + L - c - 4) = make_float4(q0[3], q0[2], q0[1], q0[0]);
      *reinterpret_cast<float4*>(row1 + L - c - 4) = make_float4(q1[3], q1[2], q1[1], q1[0]);
      *reinterpret_cast<float4*>(row0 + c) = make_float4(r0[3], r0[2], r0[1], r0[0]);
      *reinterpret_cast<float4*>(row1 + c) = make_float4(r1[3], r1[2], r1[1], r1[0]);
    }
  }
}

// Inverse preprocess: sf holds the two source rows (L floats each, raw);
// zero_a: the first row is zero (IDXST_IDCT, packed item).  DST-II reads the
// columns reversed; IDCT_IDXST swaps the reads at k2 and N2-k2 (column 0 zero).
template <int L, int TPS, bool MAPPED>
__device__ __forceinline__ void inv_pre_loop(const float* sf, const Dct2dArgs& a, float2 ia, float2 ih, bool packed,
                                             bool zero_a, int g, float2* v) {
  const bool rev = MAPPED && a.vkind == 1, swapc = MAPPED && a.vkind == 2;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int k2 = g + j * TPS;
    const int km = (L - k2) & (L - 1);
    float c1, c3, c4, c2;
    if constexpr (!MAPPED) {
      c1 = zero_a ? 0.f : sf[k2];
      c3 = sf[L + k2];
      c4 = (k2 && !zero_a) ? sf[km] : 0.f;
      c2 = k2 ? sf[L + km] : 0.f;
    } else {
      const int ka = swapc ? km : k2, kb = swapc ? k2 : km;
      const int pa = rev ? L - 1 - ka : ka, pb = rev ? L - 1 - kb : kb;
      const bool z0 = swapc && !k2;
      c1 = (zero_a || z0) ? 0.f : sf[pa];
      c3 = z0 ? 0.f : sf[L + pa];
      c4 = (k2 && !zero_a) ? sf[pb] : 0.f;
      c2 = k2 ? sf[L + pb] : 0.f;
    }
    const float2 bk = __ldg(a.ib + k2);
    if (packed) {
      const float2 v0 = cmul(cmul(make_float2(c1, -c4), bk), ia);
      const float2 vh = cmul(cmul(make_float2(c3 - c2, -(c3 + c2)), bk), ih);
      v[j] = make_float2(v0.x - vh.y, v0.y + vh.x);
    } else {
      v[j] = cmul(cmul(make_float2(c1 - c2, -(c3 + c4)), bk), ia);
    }
  }
}

// Inverse preprocess: sf holds the two source rows (L floats each, raw);
// zero_a: the first row is zero (IDXST_IDCT, packed item).  DST-II reads the
// columns reversed; IDCT_IDXST swaps the reads at k2 and N2-k2 (column 0 zero).
// The kind is tested once, outside the unrolled loop.
template <int L, int TPS>
__device__ __forceinline__ void inv_pre(const float* sf, const Dct2dArgs& a, int k1, bool packed, bool zero_a,
                                        int g, float2* v) {
  const float2 ia = __ldg(a.ia + k1);
  const float2 ih = __ldg(a.ia + a.n1 / 2);
  if (a.vkind == 1 || a.vkind == 2)
    inv_pre_loop<L, TPS, true>(sf, a, ia, ih, packed, zero_a, g, v);
  else
    inv_pre_loop<L, TPS, false>(sf, a, ia, ih, packed, zero_a, g, v);
}

// Inverse pairing: row IFFT in s -> workspace rows of k1 and kmir.
template <int L, int TPS>
__device__ __forceinline__ void inv_pair(const float2* s, float2* zr0, float2* zr1, bool packed, int g) {
  for (int h = g; h < L / 4; h += TPS) {  // two columns p = 2h, 2h + 1 per 16-byte store
    const int p = 2 * h;
    const float2 u0 = s[pidx<float2>(p)], u1 = s[pidx<float2>(p + 1)];
    const float2 w0 = s[pidx<float2>(L - 1 - p)], w1 = s[pidx<float2>(L - 2 - p)];
    float4 o0, o1;
    if (packed) {
      o0 = make_float4(u0.x, w0.x, u1.x, w1.x);
      o1 = make_float4(u0.y, w0.y, u1.y, w1.y);
    } else {
      o0 = make_float4(u0.x - w0.y, u0.y + w0.x, u1.x - w1.y, u1.y + w1.x);
      o1 = make_float4(u0.x + w0.y, w0.x - u0.y, u1.x + w1.y, w1.x - u1.y);
    }
    *reinterpret_cast<float4*>(zr0 + p) = o0;
    *reinterpret_cast<float4*>(zr1 + p) = o1;
  }
}

// Everything of one item after its rows are in shared memory (st: raw rows;
// s: the item's FFT buffer).  Contains __syncthreads: all threads call it.
template <int L, bool INV>
__device__ __forceinline__ void row_item(const Dct2dArgs& a, int b, int k1, const float* st, float2* s, int g,
                                         bool zero_a) {
  using R = RowGeom<L>;
  const bool packed = (k1 == 0);
  const int kmir = row_mirror(k1, a.n1);
  float2 v[16];
  if constexpr (!INV)
    fwd_split<L, R::TPS>(reinterpret_cast<const float2*>(st), packed, g, v);
  else
    inv_pre<L, R::TPS>(st, a, k1, packed, zero_a, g, v);
  __syncthreads();  // st may alias s: every read of the rows precedes the first stage
  first_stage_regs<L, INV>(v, s, g);
  __syncthreads();
  fft_stages<L, 16, INV>(s, g, a.tw2);
  if constexpr (!INV) {
    fwd_post<L, R::TPS>(s, a, a.out + (long long)b * a.out_bstride, k1, kmir, packed, g);
  } else {
    float2* Zw = a.work + (long long)b * a.work_bstride;
    inv_pair<L, R::TPS>(s, Zw + (long long)fs2_prow(k1, a.fsA, a.fsB) * (L / 2),
                        Zw + (long long)fs2_prow(kmir, a.fsA, a.fsB) * (L / 2), packed, g);
  }
}

template <int L, bool INV>
__global__ void __launch_bounds__(RowGeom<L>::THREADS, RowGeom<L>::MINB) k_fs2_rows(Dct2dArgs a) {
  using R = RowGeom<L>;
  extern __shared__ float4 srw[];
  const int li = threadIdx.x / R::TPS, g = threadIdx.x % R::TPS;
  float2* s = reinterpret_cast<float2*>(srw) + li * R::LP;
  const int k1 = blockIdx.x * R::NI + li;
  const float *ra, *rb;
  row_sources<L, INV>(a, blockIdx.z, k1, &ra, &rb);
  stage_two_rows<L, R::TPS>(reinterpret_cast<float*>(s), ra, rb, g);  // raw rows in the FFT buffer
  __syncthreads();
  row_item<L, INV>(a, blockIdx.z, k1, reinterpret_cast<const float*>(s), s, g, ra == nullptr);
}


// ----------------------------------------------------------------------------
// Row passes, two-item form (N2 <= 8192, the default).  A thread group of
// L/16 threads transforms two row items at once in packed two-lane FP32
// arithmetic (fft_soa.cuh): lane a is item k1, lane b item k1 + 1.  The
// forward Hermitian split is fused into the loads (each thread reads its 16
// points of the four column-spectrum rows straight from the workspace, no
// staging copy), and the split's factor 1/2 is folded into the a-twiddle of
// the combine.  The inverse reads its four-read preprocess inputs straight
// from the input rows.  Item 0 (the packed rows 0 and N1/2) takes the
// packed formulas in lane a of the first group.
// ----------------------------------------------------------------------------
template <int L>
struct RowX2Geom {
  static constexpr int TPS = fft_tps(L);                          // threads per item pair
  static constexpr int NP = (256 / TPS) > 0 ? 256 / TPS : 1;      // item pairs per CTA
  static constexpr int THREADS = NP * TPS;
  static constexpr int LP = L + L / 16;                           // padded float4 per item pair
  static constexpr size_t SMEM = (size_t)NP * LP * sizeof(float4);
  // CTAs per SM: two (up to 128 registers) measured faster than three at 80
  // registers, where the compiler serialises the loads of the split
  static constexpr int MINB = THREADS >= 512 ? 1 : 2;
  static constexpr int MINB_INV = THREADS >= 512 ? 1 : 2;
};

// Column-spectrum rows of item k (row k1 and its mirror) in the workspace.
template <int L>
__device__ __forceinline__ void fwd_rows_of(const Dct2dArgs& a, const float2* Zw, int k, const float2** z,
                                            const float2** m) {
  *z = Zw + (long long)fs2_prow(k, a.fsA, a.fsB) * (L / 2);
  *m = Zw + (long long)fs2_prow(row_mirror(k, a.n1), a.fsA, a.fsB) * (L / 2);
}

// Forward split of two items from the workspace into SoA registers: point
// n2 = t + TPS j of u = V_col(k1, :) is (z(p) + conj m(p)) / 2 for n2 < L/2
// (p = n2) and (z(p) - conj m(p)) / 2i above (p = L-1-n2); the 1/2 is left out
// here.  Packed lane a (item 0): u = V_col(0, :) + i V_col(N1/2, :).  Each
// workspace value is read once: the thread reads its low-half points, forms
// both the low value and the high value it implies (for point L-1-n2, which
// belongs to the mirror butterfly TPS-1-t at j' = 15 - j), and the two mirror
// lanes swap the high values.
// Split of point p for both lanes from the column-spectrum values A = z_a(p),
// Am = m_a(p), B = z_b(p), Bm = m_b(p): the low value (point p) into lo, the
// high value (point L-1-p) exchanged with the mirror lane into hi.
template <int MASK>
__device__ __forceinline__ void split_point(float2 A, float2 Am, float2 B, float2 Bm, bool packed, soa::C2& lo,
                                            soa::C2& hi) {
  const float lra = packed ? A.x : A.x + Am.x, lia = packed ? Am.x : A.y - Am.y;
  const float hra = packed ? A.y : A.y + Am.y, hia = packed ? Am.y : Am.x - A.x;
  lo = soa::C2{make_float2(lra, B.x + Bm.x), make_float2(lia, B.y - Bm.y)};
  const float h0 = hra, h1 = B.y + Bm.y, h2 = hia, h3 = Bm.x - B.x;
  hi = soa::C2{make_float2(__shfl_xor_sync(0xffffffffu, h0, MASK), __shfl_xor_sync(0xffffffffu, h1, MASK)),
               make_float2(__shfl_xor_sync(0xffffffffu, h2, MASK), __shfl_xor_sync(0xffffffffu, h3, MASK))};
}

template <int L>
__device__ __forceinline__ void fwd_split_x2(const float2* __restrict__ za, const float2* __restrict__ ma,
                                             const float2* __restrict__ zb, const float2* __restrict__ mb, int t,
                                             bool packed, soa::C2* v) {
  constexpr int TPS = fft_tps(L);
  constexpr int MASK = rowp::rev_lane_mask<TPS>();
  const uint64_t pol = l2::evict_first();  // last use of the workspace
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int p = t + TPS * j;
    const float2 A = l2::ld_once(za + p, pol), Am = l2::ld_once(ma + p, pol), B = l2::ld_once(zb + p, pol),
                 Bm = l2::ld_once(mb + p, pol);
    // low point n2 = p (this thread), high point L-1-p (the mirror lane)
    split_point<MASK>(A, Am, B, Bm, packed, v[j], v[15 - j]);
  }
}

// Output rows k1, N1-k1 (lane a; rows 0 and N1/2 of the packed item) and kb, N1-kb
// (lane b) of a group.
struct OutRows {
  float *a0, *a1, *b0, *b1;
};
// The output row of item k (mirror: its second row); DST-II (rev): output (k1, k2)
// goes to (N1-1-k1, N2-1-k2).
__device__ __forceinline__ int fwd_out_row(int k, bool mirror, int N1, bool rev) {
  const int r = mirror ? row_mirror(k, N1) : k;
  return rev ? N1 - 1 - r : r;
}

// Forward postprocess of both items (rowp::fwd_post) into their output rows,
// rows_of().  GENERAL: plans with the DST-II order or a magnitude threshold.
template <int L, bool GENERAL, bool FIRST, bool SMEM, bool EXACT, typename Rows>
__device__ __forceinline__ void fwd_post_rows(soa::C2* v, const Dct2dArgs& a, const Rows& rows_of, int k1, int kb,
                                              bool packed, int g) {
  const float2 fa0 = __ldg(a.fa + k1), fa1 = __ldg(a.fa + kb);
  // 1/2 of the split folded into the a-twiddle (not for the packed item)
  const float2 avr = make_float2(packed ? 1.f : 0.5f * fa0.x, 0.5f * fa1.x);
  const float2 avi = make_float2(packed ? 0.f : 0.5f * fa0.y, 0.5f * fa1.y);
  rowp::FwdOut<L, GENERAL, SMEM> out;
  const OutRows rows = rows_of();
  out.a0 = rows.a0;
  out.a1 = rows.a1;
  out.b0 = rows.b0;
  out.b1 = rows.b1;
  out.pol = l2::evict_first();  // the output is streamed out
  out.eps = a.thresh;           // magnitude threshold of Section V-A, Eq. image-compression (0: off)
  out.rev = GENERAL && a.vkind == 1;
  rowp::fwd_post<L, FIRST, EXACT>(v, out, avr, avi, a.fb4, g, packed);
}
template <int L, bool GENERAL, bool SMEM, bool EXACT, typename Rows>
__device__ __forceinline__ void fwd_post_x2(soa::C2* v, const Dct2dArgs& a, const Rows& rows_of, int k1, int kb,
                                            bool packed, int g) {
  if (rowp::warp_has_first<fft_tps(L)>(packed))
    fwd_post_rows<L, GENERAL, true, SMEM, EXACT>(v, a, rows_of, k1, kb, packed, g);
  else
    fwd_post_rows<L, GENERAL, false, SMEM, EXACT>(v, a, rows_of, k1, kb, false, g);
}
// The same into rows of y, `stride` floats apart.
template <int L, bool GENERAL, bool SMEM, bool EXACT>
__device__ __forceinline__ void fwd_post_x2(soa::C2* v, const Dct2dArgs& a, float* y, long long stride, int k1, int kb,
                                            bool packed, int g) {
  const bool rev = GENERAL && a.vkind == 1;
  auto row = [&](int k, bool mirror) { return y + fwd_out_row(k, mirror, a.n1, rev) * stride; };
  fwd_post_x2<L, GENERAL, SMEM, EXACT>(
      v, a, [&] { return OutRows{row(k1, false), row(k1, true), row(kb, false), row(kb, true)}; }, k1, kb, packed, g);
}

// Row FFT of both items from registers (v: points t + TPS j of the thread's
// first-stage butterfly t) and the postprocess.
template <int L, bool GENERAL, bool EXACT>
__device__ __forceinline__ void fwd_fft_post_x2(soa::C2* v, float4* s, const Dct2dArgs& a, float* y, int k1, int kb,
                                                bool packed, int t, int g, int group) {
  soa::first_stage<L, false>(v, s, t);
  rowp::stages_to_regs<L, 16, false, true, EXACT>(s, g, group, a.tw2x, v);
  pdl::launch_dependents();
  fwd_post_x2<L, GENERAL, false, EXACT>(v, a, y, L, k1, kb, packed, g);
}

template <int L, bool GENERAL>
__global__ void __launch_bounds__(RowX2Geom<L>::THREADS, RowX2Geom<L>::MINB) k_fs2_rows_fwd_x2(Dct2dArgs a) {
  using R = RowX2Geom<L>;
  extern __shared__ float4 sxf[];
  const int pi = threadIdx.x / R::TPS, g = threadIdx.x % R::TPS;
  float4* s = sxf + pi * R::LP;
  const int k1 = 2 * (blockIdx.x * R::NP + pi);  // items k1 (lane a), k1 + 1 (lane b)
  const float2* Zw = a.work + (long long)blockIdx.z * a.work_bstride;
  const float2 *za, *ma, *zb, *mb;
  fwd_rows_of<L>(a, Zw, k1, &za, &ma);
  fwd_rows_of<L>(a, Zw, k1 + 1, &zb, &mb);
  soa::C2 v[16];
  const bool packed = (k1 == 0);
  const int t = rowp::rev_lane_butterfly<R::TPS>(g);
  pdl::wait_prior_grid();
  // A workspace larger than L2 comes from DRAM: with one CTA per SM (L = 8192) the
  // memory would idle while all of them compute, so each sends for the rows of the
  // CTA that follows it on an SM (8192^2 forward 354 -> 334 us).
  if (a.ahead && g == 0 && (int)blockIdx.x + a.ahead < (int)gridDim.x) {
    const int kn = k1 + 2 * R::NP * a.ahead;
    const float2* next[4];
    fwd_rows_of<L>(a, Zw, kn, &next[0], &next[1]);
    fwd_rows_of<L>(a, Zw, kn + 1, &next[2], &next[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) tma::prefetch_l2(next[i], L * (uint32_t)sizeof(float));
  }
  if (rowp::warp_has_first<R::TPS>(packed))
    fwd_split_x2<L>(za, ma, zb, mb, t, packed, v);
  else
    fwd_split_x2<L>(za, ma, zb, mb, t, false, v);
  fwd_fft_post_x2<L, GENERAL, false>(v, s, a, a.out + (long long)blockIdx.z * a.out_bstride, k1, k1 + 1, packed, t, g, pi);
}

// Inverse four-read preprocess (Eq. 2d_idct_pre, conjugated twiddle, 1/(N1 N2)
// in the a-table) of one item, from C(k1,k2), C(kmir,k2), C(k1,N2-k2) and
// C(kmir,N2-k2) (zero past the edge).  The kind's maps are folded into the reads:
// DST-II reads rows N1-1-k and columns reversed; IDCT_IDXST swaps the reads at
// k2 and N2-k2 (column 0 zero); IDXST_IDCT swaps the item's two rows (row 0 zero).
struct InvRows {
  const float* ra;  // row of c1 / c4 (null: zero row)
  const float* rb;  // row of c3 / c2
};

// Input rows of item k (rows L floats apart).
__device__ __forceinline__ InvRows inv_rows_of(const Dct2dArgs& a, const float* C, int k, int L, int vkind) {
  const int N1 = a.n1;
  const int kmir = row_mirror(k, N1);
  int r0 = k, r1 = kmir;
  if (vkind == 1) {
    r0 = N1 - 1 - k;
    r1 = N1 - 1 - kmir;
  }
  InvRows r{C + (long long)r0 * L, C + (long long)r1 * L};
  if (vkind == 3) {
    if (k) {
      const float* t = r.ra;
      r.ra = r.rb;
      r.rb = t;
    } else {
      r.ra = nullptr;
    }
  }
  return r;
}

// Reads of one item's two rows, first (c1, c4) and second (c3, c2), at a column:
// from global memory with the L2 policy, or (STAGED) from copies of the rows
// already in shared memory.
template <bool STAGED>
struct RowReads {
  InvRows r;
  uint64_t pol;
  __device__ __forceinline__ bool has_a() const { return r.ra != nullptr; }
  __device__ __forceinline__ float a(int c) const { return STAGED ? r.ra[c] : l2::ld(r.ra + c, pol); }
  __device__ __forceinline__ float b(int c) const { return STAGED ? r.rb[c] : l2::ld(r.rb + c, pol); }
};

// The reads of columns k2 and km = L - k2 of one item (edge: k2 = 0, whose
// mirror reads are zero); ROW0: the item's first row may be missing (zero).
template <int L, bool MAPPED, bool ROW0, typename Reads>
__device__ __forceinline__ rowp::Quad inv_quad(const Reads& r, int k2, int km, bool edge, bool rev, bool swapc) {
  const bool has = !ROW0 || r.has_a();
  rowp::Quad q;
  if constexpr (!MAPPED) {
    q.c1 = has ? r.a(k2) : 0.f;
    q.c3 = r.b(k2);
    q.c4 = (has && !edge) ? r.a(km) : 0.f;
    q.c2 = !edge ? r.b(km) : 0.f;
  } else {
    const int ka = swapc ? km : k2, kb = swapc ? k2 : km;
    const int pa = rev ? L - 1 - ka : ka, pb = rev ? L - 1 - kb : kb;
    const bool z0 = swapc && edge;
    q.c1 = (has && !z0) ? r.a(pa) : 0.f;
    q.c3 = !z0 ? r.b(pa) : 0.f;
    q.c4 = (has && !edge) ? r.a(pb) : 0.f;
    q.c2 = !edge ? r.b(pb) : 0.f;
  }
  return q;
}

// Preprocess of both items: points t + TPS j of the returned butterfly t in v.
template <int L, bool MAPPED, bool FIRST, bool EXACT, typename Reads>
__device__ __forceinline__ int inv_pre_x2(const Dct2dArgs& a, const Reads& A, const Reads& B, int vkind, int k1, int kb,
                                          bool packed, int g, soa::C2* v) {
  const bool rev = MAPPED && vkind == 1, swapc = MAPPED && vkind == 2;
  auto quads = [&](int k2, int km, bool edge, rowp::Quad& qa, rowp::Quad& qb) {
    qa = inv_quad<L, MAPPED, FIRST>(A, k2, km, edge, rev, swapc);
    qb = inv_quad<L, MAPPED, false>(B, k2, km, edge, rev, swapc);
  };
  return rowp::inv_pre<L, FIRST, EXACT>(quads, a.ib, a.ib4, __ldg(a.ia + k1), __ldg(a.ia + kb),
                                        __ldg(a.ia + a.n1 / 2), packed, g, v);
}

// Inverse pairing of both items: row IFFT u in the registers of the last stage ->
// workspace rows k1 and its mirror: Z(k1, p) = u(p) + i u(L-1-p), Z(kmir, p) =
// conj(u(p)) + i conj(u(L-1-p)), the pairs of points p and L-1-p as rowp::inv_pairs
// joins them; packed lane a: the real and imaginary parts go to rows 0 and N1/2.
template <int L>
__device__ __forceinline__ void inv_pair_x2(const soa::C2* v, const Dct2dArgs& a, float2* Zw, int k1, bool packed,
                                            int g) {
  float2* za = Zw + (long long)fs2_prow(k1, a.fsA, a.fsB) * (L / 2);
  float2* ma = Zw + (long long)fs2_prow(row_mirror(k1, a.n1), a.fsA, a.fsB) * (L / 2);
  float2* zb = Zw + (long long)fs2_prow(k1 + 1, a.fsA, a.fsB) * (L / 2);
  float2* mb = Zw + (long long)fs2_prow(row_mirror(k1 + 1, a.n1), a.fsA, a.fsB) * (L / 2);
  const uint64_t pol = l2::evict_last();  // read again by the next column step
  rowp::inv_pairs<L>(v, g, [&](int base, int off, const soa::C2& u, const soa::C2& w) {
    l2::st(zb + base + off, make_float2(u.re.y - w.im.y, u.im.y + w.re.y), pol);
    l2::st(mb + base + off, make_float2(u.re.y + w.im.y, w.re.y - u.im.y), pol);
    l2::st(za + base + off,
           packed ? make_float2(u.re.x, w.re.x) : make_float2(u.re.x - w.im.x, u.im.x + w.re.x), pol);
    l2::st(ma + base + off,
           packed ? make_float2(u.im.x, w.im.x) : make_float2(u.re.x + w.im.x, w.re.x - u.im.x), pol);
  });
}

// MAPPED: the DST-II / IDCT_IDXST index maps folded into the reads (a separate
// instantiation, so the plain DCT-II inverse carries no code for them).
template <int L, bool MAPPED>
__global__ void __launch_bounds__(RowX2Geom<L>::THREADS, RowX2Geom<L>::MINB_INV) k_fs2_rows_inv_x2(Dct2dArgs a) {
  using R = RowX2Geom<L>;
  extern __shared__ float4 sxi[];
  const int pi = threadIdx.x / R::TPS, g = threadIdx.x % R::TPS;
  float4* s = sxi + pi * R::LP;
  const int k1 = 2 * (blockIdx.x * R::NP + pi);
  const float* C = a.in + (long long)blockIdx.z * a.in_bstride;
  const uint64_t pol = l2::evict_first();  // the input is streamed in
  const RowReads<false> A{inv_rows_of(a, C, k1, L, a.vkind), pol}, B{inv_rows_of(a, C, k1 + 1, L, a.vkind), pol};
  const bool packed = (k1 == 0);
  pdl::wait_prior_grid();
  soa::C2 v[16];
  int t;
  if (rowp::warp_has_first<R::TPS>(packed))
    t = inv_pre_x2<L, MAPPED, true, false>(a, A, B, a.vkind, k1, k1 + 1, packed, g, v);
  else
    t = inv_pre_x2<L, MAPPED, false, false>(a, A, B, a.vkind, k1, k1 + 1, false, g, v);
  soa::first_stage<L, true>(v, s, t);
  rowp::stages_to_regs<L, 16, true, false, false>(s, g, pi, a.tw2x, v);
  pdl::launch_dependents();
  float2* Zw = a.work + (long long)blockIdx.z * a.work_bstride;
  if (rowp::warp_has_first<R::TPS>(packed))
    inv_pair_x2<L>(v, a, Zw, k1, packed, g);
  else
    inv_pair_x2<L>(v, a, Zw, k1, false, g);
}

}  // namespace gbdct
