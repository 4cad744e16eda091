// dct2d_tp_kernels.cuh - two-pass family: each direction of the 2D DCT is two
// launches (a column pass and a row pass), the column FFT of length N1 split
// once by decimation in time.
//
// Method: arXiv 2110.01172, Algorithm 2 (reorder, 2D real FFT, postprocess)
// with the fused pre/postprocess of Section III, as in the four-step family
// (dct2d_fs2_kernels.cuh); only the column FFT is organised differently.  With
// M = N1/2 and v the row-reordered input (Eq. 2d_dct_pre), the column DFT of
// length N1 is (radix-2 decimation in time)
//   V[k] = E[k mod M] + W_N1^k O[k mod M],  E = DFT_M(v[2m]),  O = DFT_M(v[2m+1]).
// The column pass computes E and O: a CTA owns a strip of NP complex column
// pairs (NP * 16 bytes of every row) and all M rows of one parity, so the whole
// half-length column FFT runs in shared memory and only E and O are written.
// The row pass applies the radix-2 step while it loads: item k1 needs rows k1
// and N1-k1 of V, and pairing item k1 with item M-k1 makes the four rows of a
// two-item group come from exactly four workspace rows (w = W_N1^k1):
//   V[k1]    = E[k1]   + w O[k1]          V[M+k1] = E[k1]   - w O[k1]
//   V[N1-k1] = E[M-k1] + conj(w) O[M-k1]  V[M-k1] = E[M-k1] - conj(w) O[M-k1]
// The first group pairs the packed item 0 (rows 0 and M = E[0] +- O[0]) with
// item M/2 (rows M/2 and 3M/2 = E[M/2] +- W_N1^{M/2} O[M/2]).
// The inverse is the mirror image: the inverse row pass ends with
//   E'[k] = V[k] + V[M+k],  O'[k] = W_N1^{-k} (V[k] - V[M+k])   (k < M)
// and the inverse column pass takes IDFT_M of E' and O' to the even and odd
// positions of the reordered sequence, stored with the inverse reorder of
// Eq. (2d_idct_post).
//
// Workspace: N1 rows of N2/2 complex; rows [0, M) hold E (E'), rows [M, N1) O (O').
// Supported: N1 in {128, ..., 8192}, N2 in {128, ..., 8192}; default plans (above 16384
// values) and the solves of gbdct_poisson.cu also run sides of 64, with exact kernels
// (Dct2dArgs::exact).
#pragma once

#include "dct2d_fs2_kernels.cuh"
#include "launch_dep.cuh"
#include "tma_util.cuh"

namespace gbdct {

// ----------------------------------------------------------------------------
// Column pass.  A column pair (two adjacent complex columns, one float4 per
// row) is one two-lane sequence of the SoA engine (fft_soa.cuh); the NP pairs
// of a CTA are interleaved point by point in shared memory and thread
// t = g * NP + pi is rank g of pair pi, so a warp's loads and stores cover
// 32/NP rows x NP*16 contiguous bytes.  NP (the strip width, a tile
// parameter the autotuner can choose) keeps the CTA at 64 to 512 threads
// and its shared memory within one SM.
// ----------------------------------------------------------------------------
template <int M, int NP_>
struct TpColGeom {
  static constexpr int TPS = fft_tps(M);  // threads per column pair
  static constexpr int NP = NP_;          // column pairs per CTA
  static constexpr int THREADS = NP * TPS;
  static constexpr int LP = M + M / 16;   // padded points per pair
  static constexpr size_t SMEM = (size_t)NP * LP * sizeof(float4);
  // CTAs per SM: three at 256 threads (80 registers, a few spilled) measured
  // faster than two at 128 registers (4096^2: 35.5 / 33.3 us vs 37.6 / 37.4),
  // the CTAs' strip loads overlapping the others' FFTs; else 128 registers
  static constexpr int MINB = THREADS == 256 ? 3 : (THREADS <= 512 ? 512 / THREADS : 1);
  static constexpr bool VALID = THREADS >= (M == 32 ? 32 : 64) && THREADS <= 512 && SMEM <= 227 * 1024 - 256;
  // widths the default rule can pick, which a Poisson solve runs
  static constexpr bool POISSON = VALID && (THREADS <= 128 || NP == 2);
  // bulk tensor copy form: + 128-byte alignment slack, the mbarrier and a flag
  static constexpr size_t SMEM_TMA = SMEM + 256;
  static constexpr int HALF = M / 2;                    // rows of one reorder residue
  static constexpr int ZB = HALF < 256 ? HALF : 256;    // rows per tensor copy (box height)
};
// Default strip width: 128 threads per CTA, but at least two column pairs
// (32 bytes of every row); measured fastest at every size (4096^2: NP = 2,
// 256 threads, 74 / 76 us vs 87 / 87 us at 512 threads).
__host__ __device__ constexpr int tp_default_np(int M) { return 128 / fft_tps(M) > 2 ? 128 / fft_tps(M) : 2; }

__device__ __forceinline__ soa::C2 aos_to_soa(float4 q) { return {make_float2(q.x, q.z), make_float2(q.y, q.w)}; }
__device__ __forceinline__ float4 soa_to_aos(soa::C2 y) { return make_float4(y.re.x, y.im.x, y.re.y, y.im.y); }

// Forward (INV = false): reorder + E or O (blockIdx.y = parity of the
// reordered row) -> workspace.  Inverse: E' or O' -> IDFT_M -> output rows
// with the inverse reorder.
template <int M, int NP, bool INV, bool POIS, bool EXACT>
__global__ void __launch_bounds__(TpColGeom<M, NP>::THREADS, TpColGeom<M, NP>::MINB)
    k_tp_cols(Dct2dArgs a, PoissonArgs ps) {
  using G = TpColGeom<M, NP>;
  constexpr int TPS = G::TPS;
  extern __shared__ float4 stc[];
  const int pi = threadIdx.x % G::NP, g = threadIdx.x / G::NP;
  const int par = blockIdx.y;
  const int vcol = blockIdx.x * G::NP + pi;  // float4 column of the strip
  const int N1 = 2 * M;
  const long long hv = a.n2 / 4;             // float4 per row (input, output and workspace)
  float4* W = reinterpret_cast<float4*>(a.work + (long long)blockIdx.z * a.work_bstride) + (long long)par * M * hv +
              vcol;
  float4* s = stc + pi;
  const uint64_t pol_stream = l2::evict_first();
  pdl::wait_prior_grid();
  soa::C2 v[16];
  if constexpr (!INV) {
    const float4* xin = reinterpret_cast<const float4*>(a.in + (long long)blockIdx.z * a.in_bstride) + vcol;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int row = reorder_src(2 * (g + TPS * j) + par, N1);
      float4 q = l2::ld_once(xin + (long long)row * hv, pol_stream);
      if (a.vkind == 1) {  // DST-II: (-1)^(n1 + n2); real columns alternate in parity
        const float sr = (row & 1) ? -1.f : 1.f;
        q = vsign(q, sr, -sr);
      }
      v[j] = aos_to_soa(q);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = aos_to_soa(l2::ld_once(W + (long long)(g + TPS * j) * hv, pol_stream));
  }
  soa::first_stage<M, INV, G::NP>(v, s, g);
  __syncthreads();
  soa::stages<M, 16, INV, G::NP, 0, EXACT>(s, g, a.tw1x);
  pdl::launch_dependents();
  if constexpr (!INV) {
    const uint64_t pol_keep = l2::work_policy(a.stream_work);  // read again by the row pass
#pragma unroll 4
    for (int r = 0; r < 16; ++r) {
      const int k = g + TPS * r;
      l2::st(W + (long long)k * hv, soa_to_aos(soa::unpack(s[G::NP * soa::pidx4(k)])), pol_keep);
    }
  } else {
    const int vkind = POIS ? poisson_vkind(blockIdx.z) : a.vkind;
    float* out = a.out + (long long)blockIdx.z * a.out_bstride;
    if constexpr (POIS) out = blockIdx.z == 0 ? ps.out[0] : blockIdx.z == 1 ? ps.out[1] : ps.out[2];
    float4* xo = reinterpret_cast<float4*>(out) + vcol;
#pragma unroll 4
    for (int r = 0; r < 16; ++r) {
      const int m = g + TPS * r;
      const int row = reorder_src(2 * m + par, N1);
      float4 y = soa_to_aos(soa::unpack(s[G::NP * soa::pidx4(m)]));
      if (vkind) {  // output signs: (-1)^(n1+n2) DST-II, (-1)^n2 IDCT_IDXST, (-1)^n1 IDXST_IDCT
        const float sr = (vkind != 2 && (row & 1)) ? -1.f : 1.f;
        const float sc = (vkind != 3) ? -sr : sr;
        y = vsign(y, sr, sc);
      }
      l2::st(xo + (long long)row * hv, y, pol_stream);
    }
  }
}

// The same pass with the strip moved by bulk tensor copies (TMA) instead of
// per-thread loads and stores, which at 16 * NP bytes per row would cost the
// LSU one wavefront per row touched.  The reorder makes the M rows of one
// parity two regular row sets: with the input viewed as (x, row % 4, row / 4,
// batch), the first half of the reordered positions (m < M/2) is row 4m + 2par
// (residue 2par, z = m) and the second half is row 2N1 - 4m - 2par - 1
// (residue 3 - 2par, z = M - 1 - m), so each is a run of boxes of ZB rows at
// one residue.  The strip lands dense in shared memory (second half in z
// order), the threads take their points from there, and the last FFT stage
// writes its outputs dense (inverse: second half reversed) and interleaved
// (re_a, im_a, re_b, im_b) for the bulk tensor stores.  mx: 4D map of the input (forward) or output (inverse), box
// {4 NP, 1, ZB, 1}; mw: 3D map of the workspace (x, row, batch), box
// {4 NP, ZB, 1}.  One thread issues the copies and waits on the mbarrier
// (bounded; a wait that gives up records the device error, waits again for
// the copies to land and leaves the strip unwritten).
__device__ __forceinline__ float4* align128(float4* p) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  return reinterpret_cast<float4*>((a + 127) & ~uintptr_t(127));
}

// POIS: batch entry z of the workspace goes to output array z (its own map, one
// array each), with that entry's kind.
template <int N>
struct ColMaps {
  CUtensorMap x[N];  // input (forward) or output (inverse)
  CUtensorMap w;     // workspace
};

template <int M, int NP, bool INV, bool POIS, bool EXACT>
__global__ void __launch_bounds__(TpColGeom<M, NP>::THREADS, TpColGeom<M, NP>::MINB)
    k_tp_cols_tma(Dct2dArgs a, const __grid_constant__ ColMaps<POIS ? 3 : 1> maps) {
  using G = TpColGeom<M, NP>;
  constexpr int TPS = G::TPS, HALF = G::HALF, ZB = G::ZB;
  extern __shared__ float4 stt_raw[];
  float4* buf = align128(stt_raw);
  uint64_t* bar = reinterpret_cast<uint64_t*>(buf + NP * G::LP);
  int* flag = reinterpret_cast<int*>(bar + 1);
  const int pi = threadIdx.x % NP, g = threadIdx.x / NP;
  const int par = blockIdx.y, b = blockIdx.z;
  const CUtensorMap& mx = maps.x[POIS ? b : 0];
  const CUtensorMap& mw = maps.w;
  const int xb = POIS ? 0 : b;  // batch coordinate within the input or output map
  const int vkind = POIS ? poisson_vkind(b) : a.vkind;
  const int x0 = blockIdx.x * NP * 4;  // first float column of the strip
  if (threadIdx.x == 0) {
    tma::bar_init(bar, 1);
    tma::fence_barrier_init();
  }
  pdl::wait_prior_grid();
  if (threadIdx.x == 0) {
    tma::bar_expect_tx(bar, (uint32_t)(M * NP * sizeof(float4)));
    const uint64_t pol = l2::evict_first();  // input streamed once / last use of the workspace
    if constexpr (!INV) {
      for (int z = 0; z < HALF; z += ZB) {
        tma::load_4d(buf + z * NP, &mx, x0, 2 * par, z, xb, bar, pol);
        tma::load_4d(buf + (HALF + z) * NP, &mx, x0, 3 - 2 * par, z, xb, bar, pol);
      }
    } else {
      for (int z = 0; z < M; z += ZB) tma::load_3d(buf + z * NP, &mw, x0, par * M + z, b, bar, pol);
    }
    const uint32_t polls = a.polls ? a.polls : tma::kDefaultPolls;
    int ok = tma::bar_wait_from_issue(bar, 0, polls);
    if (!ok) {
      atomicExch(a.err, 1);
      tma::bar_wait(bar, 0, tma::kDefaultPolls);  // the copies must land before the CTA exits
    }
    *flag = ok;
  }
  __syncthreads();
  if (!*flag) return;
  // every thread observes the completed phase (acquire of the copied data);
  // it has completed, so the first, non-blocking poll succeeds
  if (threadIdx.x) tma::test_wait(bar, 0);
  soa::C2 v[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int m = g + TPS * j;  // in the first half for j < 8
    if constexpr (!INV) {
      float4 q = j < 8 ? buf[NP * m + pi] : buf[NP * (3 * HALF - 1 - TPS * j) + pi - NP * g];
      if (a.vkind == 1) {  // DST-II: (-1)^(n1 + n2); rows of the first half even, second half odd
        const float sr = j < 8 ? 1.f : -1.f;
        q = vsign(q, sr, -sr);
      }
      v[j] = aos_to_soa(q);
    } else {
      v[j] = aos_to_soa(buf[NP * m + pi]);
    }
  }
  __syncthreads();
  float4* s = buf + pi;
  soa::first_stage<M, INV, NP>(v, s, g);
  __syncthreads();
  soa::stages<M, 16, INV, NP, INV ? 2 : 1, EXACT>(s, g, a.tw1x);
  if constexpr (INV) {
    if (vkind) {  // output signs: (-1)^(n1+n2) DST-II, (-1)^n2 IDCT_IDXST, (-1)^n1 IDXST_IDCT
#pragma unroll 4
      for (int r = 0; r < 16; ++r) {
        const int pos = g + TPS * r;  // slots of the second half hold odd rows
        const float sr = (vkind != 2 && pos >= HALF) ? -1.f : 1.f;
        const float sc = (vkind != 3) ? -sr : sr;
        buf[NP * pos + pi] = vsign(buf[NP * pos + pi], sr, sc);
      }
    }
  }
  tma::fence_proxy_async();
  __syncthreads();
  pdl::launch_dependents();
  if (threadIdx.x == 0) {
    if constexpr (!INV) {
      const uint64_t pol = l2::work_policy(a.stream_work);  // read again by the row pass
      for (int z = 0; z < M; z += ZB) tma::store_3d(&mw, buf + z * NP, x0, par * M + z, b, pol);
    } else {
      const uint64_t pol = l2::evict_first();
      for (int z = 0; z < HALF; z += ZB) {
        tma::store_4d(&mx, buf + z * NP, x0, 2 * par, z, xb, pol);
        tma::store_4d(&mx, buf + (HALF + z) * NP, x0, 3 - 2 * par, z, xb, pol);
      }
    }
    tma::commit_group();
    tma::wait_group_read();
  }
}

// ----------------------------------------------------------------------------
// Row passes (L = N2), two items per thread group as in the four-step family:
// group c pairs item c (lane a; the packed item 0 when c = 0) with item
// M - c (lane b; item M/2 when c = 0).
// ----------------------------------------------------------------------------
__device__ __forceinline__ int tp_item_b(int c, int M) { return c ? M - c : M / 2; }

// Row-pass geometry: NP item pairs per CTA, TPS = L/16 threads each.  Wide
// CTAs have 256 threads (the four-step family's row geometry); narrow ones 64,
// for grids that would otherwise leave SMs idle (a single transform with few
// rows: 1024^2 has 256 item pairs, 64 wide CTAs for 152 SMs).  SMEM_STAGED
// adds one 8-byte barrier per group and the CTA's 4-byte flag (16 bytes of
// slack) for the inverse pass's staged rows.  (Staging the forward row pass's
// workspace rows the same way measured slower, 36.2 vs 33.5 us at 4096^2: its
// loads already hit L2 and are read once.)
template <int L, bool NARROW>
struct TpRows {
  static constexpr int TPS = fft_tps(L);
  static constexpr int NP = ((NARROW ? 64 : 256) / TPS) > 0 ? (NARROW ? 64 : 256) / TPS : 1;
  static constexpr int THREADS = NP * TPS;
  static constexpr int LP = L + L / 16;
  static constexpr size_t SMEM = (size_t)NP * LP * sizeof(float4);
  static constexpr size_t SMEM_STAGED = SMEM + (((size_t)NP * 8 + 16 + 15) & ~size_t(15));
  static constexpr size_t SMEM_DEN = SMEM_STAGED + (size_t)NP * 16 * L;  // + a Poisson solve's denominators
  static constexpr int MINB = THREADS >= 512 ? 1 : 512 / THREADS;  // up to 128 registers
};

// The radix-2 twiddles of a group: forward W_N1^c on O[c] and W_N1^-c on O[kb] (first
// group: 1 and W_N1^{M/2}), inverse W_N1^-c and -W_N1^c on the differences (1 and i).
// REST: with the rests that the table's rounding left, both products in one packed
// multiplication.
template <bool INV, bool REST>
struct R2 {
  float2 w1, w2;       // without rests: the two twiddles (inverse: w1 for both)
  soa::C2 w, r;        // with rests: lane by lane
  bool first;

  __device__ __forceinline__ R2(const Dct2dArgs& a, int c, bool f) : first(f) {
    const int k = !INV && f ? a.n1 / 4 : c;
    const float2 t = __ldg(a.r2w + k);
    if constexpr (!REST) {
      w1 = !INV && f ? make_float2(1.f, 0.f) : t;
      w2 = f ? t : conjf2(t);
    } else {
      const float2 u = __ldg(a.r2r + k);
      if constexpr (!INV) {
        w = f ? soa::C2{make_float2(1.f, t.x), make_float2(0.f, t.y)} : soa::C2{soa::bc(t.x), make_float2(t.y, -t.y)};
        r = f ? soa::C2{make_float2(0.f, u.x), make_float2(0.f, u.y)} : soa::C2{soa::bc(u.x), make_float2(u.y, -u.y)};
      } else {
        w = f ? soa::C2{make_float2(1.f, 0.f), make_float2(0.f, 1.f)} : soa::C2{make_float2(t.x, -t.x), soa::bc(-t.y)};
        r = f ? soa::C2{soa::bc(0.f), soa::bc(0.f)} : soa::C2{make_float2(u.x, -u.x), soa::bc(-u.y)};
      }
    }
  }
  __device__ __forceinline__ void mul(float2& a, float2& b) const {
    if constexpr (REST) {
      const soa::C2 o = soa::mulw(soa::C2{make_float2(a.x, b.x), make_float2(a.y, b.y)}, w.re, w.im, r.re, r.im);
      a = make_float2(o.re.x, o.im.x);
      b = make_float2(o.re.y, o.im.y);
    } else if constexpr (!INV) {
      a = cmul(a, w1);
      b = cmul(b, w2);
    } else {
      a = first ? a : cmulc(a, w1);
      b = first ? make_float2(-b.y, b.x) : cmul(make_float2(-b.x, -b.y), w1);
    }
  }
};

// The thread's points of both items in v, straight from the group's four
// workspace rows (SMEM: in shared memory).
template <int L, bool FIRST, bool SMEM, bool REST>
__device__ __forceinline__ void tp_fwd_load(const float2* e1r, const float2* o1r, const float2* e2r, const float2* o2r,
                                            const R2<false, REST>& w, bool first, int t, soa::C2* v) {
  constexpr int TPS = fft_tps(L);
  constexpr int MASK = rowp::rev_lane_mask<TPS>();
  const uint64_t pol = l2::evict_first();  // last use of the workspace
  auto ld = [&](const float2* r) { return SMEM ? *r : l2::ld_once(r, pol); };
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int p = t + TPS * j;
    const float2 e1 = ld(e1r + p), e2 = ld(e2r + p);
    float2 o1 = ld(o1r + p), o2 = ld(o2r + p);
    w.mul(o1, o2);
    const float2 P = cadd(e1, o1), Q = csub(e1, o1), Rr = cadd(e2, o2), S = csub(e2, o2);
    // (z_a, m_a, z_b, m_b) = (V[c], V[N1-c], V[M-c], V[M+c]); first group:
    // (V[0], V[M], V[M/2], V[3M/2])
    const bool f = FIRST && first;
    const float2 Am = f ? Q : Rr, B = f ? Rr : S, Bm = f ? S : Q;
    split_point<MASK>(P, Am, B, Bm, f, v[j], v[15 - j]);
  }
}

// The group's finished rows gathered in its shared buffer and stored whole by the
// CTA, for outputs that are not device memory: the registers' stores cover L/16
// columns at a time, which L2 joins but the host link does not (device to page-locked
// host memory, stored from registers / gathered: 64 x (512 x 64) 230 / 53 us, 64 x (512
// x 128) 292 / 98).
template <int L, bool NARROW, bool EXACT>
__device__ __forceinline__ void tp_fwd_gathered(soa::C2* v, float4* smem, const Dct2dArgs& a, int c, int kb, bool first,
                                                int g, int pi) {
  using R = TpRows<L, NARROW>;
  float* st = reinterpret_cast<float*>(smem + pi * R::LP);  // 4 L of its 4.25 L floats
  rowp::group_sync<R::TPS>(pi);                             // the rows overlay the points of the last stage
  fwd_post_x2<L, true, true, EXACT>(
      v, a, [&] { return OutRows{st, st + L, st + 2 * L, st + 3 * L}; }, c, kb, first, g);
  __syncthreads();
  float* y = a.out + (long long)blockIdx.z * a.out_bstride;
  const uint64_t pol = l2::evict_first();
#pragma unroll 4
  for (int i = 0; i < R::NP * L / R::THREADS; ++i) {
    const int f = threadIdx.x + R::THREADS * i, row = f / (L / 4), col = f % (L / 4), slot = row & 3;
    const int cc = blockIdx.x * R::NP + row / 4, item = slot < 2 ? cc : tp_item_b(cc, a.n1 / 2);
    const int k = fwd_out_row(item, slot & 1, a.n1, a.vkind == 1);
    l2::st(reinterpret_cast<float4*>(y + (long long)k * L) + col, smem[row / 4 * R::LP + slot * (L / 4) + col], pol);
  }
}

// GENERAL: plans with the DST-II order or a magnitude threshold (row_pairs.cuh).
// HOST: the output is not device memory.
template <int L, bool NARROW, bool GENERAL, bool EXACT, bool HOST>
__global__ void __launch_bounds__(TpRows<L, NARROW>::THREADS, TpRows<L, NARROW>::MINB) k_tp_rows_fwd(Dct2dArgs a) {
  using R = TpRows<L, NARROW>;
  constexpr int TPS = R::TPS;
  extern __shared__ float4 sxt[];
  const int pi = threadIdx.x / TPS, g = threadIdx.x % TPS;
  float4* s = sxt + pi * R::LP;
  const int M = a.n1 / 2;
  const int c = blockIdx.x * R::NP + pi;
  const bool first = (c == 0);
  const int kb = tp_item_b(c, M);
  const float2* Zw = a.work + (long long)blockIdx.z * a.work_bstride;
  const float2* e1r = Zw + (long long)c * (L / 2);
  const float2* o1r = Zw + (long long)(M + c) * (L / 2);
  const float2* e2r = Zw + (long long)kb * (L / 2);
  const float2* o2r = Zw + (long long)(M + kb) * (L / 2);
  const R2<false, EXACT> w(a, c, first);
  const int t = rowp::rev_lane_butterfly<TPS>(g);
  pdl::wait_prior_grid();
  soa::C2 v[16];
  if (rowp::warp_has_first<TPS>(first))
    tp_fwd_load<L, true, false, EXACT>(e1r, o1r, e2r, o2r, w, first, t, v);
  else
    tp_fwd_load<L, false, false, EXACT>(e1r, o1r, e2r, o2r, w, false, t, v);
  if constexpr (HOST) {
    soa::first_stage<L, false>(v, s, t);
    rowp::stages_to_regs<L, 16, false, true, EXACT>(s, g, pi, a.tw2x, v);
    pdl::launch_dependents();
    tp_fwd_gathered<L, NARROW, EXACT>(v, sxt, a, c, kb, first, g, pi);
  } else {
    fwd_fft_post_x2<L, GENERAL, EXACT>(v, s, a, a.out + (long long)blockIdx.z * a.out_bstride, c, kb, first, t, g, pi);
  }
}

// Inverse pairing of both items into E' / O' rows: from the row IFFT u in v,
// Z(k, p) of the items' rows as in the four-step family's pairing, then
//   E'[c] = V[c] + V[M+c],      O'[c] = conj(w) (V[c] - V[M+c])
//   E'[M-c] = V[M-c] + V[N1-c], O'[M-c] = w (V[N1-c] - V[M-c])
// and for the first group E'[0], O'[0] from V[0] +- V[M], E'[M/2] = V[M/2] +
// V[3M/2], O'[M/2] = i (V[M/2] - V[3M/2]).
// Rows of Zw are `stride` complex values apart (SMEM: in shared memory).
template <int L, bool SMEM, bool REST>
__device__ __forceinline__ void tp_inv_pair(const soa::C2* v, const Dct2dArgs& a, float2* Zw, long long stride, int c,
                                            int kb, bool first, int g) {
  const int M = a.n1 / 2;
  float2* e1r = Zw + c * stride;
  float2* o1r = Zw + (M + c) * stride;
  float2* e2r = Zw + kb * stride;
  float2* o2r = Zw + (M + kb) * stride;
  const R2<true, REST> cw(a, c, first);
  const uint64_t pol = l2::work_policy(a.stream_work);  // read again by the column pass
  rowp::inv_pairs<L>(v, g, [&](int base, int off, const soa::C2& u, const soa::C2& w) {
    const float2 zb0 = make_float2(u.re.y - w.im.y, u.im.y + w.re.y);  // V[kb]
    const float2 zb1 = make_float2(u.re.y + w.im.y, w.re.y - u.im.y);  // V[mirror of kb]
    const float2 za0 = first ? make_float2(u.re.x, w.re.x) : make_float2(u.re.x - w.im.x, u.im.x + w.re.x);
    const float2 za1 = first ? make_float2(u.im.x, w.im.x) : make_float2(u.re.x + w.im.x, w.re.x - u.im.x);
    const float2 x1 = first ? za1 : zb1;  // V[c + M]
    const float2 x2 = first ? zb1 : za1;  // V[kb + M]
    float2 o1 = csub(za0, x1), o2 = csub(zb0, x2);
    cw.mul(o1, o2);
    auto st = [&](float2* p, float2 z) {
      if constexpr (SMEM)
        *p = z;
      else
        l2::st(p, z, pol);
    };
    st(e1r + base + off, cadd(za0, x1));
    st(o1r + base + off, o1);
    st(e2r + base + off, cadd(zb0, x2));
    st(o2r + base + off, o2);
  });
}

// STAGED: the group's (up to) four input rows are first copied whole into its
// shared buffer by contiguous bulk copies (one mbarrier per group, bounded
// wait as in the column pass), so few registers hold loads in flight; the
// buffer (17 L bytes) holds the 16 L bytes of the rows until the first FFT
// stage overwrites it.  Device buffers only.  Otherwise the preprocess loads
// its points straight from global memory, every value once: faster for short
// rows, whose groups would all wait for the slowest group's copies (inverse,
// staged vs direct: 25 x 512^2 22.3 vs 20.6 us, 64 x 256^2 13.9 vs 13.5, 1024^2
// 8.9 vs 8.6, 2048^2 17.5 vs 17.3, but 4096^2 62.3 vs 63.3).  A Poisson solve,
// which also loads a denominator for every value, stages at every length (512^2
// 19.8 vs 21.0 us per call).
template <int L>
constexpr bool tp_inv_staged() { return L >= 4096; }

// The scaled reads of entry Z of a Poisson solve: RowReads' value times the
// eigenvalue denominator and (entry 1) the row's wu or (entry 2) the column's wv.
// DEN: the denominators' rows are in shared memory, `den` floats behind the
// values' rows.
template <bool STAGED, bool DEN, int Z>
struct PoissonReads {
  RowReads<STAGED> r;
  const float *ia, *ib;  // the denominators of the two rows
  const float* wv;       // entry 2
  float ua, ub;          // entry 1: wu of the two rows
  __device__ __forceinline__ PoissonReads(const RowReads<STAGED>& reads, const InvRows& src, const float* spectrum,
                                          const PoissonArgs& ps, int n1, int L, int den)
      : r(reads), ia(src.ra ? ps.inv + (src.ra - spectrum) : nullptr), ib(ps.inv + (src.rb - spectrum)),
        wv(ps.w + n1), ua(1.f), ub(1.f) {
    if constexpr (Z == 1) {
      if (src.ra) ua = __ldg(ps.w + (src.ra - spectrum) / L);
      ub = __ldg(ps.w + (src.rb - spectrum) / L);
    }
    if constexpr (DEN) {
      ia = src.ra ? reads.r.ra + den : nullptr;
      ib = reads.r.rb + den;
    }
  }
  __device__ __forceinline__ bool has_a() const { return ia != nullptr; }
  __device__ __forceinline__ float scaled(float v, const float* i, int c, float u) const {
    v *= DEN ? i[c] : __ldg(i + c);
    if constexpr (Z == 1) v *= u;
    if constexpr (Z == 2) v *= __ldg(wv + c);
    return v;
  }
  __device__ __forceinline__ float a(int c) const { return scaled(r.a(c), ia, c, ua); }
  __device__ __forceinline__ float b(int c) const { return scaled(r.b(c), ib, c, ub); }
};

// Whether a Poisson solve's staged rows take the denominators' rows with them:
// in narrow CTAs, whose solves are bound by latency (the copies leave while the
// forward transform finishes; with each entry's kind and factors as constants,
// GPU time of a solve 256^2 18.5 -> 15.7 us, 512^2 18.3 -> 16.9, 1024^2 25.7 ->
// 24.0); wide ones would be left with one CTA per SM.
template <int L, bool NARROW>
constexpr bool tp_den_staged() { return NARROW && L <= 2048; }

// Preprocess of a group from its rows' reads.
template <int L, bool MAPPED, bool EXACT, typename Reads>
__device__ __forceinline__ int tp_inv_pre(const Dct2dArgs& a, const Reads& A, const Reads& B, int vkind, int c, int kb,
                                          bool first, int g, soa::C2* v) {
  return rowp::warp_has_first<fft_tps(L)>(first)
             ? inv_pre_x2<L, MAPPED, true, EXACT>(a, A, B, vkind, c, kb, first, g, v)
             : inv_pre_x2<L, MAPPED, false, EXACT>(a, A, B, vkind, c, kb, false, g, v);
}

// The same for a Poisson solve: its entries' kinds and factors as constants.
template <int L, bool STAGED, bool DEN, bool EXACT>
__device__ __forceinline__ int tp_poisson_pre(const Dct2dArgs& a, const PoissonArgs& ps, const RowReads<STAGED>& A,
                                              const RowReads<STAGED>& B, const InvRows& srcA, const InvRows& srcB,
                                              const float* C, int den, int c, int kb, bool first, int g, soa::C2* v) {
  auto pre = [&](auto zc) {
    constexpr int Z = decltype(zc)::value;
    return tp_inv_pre<L, Z == 2, EXACT>(a, PoissonReads<STAGED, DEN, Z>(A, srcA, C, ps, a.n1, L, den),
                                 PoissonReads<STAGED, DEN, Z>(B, srcB, C, ps, a.n1, L, den), poisson_vkind(Z), c, kb,
                                 first, g, v);
  };
  return blockIdx.z == 0   ? pre(std::integral_constant<int, 0>{})
         : blockIdx.z == 1 ? pre(std::integral_constant<int, 1>{})
                           : pre(std::integral_constant<int, 2>{});
}

// POIS: blockIdx.z counts the three inverses of a Poisson solve, which read the
// one spectrum; its scaling is applied to the values as they are read (the
// products rounded in the order a inv, then times wu or wv).
template <int L, bool MAPPED, bool STAGED, bool NARROW, bool POIS, bool EXACT>
__global__ void __launch_bounds__(TpRows<L, NARROW>::THREADS, TpRows<L, NARROW>::MINB)
    k_tp_rows_inv(Dct2dArgs a, PoissonArgs ps) {
  using R = TpRows<L, NARROW>;
  extern __shared__ float4 sxti[];
  const int pi = threadIdx.x / R::TPS, g = threadIdx.x % R::TPS;
  float4* s = sxti + pi * R::LP;
  const int M = a.n1 / 2;
  const int c = blockIdx.x * R::NP + pi;
  const bool first = (c == 0);
  const int kb = tp_item_b(c, M);
  const float* C = a.in + (POIS ? 0 : (long long)blockIdx.z * a.in_bstride);
  const int vkind = POIS ? poisson_vkind(blockIdx.z) : a.vkind;
  const InvRows A = inv_rows_of(a, C, c, L, vkind), B = inv_rows_of(a, C, kb, L, vkind);
  soa::C2 v[16];
  int t;
  if constexpr (STAGED) {
    uint64_t* bar = reinterpret_cast<uint64_t*>(sxti + R::NP * R::LP) + pi;
    int* flag = reinterpret_cast<int*>(reinterpret_cast<uint64_t*>(sxti + R::NP * R::LP) + R::NP);
    float* st = reinterpret_cast<float*>(s);
    constexpr bool DEN = POIS && tp_den_staged<L, NARROW>();
    // the denominators' rows, behind the barriers and the flag
    float* dst = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(sxti) + R::SMEM_STAGED) + pi * 4 * L;
    if (threadIdx.x == 0) *flag = 1;
    if (g == 0) {
      tma::bar_init(bar, 1);
      tma::fence_barrier_init();
    }
    if constexpr (!DEN) pdl::wait_prior_grid();
    __syncthreads();
    const float* src[4] = {A.ra, A.rb, B.ra, B.rb};  // rb rows are never null
    if (g == 0) {
      uint32_t bytes = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) bytes += src[i] ? (DEN ? 2 : 1) * L * (uint32_t)sizeof(float) : 0u;
      tma::bar_expect_tx(bar, bytes);
    }
    if constexpr (DEN) {
      // a table of the solver: sent for while the forward transform finishes
      if (g == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (src[i])
            tma::bulk_load(dst + i * L, ps.inv + (src[i] - C), L * (uint32_t)sizeof(float), bar, l2::evict_last());
      }
      pdl::wait_prior_grid();
    }
    if (g == 0) {
      const uint64_t pol = l2::evict_first();  // the input is streamed in
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (src[i]) tma::bulk_load(st + i * L, src[i], L * (uint32_t)sizeof(float), bar, pol);
      const uint32_t polls = a.polls ? a.polls : tma::kDefaultPolls;
      if (!tma::bar_wait_from_issue(bar, 0, polls)) {
        atomicExch(a.err, 1);
        tma::bar_wait(bar, 0, tma::kDefaultPolls);  // the copies must land before the CTA exits
        *flag = 0;
      }
    }
    __syncthreads();
    if (!*flag) return;
    tma::test_wait(bar, 0);  // completed: every thread observes the copied rows
    const RowReads<true> As{{A.ra ? st : nullptr, st + L}, 0}, Bs{{B.ra ? st + 2 * L : nullptr, st + 3 * L}, 0};
    if constexpr (POIS)
      t = tp_poisson_pre<L, true, DEN, EXACT>(a, ps, As, Bs, A, B, C, (int)(dst - st), c, kb, first, g, v);
    else
      t = tp_inv_pre<L, MAPPED, EXACT>(a, As, Bs, vkind, c, kb, first, g, v);
    rowp::group_sync<R::TPS>(pi);  // the first stage overwrites the staged rows
  } else {
    pdl::wait_prior_grid();
    const uint64_t pol = l2::evict_first();  // the input is streamed in
    const RowReads<false> Ag{A, pol}, Bg{B, pol};
    if constexpr (POIS)
      t = tp_poisson_pre<L, false, false, EXACT>(a, ps, Ag, Bg, A, B, C, 0, c, kb, first, g, v);
    else
      t = tp_inv_pre<L, MAPPED, EXACT>(a, Ag, Bg, vkind, c, kb, first, g, v);
  }
  soa::first_stage<L, true>(v, s, t);
  rowp::stages_to_regs<L, 16, true, false, EXACT>(s, g, pi, a.tw2x, v);
  pdl::launch_dependents();
  float2* Zw = a.work + (long long)blockIdx.z * a.work_bstride;
  if (rowp::warp_has_first<R::TPS>(first))
    tp_inv_pair<L, false, EXACT>(v, a, Zw, L / 2, c, kb, first, g);
  else
    tp_inv_pair<L, false, EXACT>(v, a, Zw, L / 2, c, kb, false, g);
}

}  // namespace gbdct
