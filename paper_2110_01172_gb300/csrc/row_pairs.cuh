// row_pairs.cuh - the row passes' work on mirror pairs of points, in registers.
//
// The forward postprocess combines the row spectrum at columns c and L - c
// (Section III-B, Eqs. four-elements, s-t), the inverse preprocess makes the
// points k2 and L - k2 from the same four reads (Eq. 2d_idct_pre), and the
// inverse pairing joins the points p and L - 1 - p.  In the Stockham stages the
// points of one butterfly t of NS = L / R are t + NS m, so both mirrors map
// whole butterflies onto whole butterflies:
//   L - (t + NS m)     = (NS - t)     + NS (R - 1 - m)   (t > 0)
//   L - 1 - (t + NS m) = (NS - 1 - t) + NS (R - 1 - m).
// The threads' butterflies of the first or last stage are therefore chosen
// such that a butterfly and its mirror are held either by the same thread
// (radices below 16: a thread has 16 / R butterflies) or by two lanes of one
// warp, which swap half of their values with shuffles.  The pair work then
// needs no shared-memory pass of its own: the row pass moves its points
// through shared memory twice instead of three times, and the inverse reads
// every input value once.  Together with immediate-offset addresses the forward
// row pass of a 4096^2 transform executes 13.1 M warp instructions instead of
// 17.2 M, the inverse 15.3 M instead of 18.3 M.  What bounds the passes is the
// latency of their phases (loads, FFT, stores) at 16 warps per SM: the
// shared-memory pipe is busy for half of the time, the FMA pipe for 38 %.
// Measured, forward / inverse row pass: 4096^2 32.4 / 36.2 -> 30.5 / 34.5 us,
// 25 x 512^2 13.7 / 14.5 -> 10.7 / 13.0, 1024 x 8192 22.7 / 24.7 -> 21.0 / 23.0,
// 8192^2 (four-step family) 169 / 198 -> 160 / 188.
#pragma once

#include "fft_soa.cuh"
#include "l2_hint.cuh"

namespace gbdct {
namespace rowp {

constexpr float kRH = 0.70710678118654752f;  // sqrt(1/2)

// Barrier of one thread group (TPS threads; `group` its index in the CTA).
// Groups of a CTA work on separate rows and need no common barrier.
template <int TPS>
__device__ __forceinline__ void group_sync(int group) {
  if constexpr (TPS <= 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(TPS) : "memory");
  }
}

// Butterfly of thread g among T (one per thread) such that t and T - 1 - t sit
// in lanes l and l ^ rev_lane_mask<T>() of one warp.
template <int T>
__device__ __forceinline__ int rev_lane_butterfly(int g) {
  if constexpr (T >= 32) {
    const int w = g >> 5, l = g & 31;
    return l < 16 ? 16 * w + l : T + 15 - 16 * w - l;
  } else {
    return g;
  }
}
template <int T>
constexpr int rev_lane_mask() { return T >= 32 ? 16 : T - 1; }

// Butterfly of thread g among T (one per thread) such that t and T - t sit in
// one warp; 0 and T / 2 are their own mirrors and take the two lanes that
// would otherwise mirror each other.
template <int T>
__device__ __forceinline__ int neg_lane_butterfly(int g) {
  if constexpr (T >= 32) {
    const int w = g >> 5, l = g & 31;
    return l < 16 ? 16 * w + l : (g == 16 ? T / 2 : T + 16 - 16 * w - l);
  } else {
    return g;
  }
}
// The lane of the mirror butterfly (the lane itself for 0 and T / 2).
template <int T>
__device__ __forceinline__ int neg_lane_source(int g) {
  const int lane = threadIdx.x & 31;
  if constexpr (T >= 32) {
    return (g == 0 || g == 16) ? lane : lane ^ 16;
  } else {
    return (lane & ~(T - 1)) | ((T - g) & (T - 1));
  }
}

__device__ __forceinline__ soa::C2 shfl(soa::C2 v, int src) {
  return {make_float2(__shfl_sync(0xffffffffu, v.re.x, src), __shfl_sync(0xffffffffu, v.re.y, src)),
          make_float2(__shfl_sync(0xffffffffu, v.im.x, src), __shfl_sync(0xffffffffu, v.im.y, src))};
}
__device__ __forceinline__ soa::C2 shfl_xor(soa::C2 v, int mask) {
  return {make_float2(__shfl_xor_sync(0xffffffffu, v.re.x, mask), __shfl_xor_sync(0xffffffffu, v.re.y, mask)),
          make_float2(__shfl_xor_sync(0xffffffffu, v.im.x, mask), __shfl_xor_sync(0xffffffffu, v.im.y, mask))};
}

// Shape of the last stage of length L: NB butterflies of radix R per thread,
// inputs and outputs t + NS m.
template <int L>
struct Last {
  static constexpr int NS = last_stage_ns(L);
  static constexpr int R = stage_radix(L, NS);
  static constexpr int NB = fft_points(L) / R;
  static constexpr int TPS = fft_tps(L);
  static_assert(NB == 1 || NB % 2 == 0, "butterflies come in mirror pairs");
};

// Butterfly q of thread g in the last stage.  NEG: mirrored by NS - t (forward
// postprocess), else by NS - 1 - t (inverse pairing); for NB > 1 butterfly
// NB / 2 + i is the mirror of butterfly i.
template <int L, bool NEG>
__device__ __forceinline__ int last_butterfly(int g, int q) {
  using S = Last<L>;
  if constexpr (S::NB == 1) {
    return NEG ? neg_lane_butterfly<S::NS>(g) : rev_lane_butterfly<S::NS>(g);
  } else {
    if (q < S::NB / 2) return g + q * S::TPS;
    const int t = g + (q - S::NB / 2) * S::TPS;
    if (!NEG) return S::NS - 1 - t;
    return t ? S::NS - t : S::NS / 2;
  }
}

// Stages NS .. L of a group's rows in s; the last stage leaves its outputs in
// v (output m of butterfly q at v[q R + m]).  Called once the thread has written
// its outputs of the stage before; the barrier that follows is in here, after
// the loads of the stage's twiddles, so that their latency passes in its wait.
template <int L, int NS, bool INV, bool NEG, bool EXACT>
__device__ __forceinline__ void stages_to_regs(float4* __restrict__ s, int g, int group,
                                               const float4* __restrict__ tw, soa::C2* v) {
  constexpr int R = stage_radix(L, NS);
  constexpr int TPS = fft_tps(L);
  constexpr int NB = fft_points(L) / R;
  constexpr bool LAST = NS * R == L;
  soa::Tw<R> w[NB];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int t = LAST ? last_butterfly<L, NEG>(g, q) : g + q * TPS;
    w[q].load(tw + tw_offset(L, NS) + (t & (NS - 1)), NS);
  }
  group_sync<TPS>(group);
#pragma unroll
  for (int q = 0; q < NB; ++q)
    soa::load_butterfly<L, NS, 1>(v + q * R, s, LAST ? last_butterfly<L, NEG>(g, q) : g + q * TPS);
  if constexpr (!LAST) group_sync<TPS>(group);
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int t = LAST ? last_butterfly<L, NEG>(g, q) : g + q * TPS;
    soa::twiddle<R, INV, EXACT>(v + q * R, w[q], tw + tw_offset(L, NS) + (t & (NS - 1)), NS);
    soa::dft<R, INV>(v + q * R);
    if constexpr (!LAST) soa::store_butterfly<L, NS, 1>(v + q * R, s, g + q * TPS);
  }
  if constexpr (!LAST) stages_to_regs<L, NS * R, INV, NEG, EXACT>(s, g, group, tw, v);
}

// Whether any group of the calling warp is the transform's first one (the
// group with the packed item): warp-uniform, so the code for the packed item
// may be a branch of its own although the pair work shuffles across the warp.
template <int TPS>
__device__ __forceinline__ bool warp_has_first(bool first) {
  return TPS >= 32 ? first : __any_sync(0xffffffffu, first);
}

// ---------------------------------------------------------------------------
// Forward postprocess
// ---------------------------------------------------------------------------

// Combine of both items (lanes) from the row spectrum at a column P = Y(c) and
// its mirror M = Y(L - c), b = b_c / 2 as (br, br, bi, bi): with u = aP +
// conj(aM), w = aP - conj(aM), s = b u, t = b w the outputs are
// y(k1, c) = Re s, y(kmir, c) = -Im t, y(k1, L-c) = -Im s, y(kmir, L-c) = -Re t.
// FIRST && packed: lane a is the packed item of rows 0 and N1/2 (a = 1 for row
// 0 and w = sqrt(1/2) (M.x - P.x, -(P.y + M.y)) for row N1/2).
struct Outs {
  float2 lo0, lo1, hi0, hi1;  // (lane a, lane b): rows k1 and kmir at c, then at L - c
};
// EXACT: b = (br, bi) and the rests (br, bi) that its rounding left.
template <bool FIRST, bool EXACT>
__device__ __forceinline__ Outs combine(soa::C2 P, soa::C2 M, float2 avr, float2 avi, float4 b, bool packed) {
  const soa::C2 aP = soa::mulw(P, avr, avi), aM = soa::mulw(M, avr, avi);
  const float2 ur = soa::add2(aP.re, aM.re), nui = soa::sub2(aM.im, aP.im);
  float2 nwr = soa::sub2(aM.re, aP.re), wi = soa::add2(aP.im, aM.im);
  if (FIRST && packed) {
    nwr.x = kRH * (P.re.x - M.re.x);
    wi.x = -kRH * (P.im.x + M.im.x);
  }
  Outs o;
  if constexpr (EXACT) {
    const float2 br = soa::bc(b.x), bi = soa::bc(b.y), rr = soa::bc(b.z), ri = soa::bc(b.w), nwi = soa::ng(wi);
    o.lo0 = soa::fma2(nui, bi, soa::fma2(ur, br, soa::fma2(nui, ri, soa::mul2(ur, rr))));
    o.hi0 = soa::fma2(nui, br, soa::fma2(ur, soa::ng(bi), soa::fma2(nui, rr, soa::mul2(ur, soa::ng(ri)))));
    o.lo1 = soa::fma2(nwi, br, soa::fma2(nwr, bi, soa::fma2(nwi, rr, soa::mul2(nwr, ri))));
    o.hi1 = soa::fma2(wi, bi, soa::fma2(nwr, br, soa::fma2(wi, ri, soa::mul2(nwr, rr))));
    return o;
  }
  const float2 br = make_float2(b.x, b.y), bi = make_float2(b.z, b.w), nbi = soa::ng(bi);
  o.lo0 = soa::fma2(nui, bi, soa::mul2(ur, br));
  o.hi0 = soa::fma2(nui, br, soa::mul2(ur, nbi));
  o.lo1 = soa::fma2(soa::ng(wi), br, soa::mul2(nwr, bi));
  o.hi1 = soa::fma2(wi, bi, soa::mul2(nwr, br));
  return o;
}

// Where the outputs of a forward row group go.  GENERAL: the DST-II order
// (output (k1, k2) stored at (N1-1-k1, N2-1-k2)) and the magnitude threshold of
// Section V-A (outputs below eps stored as zero; 0: off); otherwise the
// DCT-II order and no threshold, with every column offset an immediate.
// SMEM: the rows are in shared memory.
template <int L, bool GENERAL, bool SMEM = false>
struct FwdOut {
  float *a0, *a1, *b0, *b1;  // rows k1 and kmir of lane a, of lane b
  uint64_t pol;
  float eps;
  bool rev;

  __device__ __forceinline__ void put(float* p, float v) const {
    if constexpr (GENERAL) v = fabsf(v) < eps ? 0.f : v;
    if constexpr (SMEM)
      *p = v;
    else
      l2::st(p, v, pol);
  }
  // the outputs of columns c = base + off and L - c (off a compile-time constant)
  __device__ __forceinline__ void store(const Outs& o, int base, int off, bool mirror) const {
    const int c0 = (GENERAL && rev) ? L - 1 - base - off : base + off;
    put(a0 + c0, o.lo0.x);
    put(b0 + c0, o.lo0.y);
    put(a1 + c0, o.lo1.x);
    put(b1 + c0, o.lo1.y);
    if (!mirror) return;
    const int c1 = (GENERAL && rev) ? base + off - 1 : L - base - off;
    put(a0 + c1, o.hi0.x);
    put(b0 + c1, o.hi0.y);
    put(a1 + c1, o.hi1.x);
    put(b1 + c1, o.hi1.y);
  }
};

// Calls column(P, M, base, off, mirror) for every pair of points c = base + off
// (off a compile-time constant) and L - c of the last stage's outputs in v; mirror
// is false for c = 0 and L / 2, which pair with themselves.  t, src: the thread's
// last-stage butterfly and the lane of its mirror (one butterfly per thread only).
template <int L, typename Column>
__device__ __forceinline__ void neg_pairs(soa::C2* v, int g, int t, int src, const Column& column) {
  using S = Last<L>;
  constexpr int NS = S::NS, R = S::R;
  if constexpr (S::NB == 1) {
    static_assert(R == 16, "one butterfly per thread has the full radix");
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      // butterfly 0 mirrors onto itself with m <-> 16 - m
      soa::C2 x = v[15 - m];
      const soa::C2 z = v[(16 - m) & 15];
      if (t == 0) x = z;
      const soa::C2 M = shfl(x, src);
      column(v[m], M, t, NS * m, m > 0 || t != 0);
    }
    if (t == 0) column(v[8], v[8], 0, L / 2, false);
  } else {
#pragma unroll
    for (int i = 0; i < S::NB / 2; ++i) {
      t = g + i * S::TPS;
      soa::C2* A = v + i * R;
      soa::C2* B = v + (S::NB / 2 + i) * R;
      // slots: P = A[m], M = B[R - 1 - m], column t + NS m.  Butterfly 0 is its
      // own mirror (m <-> R - m) and its partner here is butterfly NS / 2, its own
      // mirror too (m <-> R - 1 - m): regrouped so that the slots' pairs stay
      // (slot 0 is column 0 with itself; column L / 2 is left over).
      soa::C2 half = A[R / 2];
      if (i == 0 && t == 0) {
        soa::C2 h[R];
#pragma unroll
        for (int m = 0; m < R; ++m) h[m] = B[m];
#pragma unroll
        for (int m = 0; m < R / 2; ++m) {
          B[R / 2 + m] = m == R / 2 - 1 ? A[0] : A[R / 2 + 1 + m];
          B[m] = h[R / 2 + m];
        }
#pragma unroll
        for (int m = 0; m < R / 2; ++m) A[R / 2 + m] = h[m];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int base = h == 0 ? t : ((i == 0 && t == 0) ? NS / 2 : t + L / 2);
#pragma unroll
        for (int m = 0; m < R / 2; ++m)
          column(A[h * (R / 2) + m], B[R - 1 - h * (R / 2) - m], base, NS * m, i > 0 || h > 0 || m > 0 || t != 0);
      }
      if (i == 0 && t == 0) column(half, half, 0, L / 2, false);
    }
  }
}

// Postprocess of a group's two rows from the last stage's registers.
template <int L, bool FIRST, bool EXACT, typename Out>
__device__ __forceinline__ void fwd_post(soa::C2* v, const Out& out, float2 avr, float2 avi,
                                         const float4* __restrict__ fb4, int g, bool packed) {
  constexpr int NS = Last<L>::NS;
  neg_pairs<L>(v, g, neg_lane_butterfly<NS>(g), neg_lane_source<NS>(g),
               [&](soa::C2 P, soa::C2 M, int base, int off, bool mirror) {
                 out.store(combine<FIRST, EXACT>(P, M, avr, avi, __ldg(fb4 + base + off), packed), base, off, mirror);
               });
}

// ---------------------------------------------------------------------------
// Inverse preprocess
// ---------------------------------------------------------------------------

// The four reads of a point k2 and its mirror km = L - k2 of one item: c1 =
// C(k1,k2), c3 = C(kmir,k2), c4 = C(k1,km), c2 = C(kmir,km).
struct Quad {
  float c1, c3, c4, c2;
};

// v(k2) and v(km) of both items from their reads.  v = x b ia with x = (c1 -
// c2, -(c3 + c4)); at the mirror the reads trade places and b_km = i conj(b_k2).
// FIRST && packed: lane a packs rows 0 and N1/2 as the real and imaginary
// parts of one sequence.
// EXACT: b = (br, bi) and the rests that its rounding left (else 0).
template <bool FIRST, bool EXACT>
__device__ __forceinline__ void inv_pair_points(const Quad& qa, const Quad& qb, float4 b4, float2 iaA, float2 iar,
                                                float2 iai, float2 ih, bool packed, soa::C2& lo,
                                                soa::C2& hi) {
  const float2 b = make_float2(b4.x, b4.y), br = soa::bc(b.x), bi = soa::bc(b.y);
  const float2 rr = soa::bc(b4.z), ri = soa::bc(b4.w);
  const soa::C2 x{make_float2(qa.c1 - qa.c2, qb.c1 - qb.c2), make_float2(-(qa.c3 + qa.c4), -(qb.c3 + qb.c4))};
  lo = soa::mulw(EXACT ? soa::mulw(x, br, bi, rr, ri) : soa::mulw(x, br, bi), iar, iai);
  const soa::C2 y{make_float2(qa.c2 + qa.c1, qb.c2 + qb.c1), make_float2(qa.c4 - qa.c3, qb.c4 - qb.c3)};
  hi = soa::mulw(EXACT ? soa::mulw(y, br, soa::ng(bi), rr, soa::ng(ri)) : soa::mulwc(y, br, bi), iar, iai);
  if (FIRST && packed) {
    const float2 v0 = cmul(cmul(make_float2(qa.c1, -qa.c4), b), iaA);
    const float2 vh = cmul(cmul(make_float2(qa.c3 - qa.c2, -(qa.c3 + qa.c2)), b), ih);
    lo.re.x = v0.x - vh.y;
    lo.im.x = v0.y + vh.x;
    // the mirror: i (c4 - i c1) = c1 + i c4 times conj(b)
    const float2 w0 = cmul(cmulc(make_float2(qa.c1, qa.c4), b), iaA);
    const float2 wh = cmul(cmulc(make_float2(qa.c2 + qa.c3, qa.c2 - qa.c3), b), ih);
    hi.re.x = w0.x - wh.y;
    hi.im.x = w0.y + wh.x;
  }
}

// Points t + TPS j (t the thread's first-stage butterfly, returned) of both
// items in v.  quads(k2, km, qa, qb) reads one pair of columns of both items
// (km = 0 past the edge for k2 = 0, where the mirror reads are zero).
template <int L, bool FIRST, bool EXACT, typename Quads>
__device__ __forceinline__ int inv_pre(const Quads& quads, const float2* __restrict__ ib,
                                       const float4* __restrict__ ib4, float2 iaA, float2 iaB,
                                       float2 ih, bool packed, int g, soa::C2* v) {
  constexpr int T = fft_tps(L);
  const int t = neg_lane_butterfly<T>(g), src = neg_lane_source<T>(g);
  const float2 iar = make_float2(iaA.x, iaB.x), iai = make_float2(iaA.y, iaB.y);
  auto twiddle = [&](int k) {
    if constexpr (EXACT) return __ldg(ib4 + k);
    const float2 w = __ldg(ib + k);
    return make_float4(w.x, w.y, 0.f, 0.f);
  };
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    Quad qa, qb;
    quads(t + T * j, L - t - T * j, j == 0 && t == 0, qa, qb);
    soa::C2 hi;
    inv_pair_points<FIRST, EXACT>(qa, qb, twiddle(t + T * j), iaA, iar, iai, ih, packed, v[j], hi);
    v[15 - j] = shfl(hi, src);  // point L - k2 belongs to the mirror butterfly, at 15 - j
  }
  if (t == 0) {  // butterfly 0 mirrors onto itself with j <-> 16 - j; point L / 2 pairs with itself
#pragma unroll
    for (int j = 15; j > 8; --j) v[j] = v[j - 1];
    Quad qa, qb;
    quads(L / 2, L / 2, false, qa, qb);
    soa::C2 hi;
    inv_pair_points<FIRST, EXACT>(qa, qb, twiddle(L / 2), iaA, iar, iai, ih, packed, v[8], hi);
  }
  return t;
}

// ---------------------------------------------------------------------------
// Inverse pairing
// ---------------------------------------------------------------------------

// Calls emit(p, u, w) with u the row IFFT's point p < L / 2 and w its point
// L - 1 - p, from the last stage's registers (base + off = p, off a
// compile-time constant).
template <int L, typename Emit>
__device__ __forceinline__ void inv_pairs(const soa::C2* v, int g, const Emit& emit) {
  using S = Last<L>;
  constexpr int NS = S::NS, R = S::R;
  if constexpr (S::NB == 1) {
    const int t = rev_lane_butterfly<NS>(g);
#pragma unroll
    for (int m = 0; m < 8; ++m) emit(t, NS * m, v[m], shfl_xor(v[15 - m], rev_lane_mask<NS>()));
  } else {
#pragma unroll
    for (int i = 0; i < S::NB / 2; ++i) {
      const int t = g + i * S::TPS;
      const soa::C2* A = v + i * R;
      const soa::C2* B = v + (S::NB / 2 + i) * R;
#pragma unroll
      for (int m = 0; m < R / 2; ++m) {
        emit(t, NS * m, A[m], B[R - 1 - m]);
        emit(NS - 1 - t, NS * m, B[m], A[R - 1 - m]);
      }
    }
  }
}

}  // namespace rowp
}  // namespace gbdct
