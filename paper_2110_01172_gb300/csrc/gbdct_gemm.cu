// gbdct_gemm.cu - split-BF16 DFT-GEMM precision mode (see gemm_path.cuh): the
// two dense products of the separable definition on the tensor cores, by the
// hand-written tcgen05 kernel of tc_gemm.cuh.
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <mutex>
#include <new>

#include "gemm_path.cuh"
#include "tc_gemm.cuh"

namespace gbdct {

struct GemmPath {
  int n1 = 0, n2 = 0, batch = 0, nsm = 0;
  int* err = nullptr;                          // the plan's device error word
  uint32_t polls = tc::kDefaultPolls;          // bound of every device-side wait
  // Half-size matrices of one side, split: rows [forward p0, forward p1, inverse
  // p0, inverse p1] of N/2 each, N/2 columns; hi then lo, side 1 then side 2
  __nv_bfloat16* mats = nullptr;
  __nv_bfloat16 *xh = nullptr, *xl = nullptr;  // split input quadrants, [p2][batch][p1][n1/2][n2/2]
  __nv_bfloat16 *th = nullptr, *tl = nullptr;  // split intermediate, [p1][batch][p2][n2/2][n1/2]
  size_t bytes = 0;
  // tensor maps, hi / lo (box 64 x 128 for A operands; 64 x 128 and 64 x 64 for B operands)
  CUtensorMap xa[2], ta[2];        // input quadrants and intermediate as A
  CUtensorMap m1[2][2], m2[2][2];  // [BN 128 / 64][hi / lo] matrices of side 1 and 2 as B
};

namespace {

// Matrix entry in FP64 from the integer-reduced angle m = k (2j+1) mod 4N.
__device__ double cos_half(long long m, int n) { return cospi((double)(m % (4LL * n)) / (2.0 * n)); }

// The half-size matrices of side n (see GemmPath::mats): with j < n/2 the position,
// k = 2i + p the frequency, forward row i, column j: cos(pi k (2j+1) / 2n);
// inverse row j, column i: (2/n) w_k cos(pi k (2j+1) / 2n), w_0 = 1/2.
__global__ void k_gemm_mats(__nv_bfloat16* hi, __nv_bfloat16* lo, int n) {
  const int h = n / 2;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4LL * h * h) return;
  const int c = (int)(idx % h), r = (int)(idx / h % h), m = (int)(idx / ((long long)h * h));
  const bool inv = m >= 2;
  const int k = 2 * (inv ? c : r) + (m & 1), j = inv ? r : c;
  double v = cos_half((long long)k * (2 * j + 1), n);
  if (inv) v *= (2.0 / n) * (k ? 1.0 : 0.5);
  const __nv_bfloat16 hv = __float2bfloat16_rn((float)v);
  hi[idx] = hv;
  lo[idx] = __float2bfloat16_rn((float)(v - (double)__bfloat162float(hv)));
}

// Four values as bf16 hi and lo parts.
__device__ __forceinline__ void put_split(__nv_bfloat16* hi, __nv_bfloat16* lo, long long i, const float (&v)[4]) {
  __nv_bfloat16 h[4], l[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    h[j] = __float2bfloat16_rn(v[j]);
    l[j] = __float2bfloat16_rn(v[j] - __bfloat162float(h[j]));
  }
  auto pack = [](const __nv_bfloat16* q) {
    const __nv_bfloat162 a = __halves2bfloat162(q[0], q[1]), b = __halves2bfloat162(q[2], q[3]);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  };
  *reinterpret_cast<uint2*>(hi + i) = pack(h);
  *reinterpret_cast<uint2*>(lo + i) = pack(l);
}

__device__ __forceinline__ float4 rev4(float4 v) { return make_float4(v.w, v.z, v.y, v.x); }

// Sums and differences of four float4: s[p1][p2] = (a +- b) +- (c +- d), minus for p = 1
// (p2 within a pair, p1 between the pairs).
__device__ __forceinline__ void mirror_sums(float4 a, float4 b, float4 c, float4 d, float (&s)[2][2][4]) {
  const float va[4] = {a.x, a.y, a.z, a.w}, vb[4] = {b.x, b.y, b.z, b.w};
  const float vc[4] = {c.x, c.y, c.z, c.w}, vd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float e0 = va[j] + vb[j], e1 = vc[j] + vd[j], o0 = va[j] - vb[j], o1 = vc[j] - vd[j];
    s[0][0][j] = e0 + e1;
    s[1][0][j] = e0 - e1;
    s[0][1][j] = o0 + o1;
    s[1][1][j] = o0 - o1;
  }
}

// One thread: four columns j2 .. j2+3 of row i1 of every quadrant of one transform.
struct Quads {
  int i1, j2, b;
  bool live;
  __device__ __forceinline__ Quads(int n1, int n2, int batch) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int w = n2 / 8;  // groups of four columns in a quadrant's row
    j2 = 4 * (int)(idx % w);
    i1 = (int)(idx / w % (n1 / 2));
    const long long bb = idx / w / (n1 / 2);
    live = bb < batch;
    b = live ? (int)bb : 0;
  }
};

// The split input quadrants.  Forward: q[p1][p2] = mirror sums of the input over
// both axes (x_j +- x_{N-1-j}); inverse: the spectrum's entries of parity (p1, p2).
template <bool INV>
__global__ void __launch_bounds__(256) k_split(const float* __restrict__ in, __nv_bfloat16* __restrict__ hi,
                                               __nv_bfloat16* __restrict__ lo, int n1, int n2, int batch) {
  const Quads t(n1, n2, batch);
  pdl::wait_prior_grid();
  pdl::launch_dependents();
  if (!t.live) return;
  const float* x = in + (long long)t.b * n1 * n2;
  auto ld = [&](int r, int c) { return *reinterpret_cast<const float4*>(x + (long long)r * n2 + c); };
  float q[2][2][4];
  if constexpr (!INV) {
    mirror_sums(ld(t.i1, t.j2), rev4(ld(t.i1, n2 - 4 - t.j2)), ld(n1 - 1 - t.i1, t.j2),
                rev4(ld(n1 - 1 - t.i1, n2 - 4 - t.j2)), q);
  } else {
#pragma unroll
    for (int p1 = 0; p1 < 2; ++p1) {
      const float4 u = ld(2 * t.i1 + p1, 2 * t.j2), v = ld(2 * t.i1 + p1, 2 * t.j2 + 4);
      q[p1][0][0] = u.x, q[p1][0][1] = u.z, q[p1][0][2] = v.x, q[p1][0][3] = v.z;
      q[p1][1][0] = u.y, q[p1][1][1] = u.w, q[p1][1][2] = v.y, q[p1][1][3] = v.w;
    }
  }
  const int h1 = n1 / 2, h2 = n2 / 2;
#pragma unroll
  for (int p2 = 0; p2 < 2; ++p2)
#pragma unroll
    for (int p1 = 0; p1 < 2; ++p1)
      put_split(hi, lo, ((((long long)p2 * batch + t.b) * 2 + p1) * h1 + t.i1) * h2 + t.j2, q[p1][p2]);
}

// Inverse: the output from the quadrants y[b][p1][p2] of the second product, whose
// entries of odd frequency parity change sign at the mirror position.
__global__ void __launch_bounds__(256) k_join(const float* __restrict__ y, float* __restrict__ out, int n1, int n2,
                                              int batch) {
  const Quads t(n1, n2, batch);
  pdl::wait_prior_grid();
  pdl::launch_dependents();
  if (!t.live) return;
  const long long quad = (long long)(n1 / 2) * (n2 / 2);
  const float* q = y + (long long)t.b * n1 * n2 + (long long)t.i1 * (n2 / 2) + t.j2;
  auto ld = [&](int p1, int p2) { return *reinterpret_cast<const float4*>(q + (2 * p1 + p2) * quad); };
  float s[2][2][4];  // [mirror of axis 0][mirror of axis 1]
  mirror_sums(ld(0, 0), ld(0, 1), ld(1, 0), ld(1, 1), s);
  float* o = out + (long long)t.b * n1 * n2;
  auto f4 = [](const float (&v)[4]) { return make_float4(v[0], v[1], v[2], v[3]); };
  const long long r0 = (long long)t.i1 * n2, r1 = (long long)(n1 - 1 - t.i1) * n2;
  *reinterpret_cast<float4*>(o + r0 + t.j2) = f4(s[0][0]);
  *reinterpret_cast<float4*>(o + r0 + n2 - 4 - t.j2) = rev4(f4(s[0][1]));
  *reinterpret_cast<float4*>(o + r1 + t.j2) = f4(s[1][0]);
  *reinterpret_cast<float4*>(o + r1 + n2 - 4 - t.j2) = rev4(f4(s[1][1]));
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() { return tma::encoder(); }

// 2D bf16 map of a row-major rows x cols matrix, box 64 (cols) x box_rows, 128-byte swizzle.
bool map2d(CUtensorMap* m, const void* base, long long rows, long long cols, int box_rows) {
  const PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {(cuuint32_t)tc::BK, (cuuint32_t)box_rows};
  const cuuint32_t es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The largest grid that a plan can ask for: 65535 transforms, sides of kGemmMaxSide.
static_assert(tc::tile_grid(65535LL * kGemmMaxSide, kGemmMaxSide / 2, 64) <= 0x7fffffffLL, "tiles fit the grid's x axis");

// One product: A (map pair a) times the side's matrices, rows x cols outputs (cols /
// BN a power of two) for each of the two parities in blockIdx.z.
template <int BN>
cudaError_t launch(const CUtensorMap (&a)[2], const CUtensorMap (&b)[2][2], tc::Epi e, int rows, int cols, int kdim,
                   uint32_t polls, int* err, cudaStream_t s) {
  using Cf = tc::Cfg<BN>;
  const CUtensorMap(&m)[2] = b[BN == 128 ? 0 : 1];
  e.lg_cols = 0;
  while ((BN << e.lg_cols) < cols) ++e.lg_cols;
  const dim3 grid((unsigned)tc::tile_grid(rows, cols, BN), 1, 2);
  return pdl::launch(tc::k_tc_dftgemm<BN>, grid, dim3(128), (size_t)Cf::SMEM, s, a[0], a[1], m[0], m[1], e,
                     kdim / tc::BK, polls, err);
}

// BN = 128 when that already gives at least one tile per SM, else 64.
bool wide_tiles(long long rows, long long cols, int nsm) {
  return cols % 128 == 0 && (rows / tc::BM) * (cols / 128) * 2 >= nsm;
}

}  // namespace

GemmPath* gemm_create(int n1, int n2, int batch, int* err, gbdct_status* st) {
  *st = GBDCT_ERR_UNSUPPORTED;
  if (n1 < kGemmMinSide || n2 < kGemmMinSide || n1 > kGemmMaxSide || n2 > kGemmMaxSide || batch < 1) return nullptr;
  GemmPath* g = new (std::nothrow) GemmPath();
  if (!g) {
    *st = GBDCT_ERR_OOM;
    return nullptr;
  }
  g->n1 = n1;
  g->n2 = n2;
  g->batch = batch;
  g->err = err;
  int dev = 0;
  cudaError_t ce = cudaGetDevice(&dev);
  if (ce == cudaSuccess) ce = cudaDeviceGetAttribute(&g->nsm, cudaDevAttrMultiProcessorCount, dev);
  // elements of one side's matrices (hi or lo), and of the array
  const size_t m1 = (size_t)n1 * n1, m2 = (size_t)n2 * n2, e = (size_t)batch * n1 * n2;
  if (ce == cudaSuccess) ce = cudaMalloc(&g->mats, 2 * (m1 + m2) * sizeof(__nv_bfloat16));
  if (ce == cudaSuccess) ce = cudaMalloc(&g->xh, 4 * e * sizeof(__nv_bfloat16));  // xh, xl, th, tl
  g->bytes = 2 * (m1 + m2) * sizeof(__nv_bfloat16) + 4 * e * sizeof(__nv_bfloat16);
  if (ce == cudaSuccess) {
    g->xl = g->xh + e;
    g->th = g->xl + e;
    g->tl = g->th + e;
    __nv_bfloat16* m = g->mats;
    k_gemm_mats<<<(unsigned)((m1 + 255) / 256), 256>>>(m, m + m1, n1);
    __nv_bfloat16* q = m + 2 * m1;
    k_gemm_mats<<<(unsigned)((m2 + 255) / 256), 256>>>(q, q + m2, n2);
    ce = cudaGetLastError();
    if (ce == cudaSuccess) ce = cudaDeviceSynchronize();
  }
  if (ce == cudaSuccess) ce = cudaFuncSetAttribute(reinterpret_cast<const void*>(tc::k_tc_dftgemm<128>),
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, tc::Cfg<128>::SMEM);
  if (ce == cudaSuccess) ce = cudaFuncSetAttribute(reinterpret_cast<const void*>(tc::k_tc_dftgemm<64>),
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, tc::Cfg<64>::SMEM);
  bool maps = ce == cudaSuccess;
  if (maps) {
    const __nv_bfloat16* m = g->mats;
    const __nv_bfloat16* q = m + 2 * m1;
    const long long xr = 2LL * batch * n1, tr = 2LL * batch * n2;  // both parities stacked
    for (int l = 0; l < 2 && maps; ++l) {
      maps = map2d(&g->xa[l], l ? g->xl : g->xh, xr, n2 / 2, tc::BM) &&
             map2d(&g->ta[l], l ? g->tl : g->th, tr, n1 / 2, tc::BM);
      for (int w = 0; w < 2 && maps; ++w)
        maps = map2d(&g->m1[w][l], m + l * m1, 2LL * n1, n1 / 2, w ? 64 : 128) &&
               map2d(&g->m2[w][l], q + l * m2, 2LL * n2, n2 / 2, w ? 64 : 128);
    }
  }
  if (ce != cudaSuccess || !maps) {
    gemm_destroy(g);
    *st = ce == cudaErrorMemoryAllocation ? GBDCT_ERR_OOM : GBDCT_ERR_CUDA;
    return nullptr;
  }
  *st = GBDCT_OK;
  return g;
}

void gemm_set_wait_polls(GemmPath* g, uint32_t polls) {
  if (g) g->polls = polls ? polls : tc::kDefaultPolls;
}

gbdct_status gemm_exec(GemmPath* g, bool inverse, const float* in, float* out, cudaStream_t s) {
  const int n1 = g->n1, n2 = g->n2, h1 = n1 / 2, h2 = n2 / 2, batch = g->batch;
  const long long threads = (long long)batch * h1 * (n2 / 8);
  const dim3 blocks((unsigned)((threads + 255) / 256));
  cudaError_t ce = inverse ? pdl::launch(k_split<true>, blocks, dim3(256), 0, s, in, g->xh, g->xl, n1, n2, batch)
                           : pdl::launch(k_split<false>, blocks, dim3(256), 0, s, in, g->xh, g->xl, n1, n2, batch);
  // first product, along axis 1 (rows (b, p1, i1), for each parity p2)
  const tc::Epi e1{tc::EPI_SPLIT_T, n1, n2, batch, batch * n1, h2, inverse ? n2 : 0, 0, g->th, g->tl, nullptr};
  if (ce == cudaSuccess)
    ce = wide_tiles((long long)batch * n1, h2, g->nsm)
             ? launch<128>(g->xa, g->m2, e1, batch * n1, h2, h2, g->polls, g->err, s)
             : launch<64>(g->xa, g->m2, e1, batch * n1, h2, h2, g->polls, g->err, s);
  // second product, along axis 0 (rows (b, p2, j2), for each parity p1); the
  // inverse's quadrants reuse the split input's memory
  float* y = reinterpret_cast<float*>(g->xh);
  const tc::Epi e2{inverse ? tc::EPI_QUADRANT : tc::EPI_DCT, n1, n2, batch, batch * n2, h1, inverse ? n1 : 0, 0, nullptr,
                   nullptr, inverse ? y : out};
  if (ce == cudaSuccess)
    ce = wide_tiles((long long)batch * n2, h1, g->nsm)
             ? launch<128>(g->ta, g->m1, e2, batch * n2, h1, h1, g->polls, g->err, s)
             : launch<64>(g->ta, g->m1, e2, batch * n2, h1, h1, g->polls, g->err, s);
  if (ce == cudaSuccess && inverse) ce = pdl::launch(k_join, blocks, dim3(256), 0, s, static_cast<const float*>(y), out, n1, n2, batch);
  return ce == cudaSuccess ? GBDCT_OK : GBDCT_ERR_CUDA;
}

size_t gemm_workspace_bytes(const GemmPath* g) { return g ? g->bytes : 0; }

void gemm_destroy(GemmPath* g) {
  if (!g) return;
  cudaFree(g->mats);
  cudaFree(g->xh);
  delete g;
}

}  // namespace gbdct
