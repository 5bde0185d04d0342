// Random projection B = A Omega (Sec. 5.1, Algorithm 2).
//
// Algorithm 2 has every mapper keep an in-memory partial sum
// Bbar = sum_{i in block} A_:i Omega_i: over its columns and the reducers add
// the c partials row by row.  Here the column range is split into S slices;
// each slice's partial product is one tile grid of the GEMM, and a second
// kernel adds the S partials in a fixed order (reproducible results).
#include "project.cuh"
#include "tc.cuh"

#include <algorithm>
#include <cstring>

using namespace css;

namespace {

template <typename TA> __device__ __forceinline__ typename AccOf<TA>::type cvt(TA v);
template <> __device__ __forceinline__ double cvt<double>(double v) { return v; }
template <> __device__ __forceinline__ float cvt<float>(float v) { return v; }
template <> __device__ __forceinline__ float cvt<__nv_bfloat16>(__nv_bfloat16 v) {
  return __uint_as_float(((uint32_t)__bfloat16_as_ushort(v)) << 16);
}

constexpr int kSlices = 8;
constexpr int kMaxTcSlices = 32;

// partial[s][i + j*m] = sum over columns l of slice s of A[i, l] * Omega[l, j]
template <typename TA, int TT, int KC>
__global__ void __launch_bounds__(256) project_simt_kernel(const TA* __restrict__ A, long long lda,
                                                          const TA* __restrict__ Om, long long ldo,
                                                          int m, int n, int r, int slice_len,
                                                          typename AccOf<TA>::type* __restrict__ partial) {
  using Acc = typename AccOf<TA>::type;
  constexpr int BT = 16 * TT;
  __shared__ __align__(16) Acc As[KC][BT];
  __shared__ __align__(16) Acc Os[KC][BT + 1];
  const int i0 = blockIdx.x * BT, j0 = blockIdx.y * BT, sl = blockIdx.z;
  const int l_begin = sl * slice_len, l_end = min(n, l_begin + slice_len);
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  Acc acc[TT][TT];
#pragma unroll
  for (int a = 0; a < TT; ++a)
#pragma unroll
    for (int b = 0; b < TT; ++b) acc[a][b] = Acc(0);
  for (int l0 = l_begin; l0 < l_end; l0 += KC) {
    for (int e = tid; e < KC * BT; e += 256) {
      const int kk = e / BT, rr = e % BT;           // A: rows contiguous
      const int l = l0 + kk;
      As[kk][rr] = (l < l_end && i0 + rr < m) ? cvt<TA>(A[(long long)l * lda + i0 + rr]) : Acc(0);
      const int jj = e / KC, k2 = e % KC;           // Omega: columns of length n contiguous
      const int l2 = l0 + k2;
      Os[k2][jj] = (l2 < l_end && j0 + jj < r) ? cvt<TA>(Om[(long long)(j0 + jj) * ldo + l2]) : Acc(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KC; ++kk) {
      Acc a[TT], b[TT];
#pragma unroll
      for (int q = 0; q < TT; ++q) { a[q] = As[kk][ty * TT + q]; b[q] = Os[kk][tx * TT + q]; }
#pragma unroll
      for (int q = 0; q < TT; ++q)
#pragma unroll
        for (int w = 0; w < TT; ++w) acc[q][w] = fma(a[q], b[w], acc[q][w]);
    }
    __syncthreads();
  }
  Acc* out = partial + (long long)sl * m * r;
#pragma unroll
  for (int q = 0; q < TT; ++q)
#pragma unroll
    for (int w = 0; w < TT; ++w) {
      const int i = i0 + ty * TT + q, j = j0 + tx * TT + w;
      if (i < m && j < r) out[(long long)j * m + i] = acc[q][w];
    }
}

// The same partial sums with FP32 accumulation: 128 x (16 CT) outputs per
// block, 8 x CT per thread, so that each column of the chunk costs a thread
// two or more 16-byte shared-memory reads for 8 CT multiply-adds (the 4 x 4
// kernel above spends one 4-byte read on two).  The next 16 columns are in
// registers while the current ones are multiplied.  Bound by the FP32 rate
// where r fills its tiles: FP32 1500 x 50001, r = 200: 1.89 -> 0.94 ms
// (0.44 at the FP32 rate, a quarter of it for padding r to 256).
constexpr int kPR = 128;   // rows of a tile
constexpr int kPK = 16;    // columns of A per chunk

template <typename TA, int CT>
__global__ void __launch_bounds__(256, 2) project_f32_kernel(const TA* __restrict__ A, long long lda,
                                                             const TA* __restrict__ Om, long long ldo, int m, int n,
                                                             int r, int slice_len, float* __restrict__ partial) {
  constexpr int BN = 16 * CT, OP = BN + 4;   // Omega is staged transposed: its rows are padded
  constexpr int VA = kPR * kPK / 256, VO = BN * kPK / 256;
  __shared__ __align__(16) float As[2][kPK][kPR];
  __shared__ __align__(16) float Os[2][kPK][OP];
  const int i0 = blockIdx.x * kPR, j0 = blockIdx.y * BN, sl = blockIdx.z;
  const int l_begin = sl * slice_len, l_end = min(n, l_begin + slice_len);
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  float acc[8][CT];
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int w = 0; w < CT; ++w) acc[q][w] = 0.f;
  float ra[VA], ro[VO];
  // A: row tid % 128 of columns tid / 128 + 2 v.  Omega: entry tid % 16 of the
  // chunk of columns tid / 16 + 16 v
  const int ar = tid % kPR, ak = tid / kPR, ok = tid % kPK, oj = tid / kPK;
  const bool row_in = i0 + ar < m;
  const TA* pa = A + (long long)ak * lda + i0 + ar;
  const TA* po = Om + (long long)(j0 + oj) * ldo + ok;
  auto fetch = [&](int l0) {
#pragma unroll
    for (int v = 0; v < VA; ++v)
      ra[v] = (row_in && l0 + ak + 2 * v < l_end) ? cvt<TA>(__ldg(pa + (long long)(l0 + 2 * v) * lda)) : 0.f;
#pragma unroll
    for (int v = 0; v < VO; ++v)
      ro[v] = (j0 + oj + 16 * v < r && l0 + ok < l_end) ? cvt<TA>(__ldg(po + (long long)(16 * v) * ldo + l0)) : 0.f;
  };
  auto stage = [&](int b) {
#pragma unroll
    for (int v = 0; v < VA; ++v) As[b][ak + 2 * v][ar] = ra[v];
#pragma unroll
    for (int v = 0; v < VO; ++v) Os[b][ok][oj + 16 * v] = ro[v];
  };
  // this thread's rows: 4 ty + {0..3} and 64 + those; its columns likewise
  // (CT = 8), 4 tx + {0..3} (CT = 4) or 2 tx + {0, 1} (CT = 2)
  auto row_of = [&](int q) { return (q < 4 ? 0 : 64) + ty * 4 + (q & 3); };
  auto col_of = [&](int w) { return CT == 8 ? (w < 4 ? 0 : 64) + tx * 4 + (w & 3) : tx * CT + w; };
  if (l_begin < l_end) {
    fetch(l_begin);
    stage(0);
  }
  __syncthreads();
  int b = 0;
  for (int l0 = l_begin; l0 < l_end; l0 += kPK) {
    const bool more = l0 + kPK < l_end;
    if (more) fetch(l0 + kPK);
#pragma unroll
    for (int kk = 0; kk < kPK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[b][kk][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[b][kk][64 + ty * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      float o[CT];
      if constexpr (CT == 2) {
        const float2 t = *reinterpret_cast<const float2*>(&Os[b][kk][tx * 2]);
        o[0] = t.x; o[1] = t.y;
      } else {
#pragma unroll
        for (int h = 0; h < CT / 4; ++h) {
          const float4 t = *reinterpret_cast<const float4*>(&Os[b][kk][64 * h + tx * 4]);
          o[4 * h] = t.x; o[4 * h + 1] = t.y; o[4 * h + 2] = t.z; o[4 * h + 3] = t.w;
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int w = 0; w < CT; ++w) acc[q][w] = fmaf(a[q], o[w], acc[q][w]);
    }
    if (more) stage(b ^ 1);
    __syncthreads();
    b ^= 1;
  }
  float* out = partial + (long long)sl * m * r;
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int w = 0; w < CT; ++w) {
      const int i = i0 + row_of(q), j = j0 + col_of(w);
      if (i < m && j < r) out[(long long)j * m + i] = acc[q][w];
    }
}

// Reducers: B[i, j] = sum_s partial[s][i, j], slices in order.
template <typename Acc>
__global__ void project_reduce_kernel(const Acc* __restrict__ partial, int S, int m, int r,
                                      Acc* __restrict__ B, long long ldb) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)m * r) return;
  const int i = (int)(idx % m), j = (int)(idx / m);
  Acc s = Acc(0);
  for (int q = 0; q < S; ++q) s += partial[(long long)q * m * r + idx];
  B[(long long)j * ldb + i] = s;
}

cudaError_t project_simt_f64(const void* A, long long lda, const void* Om, long long ldo, int m, int n,
                             int r, void* B, long long ldb, void* partial, cudaStream_t s) {
  constexpr int TT = 4, KC = 16, BT = 16 * TT;
  const int S = kSlices;
  const int slice_len = (n + S - 1) / S;
  dim3 grid((m + BT - 1) / BT, (r + BT - 1) / BT, S);
  project_simt_kernel<double, TT, KC><<<grid, 256, 0, s>>>((const double*)A, lda, (const double*)Om, ldo, m, n, r,
                                                          slice_len, (double*)partial);
  const long long tot = (long long)m * r;
  project_reduce_kernel<double><<<(unsigned)((tot + 255) / 256), 256, 0, s>>>((const double*)partial, S, m, r,
                                                                            (double*)B, ldb);
  return cudaGetLastError();
}

template <typename TA>
cudaError_t project_f32(const void* A, long long lda, const void* Om, long long ldo, int m, int n, int r, void* B,
                        long long ldb, void* partial, int sms, cudaStream_t s) {
  // the narrowest tile whose padding costs no more than the wider one's
  const int w32 = (r + 31) / 32 * 32, w64 = (r + 63) / 64 * 64, w128 = (r + 127) / 128 * 128;
  const int BN = w32 < w64 && r <= 32 ? 32 : w64 < w128 ? 64 : 128;
  const int mt = (m + kPR - 1) / kPR, nt = (r + BN - 1) / BN;
  // at least kSlices partial sums (a longer FP32 chain would round more), and
  // of the counts up to kMaxTcSlices that leave a slice 128 columns the one whose waves of
  // two blocks an SM are fullest
  int S = kSlices;
  for (int c = kSlices + 1; c <= std::min(kMaxTcSlices, n / 128); ++c) {
    const auto waves = [&](long long k) { return ((long long)mt * nt * k + 2 * sms - 1) / (2 * sms); };
    if (waves(c) * S < waves(S) * c) S = c;
  }
  const int slice_len = ((n + S - 1) / S + kPK - 1) / kPK * kPK;
  const dim3 grid(mt, nt, S);
  const TA *a = (const TA*)A, *o = (const TA*)Om;
  float* p = (float*)partial;
  if (BN == 32) project_f32_kernel<TA, 2><<<grid, 256, 0, s>>>(a, lda, o, ldo, m, n, r, slice_len, p);
  else if (BN == 64) project_f32_kernel<TA, 4><<<grid, 256, 0, s>>>(a, lda, o, ldo, m, n, r, slice_len, p);
  else project_f32_kernel<TA, 8><<<grid, 256, 0, s>>>(a, lda, o, ldo, m, n, r, slice_len, p);
  const long long tot = (long long)m * r;
  project_reduce_kernel<float><<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(p, S, m, r, (float*)B, ldb);
  return cudaGetLastError();
}

size_t accsz(int dt) { return dt == CSS_F64 ? 8 : 4; }

}  // namespace

size_t project_workspace_bytes(int dtype, int64_t m, int64_t n, int64_t r) {
  (void)n;
  const size_t sl = std::max(kSlices, kMaxTcSlices);
  return kStatusBytes + align_up((size_t)sl * m * r * accsz(dtype));
}

extern "C" css_status css_project(const void* A, css_dtype dtype, int64_t m, int64_t n, int64_t lda,
                                  const void* Omega, int64_t r, int64_t ldo, void* Bout, int64_t ldb,
                                  void* ws, size_t ws_bytes, const css_opts* opts,
                                  css_stream_t stream) {
  (void)opts;
  if (!A || !Omega || !Bout) return CSS_ERR_INVALID_ARG;
  if (dtype != CSS_F64 && dtype != CSS_F32 && dtype != CSS_BF16) return CSS_ERR_INVALID_ARG;
  if (m < 1 || n < 1 || r < 1 || lda < m || ldo < n || ldb < m) return CSS_ERR_INVALID_ARG;
  if (m > INT32_MAX || n > INT32_MAX || r > INT32_MAX) return CSS_ERR_INVALID_ARG;
  if (!ws || ((uintptr_t)ws % kWsAlign) != 0) return CSS_ERR_WORKSPACE;
  if (ws_bytes < project_workspace_bytes(dtype, m, n, r)) return CSS_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  void* partial = (char*)ws + kStatusBytes;
  int* err = (int*)ws;
  css_opts o0;
  css_opts_default(&o0);
  const css_opts& oo = opts ? *opts : o0;
  cudaError_t e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // BF16 input: tcgen05 split-K GEMM (Algorithm 2's per-block partial sums in
  // TMEM), then the same fixed-order reduction as the SIMT path
  if (dtype == CSS_BF16 && oo.init_path != 1 && css::tc::supported(A, lda, (int)m, (int)r) &&
      css::tc::supported(Omega, ldo, (int)n, (int)r)) {
    const int slices = std::min(kMaxTcSlices, css::tc::project_slices((int)m, sms > 0 ? sms : 1));
    if ((e = cudaMemsetAsync(err, 0, sizeof(int), s)) != cudaSuccess) return CSS_ERR_CUDA;
    e = css::tc::project_partials(A, lda, (int)m, (int)n, Omega, ldo, (int)r, slices, (float*)partial, err,
                                  oo.spin_budget_ns ? oo.spin_budget_ns : 2000000000ull, s);
    if (e != cudaSuccess) return CSS_ERR_CUDA;
    const long long tot = m * r;
    project_reduce_kernel<float><<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(
        (const float*)partial, slices, (int)m, (int)r, (float*)Bout, ldb);
    if ((e = cudaGetLastError()) != cudaSuccess) return CSS_ERR_CUDA;
    if (oo.sync) {
      int h = 0;
      if (cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        return CSS_ERR_CUDA;
      if (h) return (css_status)h;
    }
    return CSS_OK;
  }
  switch (dtype) {
    case CSS_F64: e = project_simt_f64(A, lda, Omega, ldo, (int)m, (int)n, (int)r, Bout, ldb, partial, s); break;
    case CSS_F32: e = project_f32<float>(A, lda, Omega, ldo, (int)m, (int)n, (int)r, Bout, ldb, partial, sms, s); break;
    default: e = project_f32<__nv_bfloat16>(A, lda, Omega, ldo, (int)m, (int)n, (int)r, Bout, ldb, partial, sms, s); break;
  }
  if (e != cudaSuccess) return CSS_ERR_CUDA;
  const css_opts o = [&] { css_opts t; css_opts_default(&t); return opts ? *opts : t; }();
  if (o.sync) {
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return CSS_ERR_CUDA;
  }
  return CSS_OK;
}
