// Initial scores of FP64 problems from integer digits on the tensor cores
// (slice_gemm.cu): C = A A^T, then f_i = a_i^T (C a_i) (Algorithm 1).  The
// digit products keep 2^-64 of the rows' largest products, so C and C A are
// as accurate as FP64 sums.  Equal columns get equal bits (each entry is an
// exact integer sum rounded once, and the columns' dots run in one order).
// Infinities become NaN: the selection reports either as non-finite data.
//
// The FP64 tiles of init_simt.cu are bound by an SM's FP64 rate (two lanes a
// clock), and a small problem has too few of them: 500 x 1000 took 1.63 ms
// with 36 blocks in C = A A^T; here
// 0.23 ms; 1024 x 8192: 23.4 -> 1.03 ms.
#include <algorithm>

#include "init.cuh"
#include "slice_gemm.cuh"

namespace css {
namespace {

constexpr long long kChunk = 16384;               // columns whose products are held at a time
constexpr size_t kMaxDigits = (size_t)1 << 34;    // scratch bound: beyond it the FP64 tiles run

// Columns per chunk: digits of at most 1 GB.
long long chunk_cols(long long m, long long n) {
  const long long fit = std::max<long long>(128, ((1ll << 30) / (16 * std::max<long long>(m, 64))) / 128 * 128);
  return std::min(std::min(kChunk, fit), n);
}

struct Layout {
  sg::Digits rows, cols, left;   // A by rows, A's chunk by columns (in the same space), C
  double* D;
  sg::Scratch sc;
};

Layout carve(WsCarver& c, long long m, long long n) {
  Layout L{};
  const long long nb = chunk_cols(m, n);
  const size_t at = c.off;
  L.rows = sg::carve_digits(c, m, n);
  const size_t end = c.off;
  c.off = at;
  L.cols = sg::carve_digits(c, nb, m);
  c.off = std::max(c.off, end);
  L.left = sg::carve_digits(c, m, m);
  L.D = c.take<double>((size_t)m * nb);
  size_t words = std::max(sg::sum_words(m, m, n, 1), sg::sum_words(m, nb, m, 0));
  if (n % nb) words = std::max(words, sg::sum_words(m, n % nb, m, 0));
  L.sc = sg::carve_scratch(c, words);
  return L;
}

// f[i] = sum_r D[r, i] A[r, i]: one warp a column, memory-bound.
__global__ void __launch_bounds__(256) column_dots_kernel(const double* __restrict__ D, const double* __restrict__ A,
                                                          long long lda, int m, int n, double* __restrict__ f) {
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const double *d = D + (long long)i * m, *a = A + (long long)i * lda;
  double s = 0.0;
#pragma unroll 4
  for (int r = lane; r < m; r += 32) s = fma(d[r], a[r], s);
  s = warp_sum(s);
  if (lane == 0) f[i] = s;
}

}  // namespace

size_t css_f0_f64_bytes(int64_t m, int64_t n) {
  WsCarver c(nullptr, (size_t)-1);
  if ((size_t)m * (size_t)n > kMaxDigits / 16) return 0;
  carve(c, m, n);
  return c.off;
}

cudaError_t css_f0_f64(const double* A, long long lda, int m, int n, double* C, long long ldc, void* scratch,
                       double* f, int* err, unsigned long long spin_ns, cudaStream_t s) {
  WsCarver c(scratch, (size_t)-1);
  Layout L = carve(c, m, n);
  const sg::Source rows{A, CSS_F64, 1, lda, m, n}, cs{C, CSS_F64, ldc, 1, m, m};
  cudaError_t e = sg::split(rows, L.rows, s);
  if (e == cudaSuccess) e = sg::gemm(L.rows, L.rows, sg::Store{C, 1, ldc, 1}, L.sc, err, spin_ns, s);
  if (e == cudaSuccess) e = sg::split(cs, L.left, s);
  if (e != cudaSuccess) return e;
  const long long nb = chunk_cols(m, n);
  for (long long c0 = 0; c0 < n; c0 += nb) {
    const int nc = (int)std::min<long long>(nb, n - c0);
    const sg::Source cols{A + c0 * lda, CSS_F64, lda, 1, nc, m};
    e = sg::split(cols, L.cols, s);
    if (e == cudaSuccess) e = sg::gemm(L.left, L.cols, sg::Store{L.D, 1, m, 0}, L.sc, err, spin_ns, s);
    if (e != cudaSuccess) return e;
    column_dots_kernel<<<(nc + 7) / 8, 256, 0, s>>>(L.D, A + c0 * lda, lda, m, nc, f + c0);
  }
  return cudaGetLastError();
}

}  // namespace css
