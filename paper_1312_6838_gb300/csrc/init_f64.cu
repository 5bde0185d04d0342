// Initial scores of FP64 problems from integer digits on the tensor cores
// (slice_gemm.cu): C = A A^T, then f_i = a_i^T (C a_i) (Algorithm 1).  The
// products drop less than 2^-58 of the rows' largest products a term, so C and
// C A are as accurate as FP64 sums (C relative to sqrt(C_ii C_jj); C A with
// A's rows brought to one size).  Equal columns get equal bits (each entry is an
// exact integer sum rounded once, and the columns' dots run in one order).
// Infinities become NaN: the selection reports either as non-finite data.
//
// The FP64 tiles of init_simt.cu are bound by an SM's FP64 rate (two lanes a
// clock), and a small problem has too few of them: 500 x 1000 took 1.63 ms
// with 36 blocks in C = A A^T; here 0.23 ms; 1024 x 8192: 23.4 -> 1.03 ms.
// Whole selections, us with the tiles and here: 64 x 128, k = 8 587 and 519;
// 1000 x 500, k = 50 4114 and 2782; 64 x 20000, k = 16 21955 and 1215; the tiles
// only win at a single tile (32 x 64, k = 8: 468 and 493).
#include <algorithm>

#include "init.cuh"
#include "slice_gemm.cuh"

namespace css {
namespace {

constexpr long long kChunk = 16384;                // most columns whose products are held at a time
// Digits of a part of A by rows; of one by columns, and of a part of C's rows.
constexpr long long kRowBytes = 256ll << 20, kPartBytes = 1ll << 30;
constexpr size_t kMaxEntries = (size_t)1 << 30;   // of A; beyond it the FP64 tiles run (not measured there)

struct Layout {
  sg::Digits rows, cols, left;   // parts of A by rows and by columns (in one space), and of C
  long long part_k, part_cols, part_left;
  double* D;
  int* kexp;   // of the sizes of A's rows
  sg::Scratch sc;
};

Layout carve(WsCarver& c, long long m, long long n) {
  Layout L{};
  L.part_k = std::min(n, sg::part_k(m, kRowBytes));
  L.part_cols = std::min(std::min(n, kChunk), sg::part_rows(m, kPartBytes));
  L.part_left = std::min(m, sg::part_rows(m, kPartBytes));
  const size_t at = c.off;
  L.rows = sg::carve_digits(c, m, L.part_k);
  const size_t end = c.off;
  c.off = at;
  L.cols = sg::carve_digits(c, L.part_cols, m);
  c.off = std::max(c.off, end);
  L.left = sg::carve_digits(c, L.part_left, m);
  L.D = c.take<double>((size_t)(L.part_left * L.part_cols));
  L.kexp = c.take<int>((size_t)m);
  size_t words = std::max(sg::sum_words(m, m, L.part_k, 1), sg::sum_words(L.part_left, L.part_cols, m, 0));
  if (n % L.part_cols) words = std::max(words, sg::sum_words(L.part_left, n % L.part_cols, m, 0));
  L.sc = sg::carve_scratch(c, words);
  return L;
}

// f[i] = sum_r D[r, i] A[r, i], or f[i] += that: one warp a column, memory-bound.
__global__ void __launch_bounds__(256) column_dots_kernel(const double* __restrict__ D, const double* __restrict__ A,
                                                          long long lda, int m, int n, double* __restrict__ f,
                                                          bool add) {
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const double *d = D + (long long)i * m, *a = A + (long long)i * lda;
  double s = 0.0;
#pragma unroll 4
  for (int r = lane; r < m; r += 32) s = fma(d[r], a[r], s);
  s = warp_sum(s);
  if (lane == 0) f[i] = add ? f[i] + s : s;
}

}  // namespace

size_t css_f0_f64_bytes(int64_t m, int64_t n) {
  WsCarver c(nullptr, (size_t)-1);
  if ((size_t)m * (size_t)n > kMaxEntries) return 0;
  carve(c, m, n);
  return c.off;
}

cudaError_t css_f0_f64(const double* A, long long lda, int m, int n, double* C, long long ldc, void* scratch,
                       double* f, int* err, unsigned long long spin_ns, cudaStream_t s, int stall) {
  WsCarver c(scratch, (size_t)-1);
  Layout L = carve(c, m, n);
  L.sc.stall = stall;
  cudaError_t e = cudaSuccess;
  for (long long c0 = 0; e == cudaSuccess && c0 < n; c0 += L.part_k) {
    const sg::Source rows{A + c0 * lda, CSS_F64, 1, lda, m, (int)std::min(L.part_k, n - c0)};
    e = sg::split(rows, L.rows, s);
    const sg::Store st{C, 1, ldc, 1, nullptr, nullptr, c0 > 0};
    if (e == cudaSuccess) e = sg::gemm(L.rows, L.rows, st, L.sc, err, spin_ns, s);
  }
  // C A with A's rows at one size: (C S^-1)(S A), S^2 the diagonal of C
  if (e == cudaSuccess) sg::gram_exponents(C, ldc, m, L.kexp, s);
  for (long long c0 = 0; e == cudaSuccess && c0 < n; c0 += L.part_cols) {
    const int nc = (int)std::min(L.part_cols, n - c0);
    const sg::Source cols{A + c0 * lda, CSS_F64, lda, 1, nc, m, L.kexp, 1};
    e = sg::split(cols, L.cols, s);
    for (long long r0 = 0; e == cudaSuccess && r0 < m; r0 += L.part_left) {
      const int mr = (int)std::min<long long>(L.part_left, m - r0);
      const sg::Source cs{C + r0 * ldc, CSS_F64, ldc, 1, mr, m, L.kexp, -1};
      if (c0 == 0 || L.part_left < m) e = sg::split(cs, L.left, s);
      if (e == cudaSuccess) e = sg::gemm(L.left, L.cols, sg::Store{L.D, 1, mr, 0}, L.sc, err, spin_ns, s);
      column_dots_kernel<<<(nc + 7) / 8, 256, 0, s>>>(L.D, A + c0 * lda + r0, lda, mr, nc, f + c0, r0 > 0);
    }
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace css
