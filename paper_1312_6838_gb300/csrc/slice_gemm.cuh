// Internal interface of the slice GEMM (slice_gemm.cu): products of FP64,
// FP32 or BF16 matrices to FP64 accuracy on the BF16 tensor cores.
#pragma once

#include <algorithm>

#include "css_common.cuh"

namespace css {
namespace sg {

// A rows x K operand in its own type: element (row, k) at p[row * rs + k * ks],
// times 2^(kexp_sign kexp[k]) where kexp is given (FP64 only).
struct Source {
  const void* p;
  int dtype;            // css_dtype
  long long rs, ks;
  int rows, K;
  const int* kexp;
  int kexp_sign;
};
// Balances operands whose inner index runs over very different sizes: digits
// hold a row's entries relative to its largest one, so where a few inner
// indices are by far the largest in X and a row of Y is zero there, what is
// left of X's rows would be too coarse for it.  e[k] = the exponent of
// sqrt(G_kk) of a Gram matrix over the inner index: X 2^e and Y 2^-e (or the
// reverse) have the same product.
void gram_exponents(const double* G, long long ld, int K, int* e, cudaStream_t s);

// The operand as digits (see slice_gemm.cu).
struct Digits {
  unsigned char* d;     // tiles of 128 rows x 16 k x 8 slices
  unsigned char* ns;    // non-zero leading slices per (row tile, 64 k)
  int* ex;              // largest biased exponent of each row
  int rows, K, dtype;
};

// Carves the digits of a rows x K operand (whole tiles of 128 rows) from a
// workspace (rows may be the
// largest of several operands that use the same space one after another).
Digits carve_digits(WsCarver& c, long long rows, long long K);
// Digits take 16 bytes an entry of whole 128-row x 64-k blocks.  Operands of
// more than this many bytes are formed a part at a time: by parts of the inner
// dimension whose products are added (Store::add; this also keeps the integer
// sums far inside 64 bits: K is at most 2^20 a part, and 2^25 fit), or by rows.
constexpr long long kDigitBudget = 1280ll << 20;
// Inner indices a part that `rows` rows allow, and rows that K allows.
inline long long part_k(long long rows, long long budget = kDigitBudget) {
  return std::max<long long>(64, budget / (2048 * ((rows + 127) / 128)) / 64 * 64);
}
inline long long part_rows(long long K, long long budget = kDigitBudget) {
  return std::max<long long>(128, budget / (1024 * ((K + 63) / 64)) / 128 * 128);
}
// Splits src into digits (src.rows <= the carved rows).
cudaError_t split(const Source& src, Digits& D, cudaStream_t s);

// Scratch of gemm: per-CTA partial sums, and the integer sums of a product
// whose inner dimension is cut into slices (taken when they fit).
struct Scratch {
  long long* part;
  unsigned long long* sums;
  size_t cap;           // 8-byte words of sums
  int stall;            // test hook: the products also wait on a phase nothing completes
};
// Words of integer sums that an M x N product over K can use (0: none).
size_t sum_words(long long M, long long N, long long K, int lower);
Scratch carve_scratch(WsCarver& c, size_t words);

// out[i * rs + j * cs] = cscale[j] sum_k X[i, k] Y[j, k] (FP64, or FP32 to
// out32; cscale may be null).  lower: X and Y are the same operand; only tiles
// touching i >= j are computed and both triangles written.  add: out += that
// (FP64 only).
struct Store {
  double* out;
  long long rs, cs;
  int lower;
  const double* cscale;
  float* out32;
  int add;
};
// Rows with an infinity or a NaN give NaN; with the operands' sources their
// results beside infinities are as FP64 arithmetic gives them.
cudaError_t gemm(const Digits& X, const Digits& Y, const Store& st, const Scratch& w, int* err,
                 unsigned long long spin_ns, cudaStream_t s, const Source& sx = Source{},
                 const Source& sy = Source{});

// R = A - X Y^T for FP32 or BF16 A (M x N, leading dimension lda): writes R
// (FP32, leading dimension M) when R != null, dA = g2 R when dA != null, and
// adds its share of ||R||^2 to a partial sum per CTA (residual_parts of them).
struct Residual {
  const void* A;
  int dtype;
  long long lda;
  float* R;
  void* dA;
  long long ldda;
  double g2;
  double* loss_part;
};
int residual_parts();
cudaError_t gemm_residual(const Digits& X, const Digits& Y, const Residual& r, const Scratch& w, int* err,
                          unsigned long long spin_ns, cudaStream_t s);

}  // namespace sg
}  // namespace css
