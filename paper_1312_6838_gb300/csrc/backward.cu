// Reconstruction at a fixed selected set S: the embedding Q = orth(A_S),
// W = Q^T A of Sec. 3.2 (css_embed), and the loss and gradient of the
// reconstruction error (css_residual_backward).
//
// Loss and gradient:
//   L(A) = ||A - P^(S) A||_F^2,  P^(S) = A_S (A_S^T A_S)^-1 A_S^T   (Eq. Projection)
//   T = (A_S^T A_S)^-1 A_S^T A,  R = A - A_S T
//   dL/dA = 2 R  (columns outside S),  dL/dA_S = -2 R T^T
//
// With the Cholesky factor A_S^T A_S = L L^T in FP64 and Q = A_S L^-T
// (orthonormal; formed anew by each call, so that nothing of a forward pass is
// kept for the gradient):
//   W = Q^T A,  R = A - Q W,  T = L^-T W,  R T^T = (R W^T) L^-1.
// R is a small difference of large terms (the part of A outside span(A_S)),
// so W, Q W and R W^T are sums of exact digit products on the slice GEMM
// (slice_gemm.cu); R of FP32/BF16 input is formed from pairs of FP32 values
// and held in FP32.  Its product with W^T keeps all digits all the same: W's
// rows hold the selected columns, where R is zero, and where those are the
// largest the columns that count lie far below the rows' largest entries (four
// digits a factor: selected columns 1e4 times the rest, their gradient off by
// 1.2e-4; all digits: 5e-8, forward and backward 3.79 -> 4.12 ms).
#include <algorithm>
#include <vector>

#include "backward.cuh"
#include "slice_gemm.cuh"

using namespace css;

namespace {

template <typename TA> __device__ __forceinline__ double to_d(TA v);
template <> __device__ __forceinline__ double to_d<double>(double v) { return v; }
template <> __device__ __forceinline__ double to_d<float>(float v) { return (double)v; }
template <> __device__ __forceinline__ double to_d<__nv_bfloat16>(__nv_bfloat16 v) {
  return (double)__uint_as_float(((uint32_t)__bfloat16_as_ushort(v)) << 16);
}
template <typename TA> __device__ __forceinline__ TA from_d(double v);
template <> __device__ __forceinline__ double from_d<double>(double v) { return v; }
template <> __device__ __forceinline__ float from_d<float>(double v) { return (float)v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_d<__nv_bfloat16>(double v) {
  return __float2bfloat16_rn((float)v);
}

// ------------------------------------------------------- small FP64 steps --
template <typename TA>
__global__ void gather_cols_kernel(const TA* __restrict__ A, long long lda, int m,
                                   const int* __restrict__ sel, int k, double* __restrict__ AS) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)m * k) return;
  const int i = (int)(idx % m), j = (int)(idx / m);
  AS[idx] = to_d<TA>(A[(long long)sel[j] * lda + i]);
}


// G = A_S^T A_S split over the m rows: block (pair, slice) forms the 32 x 32
// tile (ti >= tj) of one row slice, 2 x 2 outputs per thread; gram_fin then
// adds the slices in order and mirrors (bit-reproducible).  Enough blocks to
// fill the GPU even for small k, where one block per output tile would not.
constexpr int kGT = 32, kGK = 32;

struct GramPlan {
  int tiles, npairs, nslices, slice;
};

GramPlan gram_plan(int m, int k) {
  GramPlan g{};
  g.tiles = (k + kGT - 1) / kGT;
  g.npairs = g.tiles * (g.tiles + 1) / 2;
  const int want = std::max(1, (2 * 148 + g.npairs - 1) / g.npairs);
  g.nslices = std::max(1, std::min(want, (m + 127) / 128));
  g.slice = (m + g.nslices - 1) / g.nslices;
  return g;
}

__global__ void __launch_bounds__(256) gram_part_kernel(const double* __restrict__ AS, int m, int k, int slice,
                                                        int npairs, double* __restrict__ part) {
  __shared__ double xa[kGT][kGK + 1], xb[kGT][kGK + 1];
  const int pidx = blockIdx.x, sl = blockIdx.y;
  int ti = (int)((sqrtf(8.f * pidx + 1.f) - 1.f) * 0.5f);
  while (ti * (ti + 1) / 2 > pidx) --ti;
  while ((ti + 1) * (ti + 2) / 2 <= pidx) ++ti;
  const int tj = pidx - ti * (ti + 1) / 2;
  const int a0 = ti * kGT, b0 = tj * kGT;
  const int rb = sl * slice, re = min(m, rb + slice);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc00 = 0.0, acc01 = 0.0, acc10 = 0.0, acc11 = 0.0;
  for (int r0 = rb; r0 < re; r0 += kGK) {
    for (int e = threadIdx.x; e < kGT * kGK; e += 256) {
      const int col = e / kGK, rr = e % kGK;
      const bool okr = r0 + rr < re;
      xa[col][rr] = (okr && a0 + col < k) ? AS[(long long)(a0 + col) * m + r0 + rr] : 0.0;
      xb[col][rr] = (okr && b0 + col < k) ? AS[(long long)(b0 + col) * m + r0 + rr] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < kGK; ++kk) {
      const double u0 = xa[ty * 2][kk], u1 = xa[ty * 2 + 1][kk];
      const double v0 = xb[tx * 2][kk], v1 = xb[tx * 2 + 1][kk];
      acc00 = fma(u0, v0, acc00);
      acc01 = fma(u0, v1, acc01);
      acc10 = fma(u1, v0, acc10);
      acc11 = fma(u1, v1, acc11);
    }
    __syncthreads();
  }
  double* out = part + ((long long)sl * npairs + pidx) * (kGT * kGT);
  out[(ty * 2) * kGT + tx * 2] = acc00;
  out[(ty * 2) * kGT + tx * 2 + 1] = acc01;
  out[(ty * 2 + 1) * kGT + tx * 2] = acc10;
  out[(ty * 2 + 1) * kGT + tx * 2 + 1] = acc11;
}

__global__ void gram_fin_kernel(const double* __restrict__ part, int nslices, int npairs, int k,
                                double* __restrict__ G) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)k * k) return;
  const int r = (int)(idx % k), c = (int)(idx / k);
  const int a = max(r, c), b = min(r, c);
  const int pidx = (a / kGT) * (a / kGT + 1) / 2 + b / kGT;
  const int off = (a % kGT) * kGT + (b % kGT);
  double s = 0.0;
  for (int q = 0; q < nslices; ++q) s += part[((long long)q * npairs + pidx) * (kGT * kGT) + off];
  G[idx] = s;
}

size_t gram_part_doubles(int m, int k) {
  const GramPlan g = gram_plan(m, k);
  return (size_t)g.nslices * g.npairs * kGT * kGT;
}

void gram(const double* AS, int m, int k, double* part, double* G, cudaStream_t s) {
  const GramPlan g = gram_plan(m, k);
  gram_part_kernel<<<dim3(g.npairs, g.nslices), 256, 0, s>>>(AS, m, k, g.slice, g.npairs, part);
  gram_fin_kernel<<<(unsigned)(((long long)k * k + 255) / 256), 256, 0, s>>>(part, g.nslices, g.npairs, k, G);
}

// Cholesky G = L L^T in place (lower triangle of the column-major k x k G) and
// X = L^-1 together, blocked and right-looking, kCb columns a panel, as
// stream-ordered launches.  With D the panel's diagonal block of L:
//   chol_diag_kernel: one block forms D and D^-1 in shared memory, a column of
//     one and a row of the other a step (the steps depend on one another, so
//     they are short loops: unrolled into registers of one warp, the code's
//     own fetches took 69 us a panel);
//   chol_rows_kernel: below the panel L_i = G_i D^-T, left of it X_j = D^-1 X_j;
//   chol_update_kernel: G_IJ -= L_I L_J^T and X_I -= L_I X_j below the panel.
// FP64 runs at two lanes per clock per SM on this part, so the products are
// cut into CTAs of 256 outputs, 32 multiply-adds each (2 us), and D is applied
// as an inverse instead of by substitution.  A pivot at or below 1e-12 of its
// column's initial squared norm (diag0, saved first) means the selected
// columns are linearly dependent to working precision: the pivot is replaced
// by 1 and status[0] = 1.  Factor and inverse together, measured: k = 128
// 472 -> 172 us (one block in shared memory, then a substitution per
// column), k = 256 656 -> 346 us (blocked with substitutions).
constexpr int kCb = 32;

__global__ void chol_save_kernel(const double* __restrict__ G, int k, double* __restrict__ diag0) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < k) diag0[j] = G[(long long)j * k + j];
}

__global__ void __launch_bounds__(256) chol_diag_kernel(double* __restrict__ G, double* __restrict__ X, int k, int j0,
                                                        const double* __restrict__ diag0,
                                                        int* __restrict__ status) {
  __shared__ double D[kCb][kCb + 1], V[kCb][kCb + 1];   // the block, and D^-1 as it forms
  const int t = threadIdx.x, b = min(kCb, k - j0);
  for (int e = t; e < kCb * kCb; e += 256) {
    const int r = e % kCb, c = e / kCb;
    D[r][c] = r < b && c <= r ? G[(long long)(j0 + c) * k + j0 + r] : 0.0;
    V[r][c] = r == c ? 1.0 : 0.0;
  }
  __syncthreads();
  // (a single panel's initial diagonal is its own)
  const double least = t < b ? 1e-12 * (diag0 ? diag0[j0 + t] : D[t][t]) : 0.0;
  __syncthreads();
  bool bad = false;
  for (int c = 0; c < b; ++c) {
    if (t < kCb) {
      // column c of L and row c of D^-1 are done but for the pivot
      const double d = D[c][c];
      const bool ok = d > __shfl_sync(0xffffffffu, least, c);
      bad |= !ok;
      const double r = ok ? rsqrt(d) : 1.0;
      __syncwarp();
      if (t == c) D[c][c] = ok ? d * r : 1.0;
      else if (t > c) D[t][c] *= r;
      if (t <= c) V[c][t] *= r;
    }
    __syncthreads();
    // rows below: column c out of the block's trailing part and of D^-1
    const int q = t / 8;
    if (q > c && q < b) {
      const double l = D[q][c];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // (one multiply-add for both: a branch would issue two)
        const int x = t % 8 + 8 * i;
        double* to = x <= c ? &V[q][x] : &D[q][x];
        const double by = x <= c ? V[c][x] : D[x][c];
        if (x <= q) *to = fma(-l, by, *to);
      }
    }
    __syncthreads();
  }
  if (t == 0 && bad) status[0] = 1;
  for (int e = t; e < kCb * kCb; e += 256) {
    const int r = e % kCb, c = e / kCb;
    if (r < b && c <= r) G[(long long)(j0 + c) * k + j0 + r] = D[r][c];
    if (r < b && c < b) X[(long long)(j0 + c) * k + j0 + r] = V[r][c];   // (zero above the diagonal)
  }
}

// Blocks 0 .. nlow - 1: eight rows of L below the panel; the others: eight
// columns of X's panel rows.
__global__ void __launch_bounds__(256) chol_rows_kernel(double* __restrict__ G, double* __restrict__ X, int k, int j0,
                                                        int nlow) {
  __shared__ double D[kCb][kCb + 1], V[8][kCb + 1];
  const int b = min(kCb, k - j0), t = threadIdx.x;
  const bool low = (int)blockIdx.x < nlow;
  for (int e = t; e < kCb * kCb; e += 256) {
    const int r = e % kCb, c = e / kCb;
    D[r][c] = r < b && c <= r ? X[(long long)(j0 + c) * k + j0 + r] : 0.0;
  }
  const int at = low ? j0 + b + blockIdx.x * 8 : ((int)blockIdx.x - nlow) * 8;   // first row of L, or column of X
  const int v = low ? t % 8 : t / kCb, q = low ? t / 8 : t % kCb;
  const bool in = q < b && at + v < (low ? k : j0);
  double* p = low ? G + (long long)(j0 + q) * k + at + v : X + (long long)(at + v) * k + j0 + q;
  V[v][q] = in ? *p : 0.0;
  __syncthreads();
  double acc = 0.0;
#pragma unroll 8
  for (int e = 0; e < kCb; ++e) acc = fma(V[v][e], D[q][e], acc);
  if (in) *p = acc;
}

// 16 x 16 outputs a block: lower tiles of G's trailing part, then the tiles
// of X's rows below the panel (columns up to the panel's last).
__global__ void __launch_bounds__(256) chol_update_kernel(double* __restrict__ G, double* __restrict__ X, int k,
                                                          int j0, int ntri, int xcols) {
  __shared__ double P[16][kCb + 1], Q[16][kCb + 1];
  const int t0 = j0 + kCb, t = threadIdx.x, bid = blockIdx.x;   // (a panel with rows below it is full)
  const bool tri = bid < ntri;
  int ti, tj;
  if (tri) {
    ti = (int)((sqrtf(8.f * bid + 1.f) - 1.f) * 0.5f);
    while (ti * (ti + 1) / 2 > bid) --ti;
    while ((ti + 1) * (ti + 2) / 2 <= bid) ++ti;
    tj = bid - ti * (ti + 1) / 2;
  } else {
    ti = (bid - ntri) / xcols;
    tj = (bid - ntri) % xcols;
  }
  const int r0 = t0 + ti * 16, c0 = (tri ? t0 : 0) + tj * 16;
  for (int e = t; e < 16 * kCb; e += 256) {
    const int r = e % 16, q = e / 16;
    P[r][q] = r0 + r < k ? G[(long long)(j0 + q) * k + r0 + r] : 0.0;
    if (tri) Q[r][q] = c0 + r < k ? G[(long long)(j0 + q) * k + c0 + r] : 0.0;
  }
  if (!tri)
    for (int e = t; e < 16 * kCb; e += 256) {
      const int q = e % kCb, c = e / kCb;
      Q[c][q] = X[(long long)(c0 + c) * k + j0 + q];
    }
  __syncthreads();
  const int r = t % 16, c = t / 16;
  const int i = r0 + r, l = c0 + c;
  if (i >= k || (tri && l > i)) return;
  double acc = 0.0;
#pragma unroll 8
  for (int q = 0; q < kCb; ++q) acc = fma(P[r][q], Q[c][q], acc);
  (tri ? G : X)[(long long)l * k + i] -= acc;
}

// Cholesky of the k x k matrix in G (overwritten by L) and L^-1 into Linv
// (status[0] = 1 for a rank-deficient G).  diag0: k doubles of scratch.
void chol_inv(double* G, int k, double* Linv, double* diag0, int* status, cudaStream_t s) {
  if (k > kCb) {
    cudaMemsetAsync(Linv, 0, (size_t)k * k * sizeof(double), s);
    chol_save_kernel<<<(k + 255) / 256, 256, 0, s>>>(G, k, diag0);
  } else {
    diag0 = nullptr;
  }
  for (int j0 = 0; j0 < k; j0 += kCb) {
    const int below = std::max(0, k - j0 - kCb);
    chol_diag_kernel<<<1, 256, 0, s>>>(G, Linv, k, j0, diag0, status);
    const int nlow = (below + 7) / 8, nx = j0 / 8;
    if (nlow + nx > 0) chol_rows_kernel<<<nlow + nx, 256, 0, s>>>(G, Linv, k, j0, nlow);
    if (below > 0) {
      const int T = (below + 15) / 16, ntri = T * (T + 1) / 2, xcols = (j0 + kCb) / 16;
      chol_update_kernel<<<ntri + T * xcols, 256, 0, s>>>(G, Linv, k, j0, ntri, xcols);
    }
  }
}

// Q = A_S L^-T (m x k): Q[i, j] = sum_{l <= j} A_S[i, l] Linv[j, l].
__global__ void q_kernel(const double* __restrict__ AS, const double* __restrict__ Linv, int m, int k,
                         double* __restrict__ Q) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)m * k) return;
  const int i = (int)(idx % m), j = (int)(idx / m);
  double acc = 0.0;
  for (int l = 0; l <= j; ++l) acc = fma(AS[(long long)l * m + i], Linv[(long long)l * k + j], acc);
  Q[idx] = acc;
}

// Above this many columns G = A_S^T A_S and Q = A_S L^-T run on the slice GEMM.
// css_embed with n = 256 (two rounds of both), us with the FP64 kernels and with
// slices: m = 512, l = 128 679 and 862, l = 256 1065 and 1210; m = 1024, l = 128
// 703 and 864, l = 256 1168 and 1212; m = 4096, l = 65 613 and 714, l = 128 859
// and 870, l = 160 1076 and 956, l = 256 2109 and 1228; m = 16384, l = 32 470 and
// 584, l = 65 971 and 776, l = 256 5569 and 1546.  (The two meet near m l^2 =
// 2^26, so the line fits 4096 rows; for 129 to 256 columns of 512 it costs 25 to
// 14 %, for 65 to 128 of 16384 it gives away 20 to 43 %.)
constexpr int kSliceK = 128;

// A_S's orthonormal basis by Cholesky: G = A_S^T A_S = L L^T, Q = A_S L^-T.
constexpr int kErr = kAuxErrOffset / sizeof(int);

struct OrthSpace {
  double *G, *gpart, *Linv;
  sg::Digits DS, DSr, DL;   // parts of A_S both ways (in one space), L^-1
  long long part_k, part_rows;
  int* kexp;                // of the sizes of A_S's columns
  sg::Scratch sc;
  int* status;              // [0] rank deficient, [kErr] error of the products
};
OrthSpace carve_orth(WsCarver& c, int* status, long long m, int k) {
  OrthSpace w{};
  w.status = status;
  w.G = c.take<double>((size_t)k * k);
  w.gpart = c.take<double>(gram_part_doubles((int)m, k));
  w.Linv = c.take<double>((size_t)k * k);
  return w;
}
void carve_orth_digits(WsCarver& c, long long m, int k, OrthSpace& w) {
  if (k <= kSliceK) return;
  w.part_k = std::min<long long>(m, sg::part_k(k));
  w.part_rows = std::min<long long>((m + 127) / 128 * 128, sg::part_rows(k));
  const size_t at = c.off;
  w.DS = sg::carve_digits(c, k, w.part_k);
  const size_t end = c.off;
  c.off = at;
  w.DSr = sg::carve_digits(c, w.part_rows, k);
  c.off = std::max(c.off, end);
  w.DL = sg::carve_digits(c, k, k);
  w.kexp = c.take<int>(k);
  w.sc = sg::carve_scratch(c, std::max(sg::sum_words(k, k, w.part_k, 1), sg::sum_words(w.part_rows, k, k, 0)));
}
cudaError_t orth(const double* AS, int m, int k, double* Q, OrthSpace& w, unsigned long long spin_ns,
                 cudaStream_t s) {
  cudaError_t e;
  const long long mk = (long long)m * k;
  if (k <= kSliceK) {
    gram(AS, m, k, w.gpart, w.G, s);
    chol_inv(w.G, k, w.Linv, w.gpart, w.status, s);
    q_kernel<<<(unsigned)((mk + 255) / 256), 256, 0, s>>>(AS, w.Linv, m, k, Q);
    return cudaGetLastError();
  }
  for (long long r0 = 0; r0 < m; r0 += w.part_k) {
    const sg::Source a{AS + r0, CSS_F64, m, 1, k, (int)std::min(w.part_k, m - r0)};
    if ((e = sg::split(a, w.DS, s)) != cudaSuccess) return e;
    const sg::Store st{w.G, 1, k, 1, nullptr, nullptr, r0 > 0};
    if ((e = sg::gemm(w.DS, w.DS, st, w.sc, w.status + kErr, spin_ns, s)) != cudaSuccess) return e;
  }
  // Q = (A_S D^-1)(D L^-T), D^2 the diagonal of G: columns of very different
  // sizes (a greedy choice on graded data) at one size
  sg::gram_exponents(w.G, k, k, w.kexp, s);
  chol_inv(w.G, k, w.Linv, w.gpart, w.status, s);
  const sg::Source li{w.Linv, CSS_F64, 1, k, k, k, w.kexp, 1};
  if ((e = sg::split(li, w.DL, s)) != cudaSuccess) return e;
  for (long long r0 = 0; r0 < m; r0 += w.part_rows) {
    const sg::Source ar{AS + r0, CSS_F64, 1, m, (int)std::min(w.part_rows, m - r0), k, w.kexp, -1};
    if ((e = sg::split(ar, w.DSr, s)) != cudaSuccess) return e;
    if ((e = sg::gemm(w.DSr, w.DL, sg::Store{Q + r0, 1, m, 0}, w.sc, w.status + kErr, spin_ns, s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The call's status once its work is enqueued (opts->sync): [0] A_S is rank
// deficient, [kErr] a product's wait ran out (where css_read_status looks).
css_status finish(const int* status, const css_opts& o, cudaStream_t s) {
  if (!o.sync) return CSS_OK;
  int st[kErr + 1] = {};
  if (cudaMemcpyAsync(st, status, sizeof(st), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CSS_ERR_CUDA;
  if (st[kErr]) return (css_status)st[kErr];
  return st[0] ? CSS_ERR_INVALID_ARG : CSS_OK;   // A_S is rank deficient
}

// -------------------------------------------------- products in digits -----
// W = Q^T A, R = A - Q W and P = R W^T run on the slice GEMM (slice_gemm.cu),
// a range of columns of A at a time, which bounds the workspace: as many tiles
// of 128 columns as kDigitBudget of A's digits hold, cut to a whole number of
// rounds over the 152 SMs.  Where not even one tile's do (m above 655360) the
// rows are taken in parts as well.
constexpr int kRound = 152;

// Rows a part of W = Q^T A.
long long w_rows(long long m, int k) { return std::min(m, sg::part_k(std::max(k, 128))); }

long long chunk_cols(long long m, long long n, int k) {
  const long long tiles = (n + 127) / 128, tn = (k + 127) / 128;
  const long long per_tile = 128 * 16 * ((w_rows(m, k) + 63) / 64 * 64);
  long long c = std::max<long long>(1, sg::kDigitBudget / per_tile);
  if (c * tn > kRound) c = c * tn / kRound * kRound / tn;
  return std::min(c, tiles) * 128;
}

// W = Q^T A: element (j, c) to W[j * wj + c * wc].  DQ: whether the digits of
// the whole of Q are already there.
cudaError_t w_product(const double* Q, const void* A, int dtype, long long lda, int m, int n, int k, double* W,
                      long long wj, long long wc, sg::Digits& DQ, bool have_q, sg::Digits& DA, const sg::Scratch& sc,
                      int* err, unsigned long long spin_ns, cudaStream_t s) {
  const long long cols = chunk_cols(m, n, k), rows = w_rows(m, k);
  const long long esz = dtype == CSS_F64 ? 8 : dtype == CSS_F32 ? 4 : 2;
  for (long long c0 = 0; c0 < n; c0 += cols) {
    for (long long r0 = 0; r0 < m; r0 += rows) {
      const int mm = (int)std::min(rows, m - r0);
      const sg::Source q{Q + r0, CSS_F64, m, 1, k, mm};
      const sg::Source a{(const char*)A + (c0 * lda + r0) * esz, dtype, lda, 1, (int)std::min(cols, n - c0), mm};
      cudaError_t e = cudaSuccess;
      if (rows < m || (c0 == 0 && !have_q)) e = sg::split(q, DQ, s);
      if (e == cudaSuccess) e = sg::split(a, DA, s);
      if (e != cudaSuccess) return e;
      const sg::Store st{W + c0 * wc, wc, wj, 0, nullptr, nullptr, r0 > 0};
      if ((e = sg::gemm(DA, DQ, st, sc, err, spin_ns, s, a, q)) != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// ------------------------------------------ products of small calls in FP64 --
// out(i, j) = sum_q x(i, q) y(j, q) in FP64: 8 x 8 outputs a block, four threads
// an output (q mod 4), the next 32 q in registers.  COMP: products and sums with
// their rounding errors (Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26, 2005),
// so that FP64 input loses nothing against digits; FP32 and BF16 input has its
// results rounded to FP32 anyway.  Digits take five launches a product, which is
// what a small call waits for; FP64's two lanes a clock and SM set the other side.
constexpr int kSo = 8, kSq = 32, kSp = kSq + 4;   // (rows padded: no bank conflicts)
template <typename TX, bool COMP>
__global__ void __launch_bounds__(256) small_sums_kernel(const TX* __restrict__ x, long long xr, long long xq,
                                                         const double* __restrict__ y, long long yr, long long yq,
                                                         int M, int N, int K, double* __restrict__ out, long long os,
                                                         long long oc) {
  __shared__ double sx[2][kSo * kSp], sy[2][kSo * kSp];
  const int t = threadIdx.x, tm = (M + kSo - 1) / kSo;
  const int i0 = (int)(blockIdx.x % tm) * kSo, j0 = (int)(blockIdx.x / tm) * kSo;
  // staging: one entry of each operand a thread, along its contiguous index
  const int xrow = xq == 1 ? t / kSq : t % kSo, xk = xq == 1 ? t % kSq : t / kSo;
  const int yrow = yq == 1 ? t / kSq : t % kSo, yk = yq == 1 ? t % kSq : t / kSo;
  auto get_x = [&](int q0) {
    return i0 + xrow < M && q0 + xk < K ? to_d<TX>(x[(i0 + xrow) * xr + (q0 + xk) * xq]) : 0.0;
  };
  auto get_y = [&](int q0) { return j0 + yrow < N && q0 + yk < K ? y[(j0 + yrow) * yr + (q0 + yk) * yq] : 0.0; };
  const int g = t & 3, i = t >> 2 & 7, j = t >> 5;
  double s = 0.0, c = 0.0, vx = get_x(0), vy = get_y(0);
  int b = 0;
  for (int q0 = 0; q0 < K; q0 += kSq) {
    sx[b][xrow * kSp + xk] = vx;
    sy[b][yrow * kSp + yk] = vy;
    __syncthreads();   // (the other buffer's readers are past the last one)
    vx = get_x(q0 + kSq);
    vy = get_y(q0 + kSq);
#pragma unroll
    for (int e = 0; e < kSq; e += 4) {
      const double u = sx[b][i * kSp + e + g], v = sy[b][j * kSp + e + g];
      if constexpr (COMP) {
        const double p = __dmul_rn(u, v), n = __dadd_rn(s, p), z = __dsub_rn(n, s);
        c += (__dsub_rn(s, __dsub_rn(n, z)) + __dsub_rn(p, z)) + fma(u, v, -p);
        s = n;
      } else {
        s = fma(u, v, s);
      }
    }
    b ^= 1;
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    const double p = __shfl_xor_sync(0xffffffffu, s, o), pc = __shfl_xor_sync(0xffffffffu, c, o);
    const double n = __dadd_rn(s, p), z = __dsub_rn(n, s);
    if constexpr (COMP) c = (c + pc) + (__dsub_rn(s, __dsub_rn(n, z)) + __dsub_rn(p, z));
    s = n;
  }
  // (beside infinities the errors are NaN)
  if (g == 0 && i0 + i < M && j0 + j < N) out[(i0 + i) * os + (j0 + j) * oc] = COMP && isfinite(s) ? s + c : s;
}
template <typename TX, bool COMP>
void small_sums(const TX* x, long long xr, long long xq, const double* y, long long yr, long long yq, int M, int N,
                int K, double* out, long long os, long long oc, cudaStream_t s) {
  const unsigned blocks = (unsigned)((M + kSo - 1) / kSo) * ((N + kSo - 1) / kSo);
  small_sums_kernel<TX, COMP><<<blocks, 256, 0, s>>>(x, xr, xq, y, yr, yq, M, N, K, out, os, oc);
}
// Multiply-adds of a product up to which css_residual_backward's run there, and
// the longest sum (one block's chain).  css.residual forward, then with backward,
// us with digits and here (before digits): FP32 64 x 128, k = 8 276, 772 and 175,
// 539 (208, 606); 256 x 1024, k = 16 335, 904 and 246, 686 (295, 778); 257 x
// 1000, k = 31 351, 990 and 258, 711 (338, 859); 300 x 4000, k = 8 343, 928 and
// 328, 920 (314, 825); beyond 1e7 digits were not slower than what they replaced.
// FP64: 64 x 128, k = 8 290, 839 and 186, 581 (230, 661); 128 x 256, k = 16 347,
// 982 and 245, 724; 256 x 512, k = 8 338, 935 and 333, 961.
constexpr double kSmallMacs = 1e7, kSmallMacsF64 = 524288.0;
constexpr long long kSmallDim = 4096;
bool small_residual(int dt, long long m, long long n, int k) {
  return k <= kSliceK && std::max(m, n) <= kSmallDim &&
         (double)m * n * k <= (dt == CSS_F64 ? kSmallMacsF64 : kSmallMacs);
}

// V = Q W on entry, R = A - V on return (in place), dA = g2 R when dA != null,
// and each block's share of ||R||^2 added to its partial sum (FP64 input, and
// small calls).
constexpr int kLossBlocks = 152 * 8;
template <typename TA>
__global__ void __launch_bounds__(256) residual_f64_kernel(const TA* __restrict__ A, long long lda, int m,
                                                           long long mn, double* __restrict__ R,
                                                           TA* __restrict__ dA, long long ldda, double g2,
                                                           double* __restrict__ loss_part) {
  __shared__ double red[32];
  double sq = 0.0;
  for (long long idx = (long long)blockIdx.x * 256 + threadIdx.x; idx < mn; idx += (long long)gridDim.x * 256) {
    const long long c = idx / m, i = idx - c * m;
    const double r = to_d<TA>(A[c * lda + i]) - R[idx];
    R[idx] = r;
    if (dA) dA[c * ldda + i] = from_d<TA>(g2 * r);
    sq = fma(r, r, sq);
  }
  sq = block_sum(sq, red);
  if (threadIdx.x == 0) loss_part[blockIdx.x] += sq;
}

__global__ void sum_kernel(const double* __restrict__ part, long long cnt, double scale,
                           double* __restrict__ out) {
  __shared__ double red[32];
  double a = 0.0;
  for (long long i = threadIdx.x; i < cnt; i += blockDim.x) a += part[i];
  a = block_sum(a, red);
  if (threadIdx.x == 0) out[0] = a * scale;
}

// dA[:, S[j]] = -2 g sum_{l >= j} P[i, l] Linv[l, j].
template <typename TA>
__global__ void das_kernel(const double* __restrict__ P, const double* __restrict__ Linv, int m, int k,
                           const int* __restrict__ sel, double g2, TA* __restrict__ dA, long long ldda) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)m * k) return;
  const int i = (int)(idx % m), j = (int)(idx / m);
  double acc = 0.0;
  for (int l = j; l < k; ++l) acc += P[(long long)l * m + i] * Linv[(long long)j * k + l];
  dA[(long long)sel[j] * ldda + i] = from_d<TA>(-g2 * acc);
}

struct BwLayout {
  int* status;   // [0] A_S is rank deficient, [kErr] error of the products
  double *AS, *Q, *Psum, *loss_part;
  OrthSpace o;
  bool small;             // products in FP64, in one part
  long long cols, rows;   // of a part
  double* W;     // a part's columns
  void* R;       // a part of the residual: FP32, FP64 for FP64 input and small calls
  sg::Digits DQ, DQr, DW, DWr, DA, DR;   // operands of a part's products (r: the other way round)
  sg::Scratch sc;
  size_t bytes;
};

BwLayout bw_layout(void* ws, size_t cap, int dt, int64_t m, int64_t n, int32_t k, bool grad) {
  WsCarver c(ws, cap);
  BwLayout L{};
  L.status = c.take<int>(64);
  L.AS = c.take<double>((size_t)m * k);
  L.o = carve_orth(c, L.status, m, k);
  L.Q = c.take<double>((size_t)m * k);
  L.Psum = grad ? c.take<double>((size_t)m * k) : nullptr;
  L.loss_part = c.take<double>((size_t)std::max(kLossBlocks, sg::residual_parts()));
  L.small = small_residual(dt, m, n, k);
  if (L.small) {
    L.W = c.take<double>((size_t)k * n);
    L.R = c.take<double>((size_t)m * n);
    L.bytes = c.off;
    return L;
  }
  // the basis is formed before the first part's digits
  const size_t at = c.off;
  carve_orth_digits(c, m, k, L.o);
  const size_t end = c.off;
  c.off = at;
  L.cols = chunk_cols(m, n, k);
  L.rows = std::min<long long>((m + 127) / 128 * 128, sg::part_rows(std::max<long long>(L.cols, k)));
  const long long cols = std::min<long long>(L.cols, n), rows = std::min<long long>(L.rows, m);
  L.W = c.take<double>((size_t)k * cols);
  const size_t rs = dt == CSS_F64 ? 8 : 4;
  L.R = grad || dt == CSS_F64 ? (void*)c.take<char>((size_t)rows * cols * rs) : nullptr;
  L.DQ = sg::carve_digits(c, k, w_rows(m, k));
  L.DQr = sg::carve_digits(c, rows, k);
  L.DWr = sg::carve_digits(c, cols, k);
  L.DW = grad ? sg::carve_digits(c, k, cols) : sg::Digits{};
  size_t words = std::max(sg::sum_words(cols, k, w_rows(m, k), 0), sg::sum_words(128, k, w_rows(m, k), 0));
  if (grad) words = std::max(words, sg::sum_words(rows, k, cols, 0));
  L.sc = sg::carve_scratch(c, words);
  // A's digits are done with when R's are formed
  const size_t da = c.off;
  L.DA = sg::carve_digits(c, cols, w_rows(m, k));
  const size_t da_end = c.off;
  c.off = da;
  if (grad) L.DR = sg::carve_digits(c, rows, cols);
  L.bytes = std::max({c.off, da_end, end});
  return L;
}

template <typename TA>
css_status run_backward(const TA* A, int m, int n, long long lda, const int* sel, int k,
                        double grad_out, TA* dA, long long ldda, double* loss, BwLayout& L,
                        const css_opts& o, cudaStream_t s) {
  constexpr int dt = sizeof(TA) == 8 ? CSS_F64 : sizeof(TA) == 4 ? CSS_F32 : CSS_BF16;
  const unsigned long long spin = o.spin_budget_ns ? o.spin_budget_ns : 2000000000ull;
  const long long mn = (long long)m * n;
  const int parts = L.small ? (int)std::min<long long>(kLossBlocks, (mn + 255) / 256)
                    : dt == CSS_F64 ? kLossBlocks : sg::residual_parts();
  cudaMemsetAsync(L.status, 0, (kErr + 1) * sizeof(int), s);
  L.sc.stall = L.o.sc.stall = o.test_unmet_wait == 2;
  cudaMemsetAsync(L.loss_part, 0, parts * sizeof(double), s);
  int* err = L.status + kErr;
  const long long mk = (long long)m * k;
  gather_cols_kernel<TA><<<(unsigned)((mk + 255) / 256), 256, 0, s>>>(A, lda, m, sel, k, L.AS);
  if (orth(L.AS, m, k, L.Q, L.o, spin, s) != cudaSuccess) return CSS_ERR_CUDA;
  if (L.small) {
    constexpr bool kComp = dt == CSS_F64;
    double* const R = (double*)L.R;
    small_sums<TA, kComp>(A, lda, 1, L.Q, m, 1, n, k, m, L.W, k, 1, s);
    small_sums<double, kComp>(L.Q, 1, m, L.W, k, 1, m, n, k, R, 1, m, s);
    residual_f64_kernel<TA><<<parts, 256, 0, s>>>(A, lda, m, mn, R, dA, ldda, 2.0 * grad_out, L.loss_part);
    if (dA) small_sums<double, kComp>(R, 1, m, L.W, 1, k, m, k, n, L.Psum, 1, m, s);
  }
  for (long long c0 = 0; !L.small && c0 < n; c0 += L.cols) {
    const int nc = (int)std::min(L.cols, n - c0);
    const TA* Ac = A + c0 * lda;
    const sg::Source w{L.W, CSS_F64, 1, k, k, nc}, wr{L.W, CSS_F64, k, 1, nc, k};
    if (w_product(L.Q, Ac, dt, lda, m, nc, k, L.W, 1, k, L.DQ, c0 > 0, L.DA, L.sc, err, spin, s) != cudaSuccess ||
        sg::split(wr, L.DWr, s) != cudaSuccess || (dA && sg::split(w, L.DW, s) != cudaSuccess))
      return CSS_ERR_CUDA;
    for (long long r0 = 0; r0 < m; r0 += L.rows) {
      const int mr = (int)std::min<long long>(L.rows, m - r0);
      const sg::Source qr{L.Q + r0, CSS_F64, 1, m, mr, k};
      TA* const dAc = dA ? dA + c0 * ldda + r0 : nullptr;
      if ((c0 == 0 || L.rows < m) && sg::split(qr, L.DQr, s) != cudaSuccess) return CSS_ERR_CUDA;
      if constexpr (dt == CSS_F64) {
        const sg::Store st{(double*)L.R, 1, mr, 0};
        if (sg::gemm(L.DQr, L.DWr, st, L.sc, err, spin, s, qr, wr) != cudaSuccess) return CSS_ERR_CUDA;
        residual_f64_kernel<TA><<<kLossBlocks, 256, 0, s>>>(Ac + r0, lda, mr, (long long)mr * nc, (double*)L.R, dAc,
                                                            ldda, 2.0 * grad_out, L.loss_part);
      } else {
        const sg::Residual r{Ac + r0, dt, lda, dA ? (float*)L.R : nullptr, dAc, ldda, 2.0 * grad_out, L.loss_part};
        if (sg::gemm_residual(L.DQr, L.DWr, r, L.sc, err, spin, s) != cudaSuccess) return CSS_ERR_CUDA;
      }
      if (!dA) continue;
      const sg::Source r{L.R, dt == CSS_F64 ? CSS_F64 : CSS_F32, 1, mr, mr, nc};
      const sg::Store st{L.Psum + r0, 1, m, 0, nullptr, nullptr, c0 > 0};
      if (sg::split(r, L.DR, s) != cudaSuccess || sg::gemm(L.DR, L.DW, st, L.sc, err, spin, s) != cudaSuccess)
        return CSS_ERR_CUDA;
    }
  }
  if (loss) sum_kernel<<<1, 512, 0, s>>>(L.loss_part, parts, 1.0, loss);
  if (dA)
    das_kernel<TA><<<(unsigned)((mk + 255) / 256), 256, 0, s>>>(L.Psum, L.o.Linv, m, k, sel, 2.0 * grad_out, dA,
                                                               ldda);
  if (cudaGetLastError() != cudaSuccess) return CSS_ERR_CUDA;
  return finish(L.status, o, s);
}

// ------------------------------------------------ embedding (Sec. 3.2) -----
// Copy of an m x l FP64 matrix to a caller buffer with leading dimension ld.
__global__ void copy_cols_kernel(const double* __restrict__ src, int m, int l, double* __restrict__ dst,
                                 long long ld) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)m * l) return;
  const int i = (int)(idx % m), j = (int)(idx / m);
  dst[(long long)j * ld + i] = src[idx];
}

struct EmbLayout {
  int* status;
  double *AS, *Q1, *Q;
  OrthSpace o;
  sg::Digits DQ, DA;
  sg::Scratch sc;
  size_t bytes;
};

EmbLayout emb_layout(void* ws, size_t cap, int64_t m, int64_t n, int32_t l) {
  WsCarver c(ws, cap);
  EmbLayout L{};
  L.status = c.take<int>(64);
  L.AS = c.take<double>((size_t)m * l);
  L.o = carve_orth(c, L.status, m, l);
  L.Q1 = c.take<double>((size_t)m * l);
  L.Q = c.take<double>((size_t)m * l);
  // the basis is formed before W's digits
  const size_t at = c.off;
  carve_orth_digits(c, m, l, L.o);
  const size_t end = c.off;
  c.off = at;
  const long long cols = chunk_cols(m, n, l), rows = w_rows(m, l);
  L.DQ = sg::carve_digits(c, l, rows);
  L.DA = sg::carve_digits(c, std::min<long long>(cols, n), rows);
  L.sc = sg::carve_scratch(c, std::max(sg::sum_words(cols, l, rows, 0), sg::sum_words(128, l, rows, 0)));
  L.bytes = std::max(c.off, end);
  return L;
}

// CholeskyQR2: A_S^T A_S = L1 L1^T, Q1 = A_S L1^-T; Q1^T Q1 = L2 L2^T,
// Q = Q1 L2^-T.  Then W = Q^T A (row t at W + t * ldw).
template <typename TA>
css_status run_embed(const TA* A, int m, int n, long long lda, const int* sel, int l, double* Qout,
                     long long ldq, double* W, long long ldw, EmbLayout& L, const css_opts& o,
                     cudaStream_t s) {
  constexpr int dt = sizeof(TA) == 8 ? CSS_F64 : sizeof(TA) == 4 ? CSS_F32 : CSS_BF16;
  cudaMemsetAsync(L.status, 0, (kErr + 1) * sizeof(int), s);
  L.sc.stall = L.o.sc.stall = o.test_unmet_wait == 2;
  const long long ml = (long long)m * l;
  const unsigned gb = (unsigned)((ml + 255) / 256);
  gather_cols_kernel<TA><<<gb, 256, 0, s>>>(A, lda, m, sel, l, L.AS);
  const unsigned long long spin = o.spin_budget_ns ? o.spin_budget_ns : 2000000000ull;
  if (orth(L.AS, m, l, L.Q1, L.o, spin, s) != cudaSuccess || orth(L.Q1, m, l, L.Q, L.o, spin, s) != cudaSuccess)
    return CSS_ERR_CUDA;
  if (W && w_product(L.Q, A, dt, lda, m, n, l, W, ldw, 1, L.DQ, false, L.DA, L.sc, L.status + kErr, spin, s) != cudaSuccess)
    return CSS_ERR_CUDA;
  if (Qout) copy_cols_kernel<<<gb, 256, 0, s>>>(L.Q, m, l, Qout, ldq);
  if (cudaGetLastError() != cudaSuccess) return CSS_ERR_CUDA;
  return finish(L.status, o, s);
}

// The selected indices are device memory the caller wrote on `s`: read back
// in stream order (one synchronisation) and checked on the host.
css_status check_selection(const int32_t* sel, int32_t k, int64_t n, cudaStream_t s) {
  std::vector<int32_t> h(k);
  if (cudaMemcpyAsync(h.data(), sel, sizeof(int32_t) * k, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return CSS_ERR_CUDA;
  std::vector<char> seen(n, 0);
  for (int32_t v : h) {
    if (v < 0 || v >= n || seen[v]) return CSS_ERR_INVALID_ARG;
    seen[v] = 1;
  }
  return CSS_OK;
}

}  // namespace

size_t embed_workspace_bytes(int64_t m, int64_t n, int32_t l) {
  return emb_layout(nullptr, (size_t)-1, m, n, l).bytes;
}

extern "C" css_status css_embed(const void* A, css_dtype dtype, int64_t m, int64_t n, int64_t lda,
                                const int32_t* sel, int32_t l, double* Q, int64_t ldq, double* W,
                                int64_t ldw, void* ws, size_t ws_bytes, const css_opts* opts,
                                css_stream_t stream) {
  css_opts o;
  css_opts_default(&o);
  if (opts) o = *opts;
  if (!A || !sel || (!Q && !W)) return CSS_ERR_INVALID_ARG;
  if (dtype != CSS_F64 && dtype != CSS_F32 && dtype != CSS_BF16) return CSS_ERR_INVALID_ARG;
  if (m < 1 || n < 1 || lda < m || l < 1 || l > 1024 || l > m || l > n) return CSS_ERR_INVALID_ARG;
  if (m > INT32_MAX || n > INT32_MAX) return CSS_ERR_INVALID_ARG;
  if ((Q && ldq < m) || (W && ldw < n)) return CSS_ERR_INVALID_ARG;
  if (!ws || ((uintptr_t)ws % kWsAlign) != 0) return CSS_ERR_WORKSPACE;
  EmbLayout L = emb_layout(ws, ws_bytes, m, n, l);
  if (L.bytes > ws_bytes) return CSS_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  css_status cs = check_selection(sel, l, n, s);
  if (cs != CSS_OK) return cs;
  switch (dtype) {
    case CSS_F64:
      return run_embed<double>((const double*)A, (int)m, (int)n, lda, sel, l, Q, ldq, W, ldw, L, o, s);
    case CSS_F32:
      return run_embed<float>((const float*)A, (int)m, (int)n, lda, sel, l, Q, ldq, W, ldw, L, o, s);
    default:
      return run_embed<__nv_bfloat16>((const __nv_bfloat16*)A, (int)m, (int)n, lda, sel, l, Q, ldq, W, ldw,
                                      L, o, s);
  }
}

size_t backward_workspace_bytes(int dtype, int64_t m, int64_t n, int32_t k) {
  return bw_layout(nullptr, (size_t)-1, dtype, m, n, k, true).bytes;
}

extern "C" css_status css_residual_backward(const void* A, css_dtype dtype, int64_t m, int64_t n,
                                            int64_t lda, const int32_t* sel, int32_t k,
                                            double grad_out, void* dA, int64_t ldda, double* loss,
                                            void* ws, size_t ws_bytes, const css_opts* opts,
                                            css_stream_t stream) {
  css_opts o;
  css_opts_default(&o);
  if (opts) o = *opts;
  if (!A || !sel || (!dA && !loss)) return CSS_ERR_INVALID_ARG;
  if (dtype != CSS_F64 && dtype != CSS_F32 && dtype != CSS_BF16) return CSS_ERR_INVALID_ARG;
  if (m < 1 || n < 1 || lda < m || k < 1 || k > 1024 || k > m || k > n) return CSS_ERR_INVALID_ARG;
  if (dA && ldda < m) return CSS_ERR_INVALID_ARG;
  if (m > INT32_MAX || n > INT32_MAX) return CSS_ERR_INVALID_ARG;
  if (!ws || ((uintptr_t)ws % kWsAlign) != 0) return CSS_ERR_WORKSPACE;
  BwLayout L = bw_layout(ws, ws_bytes, dtype, m, n, k, dA != nullptr);
  if (L.bytes > ws_bytes) return CSS_ERR_WORKSPACE;
  // the selected indices: in range and distinct (a small stream-ordered copy)
  cudaStream_t s = (cudaStream_t)stream;
  const css_status cs = check_selection(sel, k, n, s);
  if (cs != CSS_OK) return cs;
  switch (dtype) {
    case CSS_F64:
      return run_backward<double>((const double*)A, (int)m, (int)n, lda, sel, k, grad_out,
                                  (double*)dA, ldda, loss, L, o, s);
    case CSS_F32:
      return run_backward<float>((const float*)A, (int)m, (int)n, lda, sel, k, grad_out,
                                 (float*)dA, ldda, loss, L, o, s);
    default:
      return run_backward<__nv_bfloat16>((const __nv_bfloat16*)A, (int)m, (int)n, lda, sel, k,
                                         grad_out, (__nv_bfloat16*)dA, ldda, loss, L, o, s);
  }
}
