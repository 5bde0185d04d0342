// Products to FP64 accuracy on the BF16 tensor cores.
//
// FP64 multiply-adds issue at two lanes per clock and SM on this part and
// double-float ones cost about eleven FP32 operations, while the BF16 tensor
// cores run some 1500 times the FP64 rate.  So a dense product whose result
// must keep 48 to 53 bits is formed from integer digits (the error-free
// transformation of Ozaki, Ogita, Oishi and Rump, Numerical Algorithms 59,
// 2012, with tensor cores as in Mukunoki, Ozaki, Ogita and Imamura, 2020):
//
//   row i of an operand is scaled by a power of two so that every entry is at
//   most 1/2, and written in base 256 with balanced digits,
//     x = sum_{s=1..8} d_s 256^-s,   |d_s| <= 128  (exact in BF16).
//   x y = sum over w = s + t of 256^-w d_s e_t, and w = 2..9 is kept.  The
//   seven pairs of w = 10 are at most 2^14 each, so with the rounding to eight
//   digits less than 2^-62 of the scaled entries is dropped, and with row
//   maxima in [1/4, 1/2) less than 2^-58 of the product of the two rows'
//   largest entries, a term.
//
// This is fixed point per row: an entry down to about 2^-10 of its row's
// largest keeps FP64's 53 bits, a smaller one fewer.  Sums are normwise more
// accurate than FP64 ones (below); where an inner index that dominates X's rows
// meets zeros in Y, callers balance the operands first (gram_exponents).
//
// Each w has its own TMEM accumulator.  A product of digits is at most 2^14,
// so an accumulator that has taken at most 1024 of them holds an integer of
// at most 2^24, which FP32 accumulation represents exactly whatever its
// rounding; it is then drained into 64-bit integers (or double-float for the
// residual).  The whole sum is exact but for the dropped digits and the
// conversion of the result, so it does not depend on the order of the work,
// and split-K partial sums may meet in integer atomics.
//
// Measured: W = Q^T A of a 4096 x 65536 BF16 matrix with l = 256 (68.7 G
// multiply-adds) 24 ms as double-float on the FP32 pipe; here 2.3 ms and 0.7 ms
// for the split of A; its error against 64 bits fell from 1.1e-12 to 2.2e-15.
// The tensor pipe is active 57 % of the time there (ncu; 61 to 66 % with k = 128
// and in Gram matrices), and 27 % in the residual's product, whose epilogue reads
// A and writes R and dA; the rest is the drains, during which the accumulators
// cannot take products.  G = W W^T, 256 x 65536: 4.26 ms
// in FP64 instructions, 0.17 ms here.
//
// Slices that are zero in a block of 128 rows x 64 k are not stored, loaded
// or multiplied: BF16 entries of similar size have three non-zero slices,
// FP32 ones five.
//
// One CTA of the product owns a 128 x 128 tile of the result: four
// accumulators of 128 columns are all of TMEM, so the eight w run as two
// halves, low digits first.  (With all eight resident at 64 columns the
// 128 x 64 x 16 MMAs would read 6 KB of shared memory in the time of 4 KB.)
#include "slice_gemm.cuh"

#include <algorithm>

#include "tc_ptx.cuh"

namespace css {
namespace sg {
namespace {

using namespace css::tc;

// A value held as the unevaluated sum s + c of two FP32 numbers.
struct DF {
  float s, c;
};

constexpr int kT = 128;                 // rows of an operand tile
constexpr int kS = 8;                   // slices
constexpr int kSliceBytes = kT * 16 * 2;   // one slice of a tile's 16 k
constexpr int kKb = 64;                 // k per zero-slice count
constexpr int kBudget = 1024;           // digit products per accumulator between drains

__host__ __device__ inline long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }

__host__ __device__ inline int exp_bias(int dtype) { return dtype == CSS_F64 ? 1023 : 127; }
// in the place of the largest exponent of a row that holds an infinity, a NaN
constexpr int kExInf = 1 << 20, kExNan = 1 << 21;
// entries of a row with largest biased exponent e are at most 2^(scale_exp - 1)
__device__ __forceinline__ int scale_exp(int e, int dtype) { return e - exp_bias(dtype) + 2; }

__device__ __forceinline__ int biased_exp(double v) {
  const int h = __double2hiint(v), e = (h >> 20) & 0x7ff;
  return e < 0x7ff ? e : (h & 0xfffff) | __double2loint(v) ? kExNan : kExInf;
}
__device__ __forceinline__ int biased_exp(float v) {
  const int b = __float_as_int(v), e = (b >> 23) & 0xff;
  return e < 0xff ? e : b & 0x7fffff ? kExNan : kExInf;
}
// with 2^ke applied: zeros have none, subnormals that of their range
__device__ __forceinline__ int scaled_exp(double v, int ke) {
  const int e = biased_exp(v);
  return e >= kExInf ? e : v == 0.0 ? 0 : max(e, 1) + ke;
}
__device__ __forceinline__ float load_val(const float* p) { return __ldg(p); }
__device__ __forceinline__ double load_val(const double* p) { return __ldg(p); }
__device__ __forceinline__ float load_val(const __nv_bfloat16* p) {
  return __uint_as_float(((uint32_t)__ldg((const unsigned short*)p)) << 16);
}

// 8 consecutive elements at p
template <bool VEC>
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&v)[8]) {
  if (VEC) {
    const uint4 r = __ldg(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { v[2 * i] = bf16_lo(w[i]); v[2 * i + 1] = bf16_hi(w[i]); }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = load_val(p + i);
  }
}
template <bool VEC>
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  if (VEC) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 r = __ldg(reinterpret_cast<const float4*>(p) + i);
      v[4 * i] = r.x; v[4 * i + 1] = r.y; v[4 * i + 2] = r.z; v[4 * i + 3] = r.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = load_val(p + i);
  }
}
template <bool VEC>
__device__ __forceinline__ void load8(const double* p, double (&v)[8]) {
  if (VEC) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double2 r = __ldg(reinterpret_cast<const double2*>(p) + i);
      v[2 * i] = r.x; v[2 * i + 1] = r.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = load_val(p + i);
  }
}

// The block's 128 rows x 64 k in registers: each thread four chunks of 8
// consecutive k.  KC (k contiguous): chunk q = row tid / 8 + 32 q, k chunk
// tid % 8, so that eight lanes read a row's 64 k.  Otherwise rows are
// contiguous: row tid % 128, k chunk tid / 128 + 2 q.  Zero outside.
template <typename T, typename V, bool KC, bool VEC>
__device__ __forceinline__ void load_block(const T* p, long long rs, long long ks, int rows, int K, int r0, int k0,
                                           V (&v)[4][8]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int row = r0 + (KC ? (int)threadIdx.x / 8 + 32 * q : (int)threadIdx.x % 128);
    const int k = k0 + 8 * (KC ? (int)threadIdx.x % 8 : (int)threadIdx.x / 128 + 2 * q);
#pragma unroll
    for (int e = 0; e < 8; ++e) v[q][e] = V(0);
    if (row >= rows) continue;
    const T* src = p + row * rs + k * ks;
    if (KC && k + 8 <= K) {
      load8<VEC>(src, v[q]);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (k + e < K) v[q][e] = load_val(src + e * ks);
    }
  }
}

// First k of this thread's chunk q, and the exponent applied at k.
template <bool KC>
__device__ __forceinline__ int k_of(int k0, int q) {
  return k0 + 8 * (KC ? (int)threadIdx.x % 8 : (int)threadIdx.x / 128 + 2 * q);
}
__device__ __forceinline__ int k_exp(const int* kexp, int sign, int k, int K) {
  return k < K ? sign * __ldg(kexp + k) : 0;
}

// Largest biased exponents of this thread's entries of a block, by chunk.
template <bool KC, bool SC, typename V>
__device__ __forceinline__ void block_exps(const V (&v)[4][8], const int* kexp, int sign, int k0, int K, int (&best)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if constexpr (SC) best[q] = max(best[q], scaled_exp(v[q][e], k_exp(kexp, sign, k_of<KC>(k0, q) + e, K)));
      else best[q] = max(best[q], biased_exp(v[q][e]));
    }
}

// Largest biased exponent of every row (ex zeroed before): a block takes 128
// rows and every gridDim.y-th 64 k of them.  Memory-bound.
template <typename T, typename V, bool KC, bool VEC, bool SC>
__global__ void __launch_bounds__(256) row_exp_kernel(const T* __restrict__ p, long long rs, long long ks, int rows,
                                                      int K, const int* __restrict__ kexp, int sign,
                                                      int* __restrict__ ex) {
  const int r0 = blockIdx.x * kT;
  int best[4] = {0, 0, 0, 0};
  for (int k0 = blockIdx.y * kKb; k0 < K; k0 += gridDim.y * kKb) {
    V v[4][8];
    load_block<T, V, KC, VEC>(p, rs, ks, rows, K, r0, k0, v);
    block_exps<KC, SC>(v, kexp, sign, k0, K, best);
  }
  if (KC) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) best[q] = max(best[q], __shfl_xor_sync(0xffffffffu, best[q], o));
      const int row = r0 + threadIdx.x / 8 + 32 * q;
      if (threadIdx.x % 8 == 0 && row < rows && best[q] > 0) atomicMax(ex + row, best[q]);
    }
  } else {
    const int row = r0 + threadIdx.x % 128, b = max(max(best[0], best[1]), max(best[2], best[3]));
    if (row < rows && b > 0) atomicMax(ex + row, b);
  }
}

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

// Digits of one block of 128 rows x 64 k; slices are written until what is
// left can give no digit, and their number goes to ns.  Rows with an infinity
// or a NaN get zero digits (see restore_kernel).  WHOLE: of all k of 128 rows,
// whose exponents are formed here too (see kWholeK).
template <typename T, typename V, bool KC, bool VEC, bool SC, bool WHOLE>
__global__ void __launch_bounds__(256) split_kernel(const T* __restrict__ p, long long rs, long long ks, int rows,
                                                    int K, int k64, int dtype, const int* __restrict__ kexp, int sign,
                                                    int* __restrict__ ex, unsigned char* __restrict__ d,
                                                    unsigned char* __restrict__ ns) {
  // (one grid dimension: K / 64 may exceed the others' 65535)
  const unsigned tiles = (unsigned)(rows + kT - 1) / kT, tile = blockIdx.x % tiles;
  const int r0 = (int)tile * kT;
  int es[4] = {0, 0, 0, 0};
  if constexpr (WHOLE) {
    int best[4] = {0, 0, 0, 0};
    for (int k0 = 0; k0 < K; k0 += kKb) {
      V v[4][8];
      load_block<T, V, KC, VEC>(p, rs, ks, rows, K, r0, k0, v);
      block_exps<KC, SC>(v, kexp, sign, k0, K, best);
    }
    if (KC) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) best[q] = max(best[q], __shfl_xor_sync(0xffffffffu, best[q], o));
        es[q] = best[q];
        const int row = r0 + threadIdx.x / 8 + 32 * q;
        if (threadIdx.x % 8 == 0 && row < rows) ex[row] = best[q];
      }
    } else {
      __shared__ int s_best[2][kT];
      s_best[threadIdx.x / kT][threadIdx.x % kT] = max(max(best[0], best[1]), max(best[2], best[3]));
      __syncthreads();
      const int row = threadIdx.x % kT, b = max(s_best[0][row], s_best[1][row]);
#pragma unroll
      for (int q = 0; q < 4; ++q) es[q] = b;
      if (threadIdx.x < kT && r0 + row < rows) ex[r0 + row] = b;
    }
  }
  for (int kb = WHOLE ? 0 : (int)(blockIdx.x / tiles), kend = WHOLE ? k64 : kb + 1; kb < kend; ++kb) {
    V v[4][8];
    load_block<T, V, KC, VEC>(p, rs, ks, rows, K, r0, kb * kKb, v);
    unsigned char* out[4];
    unsigned long long G[4][8];   // FP64: the balanced digits of |x|, biased by 128 but for the first
    uint32_t neg[4] = {0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int rl = KC ? (int)threadIdx.x / 8 + 32 * q : (int)threadIdx.x % 128;
      const int kc = KC ? (int)threadIdx.x % 8 : (int)threadIdx.x / 128 + 2 * q;
      out[q] = d + (((long long)tile * k64 + kb) * 4 + kc / 2) * (kS * kSliceBytes) + (kc % 2) * (kT * 16) + rl * 16;
      const int e = WHOLE ? es[q] : r0 + rl < rows ? ex[r0 + rl] : 0;
      const bool dead = e >= kExInf;
      if constexpr (sizeof(V) == 4) {
        // two factors, so that neither leaves FP32's range
        const int sh = 8 - scale_exp(e, dtype), h1 = sh / 2;
        const float f1 = pow2f(h1), f2 = pow2f(sh - h1);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[q][i] = dead ? 0.f : v[q][i] * f1 * f2;
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const unsigned long long b = (unsigned long long)__double_as_longlong(v[q][i]);
          const int be = (int)(b >> 52) & 0x7ff;
          unsigned long long mant = b & 0xfffffffffffffull;
          if (be > 0) mant |= 1ull << 52;
          // |x| 2^(64 - scale), rounded to an integer below 2^63
          const int ke = SC ? k_exp(kexp, sign, k_of<KC>(kb * kKb, q) + i, K) : 0;
          const int sh = max(be, 1) + ke - e + 10;
          unsigned long long F = 0;
          if (!dead) {
            if (sh >= 0) F = mant << sh;
            else if (sh > -64) F = (mant + (1ull << (-sh - 1))) >> -sh;
          }
          if (b >> 63) neg[q] |= 1u << i;
          G[q][i] = F;
        }
      }
    }
    int s = 0;
    for (; s < kS; ++s) {
      int any = 0;
      if constexpr (sizeof(V) == 4) {
        const float least = 0.5f * pow2f(-8 * (kS - 1 - s));
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int i = 0; i < 8; ++i) any |= fabsf(v[q][i]) >= least;
      } else {
        const unsigned long long mask = s == 0 ? ~0ull : (1ull << (64 - 8 * s)) - 1;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int i = 0; i < 8; ++i) any |= (G[q][i] & mask) != 0;
      }
      if (!__syncthreads_or(any)) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float dg[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int x = 2 * i + j;
            if constexpr (sizeof(V) == 4) {
              const float f = (v[q][x] + 12582912.f) - 12582912.f;   // round to nearest integer
              v[q][x] = (v[q][x] - f) * 256.f;
              dg[j] = f;
            } else {
              const unsigned long long b = G[q][x] + 0x0080808080808080ull;
              const uint32_t byte = (uint32_t)(b >> (56 - 8 * s)) & 0xffu;
              float f = __uint_as_float(0x4b000000u | byte) - (s == 0 ? 8388608.f : 8388736.f);
              dg[j] = (neg[q] >> x) & 1u ? -f : f;
            }
          }
          // digits have at most 8 bits, so their upper halves are their BF16
          w[i] = __byte_perm(__float_as_uint(dg[0]), __float_as_uint(dg[1]), 0x7632);
        }
        *reinterpret_cast<uint4*>(out[q] + s * kSliceBytes) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    if (threadIdx.x == 0) ns[(long long)tile * k64 + kb] = (unsigned char)s;
  }
}

// ------------------------------------------------------------- product -----
constexpr int kStages = 3;
constexpr int kOperandSlot = kS * kSliceBytes;          // 32 KB
constexpr int kStageBytes = 2 * kOperandSlot;
constexpr int kEpiWarps = 8;
constexpr int kThreads = (4 + kEpiWarps) * 32;
// 168 registers a thread at launch; the epilogue's two warpgroups take those
// that the first one (producer, MMA issuer, two idle warps) gives back
constexpr int kRegsIssue = 56, kRegsEpi = 224;
static_assert(4 * kRegsIssue + kEpiWarps * kRegsEpi <= (4 + kEpiWarps) * 168, "within the launch's registers");
constexpr int kSmem = kStages * kStageBytes + 256 + 1024;
constexpr int kCtas = 152;

enum Ep { kEpStore = 0, kEpSplitK = 1, kEpResidual = 2 };

struct Args {
  const unsigned char *xd, *yd, *xns, *yns;
  const int *xe, *ye;
  int xdt, ydt;
  int M, N, K;
  int k16, k64;        // 16-k blocks in use, 64-k blocks stored
  int tn, tiles;       // tiles along N; tiles in all
  int lower;
  int ksplit, k16_per; // K slices and their 16-k blocks (a multiple of 4)
  Store st;
  Source sx, sy;
  long long* part;
  unsigned long long* sums;
  Residual r;
  int* err;
  unsigned long long spin_ns;
  int stall;           // test hook: the epilogue first waits on a phase nothing completes
};

struct Item {
  int tm, tn, k0, k1;
};
__device__ __forceinline__ Item item_of(const Args& P, int it) {
  Item w;
  const int tile = it / P.ksplit, sl = it % P.ksplit;
  if (P.lower) {
    int a = (int)((sqrtf(8.f * tile + 1.f) - 1.f) * 0.5f);
    while (a * (a + 1) / 2 > tile) --a;
    while ((a + 1) * (a + 2) / 2 <= tile) ++a;
    w.tm = a;
    w.tn = tile - a * (a + 1) / 2;
  } else {
    w.tm = tile / P.tn;
    w.tn = tile % P.tn;
  }
  w.k0 = sl * P.k16_per;
  w.k1 = min(P.k16, w.k0 + P.k16_per);
  return w;
}

// Shared-memory descriptors of a K-major operand without swizzle: 8 x 16-byte
// core matrices, 128 bytes apart along the rows, 2 KB apart along k.  Only the
// address field (16-byte units) changes from one MMA to the next.
constexpr uint32_t kDescHi = (128u >> 4) | 1u << 14;
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return (saddr >> 4) | (uint32_t)((kT * 16) >> 4) << 16; }
constexpr uint32_t kDescSlice = kSliceBytes >> 4;
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Element (i, j) of the product as FP64 arithmetic gives it, by a warp.
template <typename TX>
__device__ double warp_dot_x(const Source& x, const Source& y, int i, int j) {
  const TX* p = (const TX*)x.p + i * x.rs;
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int k0 = 0; k0 < x.K; k0 += 1024) {
    const int ke = min(x.K, k0 + 1024);
#pragma unroll 4
    for (int k = k0 + lane; k < ke; k += 32) {
      const long long o = j * y.rs + k * y.ks;
      const double b = y.dtype == CSS_F64   ? ((const double*)y.p)[o]
                       : y.dtype == CSS_F32 ? (double)((const float*)y.p)[o]
                                            : (double)load_val((const __nv_bfloat16*)y.p + o);
      s = fma((double)load_val(p + k * x.ks), b, s);
    }
    if (__any_sync(0xffffffffu, isnan(s))) break;
  }
  return warp_sum(s);
}
__device__ double warp_dot(const Source& x, const Source& y, int i, int j) {
  if (x.dtype == CSS_F64) return warp_dot_x<double>(x, y, i, j);
  if (x.dtype == CSS_F32) return warp_dot_x<float>(x, y, i, j);
  return warp_dot_x<__nv_bfloat16>(x, y, i, j);
}

// The result from its integer sums, (hi 2^32 + lo) 2^(e - 72), rounded once to
// nearest even.  In integer instructions: an FP64 instruction occupies the SM's
// FP64 pipe for 16 clocks, and conversions, scaling and the sum would take
// seven of them an entry.
__device__ __forceinline__ double combine(long long hi, long long lo, int e) {
  unsigned long long b = (unsigned long long)hi << 32;
  long long t = hi >> 32;
  const unsigned long long l = (unsigned long long)lo;
  b += l;
  t += (b < l) + (lo >> 63);
  const bool neg = t < 0;
  unsigned long long a = (unsigned long long)t;
  if (neg) {
    b = ~b + 1;
    a = ~a + (b == 0);
  }
  if ((a | b) == 0) return 0.0;
  // normalised: the leading bit at the top of a
  int n = 0;
  if (a == 0) {
    a = b;
    b = 0;
    n = 64;
  }
  const int z = __clzll((long long)a);
  if (z > 0) {
    a = a << z | b >> (64 - z);
    b <<= z;
  }
  n += z;
  unsigned long long mant = a >> 11;
  const unsigned int rest = (unsigned int)a & 0x7ffu;
  mant += rest > 0x400u || (rest == 0x400u && (b != 0 || (mant & 1)));
  const int ex = 127 - n - 72 + e;
  double v;
  if (ex > -1022 && ex < 1023)
    v = __longlong_as_double((long long)((unsigned long long)(ex + 1022) << 52) + (long long)mant);
  else
    v = scalbn((double)mant, ex - 52);
  return neg ? -v : v;
}

// What stands for an entry without digits: NaN, or nothing where restore_kernel
// will add to what is there.
__device__ __forceinline__ double unformed(const Args& P, int ex) {
  return ex < kExNan && P.st.add && P.sx.p ? 0.0 : __longlong_as_double(0x7fffffffffffffffll);
}

__device__ __forceinline__ void store(const Store& st, int row, int c, double v) {
  if (st.cscale) v *= __ldg(st.cscale + c);
  if (st.out32) {
    st.out32[row * st.rs + c * st.cs] = (float)v;
  } else {
    double* p = st.out + row * st.rs + c * st.cs;
    *p = st.add ? *p + v : v;
  }
}

// sum_i (h_i + l_i)^2 over eight pairs of FP32 values, in FP64's range: the
// squares are formed at the power of two that takes the largest |h_i| to
// [1, 2), so that one below 2^-126 of the largest is all that underflows, and
// summed as a pair.  (Squares in FP64 would cost four FP64 instructions an
// entry, at two lanes a clock and SM; here half of one.)
__device__ __forceinline__ double sum_squares(const float (&h)[8], const float (&l)[8]) {
  int top = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) top = max(top, __float_as_int(h[i]) & 0x7fffffff);
  if (top == 0) return 0.0;
  // two factors, because 2^149 leaves FP32's range (an infinity or a NaN stays one)
  const int e = max(1, top >> 23) - 127, e1 = e / 2;
  const float f1 = pow2f(-e1), f2 = pow2f(e1 - e);
  float sh = 0.f, sl = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float x = h[i] * f1 * f2, y = l[i] * f1 * f2;
    const float p = x * x, pe = fmaf(x, x, -p) + 2.f * x * y;
    const float ns = sh + p, nb = ns - sh;
    sl += ((sh - (ns - nb)) + (p - nb)) + pe;
    sh = ns;
  }
  // an infinite square leaves inf - inf in the low part
  const double s = isfinite(sh) ? to_f64(sh) + to_f64(sl) : to_f64(sh);
  return s * __longlong_as_double((long long)(2 * e + 1023) << 52);
}

// 32 columns of this warp's TMEM lanes
constexpr int kLd = 32;
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

template <int EP>
__global__ void __launch_bounds__(kThreads, 1) slice_gemm_kernel(const __grid_constant__ Args P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* acc_full = empty + kStages;
  uint64_t* acc_empty = acc_full + 1;      // one per accumulator
  uint64_t* done = acc_empty + 4;
  uint64_t* never = done + 1;
  uint32_t* s_tmem = (uint32_t*)(never + 1);
  int* s_chunk = (int*)(s_tmem + 1);       // accumulators in use | last chunk of the half << 4
  int* s_ns = s_chunk + 1;                 // per stage: slices of X | of Y << 8
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int items = P.tiles * P.ksplit;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), 1);
    }
    mbar_init(smem_u32(acc_full), 2);      // the MMAs' commit, and the issuer's own arrival
    for (int g = 0; g < 4; ++g) mbar_init(smem_u32(&acc_empty[g]), kEpiWarps);
    mbar_init(smem_u32(done), 1);
    mbar_init(smem_u32(never), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *s_tmem;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
  if (warp == 0) {
    // ------------------------------------------------------------ producer
    // (the whole warp walks the stages: its lanes hold the slice counts of
    // the next 32 blocks of 64 k)
    int st = 0;
    bool ok = true;
    for (int it = blockIdx.x; ok && it < items; it += gridDim.x) {
      const Item w = item_of(P, it);
      for (int half = 1; ok && half >= 0; --half) {
        const int kps = half ? 1 : 2, cap = half ? kS : 4;
        int cnt = 0;
        for (int k = w.k0; ok && k < w.k1; k += kps, ++st) {
          if ((k - w.k0) % 128 == 0) {
            const int kb = k / 4 + lane;
            cnt = 0;
            if (kb < P.k64)
              cnt = P.xns[(long long)w.tm * P.k64 + kb] | P.yns[(long long)w.tn * P.k64 + kb] << 8;
          }
          const int both = __shfl_sync(0xffffffffu, cnt, ((k - w.k0) / 4) & 31);
          const int nx = min(both & 0xff, cap), ny = min(both >> 8, cap);
          const int slot = st % kStages;
          if (lane == 0) {
            ok = mbar_wait(smem_u32(&empty[slot]), (uint32_t)((st / kStages) & 1) ^ 1u, P.err, P.spin_ns);
            if (ok) {
              s_ns[slot] = nx | ny << 8;
              const uint32_t fb = smem_u32(&full[slot]);
              const int nk = min(kps, w.k1 - k);
              if (nx > 0 && ny > 0) {
                mbar_expect_tx(fb, (uint32_t)(nk * (nx + ny) * kSliceBytes));
                for (int q = 0; q < nk; ++q) {
                  uint8_t* dst = smem + slot * kStageBytes + q * 4 * kSliceBytes;
                  const long long kx = (long long)w.tm * P.k64 * 4 + k + q, ky = (long long)w.tn * P.k64 * 4 + k + q;
                  bulk_load(smem_u32(dst), P.xd + kx * kOperandSlot, (uint32_t)(nx * kSliceBytes), fb);
                  bulk_load(smem_u32(dst + kOperandSlot), P.yd + ky * kOperandSlot, (uint32_t)(ny * kSliceBytes), fb);
                }
              } else {
                mbar_arrive(fb);
              }
            }
          }
          ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
          if (!ok) break;   // this stage was not issued
        }
      }
    }
    // every copy issued has landed before the CTA exits
    if (lane == 0)
      for (int i = max(0, st - kStages); i < st; ++i)
        mbar_drain(smem_u32(&full[i % kStages]), (uint32_t)((i / kStages) & 1));
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA issuer
    const uint32_t idesc = make_idesc(kT, kT, false, false);
    const uint32_t elected = elect_one();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t base = smem_u32(smem);
    int st = 0, slot = 0;
    uint32_t chunk = 0, ph = 0;
    bool ok = true;
    // the accumulators not yet waited for in this chunk, then its end
    auto finish_chunk = [&](int used, int ready, int last) {
      for (int g = 0; ok && g < 4; ++g)
        if (!(ready >> g & 1)) ok = mbar_wait_warp(smem_u32(&acc_empty[g]), (chunk & 1) ^ 1u, P.err, P.spin_ns);
      if (!ok) return;
      if (elected) {
        *s_chunk = used | last;
        umma_commit(smem_u32(acc_full));
        mbar_arrive(smem_u32(acc_full));
      }
      __syncwarp();
      ++chunk;
    };
    for (int it = blockIdx.x; ok && it < items; it += gridDim.x) {
      const Item w = item_of(P, it);
      for (int half = 1; ok && half >= 0; --half) {
        const int kps = half ? 1 : 2, w0 = half ? 6 : 2;
        int used = 0, budget = 0, ready = 0;   // accumulators written, and waited for, in this chunk
        for (int k = w.k0; k < w.k1; k += kps, ++st) {
          ok = mbar_wait_warp(smem_u32(&full[slot]), ph, P.err, P.spin_ns);
          if (!ok) break;
          fence_after();
          const int both = __shfl_sync(0xffffffffu, s_ns[slot], 0);
          const int nx = both & 0xff, ny = both >> 8;
          const int nk = min(kps, w.k1 - k);
          const int cost = nk * 16 * min(nx, ny);
          if (budget + cost > kBudget) {
            // drain before the accumulators can leave FP32's integers
            finish_chunk(used, ready, 0);
            if (!ok) break;
            used = budget = ready = 0;
          }
          budget += cost;
          const uint32_t dx = desc_lo(base + slot * kStageBytes), dy = dx + (kOperandSlot >> 4);
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const int wt = w0 + g;
            const int s_lo = max(1, wt - ny), s_hi = min(nx, wt - 1);
            if (s_lo > s_hi) continue;
            if (!(ready >> g & 1)) {
              ok = ok && mbar_wait_warp(smem_u32(&acc_empty[g]), (chunk & 1) ^ 1u, P.err, P.spin_ns);
              if (!ok) break;
              ready |= 1 << g;
              fence_after();
            }
            uint32_t acc = used >> g & 1;
            used |= 1 << g;
            for (int q = 0; q < nk; ++q) {
              uint32_t xl = dx + (q * 4 + s_lo - 1) * kDescSlice, yl = dy + (q * 4 + wt - s_lo - 1) * kDescSlice;
              for (int s = s_lo; s <= s_hi; ++s) {
                umma_elected(elected, tm + g * kT, xl, yl, kDescHi, idesc, acc);
                acc = 1;
                xl += kDescSlice;
                yl -= kDescSlice;
              }
            }
          }
          if (!ok) break;
          if (elected) umma_commit(smem_u32(&empty[slot]));
          __syncwarp();
          if (++slot == kStages) {
            slot = 0;
            ph ^= 1u;
          }
        }
        if (ok) finish_chunk(used, ready, 16);
      }
    }
    if (elected) {
      umma_commit(smem_u32(done));
      mbar_drain(smem_u32(done), 0u);   // no MMA is in flight when TMEM is released
    }
    __syncwarp();
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    // ------------------------------------------------------------ epilogue
    const int q = warp & 3, ch = (warp - 4) >> 2;   // TMEM lane quarter, column half
    const int r_tile = q * 32 + lane;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * 64);
    uint32_t chunk = 0;
    bool ok = true;
    if (P.stall) ok = mbar_wait_warp(smem_u32(never), 0u, P.err, P.spin_ns);
    double loss = 0.0;            // residual: ||R||^2 of this thread's entries
    for (int it = blockIdx.x; ok && it < items; it += gridDim.x) {
      const Item w = item_of(P, it);
      const int row = w.tm * kT + r_tile, col0 = w.tn * kT + ch * 64;
      // exponents: this thread's row, and the 64 columns over the lanes
      int exr = 0, ey2[2] = {0, 0};
      if (EP != kEpSplitK) {
        if (row < P.M) exr = __ldg(P.xe + row);
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (col0 + 32 * i + lane < P.N) ey2[i] = __ldg(P.ye + col0 + 32 * i + lane);
      }
      long long acc[EP == kEpResidual ? 1 : 64];
      DF df[EP == kEpResidual ? 64 : 1];
      if constexpr (EP == kEpResidual) {
#pragma unroll
        for (int j = 0; j < 64; ++j) df[j] = DF{0.f, 0.f};
      }
      // this thread's 64 entries in the CTA's scratch (hi, then lo halves): the
      // results are formed from there in short loops, because 64 unrolled
      // copies of that code do not stay in the instruction cache
      long long* mine = P.part + (long long)blockIdx.x * (2 * kT * kT) + (long long)(ch * 64) * kT + r_tile;
      for (int half = 1; ok && half >= 0; --half) {
        if constexpr (EP != kEpResidual) {
#pragma unroll
          for (int j = 0; j < 64; ++j) acc[j] = 0;
        }
        bool last = false;
        while (!last) {
          ok = mbar_wait(smem_u32(acc_full), chunk & 1, P.err, P.spin_ns);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          const int info = *(volatile int*)s_chunk;
          last = (info & 16) != 0;
          fence_after();
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const float unit = half ? pow2f(-32 - 8 * g) : pow2f(-8 * g);   // residual: in units of 2^-16
            if (info >> g & 1) {
#pragma unroll
              for (int j0 = 0; j0 < 64; j0 += kLd) {
                float v[kLd];
                tmem_ld(tbase + (uint32_t)(g * kT + j0), v);
#pragma unroll
                for (int jj = 0; jj < kLd; ++jj) {
                  if constexpr (EP == kEpResidual) {
                    const float x = v[jj] * unit;
                    DF& a = df[j0 + jj];
                    const float s = a.s + x, bb = s - a.s;
                    a.c += (a.s - (s - bb)) + (x - bb);
                    a.s = s;
                  } else {
                    acc[j0 + jj] += (long long)__float2int_rn(v[jj]) * (1ll << (24 - 8 * g));
                  }
                }
              }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[g]));
          }
          ++chunk;
        }
        if (!ok) break;
        if constexpr (EP == kEpStore) {
          long long* part = mine + (half ? (long long)kT * kT : 0);
#pragma unroll
          for (int j = 0; j < 64; ++j) __stcg(part + (long long)j * kT, acc[j]);
        } else if constexpr (EP == kEpSplitK) {
          unsigned long long* sums = P.sums + (half ? 0 : (long long)P.M * P.N);
          if (row < P.M) {
#pragma unroll
            for (int j = 0; j < 64; ++j) {
              const int c = col0 + j;
              if (c < P.N) atomicAdd(sums + (long long)c * P.M + row, (unsigned long long)acc[j]);
            }
          }
        }
      }
      if (!ok) break;
      if constexpr (EP == kEpStore) {
        const int ex = scale_exp(exr, P.xdt);
#pragma unroll 1
        for (int j0 = 0; j0 < 64; j0 += 8) {
          long long hv[8], lv[8];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            hv[jj] = __ldcg(mine + (long long)(j0 + jj) * kT);
            lv[jj] = __ldcg(mine + (long long)(kT + j0 + jj) * kT);
          }
          const int ey = j0 < 32 ? ey2[0] : ey2[1];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const int c = col0 + j0 + jj;
            const int eyr = __shfl_sync(0xffffffffu, ey, (j0 + jj) & 31);
            if (row >= P.M || c >= P.N) continue;
            double v = combine(hv[jj], lv[jj], ex + scale_exp(eyr, P.ydt));
            if (max(exr, eyr) >= kExInf) v = unformed(P, max(exr, eyr));
            store(P.st, row, c, v);
            if (P.lower && w.tm != w.tn) store(P.st, c, row, v);
          }
        }
      }
      if constexpr (EP == kEpResidual) {
        float2* pairs = reinterpret_cast<float2*>(mine);
#pragma unroll
        for (int j = 0; j < 64; ++j) __stcg(pairs + (long long)j * kT, make_float2(df[j].s, df[j].c));
        const Residual& R = P.r;
        const int ex = scale_exp(exr, P.xdt) - 16;
        const float gh = (float)R.g2, gl = (float)(R.g2 - (double)gh);
        const bool g_plain = fabsf(gh) < 1e30f && fabsf(gh) > 1e-30f;
        const bool f32 = R.dtype == CSS_F32;
        const bool row_ok = row < P.M;
#pragma unroll 1
        for (int j0 = 0; j0 < 64; j0 += 8) {
          float av[8];
          float2 pv[8];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const int c = col0 + j0 + jj;
            pv[jj] = __ldcg(pairs + (long long)(j0 + jj) * kT);
            av[jj] = 0.f;
            if (row_ok && c < P.N)
              av[jj] = f32 ? load_val((const float*)R.A + (long long)c * R.lda + row)
                           : load_val((const __nv_bfloat16*)R.A + (long long)c * R.lda + row);
          }
          const int ey = j0 < 32 ? ey2[0] : ey2[1];
          float rhi[8], rlo[8];
          unsigned far = 0;   // entries near or beyond FP32's limit, or not numbers
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const int c = col0 + j0 + jj;
            const int eyr = __shfl_sync(0xffffffffu, ey, (j0 + jj) & 31);
            rhi[jj] = rlo[jj] = 0.f;
            if (!row_ok || c >= P.N) continue;
            const int e = ex + scale_exp(eyr, P.ydt);
            const int e1 = max(-126, min(127, e)), e2 = max(-126, min(127, e - e1));
            const float f1 = pow2f(e1), f2 = pow2f(e2);
            float vh = pv[jj].x * f1 * f2;
            const float vl = pv[jj].y * f1 * f2;
            if (max(exr, eyr) >= kExInf) vh = __int_as_float(0x7fffffff);
            const float a = av[jj];
            // r = a - vh - vl as a normalised pair
            const float s = a - vh, bb = s - a;
            const float t = ((a - (s - bb)) + (-vh - bb)) - vl;
            const float rh = s + t, rl = t - (rh - s);
            const bool near = fabsf(s) < 0x1p126f;
            far |= (unsigned)!near << jj;
            rhi[jj] = near ? rh : 0.f;
            rlo[jj] = near ? rl : 0.f;
            if (R.R) R.R[(long long)c * P.M + row] = rh;
            if (R.dA) {
              float g;
              if (g_plain) {
                g = gh * rh;
                // (an infinite product would meet its negative in the low part)
                const float low = fmaf(gh, rh, -g) + (gh * rl + gl * rh);
                g = fabsf(g) < __int_as_float(0x7f800000) ? g + low : g;
              } else {
                g = (float)(R.g2 * ((double)rh + (double)rl));
              }
              if (f32) ((float*)R.dA)[(long long)c * R.ldda + row] = g;
              else ((__nv_bfloat16*)R.dA)[(long long)c * R.ldda + row] = __float2bfloat16_rn(g);
            }
          }
          loss += sum_squares(rhi, rlo);
          // these again, in FP64 (a loop of its own: a branch an entry above
          // cost FP32 4096 x 16384, k = 128, forward and backward, 5.1 -> 6.4 ms)
          if (__any_sync(0xffffffffu, far != 0)) {
#pragma unroll 1
            for (int jj = 0; jj < 8; ++jj) {
              const int c = col0 + j0 + jj, eyr = __shfl_sync(0xffffffffu, ey, (j0 + jj) & 31);
              if (!(far >> jj & 1)) continue;
              const float2 p = __ldcg(pairs + (long long)(j0 + jj) * kT);
              const double f = __longlong_as_double(
                  (long long)(max(-1000, min(1000, ex + scale_exp(eyr, P.ydt))) + 1023) << 52);
              const double av = f32 ? (double)load_val((const float*)R.A + (long long)c * R.lda + row)
                                    : (double)load_val((const __nv_bfloat16*)R.A + (long long)c * R.lda + row);
              double r = (av - (double)p.x * f) - (double)p.y * f;
              if (max(exr, eyr) >= kExInf) r = __longlong_as_double(0x7fffffffffffffffll);
              loss = fma(r, r, loss);
              if (R.R) R.R[(long long)c * P.M + row] = (float)r;
              if (R.dA) {
                const float g = (float)(R.g2 * r);
                if (f32) ((float*)R.dA)[(long long)c * R.ldda + row] = g;
                else ((__nv_bfloat16*)R.dA)[(long long)c * R.ldda + row] = __float2bfloat16_rn(g);
              }
            }
          }
        }
      }
    }
    if constexpr (EP == kEpResidual) {
      // the CTA's share of ||R||^2, in a fixed order
      __shared__ double s_loss[kEpiWarps];
      const double t = warp_sum(loss);
      if (lane == 0) s_loss[warp - 4] = t;
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (warp == 4 && lane == 0) {
        double sum = 0.0;
        for (int i = 0; i < kEpiWarps; ++i) sum += s_loss[i];
        P.r.loss_part[blockIdx.x] += sum;
      }
    }
    fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// The split-K sums (lo half first) to FP64.
__global__ void __launch_bounds__(256) finish_kernel(const __grid_constant__ Args P) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long long)P.M * P.N) return;
  const int row = (int)(idx % P.M), c = (int)(idx / P.M);
  // lower: the tiles above the diagonal were not computed
  const bool up = P.lower && row / kT < c / kT;
  const long long at = up ? (long long)row * P.M + c : idx;
  const int exr = P.xe[row], eyr = P.ye[c];
  double v = combine((long long)P.sums[(long long)P.M * P.N + at], (long long)P.sums[at],
                     scale_exp(exr, P.xdt) + scale_exp(eyr, P.ydt));
  if (max(exr, eyr) >= kExInf) v = unformed(P, max(exr, eyr));
  store(P.st, row, c, v);
}

// A row (of X or Y) with an infinity or a NaN has no digits, and its results
// were stored as NaN.  That is what they are beside a NaN; beside infinities
// they depend on the signs and zeros they meet, so these are formed from the
// sources, a warp an entry.  Most calls find nothing (3 us).  (Inside the
// product, one thread walking K while the others' bounded waits ran, it ended
// FP64 selections of 2304 x 16384 with an infinity in a timeout; called after
// its loops it cost the kernel spills, css_embed of 4096 x 65536 2 %.)
__global__ void __launch_bounds__(256) restore_kernel(const __grid_constant__ Args P) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tn = (P.N + kT - 1) / kT, tiles = (P.M + kT - 1) / kT * tn;
  for (int it = blockIdx.x; it < tiles; it += gridDim.x) {
    const int r0 = it / tn * kT, c0 = it % tn * kT;
    const int at = (threadIdx.x < kT ? r0 : c0) + threadIdx.x % kT;
    const int ex = at >= (threadIdx.x < kT ? P.M : P.N) ? 0 : threadIdx.x < kT ? P.xe[at] : P.ye[at];
    if (!__syncthreads_or(ex >= kExInf && ex < kExNan)) continue;
    for (int row = r0 + warp; row < min(P.M, r0 + kT); row += 8) {
      for (int cb = c0; cb < min(P.N, c0 + kT); cb += 32) {
        const int e = cb + lane < P.N ? max(P.xe[row], P.ye[cb + lane]) : 0;
        for (unsigned todo = __ballot_sync(0xffffffffu, e >= kExInf && e < kExNan); todo; todo &= todo - 1) {
          const int c = cb + __ffs(todo) - 1;
          const double v = warp_dot(P.sx, P.sy, row, c);
          if (lane == 0) store(P.st, row, c, v);
        }
      }
    }
  }
}

int k_blocks(long long K) { return (int)ceil_div(K, kKb); }

// Up to this many k a block forms a row tile's exponents and digits: one launch
// instead of three, which is what small calls wait for (css.embed of 64 x 128,
// l = 8, FP32 229 -> 212 us; css.residual of it 300 -> 267, a launch less of the
// Cholesky panel in it).
constexpr int kWholeK = 128;

template <typename T, typename V, bool KC, bool VEC, bool SC = false>
void launch_split(const Source& src, const Digits& D, cudaStream_t s) {
  const int k64 = k_blocks(src.K);
  const unsigned tiles = (unsigned)ceil_div(src.rows, kT);
  const unsigned ky = (unsigned)std::min<long long>(k64, std::max<long long>(1, ceil_div(152 * 8, tiles)));
  const T* p = (const T*)src.p;
  if (src.K <= kWholeK) {
    split_kernel<T, V, KC, VEC, SC, true><<<tiles, 256, 0, s>>>(p, src.rs, src.ks, src.rows, src.K, k64, src.dtype,
                                                                src.kexp, src.kexp_sign, D.ex, D.d, D.ns);
    return;
  }
  cudaMemsetAsync(D.ex, 0, sizeof(int) * (size_t)src.rows, s);
  row_exp_kernel<T, V, KC, VEC, SC><<<dim3(tiles, ky), 256, 0, s>>>(p, src.rs, src.ks, src.rows, src.K, src.kexp,
                                                                    src.kexp_sign, D.ex);
  split_kernel<T, V, KC, VEC, SC, false><<<tiles * (unsigned)k64, 256, 0, s>>>(
      p, src.rs, src.ks, src.rows, src.K, k64, src.dtype, src.kexp, src.kexp_sign, D.ex, D.d, D.ns);
}
template <typename T, typename V>
void launch_split_of(const Source& src, const Digits& D, cudaStream_t s) {
  const bool vec = ((uintptr_t)src.p & 15u) == 0 && (src.rs * (long long)sizeof(T)) % 16 == 0;
  if constexpr (sizeof(T) == 8) {
    if (src.kexp) {
      if (src.ks == 1 && vec) launch_split<T, V, true, true, true>(src, D, s);
      else if (src.ks == 1) launch_split<T, V, true, false, true>(src, D, s);
      else launch_split<T, V, false, false, true>(src, D, s);
      return;
    }
  }
  if (src.ks == 1 && vec) launch_split<T, V, true, true>(src, D, s);
  else if (src.ks == 1) launch_split<T, V, true, false>(src, D, s);
  else launch_split<T, V, false, false>(src, D, s);
}

Args base_args(const Digits& X, const Digits& Y, int* err, unsigned long long spin_ns) {
  Args P{};
  P.xd = X.d;
  P.yd = Y.d;
  P.xns = X.ns;
  P.yns = Y.ns;
  P.xe = X.ex;
  P.ye = Y.ex;
  P.xdt = X.dtype;
  P.ydt = Y.dtype;
  P.M = X.rows;
  P.N = Y.rows;
  P.K = X.K;
  P.k64 = k_blocks(X.K);
  P.k16 = (int)ceil_div(X.K, 16);
  P.tn = (int)ceil_div(P.N, kT);
  P.tiles = (int)ceil_div(P.M, kT) * P.tn;
  P.ksplit = 1;
  P.k16_per = P.k64 * 4;
  P.err = err;
  P.spin_ns = spin_ns;
  return P;
}

template <int EP>
cudaError_t launch_gemm(const Args& P, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(slice_gemm_kernel<EP>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  slice_gemm_kernel<EP><<<std::min(kCtas, P.tiles * P.ksplit), kThreads, kSmem, s>>>(P);
  return cudaGetLastError();
}

// (without sources the results beside infinities stay NaN)
cudaError_t restore(const Args& P, cudaStream_t s) {
  if (!P.sx.p || !P.sy.p) return cudaSuccess;
  const long long tiles = ceil_div(P.M, kT) * ceil_div(P.N, kT);
  restore_kernel<<<(unsigned)std::min<long long>(8 * kCtas, tiles), 256, 0, s>>>(P);
  return cudaGetLastError();
}

// K slices for `tiles` result tiles: enough items for every SM, slices of at
// least 256 k (a few drains each; below that the atomics of the sums show).
int k_slices(long long tiles, long long K) {
  if (tiles * 2 > kCtas) return 1;
  return (int)std::max<long long>(1, std::min(kCtas / tiles, K / 256));
}

}  // namespace

Digits carve_digits(WsCarver& c, long long rows, long long K) {
  Digits D{};
  const long long tiles = ceil_div(rows, kT), k64 = k_blocks(K);
  D.d = c.take<unsigned char>((size_t)(tiles * k64 * 4 * kS * kSliceBytes));
  D.ns = c.take<unsigned char>((size_t)(tiles * k64));
  D.ex = c.take<int>((size_t)(tiles * kT));
  return D;
}

cudaError_t split(const Source& src, Digits& D, cudaStream_t s) {
  D.rows = src.rows;
  D.K = src.K;
  D.dtype = src.dtype;
  switch (src.dtype) {
    case CSS_F64: launch_split_of<double, double>(src, D, s); break;
    case CSS_F32: launch_split_of<float, float>(src, D, s); break;
    default: launch_split_of<__nv_bfloat16, float>(src, D, s); break;
  }
  return cudaGetLastError();
}

__global__ void gram_exponents_kernel(const double* __restrict__ G, long long ld, int K, int* __restrict__ e) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k >= K) return;
  const int b = biased_exp(G[k * ld + k]);
  // (a zero, an infinity or a NaN: nothing to balance)
  e[k] = b > 0 && b < kExInf ? (b - 1023) >> 1 : 0;
}
void gram_exponents(const double* G, long long ld, int K, int* e, cudaStream_t s) {
  gram_exponents_kernel<<<(K + 255) / 256, 256, 0, s>>>(G, ld, K, e);
}

size_t sum_words(long long M, long long N, long long K, int lower) {
  const long long tm = ceil_div(M, kT), tiles = lower ? tm * (tm + 1) / 2 : tm * ceil_div(N, kT);
  return k_slices(tiles, K) > 1 ? (size_t)(2 * M * N) : 0;
}

Scratch carve_scratch(WsCarver& c, size_t words) {
  Scratch w{};
  w.part = c.take<long long>((size_t)2 * kCtas * kT * kT);
  w.sums = c.take<unsigned long long>(words);
  w.cap = words;
  return w;
}

cudaError_t gemm(const Digits& X, const Digits& Y, const Store& st, const Scratch& w, int* err,
                 unsigned long long spin_ns, cudaStream_t s, const Source& sx, const Source& sy) {
  Args P = base_args(X, Y, err, spin_ns);
  P.st = st;
  P.sx = sx;
  P.sy = sy;
  P.part = w.part;
  P.stall = w.stall;
  P.lower = st.lower;
  if (st.lower) P.tiles = P.tn * (P.tn + 1) / 2;
  const size_t words = sum_words(P.M, P.N, P.K, P.lower);
  P.ksplit = words && words <= w.cap ? k_slices(P.tiles, P.K) : 1;
  if (P.ksplit == 1) {
    cudaError_t e = launch_gemm<kEpStore>(P, s);
    return e == cudaSuccess ? restore(P, s) : e;
  }
  P.sums = w.sums;
  P.k16_per = (int)ceil_div(ceil_div(P.k16, P.ksplit), 4) * 4;
  P.ksplit = (int)ceil_div(P.k16, P.k16_per);
  const size_t mn = (size_t)P.M * P.N;
  cudaError_t e = cudaMemsetAsync(P.sums, 0, 2 * mn * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  if ((e = launch_gemm<kEpSplitK>(P, s)) != cudaSuccess) return e;
  finish_kernel<<<(unsigned)((mn + 255) / 256), 256, 0, s>>>(P);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return restore(P, s);
}

int residual_parts() { return kCtas; }

cudaError_t gemm_residual(const Digits& X, const Digits& Y, const Residual& r, const Scratch& w, int* err,
                          unsigned long long spin_ns, cudaStream_t s) {
  Args P = base_args(X, Y, err, spin_ns);
  P.part = w.part;
  P.stall = w.stall;
  P.r = r;
  return launch_gemm<kEpResidual>(P, s);
}

}  // namespace sg
}  // namespace css
