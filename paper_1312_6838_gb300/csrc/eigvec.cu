// An estimate X of the eigenvectors of the Gram matrix G = W W^T (l x l), so
// that the FP64 Jacobi rounds of lowrank.cu start from X^T G X, which is
// diagonal to rounding for all eigenvalues that FP32 separates.
//
// The cyclic rounds cost about 4 us each whatever they rotate (an L2 trip, a
// grid barrier and FP64 at two lanes per clock and SM), and starting from G
// they take some twelve sweeps of l - 1 rounds: 11.9 of the 13.1 ms of
// css_lowrank at l = 256 (here 2.44 in all: 1.5 for part 1 and 0.9 for parts 2
// and 3, and no sweep is left).  From l = 17 on (l = 31: 1.15 -> 0.39 ms; at
// l = 16 the rounds take 0.37).  A spectrum that FP32 does not resolve leaves
// more sweeps: singular values 1 / i at l = 256 14.2 -> 9.4 ms.  Here:
//   1. estimate_kernel: block Jacobi in FP32 (the ordering of Brent and Luk
//      over 32-column blocks; Golub and Van Loan, Matrix Computations,
//      Sec. 8.5).  A block pair's 64 x 64 matrix is swept once in one CTA's
//      shared memory, 63 rounds without a grid barrier, and the sweep's 64 x 64
//      rotation is then applied to the rest of A and to X by all CTAs: two
//      barriers for 63 rounds.  FP32 issues 64 times the FP64 rate.
//   2. Four steps of the refinement of Ogita and Aishima (Japan J. Indust.
//      Appl. Math. 35, 2018) in FP64: X <- X + X E with E from I - X^T X and
//      X^T G X, which squares the error of every separated pair.  A pair whose
//      correction would not be small keeps its subspace (E only restores
//      orthogonality there) and is left to the Jacobi rounds.
//   3. Two Newton steps X <- X (3 I - X^T X) / 2, so that X is orthogonal to
//      rounding whatever E was, and H = X^T G X.
// The eigenvalues of H are those of G, so the result does not depend on the
// estimate's quality; only the number of Jacobi sweeps does.
#include <algorithm>

#include "eigvec.cuh"

namespace css {
namespace {

constexpr int kB = 32;            // columns of a block
constexpr int kP = 2 * kB;        // columns of a block pair
constexpr int kR = kP - 1;        // rounds of a pair's sweep
constexpr int kNT = 17 * 32;      // 16 warps of updates, one of rotation angles
constexpr int kUp = 16 * 32;
constexpr size_t kSmem = sizeof(float) * (2 * kP * kP + 2 * kP * 16);
static_assert(kSmem >= sizeof(float) * (2 * 4 * kB * (kB + 1) + 4 * kB) && kSmem <= 48 * 1024, "a sweep's arrays fit");
constexpr float kSmallPair = 1e-4f;   // see the sweeps' end

struct EstArgs {
  const double* G;
  int l, lp, L;
  Estimate w;
  DevStatus* st;
};

// Block pair j of round r of the tournament on nb blocks: lower and higher.
__device__ __forceinline__ int2 block_pair(int r, int j, int nb) {
  const int a = j == 0 ? r : (r + j) % (nb - 1);
  const int b = j == 0 ? nb - 1 : (r + nb - 1 - j) % (nb - 1);
  return make_int2(min(a, b), max(a, b));
}
// Global index of local index i of a block pair.
__device__ __forceinline__ int pair_at(int2 bp, int i) { return (i < kB ? bp.x : bp.y) * kB + (i & (kB - 1)); }

// Indices (a, b) of pair j in round r of the tournament on 64 indices.
__device__ __forceinline__ void ab_of(int r, int j, int& a, int& b) {
  a = r + j;
  if (a >= kR) a -= kR;
  b = r - j;
  if (b < 0) b += kR;
  if (j == 0) b = kR;
}
// The angles only have to be close (a rotation is as orthogonal as its c and
// s, and X is made orthogonal in FP64 later), and their chain is what a round
// waits for.
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The rotations of a pair's sweep pass through global memory from the CTA that
// sweeps to the one that forms Q, as single 8-byte words that are zero until
// they are written (c is never 0) and zeroed again once they are read.
__device__ __forceinline__ void put_rotation(unsigned long long* p, float c, float s) {
  const unsigned long long v = (unsigned long long)__float_as_uint(s) << 32 | __float_as_uint(c);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ float2 get_rotation(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}

// Q = J_1 ... J_63 of a pair from its rotations, while they are being formed:
// four rows a warp, in registers.  Lane j holds the entries at the round's
// indices a_j and b_j, which move by one lane from round to round.  (In the
// sweeping CTA this took as many issue slots as the sweep: l = 256 3.05 ms,
// apart 2.69.)
__device__ void build_q(const EstArgs& A, unsigned long long* log, float* Qg) {
  constexpr int kBatch = 7;
  static_assert(kR % kBatch == 0, "whole batches");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  {
    int a, b;
    ab_of(0, lane, a, b);
    float xa[4], xb[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      xa[q] = a == warp * 4 + q ? 1.f : 0.f;
      xb[q] = b == warp * 4 + q ? 1.f : 0.f;
    }
    const uint64_t t0 = globaltimer_ns();
    const bool stall = A.st->stall_where == kRotationWait;   // test hook
    bool stop = false;   // every warp still meets the others below
    for (int r0 = 0; r0 < kR && !stop; r0 += kBatch) {
      float2 v[kBatch];
      for (uint32_t spins = 1; !stop; ++spins) {
        bool have = true;
#pragma unroll
        for (int i = 0; i < kBatch; ++i) v[i] = get_rotation(log + (r0 + i) * kB + lane);
#pragma unroll
        for (int i = 0; i < kBatch; ++i) have &= v[i].x != 0.f;
        if (stall) have = false;
        if (__all_sync(0xffffffffu, have)) break;
        if ((spins & 63u) == 0u) {
          if (ld_volatile_i32(&A.st->code) != 0) {
            stop = true;
          } else if (globaltimer_ns() - t0 > A.st->spin_budget_ns) {
            set_error(A.st, (int32_t)CSS_ERR_TIMEOUT, kRotationWait);
            stop = true;
          }
        }
        stop = __any_sync(0xffffffffu, stop);   // the next barrier sees the status
      }
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float na = fmaf(v[i].x, xa[q], -(v[i].y * xb[q])), nb = fmaf(v[i].y, xa[q], v[i].x * xb[q]);
          const float da = __shfl_down_sync(0xffffffffu, na, 1);
          const float ub = __shfl_up_sync(0xffffffffu, lane == 0 ? na : nb, 1);
          xa[q] = lane == 31 ? nb : da;
          xb[q] = lane == 0 ? nb : ub;
        }
      }
    }
    // after 63 rounds the indices are those of round 0 again
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      __stcg(Qg + (warp * 4 + q) * kP + a, xa[q]);
      __stcg(Qg + (warp * 4 + q) * kP + b, xb[q]);
    }
  }
  asm volatile("bar.sync 1, %0;" ::"n"(kUp) : "memory");
  for (int e = threadIdx.x; e < kR * kB; e += kUp) log[e] = 0ull;
}

// Where the index of slot s (first or second of its pair) goes from one round
// to the next, as slot * 2 + second (see ab_of): a_j -> a_{j-1}, a_0 -> b_1,
// b_j -> b_{j+1}, b_31 -> a_31; b_0 stays.
__device__ __forceinline__ int moves_to(int s, int second) {
  if (!second) return s == 0 ? 3 : (s - 1) * 2;
  return s == 0 ? 1 : s == kB - 1 ? s * 2 : (s + 1) * 2 + 1;
}
// Place of the entry between two indices (slot * 2 + second) of different
// pairs: one plane per (second of the lower slot, second of the higher).
constexpr int kRow = kB + 1;            // one unused word a row
constexpr int kPlane = kB * kRow;
__device__ __forceinline__ int entry_at(int p, int q) {
  const int lo = min(p, q), hi = max(p, q);
  return ((lo & 1) * 2 + (hi & 1)) * kPlane + (hi >> 1) * kRow + (lo >> 1);
}
__device__ __forceinline__ int local_index(int slot, int second) {   // in round 0 (and 63)
  return !second ? slot : slot == 0 ? kR : kR - slot;
}

// One sweep of rotations over the 64 x 64 matrix of a block pair.  In round r,
// 496 threads apply its rotations to one off-diagonal 2 x 2 block each, from
// one copy of the entries to the other, while warp 16 forms round r + 1's:
// lane j forms the entry that its next pair (a_{j+1}, b_{j-1} of round r) will
// have from the four it comes from, and holds the diagonal in registers.  The
// entries are kept by slot, not by index, so that every address is the same in
// all rounds and a warp's accesses fall into different banks.  A round is one
// chain of shared-memory loads and an angle, and one barrier: 22 us a sweep
// with entries kept by index, now 15.
__device__ void sweep_pair(const EstArgs& A, const float* Ac, float* An, unsigned long long* log, int2 bp, float* smem,
                           float& off, float& top) {
  float* S = smem;   // two copies of the off-diagonal entries
  float2* cs = reinterpret_cast<float2*>(smem + 2 * 4 * kPlane);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, L = A.L;
  if (warp == 16) {
    const int ga = pair_at(bp, local_index(lane, 0)), gb = pair_at(bp, local_index(lane, 1));
    float da = __ldcg(Ac + (long long)ga * L + ga), db = __ldcg(Ac + (long long)gb * L + gb);
    float g = __ldcg(Ac + (long long)max(ga, gb) * L + min(ga, gb)), c, s;
    // the rotation of this lane's pair in round r, the diagonal after it, and
    // what is left of g
    auto turn = [&](int r) {
      off = fmaxf(off, fabsf(g));
      top = fmaxf(top, fmaxf(da, db));
      c = 1.f;
      s = 0.f;
      if (fabsf(g) > 1e-12f && g * g > 1e-16f * fabsf(da * db)) {
        // t = tan(theta): the smaller root of t^2 + 2 tau t - 1 = 0
        const float d = db - da, g2 = 2.f * g;
        const float t = copysignf(g2, __int_as_float(__float_as_int(d) ^ __float_as_int(g2))) *
                        rcp_approx(fabsf(d) + sqrt_approx(fmaf(d, d, g2 * g2)));
        const float x = fmaf(t, t, 1.f);
        c = rsqrt_approx(x);
        c = fmaf(0.5f * c, fmaf(-x * c, c, 1.f), c);
        s = t * c;
        da = fmaf(-t, g, da);
        db = fmaf(t, g, db);
        g = 0.f;
      }
      cs[(r & 1) * kB + lane] = make_float2(c, s);
      put_rotation(log + r * kB + lane, c, s);
    };
    // the slots that round r + 1's a_j and b_j come from: a_{j+1} (b_31 for the
    // last lane) and b_{j-1} (a_0 for lane 1, b_0 for lane 0)
    const int jx = min(lane + 1, kB - 1), jy = max(lane - 1, 0);
    const bool x_first = lane < kB - 1, y_first = lane == 1;
    const int blk = jx * kRow + jy, mine = entry_at(moves_to(lane, 0), moves_to(lane, 1));
    turn(0);
    __syncthreads();
    for (int r = 0; r < kR; ++r) {
      const float* Sc = S + (r & 1) * 4 * kPlane + blk;
      const float e0 = Sc[0], e1 = Sc[kPlane], e2 = Sc[2 * kPlane], e3 = Sc[3 * kPlane];
      S[(~r & 1) * 4 * kPlane + mine] = g;
      const float cx = __shfl_sync(0xffffffffu, c, jx), sx = __shfl_sync(0xffffffffu, s, jx);
      const float cy = __shfl_sync(0xffffffffu, c, jy), sy = __shfl_sync(0xffffffffu, s, jy);
      const float dd = __shfl_down_sync(0xffffffffu, da, 1);
      const float du = __shfl_up_sync(0xffffffffu, lane == 0 ? da : db, 1);
      const float ua = x_first ? cx : sx, ub = x_first ? -sx : cx;
      const float va = y_first ? cy : sy, vb = y_first ? -sy : cy;
      g = ua * fmaf(va, e0, vb * e2) + ub * fmaf(va, e1, vb * e3);
      da = lane == kB - 1 ? db : dd;
      db = lane == 0 ? db : du;
      if (r < kR - 1) turn(r + 1);
      __syncthreads();
    }
    // all indices are back in their slots of round 0
    __stcg(An + (long long)ga * L + ga, da);
    __stcg(An + (long long)gb * L + gb, db);
    __stcg(An + (long long)ga * L + gb, g);
    __stcg(An + (long long)gb * L + ga, g);
  } else {
    // this thread's off-diagonal block (jr < jc); the others repeat the last
    // one and put what they form into unused words
    const int e = min(tid, kB * (kB - 1) / 2 - 1);
    int jc = (int)((1.f + sqrtf(1.f + 8.f * e)) * 0.5f);
    while (jc * (jc - 1) / 2 > e) --jc;
    while ((jc + 1) * jc / 2 <= e) ++jc;
    const int jr = e - jc * (jc - 1) / 2, blk = jc * kRow + jr;
    const bool upd = e == tid;
    int to[4];
    int gr[2], gc[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      gr[q] = pair_at(bp, local_index(jr, q));
      gc[q] = pair_at(bp, local_index(jc, q));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int p1 = moves_to(jr, q >> 1), p2 = moves_to(jc, q & 1);
      // an entry that becomes its pair's own is warp 16's
      to[q] = !upd || (p1 >> 1) == (p2 >> 1) ? q * kPlane + jc * kRow + kB : entry_at(p1, p2);
      if (upd) {
        const int hi = max(gr[q >> 1], gc[q & 1]), lo = min(gr[q >> 1], gc[q & 1]);
        S[q * kPlane + blk] = __ldcg(Ac + (long long)hi * L + lo);
      }
    }
    __syncthreads();
    for (int r = 0; r < kR; ++r) {
      const float* Sc = S + (r & 1) * 4 * kPlane + blk;
      float* Sn = S + (~r & 1) * 4 * kPlane;
      const float b00 = Sc[0], b01 = Sc[kPlane], b10 = Sc[2 * kPlane], b11 = Sc[3 * kPlane];
      const float2 u = cs[(r & 1) * kB + jr], v = cs[(r & 1) * kB + jc];
      const float x00 = fmaf(u.x, b00, -(u.y * b10)), x10 = fmaf(u.y, b00, u.x * b10);
      const float x01 = fmaf(u.x, b01, -(u.y * b11)), x11 = fmaf(u.y, b01, u.x * b11);
      Sn[to[0]] = fmaf(v.x, x00, -(v.y * x01));
      Sn[to[1]] = fmaf(v.y, x00, v.x * x01);
      Sn[to[2]] = fmaf(v.x, x10, -(v.y * x11));
      Sn[to[3]] = fmaf(v.y, x10, v.x * x11);
      __syncthreads();
    }
    if (upd) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float v = S[(kR & 1) * 4 * kPlane + q * kPlane + blk];
        __stcg(An + (long long)gr[q >> 1] * L + gc[q & 1], v);
        __stcg(An + (long long)gc[q & 1] * L + gr[q >> 1], v);
      }
    }
  }
  __syncthreads();   // smem is used again
}

// out[r][4 g ..] = sum_k a[k * as + r * ar] b[k * bs + 4 g ..] over 64 k
__device__ __forceinline__ float4 dot64(const float* a, int as, const float* b, int bs) {
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 16
  for (int k = 0; k < kP; ++k) {
    const float av = a[k * as];
    const float4 bv = *reinterpret_cast<const float4*>(b + k * bs);
    o.x = fmaf(av, bv.x, o.x);
    o.y = fmaf(av, bv.y, o.y);
    o.z = fmaf(av, bv.z, o.z);
    o.w = fmaf(av, bv.w, o.w);
  }
  return o;
}

__global__ void __launch_bounds__(kNT, 1) estimate_kernel(EstArgs A) {
  extern __shared__ __align__(16) float smem[];
  __shared__ double s_red[32];
  __shared__ uint32_t s_epoch;
  const int tid = threadIdx.x, L = A.L, nb = L / kB, np = nb / 2, ncta = gridDim.x;
  if (tid == 0) s_epoch = 0u;
  // trace(G) = ||W||_F^2, the same sum in every CTA
  double tr = 0.0;
  for (int i = tid; i < A.l; i += kNT) tr += A.G[(long long)i * A.lp + i];
  tr = block_sum(tr, s_red);
  if (!isfinite(tr)) {
    if (blockIdx.x == 0 && tid == 0) set_error(A.st, (int32_t)CSS_ERR_NONFINITE, 0);
    return;
  }
  // (a trace whose inverse overflows: X stays the identity)
  const double inv_tr = tr > 0.0 && 1.0 / tr < 1e308 ? 1.0 / tr : 0.0;
  for (int e = blockIdx.x * kNT + tid; e < L * L; e += ncta * kNT) {
    const int r = e % L, c = e / L;
    __stcg(A.w.A0 + e, r < A.l && c < A.l ? (float)(A.G[(long long)c * A.lp + r] * inv_tr) : 0.f);
    __stcg(A.w.X32 + e, r == c ? 1.f : 0.f);
  }
  for (int e = blockIdx.x * kNT + tid; e < np * kR * kB; e += ncta * kNT) A.w.log[e] = 0ull;
  if (!team_barrier(A.w.bar, ncta, A.st, 43, &s_epoch)) return;
  const int ntile = np * (np - 1) / 2 * 4, nx = np * (L / 16);
  float *Ac = A.w.A0, *An = A.w.A1;
  for (int sweep = 0; sweep < kEstimateSweeps; ++sweep) {
    float off = 0.f, top = 0.f;
    for (int r = 0; r < nb - 1; ++r) {
      // (the launch has at least two CTAs a pair)
      if (blockIdx.x < np)
        sweep_pair(A, Ac, An, A.w.log + blockIdx.x * kR * kB, block_pair(r, blockIdx.x, nb), smem, off, top);
      else if (blockIdx.x < 2 * np && tid < kUp)
        build_q(A, A.w.log + (blockIdx.x - np) * kR * kB, A.w.Q + (long long)(blockIdx.x - np) * kP * kP);
      if (r == nb - 2 && blockIdx.x < np && tid >= kUp) {
        // non-negative floats order like their bits
        atomicMax(A.w.most + 2 * sweep, __float_as_uint(off));
        atomicMax(A.w.most + 2 * sweep + 1, __float_as_uint(top));
      }
      if (!team_barrier(A.w.bar, ncta, A.st, 44, &s_epoch)) return;
      // A <- J^T A J on the tiles between two pairs (i < j, 16 columns of
      // pair j an item, the mirror image written too), X <- X J (16 rows)
      for (int it = blockIdx.x; it < ntile + nx; it += ncta) {
        float *T = smem, *Qi = smem + kP * kP, *Qj = smem, *M = smem + 2 * kP * kP, *Qs = M + kP * 16;
        if (it < ntile) {
          int j = 1, i = it >> 2;
          while (i >= j) { i -= j; ++j; }
          const int2 bi = block_pair(r, i, nb), bj = block_pair(r, j, nb);
          const int s0 = (it & 3) * 16;
          for (int e = tid; e < kP * kP; e += kNT) {
            T[e] = __ldcg(Ac + (long long)pair_at(bj, e / kP) * L + pair_at(bi, e & (kP - 1)));
            Qi[e] = __ldcg(A.w.Q + (long long)i * kP * kP + e);
          }
          for (int e = tid; e < kP * 16; e += kNT)
            Qs[e] = __ldcg(A.w.Q + (long long)j * kP * kP + (e >> 4) * kP + s0 + (e & 15));
          __syncthreads();
          const int row = tid & (kP - 1), g = tid / kP;   // 256 threads: a row, 4 columns
          if (tid < 4 * kP) *reinterpret_cast<float4*>(M + row * 16 + 4 * g) = dot64(T + row, kP, Qs + 4 * g, 16);
          __syncthreads();
          if (tid < 4 * kP) {
            const float4 o = dot64(Qi + row, kP, M + 4 * g, 16);
            const int gr = pair_at(bi, row), gc = pair_at(bj, s0 + 4 * g);
            __stcg(An + (long long)gc * L + gr, o.x);
            __stcg(An + (long long)(gc + 1) * L + gr, o.y);
            __stcg(An + (long long)(gc + 2) * L + gr, o.z);
            __stcg(An + (long long)(gc + 3) * L + gr, o.w);
            __stcg(reinterpret_cast<float4*>(An + (long long)gr * L + gc), o);
          }
        } else {
          const int j = (it - ntile) % np, r0 = (it - ntile) / np * 16;
          const int2 bj = block_pair(r, j, nb);
          for (int e = tid; e < kP * kP; e += kNT) Qj[e] = __ldcg(A.w.Q + (long long)j * kP * kP + e);
          // Xs[k][row], 16 rows
          for (int e = tid; e < kP * 16; e += kNT)
            M[e] = __ldcg(A.w.X32 + (long long)pair_at(bj, e >> 4) * L + r0 + (e & 15));
          __syncthreads();
          if (tid < 256) {
            const int row = tid & 15, g = tid >> 4;
            const float4 o = dot64(M + row, 16, Qj + 4 * g, kP);
            float* x = A.w.X32 + (long long)pair_at(bj, 4 * g) * L + r0 + row;
            __stcg(x, o.x);
            __stcg(x + L, o.y);
            __stcg(x + 2 * L, o.z);
            __stcg(x + 3 * L, o.w);
          }
        }
        __syncthreads();
      }
      if (!team_barrier(A.w.bar, ncta, A.st, 45, &s_epoch)) return;
      float* t = Ac;
      Ac = An;
      An = t;
    }
    // The entries that this sweep annihilated were small: they are now at
    // FP32 rounding (convergence is quadratic), which is all that the
    // refinement wants.
    const float o = __uint_as_float(__ldcg(A.w.most + 2 * sweep)), d = __uint_as_float(__ldcg(A.w.most + 2 * sweep + 1));
    if (o <= kSmallPair * d) break;
  }
  for (int e = blockIdx.x * kNT + tid; e < A.l * A.l; e += ncta * kNT)
    A.w.X0[e] = (double)__ldcg(A.w.X32 + (long long)(e / A.l) * L + e % A.l);
}

// --------------------------------------------------------- FP64 products --
// out = op(A) B for l x l operands, 32 x 16 outputs a CTA (l = 256: 128 CTAs,
// 8192 multiply-adds a lane pair: bound by the FP64 rate, 34 us).
constexpr int kTM = 32, kTN = 16, kTK = 32;

// mode 0: A(i, k) = A[k lda + i];  1: A(i, k) = A[i lda + k], lower tiles, mirrored
template <int MODE>
__device__ __forceinline__ void product(const double* __restrict__ A, int lda, const double* __restrict__ B,
                                        const double* __restrict__ add, double f, bool minus_from_i, double* out,
                                        int ldo, int l, int ti, int tj) {
  __shared__ __align__(16) double sa[kTK][kTM + 1];
  __shared__ __align__(16) double sb[kTK][kTN + 2];
  const int r0 = ti * kTM, c0 = tj * kTN, tid = threadIdx.x;
  double ra[kTM * kTK / 128], rb[kTN * kTK / 128];
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < kTM * kTK / 128; ++q) {
      const int e = tid + q * 128;
      const int i = r0 + (MODE == 1 ? e / kTK : e % kTM), k = k0 + (MODE == 1 ? e % kTK : e / kTM);
      ra[q] = i < l && k < l ? __ldg(A + (MODE == 1 ? (long long)i * lda + k : (long long)k * lda + i)) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kTN * kTK / 128; ++q) {
      const int e = tid + q * 128, k = k0 + e % kTK, j = c0 + e / kTK;
      rb[q] = j < l && k < l ? __ldg(B + (long long)j * l + k) : 0.0;
    }
  };
  const int row = tid & 31, g = (tid >> 5) * 4;
  double o[4] = {0.0, 0.0, 0.0, 0.0};
  load(0);
  for (int k0 = 0; k0 < l; k0 += kTK) {
#pragma unroll
    for (int q = 0; q < kTM * kTK / 128; ++q) {
      const int e = tid + q * 128;
      if (MODE == 1) sa[e % kTK][e / kTK] = ra[q];
      else sa[e / kTM][e % kTM] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < kTN * kTK / 128; ++q) {
      const int e = tid + q * 128;
      sb[e % kTK][e / kTK] = rb[q];
    }
    __syncthreads();
    if (k0 + kTK < l) load(k0 + kTK);
#pragma unroll 8
    for (int k = 0; k < kTK; ++k) {
      const double av = sa[k][row];
      const double2 b0 = *reinterpret_cast<const double2*>(&sb[k][g]), b1 = *reinterpret_cast<const double2*>(&sb[k][g + 2]);
      o[0] = fma(av, b0.x, o[0]);
      o[1] = fma(av, b0.y, o[1]);
      o[2] = fma(av, b1.x, o[2]);
      o[3] = fma(av, b1.y, o[3]);
    }
    __syncthreads();
  }
  const int i = r0 + row;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int j = c0 + g + c;
    if (i >= l || j >= l || (MODE == 1 && j > i)) continue;
    double v = o[c];
    if (minus_from_i) v = (i == j ? 1.0 : 0.0) - v;
    if (add) v = fma(f, v, add[(long long)j * l + i]);
    out[(long long)j * ldo + i] = v;
    if (MODE == 1) out[(long long)i * ldo + j] = v;
  }
}

__global__ void __launch_bounds__(128) product_kernel(const double* A, int lda, const double* B, const double* add,
                                                      double f, double* out, int l) {
  product<0>(A, lda, B, add, f, false, out, l, l, blockIdx.x, blockIdx.y);
}
// R = I - X^T X and H = X^T Y (either may be null), symmetric: the tiles that
// touch the lower triangle, row tile I has 2 I + 2 of them.
__global__ void __launch_bounds__(128) inner_kernel(const double* X, const double* Y, double* R, double* H, int ldh,
                                                    int l) {
  const int both = R && H, t = both ? blockIdx.x >> 1 : blockIdx.x;
  int I = (int)((sqrtf(4.f * t + 1.f) - 1.f) * 0.5f);
  while (I * (I + 1) > t) --I;
  while ((I + 1) * (I + 2) <= t) ++I;
  const int J = t - I * (I + 1);
  if (J * kTN >= l) return;
  if (R && (!both || (blockIdx.x & 1))) product<1>(X, l, X, nullptr, 1.0, true, R, l, l, I, J);
  else product<1>(X, l, Y, nullptr, 1.0, false, H, ldh, l, I, J);
}

// E: e_ij = r_ij / 2 + k_ij, k_ij = (h_ij + (d_i + d_j) r_ij / 2) /
// (d_j - d_i) antisymmetric, where |k| < lim and the gap is above `floor` of
// the largest diagonal entry; else k = 0.  d_i = h_ii / (1 - r_ii).
__global__ void __launch_bounds__(256) correction_kernel(const double* __restrict__ H, int ldh,
                                                         const double* __restrict__ R, double* __restrict__ E, int l,
                                                         double lim, double floor) {
  __shared__ double s_top[8];
  double top = 0.0;
  for (int i = threadIdx.x; i < l; i += 256) top = fmax(top, fabs(H[(long long)i * ldh + i]));
  for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
  if ((threadIdx.x & 31) == 0) s_top[threadIdx.x >> 5] = top;
  __syncthreads();
  for (int q = 0; q < 8; ++q) top = fmax(top, s_top[q]);
  const int j = blockIdx.x;
  const double rj = R[(long long)j * l + j], dj = H[(long long)j * ldh + j] / (1.0 - rj);
  for (int i = threadIdx.x; i < l; i += 256) {
    const double r = R[(long long)j * l + i];
    double k = 0.0;
    if (i != j) {
      const double ri = R[(long long)i * l + i], di = H[(long long)i * ldh + i] / (1.0 - ri);
      const double num = fma(0.5 * (di + dj), r, H[(long long)j * ldh + i]), gap = dj - di;
      if (fabs(gap) > floor * top && fabs(num) < lim * fabs(gap)) k = num / gap;
    }
    E[(long long)j * l + i] = fma(0.5, r, k);
  }
}

}  // namespace

Estimate carve_estimate(WsCarver& c, int l) {
  Estimate w{};
  if (l < kEstimateMinL) return w;
  const size_t L = (size_t)(l + kP - 1) / kP * kP;
  w.bar = c.take<uint32_t>(kEstimateZeroed);
  w.most = w.bar ? w.bar + 32 : nullptr;
  w.A0 = c.take<float>(L * L);
  w.A1 = c.take<float>(L * L);
  w.X32 = c.take<float>(L * L);
  w.Q = c.take<float>(L * kP);
  w.log = c.take<unsigned long long>(L / kP * kR * kB);
  w.X0 = c.take<double>((size_t)l * l);
  w.X1 = c.take<double>((size_t)l * l);
  w.Y = c.take<double>((size_t)l * l);
  w.E = c.take<double>((size_t)l * l);
  return w;
}

cudaError_t estimate_eigvecs(const double* G, double* H, int l, int lp, const Estimate& w, DevStatus* st, int sms,
                             const double** X, cudaStream_t s) {
  EstArgs a{G, l, lp, (l + kP - 1) / kP * kP, w, st};
  cudaError_t e = cudaMemsetAsync(w.bar, 0, sizeof(uint32_t) * kEstimateZeroed, s);
  if (e != cudaSuccess) return e;
  const int np = a.L / kP;
  const int items = np * (np - 1) / 2 * 4 + np * (a.L / 16);
  void* args[] = {&a};
  e = cudaLaunchCooperativeKernel((const void*)estimate_kernel, dim3(std::min(sms, items)), dim3(kNT), args, kSmem, s);
  if (e != cudaSuccess) return e;
  const dim3 grid((l + kTM - 1) / kTM, (l + kTN - 1) / kTN);
  const int lower = grid.x * (grid.x + 1);
  double *x = w.X0, *xn = w.X1;
  auto step = [&](const double* E, double f) {   // X <- X + f X E
    product_kernel<<<grid, 128, 0, s>>>(x, l, E, x, f, xn, l);
    double* t = x;
    x = xn;
    xn = t;
  };
  // errors of a separated pair: FP32 rounding over the relative gap, then
  // squared step by step; the limits keep E's norm small
  const double lim[4] = {0.1, 0.03, 1e-3, 1e-6};
  for (int q = 0; q < 4; ++q) {
    product_kernel<<<grid, 128, 0, s>>>(G, lp, x, nullptr, 1.0, w.Y, l);
    inner_kernel<<<2 * lower, 128, 0, s>>>(x, w.Y, w.E, H, lp, l);
    correction_kernel<<<l, 256, 0, s>>>(H, lp, w.E, w.Y, l, lim[q], 2e-6);
    step(w.Y, 1.0);
  }
  for (int q = 0; q < 2; ++q) {
    inner_kernel<<<lower, 128, 0, s>>>(x, nullptr, w.E, nullptr, lp, l);
    step(w.E, 0.5);
  }
  product_kernel<<<grid, 128, 0, s>>>(G, lp, x, nullptr, 1.0, w.Y, l);
  inner_kernel<<<lower, 128, 0, s>>>(x, w.Y, nullptr, H, lp, l);
  *X = x;
  return cudaGetLastError();
}

}  // namespace css
