// Device helpers shared by the kernels that finish a sketched Gram-Schmidt
// reduction (the sketch kernel fuses the first pass; k_arnoldi.cu holds
// the others): block partial dot products with the stored sketched basis,
// the last-block combine, the Givens update of Eq. 11S and the scalar
// epilogue of each pass (Section 4.3; the Block GMRES algorithm's steps).
#pragma once

#include <type_traits>

#include "rtg_internal.cuh"

namespace rtg {

constexpr int GS_MAXW = 8;   // warps per block of the reducing kernels (256 threads)
constexpr int kRedCols = 2 * kMaxK + 4;   // columns of one reduction (see gs_ncols)
// Gram matrices of up to this many rows are staged in shared memory by the
// step finish (rows of gram_smem_ld(r) <= r + 2 doubles; it needs
// (kMaxK + 6) + r (r + 2) + GS_MAXW r + 4 doubles of scratch)
constexpr int kGramSmemRows = 56;
static_assert((kMaxK + 6) + kGramSmemRows * (kGramSmemRows + 2) + GS_MAXW * kGramSmemRows + 4 <=
                  GS_MAXW * kRedCols,
              "Gram staging must fit the reduction scratch");
// row stride of the staged n x n Gram matrix: even, so that 16-byte copies
// land on 16-byte boundaries
__device__ __forceinline__ int gram_smem_ld(int n) { return (n + 2) & ~1; }

template <typename A>
__device__ __forceinline__ A warp_sum(A v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Last-block ticket: an atomic increment (wrapping to zero after `last`)
// with acquire-release semantics at GPU scope.  The barrier before it makes
// the block's writes (its partial row) precede the release; the barrier
// after it orders the last block's reads after the acquire.  Cheaper than
// two full fences around a relaxed atomic.
__device__ __forceinline__ unsigned ticket_acq_rel(unsigned* counter, unsigned last) {
  unsigned old;
  asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;" : "=r"(old) : "l"(counter), "r"(last) : "memory");
  return old;
}

// Condition of the device-side loop.  A lock-step batch (o.group_left set)
// keeps looping while any of its problems runs: each problem's stop is
// counted once, and the count reaching zero ends the loop.
// (The count is kept on direct launches too: the host reads it per step.)
__device__ __forceinline__ void set_cond(const StepOpts& o, int keep_going, Ctl* ctl = nullptr) {
  const cudaGraphConditionalHandle h = static_cast<cudaGraphConditionalHandle>(o.cond);
  if (o.group_left == nullptr) {
    if (o.use_cond) cudaGraphSetConditional(h, keep_going ? 1u : 0u);
    return;
  }
  if (!keep_going && ctl != nullptr && atomicExch(&ctl->counted, 1) == 0 && atomicSub(o.group_left, 1u) == 1u &&
      o.use_cond)
    cudaGraphSetConditional(h, 0u);
}

// Double-float ("float-float") accumulation for FP32 data: the FP64 pipe
// of this GPU runs at 1/64 of the FP32 rate with a long dependent latency,
// so sums of products of FP32 values are kept as unevaluated pairs
// hi + lo of floats with error-free transformations (exact product by
// FMA, Knuth's two-sum), about 48 significant bits.  IEEE intrinsics keep
// the compiler from contracting or reassociating them.
struct FF {
  float hi, lo;
};
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ FF ff_add(FF x, FF y) {
  const FF s = ff_two_sum(x.hi, y.hi);
  const float e = __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo));
  return ff_two_sum(s.hi, e);
}
// Sum of two pairs inside a reduction: the two-sum of the high parts is
// exact and the low parts are added in FP32, without renormalising the
// result (the pair still stands for hi + lo; every reduction here ends in
// a conversion to double, which needs no normalised pair).  8 FP32
// operations instead of ff_add's 14.
__device__ __forceinline__ FF ff_add_lazy(FF x, FF y) {
  const FF s = ff_two_sum(x.hi, y.hi);
  return {s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo))};
}
__device__ __forceinline__ FF ff_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ FF ff_warp_sum(FF v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    FF w;
    w.hi = __shfl_xor_sync(0xffffffffu, v.hi, o);
    w.lo = __shfl_xor_sync(0xffffffffu, v.lo, o);
    v = ff_add_lazy(v, w);
  }
  return v;
}
__device__ __forceinline__ double ff_to_double(FF v) {
  return static_cast<double>(v.hi) + static_cast<double>(v.lo);
}

// Dot-product accumulator: float-float for FP32 data, FP64 for FP64 data.
template <typename T>
struct DotAcc;
template <>
struct DotAcc<float> {
  FF v{0.f, 0.f};
  __device__ __forceinline__ void add(float a, float b) { v = ff_add_lazy(v, ff_prod(a, b)); }
  __device__ __forceinline__ double warp_total() { return ff_to_double(ff_warp_sum(v)); }
};
template <>
struct DotAcc<double> {
  double v = 0.0;
  __device__ __forceinline__ void add(double a, double b) { v = fma(a, b, v); }
  __device__ __forceinline__ double warp_total() { return warp_sum(v); }
};

// Type of the combined partial sums: float-float for FP32 data, FP64 for
// FP64 data.
template <typename T>
struct Sum;
template <>
struct Sum<float> {
  using V = FF;
  static __device__ __forceinline__ V zero() { return {0.f, 0.f}; }
  static __device__ __forceinline__ V add(V a, V b) { return ff_add_lazy(a, b); }
  static __device__ __forceinline__ V ldcg(const V* p) {
    const float2 f = __ldcg(reinterpret_cast<const float2*>(p));
    return {f.x, f.y};
  }
};
template <>
struct Sum<double> {
  using V = double;
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V add(V a, V b) { return a + b; }
  static __device__ __forceinline__ V ldcg(const V* p) { return __ldcg(p); }
};

// __double2float_rn on the integer pipe for values in FP32's normal range
// (the conversion instruction takes about 1000 cycles on this GPU): the
// significand's upper 24 bits, rounded to nearest even, and the exponent
// moved; a carry out of the significand lands in the exponent.
__device__ __forceinline__ float double_to_float_rn(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const unsigned e = static_cast<unsigned>(b >> 52) & 0x7ffu;
  if (e < 1023u - 126u || e > 1023u + 126u) return b << 1 == 0ull ? __uint_as_float(static_cast<unsigned>(b >> 32)) : __double2float_rn(x);
  const unsigned long long m = (b & 0x7fffffffffffffffull) - (static_cast<unsigned long long>(1023 - 127) << 52);
  const unsigned long long r = (m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29;
  return __uint_as_float(static_cast<unsigned>(r) | (static_cast<unsigned>(b >> 32) & 0x80000000u));
}

// x as the FP32 value nearest to it and the FP32 value nearest to the rest, as
// the two conversions would give them, without the FP64 pipe's round trips:
// the rest of a 53-bit significand after its rounding to 24 bits is an
// integer of at most 29 bits.
__device__ __forceinline__ FF double_split_rn(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int e = static_cast<int>(b >> 52) & 0x7ff;
  if (e < 1023 - 60 || e > 1023 + 126) {
    const float hi = double_to_float_rn(x);
    return {hi, double_to_float_rn(x - static_cast<double>(hi))};
  }
  const float hi = double_to_float_rn(x);
  const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  const unsigned long long top = (m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29;   // as rounded (up to 2^24)
  const int rest = static_cast<int>(static_cast<long long>(m) - static_cast<long long>(top << 29));
  const float lo = static_cast<float>(rest) * __int_as_float((e - 1023 - 52 + 127) << 23);   // exact scaling
  return {hi, b >> 63 ? -lo : lo};
}

// A coefficient in the data's type.
template <typename T>
__device__ __forceinline__ T coef_as(double x) {
  if constexpr (sizeof(T) == 4) return double_to_float_rn(x);
  else return x;
}

// Columns of the per-block partial sums of one Gram-Schmidt reduction:
// [0, J] s . Q_i, [J+1] s . s, [J+2, 2J+2] Q_J . Q_i (the new row of the
// Gram matrix G = Q^T Q).  The start of a process (J = -1) has only s . s.
__device__ __forceinline__ int gs_ncols(int J) { return J < 0 ? 1 : 2 * J + 3; }

// Reduce-scatter of NV = 2, 4, ..., 32 float-float values across a warp: in
// log2(NV) halving rounds inside aligned groups of NV lanes each lane keeps one
// half of its values and hands the other half to its partner, adding what it
// receives; then butterfly sums across the groups; afterwards v[0] of lane l is
// the warp total of value l % NV.  NV = 32: 31 exchanges per lane instead of 32
// x 5 for separate warp sums, and the adds of a round are independent.  The tree
// is fixed, so the sums are deterministic.
template <int NV>
__device__ __forceinline__ void ff_reduce_scatter(FF (&v)[NV]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int half = NV / 2; half >= 1; half >>= 1) {
    const bool up = (lane & half) != 0;
#pragma unroll
    for (int k = 0; k < half; ++k) {
      const FF give = up ? v[k] : v[k + half];
      const FF keep = up ? v[k + half] : v[k];
      FF got;
      got.hi = __shfl_xor_sync(0xffffffffu, give.hi, half);
      got.lo = __shfl_xor_sync(0xffffffffu, give.lo, half);
      v[k] = ff_add_lazy(keep, got);
    }
  }
#pragma unroll
  for (int o = NV; o < 32; o <<= 1) {
    FF got;
    got.hi = __shfl_xor_sync(0xffffffffu, v[0].hi, o);
    got.lo = __shfl_xor_sync(0xffffffffu, v[0].lo, o);
    v[0] = ff_add_lazy(v[0], got);
  }
}

// One group of W columns i0 .. i0 + W - 1 (those <= J) of the FP32 partial
// sums: s . Q_i and Q_J . Q_i over this thread's ITEMS entries, reduced
// across the warp by one reduce-scatter of 2 W float-float values; lane
// l < 2 W writes column i0 + l % W of its warp's row (s . Q_i for l < W).
template <int W, int ITEMS>
__device__ __forceinline__ void ff_dot_group(const float* Q, int64_t d, const float (&sv)[ITEMS],
                                             const float (&qJ)[ITEMS], const int64_t* idx, int cnt, int i0, int J,
                                             FF (*rf)[kRedCols], int warp, int lane) {
  float qv[W][ITEMS];
#pragma unroll
  for (int g = 0; g < W; ++g)
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
      const bool ok = k < cnt && idx[k] >= 0 && i0 + g <= J;
      qv[g][k] = ok ? Q[static_cast<int64_t>(i0 + g) * d + idx[k]] : 0.f;
    }
  FF v[2 * W];
#pragma unroll
  for (int g = 0; g < W; ++g) {
    // the first product starts the pair (an exact product is already a
    // normalised pair, so adding it to zero would change nothing)
    FF p = ff_prod(sv[0], qv[g][0]), q = ff_prod(qJ[0], qv[g][0]);
#pragma unroll
    for (int k = 1; k < ITEMS; ++k) {
      p = ff_add_lazy(p, ff_prod(sv[k], qv[g][k]));
      q = ff_add_lazy(q, ff_prod(qJ[k], qv[g][k]));
    }
    v[g] = p;
    v[W + g] = q;
  }
  ff_reduce_scatter<2 * W>(v);
  if (lane < 2 * W) {
    const int g = lane % W;
    if (i0 + g <= J) rf[warp][lane < W ? i0 + g : J + 2 + i0 + g] = v[0];
  }
}

// Sum of the per-warp values of one column in a fixed order.
__device__ __forceinline__ double warps_total(const double (*red)[kRedCols], int nw, int i) {
  if (nw == 8)
    return ((red[0][i] + red[1][i]) + (red[2][i] + red[3][i])) +
           ((red[4][i] + red[5][i]) + (red[6][i] + red[7][i]));
  double acc = 0.0;
  for (int u = 0; u < nw; ++u) acc += red[u][i];
  return acc;
}

// Sum of the per-warp float-float values of one column in a fixed order.
__device__ __forceinline__ FF ff_warps_total(const FF (*red)[kRedCols], int nw, int i) {
  if (nw == 8)
    return ff_add_lazy(ff_add_lazy(ff_add_lazy(red[0][i], red[1][i]), ff_add_lazy(red[2][i], red[3][i])),
                       ff_add_lazy(ff_add_lazy(red[4][i], red[5][i]), ff_add_lazy(red[6][i], red[7][i])));
  FF acc{0.f, 0.f};
  for (int u = 0; u < nw; ++u) acc = ff_add_lazy(acc, red[u][i]);
  return acc;
}

// Per-block partial sums of the columns above: products of the stored
// values accumulated in double-float (FP32 data) or FP64 (FP64 data).
// Each thread passes up to ITEMS entries (vals at sketch indices idx);
// entries past cnt or with a negative index are ignored.  Writes this block's
// entry (linear block id) of every column of w.part, which is stored column
// by column (w.part_rows entries each, so that the combine reads a column's
// entries side by side): float-float pairs for FP32 data, doubles for FP64
// data.
// red: shared [GS_MAXW][kRedCols] doubles (float-float pairs for FP32).
// FP64 data: blocks with the same entries may share the columns, block y of
// gridDim.y taking the columns y, y + gridDim.y, ... (and s . s by block 0):
// the FP64 work of a column is some 2000 cycles of its SM.
template <typename T, int ITEMS>
__device__ void block_partials(const Work& w, const T* vals, const int64_t* idx, int cnt, int J,
                               double (*red)[kRedCols]) {
  const T* Q = static_cast<const T*>(w.Q);
  const int64_t d = w.d;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  const int ncols = gs_ncols(J);
  T sv[ITEMS], qJ[ITEMS];
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const bool ok = k < cnt && idx[k] >= 0;
    sv[k] = ok ? vals[k] : static_cast<T>(0);
    qJ[k] = (ok && J >= 0) ? Q[static_cast<int64_t>(J) * d + idx[k]] : static_cast<T>(0);
  }
  FF (*rf)[kRedCols] = reinterpret_cast<FF (*)[kRedCols]>(red);
  if (sizeof(T) == 4 || blockIdx.y == 0) {   // s . s
    DotAcc<T> a;
    if constexpr (sizeof(T) == 4) a.v = ff_prod(sv[0], sv[0]);
    else a.add(sv[0], sv[0]);
#pragma unroll
    for (int k = 1; k < ITEMS; ++k) {
      if (sizeof(T) == 8 && k >= cnt) break;   // (the entries past it are zero)
      a.add(sv[k], sv[k]);
    }
    if constexpr (sizeof(T) == 4) {
      const FF t = ff_warp_sum(a.v);
      if (lane == 0) rf[warp][J + 1] = t;
    } else {
      const double t = a.warp_total();
      if (lane == 0) red[warp][J + 1] = t;
    }
  }
  if constexpr (sizeof(T) == 4) {
    // 16 columns of Q at a time (the last group only as wide as it needs,
    // rounded up to a power of two): s . Q_i and Q_J . Q_i for each
    for (int i0 = 0; i0 <= J; i0 += 16) {
      const int nv = J + 1 - i0;
      if (nv > 8) ff_dot_group<16, ITEMS>(Q, d, sv, qJ, idx, cnt, i0, J, rf, warp, lane);
      else if (nv > 4) ff_dot_group<8, ITEMS>(Q, d, sv, qJ, idx, cnt, i0, J, rf, warp, lane);
      else if (nv > 2) ff_dot_group<4, ITEMS>(Q, d, sv, qJ, idx, cnt, i0, J, rf, warp, lane);
      else if (nv > 1) ff_dot_group<2, ITEMS>(Q, d, sv, qJ, idx, cnt, i0, J, rf, warp, lane);
      else ff_dot_group<1, ITEMS>(Q, d, sv, qJ, idx, cnt, i0, J, rf, warp, lane);
    }
  } else {
    // four columns of Q at a time: all their loads go out before any use
    constexpr int GRP = 4;
    const int step = gridDim.y;
    for (int i0 = blockIdx.y; i0 <= J; i0 += GRP * step) {
      T qv[GRP][ITEMS];
#pragma unroll
      for (int g = 0; g < GRP; ++g)
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
          const bool ok = k < cnt && idx[k] >= 0 && i0 + g * step <= J;
          qv[g][k] = ok ? Q[static_cast<int64_t>(i0 + g * step) * d + idx[k]] : static_cast<T>(0);
        }
#pragma unroll
      for (int g = 0; g < GRP; ++g) {
        const int i = i0 + g * step;
        if (i > J) break;
        double p = 0.0, q = 0.0;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
          if (k >= cnt) break;   // (the entries past it are zero)
          p = fma(sv[k], qv[g][k], p);
          q = fma(qJ[k], qv[g][k], q);
        }
        // both warp sums in one tree: the lower half-warp goes on with p, the upper with q
        const bool up = (lane & 16) != 0;
        double v = (up ? q : p) + __shfl_xor_sync(0xffffffffu, up ? p : q, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((lane & 15) == 0) red[warp][up ? J + 2 + i : i] = v;
      }
    }
  }
  __syncthreads();
  const int64_t row = sizeof(T) == 4 ? blockIdx.x + gridDim.x * blockIdx.y : blockIdx.x;
  for (int i = threadIdx.x; i < ncols; i += blockDim.x) {
    if constexpr (sizeof(T) == 8) {   // this block's columns
      const int c = i <= J ? i : i - (J + 2);
      if (c < 0 ? blockIdx.y != 0 : c % gridDim.y != blockIdx.y) continue;
    }
    const int64_t at = static_cast<int64_t>(i) * w.part_rows + row;
    if constexpr (sizeof(T) == 4) reinterpret_cast<FF*>(w.part)[at] = ff_warps_total(rf, nw, i);
    else w.part[at] = warps_total(red, nw, i);
  }
}

// One thread's share of a column: entries g, g + G, ... below n, U loads in
// flight per round, each round summed as a tree.
template <typename T, int U>
__device__ __forceinline__ typename Sum<T>::V column_share(const typename Sum<T>::V* p, unsigned g, unsigned G,
                                                           unsigned n) {
  using A = Sum<T>;
  typename A::V acc = A::zero();
  for (unsigned b = g; b < n; b += U * G) {
    typename A::V v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = b + u * G < n ? A::ldcg(p + b + u * G) : A::zero();
#pragma unroll
    for (int h = U / 2; h > 0; h >>= 1)
#pragma unroll
      for (int u = 0; u < h; ++u) v[u] = A::add(v[u], v[u + h]);
    acc = A::add(acc, v[0]);
  }
  return acc;
}

// Ticket: returns true in every thread of the last block to finish, after
// tot[0..ncols) holds the sum of all blocks' entries of each column (summed in
// float-float for T = float, in FP64 for double; 256 threads).  The order is
// fixed, so the result is deterministic.  FP32 data: a column is summed by G
// neighbouring lanes (a power of two), each taking every G-th entry with as
// many loads in flight as it has entries (up to 16), and a shuffle tree adds
// the lanes; the total is converted once.  FP64 data: G = 256 / columns groups (at most 32), each with
// every G-th entry, then one thread per column adds the groups' sums in a
// pairwise tree (scratch: >= blockDim doubles).  The counter wraps back to
// zero by itself.  pre (optional): called by every thread of the last block
// right after the ticket, before its loads, e.g. to start asynchronous copies
// that the caller needs after the combine.
template <typename T, typename Pre = void (*)()>
__device__ inline bool last_block_combine(const Work& w, int ncols, double* tot, int* am_last, double* scratch,
                                          Pre pre = nullptr) {
  using A = Sum<T>;
  using V = typename A::V;
  __syncthreads();
  const unsigned all = gridDim.x * gridDim.y;
  const unsigned nblk = sizeof(T) == 4 ? all : gridDim.x;   // entries of a column
  if (threadIdx.x == 0) *am_last = (ticket_acq_rel(w.counter, all - 1) == all - 1);
  __syncthreads();
  if (!*am_last) return false;
  if constexpr (!std::is_same<Pre, void (*)()>::value) pre();   // e.g. start the Gram staging copies
  const V* part = reinterpret_cast<const V*>(w.part);
  if constexpr (sizeof(T) == 4) {
    // lanes per column: 32 for up to 8 columns, 16 for up to 16, ..., 1 beyond 128
    int lg = 5;
    while (lg > 0 && (ncols << lg) > static_cast<int>(blockDim.x)) --lg;
    const unsigned G = 1u << lg, g = threadIdx.x & (G - 1u);
    const int per = static_cast<int>(blockDim.x) >> lg;            // columns per round
    for (int c0 = 0; c0 < ncols; c0 += per) {
      const int c = c0 + (static_cast<int>(threadIdx.x) >> lg);
      V acc = A::zero();
      if (c < ncols) {
        const V* p = part + static_cast<int64_t>(c) * w.part_rows;
        if (nblk <= 4 * G) acc = column_share<T, 4>(p, g, G, nblk);
        else if (nblk <= 8 * G) acc = column_share<T, 8>(p, g, G, nblk);
        else acc = column_share<T, 16>(p, g, G, nblk);
      }
      for (int o = static_cast<int>(G) >> 1; o > 0; o >>= 1) {
        V other;
        other.hi = __shfl_xor_sync(0xffffffffu, acc.hi, o);
        other.lo = __shfl_xor_sync(0xffffffffu, acc.lo, o);
        acc = A::add(acc, other);
      }
      if (g == 0 && c < ncols) tot[c] = ff_to_double(acc);
    }
    __syncthreads();
  } else {
    const int nt = blockDim.x, t = threadIdx.x;
    for (int c0 = 0; c0 < ncols; c0 += nt) {
      const int nc = (ncols - c0 < nt) ? ncols - c0 : nt;
      int G = nt / nc;
      if (G > 32) G = 32;
      const int c = t % nc, g = t / nc;
      if (g < G) {
        const V* p = part + static_cast<int64_t>(c0 + c) * w.part_rows;
        // (a tree over fewer loads leaves out only additions of zero)
        if (nblk <= static_cast<unsigned>(G)) scratch[g * nc + c] = column_share<T, 1>(p, g, G, nblk);
        else scratch[g * nc + c] = column_share<T, 16>(p, g, G, nblk);
      }
      __syncthreads();
      if (t < nc) {   // pairwise tree over the G group sums (levels that would add only zeros skipped)
        const int used = static_cast<int>(nblk) < G ? static_cast<int>(nblk) : G;
        if (used <= 4) {
          V v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = u < used ? scratch[u * nc + t] : A::zero();
          tot[c0 + t] = (v[0] + v[2]) + (v[1] + v[3]);
        } else {
          V v[32];
#pragma unroll
          for (int u = 0; u < 32; ++u) v[u] = u < G ? scratch[u * nc + t] : A::zero();
#pragma unroll
          for (int h = 16; h > 0; h >>= 1)
            if (h < G) {
#pragma unroll
              for (int u = 0; u < h; ++u) v[u] = A::add(v[u], v[u + h]);
            }
          tot[c0 + t] = v[0];
        }
      }
      __syncthreads();
    }
  }
  return true;
}

// 1 / d for the kernels that scale by it, once instead of in every thread.
__device__ __forceinline__ void set_inverse(Ctl* ctl, double d) {
  const double r = 1.0 / d;
  const float f = double_to_float_rn(r);
  ctl->inv = r;
  ctl->inv_hi = f;
  ctl->inv_lo = double_to_float_rn(r - static_cast<double>(f));
}

// Start of a process (one thread): beta = ||R_0||_Theta = sqrt(s . s).
__device__ inline void gs_finish_start(const Work& w, const StepOpts& o, const double* tot) {
  Ctl* ctl = w.ctl;
  const double tol = o.desc_tol ? *o.desc_tol : o.tol;
  const double beta = sqrt(tot[0]);
  if (ctl->status != 0) {
    ctl->stop = 1;
  } else if (!isfinite(beta)) {
    ctl->status = RTG_ERR_NONFINITE;
    ctl->stop = 1;
  } else if (beta == 0.0) {
    ctl->converged = 1;
    ctl->stop = 1;
  } else {
    ctl->beta = beta;
    set_inverse(ctl, beta);
    if (ctl->cycle == 0) ctl->beta0 = beta;
    w.g[0] = beta;
    ctl->rho = beta / ctl->beta0;
    if (ctl->rho <= tol) {   // (a warm start or a restart may already meet the stop level)
      ctl->converged = 1;
      ctl->stop = 1;
    }
    if (w.m == 0) ctl->stop = 1;
  }
  set_cond(o, !ctl->stop, ctl);
}

// Starts the asynchronous copies of the stored Gram matrix rows and columns
// 0..J-1 into the finish's shared staging area, so that they travel while
// the last block combines the partial sums; the finish waits for them.  Only
// where the finish stages G
// (J + 1 <= kGramSmemRows).  G is symmetric, so column k of G (contiguous
// in global memory) is copied to row k of the staging area, in 16-byte
// copies that bypass L1 (cp.async.cg): G's addresses are rewritten with
// other values by every cycle and every solve of the plan, and only L2 is
// coherent across the SMs that run successive finishes.  When J is odd the
// last pair of a column also brings G(J, k), which the finish overwrites
// with the new row.  sh: the finish's scratch, whose staging area starts
// after kMaxK + 6 doubles (past the combine's scratch, 16-byte aligned).
__device__ inline void gs_stage_gram_async(const Work& w, int J, double* sh) {
  const int n = J + 1;
  if (J < 1 || n > kGramSmemRows) return;
  const int lg = gram_smem_ld(n), ldg = gram_ld(w.m), pairs = (J + 1) / 2;
  double* Gs = sh + (kMaxK + 2) + 4;
  for (int e = threadIdx.x; e < J * pairs; e += blockDim.x) {
    const int p = e % pairs, k = e / pairs;
    const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(&Gs[k * lg + 2 * p]));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa),
                 "l"(w.G + static_cast<int64_t>(ldg) * k + 2 * p)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// Step finish from one reduction (every thread of the last block).
// Classical Gram-Schmidt with one re-orthogonalisation pass, written with
// the Gram matrix G = Q^T Q of the stored sketched basis so that a single
// pass over Q suffices: h1 = Q^T s, h2 = Q^T (s - Q h1) = h1 - G h1,
// h = h1 + h2 and h_{j+1,j}^2 = ||s - Q h||^2 = s.s - 2 h.h1 + h.(G h), all
// in FP64 (FP64 data; gs_finish_gram_f32 is FP32 data's).  Writes the
// Hessenberg column, h_{j+1,j} (0 on breakdown), the breakdown and non-finite
// flags, and advances j.  The Givens update of
// Eq. 11S, rho_j and the stop rule follow in givens_step, off this
// kernel's critical path.  Up to kGramSmemRows rows the Gram matrix is
// staged in shared memory and every warp takes part in the two products
// with it; beyond, one warp per row reads it from global memory.  sh:
// shared scratch of GS_MAXW * kRedCols doubles, 256 threads.
__device__ inline void gs_finish_gram(const Work& w, const StepOpts& o, int J, const double* tot, double* sh) {
  Ctl* ctl = w.ctl;
  const int ld = w.m + 1, ldg = gram_ld(w.m);
  const double bd_tol = o.desc_bd_tol ? *o.desc_bd_tol : o.bd_tol;   // loaded early, used at the end
  const double* h1 = tot;
  const double s2 = tot[J + 1];
  const double* grow = tot + J + 2;
  double* col = sh;                    // h
  double* red = col + (kMaxK + 2);     // a = h.h1, b = h.(G h)
  double* G = w.G;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int n = J + 1;
  if (n <= kGramSmemRows) {
    // G staged in shared memory (even row stride); each product G x runs
    // on every warp: warp w takes a slice of the columns, lane the rows
    // lane and lane + 32, and the warps' partial rows are summed in order
    const int lg = gram_smem_ld(n);
    double* Gs = red + 4;              // n x n
    double* pr = Gs + n * lg;          // [nw][n] partial products
    double* ab = pr + nw * n;          // [2][2] the two warps' sums of a and b
    // rows and columns < J arrived by gs_stage_gram_async; J from the new row
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      Gs[J * lg + i] = grow[i];
      Gs[i * lg + J] = grow[i];
    }
    for (int i = threadIdx.x; i <= J; i += blockDim.x) {   // new row/column, for later steps
      G[i + static_cast<int64_t>(ldg) * J] = grow[i];
      G[J + static_cast<int64_t>(ldg) * i] = grow[i];
    }
    __syncthreads();
    const int ks = (n + nw - 1) / nw;
    const int k0 = warp * ks, k1 = (k0 + ks < n) ? k0 + ks : n;
    auto gmul = [&](const double* x) {   // pr[w][i] = sum over the warp's columns of G(i, k) x_k
      for (int i = lane; i < n; i += 32) {
        double u = 0.0;
        for (int k = k0; k < k1; ++k) u = fma(Gs[i * lg + k], x[k], u);
        pr[warp * n + i] = u;
      }
    };
    gmul(h1);
    __syncthreads();
    // sums of the warps' partial rows as a fixed tree (FP64 adds have a
    // long dependent latency on this GPU)
    auto wsum = [&](int i) {
      if (nw == 8)
        return ((pr[i] + pr[n + i]) + (pr[2 * n + i] + pr[3 * n + i])) +
               ((pr[4 * n + i] + pr[5 * n + i]) + (pr[6 * n + i] + pr[7 * n + i]));
      double u = 0.0;
      for (int v = 0; v < nw; ++v) u += pr[v * n + i];
      return u;
    };
    for (int i = threadIdx.x; i < n; i += blockDim.x) col[i] = 2.0 * h1[i] - wsum(i);
    __syncthreads();
    pdl_trigger();
    gmul(col);
    __syncthreads();
    if (warp < 4) {   // a = h . h1 (warps 0, 1), b = h . (G h) (warps 2, 3) over the n <= 64 rows
      // the FP64 products are split exactly into float pairs and summed by a
      // float-float warp tree on the FP32 pipe (a tree of FP64 shuffles and
      // adds is several times slower on this GPU)
      const int i = threadIdx.x & 63, which = warp >> 1;
      double p = 0.0;
      if (i < n) p = which == 0 ? col[i] * h1[i] : col[i] * wsum(i);
      FF v = double_split_rn(p);
      v = ff_warp_sum(v);
      if (lane == 0) ab[warp] = ff_to_double(v);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      red[0] = ab[0] + ab[1];
      red[1] = ab[2] + ab[3];
    }
  } else {
    for (int i = threadIdx.x; i <= J; i += blockDim.x) {
      G[i + static_cast<int64_t>(ldg) * J] = grow[i];
      G[J + static_cast<int64_t>(ldg) * i] = grow[i];
    }
    __syncthreads();
    // h = 2 h1 - G h1: one warp per row, lanes across the columns
    for (int i = warp; i <= J; i += nw) {
      double gh = 0.0;
      for (int k = lane; k <= J; k += 32) gh += __ldcg(G + i + static_cast<int64_t>(ldg) * k) * h1[k];
      gh = warp_sum(gh);
      if (lane == 0) col[i] = 2.0 * h1[i] - gh;
    }
    __syncthreads();
    double* hgh_row = red + 4;         // (G h)_i * h_i per row
    for (int i = warp; i <= J; i += nw) {
      double gh = 0.0;
      for (int k = lane; k <= J; k += 32) gh += __ldcg(G + i + static_cast<int64_t>(ldg) * k) * col[k];
      gh = warp_sum(gh);
      if (lane == 0) hgh_row[i] = gh * col[i];
    }
    __syncthreads();
    if (warp == 0) {
      double a = 0.0, b = 0.0;
      for (int i = lane; i <= J; i += 32) {
        a += col[i] * h1[i];
        b += hgh_row[i];
      }
      a = warp_sum(a);
      b = warp_sum(b);
      if (lane == 0) {
        red[0] = a;
        red[1] = b;
      }
    }
  }
  __syncthreads();
  double* Hc = w.H + static_cast<int64_t>(ld) * J;
  int bad = 0;
  for (int i = threadIdx.x; i <= J; i += blockDim.x) {
    Hc[i] = col[i];
    bad |= !isfinite(col[i]);
  }
  for (int i = J + 2 + threadIdx.x; i < ld; i += blockDim.x) Hc[i] = 0.0;
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    const double hh1 = red[0], hgh = red[1];
    const bool finite = isfinite(s2) && isfinite(hh1) && isfinite(hgh) && !bad;
    const double hn2 = s2 - 2.0 * hh1 + hgh;
    const double hn2p = hn2 > 0.0 ? hn2 : 0.0;
    const double hn = sqrt(hn2p);
    // h_{j+1,j} <= bd_tol ||S(Phi V_j)||, compared in squares (one square root fewer)
    const bool breakdown = finite && (hn2p <= bd_tol * bd_tol * s2);
    Hc[J + 1] = breakdown ? 0.0 : hn;
    ctl->pre2 = s2;
    ctl->hnext = hn;
    ctl->inv = 1.0 / hn;
    ctl->j = J + 1;
    if (!finite) ctl->status = RTG_ERR_NONFINITE;
    if (breakdown) ctl->breakdown = 1;
    ctl->skip_update = (!finite || breakdown) ? 1 : 0;
    ctl->givens = 1;
  }
}

// The step finish of FP32 data: the same in FP64, from totals summed in
// float-float, with h_{j+1,j}^2 = s.s - h.(2 h1 - G h) in one sum.  The column
// also goes out as float-float pairs (48 bits) for the basis update, and
// 1 / h_{j+1,j} with it.  On this GPU an FP64 addition returns after 60 to 150
// cycles, so what follows the second product runs on several warps beside each
// other without a block barrier: warps 0 and 1 both form the sum, warp 0 the
// root and the flags, warp 1 the reciprocal, the others write the column.
// The same chain in float-float (2^-46 a product) was no faster: 1024 x 1024,
// 12 steps, 861 us in pairs and 846 so; 512 x 512 268 and 267; queue of 48
// 2932 and 2885; video 2488 and 2467.
__device__ inline void gs_finish_gram_f32(const Work& w, const StepOpts& o, int J, const double* tot, double* sh) {
  Ctl* ctl = w.ctl;
  const int ld = w.m + 1, ldg = gram_ld(w.m);
  const double bd_tol = o.desc_bd_tol ? *o.desc_bd_tol : o.bd_tol;   // loaded early, used at the end
  const double* h1 = tot;
  const double s2 = tot[J + 1];
  const double* grow = tot + J + 2;
  double* col = sh;                     // h
  double* G = w.G;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int n = J + 1;
  const bool small = n <= kGramSmemRows;
  const int lg = gram_smem_ld(n);
  double* Gs = col + (kMaxK + 2) + 4;   // n x n, symmetric (gs_stage_gram_async)
  double* pr = Gs + n * lg;             // [nw][n] partial products
  double* row = Gs;                     // beyond kGramSmemRows: h_i (2 h1 - G h)_i per row
  auto psum = [&](int i) {   // the warps' partial rows as a fixed tree
    if (nw == 8)
      return ((pr[i] + pr[n + i]) + (pr[2 * n + i] + pr[3 * n + i])) +
             ((pr[4 * n + i] + pr[5 * n + i]) + (pr[6 * n + i] + pr[7 * n + i]));
    double u = 0.0;
    for (int v = 0; v < nw; ++v) u += pr[v * n + i];
    return u;
  };
  if (small) {
    // G staged in shared memory (even row stride); each product G x runs
    // on every warp: warp w takes a slice of the columns, lane the rows
    // lane and lane + 32, and the warps' partial rows are summed in order
    // rows and columns < J arrived by gs_stage_gram_async; J from the new row
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      Gs[J * lg + i] = grow[i];
      Gs[i * lg + J] = grow[i];
    }
    for (int i = threadIdx.x; i <= J; i += blockDim.x) {   // new row/column, for later steps
      G[i + static_cast<int64_t>(ldg) * J] = grow[i];
      G[J + static_cast<int64_t>(ldg) * i] = grow[i];
    }
    __syncthreads();
    const int ks = (n + nw - 1) / nw;
    const int k0 = warp * ks, k1 = (k0 + ks < n) ? k0 + ks : n;
    auto gmul = [&](const double* x) {   // pr[w][i] = sum over the warp's columns of G(k, i) x_k
      for (int i = lane; i < n; i += 32) {
        double u = 0.0;
        for (int k = k0; k < k1; ++k) u = fma(Gs[k * lg + i], x[k], u);
        pr[warp * n + i] = u;
      }
    };
    gmul(h1);
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) col[i] = 2.0 * h1[i] - psum(i);
    __syncthreads();
    pdl_trigger();
    gmul(col);
  } else {
    for (int i = threadIdx.x; i <= J; i += blockDim.x) {
      G[i + static_cast<int64_t>(ldg) * J] = grow[i];
      G[J + static_cast<int64_t>(ldg) * i] = grow[i];
    }
    __syncthreads();
    // h = 2 h1 - G h1: one warp per row, lanes across the columns
    for (int i = warp; i <= J; i += nw) {
      double gh = 0.0;
      for (int k = lane; k <= J; k += 32) gh = fma(__ldcg(G + i + static_cast<int64_t>(ldg) * k), h1[k], gh);
      gh = warp_sum(gh);
      if (lane == 0) col[i] = 2.0 * h1[i] - gh;
    }
    __syncthreads();
    for (int i = warp; i <= J; i += nw) {
      double gh = 0.0;
      for (int k = lane; k <= J; k += 32) gh = fma(__ldcg(G + i + static_cast<int64_t>(ldg) * k), col[k], gh);
      gh = warp_sum(gh);
      if (lane == 0) row[i] = col[i] * (2.0 * h1[i] - gh);
    }
  }
  __syncthreads();
  double* Hc = w.H + static_cast<int64_t>(ld) * J;
  if (warp > 1) {   // the column for the later kernels, beside the scalars
    for (int i = static_cast<int>(threadIdx.x) - 64; i <= J; i += blockDim.x - 64) {
      const FF h = double_split_rn(col[i]);
      Hc[i] = col[i];
      reinterpret_cast<float2*>(w.hf)[i] = make_float2(h.hi, h.lo);
    }
    for (int i = J + 2 + static_cast<int>(threadIdx.x) - 64; i < ld; i += blockDim.x - 64) Hc[i] = 0.0;
    return;
  }
  double t = 0.0;
  bool bad = false;
  for (int i = lane; i <= J; i += 32) {
    t = small ? fma(col[i], 2.0 * h1[i] - psum(i), t) : t + row[i];
    bad |= !isfinite(col[i]);
  }
  t = warp_sum(t);
  bad = __any_sync(0xffffffffu, bad);
  if (lane != 0) return;
  const double hn2 = s2 - t;
  const double hn2p = hn2 > 0.0 ? hn2 : 0.0;
  if (warp == 1) {   // (a breakdown's value is not used)
    const double r = rsqrt(hn2p);
    const FF f = double_split_rn(r);
    ctl->inv = r;
    ctl->inv_hi = f.hi;
    ctl->inv_lo = f.lo;
    return;
  }
  const bool finite = isfinite(s2) && isfinite(t) && !bad;
  const double hn = sqrt(hn2p);
  // h_{j+1,j} <= bd_tol ||S(Phi V_j)||, compared in squares (one square root fewer)
  const bool breakdown = finite && (hn2p <= bd_tol * bd_tol * s2);
  Hc[J + 1] = breakdown ? 0.0 : hn;
  ctl->pre2 = s2;
  ctl->hnext = hn;
  ctl->j = J + 1;
  if (!finite) ctl->status = RTG_ERR_NONFINITE;
  if (breakdown) ctl->breakdown = 1;
  ctl->skip_update = (!finite || breakdown) ? 1 : 0;
  ctl->givens = 1;
}

// Givens update of Eq. 11S for the Hessenberg column the last finish wrote
// (column J = j - 1), rho_j = |g_{J+1}| / beta_0, the stop rule and the
// condition of the device-side loop, which never runs more than m + 1
// bodies.  Called by every thread of one block, which runs beside the basis
// update (it does not depend on it): the block loads the column and the
// stored rotations in one round and forms their products, then one thread
// runs the dependent chain, one FP64 multiply-add per rotation.
__device__ inline void givens_step(const Work& w, const StepOpts& o) {
  // c_i y_{i+1}, s_i y_{i+1}, s_i, c_i of the stored rotations on the new
  // column, and the chain's values x_i
  __shared__ double gv_cy[kMaxK], gv_sy[kMaxK], gv_s[kMaxK], gv_c[kMaxK], gv_x[kMaxK], gv_last[2], gv_rot[2];
  __shared__ int gv_J, gv_do;
  Ctl* ctl = w.ctl;
  if (threadIdx.x == 0) {
    gv_do = ctl->givens;
    gv_J = ctl->j - 1;
  }
  __syncthreads();
  const int ld = w.m + 1;
  if (gv_do) {
    const int J = gv_J;
    const double* Hc = w.H + static_cast<int64_t>(ld) * J;
    for (int i = threadIdx.x; i < J; i += blockDim.x) {
      const double y = Hc[i + 1], c = w.cs[i], sv = w.sn[i];
      gv_c[i] = c;
      gv_s[i] = sv;
      gv_cy[i] = c * y;
      gv_sy[i] = sv * y;
    }
    if (threadIdx.x == blockDim.x - 1) gv_last[0] = Hc[0];
    if (threadIdx.x == blockDim.x - 2) gv_last[1] = Hc[J + 1];
    __syncthreads();
    // rotations 0..J-1 on the new column: one dependent multiply-add each
    // (the products with y do not depend on the chain)
    if (threadIdx.x == 0) {
      double x = gv_last[0];
      for (int i = 0; i < J; ++i) {
        gv_x[i] = x;
        x = fma(-gv_s[i], x, gv_cy[i]);
      }
      gv_last[0] = x;
    }
    __syncthreads();
    double* Rc = w.R + static_cast<int64_t>(ld) * J;
    if (threadIdx.x >= 32)
      for (int i = static_cast<int>(threadIdx.x) - 32; i < J; i += blockDim.x - 32) Rc[i] = fma(gv_c[i], gv_x[i], gv_sy[i]);
    // the new rotation: its two quotients in two lanes at once
    if (threadIdx.x < 2) {
      const double x = gv_last[0], y = gv_last[1];
      const double q = fma(x, x, y * y);
      // (hypot where the squares leave the normal range)
      const double den = (q > 1e-280 && q < 1e280) ? sqrt(q) : hypot(x, y);
      double v = threadIdx.x == 0 ? 1.0 : 0.0;
      if (den != 0.0) v = (threadIdx.x == 0 ? x : y) / den;
      gv_rot[threadIdx.x] = v;
      if (threadIdx.x == 0) Rc[J] = den;
    }
  }
  __syncwarp();
  if (threadIdx.x != 0) return;
  if (gv_do) {
    ctl->givens = 0;
    const int J = gv_J;
    const double tol = o.desc_tol ? *o.desc_tol : o.tol;
    double* Rc = w.R + static_cast<int64_t>(ld) * J;
    const double c = gv_rot[0], sv = gv_rot[1];
    Rc[J + 1] = 0.0;
    w.cs[J] = c;
    w.sn[J] = sv;
    const double gJ = w.g[J];
    w.g[J + 1] = -sv * gJ;
    w.g[J] = c * gJ;
    const double rho = fabs(sv * gJ) / ctl->beta0;
    ctl->rho = rho;
    w.rho_hist[ctl->iters_total] = rho;
    ctl->iters_total += 1;
    const bool finite = ctl->status != RTG_ERR_NONFINITE && isfinite(rho);
    if (!finite && ctl->status == 0) ctl->status = RTG_ERR_NONFINITE;
    const bool breakdown = ctl->breakdown != 0;
    const bool conv = finite && rho <= tol;
    if (conv || breakdown) ctl->converged = 1;
    // a nonzero status (a bounded wait that gave up upstream) ends the solve
    if (!finite || breakdown || conv || ctl->status != 0) {
      ctl->stop = 1;
    } else if (J + 1 >= w.m) {
      // end of a cycle: restart from the least-squares iterate while cycles
      // remain (the body's restart kernels run when rs_skip is 0), else stop
      if (ctl->cycle + 1 < w.cycles) {
        ctl->rs_skip = 0;
        if (o.use_rs_cond) cudaGraphSetConditional(static_cast<cudaGraphConditionalHandle>(o.rs_cond), 1u);
      } else {
        ctl->stop = 1;
      }
    }
  }
  // the body runs at most m times per cycle
  const int loops = ++ctl->loops;
  const int cap = w.m * w.cycles;
  if (loops > cap) {
    ctl->stop = 1;
    ctl->rs_skip = 1;
    if (o.use_cond && loops > cap + 1 && ctl->status == 0) ctl->status = RTG_ERR_TIMEOUT;
  }
  set_cond(o, !ctl->stop, ctl);
}

// new_cycle = 0: start of a solve; 1: start of a restarted cycle (gated by
// rs_skip inside the step body: it keeps the body count, the lock-step
// count of running problems and the restart flag, which the restart
// sequence clears last).
__device__ inline void reset_ctl(const Work& w0, int new_cycle, unsigned* group_left, const int* gate) {
  const BIdx bi = bidx(w0.b);
  Ctl* ctl = bsh(w0.ctl, bi.off);
  gate = bsh(gate, bi.off);
  if (gate != nullptr && *gate) return;
  unsigned* counter = bsh(w0.counter, bi.off);
  // last-block counters wrap to zero by themselves; clearing them here also
  // recovers from a solve that ended inside a kernel
  for (int i = 0; i < 8; ++i) counter[i] = 0u;
  ctl->j = 0;
  ctl->stop = 0;
  ctl->breakdown = 0;
  ctl->converged = 0;
  ctl->skip_update = 0;
  ctl->pre2 = 0.0;
  ctl->hnext = 0.0;
  ctl->givens = 0;
  if (new_cycle) {
    ctl->cycle += 1;
  } else {
    if (group_left != nullptr && bi.p == 0) *group_left = static_cast<unsigned>(w0.b.n);
    ctl->counted = 0;
    ctl->loops = 0;
    ctl->rs_skip = 1;
    ctl->status = 0;
    ctl->iters_total = 0;
    ctl->cycle = 0;
    ctl->beta0 = 0.0;
    ctl->beta = 0.0;
    ctl->rho = 1.0;
    ctl->mu = 0.0;
    ctl->true_rr = -1.0;
    ctl->true_th = -1.0;
  }
}

}  // namespace rtg
