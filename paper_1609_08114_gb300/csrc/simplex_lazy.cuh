// simplex_lazy.cuh -- the simplex method on a tableau that is never written: one
// to eight warps per LP, for LPs whose slack basis is feasible.
//
// Section 3.1 Steps 1-3 need, per pivot, one column of the tableau (Step 2), one
// row of it (the pivot row), the right-hand side and the objective row.  The
// full update writes all m n entries after every pivot to have them; this kernel
// keeps the pivots instead.  With f_s the multiplier column t_ie / p and p_s the
// pivot row of pivot s, entry (i, j) after k pivots is the chain
//
//     x <- fma(-f_s[i], p_s[j], x),   s = 1..k,
//
// that a full update would have run on it, starting again wherever row i was the
// pivot row (x = p_s[j] / p) or column j the pivot column (x = -f_s[i]).  A
// pivot needs the chain for m + n entries: k (m + n) multiply-adds instead of
// m n, in the same order, so every value -- and with it every pivot choice --
// is the one the full update gives.
//
//   * Thread t owns rows and columns t, t + NT, ... (R of each, NT threads):
//     the right-hand side, the objective row, the basic and non-basic variables
//     and the last pivot on each of its rows and columns stay in registers.
//   * History entry s holds f_s (m values) and p_s (n values), with f_s[l] =
//     -1/p and p_s[e] = 1, so that one multiply-add from -0 restarts a chain.
//     The first `ks` entries live in shared memory, the rest (few LPs take that
//     many pivots) in a slot of the workspace.
//   * An LP of more than `kmax` pivots (the planner's rule, by size) has a tableau after
//     all: the history is applied to A in one pass, into the slot, and later to
//     that tableau, whenever `ks` more pivots are kept.  The chains then start from the
//     slot's entries.  The order of operations on an entry is the same, so are the
//     values.  (20,000 x 100 x 100 with normal rows, 126 pivots: FP64 134 ms when such
//     LPs started again in the tableau kernel, 72 now, 101 with a full update per pivot;
//     plain FP32 28.9, 9.4 and 8.6.)
//   * A is read where it lies: one pass over it checks that it is finite (and
//     leaves it in L2), then a pivot reads the one row and column it needs.
//   * Refinement and certificate (FP32 + refinement): FP64 residuals from A; the
//     correction B^-1 r by running the pivots on r as another right-hand side,
//     its transpose as another objective row (k (m + n) operations), or by products
//     with the slot's tableau where there is one; the KKT certificate of the other
//     kernels.
//   * Objectives of one polytope (lpb_solve_shared): a CTA takes consecutive ones
//     and starts each from the basis of the one before, whose history, right-hand
//     side and variables it keeps, under either rule and with or without refinement:
//     the new objective row is -c run through the pivots (k n operations).  Where a
//     direction takes more than `kmax` pivots, the launch ends, and the register kernel,
//     whose warm starts cost the same from any basis, solves the objectives left (10,000
//     directions that turn slowly, 60 x 50 with normal rows, 60 pivots to the first
//     optimum: 0.71 ms on that kernel, 0.82 here, 1.2 through a tableau in the slot).
//
// What bounds it, at 50,000 x 100 with FP64 input (4.19 ms on the kernel that updates
// the whole tableau -> 2.03 ms, 0.30 of the copy bandwidth over the 83.6 KB that an LP
// must move): the serial steps of a pivot -- two arg-mins with a barrier each, the column
// and the row from where A lies, their chains -- some 5,000 cycles of which 16 warps per
// SM hide the most part (scheduler slots 41% used).  Not A's traffic alone: 50,000 directions
// of one polytope, whose A stays in L2 and is read through once, take 1.85 ms.  But L2 lets
// go of a part of A by the time a pivot gathers from it (113 KB of DRAM traffic per LP),
// which is why an LP has two warps and eight LPs an SM, and nothing is fetched ahead: one
// warp per LP and nine LPs, or fetching the next LP, read A up to three times from DRAM
// (3.4 ms).  A one-time FP32 copy of A in shared memory takes away the LPs in flight (2.45
// ms at best).  FP64 tableau, 20,000 x 100 (12.4 -> 1.37 ms): the FP64 pipe, 69% busy.
#pragma once
#include <type_traits>

#include "lpb_internal.cuh"

namespace lpb {

namespace {

// Objectives of one polytope: consecutive ones claimed at a time, and warm starts
// between two cold ones.
constexpr int kShareChunk = 16;
constexpr int kWarmMax = 32;
// Rows and (FP32) columns that a thread takes at a time when pivots are applied (the
// history's pivot rows start at a multiple of the rows).
constexpr int kApplyRows = 8;
constexpr int kApplyCols = 2;
// Residuals, in parts of the certificate's bar, at which refinement stops (the tableau
// kernel's arithmetic): a quarter of that kernel's, which asks for it in the rows of
// basic slacks too.  (Error in x against FP64, 99% quantile over 10,000 bounded LPs of
// 100 x 100: tableau kernel 2.2e-11; here 2.5e-11 with its 1e-3, 1.2e-11 with this.)
constexpr double kStop = 0.25e-3;
enum : int { kCommon = 0, kShared = 1, kRandom = 2, kPacked = 4 };

__device__ __forceinline__ float neg(float v) { return -v; }
__device__ __forceinline__ double neg(double v) { return neg_bits(v); }
__device__ __forceinline__ float mul_add(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mul_add(double a, double b, double c) { return fma(a, b, c); }
template <typename T> __device__ __forceinline__ T neg_zero();
template <> __device__ __forceinline__ float neg_zero<float>() { return __uint_as_float(0x80000000u); }
template <> __device__ __forceinline__ double neg_zero<double>() { return __hiloint2double(int(0x80000000u), 0); }

// v > eps (eps > 0) for the tableau's type; FP64 on the bits (NaN is not
// greater), which spends no FP64 instruction.
__device__ __forceinline__ bool above(float v, float eps) { return v > eps; }
__device__ __forceinline__ bool above(double v, double eps) {
  const long long b = __double_as_longlong(v);
  return b > __double_as_longlong(eps) && b <= 0x7ff0000000000000ll;
}

// Order-preserving image of a value in the unsigned integers (FP64: -0 as +0),
// and its least value over the warp.
__device__ __forceinline__ unsigned image(float v) { return f2ord(v); }
__device__ __forceinline__ unsigned long long image(double v) {
  const long long b = __double_as_longlong(v);
  return d2ord(b == static_cast<long long>(0x8000000000000000ull) ? 0.0 : v);
}
__device__ __forceinline__ float unimage(unsigned o) { return ord2f(o); }
__device__ __forceinline__ double unimage(unsigned long long o) {
  return __longlong_as_double(static_cast<long long>((o >> 63) ? (o & 0x7fffffffffffffffull) : ~o));
}
__device__ __forceinline__ unsigned warp_min(unsigned o) { return __reduce_min_sync(kFull, o); }
__device__ __forceinline__ unsigned long long warp_min(unsigned long long o) {
  const unsigned hi = __reduce_min_sync(kFull, unsigned(o >> 32));
  const unsigned lo = __reduce_min_sync(kFull, unsigned(o >> 32) == hi ? unsigned(o) : 0xffffffffu);
  return (static_cast<unsigned long long>(hi) << 32) | lo;
}
template <typename T> using Img = std::conditional_t<sizeof(T) == 8, unsigned long long, unsigned>;

// Entry of the input in FP64 (an FP32 one by integer operations: the hardware
// conversion runs on the slow FP64 unit).
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) { return f2d_exact(v); }
// The same for a zero or normal entry of A in the FP64 products, without
// branches; `low`: the least magnitude image minus one, by which the caller
// finds the subnormal ones.
__device__ __forceinline__ double widen_a(double v, unsigned &) { return v; }
__device__ __forceinline__ double widen_a(float v, unsigned &low) {
  const unsigned u = __float_as_uint(v), mag = u & 0x7fffffffu;
  low = min(low, mag - 1u);
  return __hiloint2double(int((u & 0x80000000u) | (mag == 0u ? 0u : (mag >> 3) + (896u << 20))), int(u << 29));
}

// Entry `i` of the LP's A as the tableau's type: RN = false truncates FP64 to
// FP32 (as the register kernel does), RN = true rounds (as the tableau kernel does).
template <typename T, bool F64, bool RN>
__device__ __forceinline__ T a_in(const void *A, int i) {
  if constexpr (!F64) {
    return T(__ldg(static_cast<const float *>(A) + i));
  } else {
    const double d = __ldg(static_cast<const double *>(A) + i);
    if constexpr (sizeof(T) == 8) return d;
    else if constexpr (RN) return d2f_rn(d);
    else {
      unsigned amax = 0u;
      return d2f_trunc(d, amax);
    }
  }
}

// Largest magnitude image (FP64: the high word, FP32: the word) of the LP's
// `cnt` entries of A, by 16-byte loads, kU in flight per thread.
template <bool F64, int NT>
__device__ __forceinline__ unsigned scan_a(const void *A, int cnt, int tid) {
  constexpr int ES = F64 ? 8 : 4, PER = 16 / ES, kU = 8;
  const unsigned char *p = static_cast<const unsigned char *>(A);
  int head = int((16 - (reinterpret_cast<uintptr_t>(p) & 15)) & 15) / ES;
  head = head < cnt ? head : cnt;
  unsigned amax = 0u;
  auto one = [&](int i) {
    const unsigned u = F64 ? __ldg(reinterpret_cast<const uint2 *>(p) + i).y : __ldg(reinterpret_cast<const unsigned *>(p) + i);
    amax = max(amax, u & 0x7fffffffu);
  };
  const int nv = (cnt - head) / PER;
  const uint4 *v4 = reinterpret_cast<const uint4 *>(p + size_t(head) * ES);
  auto fold = [&](const uint4 &v) {
    if (!F64) amax = max(amax, max(v.x & 0x7fffffffu, v.z & 0x7fffffffu));
    amax = max(amax, max(v.y & 0x7fffffffu, v.w & 0x7fffffffu));
  };
  int k = tid;
#pragma unroll 1
  for (; k - tid < nv; k += kU * NT) {         // past the end the last vector again
    uint4 v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = __ldg(v4 + min(k + u * NT, nv - 1));
#pragma unroll
    for (int u = 0; u < kU; ++u) fold(v[u]);
  }
  if (tid < head) one(tid);
  const int done = head + nv * PER;
  if (done + tid < cnt) one(done + tid);      // fewer than PER entries are left
  return amax;
}

// kApplyRows values of one column and the multiply-add of a pivot on them, x <- x - f p.
// FP32 in pairs: one fma.rn.f32x2 rounds its halves as two fmaf do.
template <typename T> struct Rows;
template <>
struct Rows<float> {
  unsigned long long v[kApplyRows / 2];
  static __device__ __forceinline__ unsigned long long pair(float a, float b) {
    return (static_cast<unsigned long long>(__float_as_uint(b)) << 32) | __float_as_uint(a);
  }
  __device__ __forceinline__ void load(const float *p) {           // at a 16-byte boundary
#pragma unroll
    for (int u = 0; u < kApplyRows / 4; ++u) {
      const ulonglong2 a = reinterpret_cast<const ulonglong2 *>(p)[u];
      v[2 * u] = a.x;
      v[2 * u + 1] = a.y;
    }
  }
  __device__ __forceinline__ float get(int u) const { return __uint_as_float(unsigned(u & 1 ? v[u / 2] >> 32 : v[u / 2])); }
  __device__ __forceinline__ void set(int u, float x) {
    v[u / 2] = u & 1 ? pair(__uint_as_float(unsigned(v[u / 2])), x) : pair(x, __uint_as_float(unsigned(v[u / 2] >> 32)));
  }
  __device__ __forceinline__ void sub(const Rows &f, float p) {
    const unsigned long long q = pair(-p, -p);
#pragma unroll
    for (int u = 0; u < kApplyRows / 2; ++u) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v[u]) : "l"(f.v[u]), "l"(q));
  }
};
template <>
struct Rows<double> {
  double v[kApplyRows];
  __device__ __forceinline__ void load(const double *p) {
#pragma unroll
    for (int u = 0; u < kApplyRows / 2; ++u) {
      const double2 a = reinterpret_cast<const double2 *>(p)[u];
      v[2 * u] = a.x;
      v[2 * u + 1] = a.y;
    }
  }
  __device__ __forceinline__ double get(int u) const { return v[u]; }
  __device__ __forceinline__ void set(int u, double x) { v[u] = x; }
  __device__ __forceinline__ void sub(const Rows &f, double p) {
#pragma unroll
    for (int u = 0; u < kApplyRows; ++u) v[u] = fma(neg_bits(f.v[u]), p, v[u]);
  }
};

// Full-precision reciprocal (correctly rounded, the value of 1 / x).
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip(double x) { return __drcp_rn(x); }

// Candidate of Step 1 or 2 of one warp (CTAs of several warps): the image of its
// value, its key, the last pivot on its column (row) and two values.
template <typename T>
struct __align__(16) Cand {
  Img<T> o;
  unsigned key;
  int last;
  T a, b;
};

// Shared memory of one CTA: `ks` history entries, then the small arrays.
template <typename T>
__host__ __device__ inline LazyLayout lazy_layout(int lim_m, int lim_n, int warps, int rows, int ks, int kmax, int kw) {
  LazyLayout L{};
  L.pn = (lim_m + kApplyRows - 1) & ~(kApplyRows - 1);
  L.hs = L.pn + ((lim_n + 3) & ~3);
  L.ks = ks;
  L.kmax = kmax;
  L.kw = kw;
  L.ld = lim_n;
  L.kx = ((lim_m < lim_n ? lim_m : lim_n) + 3) & ~3;
  int o = 0;
  auto take = [&](int bytes) { const int at = o; o = (o + bytes + 15) & ~15; return at; };
  L.hist = take(ks * L.hs * int(sizeof(T)));
  L.rp = take(kmax * int(sizeof(T)));
  L.at = take(kmax * 4);
  if (sizeof(T) == 4) {
    L.xq = take(2 * L.kx * 8);
    L.dv = take(2 * L.kx * 4);
    L.off = take(2 * L.kx * 4);
    L.kr = take(L.kx * 2);
    L.flag = take(2 * 32 * warps * rows);
  }
  L.red = take(warps > 1 ? 2 * warps * int(sizeof(Cand<T>)) + 8 * warps * 8 + 16 : 0);
  L.bytes = o;
  return L;
}

// The pivots of the history on the tableau in the slot (`based`; else on A), into the
// slot: kApplyRows rows of NC columns (kApplyCols; one in FP64 and at 64 registers, where
// two cost type-1 LPs of 28 x 28 10%) per thread at a time, with every pivot before they
// are stored, so that one pass over the tableau serves all of them.  Bound by the latency of
// that pass with a few warps per LP: two columns halve the round trips to L2 (20,000 x 100 x
// 100 of 126 pivots, plain FP32, inlined: 10.1 ms with one, 9.1 with two, 8.8 with four,
// which take registers from the kernel); in FP64 by that pipe.  Not inlined, and called
// outside of the pivot loop: LPs of few pivots never get here, and its code cost them 4%
// (50,000 x 100) to 15% (48 x 37) there.
template <typename T, int NT, int NC, bool F64, bool RN>
__device__ __noinline__ void apply_pivots(T *tab, const T *spill, const void *A, int m, int n, int held, bool based,
                                          int hist_at, int ats_at, int ks, int hs, int pn, int ld) {
  extern __shared__ __align__(16) unsigned char lz_smem[];
  __builtin_assume(__isGlobal(tab));
  __builtin_assume(__isGlobal(spill));
  __builtin_assume(__isGlobal(A));
  const T *hist = reinterpret_cast<const T *>(lz_smem + hist_at);
  const unsigned *ats = reinterpret_cast<const unsigned *>(lz_smem + ats_at);
  const int nj = (n + NC - 1) / NC, tasks = (m + kApplyRows - 1) / kApplyRows * nj;
#pragma unroll 1
  for (int t = threadIdx.x; t < tasks; t += NT) {
    const int ib = t / nj, j0 = t - ib * nj, i0 = ib * kApplyRows;
    int j[NC];                 // (past the end: the last column, not stored)
#pragma unroll
    for (int c = 0; c < NC; ++c) j[c] = min(j0 + c * nj, n - 1);
    Rows<T> x[NC];
#pragma unroll
    for (int u = 0; u < kApplyRows; ++u) {
      const int i = min(i0 + u, m - 1);
#pragma unroll
      for (int c = 0; c < NC; ++c) x[c].set(u, based ? tab[i * ld + j[c]] : a_in<T, F64, RN>(A, i * n + j[c]));
    }
    auto steps = [&](auto U, const T *first, int s0, int s1) {
#pragma unroll U.value
      for (int s = s0; s < s1; ++s) {
        const T *h = first + (s - s0) * hs;
        Rows<T> f;
        T p[NC];
        f.load(h + i0);
#pragma unroll
        for (int c = 0; c < NC; ++c) p[c] = h[pn + j[c]];
        const int l = int(ats[s] >> 16) - i0, e = int(ats[s] & 0xffffu);
#pragma unroll
        for (int c = 0; c < NC; ++c)
          if (j[c] == e) {
#pragma unroll
            for (int u = 0; u < kApplyRows; ++u) x[c].set(u, neg_zero<T>());
          }
        if (unsigned(l) < unsigned(kApplyRows)) {
#pragma unroll
          for (int u = 0; u < kApplyRows; ++u)
#pragma unroll
            for (int c = 0; c < NC; ++c)
              if (u == l) x[c].set(u, neg_zero<T>());
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) x[c].sub(f, p[c]);
      }
    };
    steps(std::integral_constant<int, 2>(), hist, 0, held < ks ? held : ks);
    steps(std::integral_constant<int, sizeof(T) == 8 ? 2 : 4>(), spill, ks, held);
#pragma unroll
    for (int u = 0; u < kApplyRows; ++u)
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (i0 + u < m && j0 + c * nj < n) tab[(i0 + u) * ld + j[c]] = x[c].get(u);
  }
}

// Refinement and certificate of an LP whose tableau is in the slot: as the tableau kernel
// does, at most three corrections, by products with the tableau's rows of basic
// structurals and columns of non-basic slacks, until the FP64 residuals are far below the
// certificate's bar, which they are then held against.  x and y in `xq`; returns c^T x, NaN
// where the certificate fails.
template <int W, bool F64>
__device__ __noinline__ double refine_by_tableau(const float *tab, const void *A_, const void *b_, const void *c_, int m,
                                                 int n, int ld, int k, int kx, int hist_at, int hs, int pn, int xq_at,
                                                 int off_at, int kr_at, int flag_at, int rows_at, int sums_at, double tol,
                                                 double tp, double td) {
  extern __shared__ __align__(16) unsigned char lz_smem[];
  __builtin_assume(__isGlobal(tab));
  __builtin_assume(__isGlobal(A_));
  __builtin_assume(__isGlobal(b_));
  __builtin_assume(__isGlobal(c_));
  using In = std::conditional_t<F64, double, float>;
  constexpr int NT = 32 * W;
  const In *A = static_cast<const In *>(A_), *b = static_cast<const In *>(b_), *c = static_cast<const In *>(c_);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  float *res = reinterpret_cast<float *>(lz_smem + hist_at);         // residuals by row, and by column from pn on
  const short *cp = reinterpret_cast<const short *>(res + hs), *rq = cp + kx;
  double *xq = reinterpret_cast<double *>(lz_smem + xq_at), *sums = reinterpret_cast<double *>(lz_smem + sums_at);
  const int *off = reinterpret_cast<const int *>(lz_smem + off_at);
  const short *kr = reinterpret_cast<const short *>(lz_smem + kr_at);
  const unsigned char *row_in = lz_smem + flag_at, *col_in = lz_smem + rows_at;
  auto any = [&](int v) -> int {
    if constexpr (W == 1) return __any_sync(kFull, v);
    else return __syncthreads_or(v);
  };
  int bd;
#pragma unroll 1
  for (int step = 0;; ++step) {
    if constexpr (W == 1) __syncwarp();
    else __syncthreads();
    int more = 0;
    bd = 0;
#pragma unroll 1
    for (int i = tid; i < m; i += NT) {
      double s = 0.0;
#pragma unroll 4
      for (int q = 0; q < k; ++q) s = fma(double(__ldg(A + (i * n + off[q]))), xq[q], s);
      const double r = double(__ldg(b + i)) - s;
      res[i] = __double2float_rn(r);
      bd |= !(r >= -tp);
      more |= row_in[i] && !(fabs(r) <= kStop * tp);
    }
#pragma unroll 1
    for (int j = tid; j < n; j += NT) {
      double s = 0.0;
#pragma unroll 4
      for (int q = 0; q < k; ++q) s = fma(double(__ldg(A + (off[kx + q] + j))), xq[kx + q], s);
      const double d = s - double(__ldg(c + j));
      res[pn + j] = __double2float_rn(d);
      bd |= !(d >= -td);
      more |= col_in[j] && !(fabs(d) <= kStop * td);
    }
    if constexpr (W == 1) __syncwarp();      // (several warps: the vote's barrier)
    if (!any(more) || step == 3) break;
#pragma unroll 1
    for (int t = tid; t < k; t += NT) {
      const float *row = tab + rq[t] * ld, *column = tab + cp[t];
      float dx = 0.f, dy = 0.f;
#pragma unroll 4
      for (int q = 0; q < k; ++q) {
        dx = fmaf(row[cp[q]], res[kr[q]], dx);
        dy = fmaf(-column[rq[q] * ld], res[pn + off[q]], dy);
      }
      xq[t] += double(dx);
      xq[kx + t] += double(dy);
    }
  }
  double cx = 0.0, by = 0.0;
  for (int q = tid; q < k; q += NT) {
    const double x = xq[q], y = xq[kx + q];
    bd |= int(!(x >= -tp)) | int(!(y >= -td));
    cx = fma(double(__ldg(c + off[q])), x, cx);
    by = fma(double(__ldg(b + kr[q])), y, by);
  }
  cx = warp_sum(cx);
  by = warp_sum(by);
  if constexpr (W > 1) {
    if (lane == 0) { sums[wid] = cx; sums[W + wid] = by; }
    __syncthreads();
    cx = by = 0.0;
    for (int w = 0; w < W; ++w) {
      cx += sums[w];
      by += sums[W + w];
    }
  }
  bd |= !(fabs(cx - by) <= tol * (1.0 + fabs(cx)));
  return any(bd) ? __longlong_as_double(0x7ff8000000000000ll) : cx;
}

// T: the tableau's type; W warps and R rows (columns) per thread; F64: the
// input's type; RN: the tableau kernel's arithmetic (input rounded, exact
// ratios) instead of the register kernel's (input truncated, approximate ones).
// KIND: kShared (objectives of one polytope, with warm starts), kRandom (the
// random entering rule), both, and kPacked (with RN: the arithmetic of the
// several-LPs-per-warp kernel, ratios by the rounded reciprocal, and no
// refinement) are their own instantiations, so that the common one carries none of them.
template <typename T, int W, int R, int MINB, bool F64, bool RN, int KIND>
__global__ void __launch_bounds__(32 * W, MINB) lazy_kernel(const TableauParams P, const LazyLayout L) {
  extern __shared__ __align__(16) unsigned char lz_smem[];
  using In = std::conditional_t<F64, double, float>;
  using Im = Img<T>;
  constexpr int NT = 32 * W, D = NT * R;
  constexpr bool kD = sizeof(T) == 8, SHARED = (KIND & kShared) != 0, PACKED = KIND == kPacked;
  // History entries in flight from the workspace (four with one or two warps, or in FP64, take
  // registers from the rest: 48 x 37 278 us with one, 286 with two; 50,000 x 100 2.04 and 2.08
  // ms with two and four, FP64 20,000 x 100 1.37 and 1.6 with one and four).
  constexpr int kSpillUnroll = kD || (W == 1 && !PACKED) ? 1 : RN && !PACKED ? 4 : 2;
  constexpr unsigned long long kInf = 0x7ff0000000000000ull;
  constexpr Im kNone = Im(~Im(0));
  T *hist = reinterpret_cast<T *>(lz_smem + L.hist);
  T *rps = reinterpret_cast<T *>(lz_smem + L.rp);             // 1 / p of pivot s
  unsigned *ats = reinterpret_cast<unsigned *>(lz_smem + L.at);   // its row << 16 | its column
  Cand<T> *red = reinterpret_cast<Cand<T> *>(lz_smem + L.red);    // [2][W]
  // (several warps) 2 W magnitudes, 2 W + 2 W sums or counts, a claim
  unsigned long long *mags = reinterpret_cast<unsigned long long *>(lz_smem + L.red + 2 * W * int(sizeof(Cand<T>)));
  double *sums = reinterpret_cast<double *>(mags + 2 * W);
  int *votes = reinterpret_cast<int *>(mags + 4 * W);
  float *fvote = reinterpret_cast<float *>(mags + 6 * W);
  int *claimed = reinterpret_cast<int *>(mags + 8 * W);
  // The CTA's slot: history entries beyond `ks`, then the tableau of an LP of many pivots.
  T *spill = reinterpret_cast<T *>(static_cast<unsigned char *>(P.slots) + size_t(blockIdx.x) * P.slot_bytes);
  auto tableau = [&]() {           // (formed where it is needed: few LPs get there)
    int entries = L.kmax - L.ks;
    asm volatile("" : "+r"(entries));
    return spill + size_t(entries) * size_t(L.hs);
  };
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int hs = L.hs, ks = L.ks, pn = L.pn;
  const int nitems = P.in.count ? min(*P.in.count, P.list_cap) : P.B.count;
  const T eps_p = T(P.eps_p), eps_d = T(P.eps_d);

  auto sync = [&]() {
    if constexpr (W == 1) __syncwarp();
    else __syncthreads();
  };
  auto any = [&](int v) -> int {
    if constexpr (W == 1) return __any_sync(kFull, v);
    else return __syncthreads_or(v);
  };
  // Value of v[] at row (column) idx (one warp).
  auto pick = [&](const auto &v, int idx) {
    auto x = v[0];
#pragma unroll
    for (int r = 1; r < R; ++r) {
      const auto y = v[r];
      x = (idx >> 5) == r ? y : x;
    }
    return __shfl_sync(kFull, x, idx & 31);
  };
  auto fits_lp = [&](int m, int n) {
    return m >= 1 && n >= 1 && m <= P.lim_m && n <= P.lim_n && m <= P.B.max_m && n <= P.B.max_n && m <= D && n <= D;
  };
  auto read_desc = [&](int it, int &lp_, int &m_, int &n_, long long &a_, long long &b_, long long &c_) {
    lp_ = P.in.items ? __ldg(P.in.items + it) : it;
    m_ = __ldg(P.B.m + lp_);
    n_ = __ldg(P.B.n + lp_);
    a_ = __ldg(P.B.a_off + lp_);
    b_ = __ldg(P.B.b_off + lp_);
    c_ = __ldg(P.B.c_off + lp_);
  };
  // Claims are made one LP ahead; a CTA of several warps passes them on in
  // shared memory, before the barrier of the vote on the input.  Objectives of
  // one polytope (P.shared) are claimed kShareChunk consecutive ones at a time.
  auto claim = [&](int cur) -> int {
    if (!SHARED) return atomicAdd(P.queue, 1);
    // Another CTA has met a direction of many pivots: no more of them are taken.
    if (*static_cast<volatile int32_t *>(P.over_count) != 0) return nitems;
    if (cur >= 0 && (cur + 1) % kShareChunk != 0 && cur + 1 < nitems) return cur + 1;
    return atomicAdd(P.queue, 1) * kShareChunk;
  };
  int item = 0;
  if (tid == 0) item = claim(-1);
  if constexpr (W == 1) {
    item = __shfl_sync(kFull, item, 0);
  } else {
    if (tid == 0) *claimed = item;
    __syncthreads();
    item = *claimed;
    __syncthreads();
  }
  int lp = 0, m = 0, n = 0;
  long long aoff = 0, boff = 0, coff = 0;
  if (item < nitems) read_desc(item, lp, m, n, aoff, boff, coff);
  // What a warm start of the next objective of one polytope keeps (SHARED).
  T rhs[R], obj[R];
  unsigned bkey[R], nkey[R];       // keys of each row and column: its variable << kIdxBits | its index
  int rst[R], cst[R];              // last pivot on each row and column, -1: none
  unsigned long long bm = 0ull;    // largest |b| (its bits)
  int held = 0;                    // pivots in the history
  bool based = false;              // they are pivots on the slot's tableau, not on A
  int warm_run = 0;                // objectives since a cold start; -1: the history is no basis of this polytope
  bool scanned = false;            // the shared A is known to be finite
  int cold_left = 0;               // objectives to start cold, since a warm start took many pivots
  int cold_iters = 0;              // pivots of the last cold start
  int nitem = 0;
  bool again = false;              // the same objective once more, cold
#pragma unroll 1
  while (item < nitems) {
    if (tid == 0 && !(SHARED && again)) nitem = claim(item);
    again = false;
    // ---- admission: sizes, b >= 0, finite data in the tableau's range ----
    const In *A = static_cast<const In *>(P.B.A) + aoff;
    const In *bg = static_cast<const In *>(P.B.b) + boff, *cg = static_cast<const In *>(P.B.c) + coff;
    const bool fits = fits_lp(m, n);
    int bad = !fits;
    // A warm start keeps the basis of the objective before: for a bounded number
    // of objectives (FP32 round-off grows with the pivots), and not where the
    // directions have little to do with one another.
    const bool warm = SHARED && warm_run >= 0 && warm_run < kWarmMax && held > 0 && cold_left == 0;
    if (SHARED && cold_left > 0) --cold_left;
    unsigned long long cm = 0ull;
    int ic[R], jc[R];              // own rows and columns; past the end the last one (read, never used)
    bool in_m[R], in_n[R];
    if (fits) {                    // (the same in every thread)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = tid + NT * r;
        in_m[r] = i < m;
        in_n[r] = i < n;
        ic[r] = min(i, m - 1);
        jc[r] = min(i, n - 1);
        const In b = __ldg(bg + ic[r]), c = __ldg(cg + jc[r]);
        const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(widen(b)));
        const unsigned long long a = u & 0x7fffffffffffffffull;
        const unsigned long long v = static_cast<unsigned long long>(__double_as_longlong(widen(c))) & 0x7fffffffffffffffull;
        bad |= int((u >> 63) != 0ull && a != 0ull);
        if (r == 0) bm = 0ull;
        bm = a > bm ? a : bm;
        cm = v > cm ? v : cm;
        T bt;
        if constexpr (kD) {
          bt = widen(b);
          obj[r] = neg(widen(c));
        } else if constexpr (!F64) {
          bt = b;
          obj[r] = -c;
        } else if constexpr (PACKED) {
          bt = d2f_rn(b);
          obj[r] = -d2f_rn(c);
        } else if constexpr (RN) {
          bt = __double2float_rn(b);
          obj[r] = -__double2float_rn(c);
          bad |= int(!isfinite(bt)) | int(!isfinite(obj[r]));
        } else {
          bt = d2f_tile(b, bad);
          obj[r] = -d2f_tile(c, bad);
        }
        if (!warm) {
          rhs[r] = bt;
          bkey[r] = unsigned(((n + i) << kIdxBits) | i);
          nkey[r] = unsigned((i << kIdxBits) | i);
          rst[r] = -1;
          cst[r] = -1;
        }
      }
      bad |= int(bm >= kInf) | int(cm >= kInf);
      if ((!SHARED || !scanned) && !any(bad)) {      // (an LP for Phase I is not read through)
        const unsigned amax = scan_a<F64, NT>(A, m * n, tid);
        // Not finite, or (FP32) so large that rounding could leave the float range.
        bad |= int(amax >= (F64 ? (kD ? 0x7ff00000u : 0x47efffffu) : 0x7f800000u));
      }
    }
    bm = warp_max_u64(bm);
    cm = warp_max_u64(cm);
    if constexpr (W > 1) {
      if (tid == 0) *claimed = nitem;
      if (lane == 0) { mags[wid] = bm; mags[W + wid] = cm; }
    }
    bad = any(bad);
    if constexpr (W == 1) nitem = __shfl_sync(kFull, nitem, 0);
    else nitem = *claimed;
    int nlp = 0, nm = 0, nn = 0;
    long long na = 0, nb = 0, nc = 0;
    if (nitem < nitems) read_desc(nitem, nlp, nm, nn, na, nb, nc);
    auto next = [&]() {
      item = nitem; lp = nlp; m = nm; n = nn; aoff = na; boff = nb; coff = nc;
      sync();
    };
    auto defer = [&]() {           // the tableau kernel takes it (Phase I, sizes, bad data)
      if (tid == 0) {
        P.R.status[lp] = STATUS_PENDING;
        list_push(P.defer_items, P.defer_count, P.list_cap, lp, P.err);
      }
    };
    if (bad) {
      warm_run = -1;
      defer();
      next();
      continue;
    }
    if constexpr (SHARED) {
      scanned = true;
      warm_run = warm ? warm_run + 1 : 0;
    }
    if (!warm) {
      held = 0;
      based = false;
    }

    // The block's best candidate: least image o[], then least key (kNone: no
    // candidate), with the values va, vb and the last pivot of its owner.  One
    // block barrier; `which` keeps Step 1's and Step 2's records apart, so that a
    // record is written again only after another barrier.
    auto choose = [&](int which, const Im (&o)[R], const unsigned (&keys)[R], const T (&va)[R], const T (&vb)[R],
                      const int (&last)[R]) -> Cand<T> {
      Cand<T> best;
      Im mo = o[0];
#pragma unroll
      for (int r = 1; r < R; ++r) mo = o[r] < mo ? o[r] : mo;
      best.o = warp_min(mo);
      unsigned mk = 0xffffffffu;
#pragma unroll
      for (int r = 0; r < R; ++r) mk = min(mk, o[r] == best.o ? keys[r] : 0xffffffffu);
      best.key = __reduce_min_sync(kFull, mk);
      if constexpr (W == 1) {
        const int i = int(best.key) & kIdxMask;
        best.a = pick(va, i);
        best.b = pick(vb, i);
        best.last = pick(last, i);
      } else {
        Cand<T> *rc = red + which * W;
        if (best.o == kNone) {
          if (lane == 0) { rc[wid].o = kNone; rc[wid].key = 0xffffffffu; }
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (best.key == keys[r]) rc[wid] = Cand<T>{best.o, best.key, last[r], va[r], vb[r]};
        }
        __syncthreads();
        const Im co = rc[lane & (W - 1)].o;
        best.o = warp_min(co);
        best.key = __reduce_min_sync(kFull, co == best.o ? rc[lane & (W - 1)].key : 0xffffffffu);
        const Cand<T> &c = rc[int(best.key & unsigned(NT - 1)) / 32];
        best.a = c.a;
        best.b = c.b;
        best.last = c.last;
      }
      return best;
    };
    // Entry s of the history.
    auto entry = [&](int s) -> const T * { return s < ks ? hist + s * hs : spill + (s - ks) * hs; };

    // The history's pivots on an objective row w (by column), and on a right-hand
    // side v (by row) where there is one.
    auto through_pivots = [&](float *v, float *w) __attribute__((always_inline)) {
      float *bc = reinterpret_cast<float *>(sums);       // [2 parities][v_l, w_e] (several warps)
      auto publish = [&](int s) {
        const int l = int(ats[s] >> 16), e = int(ats[s] & 0xffffu);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (v && tid + NT * r == l) bc[2 * (s & 1)] = v[r];
          if (tid + NT * r == e) bc[2 * (s & 1) + 1] = w[r];
        }
      };
      if (W > 1 && held > 0) publish(0);
#pragma unroll 1
      for (int s = 0; s < held; ++s) {
        const T *h = entry(s);
        const int l = int(ats[s] >> 16), e = int(ats[s] & 0xffffu);
        float vl = 0.f, fm;
        if constexpr (W == 1) {
          float x = w[0], y = v ? v[0] : 0.f;
#pragma unroll
          for (int r = 1; r < R; ++r) {
            const float xr = w[r], yr = v ? v[r] : 0.f;
            x = (e >> 5) == r ? xr : x;
            y = (l >> 5) == r ? yr : y;
          }
          if (v) vl = __shfl_sync(kFull, y, l & 31);
          fm = __shfl_sync(kFull, x, e & 31) * float(rps[s]);
        } else {
          __syncthreads();
          vl = bc[2 * (s & 1)];
          fm = bc[2 * (s & 1) + 1] * float(rps[s]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = tid + NT * r;
          if (v) v[r] = fmaf(-float(h[ic[r]]), vl, i == l ? -0.f : v[r]);
          w[r] = fmaf(-fm, float(h[pn + jc[r]]), i == e ? -0.f : w[r]);
        }
        if (W > 1 && s + 1 < held) publish(s + 1);
      }
      if constexpr (W > 1) __syncthreads();
    };

    // ---- Steps 1-3 ----
    const int max_iter = P.max_iter > 0 ? P.max_iter : 50 * (m + n);
    int iters = 0, status = LPB_OPTIMAL, degenerate_run = 0;
    T z = T(0);
    if constexpr (SHARED) {
      if (warm) {                  // the new objective row on the basis kept: -c through its pivots
        sync();
        through_pivots(nullptr, obj);
        if (P.mode == MODE_FP32) { // and z = c_B x_B (refinement forms its own)
          float part = 0.f;
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int v = int(bkey[r] >> kIdxBits);
            int none = 0;
            if (in_m[r] && v < n) {
              if constexpr (F64) part = fmaf(d2f_tile(__ldg(cg + v), none), rhs[r], part);
              else part = fmaf(__ldg(cg + v), rhs[r], part);
            }
          }
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(kFull, part, off);
          if constexpr (W > 1) {
            if (lane == 0) fvote[wid] = part;
            __syncthreads();
            part = 0.f;
#pragma unroll
            for (int w = 0; w < W; ++w) part += fvote[w];
          }
          z = part;
        }
      }
    }
    bool bland = false, full = false;
#pragma unroll 1
    for (;;) {
      full = false;
#pragma unroll 1
      for (;;) {
        // Step 1: the most negative reduced cost (Bland: the lowest variable).
        Im o[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          o[r] = in_n[r] && above(neg(obj[r]), eps_d) ? (bland ? Im(0) : image(obj[r])) : kNone;
          // The random rule: the least key of the variable at this pivot (FP32: of
          // its upper 31 bits, as the register kernel ranks; RN: of all but the one
          // value that stands for no candidate).
          if constexpr ((KIND & kRandom) != 0)
            if (o[r] != kNone && !bland) {
              const unsigned key = rpc_key(P.seed, P.lp_base + lp, iters, int(nkey[r] >> kIdxBits));
              o[r] = kD ? Im(key) : RN ? Im(min(key, 0xfffffffeu)) : Im(key >> 1);
            }
        }
        const Cand<T> col = choose(0, o, nkey, obj, obj, cst);
        if (col.o == kNone) break;
        if (held == (based ? L.kw : L.kmax)) { full = true; break; }
        // (a start from the wrong basis, and its pivots go to the workspace)
        if (SHARED && warm && held >= ks && 2 * iters > cold_iters) { full = true; break; }
        const int e = int(col.key) & kIdxMask, cse = col.last;
        // Column e: from A (the slot's tableau) or from the pivot that last stood on it,
        // then the pivots since.
        T a[R];
        const int e1 = held < ks ? held : ks;
        {
          int s = cse + 1;
          if (cse < 0 && based) {
            const T *tab = tableau() + e;
            const int ld = L.ld;
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = tab[ic[r] * ld];
          } else if (cse < 0) {
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = a_in<T, F64, RN>(A, ic[r] * n + e);
          } else {
            const T *h = entry(cse);
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = neg(h[ic[r]]);
          }
#pragma unroll 4
          for (; s < e1; ++s) {
            const T *h = hist + s * hs;
            const T pe = h[pn + e];
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = mul_add(neg(h[ic[r]]), pe, s == rst[r] ? neg_zero<T>() : a[r]);
          }
#pragma unroll kSpillUnroll
          for (; s < held; ++s) {
            const T *h = spill + (s - ks) * hs;
            const T pe = h[pn + e];
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = mul_add(neg(h[ic[r]]), pe, s == rst[r] ? neg_zero<T>() : a[r]);
          }
        }
        // Step 2: the min-ratio test.
        if constexpr (kD) {
          // The ratios in FP32 first (relative error below 3e-7; FP64 division is
          // slow here): only rows within 1e-5 of the smallest get the exact
          // quotient, and none does when a single row is left whose ratio is
          // clearly above the degeneracy threshold.
          float q[R], m32 = __int_as_float(0x7f800000);
          bool el[R];
#pragma unroll
          for (int r = 0; r < R; ++r) {
            el[r] = in_m[r] && above(a[r], eps_p);
            q[r] = el[r] ? __fdiv_rn(d2f_rn(rhs[r]), d2f_rn(a[r])) : __int_as_float(0x7f800000);
            if (el[r]) m32 = fminf(m32, q[r]);
          }
          m32 = ord2f(__reduce_min_sync(kFull, f2ord(m32)));
          if constexpr (W > 1) {
            if (lane == 0) fvote[wid] = m32;
            __syncthreads();
            m32 = ord2f(__reduce_min_sync(kFull, f2ord(fvote[lane & (W - 1)])));
          }
          const float cut = m32 + 1e-5f * fabsf(m32);
          int cnt = 0;
#pragma unroll
          for (int r = 0; r < R; ++r) {
            el[r] = el[r] && !(q[r] > cut);
            cnt += el[r];
          }
          int all = int(__reduce_add_sync(kFull, unsigned(cnt)));
          if constexpr (W > 1) {
            if (lane == 0) votes[wid] = all;
            __syncthreads();
            all = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) all += votes[w];
          }
          const bool one = all == 1 && m32 > 4.f * float(eps_p);
#pragma unroll
          for (int r = 0; r < R; ++r) {
            o[r] = kNone;
            if (__any_sync(kFull, el[r])) {
              const double t = one ? f2d_exact(q[r]) : rhs[r] / a[r];
              if (el[r]) o[r] = image(t);
            }
          }
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r)
            o[r] = in_m[r] && a[r] > eps_p ? image(T(PACKED ? rhs[r] * recip(a[r]) : RN ? rhs[r] / a[r] : rhs[r] * rcp_approx(float(a[r])))) : kNone;
        }
        const Cand<T> row = choose(1, o, bkey, a, rhs, rst);
        if (row.o == kNone) { status = LPB_UNBOUNDED; break; }
        if (iters >= max_iter) { status = LPB_ITER_LIMIT; break; }
        const int l = int(row.key) & kIdxMask, rsl = row.last;
        const T rp = recip(row.a), bl = row.b;
        // Row l likewise.
        T p[R];
        {
          int s = rsl + 1;
          if (rsl < 0 && based) {
            const T *tab = tableau() + l * L.ld;
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = tab[jc[r]];
          } else if (rsl < 0) {
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = a_in<T, F64, RN>(A, l * n + jc[r]);
          } else {
            const T *h = entry(rsl) + pn;
            const T rs = rps[rsl];
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = h[jc[r]] * rs;
          }
#pragma unroll 4
          for (; s < e1; ++s) {
            const T *h = hist + s * hs;
            const T nf = neg(h[l]);
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = mul_add(nf, h[pn + jc[r]], s == cst[r] ? neg_zero<T>() : p[r]);
          }
#pragma unroll kSpillUnroll
          for (; s < held; ++s) {
            const T *h = spill + (s - ks) * hs;
            const T nf = neg(h[l]);
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = mul_add(nf, h[pn + jc[r]], s == cst[r] ? neg_zero<T>() : p[r]);
          }
        }
        // Step 3 on the right-hand side and the objective row, and the pivot into
        // the history.
        T *h = held < ks ? hist + held * hs : spill + (held - ks) * hs;
        const T fm = col.a * rp;
        z = mul_add(neg(fm), bl, z);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = tid + NT * r;
          const bool is_l = i == l, is_e = i == e;
          const T f = is_l ? neg(rp) : a[r] * rp;
          const T v = is_e ? T(1) : p[r];
          rhs[r] = mul_add(neg(f), bl, is_l ? neg_zero<T>() : rhs[r]);
          obj[r] = mul_add(neg(fm), v, is_e ? neg_zero<T>() : obj[r]);
          if (in_m[r]) h[i] = f;
          if (in_n[r]) h[pn + i] = v;
          if (is_l) { bkey[r] = (col.key & ~unsigned(kIdxMask)) | unsigned(l); rst[r] = held; }
          if (is_e) { nkey[r] = (row.key & ~unsigned(kIdxMask)) | unsigned(e); cst[r] = held; }
        }
        if (tid == 0) { rps[held] = rp; ats[held] = unsigned(l << 16 | e); }
        if constexpr (W == 1) __syncwarp();     // (several warps: the next Step 1's barrier)
        ++iters;
        ++held;
        if (!above(unimage(row.o), eps_p)) {
          if (++degenerate_run >= m + n) bland = true;
        } else {
          degenerate_run = 0;
          bland = false;
        }
      }
      sync();
      // The pivots into the slot's tableau: where no more of them are kept, and for the
      // refinement of an LP whose earlier ones went there.
      const bool refines = !kD && !PACKED && P.mode == MODE_FP32_REFINE && status == LPB_OPTIMAL;
      if (SHARED || (!full && !(refines && based && held > 0))) break;
      apply_pivots<T, NT, kD || PACKED ? 1 : kApplyCols, F64, RN>(tableau(), spill, A, m, n, held, based, L.hist, L.at, ks, hs, pn, L.ld);
#pragma unroll
      for (int r = 0; r < R; ++r) rst[r] = cst[r] = -1;
      held = 0;
      based = true;
      sync();
      if (!full) break;
    }
    if (SHARED && full) {
      if (warm) {                  // the history is full after some warm starts: cold
        if (2 * iters > cold_iters) cold_left = kShareChunk - 1;
        again = true;
        warm_run = -1;
        continue;
      }
      if (tid == 0) *P.over_count = P.B.count;      // many pivots: the register kernel's launch
      break;                                        // solves what has no status yet
    }
    int bvar[R], nvar[R];          // basic variable of each row, non-basic variable of each column
#pragma unroll
    for (int r = 0; r < R; ++r) {
      bvar[r] = int(bkey[r] >> kIdxBits);
      nvar[r] = int(nkey[r] >> kIdxBits);
    }
    if (status == LPB_ITER_LIMIT) warm_run = -1;
    if (!warm) cold_iters = iters;
    if (warm && 2 * iters > cold_iters) cold_left = kShareChunk - 1;
    const int64_t yoff = P.R.y_off ? P.R.y_off[lp] : boff;    // outputs packed like b, or at y_off
    if (int32_t *bp = P.bbuf ? P.bbuf + (P.bpacked ? yoff : int64_t(lp) * P.B.max_m) : nullptr) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (in_m[r]) bp[tid + NT * r] = bvar[r];
    }
    const bool opt = status == LPB_OPTIMAL;
    if (kD || PACKED || P.mode != MODE_FP32_REFINE) {          // results straight from the tableau; zeros where there is none
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = tid + NT * r, u = opt ? nvar[r] : i, v = opt ? bvar[r] : n + i;
        if (in_n[r]) {
          if (u < n) P.R.x[coff + u] = 0.0;
          else if (P.R.y) P.R.y[yoff + (u - n)] = widen(obj[r]);
        }
        if (in_m[r]) {
          if (v < n) P.R.x[coff + v] = widen(rhs[r]);
          else if (P.R.y) P.R.y[yoff + (v - n)] = 0.0;
        }
      }
      if (tid == 0) {
        P.R.status[lp] = status;
        if (P.R.iters) P.R.iters[lp] = iters;
        P.R.obj[lp] = opt ? widen(z) : status == LPB_UNBOUNDED ? INFINITY : NAN;
      }
      next();
      continue;
    }
    if constexpr (!kD && !PACKED) {
    // ---- FP64 refinement and certificate ----
    // Numbers of the basic structurals (by row) and the non-basic slacks (by
    // column); there are as many of one as of the other.
    int qi[R], pi[R], k = 0, kn = 0;
    unsigned char *flag = lz_smem + L.flag;                    // [2][D]: row is binding, structural is basic
#pragma unroll
    for (int r = 0; r < R; ++r) flag[tid + NT * r] = flag[D + tid + NT * r] = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool b = in_m[r] && bvar[r] < n, t = in_n[r] && nvar[r] >= n;
      const unsigned mb = __ballot_sync(kFull, b), mt = __ballot_sync(kFull, t), below = (1u << lane) - 1u;
      int hb = 0, ht = 0, nb_ = __popc(mb), nt_ = __popc(mt);
      if constexpr (W > 1) {       // the warps' counts: those before this one, and all
        if (lane == 0) { votes[wid] = nb_; votes[W + wid] = nt_; }
        __syncthreads();
        nb_ = nt_ = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          if (w == wid) { hb = nb_; ht = nt_; }
          nb_ += votes[w];
          nt_ += votes[W + w];
        }
        if (R > 1) __syncthreads();
      }
      qi[r] = b ? k + hb + __popc(mb & below) : -1;
      pi[r] = t ? kn + ht + __popc(mt & below) : -1;
      k += nb_;
      kn += nt_;
    }
    if constexpr (W == 1) __syncwarp();
    bool fail = !opt;              // no optimum: confirm in FP64
    if (L.tab > 0) {               // (the limit that the operands of the warp kernel's refinement set)
      const int kb = kn | 1;
      const int st = ((m * kb * 4 + 15) & ~15) + m * kb * 8 + kn * n * 8 + (m + n) * 8;
      fail |= kn > kWarpRefK || st + (3 * m + n + 2 * kWarpRefK) * 8 + 3 * kWarpRefK * 4 > L.tab;
    }
    double cx = 0.0;
    double *xq = reinterpret_cast<double *>(lz_smem + L.xq);   // [2]: x of the basic structurals, y of the non-basic slacks
    const int kx = L.kx;
    if (!fail) {
      float *dv = reinterpret_cast<float *>(lz_smem + L.dv);     // [2]: residuals, then corrections
      int *off = reinterpret_cast<int *>(lz_smem + L.off);       // [2]: column j_q of A; start of row k_p of A
      short *kr = reinterpret_cast<short *>(lz_smem + L.kr);     // k_p
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (qi[r] >= 0) { off[qi[r]] = bvar[r]; flag[D + bvar[r]] = 1; xq[qi[r]] = widen(rhs[r]); }
        if (pi[r] >= 0) {
          kr[pi[r]] = short(nvar[r] - n);
          flag[nvar[r] - n] = 1;
          off[kx + pi[r]] = (nvar[r] - n) * n;
          xq[kx + pi[r]] = widen(obj[r]);
        }
      }
      const int kp = k > 0 ? (k + 3) & ~3 : 4;
      if (tid < kp - k) {          // the products take four at a time: entries past the end are zero
        off[k + tid] = off[kx + k + tid] = 0;
        xq[k + tid] = xq[kx + k + tid] = 0.0;
        dv[k + tid] = dv[kx + k + tid] = 0.f;
      }
      if constexpr (W > 1) {
#pragma unroll 1
        for (int w = 0; w < W; ++w) {
          bm = mags[w] > bm ? mags[w] : bm;
          cm = mags[W + w] > cm ? mags[W + w] : cm;
        }
      }
      const double tol = P.feas_tol;
      const double tp = tol * (1.0 + __longlong_as_double(static_cast<long long>(bm)));
      const double td = tol * (1.0 + __longlong_as_double(static_cast<long long>(cm)));
      constexpr float kDeltaErr = 1.f / 32768.f;
      if (based) {
        short *cp = reinterpret_cast<short *>(reinterpret_cast<float *>(hist) + hs), *rq = cp + kx;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (qi[r] >= 0) rq[qi[r]] = short(tid + NT * r);
          if (pi[r] >= 0) cp[pi[r]] = short(tid + NT * r);
        }
        cx = refine_by_tableau<W, F64>(reinterpret_cast<const float *>(tableau()), A, bg, cg, m, n, L.ld, k, kx, L.hist, hs, pn,
                                       L.xq, L.off, L.kr, L.flag, L.flag + D, L.red + 2 * W * int(sizeof(Cand<T>)) + 16 * W,
                                       tol, tp, td);
        fail = cx != cx;
      }
#pragma unroll 1
      for (int round = 0; !based; ++round) {
        sync();
        // b - A x by row and A^T y - c by column, in FP64.
        double ra[R], rd[R];
#pragma unroll
        for (int r = 0; r < R; ++r) ra[r] = rd[r] = 0.0;
        unsigned low = 0xffffffffu;
#pragma unroll 1
        for (int q = 0; q < k; q += 4) {
          In va[4][R], vb[4][R];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = off[q + u], i = off[kx + q + u];
#pragma unroll
            for (int r = 0; r < R; ++r) {
              va[u][r] = __ldg(A + (ic[r] * n + j));
              vb[u][r] = __ldg(A + (i + jc[r]));
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (q + u < k) {
              const double x = xq[q + u], y = xq[kx + q + u];
#pragma unroll
              for (int r = 0; r < R; ++r) {
                ra[r] = fma(widen_a(va[u][r], low), x, ra[r]);
                rd[r] = fma(widen_a(vb[u][r], low), y, rd[r]);
              }
            }
        }
        if (!F64 && low < 0x007fffffu) {     // subnormal entries: again, by the hardware's conversion
#pragma unroll
          for (int r = 0; r < R; ++r) {
            ra[r] = rd[r] = 0.0;
#pragma unroll 1
            for (int q = 0; q < k; ++q) {
              ra[r] = fma(double(__ldg(A + (ic[r] * n + off[q]))), xq[q], ra[r]);
              rd[r] = fma(double(__ldg(A + (off[kx + q] + jc[r]))), xq[kx + q], rd[r]);
            }
          }
        }
        // The residuals that a correction has to take up are those of the binding
        // rows and of the basic structurals' columns (a basic slack takes its own).
        float v[R], w[R], rp_[R], rd_[R];
        int more = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          ra[r] = widen(__ldg(bg + ic[r])) - ra[r];
          rd[r] = rd[r] - widen(__ldg(cg + jc[r]));
          const bool tr = in_m[r] && flag[tid + NT * r], tc = in_n[r] && flag[D + tid + NT * r];
          v[r] = __double2float_rn(ra[r]);
          w[r] = __double2float_rn(rd[r]);
          if constexpr (!RN) { rp_[r] = v[r]; rd_[r] = w[r]; }
          v[r] = tr ? v[r] : 0.f;
          w[r] = tc ? w[r] : 0.f;
          // RN: as the tableau kernel does, corrections (three at most) until the
          // residuals are far below the certificate's bar (kStop).
          if constexpr (RN)
            more |= int(tr && !dge(kStop * tp, abs_bits(ra[r]))) | int(tc && !dge(kStop * td, abs_bits(rd[r])));
        }
        bool correct = true;
        if constexpr (RN) correct = any(more) && round < 3;
        if (correct) {
          // Corrections with the FP32 basis inverse: the pivots on v as another
          // right-hand side, on w as another objective row.
          through_pivots(v, w);
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (qi[r] >= 0) dv[qi[r]] = v[r];
            if (pi[r] >= 0) dv[kx + pi[r]] = w[r];
          }
          sync();
        }
        // The corrected x and y, and c^T x and b^T y.
        int bd = 0;
        double cxp = 0.0, byp = 0.0, by;
#pragma unroll 1
        for (int q = tid; q < k; q += NT) {
          double x = xq[q], y = xq[kx + q];
          if (correct) {
            x += widen(dv[q]);
            y += widen(dv[kx + q]);
            xq[q] = x;
            xq[kx + q] = y;
          }
          bd |= int(!dge(x, neg_bits(tp))) | int(!dge(y, neg_bits(td)));
          cxp = fma(widen(__ldg(cg + off[q])), x, cxp);
          byp = fma(widen(__ldg(bg + kr[q])), y, byp);
        }
        // KKT certificate of the pair that is written out: x >= 0, A x <= b,
        // y >= 0, A^T y >= c and c^T x = b^T y, each to tol scaled by the data.
        // RN: on the residuals of that pair.  Else b - A x and A^T y - c at the
        // corrected point are the FP64 residuals plus FP32 products with the
        // corrections; their rounding (m, n <= 127 terms, and the 2^-20 truncation
        // of A) is bounded by 2^-15 times the sum of the products' magnitudes.
        if constexpr (RN) {
          if (correct) continue;
#pragma unroll
          for (int r = 0; r < R; ++r)
            bd |= int(in_m[r] && !dge(ra[r], neg_bits(tp))) | int(in_n[r] && !dge(rd[r], neg_bits(td)));
        } else {
          float dl[R], mg[R], el[R], eg[R];
#pragma unroll
          for (int r = 0; r < R; ++r) dl[r] = mg[r] = el[r] = eg[r] = 0.f;
#pragma unroll 1
          for (int q = 0; q < k; q += 4) {
            unsigned va[4][R], vb[4][R];
            const unsigned *Aw = reinterpret_cast<const unsigned *>(A);
            constexpr int es = sizeof(In) / 4;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int j = off[q + u], i = off[kx + q + u];
#pragma unroll
              for (int r = 0; r < R; ++r) {
                va[u][r] = __ldg(Aw + es * (ic[r] * n + j) + es - 1);
                vb[u][r] = __ldg(Aw + es * (i + jc[r]) + es - 1);
              }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float d = dv[q + u], g = dv[kx + q + u];
#pragma unroll
              for (int r = 0; r < R; ++r) {
                const float a = F64 ? hi2f(va[u][r]) : __uint_as_float(va[u][r]);
                const float b = F64 ? hi2f(vb[u][r]) : __uint_as_float(vb[u][r]);
                dl[r] = fmaf(a, d, dl[r]);
                mg[r] = fmaf(fabsf(a), fabsf(d), mg[r]);
                el[r] = fmaf(b, g, el[r]);
                eg[r] = fmaf(fabsf(b), fabsf(g), eg[r]);
              }
            }
          }
          // In FP32 first, with 2^-22 of the residual for its rounding; what does not
          // pass there is compared in FP64.
          const float lim_p = -__double2float_rd(tp), lim_d = -__double2float_rd(td);
          int near_bar = 0;
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const float rp = rp_[r], rq = rd_[r];
            const float sp = rp - dl[r] - fmaf(kDeltaErr, mg[r], 0x1p-22f * fabsf(rp));
            const float sd = rq + el[r] - fmaf(kDeltaErr, eg[r], 0x1p-22f * fabsf(rq));
            near_bar |= int(in_m[r] && !(sp >= lim_p)) | int(in_n[r] && !(sd >= lim_d));
          }
          if (near_bar) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const double sp = ra[r] - widen(fmaf(kDeltaErr, mg[r], dl[r]));
              const double sd = rd[r] + widen(fmaf(-kDeltaErr, eg[r], el[r]));
              bd |= int(in_m[r] && !dge(sp, neg_bits(tp))) | int(in_n[r] && !dge(sd, neg_bits(td)));
            }
          }
        }
        if constexpr (W == 1) {
          cx = warp_sum(cxp);
          by = warp_sum(byp);
        } else {                   // the sums' parts are in the first k threads
          cx = by = 0.0;
          if (32 * wid < k) {
            cxp = warp_sum(cxp);
            byp = warp_sum(byp);
            if (lane == 0) { sums[wid] = cxp; sums[W + wid] = byp; }
          }
          __syncthreads();
#pragma unroll 1
          for (int u = 0; u < W && 32 * u < k; ++u) {
            cx += sums[u];
            by += sums[W + u];
          }
        }
        bd |= !(fabs(cx - by) <= tol * (1.0 + fabs(cx)));
        fail = any(bd);
        if (RN || !fail || round == 2) break;
      }
    }
    // The corrected values of other lanes are read below (several warps: the vote's barrier).
    if constexpr (W == 1) __syncwarp();
    if (!fail) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (in_n[r]) {
          if (nvar[r] < n) P.R.x[coff + nvar[r]] = 0.0;
          else if (P.R.y) P.R.y[yoff + (nvar[r] - n)] = xq[kx + pi[r]];
        }
        if (in_m[r]) {
          if (bvar[r] < n) P.R.x[coff + bvar[r]] = xq[qi[r]];
          else if (P.R.y) P.R.y[yoff + (bvar[r] - n)] = 0.0;
        }
      }
    }
    if (fail && opt) warm_run = -1;          // the next objective starts cold
    if (tid == 0) {
      P.R.status[lp] = fail ? STATUS_PENDING : LPB_OPTIMAL;
      if (!fail) P.R.obj[lp] = cx;
      if (P.R.iters) P.R.iters[lp] = iters;
      if (fail) list_push(P.resolve_items, P.resolve_count, P.list_cap, lp, P.err);
    }
    next();
    }
  }
}

struct LazyConfig {
  int W, R;
  const void *f64, *f32;          // instantiations by input type
  const void *s64, *s32;          // ... for objectives of one polytope (FP32, else the common ones)
};

template <typename T, int W, int R, int MINB, bool RN, int KIND = kCommon>
constexpr LazyConfig lazy_config() {
  constexpr int kS = sizeof(T) == 4 && !RN ? KIND | kShared : KIND;
  return LazyConfig{W, R, reinterpret_cast<const void *>(&lazy_kernel<T, W, R, MINB, true, RN, KIND>),
                    reinterpret_cast<const void *>(&lazy_kernel<T, W, R, MINB, false, RN, KIND>),
                    reinterpret_cast<const void *>(&lazy_kernel<T, W, R, MINB, true, RN, kS>),
                    reinterpret_cast<const void *>(&lazy_kernel<T, W, R, MINB, false, RN, kS>)};
}

inline const void *lazy_fn(const LazyConfig &c, int dtype, bool shared) {
  return dtype == LPB_DTYPE_F64 ? (shared ? c.s64 : c.f64) : (shared ? c.s32 : c.f32);
}

// Smallest configuration of a table that holds LPs up to max_dim, or null.
template <int N>
const LazyConfig *lazy_pick(const LazyConfig (&t)[N], int max_dim) {
  for (const LazyConfig &c : t)
    if (32 * c.W * c.R >= max_dim) return &c;
  return nullptr;
}

template <typename T, int N>
cudaError_t lazy_occ(const LazyConfig (&t)[N], const LazyShape &q, int dtype, int *ctas, int *threads, LazyLayout *lay) {
  const LazyConfig *c = lazy_pick(t, q.max_m > q.max_n ? q.max_m : q.max_n);
  *ctas = 0;
  if (!c) return cudaSuccess;
  *lay = lazy_layout<T>(q.max_m, q.max_n, c->W, c->R, q.ks, q.kmax, q.kw);
  *threads = 32 * c->W;
  if (lay->bytes > 230000) return cudaSuccess;
  const void *fn = lazy_fn(*c, dtype, q.shared);
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, lay->bytes);
  return e != cudaSuccess ? e : cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, fn, *threads, size_t(lay->bytes));
}

template <int N>
cudaError_t lazy_launch(const LazyConfig (&t)[N], const TableauParams &p, const LazyLayout &lay, int grid, cudaStream_t s) {
  const LazyConfig *c = lazy_pick(t, p.lim_m > p.lim_n ? p.lim_m : p.lim_n);
  if (!c) return cudaErrorInvalidValue;
  const void *fn = lazy_fn(*c, p.B.dtype, p.shared != 0);
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, lay.bytes);
  if (e != cudaSuccess) return e;
  void *args[] = {const_cast<TableauParams *>(&p), const_cast<LazyLayout *>(&lay)};
  return cudaLaunchKernel(fn, dim3(grid), dim3(32 * c->W), args, size_t(lay.bytes), s);
}

}  // namespace

}  // namespace lpb
