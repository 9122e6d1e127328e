// Symmetric eigensolver for F = Q diag(eps) Q^T (eq. 19 needs the eigenpairs; eq. 36
// needs them again for the DMPT response), in FP64 and, for the mixed path, in double-float.
//
//  1. Householder tridiagonalisation (tridiag.cu).
//  2. Eigenvalues of the tridiagonal matrix by multisection on Sturm counts, several lanes
//     per eigenvalue (ascending order by construction).  FP64: FP32 counts first, then FP64
//     counts on a grid of points; mixed: double-float counts.
//  3. Eigenvectors by inverse iteration (two steps) with a partially pivoted tridiagonal
//     LU, a thread per eigenvalue; members of a cluster of close eigenvalues are made
//     orthogonal afterwards, a block per cluster.
//  4. Back-transformation Q = H_0 ... H_{n-3} Z with blocks of 128 reflectors in compact
//     WY form (I - V T V^T), carried out on Z^T.  Mixed: the two large products V^T Z and
//     Y^T Z (Y = T^T V, double-float) on the tensor cores with 4 fixed-point BF16 slices.  FP64:
//     all products on the tensor cores as digits (tc_gemm64.cu); up to 66 columns, and
//     without tensor maps, blocks of 64 and products on the FP64 pipe (gemm64.cu).  The T
//     factors are FP64 in both.
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "df.cuh"
#include "kernels.h"
#include "tc_gemm.h"

namespace kx {

constexpr int kBtBlock = 64;          // reflectors per back-transform block (products on the FP64 pipe)
constexpr int kBtBlockTc = 128;       // reflectors per back-transform block (products on the tensor cores)
constexpr double kEps = 2.220446049250313e-16;

// read-only data of this launch (written by an earlier one): cached loads
__device__ __forceinline__ dfl ldg_df(const dfl* p) {
  const float2 v = __ldg((const float2*)p);
  return dfl{v.x, v.y};
}

// Gershgorin interval, squared off-diagonals, pivmin; one block
__global__ void gersh_kernel(int n, const double* __restrict__ d, const double* __restrict__ e,
                             double* __restrict__ e2, double* __restrict__ scal, float* __restrict__ df,
                             float* __restrict__ e2f, dfl* __restrict__ d_dfl, dfl* __restrict__ e2_dfl,
                             dfl* __restrict__ e_dfl) {
  double lo = 1e300, hi = -1e300, em = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double r = 0.0;
    df[i] = (float)d[i];                 // FP32 copies for the coarse phase (no per-step conversions)
    e2f[i] = 0.0f;
    d_dfl[i] = df_from_double(d[i]);     // double-float copies for the multisection and the
    e2_dfl[i] = dfl{0.0f, 0.0f};         // inverse iteration (mixed path)
    e_dfl[i] = (i < n - 1) ? df_from_double(e[i]) : dfl{0.0f, 0.0f};
    if (i > 0) r += fabs(e[i - 1]);
    if (i < n - 1) {
      r += fabs(e[i]);
      e2[i] = e[i] * e[i];
      e2f[i] = (float)e2[i];
      e2_dfl[i] = df_from_double(e2[i]);
      em = fmax(em, e[i] * e[i]);
    }
    lo = fmin(lo, d[i] - r);
    hi = fmax(hi, d[i] + r);
  }
  // min/max reductions through negation-free warp shuffles
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    em = fmax(em, __shfl_xor_sync(0xffffffffu, em, o));
  }
  __shared__ double slo[32], shi[32], sem[32];
  int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) { slo[w] = lo; shi[w] = hi; sem[w] = em; }
  __syncthreads();
  if (threadIdx.x == 0) {
    int nw = (blockDim.x + 31) >> 5;
    for (int i = 1; i < nw; ++i) { lo = fmin(lo, slo[i]); hi = fmax(hi, shi[i]); em = fmax(em, sem[i]); }
    double tn = fmax(fabs(lo), fabs(hi));
    double pivmin = 1e-290 * fmax(1.0, em);
    lo -= 4.0 * kEps * tn + 2.0 * pivmin;
    hi += 4.0 * kEps * tn + 2.0 * pivmin;
    scal[0] = lo; scal[1] = hi; scal[2] = tn; scal[3] = pivmin;
  }
}

// Number of eigenvalues of T below x: sign changes of the leading principal
// minors p_j = (d_j - x) p_{j-1} - e_{j-1}^2 p_{j-2} (Sturm sequence), kept in
// range by exact power-of-two rescaling, so each step is two FMAs and no
// division.  An exact zero minor counts as negative (the pivmin convention).
__device__ __forceinline__ int sturm_count(int n, const double* __restrict__ d,
                                           const double* __restrict__ e2, double x, double) {
  // FP64 work per step is one multiply and one FMA; signs, zero tests and the
  // rescaling test read the bit pattern with integer instructions.
  double pm = 1.0;                    // p_{j-1}
  double p = d[0] - x;                // p_0
  long long b = __double_as_longlong(p);
  int sp = (b < 0 || (b & 0x7FFFFFFFFFFFFFFFLL) == 0) ? 1 : 0;   // 1: negative (zero counts as negative)
  int c = sp;
  for (int j = 1; j < n; ++j) {
    double pn = fma(d[j] - x, p, -e2[j - 1] * pm);
    pm = p;
    p = pn;
    b = __double_as_longlong(pn);
    int zero = (b & 0x7FFFFFFFFFFFFFFFLL) == 0;
    int sn = zero ? (sp ^ 1) : (int)((unsigned long long)b >> 63);
    c += sn ^ sp;
    sp = sn;
    int ex = (int)((b >> 52) & 0x7FF);             // biased exponent of p_j
    if (ex > 1023 + 400) {
      p *= 0x1p-400; pm *= 0x1p-400;
    } else if (ex < 1023 - 400 && (int)((__double_as_longlong(pm) >> 52) & 0x7FF) < 1023 - 400) {
      p *= 0x1p400; pm *= 0x1p400;
    }
  }
  return c;
}

// FP32 Sturm count (ratio form with a pivot floor) for the coarse phase
__device__ __forceinline__ int sturm_count_f32(int n, const float* __restrict__ d,
                                               const float* __restrict__ e2, float x, float pivmin) {
  float q = d[0] - x;
  if (fabsf(q) <= pivmin) q = -pivmin;
  int c = (q < 0.0f);
  for (int j = 1; j < n; ++j) {
    q = (d[j] - x) - e2[j - 1] / q;
    if (fabsf(q) <= pivmin) q = -pivmin;
    c += (q < 0.0f);
  }
  return c;
}

// FP64 path: eigenvalue i of T by multisection, M lanes a group: FP32 counts down to
// ~2^-22 of the Gershgorin interval, a round of FP64 counts that takes both ends in
// (and widens the bracket where the FP32 counts erred), then FP64 rounds.  A count is a
// chain of n FP64 steps on a pipe that takes ~62 cycles a warp
// instruction however many lanes are live, so lanes that count at other points of
// the same interval are free until there are more warps than FP64 pipes (kFp64Pipes);
// M = 32, 16, 8 up to 1, 1 and 2 warps a pipe, 8 beside other handles.  n = 240, 574,
// 1680: 334, 783, 3450 us; 1370, 3160, 9220 with one lane an eigenvalue.
// The FP64 counts are taken at points glo + k h of one grid, k an integer, and the
// eigenvalue is the middle of the cell whose ends have counts <= i and > i.  The cells (a
// 32nd of the tolerance, 3e-14 of the range) are ten times wider than the rounding of a count
// shifts an eigenvalue, so there is one such cell and every M, and every bracket to start from,
// ends in it: the same bits alone and beside other handles.  (Points that depended on M, down to
// the tolerance itself: 289, 669, 3030 us, and three times the error, 3e-14 of the range.)
constexpr int kFp64Pipes = 4 * 152;
template <int M>
__global__ void __launch_bounds__(32) bisect_kernel(int n, const double* __restrict__ d, const double* __restrict__ e2,
                                                  const double* __restrict__ scal, const float* __restrict__ df,
                                                  const float* __restrict__ e2f, double rel_tol,
                                                  double* __restrict__ ev) {
  const int t = blockIdx.x * 32 + threadIdx.x;
  const int i = t / M, m = t % M;             // eigenvalue of this group, point of the lane
  const int gbase = threadIdx.x & ~(M - 1);
  const unsigned gmask = (M == 32) ? 0xffffffffu : (1u << M) - 1u;
  const bool live = i < n;                    // whole groups are live or not
  const double glo = scal[0], ghi = scal[1], pivmin = scal[3];
  const double width = ghi - glo;
  // points of the group with a count above i, as bits
  auto above = [&](bool a) { return (__ballot_sync(0xffffffffu, a) >> gbase) & gmask; };
  float lo32 = (float)glo, hi32 = (float)ghi;
  const float piv32 = fmaxf((float)(1e-30 * fmax(1.0, width)), 1e-30f);
  for (float left = 0x1p22f; left > 1.0f; left /= (float)(M + 1)) {
    const float h32 = (hi32 - lo32) / (float)(M + 1);
    const unsigned g = above(live && sturm_count_f32(n, df, e2f, lo32 + (float)(m + 1) * h32, piv32) > i);
    const int f = g ? __ffs(g) - 1 : M;       // first point above, M: none
    const float nlo = (f == 0) ? lo32 : lo32 + (float)f * h32;
    hi32 = (f == M) ? hi32 : lo32 + (float)(f + 1) * h32;
    lo32 = nlo;
  }
  // rel_tol (1e-12) of the spectral range is far below what the occupations and
  // the DMPT weights resolve, and inverse iteration converges from such a shift
  // in two steps.  A looser shift costs orthogonality: after two steps the
  // component along a neighbour at distance g is ~(shift error / g)^2, which at
  // 1e-9 of the range left Q^T Q - I at 5e-7 for n = 3360.
  const double tol = fmax(2.0 * kEps * fmax(fabs(glo), fabs(ghi)), rel_tol * fmax(1.0, scal[2])) + pivmin;
  const double h = 0x1p-5 * tol;
  // cells of the grid (2^46 at most with rel_tol = 1e-12)
  const long long cells = max(1ll, (long long)fmin(ceil(width / h), 0x1p52));
  auto point = [&](long long k) { return fma((double)k, h, glo); };
  long long w = max(1ll, (long long)fmin(((double)hi32 - (double)lo32) / h, 0x1p52));
  long long lo = min(max((long long)(((double)lo32 - glo) / h) - w, 0ll), cells - 1);
  long long hi = min(max((long long)(((double)hi32 - glo) / h) + w + 1, lo + 1), cells);
  bool done = !live, ends = true;             // ends: the points of the round are 0 .. M - 1, both ends among them
  for (int it = 0; it < 260 && __any_sync(0xffffffffu, !done); ++it) {
    auto at = [&](int p) { return ends ? lo + (hi - lo) * p / (M - 1) : lo + (hi - lo) * (p + 1) / (M + 1); };
    const unsigned g = above(!done && sturm_count(n, d, e2, point(at(m)), pivmin) > i);
    if (done) continue;
    const int f = g ? __ffs(g) - 1 : M;       // first point above, M: none
    if (ends) {
      const bool low = f == 0 && lo > 0, high = f == M && hi < cells;
      if (low || high) {
        w *= 4;
        if (low) lo = max(0ll, lo - w);
        if (high) hi = min(cells, hi + w);
        continue;
      }
    }
    // (the ends of the Gershgorin interval count as below and above whatever the arithmetic says)
    const long long nlo = (f == 0) ? lo : at(f - 1);
    hi = (f == M) ? hi : max(at(f), lo + 1);
    lo = min(nlo, hi - 1);
    ends = false;
    done = hi - lo <= 1;
  }
  if (live && m == 0) ev[i] = fma((double)lo + 0.5, h, glo);
}

// Mixed path: eigenvalue i by multisection in double-float arithmetic.  A
// group of kMsLanes lanes evaluates the Sturm count at kMsLanes interior
// points of the current interval, which shrinks (kMsLanes + 1)-fold per round;
// every group starts from the Gershgorin interval, so all groups take the same
// number of rounds.  The count is the product form of sturm_count on the FP32
// pipe (about 48-bit arithmetic), kept in range by exact power-of-two scaling.
constexpr int kMsLanes = 8;

__device__ __forceinline__ int sturm_count_df(int n, const dfl* __restrict__ d, const dfl* __restrict__ e2,
                                              dfl x) {
  dfl pm = {1.0f, 0.0f};
  dfl p = df_sub(ldg_df(d), x);
  int sp = (p.hi < 0.0f || p.hi == 0.0f) ? 1 : 0;        // zero counts as negative
  int c = sp;
#pragma unroll 4
  for (int j = 1; j < n; ++j) {
    const dfl dj = ldg_df(d + j), ej = ldg_df(e2 + j - 1);
    const dfl pn = df_sub(df_mul(df_sub(dj, x), p), df_mul(ej, pm));
    const int sn = (pn.hi == 0.0f) ? (sp ^ 1) : (int)(__float_as_uint(pn.hi) >> 31);
    c += sn ^ sp;
    sp = sn;
    // keep |p| within [2^-32, 2^32] (both p and pm scale by the same power of two)
    const int ex = (int)((__float_as_uint(pn.hi) >> 23) & 0xFF);
    const float sc = (ex > 127 + 32) ? 0x1p-64f : ((ex < 127 - 32) ? 0x1p+64f : 1.0f);
    pm = dfl{KX_FMUL(p.hi, sc), KX_FMUL(p.lo, sc)};
    p = dfl{KX_FMUL(pn.hi, sc), KX_FMUL(pn.lo, sc)};
  }
  return c;
}

// Interval f of [lo, hi] cut by the kMsLanes points lo + (m + 1) h
__device__ __forceinline__ void ms_interval(double& lo, double& hi, double h, int f) {
  const double nlo = (f == 0) ? lo : lo + (double)f * h;
  hi = (f == kMsLanes) ? hi : lo + (double)(f + 1) * h;
  lo = nlo;
}

// WIDE: a block of kMsWide lanes per eigenvalue takes two rounds at once, lanes 0 .. 7 the
// first round's points and eight lanes for each of its nine intervals the second's: the
// same points and results, half the chains of n steps, two and a half times the work: n =
// 131, 240, 480, 720: 156 -> 107, 258 -> 185, 490 -> 405, 718 -> 729 us.
constexpr int kMsWideMax = 512;
constexpr int kMsWide = 96, kMsPoints = kMsLanes * (kMsLanes + 2);
template <bool WIDE>
__global__ void __launch_bounds__(WIDE ? kMsWide : 32) bisect_df_kernel(int n, const dfl* __restrict__ d,
                                                                       const dfl* __restrict__ e2,
                                                                       const double* __restrict__ scal,
                                                                       double rel_tol, double* __restrict__ ev) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = WIDE ? (int)blockIdx.x : t / kMsLanes;                 // eigenvalue of this group
  const int m = (WIDE ? (int)threadIdx.x : t) % kMsLanes;             // point m + 1 of the group
  const int sub = WIDE ? (int)threadIdx.x / kMsLanes - 1 : -1;        // interval of the round before (-1: none)
  const int gbase = (threadIdx.x & 31) & ~(kMsLanes - 1);
  const bool live = i < n;                    // whole groups are live or not (n * kMsLanes threads)
  const double glo = scal[0], ghi = scal[1], pivmin = scal[3];
  double lo = glo, hi = ghi;
  const double tol = fmax(2.0 * kEps * fmax(fabs(glo), fabs(ghi)), rel_tol * fmax(1.0, scal[2])) + pivmin;
  int rounds = 0;
  for (double w = ghi - glo; w > tol && rounds < 64; w /= (double)(kMsLanes + 1)) ++rounds;
  __shared__ unsigned s_above[2][kMsWide / 32];
  constexpr unsigned kMask = (1u << kMsLanes) - 1u;
  // counts grow with x: the first point with count > i is the new upper end
  auto first = [](unsigned g) { return g ? (__ffs(g) - 1) : kMsLanes; };   // 0-based point index, kMsLanes: none
  for (int r = 0; r < rounds; r += WIDE ? 2 : 1) {
    double l = lo, u = hi, h = (hi - lo) / (double)(kMsLanes + 1);
    if (sub >= 0) {
      ms_interval(l, u, h, sub);
      h = (u - l) / (double)(kMsLanes + 1);
    }
    const double x = l + (double)(m + 1) * h;
    const bool idle = WIDE && ((int)threadIdx.x >= kMsPoints || (sub >= 0 && r + 1 >= rounds));
    const bool above = live && !idle && sturm_count_df(n, d, e2, df_from_double(x)) > i;
    const unsigned bal = __ballot_sync(0xffffffffu, above);
    if constexpr (WIDE) {
      unsigned* w = s_above[(r >> 1) & 1];                             // (the other one was read before the barrier)
      if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = bal;
      __syncthreads();
      const int f0 = first(w[0] & kMask);
      ms_interval(lo, hi, (hi - lo) / (double)(kMsLanes + 1), f0);
      if (r + 1 < rounds) {
        const int at = kMsLanes * (f0 + 1);
        ms_interval(lo, hi, (hi - lo) / (double)(kMsLanes + 1), first(w[at >> 5] >> (at & 31) & kMask));
      }
    } else {
      ms_interval(lo, hi, h, first((bal >> gbase) & kMask));
    }
  }
  if (live && (WIDE ? threadIdx.x == 0 : m == 0)) ev[i] = 0.5 * (lo + hi);
}

__global__ void cluster_kernel(int n, const double* __restrict__ ev, const double* __restrict__ scal,
                               int* __restrict__ clus) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double ctol = 1e-7 * fmax(1.0, scal[2]);
  // a NaN gap starts a new cluster: non-finite input must not merge the whole
  // spectrum into one cluster (one block would then orthogonalise n vectors)
  clus[i] = (i == 0 || !(ev[i] - ev[i - 1] <= ctol)) ? 1 : 0;
}

__device__ __forceinline__ unsigned start_hash(int row, int col) {
  unsigned h = (unsigned)row * 0x9E3779B1u ^ ((unsigned)col * 0x85EBCA77u + 0x165667B1u);
  h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
  return h;
}
__device__ __forceinline__ double start_value(int row, int col) {
  return ((double)(start_hash(row, col) & 0xFFFFF) / 524288.0) - 1.0 + 1e-3;
}
// the same pseudo-random start entry in FP32 arithmetic (a start vector only
// needs a component along the eigenvector, not FP64 values)
__device__ __forceinline__ float start_value_f(int row, int col) {
  return __fadd_rn(__fmul_rn((float)(start_hash(row, col) & 0xFFFFF), 0x1p-19f), -0.999f);
}

// Arithmetic of the inverse iteration: FP64, or double-float (FP32 pairs, df.cuh) in
// the mixed path.  unit(): the shift separation and pivot floor in units of |T|.
template <class R>
struct IvOps;
template <>
struct IvOps<double> {
  static constexpr double kUnit = kEps;
  __device__ static __forceinline__ double from(double x) { return x; }
  __device__ static __forceinline__ double load(const double* p) { return __ldg(p); }
  __device__ static __forceinline__ double sub(double a, double b) { return a - b; }
  __device__ static __forceinline__ double mul(double a, double b) { return a * b; }
  __device__ static __forceinline__ double neg(double a) { return -a; }
  __device__ static __forceinline__ double recip(double a) { return 1.0 / a; }
  __device__ static __forceinline__ double mag(double a) { return fabs(a); }
  __device__ static __forceinline__ bool minus(double a) { return !(a >= 0.0); }
  __device__ static __forceinline__ double start(int r, int c) { return start_value(r, c); }
  __device__ static __forceinline__ double max(double a, double b) { return fmax(a, b); }
  __device__ static __forceinline__ double widen(double m) { return m; }
  __device__ static __forceinline__ void add_sq(double& s, double x) { s = fma(x, x, s); }
  __device__ static __forceinline__ double sum(double s) { return s; }
  __device__ static __forceinline__ double out(double x) { return x; }
};
template <>
struct IvOps<dfl> {
  static constexpr double kUnit = 0x1p-46;
  __device__ static __forceinline__ dfl from(double x) { return df_from_double(x); }
  __device__ static __forceinline__ dfl load(const dfl* p) {
    const float2 v = __ldg((const float2*)p);
    return dfl{v.x, v.y};
  }
  __device__ static __forceinline__ dfl sub(dfl a, dfl b) { return df_sub(a, b); }
  __device__ static __forceinline__ dfl mul(dfl a, dfl b) { return df_mul(a, b); }
  __device__ static __forceinline__ dfl neg(dfl a) { return df_neg(a); }
  __device__ static __forceinline__ dfl recip(dfl a) { return df_recip(a); }
  __device__ static __forceinline__ float mag(dfl a) { return fabsf(a.hi); }
  __device__ static __forceinline__ bool minus(dfl a) { return !(a.hi >= 0.0f); }
  __device__ static __forceinline__ dfl start(int r, int c) { return dfl{start_value_f(r, c), 0.0f}; }
  __device__ static __forceinline__ float max(float a, float b) { return fmaxf(a, b); }
  __device__ static __forceinline__ dfl widen(float m) { return dfl{m, 0.0f}; }
  __device__ static __forceinline__ void add_sq(dfl& s, dfl x) { df_acc_mul(s, x, x); }
  __device__ static __forceinline__ double sum(dfl s) { return df_to_double(df_norm(s)); }
  __device__ static __forceinline__ double out(dfl x) { return df_to_double_fast(x); }
};

// Eigenvectors of T by two steps of inverse iteration, a thread per eigenvalue; lu:
// 5 x n x n workspace.  What bounds it is the latency of the recurrences (n rows, six
// sweeps), so
//  * the sweeps carry their running values in registers and issue the loads of kIvB
//    rows ahead of the dependent arithmetic;
//  * the steps are fused: step 1 solves from the start vector without storing it, its
//    backward sweep tracks max|x|; step 2 reads x scaled by 1/max (inverse iteration is
//    linear, the scale only keeps the values in range), its backward sweep accumulates
//    ||x||^2; a last pass writes x / ||x|| in FP64;
//  * few lanes of a warp are used (kIvLanes: whole 32-byte sectors, little divergence
//    at the pivots), so that the chains spread over all SMs;
//  * members of a cluster (gaps below 1e-7 of the width) are solved like all others,
//    each from its own start vector, and made orthogonal afterwards
//    (orth_cluster_kernel): one thread doing a cluster in turn was most of the time
//    wherever there was one.  n = 1680 and 3360 (7 and 14 cages):
//    4.4 -> 2.0 and 22.6 -> 5.0 ms; FP64, which had fifteen sweeps, 574 and 1680:
//    1.42 -> 0.86 and 5.8 -> 2.8 ms.
// Shifts closer than ten units to the one before are moved up to that distance.
constexpr int kIvB = 8;
constexpr int kIvLanes = 4;
template <class R>
__global__ void __launch_bounds__(32) invit_kernel(int n, int lanes, const R* __restrict__ d, const R* __restrict__ e,
                                                 const double* __restrict__ ev, const double* __restrict__ scal,
                                                 const int* __restrict__ clus, R* __restrict__ lu,
                                                 double* __restrict__ Zout) {
  using O = IvOps<R>;
  if (threadIdx.x >= lanes) return;
  const int L = blockIdx.x * lanes + threadIdx.x;
  if (L >= n) return;
  if (n == 1) {
    Zout[0] = 1.0;
    return;
  }
  const double tiny_d = O::kUnit * fmax(scal[2], 1e-300);
  const R tiny = O::from(tiny_d);
  const size_t nn = (size_t)n * n;
  R* __restrict__ dl = lu + 0 * nn;
  R* __restrict__ rdd = lu + 1 * nn;   // reciprocal pivots
  R* __restrict__ du = lu + 2 * nn;
  R* __restrict__ du2 = lu + 3 * nn;
  int* __restrict__ pv = (int*)(lu + 4 * nn);
  R* __restrict__ Z = (R*)Zout;        // iterates in place of the FP64 output
#define LU(a, r) a[(size_t)(r) * n + L]
#define ZC(r) Z[(size_t)(r) * n + L]
  double shift = ev[L];
  if (!clus[L]) {
    int j = L;
    while (!clus[j]) --j;
    shift = ev[j];
    for (++j; j <= L; ++j) shift = (ev[j] - shift < 10.0 * tiny_d) ? shift + 10.0 * tiny_d : ev[j];
  }
  // LU of T - lam I with partial pivoting; a, u: pivot-row diagonal and superdiagonal.
  // No FP64 instruction per row in the mixed path: GB300 issues one FP64 warp
  // instruction per ~76 cycles per scheduler, which would put the FP64 pipe on the chain.
  const R lam = O::from(shift);
  R a = O::sub(O::load(d), lam), u = O::load(e);
  for (int r = 0; r < n - 1; ++r) {
    const R b = O::load(e + r);
    const R dn = O::sub(O::load(d + r + 1), lam);
    const R un = (r < n - 2) ? O::load(e + r + 1) : R{};
    if (O::mag(a) >= O::mag(b)) {
      LU(pv, r) = 0;
      if (O::mag(a) < O::mag(tiny)) a = O::minus(a) ? O::neg(tiny) : tiny;
      const R ra = O::recip(a);
      const R f = O::mul(b, ra);
      LU(dl, r) = f;
      LU(rdd, r) = ra;
      LU(du, r) = u;
      LU(du2, r) = R{};
      a = O::sub(dn, O::mul(f, u));
      u = un;
    } else {
      LU(pv, r) = 1;
      const R rb = O::recip(b);
      const R f = O::mul(a, rb);
      LU(rdd, r) = rb;
      LU(dl, r) = f;
      LU(du, r) = dn;
      const R na = O::sub(u, O::mul(f, dn));
      if (r < n - 2) {
        LU(du2, r) = un;
        u = O::neg(O::mul(f, un));
      } else {
        LU(du2, r) = R{};
      }
      a = na;
    }
  }
  if (O::mag(a) < O::mag(tiny)) a = O::minus(a) ? O::neg(tiny) : tiny;
  LU(rdd, n - 1) = O::recip(a);
  R scl = O::from(1.0);
  R nrm = R{};
  for (int it = 0; it < 2; ++it) {
    // forward (L with pivots); step 1 takes the start vector, step 2 the scaled x
    R cur = (it == 0) ? O::start(0, L) : O::mul(ZC(0), scl);
    for (int r0 = 0; r0 < n - 1; r0 += kIvB) {
      R nx[kIvB], fv[kIvB];
      int pf[kIvB];
#pragma unroll
      for (int q = 0; q < kIvB; ++q) {
        const int r = r0 + q;
        if (r < n - 1) {
          nx[q] = (it == 0) ? O::start(r + 1, L) : O::mul(ZC(r + 1), scl);
          fv[q] = LU(dl, r);
          pf[q] = LU(pv, r);
        }
      }
#pragma unroll
      for (int q = 0; q < kIvB; ++q) {
        const int r = r0 + q;
        if (r < n - 1) {
          if (pf[q] == 0) {
            ZC(r) = cur;
            cur = O::sub(nx[q], O::mul(fv[q], cur));
          } else {
            ZC(r) = nx[q];
            cur = O::sub(cur, O::mul(fv[q], nx[q]));
          }
        }
      }
    }
    // backward (U, three diagonals, reciprocal pivots), with max|x| or ||x||^2;
    // z1 = x[r + 1], z2 = x[r + 2]
    R z2 = O::mul(cur, LU(rdd, n - 1));
    ZC(n - 1) = z2;
    auto mx = O::mag(z2);
    if (it == 1) O::add_sq(nrm, z2);
    R z1 = O::mul(O::sub(ZC(n - 2), O::mul(LU(du, n - 2), z2)), LU(rdd, n - 2));
    ZC(n - 2) = z1;
    mx = O::max(mx, O::mag(z1));
    if (it == 1) O::add_sq(nrm, z1);
    for (int r0 = n - 3; r0 >= 0; r0 -= kIvB) {
      R zv[kIvB], uv[kIvB], u2[kIvB], rv[kIvB];
#pragma unroll
      for (int q = 0; q < kIvB; ++q) {
        const int r = r0 - q;
        if (r >= 0) { zv[q] = ZC(r); uv[q] = LU(du, r); u2[q] = LU(du2, r); rv[q] = LU(rdd, r); }
      }
#pragma unroll
      for (int q = 0; q < kIvB; ++q) {
        const int r = r0 - q;
        if (r >= 0) {
          const R x = O::mul(O::sub(O::sub(zv[q], O::mul(uv[q], z1)), O::mul(u2[q], z2)), rv[q]);
          ZC(r) = x;
          mx = O::max(mx, O::mag(x));
          if (it == 1) O::add_sq(nrm, x);
          z2 = z1;
          z1 = x;
        }
      }
    }
    if (it == 0) scl = (mx > 0) ? O::recip(O::widen(mx)) : O::from(1.0);
  }
  const double nd = ::sqrt(O::sum(nrm));
  const R sc = (nd > 0.0) ? O::from(1.0 / nd) : R{};
#pragma unroll 8
  for (int r = 0; r < n; ++r) Zout[(size_t)r * n + L] = O::out(O::mul(ZC(r), sc));
#undef LU
#undef ZC
}

// Gram-Schmidt within the clusters, a block per cluster (blocks of other columns
// return): every vector against the ones before it, kOrthTile at a time, twice (what
// the first pass leaves of nearly parallel vectors the second removes), then normalised.
// The columns of a cluster are neighbours, so a row's values share sectors.
constexpr int kOrthThreads = 256, kOrthTile = 32;
__global__ void __launch_bounds__(kOrthThreads) orth_cluster_kernel(int n, const int* __restrict__ clus,
                                                                  double* __restrict__ Z) {
  const int L = blockIdx.x;
  if (!clus[L] || L + 1 >= n || clus[L + 1]) return;
  int end = L + 2;
  while (end < n && !clus[end]) ++end;
  __shared__ double coef[kOrthTile];
  __shared__ double part[kOrthThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int j = L; j < end; ++j) {
    for (int pass = 0; pass < 2; ++pass)
      for (int c0 = L; c0 < j; c0 += kOrthTile) {
        const int nc = min(kOrthTile, j - c0);
        for (int c = wid; c < nc; c += kOrthThreads / 32) {
          double s = 0.0;
          for (int r = lane; r < n; r += 32) s = fma(Z[(size_t)r * n + c0 + c], Z[(size_t)r * n + j], s);
          s = warp_sum(s);
          if (lane == 0) coef[c] = s;
        }
        __syncthreads();
        for (int r = tid; r < n; r += kOrthThreads) {
          double z = Z[(size_t)r * n + j];
          for (int c = 0; c < nc; ++c) z = fma(-coef[c], Z[(size_t)r * n + c0 + c], z);
          Z[(size_t)r * n + j] = z;
        }
        __syncthreads();
      }
    double s = 0.0;
    for (int r = tid; r < n; r += kOrthThreads) s = fma(Z[(size_t)r * n + j], Z[(size_t)r * n + j], s);
    s = warp_sum(s);
    if (lane == 0) part[wid] = s;
    __syncthreads();
    s = 0.0;
    for (int w = 0; w < kOrthThreads / 32; ++w) s += part[w];
    s = (s > 0.0) ? 1.0 / ::sqrt(s) : 0.0;
    for (int r = tid; r < n; r += kOrthThreads) Z[(size_t)r * n + j] *= s;
    __syncthreads();
  }
}

// T factor of a block of kb reflectors (forward, columnwise): one block,
// T held in shared memory, each entry a dot product split over 4 partial sums
__device__ void tfactor_body(int kb, const double* __restrict__ tau, const double* __restrict__ G, int ldg,
                             double* __restrict__ T, int ldt) {
  extern __shared__ double ts[];          // kb x kb
  __shared__ double gcol[kBtBlockTc];
  const int i = threadIdx.x;
  for (int e = i; e < kb * kb; e += blockDim.x) ts[e] = 0.0;
  __syncthreads();
  for (int j = 0; j < kb; ++j) {
    if (i < j) gcol[i] = G[i * ldg + j];
    __syncthreads();
    if (i < j) {
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
      int l = i;
      for (; l + 3 < j; l += 4) {
        a0 = fma(ts[i * kb + l], gcol[l], a0);
        a1 = fma(ts[i * kb + l + 1], gcol[l + 1], a1);
        a2 = fma(ts[i * kb + l + 2], gcol[l + 2], a2);
        a3 = fma(ts[i * kb + l + 3], gcol[l + 3], a3);
      }
      for (; l < j; ++l) a0 = fma(ts[i * kb + l], gcol[l], a0);
      ts[i * kb + j] = -tau[j] * ((a0 + a1) + (a2 + a3));
    }
    if (i == j) ts[j * kb + j] = tau[j];
    __syncthreads();
  }
  for (int e = i; e < kb * kb; e += blockDim.x) T[(e / kb) * ldt + e % kb] = ts[e];
}

__global__ void tfactor_kernel(int kb, const double* __restrict__ tau, const double* __restrict__ G,
                               int ldg, double* __restrict__ T, int ldt) {
  tfactor_body(kb, tau, G, ldg, T, ldt);
}

// T factors of every block of kBtBlockTc reflectors at once (block b: reflectors
// b kBtBlockTc ..; they depend on the reflectors only, not on the vectors updated).
// Row i of T is a recurrence of its own, T_ij = -tau_j sum_l T_il G_lj, a chain of FP64
// operations: four lanes a row take one of tfactor_body's four partial sums each (the
// same sums in the same order), and kTfRows rows a CTA spread the rows over the SMs,
// one warp per FP64 pipe.  Blocks of 128: 520 us with one thread
// a row on one SM, 185 now.
constexpr int kTfRows = 32;
constexpr int kTfLd = kBtBlockTc + 3;     // rows of T: the eight of a warp in different banks
constexpr int kTfSmem = (kBtBlockTc * (kBtBlockTc + 1) + kTfRows * kTfLd + kBtBlockTc) * (int)sizeof(double);
__global__ void __launch_bounds__(4 * kTfRows) tfactor_all_kernel(int nref, const double* __restrict__ tau,
                                                                const double* __restrict__ Gall,
                                                                double* __restrict__ Tall) {
  constexpr int KB = kBtBlockTc;
  extern __shared__ double ts[];
  double* gt = ts;                        // column j of G at gt + j (KB + 1)
  double* trow = gt + KB * (KB + 1);
  double* tj = trow + kTfRows * kTfLd;
  const int k0 = blockIdx.y * KB, kb = min(KB, nref - k0), i0 = blockIdx.x * kTfRows;
  if (i0 >= kb) return;
  const double* G = Gall + (size_t)blockIdx.y * KB * KB;
  for (int e = threadIdx.x; e < KB * KB; e += blockDim.x) {
    const int l = e / KB, j = e % KB;
    if (l < j && j < kb) gt[j * (KB + 1) + l] = G[e];
  }
  for (int j = threadIdx.x; j < kb; j += blockDim.x) tj[j] = tau[k0 + j];
  __syncthreads();
  const int i = i0 + (threadIdx.x >> 2), q = threadIdx.x & 3;
  double* t = trow + (threadIdx.x >> 2) * kTfLd;
  for (int j = i0; j < kb; ++j) {
    const double* g = gt + j * (KB + 1);
    double a = 0.0;
    int l = i;
    for (; l + 3 < j; l += 4) a = fma(t[l + q], g[l + q], a);
    if (q == 0)
      for (; l < j; ++l) a = fma(t[l], g[l], a);
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    if (q == 0) t[j] = (j > i) ? -tj[j] * a : (j == i ? tj[j] : 0.0);
    __syncwarp();
  }
  __syncthreads();
  double* T = Tall + (size_t)blockIdx.y * KB * KB;
  for (int e = threadIdx.x; e < kTfRows * kb; e += blockDim.x) {
    const int r = e / kb, j = e % kb;
    if (i0 + r < kb) T[(size_t)(i0 + r) * KB + j] = (j < i0) ? 0.0 : trow[r * kTfLd + j];
  }
}

// number of blocks of kBtBlockTc reflectors (n - 2 reflectors)
static int tc_blocks(int n) { return n > 2 ? (n - 2 + kBtBlockTc - 1) / kBtBlockTc : 1; }

// Back-transformation scratch in two parts: `early` is filled by the preparation, which may run
// beside the inverse iteration, `late` is used after it
struct BtBytes {
  size_t early, late;
};
static BtBytes bt_bytes(int n);      // slices (mixed path)
static BtBytes bt64_bytes(int n);    // digits (FP64)
// Up to this size the half of the back-transformation that needs no eigenvectors (Gram
// matrices, T factors, T^T V, slices) runs on the side stream during multisection and
// inverse iteration, which leave most SMs idle there: C60 step 2.90 -> 2.64 ms, C120 4.84 ->
// 4.57, 574 basis functions in FP64 9.82 -> 9.58.  At 1680 the kernels slow one another by more
// than is gained in the mixed path (23.32 -> 23.55 ms); between, 720 to 1440, there would be 2 to
// 4 % (FP64 0.4 to 2.6 %) for the memory of a scratch of its own.
constexpr int kBtSideMax = 640;
static bool bt_splits(int n) { return n > 2 && n <= kBtSideMax; }

// One layout for sizing and binding.  Every buffer starts on a 256-byte
// boundary: the back-transformation cuts BF16 slices into the lu region and
// hands them to TMA, whose tensor maps need 16-byte aligned bases (with odd n
// an unpadded layout would leave the region 8 bytes off).
// The inverse-iteration workspace (5 n^2) also holds what the later stages need: `late`, the third
// FP64 operand (tc_gemm64.cu) and, unless the preparation runs beside the inverse iteration
// (side), `early` and the first two.  FP64 at n = 1680: 1182 MB a handle, 1284 with buffers of their own.
static size_t eig_layout(int n, EigProducts kind, bool side, void* base, EigWork* w) {
  const size_t nn = (size_t)n * n;
  side = side && bt_splits(n) && kind != kEigPlain;
  const BtBytes bt = (kind == kEigSlices) ? bt_bytes(n) : (kind == kEigDigits) ? bt64_bytes(n) : BtBytes{0, 0};
  const size_t op = (kind == kEigDigits) ? tc64_op_bytes(n, n) : 0;
  const size_t early = bt.early + 2 * op, late = bt.late + op;
  const size_t lu_bytes = std::max(5 * nn * sizeof(double), late + (side ? 0 : early));
  size_t off = 0;
  auto take = [&](size_t doubles) {
    double* q = base ? (double*)base + off : nullptr;
    off += (doubles + 31) & ~(size_t)31;
    return q;
  };
  double* A = take(nn);
  double* Vst = take(nn);
  double* d = take(n);
  double* e = take(n);
  double* e2 = take(n);
  double* tau = take(n);
  double* pbuf = take(4 * (size_t)n);
  double* lu = take((lu_bytes + 7) / 8);
  char* pre = side ? (char*)take((early + 7) / 8) : (char*)lu + (base ? late : 0);
  double* Tm = take((size_t)tc_blocks(n) * kBtBlockTc * kBtBlockTc);   // T and Gram of every reflector block
  double* Gm = take((size_t)tc_blocks(n) * kBtBlockTc * kBtBlockTc);
  double* Wt = take((size_t)kBtBlockTc * n);
  double* Wt2 = take((size_t)kBtBlockTc * n);
  double* scal = take(16);
  double* bar = take(8);
  double* clus = take(((size_t)n * sizeof(int) + 7) / 8);
  if (w) {
    w->A = A; w->Vst = Vst; w->d = d; w->e = e; w->e2 = e2; w->tau = tau; w->pbuf = pbuf; w->lu = lu;
    w->side = side;
    w->early = pre + 2 * op;
    w->late = (char*)lu + op;
    w->op64[0] = pre;
    w->op64[1] = pre + op;
    w->op64[2] = (char*)lu;
    w->Tm = Tm; w->Gm = Gm; w->Wt = Wt; w->Wt2 = Wt2; w->scal = scal;
    w->bar = (unsigned*)bar;
    w->clus = (int*)clus;
  }
  return off * sizeof(double) + 256;
}

size_t eig_work_bytes(int n, EigProducts kind, bool side) { return eig_layout(n, kind, side, nullptr, nullptr); }

// base must be 256-byte aligned (arena allocations are)
void eig_work_bind(EigWork& w, void* base, int n, EigProducts kind, bool side) { eig_layout(n, kind, side, base, &w); }

void eig_bisect(cudaStream_t s, int n, double* eps, EigWork& w, double rel_tol, bool df_path, bool shared) {
  if (n <= 0) return;
  // 2. eigenvalues
  // pbuf (4n doubles, free after the tridiagonalisation) holds the FP32 and double-float copies
  float* df = (float*)w.pbuf;
  float* e2f = df + n;
  dfl* d_dfl = (dfl*)(w.pbuf + n);
  dfl* e2_dfl = d_dfl + n;
  dfl* e_dfl = e2_dfl + n;
  gersh_kernel<<<1, 1024, 0, s>>>(n, w.d, w.e, w.e2, w.scal, df, e2f, d_dfl, e2_dfl, e_dfl);
  count_launch();
  if (df_path) {
    // one warp (4 eigenvalues) per block, so the n / 4 blocks spread over all SMs
    if (n <= kMsWideMax && !shared)
      bisect_df_kernel<true><<<n, kMsWide, 0, s>>>(n, d_dfl, e2_dfl, w.scal, rel_tol, eps);
    else
      bisect_df_kernel<false><<<(unsigned)(((long long)n * kMsLanes + 31) / 32), 32, 0, s>>>(n, d_dfl, e2_dfl, w.scal,
                                                                                           rel_tol, eps);
  } else {
    auto run = [&](auto kernel, int m) {
      kernel<<<(unsigned)(((long long)n * m + 31) / 32), 32, 0, s>>>(n, w.d, w.e2, w.scal, df, e2f, rel_tol, eps);
    };
    if (n <= kFp64Pipes && !shared)
      run(bisect_kernel<32>, 32);
    else if (n <= 2 * kFp64Pipes && !shared)
      run(bisect_kernel<16>, 16);
    else if (n <= 8 * kFp64Pipes)
      run(bisect_kernel<8>, 8);
    else
      run(bisect_kernel<4>, 4);
  }
  count_launch();
}

void eig_vectors(cudaStream_t s, int n, const double* eps, double* Q, EigWork& w, bool df_path, bool shared) {
  if (n <= 0) return;
  // 3. eigenvectors of the tridiagonal matrix
  cluster_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, eps, w.scal, w.clus);
  count_launch();
  if (df_path) {
    const dfl* d_dfl = (const dfl*)(w.pbuf + n);     // written by eig_bisect
    const dfl* e_dfl = d_dfl + 2 * (size_t)n;
    invit_kernel<dfl><<<(n + kIvLanes - 1) / kIvLanes, 32, 0, s>>>(n, kIvLanes, d_dfl, e_dfl, eps, w.scal, w.clus,
                                                                  (dfl*)w.lu, Q);
  } else {
    // (not more warps than there are FP64 pipes, which a partly filled warp holds as long as a full one)
    int lanes = shared ? 2 * kIvLanes : kIvLanes;
    while (lanes < 32 && n > lanes * kFp64Pipes) lanes *= 2;
    invit_kernel<double><<<(n + lanes - 1) / lanes, 32, 0, s>>>(n, lanes, w.d, w.e, eps, w.scal, w.clus, w.lu, Q);
  }
  count_launch();
  if (n > 1) {
    orth_cluster_kernel<<<n, kOrthThreads, 0, s>>>(n, w.clus, Q);
    count_launch();
  }
}

// tensor-core back-transformation (mixed path), carried out on Z^T so that
// every large operand is K-major: Z^T <- Z^T (I - V T V^T)^T block by block,
//   U   = Z^T_sub V_b^T     (n x kb)      tensor cores, 4 slices, split over K
//   Z^T_sub -= U Y_b        (n x m_b)     tensor cores, 4 slices
// with Y_b = T_b^T V_b formed for all blocks before the loop (it does not
// depend on Z).  The Gram matrices V_b V_b^T (for the T factors) and Y_b are
// double-float products on the FP32 pipe, one launch each for all blocks; the
// slices of V_b and Y_b^T are cut once, in two launches.
__global__ void transpose_sq_kernel(int n, const double* __restrict__ A, double* __restrict__ At) {
  __shared__ double tile[32][33];
  int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    int i = i0 + r, j = j0 + threadIdx.x;
    tile[r][threadIdx.x] = (i < n && j < n) ? A[(size_t)i * n + j] : 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    int j = j0 + r, i = i0 + threadIdx.x;
    if (i < n && j < n) At[(size_t)j * n + i] = tile[threadIdx.x][r];
  }
}

static void transpose_sq(cudaStream_t s, int n, const double* A, double* At) {
  int t = (n + 31) / 32;
  transpose_sq_kernel<<<dim3(t, t), dim3(32, 8), 0, s>>>(n, A, At);
  count_launch();
}

// G_b = V_b V_b^T (upper 32 x 32 tiles) for every block b of kBtBlockTc
// reflectors; V_b = rows k0.. of the reflector store, columns c0 = k0 + 1 ..
__global__ void __launch_bounds__(256) gram_df_kernel(int n, int nref, const double* __restrict__ Vst,
                                                      double* __restrict__ Gall) {
  constexpr int KB = kBtBlockTc, TL = 32, CH = 64;
  const int b = blockIdx.y;
  const int k0 = b * KB, kb = min(KB, nref - k0), c0 = k0 + 1, m = n - c0;
  const int ti = blockIdx.x / (KB / TL), tj = blockIdx.x % (KB / TL);
  if (ti > tj || ti * TL >= kb || tj * TL >= kb) return;
  __shared__ dfl sa[TL][CH + 1], sb[TL][CH + 1];
  const int t = threadIdx.x, ii = t >> 3, jj = (t & 7) * 4;
  dfl acc[4] = {};
  for (int l0 = 0; l0 < m; l0 += CH) {
    for (int e = t; e < TL * CH; e += blockDim.x) {
      const int r = e / CH, c = e % CH;
      const int l = l0 + c;
      const int ra = ti * TL + r, rb = tj * TL + r;
      sa[r][c] = (ra < kb && l < m) ? df_from_double_exact(Vst[(size_t)(k0 + ra) * n + c0 + l]) : dfl{0.0f, 0.0f};
      sb[r][c] = (rb < kb && l < m) ? df_from_double_exact(Vst[(size_t)(k0 + rb) * n + c0 + l]) : dfl{0.0f, 0.0f};
    }
    __syncthreads();
#pragma unroll 4
    for (int c = 0; c < CH; ++c) {
      const dfl a = sa[ii][c];
#pragma unroll
      for (int q = 0; q < 4; ++q) df_acc_mul(acc[q], a, sb[jj + q][c]);
    }
    __syncthreads();
  }
  const int i = ti * TL + ii;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = tj * TL + jj + q;
    if (i < kb && j < kb) Gall[(size_t)b * KB * KB + (size_t)i * KB + j] = df_to_double_fast(df_norm(acc[q]));
  }
}

// Y_b^T = V_b^T T_b (m_b x kb, row length KB) for every block b; T_b upper
// triangular (kb x kb, ld KB); ROWS rows of Y_b^T per CTA, T_b and the V_b
// columns in shared memory as double-float.  64 rows read T_b least often; 16 where
// that would leave SMs idle (n = 240: 8 CTAs, 167 us).
constexpr size_t y_smem(int rows) { return (size_t)(kBtBlockTc * kBtBlockTc + kBtBlockTc * rows) * sizeof(dfl); }
template <int ROWS>
__global__ void __launch_bounds__(256) y_df_kernel(int n, int nref, const double* __restrict__ Vst,
                                                   const double* __restrict__ Tall, double* __restrict__ YT) {
  constexpr int KB = kBtBlockTc;
  extern __shared__ dfl ysm[];
  dfl* sT = ysm;                   // KB x KB
  dfl* sV = ysm + KB * KB;         // KB (reflector) x ROWS (column)
  const int b = blockIdx.y;
  const int k0 = b * KB, kb = min(KB, nref - k0), c0 = k0 + 1, m = n - c0;
  const int l0 = blockIdx.x * ROWS;
  if (l0 >= m) return;
  const double* Tb = Tall + (size_t)b * KB * KB;
  for (int e = threadIdx.x; e < KB * KB; e += blockDim.x) {
    const int i = e / KB, j = e % KB;
    sT[e] = (i < kb && j < kb && i <= j) ? df_from_double_exact(Tb[(size_t)i * KB + j]) : dfl{0.0f, 0.0f};
  }
  for (int e = threadIdx.x; e < KB * ROWS; e += blockDim.x) {
    const int i = e / ROWS, c = e % ROWS;
    const int l = l0 + c;
    sV[e] = (i < kb && l < m) ? df_from_double_exact(Vst[(size_t)(k0 + i) * n + c0 + l]) : dfl{0.0f, 0.0f};
  }
  __syncthreads();
  // thread t: row c of the tile, COLS consecutive columns
  constexpr int COLS = KB * ROWS / 256;
  const int c = threadIdx.x / (KB / COLS), jb = threadIdx.x % (KB / COLS) * COLS;
  dfl acc[COLS];
#pragma unroll
  for (int q = 0; q < COLS; ++q) acc[q] = dfl{0.0f, 0.0f};
  for (int i = 0; i < kb; ++i) {
    const dfl v = sV[i * ROWS + c];
#pragma unroll
    for (int q = 0; q < COLS; ++q) df_acc_mul(acc[q], v, sT[i * KB + jb + q]);
  }
  const int l = l0 + c;
  if (l < m) {
    double* out = YT + (size_t)b * n * KB + (size_t)l * KB;
#pragma unroll
    for (int q = 0; q < COLS; ++q) out[jb + q] = (jb + q < kb) ? df_to_double_fast(df_norm(acc[q])) : 0.0;
  }
}

static int bt_blocks(int n) { return n > 2 ? (n - 2 + kBtBlockTc - 1) / kBtBlockTc : 0; }
constexpr int kBtSplitK = 6;
struct BtScratch {
  __nv_bfloat16* vs;   size_t vs_blk, vs_slice;   // V_b slices
  double* yt;                                     // Y_b^T, FP64
  __nv_bfloat16* ys;   size_t ys_blk, ys_slice;   // Y_b^T slices
  double* part;                                   // split-K partial products of U
};
static BtBytes bt_scratch_layout(int n, const EigWork* w, BtScratch* out) {
  const size_t nblk = (size_t)bt_blocks(n), KB = kBtBlockTc;
  const size_t ldn = (size_t)tc_ld(n > 1 ? n : 1);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  const size_t vs_slice = KB * ldn, vs_blk = (size_t)kTcMaxSlices * vs_slice;
  const size_t o_vs = take(nblk * vs_blk * 2);
  const size_t o_yt = take(nblk * (size_t)n * KB * 8);
  const size_t ys_slice = (size_t)n * KB, ys_blk = (size_t)kTcMaxSlices * ys_slice;
  const size_t o_ys = take(nblk * ys_blk * 2);
  if (out) {
    char* c = w->early;
    out->vs = (__nv_bfloat16*)(c + o_vs); out->vs_blk = vs_blk; out->vs_slice = vs_slice;
    out->yt = (double*)(c + o_yt);
    out->ys = (__nv_bfloat16*)(c + o_ys); out->ys_blk = ys_blk; out->ys_slice = ys_slice;
    out->part = (double*)w->late;
  }
  return BtBytes{off, (size_t)(kBtSplitK + 1) * n * KB * 8};
}
static BtBytes bt_bytes(int n) { return bt_scratch_layout(n, nullptr, nullptr); }

static void bt_attributes() {
  static PerDeviceOnce attr;
  once_per_device(attr, [] {
    return cudaFuncSetAttribute(tfactor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kBtBlockTc * kBtBlockTc * (int)sizeof(double)) == cudaSuccess &&
           cudaFuncSetAttribute(tfactor_all_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTfSmem) ==
               cudaSuccess &&
           cudaFuncSetAttribute(y_df_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)y_smem(64)) ==
               cudaSuccess &&
           cudaFuncSetAttribute(y_df_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)y_smem(16)) ==
               cudaSuccess;
  });
}

static void bt_prepare_tc(cudaStream_t s, int n, EigWork& w) {
  bt_attributes();
  const int nref = n - 2, nblk = bt_blocks(n);
  BtScratch sc;
  bt_scratch_layout(n, &w, &sc);
  // Gram matrices and T factors of all blocks, then Y_b^T = V_b^T T_b, then slices
  gram_df_kernel<<<dim3((kBtBlockTc / 32) * (kBtBlockTc / 32), nblk), 256, 0, s>>>(n, nref, w.Vst, w.Gm);
  count_launch();
  tfactor_all_kernel<<<dim3(kBtBlockTc / kTfRows, nblk), 4 * kTfRows, kTfSmem, s>>>(nref, w.tau, w.Gm, w.Tm);
  count_launch();
  if ((n + 63) / 64 * nblk >= 152)
    y_df_kernel<64><<<dim3((n + 63) / 64, nblk), 256, y_smem(64), s>>>(n, nref, w.Vst, w.Tm, sc.yt);
  else
    y_df_kernel<16><<<dim3((n + 15) / 16, nblk), 256, y_smem(16), s>>>(n, nref, w.Vst, w.Tm, sc.yt);
  count_launch();
  tc_split_blocks(s, 0, n, nref, kBtBlockTc, w.Vst, sc.vs, sc.vs_blk, sc.vs_slice, 4);
  tc_split_blocks(s, 1, n, nref, kBtBlockTc, sc.yt, sc.ys, sc.ys_blk, sc.ys_slice, 4);
}

static int eig_backtransform_tc(cudaStream_t s, int n, double* Q, EigWork& w, const TcWork& tw) {
  const int nref = n - 2;
  const int nblk = bt_blocks(n);
  const size_t stride = tc_slot_stride(tw);
  int* err = tc_error_flag(tw);
  BtScratch sc;
  bt_scratch_layout(n, &w, &sc);
  double* Zt = w.A;                      // tridiagonalisation workspace is free now
  transpose_sq(s, n, Q, Zt);
  __nv_bfloat16* sZ = tc_slot_base(tw, kSlotT0);
  __nv_bfloat16* sU = tc_slot_base(tw, kSlotT1);
  for (int b = nblk - 1; b >= 0; --b) {
    const int k0 = b * kBtBlockTc, kb = (k0 + kBtBlockTc < nref) ? kBtBlockTc : nref - k0;
    const int c0 = k0 + 1, m = n - c0;
    const int ldm = tc_ld(m);
    double* Zs = Zt + c0;                                // n x m, ld n
    tc_split_rows(s, n, m, Zs, n, 4, sZ, ldm, stride);
    const int parts = tc_gemm_grouped_rc_splitk(s, n, kb, m, sZ, ldm, stride, sc.vs + (size_t)b * sc.vs_blk, ldm,
                                                sc.vs_slice, 1.0, sc.part, kBtBlockTc, kBtSplitK, err,
                                                tw.wide);   // U parts
    if (parts <= 0) return -1;
    const int ldk = tc_ld(kb);                           // U slices fit the slot: kb <= n
    tc_reduce_split_rows(s, n, kb, sc.part, parts, kBtBlockTc, 4, sU, ldk, stride);
    if (tc_gemm_grouped_rc(s, n, m, kb, sU, ldk, stride, sc.ys + (size_t)b * sc.ys_blk, kBtBlockTc, sc.ys_slice,
                           -1.0, Zs, n, 1, err, tw.wide) != 0)                                        // Zs -= U Y_b
      return -1;
  }
  transpose_sq(s, n, Zt, Q);
  return 0;
}

// The FP64 back-transformation with FP64 tensor-core products (tc_gemm64.cu), also on
// Z^T: per block, last first, U = Z^T_sub V_b^T, Z^T_sub -= (U T_b^T) V_b.  The
// reflectors are cut once in both orientations (rows are zero left of the reflector,
// so whole rows serve every block) and give the Gram matrices of all blocks in one
// launch.  n = 1680: 64.5 -> 3.8 ms, n = 574: 9.4 -> 1.2.
struct Bt64Scratch {
  double *U, *W;       // n x kBtBlockTc
  Tc64Op u, t;         // cut U or W, and T of all blocks
};
static BtBytes bt64_scratch(int n, const EigWork* w, Bt64Scratch* out) {
  const size_t u = (size_t)n * kBtBlockTc * sizeof(double);        // a multiple of 256
  const int rt = tc_blocks(n) * kBtBlockTc;
  if (out) {
    out->t = tc64_op(w->early, rt, kBtBlockTc);
    out->U = (double*)w->late;
    out->W = (double*)(w->late + u);
    out->u = tc64_op(w->late + 2 * u, n, kBtBlockTc);
  }
  return BtBytes{tc64_op_bytes(rt, kBtBlockTc), 2 * u + tc64_op_bytes(n, kBtBlockTc)};
}
static BtBytes bt64_bytes(int n) { return bt64_scratch(n, nullptr, nullptr); }

static int bt_prepare_tc64(cudaStream_t s, int n, EigWork& w, const Tc64Work& tw) {
  constexpr int KB = kBtBlockTc;
  bt_attributes();
  const int nref = n - 2, nblk = bt_blocks(n);
  Bt64Scratch sc;
  bt64_scratch(n, &w, &sc);
  const Tc64Op V = tc64_slot(tw, 0, nref, n), Vt = tc64_slot(tw, 1, n, nref);
  tc64_cut_rows(s, V, 0, n, w.Vst, n);
  tc64_cut_cols(s, Vt, nref, w.Vst, n);
  if (tc64_gemm(s, nref, nref, 0, n, V, 0, V, 0, 0, 1.0, 0, w.Gm, KB, 1, KB, tw.err)) return -1;
  cudaMemsetAsync(w.Tm, 0, (size_t)nblk * KB * KB * sizeof(double), s);     // columns beyond a short last block
  tfactor_all_kernel<<<dim3(KB / kTfRows, nblk), 4 * kTfRows, kTfSmem, s>>>(nref, w.tau, w.Gm, w.Tm);
  count_launch();
  tc64_cut_rows(s, sc.t, 0, KB, w.Tm, KB);
  return 0;
}

static int eig_backtransform_tc64(cudaStream_t s, int n, double* Q, EigWork& w, const Tc64Work& tw) {
  constexpr int KB = kBtBlockTc;
  const int nref = n - 2, nblk = bt_blocks(n);
  Bt64Scratch sc;
  bt64_scratch(n, &w, &sc);
  const Tc64Op V = tc64_slot(tw, 0, nref, n), Vt = tc64_slot(tw, 1, n, nref), Z = tc64_slot(tw, 2, n, n);
  double* Zt = w.A;
  transpose_sq(s, n, Q, Zt);
  for (int b = nblk - 1; b >= 0; --b) {
    const int k0 = b * KB, kb = std::min(KB, nref - k0), c0 = k0 + 1, first = c0 & ~31;
    tc64_cut_rows(s, Z, first, n, Zt, n);
    if (tc64_gemm(s, n, kb, first, n, Z, 0, V, k0, 0, 1.0, 0, sc.U, KB, 0, 0, tw.err)) return -1;
    tc64_cut_rows(s, sc.u, 0, kb, sc.U, KB);
    if (tc64_gemm(s, n, kb, 0, kb, sc.u, 0, sc.t, k0, 0, 1.0, 0, sc.W, KB, 0, 0, tw.err)) return -1;
    tc64_cut_rows(s, sc.u, 0, kb, sc.W, KB);
    if (tc64_gemm(s, n, n - c0, 0, kb, sc.u, 0, Vt, c0, k0, -1.0, 1, Zt + c0, n, 0, 0, tw.err)) return -1;
  }
  transpose_sq(s, n, Zt, Q);
  return 0;
}

int eig_backtransform_prepare(cudaStream_t s, int n, EigWork& w, const TcWork* tw, const Tc64Work* t64) {
  if (n <= 2) return 0;
  if (tw) {
    bt_prepare_tc(s, n, w);
    return 0;
  }
  return t64 ? bt_prepare_tc64(s, n, w, *t64) : 0;
}

int eig_backtransform(cudaStream_t s, int n, double* Q, EigWork& w, const TcWork* tw, const Tc64Work* t64,
                      bool prepared) {
  if (!prepared && eig_backtransform_prepare(s, n, w, tw, t64) != 0) return -1;
  if (tw && n > 2) return eig_backtransform_tc(s, n, Q, w, *tw);
  if (t64 && n > 2) return eig_backtransform_tc64(s, n, Q, w, *t64);
  // 4. back-transformation, last block of reflectors first
  int nref = n - 2;
  if (nref > 0) {
    int nblk = (nref + kBtBlock - 1) / kBtBlock;
    for (int b = nblk - 1; b >= 0; --b) {
      int k0 = b * kBtBlock, k1 = (k0 + kBtBlock < nref) ? k0 + kBtBlock : nref;
      int kb = k1 - k0, c0 = k0 + 1, m = n - c0;
      const double* Vb = w.Vst + (size_t)k0 * n + c0;
      dgemm(s, 0, 1, kb, kb, m, 1.0, Vb, n, Vb, n, 0.0, w.Gm, kBtBlock);
      tfactor_kernel<<<1, kBtBlock, kb * kb * sizeof(double), s>>>(kb, w.tau + k0, w.Gm, kBtBlock, w.Tm, kBtBlock);
      count_launch();
      dgemm(s, 0, 0, kb, n, m, 1.0, Vb, n, Q + (size_t)c0 * n, n, 0.0, w.Wt, n);
      dgemm(s, 0, 0, kb, n, kb, 1.0, w.Tm, kBtBlock, w.Wt, n, 0.0, w.Wt2, n);
      dgemm(s, 1, 0, m, n, kb, -1.0, Vb, n, w.Wt2, n, 1.0, Q + (size_t)c0 * n, n);
    }
  }
  return 0;
}

}  // namespace kx
