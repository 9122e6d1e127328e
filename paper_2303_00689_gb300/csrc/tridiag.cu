// Householder tridiagonalisation T = H^T F H of the Fock matrix (eq. 19 needs
// its eigenpairs).  Per column k: x = row k of the matrix with the pending rank-2
// update (v, w of column k - 1), the reflector v_k, tau_k of x, and p = tau A v_k;
// the rank-2 update of column k is applied one column later, fused with the
// matrix-vector product, so an element of the trailing matrix is read and written
// once per column.  A persistent kernel for the FP64 path, and two in double-float
// (df.cuh: FP32 pairs, about 48 bits, on the FP32 pipe) for the mixed path: small
// matrices in one thread-block cluster, others on a grid.  What bounds them up to
// ~1500 columns is the dependent chain of a column (exchange of p between the blocks,
// reductions, product), n times, so the more blocks share the product the better, until
// the exchange between them costs more; above, the FP32 (FP64) operations.
//
// A grid that takes much of the device cannot always run beside another one (two
// handles stepped by two threads).  So a launch on its own starts with a check-in:
// either every block is there within kCheckInNs and all go on, or all leave, and a
// second launch behind it, which otherwise returns at once, does the same work with
// few blocks.  Double-float grids leave at once while the steps in flight on the device
// would fill it half as often again (g_demand; handles stepped by several threads): small
// grids then leave SMs to the other handles' kernels.  Batches and the server run small
// grids from the start and keep their total within what the device holds
// (eig_tridiag_weight).  The results do not depend on the number of blocks.
//
// Every wait is bounded in wall time (g_barrier_ns): a block that gives up, or
// that finds another block's timeout flag set, records kStatusTimeout and
// returns.
#include <limits.h>

#include <algorithm>
#include <iterator>

#include "common.cuh"
#include "df.cuh"
#include "kernels.h"
#include "tri_packet.h"

namespace kx {

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
constexpr unsigned long long kBarrierNs = 2000000000ull;   // 2 s
constexpr unsigned long long kCheckInNs = 1000000ull;      // 1 ms
// the wall-time limit of the waits (per device; tests set it through
// eig_set_barrier_limit; 0 makes every launch give up at once, even one whose
// waits would be satisfied, so a test can force the expiry path of a real step)
__device__ unsigned long long g_barrier_ns = kBarrierNs;

// what the large grids of the steps in flight on this device take, in thousandths of an SM
// (eig_tridiag_weight); every step adds its own at its start and takes it back at its end
__device__ int g_demand = 0;

int* eig_demand_word() {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_demand) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return (int*)p;
}

int eig_set_barrier_limit(unsigned long long ns) {
  return cudaMemcpyToSymbol(g_barrier_ns, &ns, sizeof(ns)) == cudaSuccess ? 0 : -1;
}

// ---- 128-bit packets: a value and what tells its column ------------------------------
struct __align__(16) Packet {
  unsigned long long x, y;
};
__device__ __forceinline__ Packet packet_load(const Packet* q) {
  Packet r;
  asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
               : "=l"(r.x), "=l"(r.y)
               : "l"(q)
               : "memory");
  return r;
}
__device__ __forceinline__ void packet_store(Packet* q, Packet v) {
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(q),
               "l"(v.x), "l"(v.y)
               : "memory");
}

struct TriArgs {
  int n, k0, k1;        // columns of this launch
  int rs;               // rows per block kept in shared memory
  int reps;             // copies of the packets (a power of two)
  const double* F;      // k0 == 0: the input; else null
  void* A;              // n x n working matrix (rows outside shared memory, hand-over between launches)
  unsigned* gate;       // check-in: arrivals, then 0 undecided / 1 go / 2 leave
  int role;             // 0: no check-in; 1: with check-in; 2: runs only if the launch before it left
  double *Vst, *d, *e, *tau;
  Packet* pk;
  double* carry;        // x of the last column of a launch, then its four scalars
  int* status;
};

// Thread 0: whether this launch is to run.  gate: arrivals, then 0 undecided / 1 go /
// 2 leave.  Role 1: all blocks are here before one gives up waiting, and none has seen a
// demand above `crowd`; role 2: the launch before this one was given up.
__device__ bool check_in(unsigned* gate, int role, int G, int crowd) {
  volatile unsigned* state = gate + 1;
  if (role == 1) {
    if (*(volatile int*)&g_demand > crowd) atomicCAS(gate + 1, 0u, 2u);
    if (atomicAdd(gate, 1u) == (unsigned)G - 1) atomicCAS(gate + 1, 0u, 1u);
    const unsigned long long t0 = global_ns();
    while (*state == 0)
      if (global_ns() - t0 > kCheckInNs) atomicCAS(gate + 1, 0u, 2u);
    return *state == 1;
  }
  return *state == 2;
}

// a poll's turn `it` without success: true when it has to give up
__device__ __forceinline__ bool poll_expired(unsigned it, unsigned long long& t0, unsigned long long limit,
                                             const int* status) {
  if ((it & 63u) != 0) return false;
  if (t0 == 0) {
    t0 = global_ns();
    return false;
  }
  return global_ns() - t0 > limit || it > (1u << 27) || ((*(volatile const int*)status) & kStatusTimeout);
}

// Named barriers.  Whole warps arrive: lanes leave the packet polls one by one, and
// without the __syncwarp the code after them ran lane by lane (5 times slower).
__device__ __forceinline__ void bar_sync(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// most rows > k0 that a block of a grid of G owns
__host__ __device__ __forceinline__ int tri_rows(int n, int k0, int G) { return (n - k0 - 1 + G - 1) / G; }

// ---- FP64 -------------------------------------------------------------------------
// n = 26, 240, 574, 1680: 97, 1310, 3400, 21900 us; with one block per 2^16 elements,
// rows dealt anew in every column and a grid barrier per column: 178, 8544, 17400,
// 49545 us.
//  * Rows i = b (mod G) belong to block b for the whole launch and live in its
//    shared memory; what does not fit stays in global memory (L2) and is touched
//    by its own block only.
//  * No grid barrier: the blocks exchange 16-byte packets, written and read as one
//    128-bit access, that say themselves which column they are of, and a reader
//    polls a packet until it is the current one: one trip through L2 (~900 cycles
//    across the two dies) per column instead of the data's, an arrival counter's,
//    a poll's and the loads'.  Packets are double-buffered by the column's parity:
//    an owner overwrites column k - 2's packet only after it has read all packets
//    of column k - 1, each of which was sent after its sender had read column
//    k - 2's.  Every block polls all packets, and on one copy of them the polls of
//    a line queue up in its L2 slice (~45 cycles a block), so there are up to 16
//    copies, about eight readers each.
//  * Every block forms the reflector itself from the packets (same data, same order:
//    bitwise the same in all blocks); its scalars (sqrt, reciprocals) and the store
//    of v_k are left to an extra warp while the others run the product, which uses
//    the unscaled x: p_i = tau scale (s_i - beta a_{i,k+1}), s_i = sum_j a_ij x_j,
//    v = scale (x - beta e_{k+1}).
// A worker thread owns fixed columns j = t (mod NTG) and keeps their x, v and w in
// registers through the packets, the reflector and the product; shared memory
// holds matrix rows and the (v, w) of the block's own rows, which every thread
// needs.  One packet per row carries s_i and, by symmetry, the next pivot row's
// a_{i,k+1}; the reader forms p_i, so the scalars are off the path from the product
// to the packets.  The highest exponent bit of s_i carries the parity of the packet's
// use, all other bits are those of s_i (tri_packet.h).  Small matrices have more warps
// than columns: RG groups of NTG threads hold the same columns and share the rows
// out.  A launch covers the columns [k0, k1): with a part of the rows outside
// shared memory the next launch starts with shorter rows, so more of them fit (all
// of them from a trailing width of ~1800 with 152 blocks on).
constexpr unsigned long long kTag = kPacketTag;
struct __align__(16) RowVecs {
  double v, w;
};

// N rows of the group, RG apart, starting with row r; column j of the u-th at
// p[u stride + j], p offset by the thread's first column.  The thread's columns
// cm <= c < ce: the pending rank-2 update, stored back, and the row sums of a x over
// the warp's columns into part.
template <int NTG, int RG, int CPL, int N>
__device__ __forceinline__ void f64_rows(double* p, ptrdiff_t stride, const RowVecs* __restrict__ PWr, int r,
                                         int t, int cm, int ce, const double (&v)[CPL], const double (&w)[CPL],
                                         const double (&x)[CPL], double* __restrict__ part, int lane) {
  constexpr int GW = NTG / 32;
  double acc[N];
#pragma unroll
  for (int u = 0; u < N; ++u) acc[u] = 0.0;
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    if (c >= cm && c < ce) {
      double y[N];
#pragma unroll
      for (int u = 0; u < N; ++u) y[u] = p[u * stride + NTG * c];
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const RowVecs q = PWr[r + u * RG];
        y[u] = fma(-q.v, w[c], fma(-q.w, v[c], y[u]));
        p[u * stride + NTG * c] = y[u];
        acc[u] = fma(y[u], x[c], acc[u]);
      }
    }
  }
  if constexpr (N == 1) {
    const double tot = warp_sum(acc[0]);
    if (lane == 0) part[(size_t)r * GW + (t >> 5)] = tot;
  } else {
    const double tot = warp_totals<N>(acc, lane);
    if ((lane & (32 / N - 1)) == 0) part[(size_t)(r + lane / (32 / N) * RG) * GW + (t >> 5)] = tot;
  }
}
// the group's rows r, r + RG, ... < r_end, all in shared memory or all in global memory
template <int NTG, int RG, int CPL, int NMAX>
__device__ __forceinline__ void f64_row_loop(double* base, ptrdiff_t row, const RowVecs* PWr, int r, int r_end,
                                             int t, int cm, int ce, const double (&v)[CPL], const double (&w)[CPL],
                                             const double (&x)[CPL], double* part, int lane) {
  double* p = base + (ptrdiff_t)r * row + t;
  const ptrdiff_t stride = row * RG;
  if constexpr (NMAX >= 8) {
#pragma unroll 1
    for (; r + 7 * RG < r_end; r += 8 * RG, p += 8 * stride)
      f64_rows<NTG, RG, CPL, 8>(p, stride, PWr, r, t, cm, ce, v, w, x, part, lane);
  }
  if constexpr (NMAX >= 4) {
#pragma unroll 1
    for (; r + 3 * RG < r_end; r += 4 * RG, p += 4 * stride)
      f64_rows<NTG, RG, CPL, 4>(p, stride, PWr, r, t, cm, ce, v, w, x, part, lane);
  }
#pragma unroll 1
  for (; r + RG < r_end; r += 2 * RG, p += 2 * stride)
    f64_rows<NTG, RG, CPL, 2>(p, stride, PWr, r, t, cm, ce, v, w, x, part, lane);
  if (r < r_end) f64_rows<NTG, RG, CPL, 1>(p, stride, PWr, r, t, cm, ce, v, w, x, part, lane);
}

__device__ __forceinline__ void f64_reflector(double x1, double sigma, double& beta, double& tau, double& scale) {
  if (sigma == 0.0) {
    beta = x1; tau = 0.0; scale = 0.0;
    return;
  }
  const double nrm = ::sqrt(x1 * x1 + sigma);
  beta = (x1 >= 0.0) ? -nrm : nrm;
  tau = (beta - x1) / beta;
  scale = 1.0 / (x1 - beta);
}

// RG groups of NTG worker threads (thread t of a group: columns t + NTG c, c < CPL)
// and one warp for the reflector scalars.  SOLO: a grid of one block; the packets
// stay in shared memory.  Barriers 0: group 0 and the scalar warp; 1: the scalars;
// 2 + g: group g.
template <int NTG, int RG, int CPL, bool SOLO>
__global__ void __launch_bounds__(NTG * RG + 32, (NTG * RG <= 256 && CPL <= 4) ? 2 : 1) tridiag_f64_kernel(TriArgs g) {
  constexpr int NT = NTG * RG, GW = NTG / 32;                      // workers; warps of a group
  static_assert(GW <= 16 && (RG & (RG - 1)) == 0, "layout");
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = g.n, G = SOLO ? 1 : (int)gridDim.x, b = SOLO ? 0 : (int)blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31;
  const bool worker = tid < NT;
  const int rg = worker ? tid / NTG : 0, t = tid - rg * NTG;       // group, thread of the group
  const int Rtot = (n > b) ? (n - b + G - 1) / G : 0;              // rows b, b + G, ...
  // shared memory: own rows' (v, w), packets (SOLO), resident rows, own rows' x (two columns'),
  // sigma partials (two columns'), p.v partials per group, row partials
  RowVecs* PWr = (RowVecs*)smem;                                           // by row r
  Packet* spk = (Packet*)(PWr + Rtot);                             // by the column's parity, then row (SOLO)
  double* rows = (double*)(spk + (SOLO ? 2 * n : 0));
  const int ms = n - g.k0 - 1;                                     // a row: columns k0 + 1 ..
  double* Xr = rows + (size_t)g.rs * ms;
  double* redB = Xr + 2 * Rtot;
  double* redA = redB + 2 * NTG + rg * (NTG + 4);
  double* part = redB + 2 * NTG + RG * (NTG + 4);                  // [r][warp of the group]
  __shared__ double s_par[2][4];                                   // beta, tau * scale, tau, scale
  __shared__ double s_x[2][2];                                     // x_k (the diagonal), x_{k+1}
  __shared__ double s_pk[RG];
  // by the column's parity: the scalar warp reads column k's word after barrier 0, when polls of
  // column k + 1 may already write theirs (k + 2's follow its arrival at barrier 1)
  __shared__ int s_fail[2];
  double* A = (double*)g.A;
  const int rres = max(Rtot - g.rs, 0);                            // rows r >= rres are resident
  double* rows0 = rows - (ptrdiff_t)rres * ms - (g.k0 + 1);        // column j of resident row r: [r ms + j]
  const unsigned long long limit = g_barrier_ns;
  if (n > 2 && limit == 0) {
    if (tid == 0) atomicOr(g.status, (int)kStatusTimeout);
    return;
  }
  if (g.role != 0) {
    if (tid == 0) s_fail[0] = check_in(g.gate, g.role, G, INT_MAX) ? 0 : 1;
    __syncthreads();
    if (s_fail[0]) return;
  }
  for (int r = g.F ? 0 : rres; r < Rtot; ++r) {
    const int i = b + r * G;
    if (i <= g.k0) continue;
    const double* src = (g.F ? g.F : A) + (size_t)i * n;
    double* dst = (r >= rres) ? rows0 + (ptrdiff_t)r * ms : A + (size_t)i * n;
    for (int j = g.k0 + 1 + tid; j < n; j += NT + 32) dst[j] = src[j];
  }
  __syncthreads();                                                 // s_fail has been read
  if (tid < 2) s_fail[tid] = 0;
  if (tid < 4) s_par[(g.k0 + 1) & 1][tid] = (g.k0 > 0) ? g.carry[n + tid] : 0.0;
  __syncthreads();
  const bool owns_last = (n - 1) % G == b;                         // alive in every column
  auto entry = [&](int r, int j) {                                 // column j of the block's row r
    return (r >= rres) ? rows0[(ptrdiff_t)r * ms + j] : A[(size_t)(b + (size_t)r * G) * n + j];
  };

  int rf = (g.k0 + 1 > b) ? (g.k0 + 1 - b + G - 1) / G : 0;        // first row > k
  if (!worker) {
    // ---- the scalar warp: reflector of column k, then the block's share of v_k
    bar_arrive(1, NT + 32);
    for (int k = g.k0; k < g.k1; ++k) {
      if (b + rf * G <= k) ++rf;
      if (rf >= Rtot) return;
      bar_sync(0, NTG + 32);                                       // x of column k is there
      const int par = k & 1;
      if (s_fail[par] || k == n - 2) return;
      const double* red = redB + par * NTG;
      double s0 = red[lane], s1 = 0.0;
#pragma unroll
      for (int q = 1; q < GW; ++q) {
        if (q & 1) s1 += red[lane + 32 * q];
        else s0 += red[lane + 32 * q];
      }
      const double sigma = warp_sum(s0 + s1);
      double beta, tau, scale;
      f64_reflector(s_x[par][1], sigma, beta, tau, scale);
      if (lane == 0) {
        s_par[par][0] = beta; s_par[par][1] = tau * scale; s_par[par][2] = tau; s_par[par][3] = scale;
      }
      bar_arrive(1, NT + 32);
      if (lane == 0 && owns_last) { g.d[k] = s_x[par][0]; g.e[k] = beta; g.tau[k] = tau; }
#pragma unroll 1
      for (int r = rf + lane; r < Rtot; r += 32) {
        const int j = b + r * G;
        g.Vst[(size_t)k * n + j] = (j == k + 1) ? 1.0 : Xr[par * Rtot + r] * scale;
      }
    }
    return;
  }

  // ---- workers
  const int gw = t >> 5;                                           // warp of the group
  const int ce = (t < n) ? (n - t + NTG - 1) / NTG : 0;            // columns of the thread
  double x[CPL], v[CPL], w[CPL];
  int own[CPL];                                                    // the block's row that is column c, or -1
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int j = t + NTG * c;
    own[c] = (j < n && j % G == b) ? j / G : -1;
    x[c] = (g.k0 > 0 && j >= g.k0 && j < n) ? g.carry[j] : 0.0;
    v[c] = w[c] = 0.0;
  }
  const Packet* in0 = g.pk + (size_t)(b & (g.reps - 1)) * 2 * n;
  for (int k = g.k0; k < g.k1; ++k) {
    if (b + rf * G <= k) ++rf;
    const int par = k & 1;
    // orders the packets before their readers, and the readers of column k - 2's, which a group
    // that is ahead overwrites at the end of this column
    if (SOLO) bar_sync(1, NT + 32);
    // packets of column k - 1, of the columns j >= k (row k of the matrix: by symmetry a_{j,k})
    Packet q[CPL];
    if (rf < Rtot) {
      if (k == 0) {
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
          const int j = t + NTG * c;
          q[c] = Packet{0ull, (j < n) ? (unsigned long long)__double_as_longlong(g.F[j]) : 0ull};
        }
      } else {
        const Packet* in = in0 + (size_t)(par ^ 1) * n;
        const unsigned long long want = (((k - 1) >> 1) & 1) ? kTag : 0ull;
        unsigned long long t0 = 0;
#pragma unroll 1
        for (unsigned it = 1;; ++it) {
          // all together: one after the other, each would cost a trip to L2 of its own
#pragma unroll
          for (int c = 0; c < CPL; ++c) {
            const int j = t + NTG * c;
            if (j >= k && j < n) q[c] = SOLO ? spk[(par ^ 1) * n + j] : packet_load(in + j);
          }
          if (SOLO) break;
          bool old = false;
#pragma unroll
          for (int c = 0; c < CPL; ++c) {
            const int j = t + NTG * c;
            old |= j >= k && j < n && (q[c].x & kTag) != want;
          }
          if (!old) break;
          if (poll_expired(it, t0, limit, g.status)) {
            atomicOr(g.status, (int)kStatusTimeout);
            s_fail[par] = 1;
            break;
          }
        }
      }
    }
    if (!SOLO) bar_sync(1, NT + 32);                               // scalars of column k - 1; every group's polls are over
    if (rf >= Rtot) return;                                        // nothing left to do for this block
    if (s_fail[par]) {
      if (rg == 0) bar_sync(0, NTG + 32);                          // lets the scalar warp go
      return;
    }
    const double beta = s_par[par ^ 1][0], ts = s_par[par ^ 1][1], tau = s_par[par ^ 1][2], scale = s_par[par ^ 1][3];
    // p = tau scale (s - beta a), v = scale x (leading element 1), p.v
    const bool prev = k > 0;
    double loc = 0.0;
    if (prev) {
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const int j = t + NTG * c;
        if (j < k || j >= n) continue;
        w[c] = ts * (__longlong_as_double((long long)packet_decode(q[c].x)) -
                     beta * __longlong_as_double((long long)q[c].y));
        v[c] = (j == k) ? 1.0 : x[c] * scale;
        if (j == k) s_pk[rg] = w[c];
        loc = fma(w[c], v[c], loc);
      }
    }
    // p.v over the group: one warp instruction of the FP64 pipe takes ~62 cycles of
    // a scheduler, so a few warps fold the NTG partials and one thread adds the rest
    constexpr int FW = (GW < 4) ? GW : 4;                          // folding warps
    redA[t] = loc;
    bar_sync(2 + rg, NTG);
    if (gw < FW) {
      double f = loc;
      for (int z = t + 32 * FW; z < NTG; z += 32 * FW) f += redA[z];
      f = warp_sum(f);
      if (lane == 0) redA[NTG + gw] = f;
    }
    bar_sync(2 + rg, NTG);
    if (t == 0) {
      double f = redA[NTG];
      for (int z = 1; z < FW; ++z) f += redA[NTG + z];
      redA[NTG] = f;
    }
    bar_sync(2 + rg, NTG);
    const double coef = 0.5 * tau * redA[NTG];
    const double wk = prev ? s_pk[rg] - coef : 0.0;                // w_k (v_k = 1)
    const double vk = prev ? 1.0 : 0.0;
    // w_{k-1}, the updated row k, sigma = sum_{j >= k+2} x_j^2; the own rows' (v, w)
    double sig = 0.0;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int j = t + NTG * c;
      if (j < k || j >= n) continue;
      if (prev) w[c] = fma(-coef, v[c], w[c]);
      x[c] = fma(-vk, w[c], fma(-wk, v[c], __longlong_as_double((long long)q[c].y)));
      if (rg == 0) {
        if (j >= k + 2) sig = fma(x[c], x[c], sig);
        else s_x[par][j - k] = x[c];
      }
      const int r = own[c];
      if (r >= 0) {
        if ((r & (RG - 1)) == rg) PWr[r] = RowVecs{v[c], w[c]};
        if (rg == 0) Xr[par * Rtot + r] = x[c];
      }
    }
    if (rg == 0) {
      redB[par * NTG + t] = sig;
      bar_sync(0, NTG + 32);
    } else {
      bar_sync(2 + rg, NTG);
    }
    if (k == n - 2) {                                              // the owner of row n - 1 alone is left
      const int r = Rtot - 1;
      if (rg == (r & (RG - 1)) && t == 0)
        g.d[n - 1] = fma(-PWr[r].v, PWr[r].w, fma(-PWr[r].w, PWr[r].v, entry(r, n - 1)));
      if (rg == 0 && t == 0) { g.d[k] = s_x[par][0]; g.e[k] = s_x[par][1]; }
      return;
    }
    // the product over the group's rows r = rg (mod RG), rf <= r < Rtot: the
    // resident rows (shared memory) and the others (L2), half of the warps
    // starting with either, so that the two memories work at the same time
    const int cm = (k >= t) ? (k - t) / NTG + 1 : 0;               // first column > k of the thread
    const int r_lo = rf + ((rg - rf) & (RG - 1));
    const int r_sm = max(rf, rres);                                // first resident row > k
    constexpr int NR = (CPL <= 2) ? 8 : (CPL <= 7) ? 4 : 2;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      if ((half ^ gw) & 1) {
        f64_row_loop<NTG, RG, CPL, NR>(rows0, ms, PWr, r_sm + ((rg - r_sm) & (RG - 1)), Rtot, t, cm, ce, v, w, x, part,
                                       lane);
      } else if (rf < rres) {
        f64_row_loop<NTG, RG, CPL, 2>(A + (size_t)b * n, (ptrdiff_t)G * n, PWr, r_lo, min(rres, Rtot), t, cm, ce, v, w,
                                      x, part, lane);
      }
    }
    bar_sync(2 + rg, NTG);
    // s_i over the group's warps, and the packets: a row per half warp, a copy per lane
    const unsigned long long tag = ((k >> 1) & 1) ? kTag : 0ull;
#pragma unroll 1
    for (int r0 = r_lo + 2 * RG * gw; r0 < Rtot; r0 += 2 * RG * GW) {
      const int r = r0 + (lane >> 4) * RG, l = lane & 15;
      constexpr int L = (GW > 8) ? 16 : (GW > 4) ? 8 : (GW > 2) ? 4 : GW;
      double s = (r < Rtot && (l & (L - 1)) < GW) ? part[(size_t)r * GW + (l & (L - 1))] : 0.0;
#pragma unroll
      for (int o = L / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (l < (SOLO ? 1 : g.reps) && r < Rtot) {
        const int i = b + r * G;
        const Packet o{packet_encode((unsigned long long)__double_as_longlong(s), tag),
                       (unsigned long long)__double_as_longlong(entry(r, k + 1))};
        if (SOLO) spk[par * n + i] = o;
        else packet_store(g.pk + ((size_t)l * 2 + par) * n + i, o);
      }
    }
  }
  // hand-over to the next launch: resident rows, x of the last column and its scalars
  bar_sync(1, NT + 32);
  for (int r = rres; r < Rtot; ++r) {
    const int i = b + r * G;
    if (i <= g.k1) continue;
    const double* src = rows0 + (ptrdiff_t)r * ms;
    for (int j = g.k1 + 1 + tid; j < n; j += NT) A[(size_t)i * n + j] = src[j];
  }
  if (owns_last && rg == 0) {
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int j = t + NTG * c;
      if (j >= g.k1 && j < n) g.carry[j] = x[c];
    }
    if (t < 4) g.carry[n + t] = s_par[(g.k1 - 1) & 1][t];
  }
}

// ---- double-float -------------------------------------------------------------------
// With the fused step a column is one grid phase:
//  * after the barrier every block reads p_{k-1} and row k in one pass, forms
//    w_{k-1} = p - (tau/2)(p.v)v and the updated row k (x = row k of A_k);
//  * the matrix-vector product uses the unscaled x (x_{k+1} = x_1) and
//    keeps a_{i,k+1}, so it need not wait for beta, tau and the scale, which
//    thread 0 forms meanwhile:
//    p_i = tau scale (sum_j a_ij x_j - beta a_{i,k+1}) since v = scale (x - beta e_{k+1});
//  * a block's rows (i = k+1+b+rG) are cut into segments of 512 columns (256
//    and 128 once the trailing matrix is narrower than 500 and 200 columns)
//    and the (row, segment) items dealt over the warps, so the warps stay
//    balanced while the trailing matrix shrinks; warp 0, which forms the
//    reflector scalars first, takes the last item of each round, so it never
//    holds more items than another warp; each lane issues the loads of its
//    item before the arithmetic;
//  * block reductions take one CTA barrier each.
// Shared memory: PW[j] = (v_{k-1}, w_{k-1}) as one 16-byte pair (during the
// first passes it holds row k and p_{k-1}), VC[j] = x_k, then v_k, plus
// reduction scratch and the (row, segment) partial sums.
// Split-phase grid barrier on a monotonically increasing arrival counter
// (reset to 0 before the launch): the e-th barrier of a block is passed once
// the counter reaches e * nblocks.  grid_arrive makes the block's earlier
// writes visible (CTA barrier, then a release reduction by thread 0), so
// independent work can run before grid_wait (an acquire load, bounded in wall
// time like grid_barrier; on expiry kStatusTimeout is set and false returned).
__device__ __forceinline__ void grid_arrive(unsigned* cnt) {
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
}
__device__ bool grid_wait(const unsigned* cnt, unsigned target, int* status) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    const unsigned long long t0 = global_ns();
    long long it = 0;
    if (g_barrier_ns == 0) atomicOr(status, (int)kStatusTimeout);
    for (; g_barrier_ns != 0;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
      if ((int)(v - target) >= 0) break;
      ++it;
      if ((it & 63) == 0 && (global_ns() - t0 > g_barrier_ns || it > (1LL << 27) ||
                             ((*(volatile int*)status) & kStatusTimeout))) {
        atomicOr(status, (int)kStatusTimeout);
        break;
      }
      __nanosleep(16);
    }
    s_ok = ((*(volatile int*)status) & kStatusTimeout) ? 0 : 1;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int kTriThreadsDf = 512;    // threads per block of the double-float kernel
constexpr int kDfRed = 32;
constexpr int kDfSeg = 512;           // columns per (row, segment) work item: 16 per lane
constexpr int kDfNarrow1 = 500;       // trailing width at and below which items are 256 columns
constexpr int kDfNarrow2 = 200;       // ... and 128 columns
static_assert(kTriThreadsDf / 32 <= kDfRed, "one reduction slot per warp");
// rows per block at the first column, for a grid of G blocks
static int tridiag_df_rmax(int n, int G) { return (n - 1 + G - 1) / G; }
static size_t tridiag_smem_df(int n, int G) {
  // at most 2 segments per row while the narrow items are in use
  const size_t rmax = (size_t)tridiag_df_rmax(n, G),
               smax = std::max<size_t>((size_t)(n - 1 + kDfSeg - 1) / kDfSeg, 2);
  return (3 * (size_t)n + 2 * kDfRed + rmax + rmax * smax) * sizeof(dfl);
}

// Loads of data other blocks wrote since the last grid barrier (and of rows
// this block does not own in every column) go past L1 to L2.
__device__ __forceinline__ dfl ldcg_df(const dfl* p) {
  const float2 v = __ldcg((const float2*)p);
  return dfl{v.x, v.y};
}
// every thread gets the sum of the kTriThreadsDf / 32 warp partials (written to
// scratch[warp] by lane 0 before a CTA barrier), added as a pairwise tree
__device__ __forceinline__ dfl df_sum_partials(const dfl* scratch) {
  constexpr int NW = kTriThreadsDf / 32;
  dfl t[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) t[w] = scratch[w];
#pragma unroll
  for (int st = 1; st < NW; st <<= 1)
#pragma unroll
    for (int w = 0; w + st < NW; w += 2 * st) t[w] = df_add(t[w], t[w + st]);
  return t[0];
}

__device__ __forceinline__ dfl lo2(float4 a) { return dfl{a.x, a.y}; }
__device__ __forceinline__ dfl hi2(float4 a) { return dfl{a.z, a.w}; }
__device__ __forceinline__ float4 pack4(dfl a, dfl b) { return make_float4(a.hi, a.lo, b.hi, b.lo); }

// The fused items of column k for one block: the pending rank-2 update
// (v_{k-1}, w_{k-1}) of rows/cols >= k+1, stored back, and sum_j a_ij x_j of
// each (row, SEG-column segment) item into part[r * S + sg] (a_{i,k+1} of the
// block's rows into ak1s).  Warp w starts at item w - 1, warp 0 at NW - 1.
// The block's rows are i = first + r G, r < R; row r at rows + r ld when they are resident
// in shared memory (RES), at rows + i ld otherwise.
template <int SEG, bool RES>
__device__ __forceinline__ void df_items(float2* __restrict__ rows, int ld, int first_row, int n, int k, int G, int R,
                                         int wid, int lane, bool prev, const float4* PW, const dfl* VC, dfl* part,
                                         dfl* ak1s) {
  constexpr int PER = SEG / 32, NW = kTriThreadsDf / 32;
  const int S = (n - (k + 1) + SEG - 1) / SEG;
  const int Q = R * S;
  for (int q = (wid == 0) ? NW - 1 : wid - 1; q < Q; q += NW) {
    const int r = q / S, sg = q - r * S;
    const int i = first_row + r * G;
    float2* row = rows + (size_t)(RES ? r : i) * ld;
    const int jb = k + 1 + sg * SEG + lane;
    const bool full = (k + 1 + (sg + 1) * SEG) <= n;
    dfl a0 = {0.0f, 0.0f}, a1 = {0.0f, 0.0f}, first = {0.0f, 0.0f};
    if (full) {
      float2 xr[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) xr[u] = RES ? row[jb + 32 * u] : __ldcg(row + jb + 32 * u);
      if (prev) {
        const float4 pwi = PW[i];
        const dfl vi = lo2(pwi), wi = hi2(pwi);
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const int j = jb + 32 * u;
          const float4 pw = PW[j];
          const dfl x = df_rank2(dfl{xr[u].x, xr[u].y}, vi, hi2(pw), wi, lo2(pw));
          row[j] = make_float2(x.hi, x.lo);
          if (u == 0) first = x;
          if (u & 1) df_acc_mul(a1, x, VC[j]); else df_acc_mul(a0, x, VC[j]);
        }
      } else {
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const int j = jb + 32 * u;
          const dfl x = dfl{xr[u].x, xr[u].y};
          if (u == 0) first = x;
          if (u & 1) df_acc_mul(a1, x, VC[j]); else df_acc_mul(a0, x, VC[j]);
        }
      }
    } else {
      float2 xr[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int j = jb + 32 * u;
        xr[u] = (j < n) ? (RES ? row[j] : __ldcg(row + j)) : make_float2(0.0f, 0.0f);
      }
      const float4 pwi = prev ? PW[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      const dfl vi = lo2(pwi), wi = hi2(pwi);
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const int j = jb + 32 * u;
        if (j < n) {
          dfl x = dfl{xr[u].x, xr[u].y};
          if (prev) {
            const float4 pw = PW[j];
            x = df_rank2(x, vi, hi2(pw), wi, lo2(pw));
            row[j] = make_float2(x.hi, x.lo);
          }
          if (u == 0) first = x;
          if (u & 1) df_acc_mul(a1, x, VC[j]); else df_acc_mul(a0, x, VC[j]);
        }
      }
    }
    const dfl acc = df_warp_sum(df_add(df_norm(a0), df_norm(a1)));
    if (lane == 0) {
      part[r * S + sg] = acc;
      if (sg == 0) ak1s[r] = first;        // lane 0, u = 0 is column k+1
    }
  }
}

// (The compiler gives it more than 64 registers a thread, so one block an SM: with two of
// them an SM a batch of 16 cages took 20.7 instead of 19.3 ms.)
template <bool GATED>
__global__ void __launch_bounds__(kTriThreadsDf) tridiag_df_kernel(int n, dfl* __restrict__ A,
                                                                 double* __restrict__ Vst,
                                                                 double* __restrict__ d,
                                                                 double* __restrict__ e,
                                                                 double* __restrict__ tau,
                                                                 dfl* __restrict__ pbuf,
                                                                 unsigned* bar, int* status, int rmax, int role,
                                                                 int crowd) {
  extern __shared__ float4 sm4[];
  float4* PW = sm4;                          // n pairs
  dfl* VC = (dfl*)(sm4 + n);                 // n
  dfl* redA = VC + n;                        // partials of p.v
  dfl* redB = redA + kDfRed;                 // partials of sigma
  dfl* ak1s = redB + kDfRed;                 // a_{i,k+1} of the block's rows (rmax)
  dfl* part = ak1s + rmax;                   // (row, segment) partial sums (rmax x smax)
  __shared__ dfl s_df[4];                    // beta, tau * scale, tau, scale
  if constexpr (GATED) {
    __shared__ int s_go;
    if (threadIdx.x == 0) s_go = check_in(bar + 2, role, (int)gridDim.x, crowd) ? 1 : 0;
    __syncthreads();
    if (!s_go) return;
  }
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  constexpr int T = kTriThreadsDf, NW = kTriThreadsDf / 32;
  const int G = gridDim.x;
  dfl tau_prev = {0.0f, 0.0f};               // tau_{k-1}
  if (n == 1) {
    if (blockIdx.x == 0 && tid == 0) d[0] = df_to_double(A[0]);
    return;
  }
  for (int k = 0;; ++k) {
    const bool prev = k > 0;
    const bool last = (k == n - 2);
    const dfl* pbp = pbuf + (size_t)((k + 1) & 1) * n;   // p_{k-1}
    // pass 1: row k and p_{k-1} in one sweep of loads (kept in PW); partial p.v
    dfl loc = {0.0f, 0.0f};
#pragma unroll 4
    for (int j = k + tid; j < n; j += T) {
      const dfl a = ldcg_df(A + (size_t)k * n + j);
      dfl p = {0.0f, 0.0f};
      if (prev) {
        p = ldcg_df(pbp + j);
        df_acc_mul(loc, p, VC[j]);           // VC = v_{k-1}
      }
      PW[j] = pack4(a, p);
    }
    dfl wk = {0.0f, 0.0f}, vk = {0.0f, 0.0f}, coef = {0.0f, 0.0f};
    if (prev) {
      loc = df_warp_sum(df_norm(loc));
      if (lane == 0) redA[wid] = loc;
      __syncthreads();
      const dfl pv = df_sum_partials(redA);
      coef = df_mul(df_mul(dfl{0.5f, 0.0f}, tau_prev), pv);
      vk = VC[k];
      wk = df_sub(hi2(PW[k]), df_mul(coef, vk));   // PW[k] is not overwritten below
    }
    // pass 2: w_{k-1} and the updated row k; sigma = sum_{j >= k+2} x_j^2
    dfl sig = {0.0f, 0.0f};
    dfl dk = {0.0f, 0.0f};
    for (int j = k + tid; j < n; j += T) {
      const float4 ap = PW[j];
      dfl x = lo2(ap);
      if (prev) {
        const dfl vj = VC[j];
        const dfl wj = (j == k) ? wk : df_sub(hi2(ap), df_mul(coef, vj));
        x = df_rank2(x, vk, wj, wk, vj);
        if (j > k) PW[j] = pack4(vj, wj);
      }
      if (j == k) {
        dk = x;
      } else {
        VC[j] = x;
        if (j >= k + 2) df_acc_mul(sig, x, x);
      }
    }
    if (last) {
      __syncthreads();
      if (blockIdx.x == 0 && tid == 0) {
        const int b = n - 1;
        dfl abb = ldcg_df(A + (size_t)b * n + b);
        if (prev) abb = df_rank2(abb, lo2(PW[b]), hi2(PW[b]), hi2(PW[b]), lo2(PW[b]));
        d[n - 2] = df_to_double(dk);
        e[n - 2] = df_to_double(VC[b]);
        d[b] = df_to_double(abb);
      }
      return;
    }
    sig = df_warp_sum(df_norm(sig));
    if (lane == 0) redB[wid] = sig;
    __syncthreads();
    // thread 0: reflector scalars (double-float: GB300's FP64 divide and square
    // root are long dependent chains) while the other warps start the product
    if (tid == 0) {
      const dfl sigma = df_sum_partials(redB);
      const dfl x1 = VC[k + 1];
      dfl beta, t, scale;
      if (sigma.hi == 0.0f) {
        beta = x1; t = dfl{0.0f, 0.0f}; scale = dfl{0.0f, 0.0f};
      } else {
        const dfl nrm = df_sqrt(df_add(df_mul(x1, x1), sigma));
        beta = (x1.hi >= 0.0f) ? df_neg(nrm) : nrm;
        t = df_mul(df_sub(beta, x1), df_recip(beta));
        scale = df_recip(df_sub(x1, beta));
      }
      s_df[0] = beta;
      s_df[1] = df_mul(t, scale);
      s_df[2] = t;
      s_df[3] = scale;
      if (blockIdx.x == 0) { d[k] = df_to_double(dk); e[k] = df_to_double(beta); tau[k] = df_to_double(t); }
    }
    // fused: pending rank-2 update (v_{k-1}, w_{k-1}) of rows/cols >= k+1 and
    // sum_j a_ij x_j over (row, segment) items
    const int R = (n - (k + 1) - (int)blockIdx.x + G - 1) / G;
    const int m1 = n - (k + 1);
    const int segw = (m1 > kDfNarrow1) ? kDfSeg : ((m1 > kDfNarrow2) ? 256 : 128);
    const int S = (m1 + segw - 1) / segw;
    if (segw == kDfSeg)
      df_items<kDfSeg, false>((float2*)A, n, k + 1 + (int)blockIdx.x, n, k, G, R, wid, lane, prev, PW, VC, part,
                            ak1s);
    else if (segw == 256)
      df_items<256, false>((float2*)A, n, k + 1 + (int)blockIdx.x, n, k, G, R, wid, lane, prev, PW, VC, part,
                            ak1s);
    else
      df_items<128, false>((float2*)A, n, k + 1 + (int)blockIdx.x, n, k, G, R, wid, lane, prev, PW, VC, part,
                            ak1s);
    __syncthreads();
    const dfl beta_df = s_df[0], ts_df = s_df[1], scale_df = s_df[3];
    tau_prev = s_df[2];
    // p_i = tau scale (sum_j a_ij x_j - beta a_{i,k+1}), segments summed as a
    // fixed tree (one warp per row while a row has at most 32 segments)
    dfl* pb = pbuf + (size_t)(k & 1) * n;
    if (S <= 32) {
      int lpr = 1;                                  // lanes per row: power of two >= S
      while (lpr < S) lpr <<= 1;
      const int rpw = 32 / lpr;                     // rows per warp
      const int sub = lane / lpr, sl = lane - sub * lpr;
      for (int r0 = wid * rpw; r0 < R; r0 += NW * rpw) {
        const int r = r0 + sub;
        dfl v = (r < R && sl < S) ? part[r * S + sl] : dfl{0.0f, 0.0f};
        for (int o = lpr >> 1; o > 0; o >>= 1) v = df_add(v, df_shfl_xor(v, o));
        if (r < R && sl == 0) pb[k + 1 + (int)blockIdx.x + r * G] = df_mul(ts_df, df_sub(v, df_mul(beta_df, ak1s[r])));
      }
    } else {
      for (int r = tid; r < R; r += T) {
        dfl* pr = part + r * S;
        for (int st = 1; st < S; st <<= 1)
          for (int sg = 0; sg + st < S; sg += 2 * st) pr[sg] = df_add(pr[sg], pr[sg + st]);
        pb[k + 1 + (int)blockIdx.x + r * G] = df_mul(ts_df, df_sub(pr[0], df_mul(beta_df, ak1s[r])));
      }
    }
    grid_arrive(bar);
    // while the other blocks finish: v_k = scale x (v_{k+1} = 1) and the
    // reflector store row k, spread over blocks
    for (int j = k + 1 + tid; j < n; j += T) {
      const dfl v = (j == k + 1) ? dfl{1.0f, 0.0f} : df_mul(VC[j], scale_df);
      VC[j] = v;
      if (j % G == (int)blockIdx.x) Vst[(size_t)k * n + j] = df_to_double_fast(v);
    }
    if (!grid_wait(bar, (unsigned)(k + 1) * (unsigned)G, status)) return;
  }
}

// The same in one thread-block cluster, for matrices that fit its shared memory: block b
// keeps rows i = b (mod G), pushes row k + 1 and its p_i into every block's shared memory
// (double-buffered by the column's parity: a buffer is rewritten two cluster barriers
// after it was filled and one after its last reader), and the cluster barrier takes the
// place of the grid's counter and polls in L2.  The blocks of a cluster are resident
// together, so there is nothing to check in or to wait for with a limit.  Same bits as
// tridiag_df_kernel.
__device__ __forceinline__ void st_cluster(void* local, int dst, float2 v) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(local)), "r"(dst));
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

__global__ void __launch_bounds__(kTriThreadsDf, 1) tridiag_cluster_kernel(int n, const double* __restrict__ F,
                                                                         double* __restrict__ Vst,
                                                                         double* __restrict__ d,
                                                                         double* __restrict__ e,
                                                                         double* __restrict__ tau, int* status) {
  extern __shared__ float4 sm4[];
  __shared__ dfl s_df[4];                    // beta, tau * scale, tau, scale
  const int G = (int)gridDim.x, rank = (int)blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  constexpr int T = kTriThreadsDf, NW = kTriThreadsDf / 32;
  const int rmax = (n - 1 + G - 1) / G;
  float4* PW = sm4;                          // n pairs
  dfl* VC = (dfl*)(sm4 + n);                 // n
  dfl* rowb = VC + n;                        // row k, 2 x n
  dfl* pbuf = rowb + 2 * n;                  // p, 2 x n
  dfl* redA = pbuf + 2 * n;                  // partials of p.v
  dfl* redB = redA + kDfRed;                 // partials of sigma
  dfl* ak1s = redB + kDfRed;                 // a_{i,k+1} of the block's rows (rmax)
  dfl* part = ak1s + rmax;                   // (row, segment) partial sums (rmax x 2)
  float2* S = (float2*)(part + 2 * rmax);    // the block's rows > 0 (rmax x n)
  if (g_barrier_ns == 0) {                   // as a wait that has no time (all blocks alike)
    if (tid == 0) atomicOr(status, (int)kStatusTimeout);
    return;
  }
  const int f0 = (rank == 0) ? G : rank;     // first row > 0 of this block
  const int R0 = (f0 < n) ? (n - 1 - f0) / G + 1 : 0;
  for (int x = tid; x < R0 * n; x += T) {
    const int r = x / n, j = x - r * n;
    const dfl a = df_from_double_bits(F[(size_t)(f0 + r * G) * n + j]);
    S[x] = make_float2(a.hi, a.lo);
  }
  for (int j = tid; j < n; j += T) rowb[j] = df_from_double_bits(F[j]);
  dfl tau_prev = {0.0f, 0.0f};               // tau_{k-1}
  // (before the first remote stores: every block of the cluster has started)
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  for (int k = 0;; ++k) {
    const bool prev = k > 0;
    const bool last = (k == n - 2);
    const dfl* pbp = pbuf + (size_t)((k + 1) & 1) * n;   // p_{k-1}
    const dfl* rowk = rowb + (size_t)(k & 1) * n;
    // pass 1: row k and p_{k-1} in one sweep of loads (kept in PW); partial p.v
    dfl loc = {0.0f, 0.0f};
#pragma unroll 4
    for (int j = k + tid; j < n; j += T) {
      const dfl a = rowk[j];
      dfl p = {0.0f, 0.0f};
      if (prev) {
        p = pbp[j];
        df_acc_mul(loc, p, VC[j]);           // VC = v_{k-1}
      }
      PW[j] = pack4(a, p);
    }
    dfl wk = {0.0f, 0.0f}, vk = {0.0f, 0.0f}, coef = {0.0f, 0.0f};
    if (prev) {
      loc = df_warp_sum(df_norm(loc));
      if (lane == 0) redA[wid] = loc;
      __syncthreads();
      const dfl pv = df_sum_partials(redA);
      coef = df_mul(df_mul(dfl{0.5f, 0.0f}, tau_prev), pv);
      vk = VC[k];
      wk = df_sub(hi2(PW[k]), df_mul(coef, vk));   // PW[k] is not overwritten below
    }
    // pass 2: w_{k-1} and the updated row k; sigma = sum_{j >= k+2} x_j^2
    dfl sig = {0.0f, 0.0f};
    dfl dk = {0.0f, 0.0f};
    for (int j = k + tid; j < n; j += T) {
      const float4 ap = PW[j];
      dfl x = lo2(ap);
      if (prev) {
        const dfl vj = VC[j];
        const dfl wj = (j == k) ? wk : df_sub(hi2(ap), df_mul(coef, vj));
        x = df_rank2(x, vk, wj, wk, vj);
        if (j > k) PW[j] = pack4(vj, wj);
      }
      if (j == k) {
        dk = x;
      } else {
        VC[j] = x;
        if (j >= k + 2) df_acc_mul(sig, x, x);
      }
    }
    if (last) {
      __syncthreads();
      if ((n - 1) % G == rank && tid == 0) {             // the owner of the last row
        const int b = n - 1;
        const float2 ab = S[(size_t)(R0 - 1) * n + b];
        dfl abb = dfl{ab.x, ab.y};
        if (prev) abb = df_rank2(abb, lo2(PW[b]), hi2(PW[b]), hi2(PW[b]), lo2(PW[b]));
        d[n - 2] = df_to_double(dk);
        e[n - 2] = df_to_double(VC[b]);
        d[b] = df_to_double(abb);
      }
      return;
    }
    sig = df_warp_sum(df_norm(sig));
    if (lane == 0) redB[wid] = sig;
    __syncthreads();
    // thread 0: reflector scalars (double-float: GB300's FP64 divide and square
    // root are long dependent chains) while the other warps start the product
    if (tid == 0) {
      const dfl sigma = df_sum_partials(redB);
      const dfl x1 = VC[k + 1];
      dfl beta, t, scale;
      if (sigma.hi == 0.0f) {
        beta = x1; t = dfl{0.0f, 0.0f}; scale = dfl{0.0f, 0.0f};
      } else {
        const dfl nrm = df_sqrt(df_add(df_mul(x1, x1), sigma));
        beta = (x1.hi >= 0.0f) ? df_neg(nrm) : nrm;
        t = df_mul(df_sub(beta, x1), df_recip(beta));
        scale = df_recip(df_sub(x1, beta));
      }
      s_df[0] = beta;
      s_df[1] = df_mul(t, scale);
      s_df[2] = t;
      s_df[3] = scale;
      if (rank == 0) { d[k] = df_to_double(dk); e[k] = df_to_double(beta); tau[k] = df_to_double(t); }
    }
    // fused: pending rank-2 update (v_{k-1}, w_{k-1}) of rows/cols >= k+1 and
    // sum_j a_ij x_j over (row, segment) items
    const int gone = (k + 1 > f0) ? (k + 1 - f0 + G - 1) / G : 0;   // rows of the list that are <= k
    const int R = max(R0 - gone, 0), first = f0 + gone * G;
    float2* Sr = S + (size_t)gone * n;
    const int m1 = n - (k + 1);
    const int segw = (m1 > kDfNarrow1) ? kDfSeg : ((m1 > kDfNarrow2) ? 256 : 128);
    const int nseg = (m1 + segw - 1) / segw;
    if (segw == kDfSeg) df_items<kDfSeg, true>(Sr, n, first, n, k, G, R, wid, lane, prev, PW, VC, part, ak1s);
    else if (segw == 256) df_items<256, true>(Sr, n, first, n, k, G, R, wid, lane, prev, PW, VC, part, ak1s);
    else df_items<128, true>(Sr, n, first, n, k, G, R, wid, lane, prev, PW, VC, part, ak1s);
    __syncthreads();
    const dfl beta_df = s_df[0], ts_df = s_df[1], scale_df = s_df[3];
    tau_prev = s_df[2];
    // row k + 1 from its owner to every block
    if (R > 0 && first == k + 1)
      for (int e = tid; e < m1 * G; e += T) {
        const int dst = e / m1, j = k + 1 + (e - dst * m1);
        st_cluster(rowb + (size_t)((k + 1) & 1) * n + j, dst, Sr[j]);
      }
    // p_i = tau scale (sum_j a_ij x_j - beta a_{i,k+1}), segments summed as a
    // fixed tree (one warp per row while a row has at most 32 segments)
    dfl* pb = pbuf + (size_t)(k & 1) * n;
    int lpr = 1;                                    // lanes per row: power of two >= S
    while (lpr < nseg) lpr <<= 1;
    const int rpw = 32 / lpr;                       // rows per warp
    const int sub = lane / lpr, sl = lane - sub * lpr;
    for (int r0 = wid * rpw; r0 < R; r0 += NW * rpw) {
      const int r = r0 + sub;
      dfl v = (r < R && sl < nseg) ? part[r * nseg + sl] : dfl{0.0f, 0.0f};
      for (int o = lpr >> 1; o > 0; o >>= 1) v = df_add(v, df_shfl_xor(v, o));
      if (r < R) {
        const dfl p = df_mul(ts_df, df_sub(v, df_mul(beta_df, ak1s[r])));
        for (int dst = sl; dst < G; dst += lpr) st_cluster(pb + first + r * G, dst, make_float2(p.hi, p.lo));
      }
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    // while the other blocks finish: v_k = scale x (v_{k+1} = 1) and the
    // reflector store row k, spread over blocks
    for (int j = k + 1 + tid; j < n; j += T) {
      const dfl v = (j == k + 1) ? dfl{1.0f, 0.0f} : df_mul(VC[j], scale_df);
      VC[j] = v;
      if (j % G == rank) Vst[(size_t)k * n + j] = df_to_double_fast(v);
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

__global__ void to_df_kernel(size_t len, const double* __restrict__ x, dfl* __restrict__ y, const unsigned* gate) {
  if (gate && *gate != 2) return;                       // for the stand-in only
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x)
    y[i] = df_from_double_bits(x[i]);
}

// ---- launch plan ----------------------------------------------------------------------
// FP64: (threads of a group, groups, columns a thread) by matrix size.  Up to 64
// columns one block does it all.  Few threads with several columns each: less to
// reduce, and the FP64 pipe is as busy (256 x 2, 3, 4 and 480 x 4 threads and columns at n =
// 343, 574, 720, 1680: 2.19, 3.95, 4.96, 24.1 ms; 128 x 3, 192 x 3, 192 x 4, 192 x 9: 1.93, 3.33,
// 4.62, 22.2), except where the rows in L2 set the time (n = 3360: 118 ms with 480 x 7, 121
// with 256 x 14).
struct TriShape {
  int n_max, ntg, rg, cpl;
  bool solo;
  const void* fn;
};
#define TRI_SHAPE(NMAX, NTG, RG, CPL, SOLO) \
  {NMAX, NTG, RG, CPL, SOLO, (const void*)tridiag_f64_kernel<NTG, RG, CPL, SOLO>}
static const TriShape kTriF64[] = {
    TRI_SHAPE(64, 64, 4, 1, true),     TRI_SHAPE(128, 128, 2, 1, false),   TRI_SHAPE(256, 128, 1, 2, false),
    TRI_SHAPE(384, 128, 1, 3, false),  TRI_SHAPE(480, 160, 1, 3, false),   TRI_SHAPE(576, 192, 1, 3, false),
    TRI_SHAPE(768, 192, 1, 4, false),  TRI_SHAPE(1120, 224, 1, 5, false),  TRI_SHAPE(1728, 192, 1, 9, false),
    TRI_SHAPE(2560, 256, 1, 10, false), TRI_SHAPE(3360, 480, 1, 7, false), TRI_SHAPE(4800, 480, 1, 10, false),
    TRI_SHAPE(10080, 480, 1, 21, false)};
constexpr size_t kTriSmemMax = 227 * 1024 - 512;       // of dynamic shared memory; the kernels have some of their own
constexpr size_t kTriSmemDf = 227 * 1024 - 48;         // the same of the double-float grid (40 bytes of its own)

struct TriLaunch {
  const void* fn = nullptr;
  int k0 = 0, k1 = 0;   // columns
  int G = 0, threads = 0, rs = 0;
  int packets = 0;      // packets per column and copy (0: none)
  size_t smem = 0;
};

// Blocks, at most one per SM.  Alone on the device 2^12 elements of the matrix
// each: fewer make the product longer than the exchange between the blocks, which
// in turn grows with their number (double-float, n = 240 / 480 / 1680: 1320, 1160,
// 1075, 1042 us with 8, 16, 31, 62 blocks / 4210, 3155, 2242, 2190, 2242 us with 8, 16,
// 62, 100, 152 / 26.5, 17.6, 12.6 ms with 31, 62, 152).  few: a grid that leaves room
// for others, 2^15 elements a block (FP64: half of the SMs at most).
static int tri_blocks(int n, int sm_count, bool df, bool few) {
  if (n <= 64) return 1;
  const int sh = few ? 15 : 12;
  const long long work = ((long long)n * n + (1LL << sh) - 1) >> sh;
  const int most = (few && !df) ? std::max(sm_count / 2, 2) : sm_count;
  return (int)std::min<long long>(std::max<long long>(work, df ? 1 : 2), most);
}

// Blocks of the cluster that does a double-float matrix, 0: none.  A column is a chain of
// 3.3 us in a cluster of up to 8 or 16 blocks and of about 5 us on a grid, until the
// rows of so few blocks take longer: n = 26, 131, 240, 300, 343: 87, 451 (8 blocks), 964, 1361,
// 1695 us (16); on a grid 139, 659, 1227, 1500, 1740 us.  16 blocks from 160 columns on:
// n = 131, 180, 240: 458, 675, 964 us, with 8 451, 702, 1049 us.
static size_t tri_cluster_smem(int n, int G) {
  const size_t rmax = (size_t)(n - 1 + G - 1) / G;
  return (7 * (size_t)n + 2 * kDfRed + 3 * rmax + rmax * n) * sizeof(dfl);
}
static cudaLaunchConfig_t tri_cluster_config(int G, size_t smem, cudaStream_t s, cudaLaunchAttribute (&at)[1]) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(kTriThreadsDf);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = G;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}
constexpr int kTriClusterMax = 320;
// Set-up, and whether a cluster of 8 and one of 16 (more than the portable size) with the shared
// memory of the largest matrix has a place on the current device (bits 0 and 1): a part of a GPU
// may have no 16 SMs that form a cluster, and a launch there would fail.
static int tri_cluster_places() {
  static PerDeviceOnce once;
  static int places[kMaxDevices];
  int dev = 0;
  if (!once_per_device(once, [] {
        const void* fn = (const void*)tridiag_cluster_kernel;
        int dev = 0, bits = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTriSmemMax) == cudaSuccess &&
            cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
          for (int k = 0; k < 2; ++k) {
            cudaLaunchAttribute at[1];
            cudaLaunchConfig_t cfg = tri_cluster_config(8 << k, tri_cluster_smem(kTriClusterMax, 8 << k), nullptr, at);
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters > 0) bits |= 1 << k;
          }
        cudaGetLastError();
        if (dev >= 0 && dev < kMaxDevices) places[dev] = bits;
        return true;
      }) ||
      cudaGetDevice(&dev) != cudaSuccess)
    return 0;
  return places[dev];
}
static int tri_cluster(int n, bool df, bool shared) {
  if (!df || shared || n < 2 || n > kTriClusterMax) return 0;
  const int places = tri_cluster_places();
  return (n > 160 && (places & 2)) ? 16 : ((places & 1) ? 8 : 0);
}
static int tri_cluster_launch(cudaStream_t s, int n, int G, const double* F, EigWork& w, int* status) {
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = tri_cluster_config(G, tri_cluster_smem(n, G), s, at);
  if (cudaLaunchKernelEx(&cfg, tridiag_cluster_kernel, n, F, w.Vst, w.d, w.e, w.tau, status) != cudaSuccess) return -2;
  count_launch();
  return 0;
}

// the FP64 launch that starts at column k0 (few: shared memory for two blocks an SM)
static TriLaunch tri_launch(int n, int k0, int sm_count, bool few) {
  TriLaunch l;
  l.k0 = k0;
  l.k1 = n - 1;
  l.G = tri_blocks(n, sm_count, false, few);
  const size_t R = (size_t)(n + l.G - 1) / l.G, row = (size_t)(n - k0 - 1) * 8;
  const TriShape* s = std::begin(kTriF64);
  while (s != std::end(kTriF64) && n > s->n_max) ++s;
  if (s == std::end(kTriF64)) return l;
  l.fn = s->fn;
  l.threads = s->ntg * s->rg + 32;
  l.packets = s->solo ? 0 : 2;
  const size_t fixed = R * 16 + (s->solo ? 2 * (size_t)n * 16 : 0) + 2 * R * 8 + 2 * (size_t)s->ntg * 8 +
                       (size_t)s->rg * (s->ntg + 4) * 8 + R * (s->ntg / 32) * 8;
  const size_t most = (few && !s->solo) ? kTriSmemMax / 2 - 1024 : kTriSmemMax;
  const int live = tri_rows(n, k0, l.G);
  const int room = (fixed < most && row > 0) ? (int)((most - fixed) / row) : 0;
  l.rs = std::min(room, live);
  // with rows outside shared memory: an eighth of the trailing matrix, after which
  // shorter rows let more of them in (a launch and the hand-over of the resident
  // rows cost about 15 us)
  if (!few && l.rs < live) l.k1 = std::min(n - 1, k0 + std::max(64, (n - k0) / 8));
  l.smem = fixed + (size_t)l.rs * row;
  return l;
}

// The opt-in dynamic shared memory, once per device, of the kernels of one precision (whatever
// the size: the limit without it, 48 KB, counts a kernel's static shared memory too).
static bool tri_attributes(bool df) {
  static PerDeviceOnce once[2];
  return once_per_device(once[df], [df] {
    auto raise = [df](const void* fn) {
      return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(df ? kTriSmemDf : kTriSmemMax)) == cudaSuccess;
    };
    bool ok = true;
    if (df) {
      ok = raise((const void*)tridiag_df_kernel<false>) && raise((const void*)tridiag_df_kernel<true>);
    } else {
      for (const TriShape& s : kTriF64) ok = ok && raise(s.fn);
    }
    if (!ok) cudaGetLastError();
    return ok;
  });
}

int eig_tridiag_weight(int n, int sm_count, bool df, bool shared) {
  if (n <= 1) return n > 0 ? 1 : 0;
  auto share = [&](const void* fn, int blocks, int threads, size_t smem) {
    int p = 0;
    if (!tri_attributes(df) || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, fn, threads, smem) != cudaSuccess || p < 1) {
      cudaGetLastError();
      p = 1;
    }
    return (int)((1000LL * blocks + p - 1) / p);
  };
  if (const int G = tri_cluster(n, df, shared)) return 1000 * G;
  if (df) {
    const int G = tri_blocks(n, sm_count, true, shared);
    return share((const void*)tridiag_df_kernel<false>, G, kTriThreadsDf, tridiag_smem_df(n, G));
  }
  int weight = 1;
  for (int k0 = 0; k0 < n - 1;) {
    const TriLaunch l = tri_launch(n, k0, sm_count, shared);
    if (!l.fn) break;
    weight = std::max(weight, share(l.fn, l.G, l.threads, l.smem));
    k0 = l.k1;
  }
  return weight;
}

__global__ void tri_one_kernel(const double* F, double* d) { d[0] = F[0]; }

int eig_tridiagonalize(cudaStream_t s, int n, const double* F, EigWork& w, int* status, int sm_count, bool df,
                       bool shared, int own) {
  // (two steps of n = 1680 together, mixed: 42.5 ms with the large grids, 33.4 with the small ones, eight
  // of 480 14.3 and 10.7; two and four of 480, a demand of 0.75 and 1.5: 5.1 and 7.7, 7.0 and 8.0.  In
  // FP64 the small grids are no gain: two of 1680 79 and 75, of 2160 141 and 164)
  int crowd = 1500 * sm_count - own;
  if (n <= 0) return 0;
  cudaMemsetAsync(w.e, 0, (size_t)n * sizeof(double), s);
  cudaMemsetAsync(w.Vst, 0, (size_t)n * n * sizeof(double), s);               // entries left of the reflectors
  if (n == 1 && !df) {
    tri_one_kernel<<<1, 1, 0, s>>>(F, w.d);
    count_launch();
    return 0;
  }
  if (const int G = tri_cluster(n, df, shared)) return tri_cluster_launch(s, n, G, F, w, status);
  if (df) {
    const size_t nn2 = (size_t)n * n;
    const int few = tri_blocks(n, sm_count, true, true), G = shared ? few : tri_blocks(n, sm_count, true, false);
    // (a grid no larger than the stand-in's needs none)
    for (int role = (G > few) ? 1 : 0;;) {
      const int blocks = (role == 2) ? few : G;
      const size_t smem = tridiag_smem_df(n, blocks);
      if (smem > kTriSmemDf || !tri_attributes(true)) return -1;
      to_df_kernel<<<(unsigned)std::min<size_t>((nn2 + 255) / 256, 8 * (size_t)sm_count), 256, 0, s>>>(
          nn2, F, (dfl*)w.A, role == 2 ? w.bar + 3 : nullptr);
      count_launch();
      cudaMemsetAsync(w.bar, 0, (role == 2 ? 2 : 4) * sizeof(unsigned), s);
      int nn = n, rmax = tridiag_df_rmax(n, blocks);
      dfl *A = (dfl*)w.A, *pb = (dfl*)w.pbuf;
      double *V = w.Vst, *d = w.d, *e = w.e, *t = w.tau;
      unsigned* bar = w.bar;
      void* args[] = {&nn, &A, &V, &d, &e, &t, &pb, &bar, &status, &rmax, &role, &crowd};
      const void* fn = role ? (const void*)tridiag_df_kernel<true> : (const void*)tridiag_df_kernel<false>;
      if (cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kTriThreadsDf), args, smem, s) != cudaSuccess)
        return -2;
      count_launch();
      if (role != 1) break;
      role = 2;
    }
    return 0;
  }
  if (!tri_attributes(false)) return -1;
  // The packets are in the inverse-iteration workspace (at least 5 n^2 doubles, free
  // until then; n > 64 here, a single block has none).  0xFF: of the parity that is
  // not the first use's.
  const int blocks = tri_blocks(n, sm_count, false, shared);
  int reps = 1;
  while (reps < 16 && 8 * reps < blocks) reps *= 2;
  Packet* pk = (Packet*)w.lu;
  for (int k0 = 0; k0 < n - 1;) {
    const TriLaunch l = tri_launch(n, k0, sm_count, shared);
    if (!l.fn) return -1;
    if (k0 == 0 && l.packets) cudaMemsetAsync(pk, 0xFF, (size_t)reps * l.packets * n * sizeof(Packet), s);
    TriArgs a{n, l.k0, l.k1, l.rs, reps, k0 == 0 ? F : nullptr, w.A, w.bar, (l.G == 1 || shared) ? 0 : 1,
              w.Vst, w.d, w.e, w.tau, pk, w.Wt, status};
    void* args[] = {&a};
    if (a.role) cudaMemsetAsync(w.bar, 0, 2 * sizeof(unsigned), s);
    if (cudaLaunchCooperativeKernel(l.fn, dim3(l.G), dim3(l.threads), args, l.smem, s) != cudaSuccess) return -2;
    count_launch();
    if (a.role) {
      const TriLaunch f = tri_launch(n, k0, sm_count, true);       // the stand-in
      a.role = 2;
      a.rs = f.rs;
      if (cudaLaunchCooperativeKernel(f.fn, dim3(f.G), dim3(f.threads), args, f.smem, s) != cudaSuccess) return -2;
      count_launch();
    }
    k0 = l.k1;
  }
  return 0;
}

}  // namespace kx
