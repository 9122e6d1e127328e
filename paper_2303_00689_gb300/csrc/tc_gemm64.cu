// FP64 matrix products on the tensor cores (sm_103a, tcgen05 + TMA): the n^3 work of
// the FP64 path (density, DMPT, back-transformation).
//
// C = alpha A B^T + beta C with every operand cut, per row, into eight balanced
// base-256 digits of the 63-bit integer round(x 2^(63 - e)), 2^e > max |row| (a splitting
// whose products are free of rounding errors: Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 2012).
// A product of two digits is an integer of at most 2^14, and the eight or fewer
// digit pairs of one weight 2^-8d (d = a + b < 8), summed over 128 columns, stay
// within 2^24: exact in the FP32 accumulator of the tensor core.  Eight
// accumulators, one per weight, are folded every 128 columns into two 64-bit
// integers, and the 36 kept pairs end as one integer hi 2^32 + lo that is rounded
// once to FP64.  What is left out (pairs with d >= 8 and the digits below 2^-63 of
// the row maximum) is under K 2^-60 of the product of the row maxima.  Where the terms
// a_ik b_jk come near that product for some k, the result is nearer to the exact product than
// K FP64 additions are; where they do not (two rows whose large elements stand in different
// columns) the error is relative to the row maxima all the same, not to sum |a||b|.  The
// operands here are orthogonal matrices and what is made of them, whose elements are known to
// 2^-53 of the row's norm at best, so that a product carries 2^-53 of the norms from them.
// Density between two fragments of 16 H atoms 10, 14 and 18 Angstrom apart (elements 1e-9,
// 2e-13, 3e-17): error 8e-17, 3e-18, 4e-20, of which the product 6e-20, 5e-20, 4e-20; with
// products on the FP64 pipe 5e-17, 3e-18, 4e-19.
//
// GB300 does 2 FP64 FMAs a clock and SM, 4096 BF16 ones: 36 digit products are far
// cheaper than one FP64 product (n = 26, 240, 574, 1680: 17, 43, 76, 568 us
// and 5 to 19 us a cut instead of 39, 280, 665, 8470 us; rms error at 1680 0.014 instead
// of 0.40 units of 2^-53 sum |a||b|).
// A CTA computes 128 x 64 (eight accumulators of 64 columns are all of the tensor
// memory), 18 warps: TMA producer, MMA issuer, 16 epilogue warps of 32 rows x 16
// columns.  A stage holds the eight digits of A and B of 32 columns (96 KB, two
// stages); its 36 x 2 products are issued weight by weight, so that the epilogue
// folds one weight of a finished chunk while the products of the next ones run.  The
// rounding uses integer instructions only: on the FP64 pipe it would take 8 us a tile.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "tc_gemm.h"
#include "tc_ptx.cuh"

namespace kx {

constexpr int k64S = kTc64Slices;
constexpr int k64BM = 128, k64BN = 64, k64BK = 32, k64Stages = 2;
constexpr int k64ChunkTiles = 4;                                  // 128 columns: exact in FP32
constexpr int k64TileA = k64BM * k64BK * 2, k64TileB = k64BN * k64BK * 2;
constexpr int k64StageBytes = k64S * (k64TileA + k64TileB);
constexpr int k64Smem = k64Stages * k64StageBytes + 1024 + 512;
constexpr int k64EpiWarps = 16, k64Threads = 32 * (2 + k64EpiWarps);
constexpr int k64LdT = k64BN + 1;                                 // output tile row in shared memory
constexpr int kNonFinite = 1025;                                  // row exponent of a row with an inf or NaN
static_assert(k64BM * k64LdT * 8 <= k64Stages * k64StageBytes, "output tile fits the stages");
static_assert(k64S * k64BN <= 512, "the accumulators fit the tensor memory");
static_assert(k64S * k64ChunkTiles * k64BK * 16384 <= 1 << 24, "a chunk's sum is exact in FP32");

// (hi 2^32 + lo) 2^k rounded to nearest even
__device__ __forceinline__ double round_product(long long hi, long long lo, int k) {
  const __int128 t = ((__int128)hi << 32) + lo;
  const bool neg = t < 0;
  unsigned __int128 m = neg ? -(unsigned __int128)t : (unsigned __int128)t;
  const unsigned long long mh = (unsigned long long)(m >> 64);
  if (m == 0) return 0.0;
  const int lz = mh ? __clzll((long long)mh) : 64 + __clzll((long long)(unsigned long long)m);
  m <<= lz;
  const unsigned long long top = (unsigned long long)(m >> 64), rest = (unsigned long long)m;
  const unsigned long long mant = top >> 11, rem = top & 0x7FF;   // 53 bits and what is below
  const bool up = rem > 0x400 || (rem == 0x400 && (rest != 0 || (mant & 1)));
  const int be = 1023 + 127 - lz + k;                             // biased exponent
  if (be >= 1 && be <= 2045) {
    const unsigned long long b = ((unsigned long long)(be - 1) << 52) + mant + (up ? 1 : 0);
    return __longlong_as_double((long long)(b | (neg ? 1ULL << 63 : 0)));
  }
  const double v = ldexp((double)(long long)(mant + (up ? 1 : 0)), be - 1075);
  return neg ? -v : v;
}

struct Gemm64Args {
  CUtensorMap a, b;            // digits stacked: rows_a * 8 and rows_b * 8 rows
  const int *exa, *exb;        // row exponents
  int rows_a, rows_b;          // rows of one digit
  int a0, b0;                  // first row of the operand used
  int bx;                      // column of B - column of A
  int kt0, kt1;                // 32-column tiles
  int M, N;
  double alpha;
  int beta;
  double* C;
  int ldc, sym;
  int diag;                    // > 0: only the diagonal blocks of this size, block after block in C
  int* err;
  const int* gate;
};

__global__ void __launch_bounds__(k64Threads, 1) tc_gemm64_kernel(const __grid_constant__ Gemm64Args g) {
  if (g.gate && *g.gate == 0) return;      // whole CTA, before any barrier or TMEM use
  const int bi = blockIdx.y, bj = g.diag ? bi * (g.diag / k64BN) + blockIdx.x : blockIdx.x;
  const int m0 = bi * k64BM, n0 = bj * k64BN;
  if (n0 >= g.N || (g.sym && m0 >= n0 + k64BN)) return;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(base + k64Stages * k64StageBytes);
  uint64_t* empty = full + k64Stages;
  uint64_t* acc_full = empty + k64Stages;
  uint64_t* acc_empty = acc_full + k64S;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + k64S);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ktiles = g.kt1 - g.kt0;
  int* err = g.err;
  double* C = g.C;
  if (g.diag) C += (ptrdiff_t)bi * g.diag * g.ldc - ((ptrdiff_t)m0 * g.ldc + m0);

  if (threadIdx.x == 0) {
    for (int st = 0; st < k64Stages; ++st) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], 1);
    }
    for (int d = 0; d < k64S; ++d) {
      mbar_init(&acc_full[d], 1);
      mbar_init(&acc_empty[d], k64EpiWarps);
    }
    mbar_fence_init();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      bool ok = true;
      for (int it = 0; it < ktiles; ++it) {
        const int st = it % k64Stages;
        if (!mbar_wait(&empty[st], ((uint32_t)(it / k64Stages) & 1u) ^ 1u, err)) { ok = false; break; }
        uint8_t* sa = base + st * k64StageBytes;
        uint8_t* sb = sa + k64S * k64TileA;
        mbar_expect_tx(&full[st], k64StageBytes);
        const int x = (g.kt0 + it) * k64BK;
#pragma unroll
        for (int a = 0; a < k64S; ++a) {
          tma_load_2d(sa + a * k64TileA, &g.a, &full[st], x, a * g.rows_a + g.a0 + m0);
          tma_load_2d(sb + a * k64TileB, &g.b, &full[st], x + g.bx, a * g.rows_b + g.b0 + n0);
        }
        issued = it + 1;
      }
      if (!ok) {
        // let our own copies land before the CTA can exit
        for (int it = (issued > k64Stages ? issued - k64Stages : 0); it < issued; ++it)
          for (long long w = 0; w < kWaitLimit && !mbar_try(&full[it % k64Stages], (uint32_t)(it / k64Stages) & 1u);
               ++w) {
          }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = make_idesc(k64BM, k64BN);
      bool ok = true;
      for (int it = 0; it < ktiles && ok; ++it) {
        const int st = it % k64Stages, chunk = it / k64ChunkTiles;
        const bool first = it % k64ChunkTiles == 0;
        const bool last = it % k64ChunkTiles == k64ChunkTiles - 1 || it == ktiles - 1;
        if (!mbar_wait(&full[st], (uint32_t)(it / k64Stages) & 1u, err)) break;
        tc_fence_after();
        // unrolled, with the descriptors of the stage as bases: one thread issues, and address
        // arithmetic between the products (a dependent chain) costs more than they take
        const uint32_t sa = smem_u32(base + st * k64StageBytes);
        const uint64_t da = smem_desc_sw64(sa), db = smem_desc_sw64(sa + k64S * k64TileA);
#pragma unroll
        for (int d = 0; d < k64S; ++d) {
          if (first && ok) {
            ok = mbar_wait(&acc_empty[d], ((uint32_t)chunk & 1u) ^ 1u, err);
            tc_fence_after();
          }
          if (!ok) break;
#pragma unroll
          for (int a = 0; a <= d; ++a)
#pragma unroll
            for (int k = 0; k < k64BK / 16; ++k)
              umma_bf16(tmem + (uint32_t)(d * k64BN), da + (uint64_t)((a * k64TileA + k * 32) >> 4),
                        db + (uint64_t)(((d - a) * k64TileB + k * 32) >> 4), idesc,
                        (a == 0 && k == 0) ? (first ? 0u : 1u) : 1u);
          if (last) umma_commit(&acc_full[d]);
        }
        umma_commit(&empty[st]);
      }
    }
  } else {
    const int quarter = warp & 3, cg = (warp - 2) >> 2;      // TMEM lanes 32 quarter .., columns 16 cg ..
    long long hi[16], lo[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) { hi[j] = 0; lo[j] = 0; }
    const bool live = m0 + quarter * 32 < g.M && n0 + cg * 16 < g.N;   // (else the warp only keeps the pipeline going)
    bool ok = true;
    const int nchunks = (ktiles + k64ChunkTiles - 1) / k64ChunkTiles;
    for (int c = 0; c < nchunks && ok; ++c) {
#pragma unroll
      for (int d = 0; d < k64S; ++d) {
        if (ok) {
          bool got = mbar_wait(&acc_full[d], (uint32_t)c & 1u, err);
          ok = __all_sync(0xffffffffu, got);
        }
        if (ok && live) {
          tc_fence_after();
          uint32_t r[16];
          tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(d * k64BN + cg * 16), r);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const long long v = __float2int_rn(__uint_as_float(r[j]));
            if (d < 4)
              hi[j] += v * (1ll << (8 * (3 - d)));
            else
              lo[j] += v * (1ll << (8 * (7 - d)));
          }
          tc_fence_before();
          __syncwarp();
        }
        if (ok && lane == 0) mbar_arrive(&acc_empty[d]);
      }
    }
    double* tile = (double*)base;      // every product is done and every copy has landed by now
    if (ok && live) {
      const int rl = quarter * 32 + lane, row = m0 + rl;
      const int ea = row < g.M ? g.exa[g.a0 + row] : 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int cl = cg * 16 + j, col = n0 + cl;
        const int eb = col < g.N ? g.exb[g.b0 + col] : 0;
        double v = round_product(hi[j], lo[j], ea + eb - 2 * 63 + 56);
        if (ea == kNonFinite || eb == kNonFinite) v = __longlong_as_double(0x7FF8000000000000LL);
        tile[rl * k64LdT + cl] = g.alpha == 1.0 ? v : (g.alpha == -1.0 ? -v : g.alpha * v);
      }
    }
    asm volatile("bar.sync 1, %0;" ::"r"(k64EpiWarps * 32) : "memory");
    if (*(volatile int*)err == 0) {
      const int t = threadIdx.x - 64;
      for (int idx = t; idx < k64BM * k64BN; idx += k64EpiWarps * 32) {
        const int rr = idx / k64BN, cc = idx % k64BN, row = m0 + rr, col = n0 + cc;
        if (row < g.M && col < g.N && !(g.sym && row > col)) {
          double* p = C + (ptrdiff_t)row * g.ldc + col;
          *p = g.beta ? *p + tile[rr * k64LdT + cc] : tile[rr * k64LdT + cc];
        }
      }
      if (g.sym)
        for (int idx = t; idx < k64BM * k64BN; idx += k64EpiWarps * 32) {
          const int rr = idx % k64BM, cc = idx / k64BM, row = m0 + rr, col = n0 + cc;
          if (row < g.M && col < g.N && row < col) {
            double* p = C + (ptrdiff_t)col * g.ldc + row;
            *p = g.beta ? *p + tile[rr * k64LdT + cc] : tile[rr * k64LdT + cc];
          }
        }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ---- cutting ---------------------------------------------------------------------------

// balanced base-256 digits of round(x 2^(63 - e)), most significant first, |x| < 2^e
__device__ __forceinline__ void digits64(double x, int e, int (&dig)[k64S]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF);
  unsigned long long M = b & 0xFFFFFFFFFFFFFULL;
  if (E != 0) M |= 1ULL << 52;
  const int sh = (E != 0 ? E : 1) - 1075 + 63 - e;              // x < 2^e: what is shifted left stays below 2^63
  unsigned long long mag = 0;
  if (e != kNonFinite) {
    if (sh >= 0)
      mag = M << min(sh, 63);
    else if (sh > -56)
      mag = (M + (1ULL << (-sh - 1))) >> -sh;
  }
  long long X = (b >> 63) ? -(long long)mag : (long long)mag;
#pragma unroll
  for (int a = k64S - 1; a > 0; --a) {
    const int r = (int)(signed char)(X & 0xFF);
    dig[a] = r;
    X = (X - r) >> 8;
  }
  dig[0] = (int)X;
}

// the digits of four consecutive columns, one 8-byte store per digit
__device__ __forceinline__ void store_digits4(const double (&x)[4], int e, __nv_bfloat16* __restrict__ p,
                                              size_t stride) {
  int d[4][k64S];
#pragma unroll
  for (int c = 0; c < 4; ++c) digits64(x[c], e, d[c]);
#pragma unroll
  for (int a = 0; a < k64S; ++a) {
    __nv_bfloat162 v[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      v[c].x = __float2bfloat16_rn((float)d[2 * c][a]);
      v[c].y = __float2bfloat16_rn((float)d[2 * c + 1][a]);
    }
    *(uint2*)(p + a * stride) = *(uint2*)v;
  }
}

// a block per row: columns [c0, cols) of X, zeros up to ld
constexpr int kCutThreads = 128;
__global__ void __launch_bounds__(kCutThreads) cut64_rows_kernel(Tc64Op op, int c0, int cols,
                                                                 const double* __restrict__ X, size_t ldx,
                                                                 const int* gate) {
  if (gate && *gate == 0) return;
  __shared__ unsigned long long s_max[kCutThreads / 32];
  const int r = blockIdx.x, tid = threadIdx.x;
  const double* x = X + (size_t)r * ldx;
  unsigned long long m = 0;
  for (int k = c0 + tid; k < cols; k += kCutThreads)
    m = max(m, (unsigned long long)__double_as_longlong(x[k]) & 0x7FFFFFFFFFFFFFFFULL);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((tid & 31) == 0) s_max[tid >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kCutThreads / 32; ++w) m = max(m, s_max[w]);
  const int e = exponent_of_max(m);
  if (tid == 0) op.ex[r] = e;
  for (int k = c0 + 4 * tid; k < op.ld; k += 4 * kCutThreads) {
    double v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = (k + c < cols) ? x[k + c] : 0.0;
    store_digits4(v, e, op.p + (size_t)r * op.ld + k, (size_t)op.rows * op.ld);
  }
}

// rows of X^T (X has `cols` rows): a block per sixteen rows, tiles of 64 columns
// through shared memory so that loads and stores are whole 128-byte lines
constexpr int kCutT = 16, kCutK = 64;
__global__ void __launch_bounds__(256) cut64_cols_kernel(Tc64Op op, int cols, const double* __restrict__ X, size_t ldx,
                                                         const int* gate) {
  if (gate && *gate == 0) return;
  __shared__ double tile[kCutK][kCutT + 1];
  __shared__ unsigned long long s_max[kCutT][kCutT];
  const int tid = threadIdx.x, cx = tid % kCutT, ky = tid / kCutT;
  const int r0 = blockIdx.x * kCutT, r = r0 + cx;
  unsigned long long m = 0;
  if (r < op.rows)
    for (int k = ky; k < cols; k += 256 / kCutT)
      m = max(m, (unsigned long long)__double_as_longlong(X[(size_t)k * ldx + r]) & 0x7FFFFFFFFFFFFFFFULL);
  s_max[ky][cx] = m;
  __syncthreads();
  m = 0;
#pragma unroll
  for (int q = 0; q < kCutT; ++q) m = max(m, s_max[q][ky]);      // of row r0 + ky, which this thread cuts
  const int e = exponent_of_max(m);
  if (cx == 0 && r0 + ky < op.rows) op.ex[r0 + ky] = e;
  for (int k0 = 0; k0 < op.ld; k0 += kCutK) {
    __syncthreads();
    for (int k = ky; k < kCutK; k += 256 / kCutT)
      tile[k][cx] = (r < op.rows && k0 + k < cols) ? X[(size_t)(k0 + k) * ldx + r] : 0.0;
    __syncthreads();
    if (r0 + ky < op.rows) {
      double v[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = tile[4 * cx + c][ky];
      store_digits4(v, e, op.p + (size_t)(r0 + ky) * op.ld + k0 + 4 * cx, (size_t)op.rows * op.ld);
    }
  }
}

// ---- host ------------------------------------------------------------------------------

size_t tc64_op_bytes(int rows, int cols) {
  const size_t digits = (size_t)k64S * rows * tc_ld(cols) * 2;
  return ((digits + 255) & ~(size_t)255) + (((size_t)rows * sizeof(int) + 255) & ~(size_t)255);
}

Tc64Op tc64_op(void* base, int rows, int cols) {
  Tc64Op op;
  op.p = (__nv_bfloat16*)base;
  op.rows = rows;
  op.ld = tc_ld(cols);
  op.ex = (int*)((char*)base + (((size_t)k64S * rows * op.ld * 2 + 255) & ~(size_t)255));
  return op;
}

bool tc64_work_bind(Tc64Work& w, char* const (&op)[3], int* err, int n, cudaStream_t s) {
  for (int k = 0; k < 3; ++k) w.op[k] = op[k];
  w.err = err;
  w.n = n;
  const Tc64Op first = tc64_slot(w, 0, n, n);
  CUtensorMap m;
  return cudaMemsetAsync(w.err, 0, sizeof(int), s) == cudaSuccess &&
         tc_encode_map_box(&m, first.p, k64S * first.rows, first.ld, first.ld, k64BK, k64BM);
}

Tc64Op tc64_slot(const Tc64Work& w, int slot, int rows, int cols) { return tc64_op(w.op[slot], rows, cols); }

void tc64_cut_rows(cudaStream_t s, const Tc64Op& op, int c0, int cols, const double* X, size_t ldx, const int* gate) {
  cut64_rows_kernel<<<op.rows, kCutThreads, 0, s>>>(op, c0, cols, X, ldx, gate);
  count_launch();
}

void tc64_cut_cols(cudaStream_t s, const Tc64Op& op, int cols, const double* X, size_t ldx, const int* gate) {
  cut64_cols_kernel<<<(op.rows + kCutT - 1) / kCutT, 256, 0, s>>>(op, cols, X, ldx, gate);
  count_launch();
}

int tc64_gemm(cudaStream_t s, int M, int N, int k0, int k1, const Tc64Op& A, int a0, const Tc64Op& B, int b0, int bx,
              double alpha, int beta, double* C, int ldc, int sym, int diag, int* err, const int* gate) {
  if (M <= 0 || N <= 0) return 0;
  static PerDeviceOnce once;
  if (!once_per_device(once, [] {
        return cudaFuncSetAttribute(tc_gemm64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, k64Smem) ==
               cudaSuccess;
      }))
    return -1;
  Gemm64Args g;
  if (!tc_encode_map_box(&g.a, A.p, k64S * A.rows, A.ld, A.ld, k64BK, k64BM) ||
      !tc_encode_map_box(&g.b, B.p, k64S * B.rows, B.ld, B.ld, k64BK, k64BN))
    return -1;
  g.exa = A.ex; g.exb = B.ex;
  g.rows_a = A.rows; g.rows_b = B.rows;
  g.a0 = a0; g.b0 = b0; g.bx = bx;
  g.kt0 = k0 / k64BK; g.kt1 = (k1 + k64BK - 1) / k64BK;
  g.M = M; g.N = N;
  g.alpha = alpha; g.beta = beta;
  g.C = C; g.ldc = ldc; g.sym = sym; g.diag = diag;
  g.err = err; g.gate = gate;
  const dim3 grid(diag ? diag / k64BN : (N + k64BN - 1) / k64BN, (M + k64BM - 1) / k64BM);
  tc_gemm64_kernel<<<grid, k64Threads, k64Smem, s>>>(g);
  count_launch();
  return 0;
}

}  // namespace kx
