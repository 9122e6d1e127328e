// Tensor-core (tcgen05) GEMMs for the mixed-precision path (internal header).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace kx {

// slots of BF16 slice matrices (each holds up to kTcMaxSlices slices of one n x n operand)
constexpr int kTcPieceSlots = 6;
constexpr int kTcMaxSlices = 4;
enum TcSlot { kSlotQs = 0, kSlotQ = 1, kSlotQt = 2, kSlotT0 = 3, kSlotT1 = 4, kSlotSpare = 5 };

struct TcWork {
  void* base = nullptr;   // host-side bookkeeping (tensor maps, piece pointers)
  bool wide = false;      // beside other handles: wide tiles, the least work
  size_t bytes = 0;
};
size_t tc_work_bytes(int n);
void tc_work_bind(TcWork& w, void* device_base, int n);
void tc_work_release(TcWork& w);
bool tc_available();                  // driver entry point for tensor maps present
bool tc_ready(const TcWork& w);       // tensor maps encoded for this handle
int* tc_error_flag(const TcWork& w);  // device word set when a bounded wait expired
// X (n x n FP64) -> `slices` fixed-point BF16 slices in slot (transpose != 0 slices X^T)
// gate (nullable device int): the kernels return at once when *gate == 0
void tc_split(cudaStream_t s, const TcWork& w, int slot, const double* X, int slices, int transpose,
              const int* gate = nullptr);
// C = alpha * sum over `terms` (1, 3, 6 or 10 for 1-4 slices) slice products A_a B_b^T
void tc_gemm(cudaStream_t s, const TcWork& w, int slotA, int slotB, int terms, double alpha, double* C,
             int sym, const int* gate = nullptr);

// The DMPT's 3-slice product (terms 6) with all slices of a k-tile staged together:
// the weight-1 slice product summed exactly per 512-K chunk, the lower-weight ones
// in FP32; within 2^-26 of sum |a||b| of the exact 6-term slice product
void tc_gemm_grouped(cudaStream_t s, const TcWork& w, int slotA, int slotB, double alpha, double* C, int sym,
                     const int* gate = nullptr);
// the 4-slice product (terms 10) the same way (density product): within ~2^-28 of
// sum |a||b| of the exact 10-term slice product
void tc_gemm_grouped4(cudaStream_t s, const TcWork& w, int slotA, int slotB, double alpha, double* C, int sym,
                      const int* gate = nullptr);
// general shapes with 4 slices (back-transformation): C (M x N, ldc) = alpha A B^T (+ C if beta),
// slice a of A's rows at Abase + a astride (row length lda), of B's likewise; < 0 on a tensor-map error
int tc_gemm_grouped_rc(cudaStream_t s, int M, int N, int K, const __nv_bfloat16* Abase, int lda, size_t astride,
                       const __nv_bfloat16* Bbase, int ldb, size_t bstride, double alpha, double* C, int ldc,
                       int beta, int* err, bool wide);
// split-K, whole exact-sum chunks a part: returns the number of parts z used (partials at P + z M ldp)
int tc_gemm_grouped_rc_splitk(cudaStream_t s, int M, int N, int K, const __nv_bfloat16* Abase, int lda,
                              size_t astride, const __nv_bfloat16* Bbase, int ldb, size_t bstride, double alpha,
                              double* P, int ldp, int splits, int* err, bool wide);

// Building blocks on caller-provided buffers (used by the allocation-free entry point)
int tc_ld(int n);                                                   // padded slice row length
bool tc_encode_map(CUtensorMap* m, void* ptr, int n, int ld);       // BF16 slice tensor map
// the slices of both operands in one launch, which clears *err
void tc_split_pair(cudaStream_t s, int n, int ld, const double* A, const double* B, int slices, int* exA, int* exB,
                   __nv_bfloat16* a, __nv_bfloat16* b, size_t stride, int* err);
void tc_gemm_on_maps(cudaStream_t s, int n, const CUtensorMap* mapsA, const CUtensorMap* mapsB, int terms,
                     double alpha, double* C, int sym, int* err);

// one-pass row slicing (row maximum and slices per warp), columns cols..ld-1 zero
void tc_split_rows(cudaStream_t s, int rows, int cols, const double* X, long long ldx, int slices,
                   __nv_bfloat16* base, int ld, size_t stride);
// all reflector blocks at once: mode 0 slices V_b (kb x m_b, rows of the reflector
// store from column b kblk + 1, row length tc_ld(m_b)), mode 1 slices Y_b^T (m_b x kb,
// src + b n kblk, row length kblk); block b at base + b blk_stride, slices slice_stride apart
void tc_split_blocks(cudaStream_t s, int mode, int n, int nref, int kblk, const double* src, __nv_bfloat16* base,
                     size_t blk_stride, size_t slice_stride, int slices);
// sum of `parts` partial products (rows x cols <= 128, at P + z rows ldp) and its slices
void tc_reduce_split_rows(cudaStream_t s, int rows, int cols, const double* P, int parts, int ldp, int slices,
                          __nv_bfloat16* base, int ld, size_t stride);
// test of the pipeline's bounded mbarrier wait: sets *err when `limit` tries expire
void tc_mbar_expiry(cudaStream_t s, int* err, long long limit);
bool tc_encode_map_box(CUtensorMap* m, void* ptr, int rows, int cols, int ld, int bk, int box_rows);

// FP64 products (tc_gemm64.cu): an operand's rows cut into eight digits each
constexpr int kTc64Slices = 8;
struct Tc64Op {
  __nv_bfloat16* p = nullptr;   // digit a of row r at p + (a rows + r) ld
  int* ex = nullptr;            // row exponents
  int rows = 0, ld = 0;
};
size_t tc64_op_bytes(int rows, int cols);              // a multiple of 256
Tc64Op tc64_op(void* base, int rows, int cols);        // base 256-byte aligned
// the device buffers of an FP64 handle: three operands of n x n (in its eigensolver workspace) and an error word
struct Tc64Work {
  char* op[3] = {};
  int* err = nullptr;
  int n = 0;
};
// clears the error word on the stream of the handle; false: no tensor map of this size
bool tc64_work_bind(Tc64Work& w, char* const (&op)[3], int* err, int n, cudaStream_t s);
Tc64Op tc64_slot(const Tc64Work& w, int slot, int rows, int cols);
// columns [c0, cols) of the rows of X (c0 a multiple of 32); the rows of X^T, X of `cols` rows
void tc64_cut_rows(cudaStream_t s, const Tc64Op& op, int c0, int cols, const double* X, size_t ldx,
                   const int* gate = nullptr);
void tc64_cut_cols(cudaStream_t s, const Tc64Op& op, int cols, const double* X, size_t ldx, const int* gate = nullptr);
// C (M x N) = alpha A B^T (+ C if beta) over the columns k0 (a multiple of 32) to k1 of
// rows a0 .. of A and b0 .. of B (there bx, a multiple of 32, columns on), zeros in both from k1 to the next multiple of 32;
// diag (a multiple of 128): the diagonal blocks of that size only, one after the
// other at C (ldc = diag); < 0 on a tensor-map error
int tc64_gemm(cudaStream_t s, int M, int N, int k0, int k1, const Tc64Op& A, int a0, const Tc64Op& B, int b0, int bx,
              double alpha, int beta, double* C, int ldc, int sym, int diag, int* err, const int* gate = nullptr);

// raw access to a slot's slice buffers (for the back-transformation)
__nv_bfloat16* tc_slot_base(const TcWork& w, int slot);
size_t tc_slot_stride(const TcWork& w);

}  // namespace kx
