// tcgen05 tensor-core GEMM for sm_103a (internal):  C[M x N] (+)= A[M x K] * B[N x K]^T
//
// A and B are K-major (row-major with K contiguous) in bf16 or fp32-as-tf32, K padded to a multiple
// of the 128-byte k-block. A persistent grid (at most one CTA per SM) walks the 128 x 256 output
// tiles (x K splits); each tile is accumulated in TMEM by tcgen05.mma issued from one thread, with
// two 256-column accumulators so that the epilogue of one tile overlaps the MMAs of the next;
// operands are staged by TMA (cp.async.bulk.tensor, 128-byte swizzle) through a 4-stage mbarrier
// pipeline; the epilogue warps read TMEM with tcgen05.ld and write FP32 rows. K splits write
// partial results at C + z * split_stride.
#pragma once
#include "gfcc_internal.cuh"

#include <algorithm>

namespace gfcc {

enum class TcKind { BF16 = 0, TF32 = 1, F16 = 2 };   // F16: exact-slice digits only

struct TcOperand {
  const void* ptr = nullptr;   // device, row-major
  long long rows = 0;          // logical rows (TMA zero-fills beyond)
  long long k_pad = 0;         // K extent in elements (multiple of the k-block)
  long long ld = 0;            // row stride in elements (0: k_pad); multiple of the k-block
  TcOperand() = default;
  TcOperand(const void* p, long long r, long long k, long long l = 0) : ptr(p), rows(r), k_pad(k), ld(l ? l : k) {}
};

// Launch C = A B^T (beta = 0) or C += A B^T (beta = 1). C is FP32 row-major with leading dimension
// ldc; rows >= M and columns >= N are not written. ksplit > 1 splits K into equal k-block ranges and
// writes partial tiles to C + z * split_stride (beta must be 0 then).
// prof_class / k_alg: profiling class of the launch and the unpadded K for its algorithmic flop count
// (0: the padded K).
void tc_gemm(TcKind kind, const TcOperand& A, const TcOperand& B, float* C, long long ldc, long long M,
             long long N, int beta, int ksplit, long long split_stride, int* err_dev, cudaStream_t s,
             int prof_class = 0, long long k_alg = 0);

// Independent products of one launch (see TcGroup in tc_gemm.cu): the arguments of tc_gemm for each.
constexpr int TC_MAX_GROUPS = 8, TC_MAX_MAPS = 3;
struct TcProduct {
  TcOperand A, B;
  float* C = nullptr;
  long long ldc = 0, M = 0, N = 0;
  int beta = 0, ksplit = 1;
  long long split_stride = 0, k_alg = 0;
};
void tc_gemm_group(TcKind kind, const TcProduct* pr, int n, int* err_dev, cudaStream_t s, int prof_class = 0);

// Exact integer GEMMs for the slices of ozaki.cuh: A and B f16 holding integers of magnitude <= 256, so
// that 256 products (TC_EXACT_CHUNK_KB k-blocks) sum exactly in FP32. For every group,
// P[z][m][n] (int32, row stride ldp, split z at P + z * split_stride) = sum over the k-blocks of split z of
// A[m][kA + k] B[n][kB + k], k < k_pad, in splits of nk_split <= TC_EXACT_MAX_KB k-blocks (|sum| < 2^31); rows
// >= M and columns >= N are not written. All groups run in one launch; longest first balances them best.
constexpr int TC_EXACT_CHUNK_KB = 4, TC_EXACT_MAX_KB = 508;
struct TcExactGroup {
  long long kA = 0, kB = 0, k_pad = 0;   // elements, multiples of 64
  long long N = 0, ldp = 0, split_stride = 0;
  int* P = nullptr;
  int nk_split = 1;
  int zs() const { return (int)std::max<long long>(1, (k_pad / 64 + nk_split - 1) / nk_split); }
};
void tc_gemm_exact(const TcOperand& A, const TcOperand& B, long long M, const TcExactGroup* eg, int n, int* err_dev,
                   cudaStream_t s, int prof_class = 0);
// k-blocks per split for n groups of M x N[i] x k_pad[i] in one launch
int tc_exact_nk_split(long long M, const long long* N, const long long* k_pad, int n);

// k-block (elements) of a kind: 64 16-bit or 32 tf32 = 128 bytes
inline int tc_kblock(TcKind k) { return k == TcKind::TF32 ? 32 : 64; }
inline int tc_pad_k(TcKind k, long long K) { int b = tc_kblock(k); return (int)((K + b - 1) / b * b); }

}  // namespace gfcc
