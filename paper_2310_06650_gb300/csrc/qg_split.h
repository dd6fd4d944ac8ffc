// Products C[row][t] = sum_k A[row][k] B[t][k] to FP64-class accuracy on the fifth-generation tensor
// cores, for a static matrix A (the inverse of the dense tail of the sparse DC factor) and a few right-hand
// sides B per evaluation.
//
// Every row of A and every right-hand side is scaled by a power of two and written as S balanced 8-bit
// digits, v = 2^e sum_i q_i 2^(-6 - 8 i), |q_i| <= 128, each a BF16 matrix of integers (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, Numerical Algorithms 59, 2012).  The digit products with i + j
// = g share one FP32 accumulator; SPLIT_CHUNK columns and at most S pairs keep it an integer of at most
// 2^24 (S 128 2^14), so every accumulation is exact, and the accumulators are added up as 64-bit integers.
// What is dropped are the digit products with i + j >= S.  An output is off by at most
//   K (S + 1) 2^(4 - 8 S) max|A[row]| max|B[t]|
// (K columns; the dropped products, and the rounding of both operands to 8 S - 2 bits below the power of two
// above their largest entry) and the rounding to the result's type: relative to the largest entries, where
// a sum in FP64 or double-FP32 is relative to sum_k |A B|.  The operands' whole range is covered, the powers of
// two being kept as exponents; a row or a right-hand side with an infinity or NaN gives NaN.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "qg_internal.h"

namespace qg {

constexpr int SPLIT_ROWS = 128;   // rows of A per tile (TMEM lanes)
constexpr int SPLIT_KB = 64;      // columns per stage (one 128-byte swizzle span)
constexpr int SPLIT_CHUNK = 128;  // columns accumulated between two flushes of the FP32 accumulators
constexpr int SPLIT_NT = 48;      // right-hand sides per pass
constexpr int SPLIT_SPREAD = 16;  // copies of the running maxima of a right-hand side (atomic contention)

// Digits: 7 carry a double-FP32 operand (its 48 bits, and 2^-54 of the row's largest entry), 8 an FP64 one.
template <typename Dc>
constexpr int split_digits() { return sizeof(Dc) == 8 && alignof(Dc) == 8 ? 8 : 7; }

// Key of |v|, increasing with it, whose leading bits are its exponent: what the scales are taken from (a maximum
// of keys is the same in any order).
#ifdef __CUDACC__
__device__ __forceinline__ unsigned split_key(double v) { return (unsigned)__double2hiint(fabs(v)); }
__device__ __forceinline__ unsigned split_key(df32 v) { return __float_as_uint(__fadd_ru(fabsf(v.hi), fabsf(v.lo))); }
#endif

// A static matrix in digits, with the tensor maps and the buffers of its right-hand sides.
struct SplitMat {
  int rows, K, T;           // A is rows x K; T right-hand sides
  int nt;                   // right-hand sides per pass, a multiple of 16 (<= SPLIT_NT)
  int ks, kbps;             // splits of K across blocks, and K blocks (of SPLIT_KB) per split
  CUtensorMap ta, tb;       // A's tiles as rows of 64; (K, T, S)
  __nv_bfloat16 *a, *b;     // tiles [row tile][K block][S][128][64] (zeroed); [S][T][ld]
  long long ld;             // K rounded up to a multiple of 8
  int *aexp, *bexp;         // e per row of A and per right-hand side
  void *part;               // [ks][row tiles][T][128] pairs of 64-bit partial sums
  unsigned *bmax;           // [SPLIT_SPREAD][T] the largest key of B's entries seen (zeroed before the producer)
};

// Elements of m.a.
long long split_elems(const SplitMat &m, int digits);

// Tensor maps of m (whose sizes and buffers are set); false when the driver's encoder is missing or refuses.
bool split_maps(SplitMat &m, int digits);

// Raises the product kernel's shared-memory limit on the current GPU (the limit belongs to a function on one
// device): once for each matrix, before its first product.
cudaError_t split_prepare(int digits);

// Digits of A from its FP64 rows (device array, row stride K); digits = 7 or 8.
cudaError_t split_matrix(const SplitMat &m, const double *src, int digits, cudaStream_t s);

// Digits of the right-hand sides z [K][T] (node-major), from the maxima in m.bmax.
template <typename Dc>
cudaError_t split_rhs(const SplitMat &m, const Dc *z, cudaStream_t s, bool pdl);

// Where the finished rows go.
template <typename Dc>
struct SplitOut {
  Dc *u, *th;               // both [pos][T]: row r is position pos0 + r
  int pos0;
  const int *pos_gb;        // generator-bus index of a position, -1 if none (adjoint pass), else NULL
  Dc *gip;                  // adjoint products [T][gi_ld]
  long long gi_ld;
};

#ifdef QG_CHECK_BOUNDS
// The index checks of qg_split.cu (qg_check.h): its table, and its first miss as 100,000 + the source line.
struct QgRange;
void split_check_upload(const QgRange *v, int n);
void split_check_first(int *line, unsigned long long *addr);
#endif

template <typename Dc>
cudaError_t split_product(const SplitMat &m, const SplitOut<Dc> &out, cudaStream_t s, bool pdl);

}  // namespace qg
