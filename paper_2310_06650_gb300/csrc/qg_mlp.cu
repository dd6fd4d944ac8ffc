// Learned warm start: a three-layer MLP (BF16 weights and activations into FP32-accumulating
// tensor-core GEMMs) that maps a load profile to an initial dispatch, voltage magnitudes and
// angles; trained on the GPU by its own forward / backward kernels and an Adam step.
//
//   Z1 = X W1^T + b1,  H1 = relu(Z1),  Z2 = H1 W2^T + b2,  H2 = relu(Z2),  Y = H2 W3^T + b3,
//   loss = mean((Y - target)^2).
// GEMM operands are rounded to BF16 where they enter a GEMM (X, H1, H2, the weights, and the
// back-propagated dY, dZ2, dZ1); accumulation is FP32; master weights, biases, moments and the
// loss are FP32 / FP64.  Every reduction has a fixed order (split-K partials are summed in a
// second pass), so results are bitwise repeatable.
//
// The GEMMs run on the fifth-generation tensor cores: C[m][n] = sum_k A[m][k] B[n][k] with both
// operands BF16 and K-contiguous, staged by TMA (128-byte swizzle) through a ring of shared-memory
// stages, multiplied by tcgen05.mma (M = 128) issued from one thread into a TMEM accumulator, and
// read back with tcgen05.ld for the FP32 partial-sum epilogue.  Every product of the network is
// put in that form: the layers run with the weights as A (their rows fill the 128 TMEM lanes) and
// the batch as B (N = 64), writing the transposed tile; the weight gradients take transposed BF16
// copies of the activations and back-propagated terms (batch-contiguous), the input gradients
// transposed BF16 copies of W2 and W3.
#include <cuda.h>  // CUtensorMap and its enums (the encoder is fetched from the driver at run time)
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "qg_internal.h"

namespace {

thread_local std::string g_mlp_error;

constexpr int UM = 128;              // tile rows: the MMA's M, one TMEM lane each
constexpr int UK = 64;               // K per stage: 64 BF16 = one 128-byte swizzle span per row
constexpr int UTHREADS = 128;        // warp 0: TMA producer, warp 1: MMA issuer, warp 2: TMEM owner; all: epilogue
constexpr unsigned long long WAIT_NS = 1000000000ull;  // a wait gives up after 1 s (error flag, clean exit)

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long gtime() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t *b, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return done != 0;
}

// Wait for the completion of the barrier's phase `parity`.  Gives up after WAIT_NS (or 2^30 polls),
// or at once when another thread of the block has given up (abort != 0 and honour_abort); returns
// whether the phase completed.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, volatile int *abort, bool honour_abort) {
  // the clock is read only once the first polls have failed: reading it costs more than a met wait
  for (int it = 0; it < 16; ++it)
    if (mbar_test(b, parity)) return true;
  const unsigned long long t0 = gtime();
  for (unsigned it = 0; it < (1u << 30); ++it) {
    if (mbar_test(b, parity)) return true;
    if (honour_abort && *abort) return false;
    if ((it & 15) == 15 && gtime() - t0 > WAIT_NS) break;
  }
  *abort = 1;
  return false;
}

// TMA: the box at (c0 = K offset in elements, c1 = row) of a 2-D BF16 tensor map into shared memory,
// completing `bytes` on the barrier.
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor of a K-major tile written by TMA with the 128-byte swizzle: rows
// of 128 bytes, 8-row groups 1024 bytes apart (stride byte offset), descriptor version 1, layout
// SWIZZLE_128B; the leading byte offset is unused for this layout.  The tile starts on a 1024-byte
// boundary, so the K step inside a row is a plain start-address offset (32 bytes per 16 elements).
__device__ __forceinline__ uint64_t umma_desc(const void *tile) {
  const uint32_t a = smem_u32(tile);
  return (uint64_t)((a & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}

// Instruction descriptor of kind::f16: D FP32, A and B BF16, both K-major, M = 128, N = BN.
template <int BN>
__host__ __device__ constexpr uint32_t umma_idesc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(UM >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// the barrier completes once every tcgen05.mma this thread issued before has completed
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// programmatic dependent launch: wait for the preceding kernels' results (a no-op without it)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive FP32 columns of this warp's 32 TMEM lanes (one lane per thread)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

template <int BN, int STAGES>
constexpr size_t umma_smem_bytes() {
  return (size_t)STAGES * (UM * UK * 2 + BN * UK * 2) + 1024;  // + alignment of the first tile to 1024 bytes
}

// Partial C[s] of split s (FP32, M x N row-major, or its transpose N x M when trans) =
//   sum over the K blocks [s kbps, (s + 1) kbps) of A[m][k] B[n][k],
// A (M x K) and B (N x K) BF16 behind the tensor maps tA (box 64 x 128) and tB (box 64 x BN); rows
// and K beyond the tensors read as zeros.  Grid (ceil(M/128), ceil(N/BN), splits), 128 threads.
// Launched as a programmatic dependent of the previous kernel: with a_static (A, the weights, is not
// written by the previous kernel, every block of which has waited for the kernels before it) the first
// stages' A tiles are requested before the wait.
// A wait that runs out sets *err, drains what this block started and returns.
template <int BN, int STAGES>
__global__ void __launch_bounds__(UTHREADS, 1)
    k_umma_gemm(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB, float *__restrict__ P,
                int M, int N, int nkb, int kbps, int trans, int a_static, int *err) {
  constexpr uint32_t A_BYTES = UM * UK * 2, B_BYTES = BN * UK * 2;
  constexpr uint32_t TMEM_COLS = BN < 32 ? 32 : BN;  // a power of two >= 32
  static_assert((BN & (BN - 1)) == 0 && BN >= 16 && BN <= 256, "BN");
  extern __shared__ unsigned char smem_raw[];
  unsigned char *base = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *sA = base, *sB = base + STAGES * A_BYTES;
  __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], accf;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort, s_issued, s_consumed;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * UM, n0 = blockIdx.y * BN;
  const int kb0 = blockIdx.z * kbps, nk = min(kbps, nkb - kb0);  // >= 1: the host sizes the splits so
  volatile int *abort = &s_abort;
  const int pre = a_static ? min(nk, STAGES) : 0;  // stages whose A tile is requested before the wait
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accf, 1);
    s_abort = 0;
    s_issued = 0;
    s_consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int kb = 0; kb < pre; ++kb) {
      mbar_expect_tx(&full[kb], A_BYTES + B_BYTES);
      tma_load_2d(sA + kb * A_BYTES, &tA, &full[kb], (kb0 + kb) * UK, m0);
    }
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  pdl_wait();  // B, and the partial buffer this kernel overwrites, belong to the kernels before it
  if (warp == 0 && lane == 0) {  // producer: stage s holds K block kb, its u-th use
    int issued = 0;
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      const uint32_t u = (uint32_t)(kb / STAGES);
      const int kx = (kb0 + kb) * UK;  // a multiple of 64 elements: 128-byte aligned
      if (kb >= pre) {
        if (kb >= STAGES && !mbar_wait(&empty[s], (u - 1) & 1, abort, true)) break;
        mbar_expect_tx(&full[s], A_BYTES + B_BYTES);
        tma_load_2d(sA + s * A_BYTES, &tA, &full[s], kx, m0);
      }
      tma_load_2d(sB + s * B_BYTES, &tB, &full[s], kx, n0);
      issued = kb + 1;
    }
    s_issued = max(issued, pre);
  } else if (warp == 1 && lane == 0) {  // MMA issuer
    constexpr uint32_t IDESC = umma_idesc<BN>();
    int consumed = 0;
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      if (!mbar_wait(&full[s], (uint32_t)(kb / STAGES) & 1, abort, true)) break;
      tc_fence_after();
      const uint64_t ad = umma_desc(sA + s * A_BYTES), bd = umma_desc(sB + s * B_BYTES);
#pragma unroll
      for (int j = 0; j < UK / 16; ++j)  // K = 16 per MMA: 32 bytes (2 descriptor units) along the row
        umma_bf16(tmem, ad + 2 * j, bd + 2 * j, IDESC, (kb | j) != 0);
      umma_commit(&empty[s]);  // stage s is free once these MMAs have read it
      consumed = kb + 1;
    }
    s_consumed = consumed;
    umma_commit(&accf);  // every MMA above has completed (also after an abort)
  }
  __syncwarp();
  // the accumulator is complete (or, after an abort, no MMA is in flight any more); the flag is read
  // after a barrier so that every warp takes the same branch into the warp-collective TMEM loads
  mbar_wait(&accf, 0, abort, false);
  tc_fence_after();
  __syncthreads();
  if (!*abort) {
    const int m = m0 + warp * 32 + lane;
    float *Ps = P + (long long)blockIdx.z * M * N;
    if (trans) {  // C^T: for each column the warp's 32 lanes (rows) write 32 consecutive floats
#pragma unroll 1
      for (int c0 = 0; c0 < BN && n0 + c0 < N; c0 += 16) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
        if (m < M)
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (n0 + c0 + i < N) Ps[(long long)(n0 + c0 + i) * M + m] = v[i];
      }
    } else {  // C: 32 x 32 pieces turned around in shared memory, each row written by the warp's lanes;
      // the stage buffers are free by now (every TMA copy was consumed, every MMA has completed)
      static_assert(4 * 32 * 33 * sizeof(float) <= STAGES * (A_BYTES + B_BYTES), "epilogue tile");
      float(*t)[33] = reinterpret_cast<float(*)[33]>(base) + warp * 32;
#pragma unroll 1
      for (int c0 = 0; c0 < BN && n0 + c0 < N; c0 += 32) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) t[lane][i] = v[i];
        tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c0 + 16), v);
#pragma unroll
        for (int i = 0; i < 16; ++i) t[lane][16 + i] = v[i];
        __syncwarp();
        const int n = n0 + c0 + lane;
        for (int r = 0; r < 32; ++r) {
          const int mr = m0 + warp * 32 + r;
          if (mr < M && n < N) Ps[(long long)mr * N + n] = t[r][lane];
        }
        __syncwarp();
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort) {
    atomicExch(err, 1);
    // copies still in flight land in this block's shared memory: wait for them (bounded) before exit
    for (int kb = s_consumed; kb < s_issued; ++kb) mbar_wait(&full[kb % STAGES], (uint32_t)(kb / STAGES) & 1, abort, false);
  }
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// One 64 x 64 tile of a BF16 operand copy from the values v of this thread (rows wid + 8 i, columns
// 2 lane and 2 lane + 1 of the tile): row-major with row stride ldd (dst) and, when dstT is given,
// transposed with row stride ldt through shared memory, so that both are written in whole 128-byte lines.
// Row strides are multiples of 8 (pad8) and the tile starts on even rows and columns, so pairs are aligned.
// Called by all 256 threads of the block.
__device__ __forceinline__ void store_tile_bf16(const float2 (&v)[8], __nv_bfloat16 *__restrict__ dst, long long ldd,
                                                __nv_bfloat16 *__restrict__ dstT, long long ldt, int r0, int c0, int rows,
                                                int cols) {
  __shared__ __nv_bfloat16 t[64][66];  // [column][row]; 33 words per column: no bank conflict either way
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = wid + 8 * i, c = 2 * lane;
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[i].x, v[i].y);
    if (dst && r0 + r < rows) {
      __nv_bfloat16 *q = dst + (long long)(r0 + r) * ldd + c0 + c;
      if (c0 + c + 1 < cols) *reinterpret_cast<__nv_bfloat162 *>(q) = h;
      else if (c0 + c < cols) *q = h.x;
    }
    if (dstT) {
      t[c][r] = h.x;
      t[c + 1][r] = h.y;
    }
  }
  if (!dstT) return;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int c = wid + 8 * i, r = 2 * lane;
    if (c0 + c >= cols) continue;
    __nv_bfloat16 *q = dstT + (long long)(c0 + c) * ldt + r0 + r;
    if (r0 + r + 1 < rows) *reinterpret_cast<__nv_bfloat162 *>(q) = *reinterpret_cast<const __nv_bfloat162 *>(&t[c][r]);
    else if (r0 + r < rows) *q = t[c][r];
  }
}

// The 64 x 64 tile at (r0, c0) of an FP32 matrix (rows x cols, row stride cols), zeros outside: this
// thread's 8 pairs, all in flight together; 8-byte loads where every row starts on an even element.
__device__ __forceinline__ void load_tile(const float *__restrict__ src, bool even, int r0, int c0, int rows, int cols,
                                          float2 (&v)[8]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, c = c0 + 2 * lane;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = r0 + wid + 8 * i;
    v[i] = make_float2(0.f, 0.f);
    if (r >= rows) continue;
    const float *q = src + (long long)r * cols + c;
    if (even && c + 1 < cols) v[i] = *reinterpret_cast<const float2 *>(q);
    else {
      if (c < cols) v[i].x = q[0];
      if (c + 1 < cols) v[i].y = q[1];
    }
  }
}

__device__ __forceinline__ bool even_rows(const float *p, int cols) {
  return (cols & 1) == 0 && (reinterpret_cast<uintptr_t>(p) & 7) == 0;
}

// BF16 operand copies of an FP32 matrix, row-major (stride ldd) and optionally transposed (stride ldt).
// Grid (ceil(cols/64), ceil(rows/64)), 256 threads.
__global__ void __launch_bounds__(256) k_tile_bf16(const float *__restrict__ src, __nv_bfloat16 *__restrict__ dst,
                                                   long long ldd, __nv_bfloat16 *__restrict__ dstT, long long ldt,
                                                   int rows, int cols) {
  pdl_wait();
  float2 v[8];
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  load_tile(src, even_rows(src, cols), r0, c0, rows, cols, v);
  store_tile_bf16(v, dst, ldd, dstT, ldt, r0, c0, rows, cols);
}

// Epilogue tile: MAX_B batch rows x TC columns of a layer's output per block of 256 threads; thread
// (column tid % TC, rows tid / TC + (256 / TC) i) sums its elements' split-K partials in split order,
// with all its rows' loads of a split in flight together.
constexpr int MAX_B = 64;
enum { EPI_HIDDEN, EPI_OUT, EPI_LOSS, EPI_BACK };

struct EpiArgs {
  const float *P;         // partials [splits][B][N]
  int splits, B, N;
  const float *bias;      // forward: added after the partials
  float *Z;               // EPI_HIDDEN: pre-activation; EPI_OUT: the network's output
  const float *target;    // EPI_LOSS
  double *lpart;          // EPI_LOSS: the block's sum of squared errors
  const float *zmask;     // EPI_BACK: elements where it is not positive are zeroed (relu')
  float *bgrad;           // EPI_LOSS, EPI_BACK: bias gradient, the column's sum in row order
  __nv_bfloat16 *Hb;      // BF16 operand for the next GEMMs, row-major with row stride ldh (may be NULL) ...
  long long ldh;
  __nv_bfloat16 *HbT;     // ... and transposed with row stride ldt
  long long ldt;
};

// What bounds it: the partials' read from L2 (a few microseconds at 16 to 36 splits) and the launch.  One
// kernel per layer: the loss's residual and gradient come with the last layer's epilogue (the output
// is not written and read again: at the rt617 network 42 us in three kernels before), bias gradients with
// the tile that holds the whole batch.
template <int MODE, int TC>
__global__ void __launch_bounds__(256) k_epi(const __grid_constant__ EpiArgs a) {
  constexpr int RS = 256 / TC, NR = MAX_B / RS;  // row stride, rows per thread
  __shared__ float s_v[MAX_B][TC + 1];
  __shared__ double red[8];
  pdl_wait();
  const int c = threadIdx.x % TC, r0 = threadIdx.x / TC, n = blockIdx.x * TC + c;
  const bool on = n < a.N;
  const int total = a.B * a.N;  // below 2^31: the host allocates 64 times it
  // elements outside the layer read element 0: every load is unconditional, 16 partials in flight
  constexpr int UN = 16 / NR;
  int at[NR];
  float v[NR], x[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int r = r0 + i * RS;
    at[i] = on && r < a.B ? r * a.N + n : 0;
    v[i] = 0.f;
    x[i] = 0.f;
    if (MODE == EPI_LOSS) x[i] = __ldg(a.target + at[i]);
    if (MODE == EPI_BACK) x[i] = __ldg(a.zmask + at[i]);
  }
  const float bias = MODE != EPI_BACK ? __ldg(a.bias + (on ? n : 0)) : 0.f;
  int sp = 0;
  for (; sp + UN <= a.splits; sp += UN) {
    float t[UN][NR];
#pragma unroll
    for (int u = 0; u < UN; ++u)
#pragma unroll
      for (int i = 0; i < NR; ++i) t[u][i] = __ldg(a.P + (long long)(sp + u) * total + at[i]);
#pragma unroll
    for (int u = 0; u < UN; ++u)
#pragma unroll
      for (int i = 0; i < NR; ++i) v[i] += t[u][i];
  }
  for (; sp < a.splits; ++sp)
#pragma unroll
    for (int i = 0; i < NR; ++i) v[i] += __ldg(a.P + (long long)sp * total + at[i]);
  const float sc = 2.0f / (float)total;
  double acc = 0.0;
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int r = r0 + i * RS;
    const bool live = on && r < a.B;
    const int e = at[i];
    if (MODE == EPI_BACK) {
      if (!(x[i] > 0.f)) v[i] = 0.f;
    } else {
      v[i] += bias;
      if (MODE == EPI_LOSS) {
        const float d = live ? v[i] - x[i] : 0.f;
        acc += (double)d * (double)d;
        v[i] = sc * d;
      } else {
        if (live) a.Z[e] = v[i];
        if (MODE == EPI_HIDDEN) v[i] = fmaxf(v[i], 0.f);
      }
    }
    if (MODE != EPI_OUT) s_v[r][c] = live ? v[i] : 0.f;
  }
  if (MODE == EPI_OUT) return;
  if (MODE == EPI_LOSS) {
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  }
  __syncthreads();
  if (MODE == EPI_LOSS && threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    a.lpart[blockIdx.x] = t;
  }
  if ((MODE == EPI_LOSS || MODE == EPI_BACK) && threadIdx.x < TC && blockIdx.x * TC + threadIdx.x < a.N) {
    float t = 0.f;
    for (int r = 0; r < a.B; ++r) t += s_v[r][threadIdx.x];
    a.bgrad[blockIdx.x * TC + threadIdx.x] = t;
  }
  if (a.Hb)
    for (int e = threadIdx.x; e < a.B * TC; e += 256) {
      const int r = e / TC, cc = e % TC;
      if (blockIdx.x * TC + cc < a.N) a.Hb[r * a.ldh + blockIdx.x * TC + cc] = __float2bfloat16_rn(s_v[r][cc]);
    }
  for (int e = threadIdx.x; e < TC * MAX_B; e += 256) {  // consecutive threads: consecutive rows of one column
    const int cc = e / MAX_B, r = e % MAX_B;
    if (r < a.B && blockIdx.x * TC + cc < a.N)
      a.HbT[(long long)(blockIdx.x * TC + cc) * a.ldt + r] = __float2bfloat16_rn(s_v[r][cc]);
  }
}

// The mean of the block partials: one block of 256 threads, strided sums then a shuffle and
// shared-memory tree (a fixed order).
__global__ void __launch_bounds__(256) k_loss_final(const double *part, int n, long long total, double *loss) {
  pdl_wait();
  __shared__ double red[8];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += part[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    *loss = t / (double)total;
  }
}

// Adam on the FP32 master parameters and the BF16 operand copies of the updated weights, in one pass:
// blocks [0, n_tiles) take 64 x 64 tiles of the three weight matrices (gradient, weight and both
// moments read, weight and moments written, with the row-major and the transposed BF16 copies from the same
// registers), the rest the biases.  Bound by HBM: 32 bytes per weight.  At the rt617 network (40 M
// weights) Adam and the five copy kernels took 220 + 187 us.
struct AdamMat {
  long long off;                        // the matrix in the parameter layout
  int rows, cols, tile0, tiles_c;       // its first tile and tiles per row of tiles
  __nv_bfloat16 *b;                     // BF16 copy, row stride ldb
  long long ldb;
  __nv_bfloat16 *t;                     // transposed copy (may be NULL), row stride ldt
  long long ldt;
};
struct AdamArgs {
  AdamMat m[3];
  int n_tiles;
  long long bias_off[3];
  int bias_n[3];
  float lr, b1, b2, c1, c2, eps;
};

// (The multiply-adds are spelled out, so that the rounding of a training run does not hang on the compiler.)
__device__ __forceinline__ void adam1(const AdamArgs &a, float &w, float g, float &m, float &v) {
  m = __fmaf_rn(1.f - a.b1, g, __fmul_rn(a.b1, m));
  v = __fmaf_rn(__fmul_rn(1.f - a.b2, g), g, __fmul_rn(a.b2, v));
  w -= a.lr * (m * a.c1) / (sqrtf(v * a.c2) + a.eps);
}

__global__ void __launch_bounds__(256, 2) k_mlp_adam(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
                                                  float *__restrict__ v, const __grid_constant__ AdamArgs a) {
  pdl_wait();
  if ((int)blockIdx.x >= a.n_tiles) {  // biases
    long long i = (long long)(blockIdx.x - a.n_tiles) * 256 + threadIdx.x;
    for (int q = 0; q < 3; ++q) {
      if (i < a.bias_n[q]) {
        const long long e = a.bias_off[q] + i;
        float wi = w[e], mi = m[e], vi = v[e];
        adam1(a, wi, g[e], mi, vi);
        w[e] = wi;
        m[e] = mi;
        v[e] = vi;
        return;
      }
      i -= a.bias_n[q];
    }
    return;
  }
  const int q = (int)blockIdx.x >= a.m[2].tile0 ? 2 : (int)blockIdx.x >= a.m[1].tile0 ? 1 : 0;
  const AdamMat &M = a.m[q];
  const int tile = blockIdx.x - M.tile0, r0 = tile / M.tiles_c * 64, c0 = tile % M.tiles_c * 64;
  const bool even = even_rows(w + M.off, M.cols);  // the four arrays are 256-byte aligned: the same for all
  float2 wv[8], gv[8], mv[8], vv[8];
  load_tile(g + M.off, even, r0, c0, M.rows, M.cols, gv);
  load_tile(m + M.off, even, r0, c0, M.rows, M.cols, mv);
  load_tile(v + M.off, even, r0, c0, M.rows, M.cols, vv);
  load_tile(w + M.off, even, r0, c0, M.rows, M.cols, wv);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, c = c0 + 2 * lane;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    adam1(a, wv[i].x, gv[i].x, mv[i].x, vv[i].x);
    adam1(a, wv[i].y, gv[i].y, mv[i].y, vv[i].y);
    const int r = r0 + wid + 8 * i;
    if (r >= M.rows) continue;
    const long long e = M.off + (long long)r * M.cols + c;
    if (even && c + 1 < M.cols) {
      *reinterpret_cast<float2 *>(w + e) = wv[i];
      *reinterpret_cast<float2 *>(m + e) = mv[i];
      *reinterpret_cast<float2 *>(v + e) = vv[i];
    } else {
      if (c < M.cols) {
        w[e] = wv[i].x;
        m[e] = mv[i].x;
        v[e] = vv[i].x;
      }
      if (c + 1 < M.cols) {
        w[e + 1] = wv[i].y;
        m[e + 1] = mv[i].y;
        v[e + 1] = vv[i].y;
      }
    }
  }
  store_tile_bf16(wv, M.b, M.ldb, M.t, M.ldt, r0, c0, M.rows, M.cols);
}

// Deterministic counter-based normal draws (Box-Muller on a splitmix64 stream) for the initial weights.
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void k_init(float *__restrict__ w, long long n, float scale, uint64_t seed, long long offset) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const uint64_t a = splitmix64(seed ^ (uint64_t)(offset + i) * 2ull);
    const uint64_t b = splitmix64(seed ^ ((uint64_t)(offset + i) * 2ull + 1ull));
    const float u1 = ((a >> 40) + 1.0f) * (1.0f / 16777217.0f);
    const float u2 = (b >> 40) * (1.0f / 16777216.0f);
    w[i] = scale * sqrtf(-2.f * logf(u1)) * cospif(2.f * u2);
  }
}

// Launch as a programmatic dependent of the previous kernel in the stream (each kernel waits with
// griddepcontrol.wait before it touches what earlier kernels wrote or read).
template <typename... KArgs, typename... Args>
cudaError_t pdl_launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

int grid_for(long long n) { return (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152 * 8)); }

long long pad8(long long n) { return (n + 7) / 8 * 8; }  // BF16 row strides: multiples of 16 bytes (TMA)

}  // namespace

struct qg_mlp {
  int n_in, n_h, n_out, max_b;
  int device = -1;  // the GPU it was created on
  long long ld_i, ld_h, ld_o, ld_b;  // padded BF16 row strides for rows of I, H, O and batch elements
  long long n_par;
  long long o_w1, o_b1, o_w2, o_b2, o_w3, o_b3;
  cudaStream_t stream = nullptr;
  std::vector<void *> allocs;
  float *w = nullptr, *gw = nullptr, *am = nullptr, *av = nullptr;
  // BF16 GEMM operands, all K-contiguous: weights [H][ld_i], [H][ld_h], [O][ld_h] and the transposed
  // W2^T [H][ld_h], W3^T [H][ld_o]; activations row-major [B][ld_*] and transposed [features][ld_b]
  __nv_bfloat16 *w1b = nullptr, *w2b = nullptr, *w3b = nullptr, *w2t = nullptr, *w3t = nullptr;
  __nv_bfloat16 *xb = nullptr, *xt = nullptr, *h1b = nullptr, *h1t = nullptr, *h2b = nullptr, *h2t = nullptr;
  __nv_bfloat16 *dyb = nullptr, *dyt = nullptr, *dz2b = nullptr, *dz2t = nullptr, *dz1t = nullptr;
  float *z1 = nullptr, *z2 = nullptr, *part = nullptr;
  double *lpart = nullptr;
  int *d_err = nullptr;  // set by a GEMM block whose pipeline wait ran out
  long long part_elems = 0;
  long long step = 0;
  std::string err;
};

namespace {

int mfail(qg_mlp *m, int code, const std::string &msg) {
  if (m) m->err = msg;
  g_mlp_error = msg;
  return code;
}

template <typename T>
int mal(qg_mlp *m, T **p, size_t n) {
  cudaError_t e = cudaMalloc((void **)p, std::max<size_t>(n, 1) * sizeof(T));
  if (e != cudaSuccess) return mfail(m, QG_ERR_CUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  m->allocs.push_back(*p);
  return QG_OK;
}

// cuTensorMapEncodeTiled from the driver (no link-time dependency on libcuda)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    cudaGetLastError();
  });
  return fn;
}

// 2-D tensor map of a BF16 matrix (rows x cols, row stride ld elements, a multiple of 8) with a box
// of 64 columns (128 bytes, the swizzle span) x box_rows rows; reads outside the matrix give zeros.
int make_map(qg_mlp *m, CUtensorMap *map, const __nv_bfloat16 *ptr, long long rows, long long cols, long long ld,
             int box_rows) {
  const auto enc = tensor_map_encoder();
  if (!enc) return mfail(m, QG_ERR_UNSUPPORTED, "cuTensorMapEncodeTiled is not available from the driver");
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)UK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16 *>(ptr), dims, strides, box,
                         estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return mfail(m, QG_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return QG_OK;
}

// Raises the kernel's shared-memory limit on the current GPU (the limit belongs to a function on one device).
template <int BN, int STAGES>
cudaError_t umma_prepare() {
  return cudaFuncSetAttribute(k_umma_gemm<BN, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)umma_smem_bytes<BN, STAGES>());
}

// Split-K partials of C = A B^T (A: M x K with row stride lda, B: N x K with row stride ldb, both BF16)
// into mm->part: [splits][M][N], or [splits][N][M] with trans; with dst, C itself (one split) into dst.  Returns the number of splits, or 0
// after recording an error.  Narrow products (N <= 64: the batch) take 64-column tiles and a
// 4-stage ring; wide ones (the weight gradients, K = the batch) 256-column tiles and 2 stages.
// a_static: A is a weight copy (not written by the kernel just before), requested before the wait.
int gemm(qg_mlp *mm, const __nv_bfloat16 *A, long long lda, int M, const __nv_bfloat16 *B, long long ldb, int N, int K,
         bool trans, bool a_static, float *dst = nullptr) {
  const bool narrow = N <= 64;
  const int BN = narrow ? 64 : 256;
  const long long tiles = (long long)((M + UM - 1) / UM) * ((N + BN - 1) / BN);
  const int nkb = (K + UK - 1) / UK;
  int splits = dst ? 1 : (int)std::max(1LL, std::min<long long>({64LL, (long long)nkb, (2LL * 152 + tiles - 1) / tiles}));
  while (splits > 1 && (long long)splits * M * N > mm->part_elems) --splits;
  const int kbps = (nkb + splits - 1) / splits;
  splits = (nkb + kbps - 1) / kbps;  // every split has at least one K block
  CUtensorMap ta, tb;
  int rc = make_map(mm, &ta, A, M, K, lda, UM);
  if (!rc) rc = make_map(mm, &tb, B, N, K, ldb, BN);
  if (rc) return 0;
  const dim3 grid((M + UM - 1) / UM, (N + BN - 1) / BN, splits);
  float *out = dst ? dst : mm->part;
  cudaError_t e;
  if (narrow) {
    e = pdl_launch(k_umma_gemm<64, 4>, grid, dim3(UTHREADS), umma_smem_bytes<64, 4>(), mm->stream, ta, tb, out, M,
                   N, nkb, kbps, trans ? 1 : 0, a_static ? 1 : 0, mm->d_err);
  } else {
    e = pdl_launch(k_umma_gemm<256, 2>, grid, dim3(UTHREADS), umma_smem_bytes<256, 2>(), mm->stream, ta, tb, out,
                   M, N, nkb, kbps, trans ? 1 : 0, a_static ? 1 : 0, mm->d_err);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    mfail(mm, QG_ERR_CUDA, std::string("tensor-core GEMM launch: ") + cudaGetErrorString(e));
    return 0;
  }
  return splits;
}

dim3 tiles64(long long rows, long long cols) { return dim3((unsigned)((cols + 63) / 64), (unsigned)((rows + 63) / 64)); }

// x (batch x I, FP32) into the BF16 operand xb [B][ld_i] and, for training (the first layer's weight
// gradient), xt [I][ld_b]
void load_x(qg_mlp *m, const float *x, int B, bool transposed) {
  pdl_launch(k_tile_bf16, tiles64(B, m->n_in), dim3(256), 0, m->stream, x, m->xb, m->ld_i,
             transposed ? m->xt : (__nv_bfloat16 *)nullptr, m->ld_b, B, m->n_in);
}

// Columns per epilogue block: narrow tiles where the layer is narrow, so that its blocks fill the SMs.
constexpr int EPI_TC_H = 8, EPI_TC_O = 32;

template <int MODE, int TC>
void epi(qg_mlp *m, const EpiArgs &a) {
  pdl_launch(k_epi<MODE, TC>, dim3((a.N + TC - 1) / TC), dim3(256), 0, m->stream, a);
}

// The two hidden layers and the last layer's GEMM, as C^T = W act^T (weights as the 128-row operand, the
// batch as N); returns the last GEMM's splits, or 0 after an error.
int forward(qg_mlp *m, int B) {
  const int H = m->n_h, I = m->n_in, O = m->n_out;
  int s = gemm(m, m->w1b, m->ld_i, H, m->xb, m->ld_i, B, I, true, true);
  if (!s) return 0;
  EpiArgs a{};
  a.P = m->part; a.B = B; a.N = H;
  a.splits = s; a.bias = m->w + m->o_b1; a.Z = m->z1; a.Hb = m->h1b; a.ldh = m->ld_h; a.HbT = m->h1t; a.ldt = m->ld_b;
  epi<EPI_HIDDEN, EPI_TC_H>(m, a);
  if (!(s = gemm(m, m->w2b, m->ld_h, H, m->h1b, m->ld_h, B, H, true, true))) return 0;
  a.splits = s; a.bias = m->w + m->o_b2; a.Z = m->z2; a.Hb = m->h2b; a.HbT = m->h2t;
  epi<EPI_HIDDEN, EPI_TC_H>(m, a);
  return gemm(m, m->w3b, m->ld_h, O, m->h2b, m->ld_h, B, H, true, true);
}

// BF16 operand copies of the FP32 master weights: W1, W2, W3 row-major (padded) and W2^T, W3^T.
void refresh_bf16(qg_mlp *m) {
  const int H = m->n_h, I = m->n_in, O = m->n_out;
  cudaStream_t s = m->stream;
  pdl_launch(k_tile_bf16, tiles64(H, I), dim3(256), 0, s, m->w + m->o_w1, m->w1b, m->ld_i, (__nv_bfloat16 *)nullptr, 0LL, H, I);
  pdl_launch(k_tile_bf16, tiles64(H, H), dim3(256), 0, s, m->w + m->o_w2, m->w2b, m->ld_h, m->w2t, m->ld_h, H, H);
  pdl_launch(k_tile_bf16, tiles64(O, H), dim3(256), 0, s, m->w + m->o_w3, m->w3b, m->ld_h, m->w3t, m->ld_o, O, H);
}

}  // namespace

extern "C" {

int qg_mlp_create(qg_mlp **out, int32_t n_in, int32_t n_hidden, int32_t n_out, int32_t max_batch, uint64_t seed) {
  g_mlp_error.clear();
  if (!out) return mfail(nullptr, QG_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (n_in < 1 || n_hidden < 1 || n_out < 1 || max_batch < 1) return mfail(nullptr, QG_ERR_INVALID_ARG, "sizes");
  if (max_batch > 64) return mfail(nullptr, QG_ERR_UNSUPPORTED, "max_batch above 64 (one 64-column GEMM tile)");
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || count < 1) return mfail(nullptr, QG_ERR_NO_DEVICE, "no CUDA device");
  if (!tensor_map_encoder()) return mfail(nullptr, QG_ERR_UNSUPPORTED, "cuTensorMapEncodeTiled is not available");
  qg_mlp *m = new qg_mlp();
  if (cudaGetDevice(&m->device) != cudaSuccess) {
    delete m;
    return mfail(nullptr, QG_ERR_NO_DEVICE, "cudaGetDevice failed");
  }
  m->n_in = n_in; m->n_h = n_hidden; m->n_out = n_out; m->max_b = max_batch;
  m->ld_i = pad8(n_in); m->ld_h = pad8(n_hidden); m->ld_o = pad8(n_out); m->ld_b = pad8(max_batch);
  m->o_w1 = 0; m->o_b1 = m->o_w1 + (long long)n_hidden * n_in;
  m->o_w2 = m->o_b1 + n_hidden; m->o_b2 = m->o_w2 + (long long)n_hidden * n_hidden;
  m->o_w3 = m->o_b2 + n_hidden; m->o_b3 = m->o_w3 + (long long)n_out * n_hidden;
  m->n_par = m->o_b3 + n_out;
  const long long B = max_batch, H = n_hidden, I = n_in, O = n_out;
  const long long li = m->ld_i, lh = m->ld_h, lo = m->ld_o, lb = m->ld_b;
  m->part_elems = std::max({64 * B * H, 65 * B * O, H * I, O * H, H * H});  // 64 splits, and an output (qg_mlp_forward)
  int rc = 0;
  if ((rc = mal(m, &m->w, m->n_par)) || (rc = mal(m, &m->gw, m->n_par)) || (rc = mal(m, &m->am, m->n_par)) ||
      (rc = mal(m, &m->av, m->n_par)) || (rc = mal(m, &m->w1b, H * li)) || (rc = mal(m, &m->w2b, H * lh)) ||
      (rc = mal(m, &m->w3b, O * lh)) || (rc = mal(m, &m->w2t, H * lh)) || (rc = mal(m, &m->w3t, H * lo)) ||
      (rc = mal(m, &m->xb, B * li)) || (rc = mal(m, &m->xt, I * lb)) || (rc = mal(m, &m->h1b, B * lh)) ||
      (rc = mal(m, &m->h1t, H * lb)) || (rc = mal(m, &m->h2b, B * lh)) || (rc = mal(m, &m->h2t, H * lb)) ||
      (rc = mal(m, &m->dyb, B * lo)) || (rc = mal(m, &m->dyt, O * lb)) || (rc = mal(m, &m->dz2b, B * lh)) ||
      (rc = mal(m, &m->dz2t, H * lb)) || (rc = mal(m, &m->dz1t, H * lb)) || (rc = mal(m, &m->z1, B * H)) ||
      (rc = mal(m, &m->z2, B * H)) || (rc = mal(m, &m->part, m->part_elems)) ||
      (rc = mal(m, &m->lpart, (O + 31) / 32)) || (rc = mal(m, &m->d_err, 1))) {
    qg_mlp_destroy(m);
    return rc;
  }
  cudaError_t e = umma_prepare<64, 4>();
  if (e == cudaSuccess) e = umma_prepare<256, 2>();
  if (e != cudaSuccess) {
    cudaGetLastError();  // a refused attribute is not a sticky error
    mfail(m, QG_ERR_CUDA, std::string("tensor-core GEMM launch: ") + cudaGetErrorString(e));
    qg_mlp_destroy(m);
    return QG_ERR_CUDA;
  }
  cudaMemset(m->gw, 0, m->n_par * sizeof(float));
  cudaMemset(m->am, 0, m->n_par * sizeof(float));
  cudaMemset(m->av, 0, m->n_par * sizeof(float));
  cudaMemset(m->w, 0, m->n_par * sizeof(float));
  cudaMemset(m->d_err, 0, sizeof(int));
  // He initialisation for the ReLU layers, a smaller scale for the linear output layer; zero biases
  k_init<<<grid_for(H * I), 256>>>(m->w + m->o_w1, H * I, sqrtf(2.f / (float)I), seed, 0);
  k_init<<<grid_for(H * H), 256>>>(m->w + m->o_w2, H * H, sqrtf(2.f / (float)H), seed, H * I);
  k_init<<<grid_for(O * H), 256>>>(m->w + m->o_w3, O * H, sqrtf(1.f / (float)H), seed, H * I + H * H);
  refresh_bf16(m);
  e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    mfail(m, QG_ERR_CUDA, std::string("init: ") + cudaGetErrorString(e));
    qg_mlp_destroy(m);
    return QG_ERR_CUDA;
  }
  *out = m;
  return QG_OK;
}

void qg_mlp_destroy(qg_mlp *m) {
  if (!m) return;
  for (void *p : m->allocs) cudaFree(p);
  delete m;
}

int64_t qg_mlp_num_params(const qg_mlp *m) { return m ? m->n_par : 0; }

int qg_mlp_set_stream(qg_mlp *m, void *stream) {
  if (!m) return QG_ERR_INVALID_ARG;
  m->stream = (cudaStream_t)stream;
  return QG_OK;
}

int qg_mlp_forward(qg_mlp *m, const float *x, int32_t batch, float *y) {
  if (!m || !x || !y || batch < 1 || batch > m->max_b) return m ? mfail(m, QG_ERR_INVALID_ARG, "forward arguments") : QG_ERR_INVALID_ARG;
  load_x(m, x, batch, false);
  const int sp = forward(m, batch);
  if (!sp) return QG_ERR_CUDA;
  // y is written in place where a kernel may write it, else past the partial sums and copied
  const long long ny = (long long)batch * m->n_out;
  const bool direct = qg::device_memory(y, sizeof(float), m->device);
  EpiArgs a{};
  a.P = m->part; a.B = batch; a.N = m->n_out; a.splits = sp; a.bias = m->w + m->o_b3;
  a.Z = direct ? y : m->part + sp * ny;
  epi<EPI_OUT, EPI_TC_O>(m, a);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && !direct)
    e = cudaMemcpyAsync(y, a.Z, sizeof(float) * ny, cudaMemcpyDeviceToDevice, m->stream);
  return e == cudaSuccess ? QG_OK : mfail(m, QG_ERR_CUDA, cudaGetErrorString(e));
}

int qg_mlp_train_step(qg_mlp *m, const float *x, const float *target, int32_t batch, double lr, double beta1,
                      double beta2, double *loss) {
  if (!m || !x || !target || batch < 1 || batch > m->max_b)
    return m ? mfail(m, QG_ERR_INVALID_ARG, "train arguments") : QG_ERR_INVALID_ARG;
  const int B = batch, H = m->n_h, I = m->n_in, O = m->n_out;
  cudaStream_t s = m->stream;
  load_x(m, x, B, true);
  int sp = forward(m, B);
  if (!sp) return QG_ERR_CUDA;
  const long long ny = (long long)B * O;
  // dY = 2 (Y - target) / (B O), the squared error and db3 = colsum(dY), from the last layer's partials
  EpiArgs a{};
  a.P = m->part; a.B = B; a.N = O; a.splits = sp; a.bias = m->w + m->o_b3; a.target = target; a.lpart = m->lpart;
  a.bgrad = m->gw + m->o_b3; a.Hb = m->dyb; a.ldh = m->ld_o; a.HbT = m->dyt; a.ldt = m->ld_b;
  epi<EPI_LOSS, EPI_TC_O>(m, a);
  if (loss)
    pdl_launch(k_loss_final, dim3(1), dim3(256), 0, s, (const double *)m->lpart, (O + EPI_TC_O - 1) / EPI_TC_O, ny, loss);
  // layer 3: dW3 = dY^T H2 (K = the batch: one split, written straight into the gradient),
  // dH2 = dY W3 masked by relu'(Z2), db2 its column sums
  if (!gemm(m, m->dyt, m->ld_b, O, m->h2t, m->ld_b, H, B, false, false, m->gw + m->o_w3)) return QG_ERR_CUDA;
  if (!(sp = gemm(m, m->w3t, m->ld_o, H, m->dyb, m->ld_o, B, O, true, true))) return QG_ERR_CUDA;
  a.N = H; a.splits = sp; a.zmask = m->z2; a.bgrad = m->gw + m->o_b2; a.Hb = m->dz2b; a.ldh = m->ld_h; a.HbT = m->dz2t;
  epi<EPI_BACK, EPI_TC_H>(m, a);
  // layer 2
  if (!gemm(m, m->dz2t, m->ld_b, H, m->h1t, m->ld_b, H, B, false, false, m->gw + m->o_w2)) return QG_ERR_CUDA;
  if (!(sp = gemm(m, m->w2t, m->ld_h, H, m->dz2b, m->ld_h, B, H, true, true))) return QG_ERR_CUDA;
  a.splits = sp; a.zmask = m->z1; a.bgrad = m->gw + m->o_b1; a.Hb = nullptr; a.HbT = m->dz1t;
  epi<EPI_BACK, EPI_TC_H>(m, a);
  // layer 1
  if (!gemm(m, m->dz1t, m->ld_b, H, m->xt, m->ld_b, I, B, false, false, m->gw + m->o_w1)) return QG_ERR_CUDA;
  // Adam and the BF16 copies of the updated weights
  if (lr > 0) {
    m->step += 1;
    AdamArgs ad{};
    const long long rows[3] = {H, H, O}, cols[3] = {I, H, H}, offs[3] = {m->o_w1, m->o_w2, m->o_w3};
    __nv_bfloat16 *const cb[3] = {m->w1b, m->w2b, m->w3b}, *const ct[3] = {nullptr, m->w2t, m->w3t};
    const long long ldb[3] = {m->ld_i, m->ld_h, m->ld_h}, ldt[3] = {0, m->ld_h, m->ld_o};
    for (int q = 0; q < 3; ++q) {
      const dim3 t = tiles64(rows[q], cols[q]);
      ad.m[q] = AdamMat{offs[q], (int)rows[q], (int)cols[q], ad.n_tiles, (int)t.x, cb[q], ldb[q], ct[q], ldt[q]};
      ad.n_tiles += (int)(t.x * t.y);
    }
    ad.bias_off[0] = m->o_b1; ad.bias_off[1] = m->o_b2; ad.bias_off[2] = m->o_b3;
    ad.bias_n[0] = H; ad.bias_n[1] = H; ad.bias_n[2] = O;
    ad.lr = (float)lr; ad.b1 = (float)beta1; ad.b2 = (float)beta2; ad.eps = 1e-8f;
    ad.c1 = (float)(1.0 / (1.0 - std::pow(beta1, (double)m->step)));
    ad.c2 = (float)(1.0 / (1.0 - std::pow(beta2, (double)m->step)));
    pdl_launch(k_mlp_adam, dim3(ad.n_tiles + (2 * H + O + 255) / 256), dim3(256), 0, s, m->w, (const float *)m->gw, m->am,
               m->av, ad);
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? QG_OK : mfail(m, QG_ERR_CUDA, cudaGetErrorString(e));
}

int qg_mlp_check(qg_mlp *m) {
  if (!m) return QG_ERR_INVALID_ARG;
  int flag = 0;
  cudaError_t e = cudaMemcpyAsync(&flag, m->d_err, sizeof(int), cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mfail(m, QG_ERR_CUDA, cudaGetErrorString(e));
  if (flag) return mfail(m, QG_ERR_CUDA, "a tensor-core GEMM pipeline wait ran out (1 s); its results are invalid");
  return QG_OK;
}

int qg_mlp_get_params(qg_mlp *m, float *w) {
  if (!m || !w) return QG_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpyAsync(w, m->w, sizeof(float) * m->n_par, cudaMemcpyDeviceToDevice, m->stream);
  return e == cudaSuccess ? QG_OK : mfail(m, QG_ERR_CUDA, cudaGetErrorString(e));
}

int qg_mlp_set_params(qg_mlp *m, const float *w) {
  if (!m || !w) return QG_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpyAsync(m->w, w, sizeof(float) * m->n_par, cudaMemcpyDeviceToDevice, m->stream);
  if (e != cudaSuccess) return mfail(m, QG_ERR_CUDA, cudaGetErrorString(e));
  refresh_bf16(m);
  return QG_OK;
}

int qg_mlp_get_grads(qg_mlp *m, float *g) {
  if (!m || !g) return QG_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpyAsync(g, m->gw, sizeof(float) * m->n_par, cudaMemcpyDeviceToDevice, m->stream);
  return e == cudaSuccess ? QG_OK : mfail(m, QG_ERR_CUDA, cudaGetErrorString(e));
}

const char *qg_mlp_last_error(const qg_mlp *m) { return m ? m->err.c_str() : g_mlp_error.c_str(); }

}  // extern "C"
