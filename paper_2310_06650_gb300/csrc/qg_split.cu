// FP64-class products on the tensor cores by error-free splitting (see qg_split.h).
//
// k_split_gemm: block (row tile, K split), 10 warps.  Warp 8's elected thread streams, per block of 64
// columns, the right-hand sides' digits (one 3-D TMA copy, [digit][t][64]) into two buffers and the row
// tile's digits (128 x 64 each, stored as contiguous 16 KB tiles in the order of the stream) through a ring
// of SPLIT_STAGES; warp 9's elected thread multiplies digit i of
// A with the digits 0 .. S - 1 - i of B in one tcgen05.mma per 16 columns (their rows are contiguous: N =
// (S - i) nt, in two parts above 256), into the accumulators of the weights i .. S - 1, which are contiguous
// in tensor memory.  After SPLIT_CHUNK columns warps 0-7 read the accumulators, all integers, and add
// them to two 64-bit sums per output, while the ring refills and no multiply runs: one set of accumulators fills
// the tensor memory (S 48 of 512 columns).  Bound by that flush, 2 us per 128 columns, on top of the stream of
// A's digits from HBM (14 or 16 bytes per entry): 3,109 x 3,109 entries, 48 right-hand sides, 7 digits: 47 us,
// 33 us for the stream alone, 143 MB at 3.0 TB/s, the tensor pipe 28% active.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "qg_check.h"
#include "qg_internal.h"
#include "qg_split.h"
#include "qg_split_feed.h"

namespace qg {
namespace {

constexpr int SPLIT_STAGES = 7;
constexpr int SPLIT_RT = 16;                    // right-hand sides per block of k_split_rhs
constexpr int SPLIT_EPI = 256;                  // epilogue threads (warps 0-7)
constexpr int SPLIT_THREADS = SPLIT_EPI + 64;   // + TMA producer warp, MMA warp
constexpr unsigned long long SPLIT_WAIT_NS = 1000000000ull;  // a wait gives up after 1 s (NaN results, clean exit)
constexpr long long SPLIT_LOST = 1ll << 62;  // a block's partial sums after a wait ran out (real ones are below 2^61)
constexpr int SPLIT_NONFINITE = 1 << 20;  // in place of an exponent: an operand is infinite or NaN
constexpr uint32_t A_BYTES = SPLIT_ROWS * SPLIT_KB * 2;

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
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
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
// Waits for the barrier's phase `parity`; gives up after SPLIT_WAIT_NS (or 2^30 polls), or at once when another
// thread of the block has given up; returns whether the phase completed.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, volatile int *abort, bool honour_abort) {
  // the clock is read only once the first polls have failed: reading it costs more than a met wait
  for (int it = 0; it < 16; ++it)
    if (mbar_test(b, parity)) return true;
  const unsigned long long t0 = gtime();
  for (unsigned it = 0; it < (1u << 30); ++it) {
    if (mbar_test(b, parity)) return true;
    if (honour_abort && *abort) return false;
    if ((it & 15) == 15 && gtime() - t0 > SPLIT_WAIT_NS) break;
  }
  *abort = 1;
  return false;
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
      : "memory");
}
// K-major tile written by TMA with the 128-byte swizzle: rows of 128 bytes, 8-row groups 1,024 bytes apart.
__device__ __forceinline__ uint64_t umma_desc(const void *tile) {
  const uint32_t a = smem_u32(tile);
  return (uint64_t)((a & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
// kind::f16: D FP32, A and B BF16, both K-major, M = 128.
__device__ __forceinline__ uint32_t umma_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(SPLIT_ROWS >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          tmem_d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void wait_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// 8 consecutive FP32 columns of this warp's 32 TMEM lanes; no wait (tmem_wait before the values are used).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// The values loaded before may be used only after the wait (the empty statements in the caller, volatile
// as this one, keep their uses behind it).
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

template <int S>
constexpr size_t split_smem_bytes() {
  return (size_t)SPLIT_STAGES * A_BYTES + 2 * (size_t)S * SPLIT_NT * SPLIT_KB * 2 + 1024;
}

// The finished value of two 64-bit sums: hi 2^-24 + lo 2^-(24 + 8 (S - 4)), times 2^(e - 12) with e the sum of the
// two operands' exponents.
template <int S>
__device__ __forceinline__ double split_value(long long hi, long long lo, int e, double) {
  constexpr double W = S == 8 ? 0x1p-32 : 0x1p-24;
  return scalbn((double)hi + (double)lo * W, e - 36);
}
template <int S>
__device__ __forceinline__ df32 split_value(long long hi, long long lo, int e, df32) {
  constexpr float W = S == 8 ? 0x1p-32f : 0x1p-24f;
  const float h = (float)hi;
  const float l = (float)(hi - (long long)h) + (float)lo * W;
  const float s = __fadd_rn(h, l), r = __fadd_rn(l, __fsub_rn(h, s));
  return {scalbnf(s, e - 36), scalbnf(r, e - 36)};
}

__device__ __forceinline__ double dc_nan(double) { return nan(""); }
__device__ __forceinline__ df32 dc_nan(df32) { return {__int_as_float(0x7fc00000), 0.f}; }

template <int S>
__global__ void __launch_bounds__(SPLIT_THREADS, 1)
    k_split_gemm(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB,
                 longlong2 *__restrict__ part, int n_rt, int K, int T, int nt, int ks, int kbps) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char *base = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *sA = base, *sB = base + SPLIT_STAGES * A_BYTES;
  __shared__ __align__(8) uint64_t fullA[SPLIT_STAGES], emptyA[SPLIT_STAGES], fullB[2], emptyB[2], accf, acce, drain;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rt = blockIdx.x / ks, kp = blockIdx.x % ks;
  const int nkb_all = (K + SPLIT_KB - 1) / SPLIT_KB;
  const int kb0 = kp * kbps, nkb = min(kbps, nkb_all - kb0);  // >= 1: sized by the host
  const uint32_t b_bytes = (uint32_t)(S * nt * SPLIT_KB * 2);
  volatile int *abort = &s_abort;
  if (threadIdx.x == 0) {
    for (int q = 0; q < SPLIT_STAGES; ++q) {
      mbar_init(&fullA[q], 1);
      mbar_init(&emptyA[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&fullB[q], 1);
      mbar_init(&emptyB[q], 1);
    }
    mbar_init(&accf, 1);
    mbar_init(&drain, 1);
    mbar_init(&acce, SPLIT_EPI / 32);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int passes = (T + nt - 1) / nt;
  constexpr int KB_PER_CHUNK = SPLIT_CHUNK / SPLIT_KB;
  const int nch = (nkb + KB_PER_CHUNK - 1) / KB_PER_CHUNK;
  if (warp == 8) {
    if (lane == 0) {  // producer: A's digits are static, B's wait for the kernel before
      struct {
        const CUtensorMap &tA, &tB;
        unsigned char *sA, *sB;
        uint64_t *fullA, *emptyA, *fullB, *emptyB;
        volatile int *abort;
        uint32_t b_bytes;
        int nt, nkb, kb0, tile0;  // K blocks of the block, the first, and its tile of digit 0
        int p, kb;                // pass and K block of the unit
        __device__ bool wait_a_free(int n) const {
          return mbar_wait(&emptyA[n % SPLIT_STAGES], (uint32_t)(n / SPLIT_STAGES - 1) & 1, abort, true);
        }
        __device__ bool wait_b_free(int u) const { return mbar_wait(&emptyB[u & 1], (uint32_t)(u / 2 - 1) & 1, abort, true); }
        __device__ void wait_inputs() const { wait_grid(); }
        __device__ void load_a(int n, int u, int i) {
          if (i == 0 && u > 0 && ++kb == nkb) {
            kb = 0;
            ++p;
          }
          const int st = n % SPLIT_STAGES;
          mbar_expect_tx(&fullA[st], A_BYTES);
          tma_load_2d(sA + st * A_BYTES, &tA, &fullA[st], 0, ((tile0 + kb) * S + i) * SPLIT_ROWS);
        }
        __device__ void load_b(int u) const {  // from a multiple of 64 elements: 128-byte aligned
          mbar_expect_tx(&fullB[u & 1], b_bytes);
          tma_load_3d(sB + (u & 1) * (size_t)b_bytes, &tB, &fullB[u & 1], (kb0 + kb) * SPLIT_KB, p * nt, 0);
        }
        __device__ void drain_a(int q) const { mbar_wait(&fullA[q % SPLIT_STAGES], (uint32_t)(q / SPLIT_STAGES) & 1, abort, false); }
        __device__ void drain_b(int u) const { mbar_wait(&fullB[u & 1], (uint32_t)(u / 2) & 1, abort, false); }
      } ops{tA, tB, sA, sB, fullA, emptyA, fullB, emptyB, abort, b_bytes, nt, nkb, kb0, rt * nkb_all + kb0, 0, 0};
      split_feed<SPLIT_STAGES>(ops, passes * nkb, S);
    }
  } else if (warp == 9) {
    if (lane == 0) {  // MMA issuer
      int n = 0;
      bool ok = true;
      for (int p = 0; p < passes && ok; ++p)
        for (int ch = 0; ch < nch && ok; ++ch) {
          const int c = p * nch + ch;
          if (c > 0 && !mbar_wait(&acce, (uint32_t)(c - 1) & 1, abort, true)) break;
          tc_fence_after();
          for (int kb = ch * KB_PER_CHUNK; kb < min(nkb, (ch + 1) * KB_PER_CHUNK) && ok; ++kb) {
            const int u = p * nkb + kb;
            if (!(ok = mbar_wait(&fullB[u & 1], (uint32_t)(u / 2) & 1, abort, true))) break;
            const uint64_t bd = umma_desc(sB + (u & 1) * (size_t)b_bytes);
            for (int i = 0; i < S; ++i, ++n) {
              const int st = n % SPLIT_STAGES;
              if (!(ok = mbar_wait(&fullA[st], (uint32_t)(n / SPLIT_STAGES) & 1, abort, true))) break;
              tc_fence_after();
              const uint64_t ad = umma_desc(sA + st * A_BYTES);
              const int cols = (S - i) * nt, n1 = cols <= 256 ? cols : 256 / nt * nt;
              const uint32_t d = tmem + (uint32_t)(i * nt), id1 = umma_idesc(n1), id2 = umma_idesc(cols - n1);
#pragma unroll
              for (int j = 0; j < SPLIT_KB / 16; ++j) {
                const uint32_t acc = (kb > ch * KB_PER_CHUNK || i > 0 || j > 0) ? 1u : 0u;
                umma_bf16(d, ad + 2 * j, bd + 2 * j, id1, acc);
                if (cols > n1) umma_bf16(d + n1, ad + 2 * j, bd + (uint64_t)(n1 * SPLIT_KB * 2 / 16) + 2 * j, id2, acc);
              }
              umma_commit(&emptyA[st]);
            }
            if (ok) umma_commit(&emptyB[u & 1]);
          }
          if (ok) umma_commit(&accf);
        }
      // every multiply issued has completed before tensor and shared memory are given back (also after an abort)
      umma_commit(&drain);
      mbar_wait(&drain, 0, abort, false);
    }
  } else {  // epilogue warps: TMEM lanes 32 (warp % 4) .. + 31, half of the columns each warpgroup
    const int half = warp >> 2, hc = nt / 2;  // nt / 2: 8, 16 or 24 columns
    const uint32_t tl = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(half * hc);
    wait_grid();  // the partial sums of the solve before have been read
    bool ok = true;
    for (int p = 0; p < passes; ++p) {
      long long hi[SPLIT_NT / 2], lo[SPLIT_NT / 2];
#pragma unroll
      for (int c = 0; c < SPLIT_NT / 2; ++c) hi[c] = lo[c] = 0;
      for (int ch = 0; ch < nch && ok; ++ch) {
        // every lane polls for itself; whether the warp goes on is one decision for all its lanes (the
        // tensor-memory loads are warp-collective)
        ok = __all_sync(0xffffffffu, mbar_wait(&accf, (uint32_t)(p * nch + ch) & 1, abort, true));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int c8 = 0; c8 < SPLIT_NT / 16; ++c8) {
          if (c8 * 8 >= hc) continue;
          uint32_t r[S][8];
#pragma unroll
          for (int g = 0; g < S; ++g) tmem_ld8(tl + (uint32_t)(g * nt + c8 * 8), r[g]);
          tmem_wait();
#pragma unroll
          for (int g = 0; g < S; ++g)
#pragma unroll
            for (int q = 0; q < 8; ++q) asm volatile("" : "+r"(r[g][q]));
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            int v[S];
#pragma unroll
            for (int g = 0; g < S; ++g) v[g] = (int)__uint_as_float(r[g][q]);
            // |v[g]| <= (g + 1) 2^21: the first two pairs still fit 32 bits
            long long h = hi[c8 * 8 + q], l = lo[c8 * 8 + q];
            h += (long long)(v[0] * 256 + v[1]) * 65536;
            h += v[2] * 256 + v[3];
#pragma unroll
            for (int g = 4; g < S; ++g) l += (long long)v[g] * (1 << 8 * (S - 1 - g));
            hi[c8 * 8 + q] = h;
            lo[c8 * 8 + q] = l;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce);
      }
      // partial sums as they are, [split][row tile][t][row]: consecutive lanes, consecutive 16-byte values
      longlong2 *dst = part + (((long long)kp * n_rt + rt) * T + p * nt + half * hc) * SPLIT_ROWS + (warp & 3) * 32 + lane;
#pragma unroll
      for (int c = 0; c < SPLIT_NT / 2; ++c)
        if (c < hc && p * nt + half * hc + c < T)
          QG_AT(dst, c * SPLIT_ROWS) = ok ? make_longlong2(hi[c], lo[c]) : make_longlong2(SPLIT_LOST, 0);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// Adds the splits' sums (integers: exact in any order) and scales: 32 rows x 8 right-hand sides per block (one
// output per thread, its splits' loads in flight together), turned to [position][t] through shared memory.
constexpr int SUM_T = 8;

template <typename Dc, int S>
__global__ void __launch_bounds__(32 * SUM_T) k_split_sum(const longlong2 *__restrict__ part, const int *__restrict__ aexp,
                                                         const int *__restrict__ bexp, int rows, int T, int ks,
                                                         int n_rt, const __grid_constant__ SplitOut<Dc> out) {
  __shared__ Dc s_v[32][SUM_T + 1];
  const int r0 = blockIdx.x * 32, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int t0 = blockIdx.y * SUM_T, tn = min(SUM_T, T - t0);
  const int ea = QG_AT(aexp, min(r0 + lane, rows - 1));
  wait_grid();
  const int t = min(t0 + wid, T - 1);
  const longlong2 *src = part + ((long long)(r0 / SPLIT_ROWS) * T + t) * SPLIT_ROWS + r0 % SPLIT_ROWS + lane;
  const int eb = QG_AT(bexp, t);
  long long hi = 0, lo = 0;
  bool lost = ea == SPLIT_NONFINITE || eb == SPLIT_NONFINITE;
#pragma unroll 8
  for (int q = 0; q < ks; ++q) {
    const longlong2 v = QG_AT(src, (long long)q * n_rt * T * SPLIT_ROWS);
    lost |= v.x == SPLIT_LOST;
    hi += v.x;
    lo += v.y;
  }
  s_v[lane][wid] = lost ? dc_nan(Dc{}) : split_value<S>(hi, lo, ea + eb, Dc{});
  __syncthreads();
  const int r = threadIdx.x / SUM_T, tt = threadIdx.x % SUM_T, pos = out.pos0 + r0 + r;
  if (r0 + r >= rows || tt >= tn) return;
  const Dc v = s_v[r][tt];
  QG_AT(out.u, (long long)pos * T + t0 + tt) = v;
  QG_AT(out.th, (long long)pos * T + t0 + tt) = v;  // forward: the angles; adjoint: eta (transformer gradients)
  if (out.pos_gb) {
    const int gb = QG_AT(out.pos_gb, pos);
    if (gb >= 0) QG_AT(out.gip, (long long)(t0 + tt) * out.gi_ld + gb) = v;
  }
}

// The exponent e with m < 2^e of the operands whose largest magnitude m has the key (split_key), over the whole
// range of the type; SPLIT_NONFINITE where there is an infinity or NaN.
__device__ __forceinline__ int split_exp(unsigned key, double) {
  return key >= 0x7ff00000u ? SPLIT_NONFINITE : max((int)(key >> 20), 1) - 1022;
}
__device__ __forceinline__ int split_exp(unsigned key, df32) {
  return key >= 0x7f800000u ? SPLIT_NONFINITE : max((int)(key >> 23), 1) - 126;
}

// Digit i of x (the value times 2^(8 S - 2 - e), |x| <= 2^(8 S - 2)), most significant first.
template <int S>
__device__ __forceinline__ void digits(long long x, float (&q)[S]) {
#pragma unroll
  for (int i = S - 1; i > 0; --i) {
    const int d = (int)(signed char)(x & 0xff);
    q[i] = (float)d;
    x = (x - d) >> 8;
  }
  q[0] = (float)(int)x;
}

// v 2^n as an integer, in two steps within the type's range (exact down to what rounds to zero).
__device__ __forceinline__ long long fixed_point(double v, int n) {
  const int h = n >> 1;
  return __double2ll_rn(v * __hiloint2double((h + 1023) << 20, 0) * __hiloint2double((n - h + 1023) << 20, 0));
}
__device__ __forceinline__ long long fixed_point(df32 v, int n) {
  const int h = n >> 1;
  const float k1 = __int_as_float((h + 127) << 23), k2 = __int_as_float((n - h + 127) << 23);
  return __float2ll_rn(v.hi * k1 * k2) + __float2ll_rn(v.lo * k1 * k2);
}

// Set-up: digits of one row of A per block, into the tiles [row tile][K block][digit][128][64] (whose pads stay 0).
template <int S>
__global__ void __launch_bounds__(256) k_split_rows(const double *__restrict__ src, int K, __nv_bfloat16 *__restrict__ a,
                                                    int *__restrict__ aexp) {
  __shared__ unsigned red[8];
  __shared__ int s_e;
  const double *row = src + (long long)blockIdx.x * K;
  unsigned mx = 0;
  for (int k = threadIdx.x; k < K; k += 256) mx = max(mx, split_key(QG_AT(row, k)));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) mx = max(mx, red[w]);
    s_e = split_exp(mx, 0.0);
    QG_AT(aexp, blockIdx.x) = s_e;
  }
  __syncthreads();
  const int rt = blockIdx.x / SPLIT_ROWS, r = blockIdx.x % SPLIT_ROWS, nkb = (K + SPLIT_KB - 1) / SPLIT_KB;
  for (int k = threadIdx.x; k < K; k += 256) {
    float q[S];
    digits<S>(s_e != SPLIT_NONFINITE ? fixed_point(QG_AT(row, k), 8 * S - 2 - s_e) : 0ll, q);
    __nv_bfloat16 *dst = a + (((long long)(rt * nkb + k / SPLIT_KB) * S) * SPLIT_ROWS + r) * SPLIT_KB + k % SPLIT_KB;
#pragma unroll
    for (int i = 0; i < S; ++i) QG_AT(dst, (long long)i * SPLIT_ROWS * SPLIT_KB) = __float2bfloat16_rn(q[i]);
  }
}

// Digits of the right-hand sides: 64 rows x SPLIT_RT columns of z [K][T] per block, turned to [digit][t][k] through shared memory.
template <typename Dc, int S>
__global__ void __launch_bounds__(256) k_split_rhs(const Dc *__restrict__ z, int K, int T, __nv_bfloat16 *__restrict__ b, long long ld,
                                                   long long slice, const unsigned *__restrict__ bmax,
                                                   int *__restrict__ bexp) {
  __shared__ Dc s_z[SPLIT_KB][SPLIT_RT + 1];
  __shared__ int s_e[SPLIT_RT];
  const int k0 = blockIdx.x * SPLIT_KB, kn = min(SPLIT_KB, K - k0), lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  wait_grid();
  const int t0 = blockIdx.y * SPLIT_RT, tn = min(SPLIT_RT, T - t0);
  for (int e = threadIdx.x; e < kn * tn; e += 256) {
    const int k = e / tn, t = e - k * tn;
    s_z[k][t] = QG_AT(z, (long long)(k0 + k) * T + t0 + t);
  }
  if ((int)threadIdx.x < tn) {
    unsigned m = 0;
#pragma unroll
    for (int q = 0; q < SPLIT_SPREAD; ++q) m = max(m, QG_AT(bmax, q * T + t0 + threadIdx.x));
    s_e[threadIdx.x] = split_exp(m, Dc{});
    if (blockIdx.x == 0) QG_AT(bexp, t0 + threadIdx.x) = s_e[threadIdx.x];
  }
  __syncthreads();
  for (int t = wid; t < tn; t += 8) {  // lanes: pairs of consecutive k, one 128-byte line per (digit, t)
    const bool ok = s_e[t] != SPLIT_NONFINITE;
    const int n = 8 * S - 2 - s_e[t];
    float q0[S], q1[S];
    const int k = 2 * lane;
    digits<S>(k < kn && ok ? fixed_point(s_z[k][t], n) : 0ll, q0);
    digits<S>(k + 1 < kn && ok ? fixed_point(s_z[k + 1][t], n) : 0ll, q1);
    if (k0 + k < (int)ld)
#pragma unroll
      for (int i = 0; i < S; ++i)
        QG_AT(reinterpret_cast<__nv_bfloat162 *>(b + i * slice + (long long)(t0 + t) * ld + k0 + k), 0) =
            __floats2bfloat162_rn(q0[i], q1[i]);
  }
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kern)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t s, bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
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

bool encode(CUtensorMap *map, __nv_bfloat16 *ptr, int rank, const cuuint64_t *dims, const cuuint64_t *strides, const cuuint32_t *box) {
  const auto enc = encoder();
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc && enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

long long split_elems(const SplitMat &m, int digits) {
  return (long long)((m.rows + SPLIT_ROWS - 1) / SPLIT_ROWS) * ((m.K + SPLIT_KB - 1) / SPLIT_KB) * digits * SPLIT_ROWS * SPLIT_KB;
}

bool split_maps(SplitMat &m, int digits) {
  const cuuint64_t da[2] = {SPLIT_KB, (cuuint64_t)(split_elems(m, digits) / SPLIT_KB)}, sa[1] = {SPLIT_KB * 2};
  const cuuint32_t ba[2] = {SPLIT_KB, SPLIT_ROWS};
  const cuuint64_t db[3] = {(cuuint64_t)m.K, (cuuint64_t)m.T, (cuuint64_t)digits};
  const cuuint64_t sb[2] = {(cuuint64_t)m.ld * 2, (cuuint64_t)m.ld * (cuuint64_t)m.T * 2};
  const cuuint32_t bb[3] = {SPLIT_KB, (cuuint32_t)m.nt, (cuuint32_t)digits};
  return encode(&m.ta, m.a, 2, da, sa, ba) && encode(&m.tb, m.b, 3, db, sb, bb);
}

#ifdef QG_CHECK_BOUNDS
void split_check_upload(const QgRange *v, int n) { check_upload(v, n); }
void split_check_first(int *line, unsigned long long *addr) {
  check_first(line, addr);
  if (*line) *line += 100000;
}
#endif

cudaError_t split_prepare(int digits) {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  return digits == 8 ? cudaFuncSetAttribute(k_split_gemm<8>, attr, (int)split_smem_bytes<8>())
                     : cudaFuncSetAttribute(k_split_gemm<7>, attr, (int)split_smem_bytes<7>());
}

cudaError_t split_matrix(const SplitMat &m, const double *src, int digits, cudaStream_t s) {
  if (digits == 8) k_split_rows<8><<<m.rows, 256, 0, s>>>(src, m.K, m.a, m.aexp);
  else k_split_rows<7><<<m.rows, 256, 0, s>>>(src, m.K, m.a, m.aexp);
  return cudaGetLastError();
}

template <typename Dc>
cudaError_t split_rhs(const SplitMat &m, const Dc *z, cudaStream_t s, bool pdl) {
  return launch(k_split_rhs<Dc, split_digits<Dc>()>, dim3((m.K + SPLIT_KB - 1) / SPLIT_KB, (m.T + SPLIT_RT - 1) / SPLIT_RT), 256, 0, s, pdl, z, m.K, m.T, m.b, m.ld,
                m.ld * m.T, (const unsigned *)m.bmax, m.bexp);
}

template <typename Dc>
cudaError_t split_product(const SplitMat &m, const SplitOut<Dc> &out, cudaStream_t s, bool pdl) {
  constexpr int S = split_digits<Dc>();
  const int n_rt = (m.rows + SPLIT_ROWS - 1) / SPLIT_ROWS;
  cudaError_t e = launch(k_split_gemm<S>, dim3(n_rt * m.ks), SPLIT_THREADS, split_smem_bytes<S>(), s, pdl, m.ta, m.tb,
                         (longlong2 *)m.part, n_rt, m.K, m.T, m.nt, m.ks, m.kbps);
  if (e == cudaSuccess)
    e = launch(k_split_sum<Dc, S>, dim3((m.rows + 31) / 32, (m.T + SUM_T - 1) / SUM_T), 32 * SUM_T, 0, s, pdl,
               (const longlong2 *)m.part, (const int *)m.aexp, (const int *)m.bexp, m.rows, m.T, m.ks, n_rt, out);
  return e;
}

template cudaError_t split_rhs<double>(const SplitMat &, const double *, cudaStream_t, bool);
template cudaError_t split_rhs<df32>(const SplitMat &, const df32 *, cudaStream_t, bool);
template cudaError_t split_product<double>(const SplitMat &, const SplitOut<double> &, cudaStream_t, bool);
template cudaError_t split_product<df32>(const SplitMat &, const SplitOut<df32> &, cudaStream_t, bool);

}  // namespace qg
