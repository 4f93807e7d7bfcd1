// Pieces every tcgen05 GEMM of this library shares: tile constants, bounded mbarrier waits with their error
// codes, ring bookkeeping, the fused output activation and the parameter block.
//
// Every wait on an mbarrier is bounded: after WaitEnv::limit_ns without progress (or as soon as another CTA
// has reported an error) the role leaves its loop, the CTA records a code in *err and exits through the common
// tail that frees TMEM.  Nothing built on these helpers can spin forever.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "ptx.cuh"

namespace w4a4 {

constexpr int kBM = 128;            // output tile rows (tokens) of one CTA
constexpr int kBN = 128;            // output tile columns (output channels)
constexpr int kBK = 128;            // K codes per pipeline stage = 2 quantization groups
constexpr int kGemmThreads = 640;
constexpr int kEpiWarp0 = 4, kEpiWarps = 16;
constexpr int kEpiCols = kBN / (kEpiWarps / 4);   // output channels per epilogue thread (32)

constexpr uint64_t kWaitLimitNs = 2000000000ull;     // 2 s: default limit of a bounded wait

enum GemmErr : int {
  kErrNone = 0,
  kErrProducerWait = 101,
  kErrMmaWait = 103,
  kErrEpilogueWait = 104,
  kErrProbeWait = 105,
};

struct WaitEnv {
  int* g_err;                // device-global error word (0 = healthy)
  volatile int* s_abort;     // CTA-local abort flag in shared memory
  uint64_t limit_ns;         // how long a wait may go without progress
};

// Slow path of a bounded wait, kept out of line so that the callers' loops stay small.  ROLE only separates the
// instantiations: an out-of-line function called from warp roles that run under different register budgets
// (setmaxnreg) would have to fit all of them.
template <int BACKOFF_NS, int ROLE>
__device__ __noinline__ bool bounded_wait_slow(uint32_t bar, uint32_t parity, int* g_err, volatile int* s_abort,
                                               uint64_t limit_ns, int code) {
  const uint64_t t0 = global_timer_ns();
  uint32_t spins = 0;
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (BACKOFF_NS > 0) __nanosleep(BACKOFF_NS);  // roles that run ahead poll lazily: issue slots belong to the epilogue
    if ((++spins & 31u) == 0) {
      if (*s_abort) return false;
      if (*reinterpret_cast<volatile int*>(g_err) != 0) {
        *s_abort = 1;
        return false;
      }
      if (global_timer_ns() - t0 > limit_ns) {
        atomicCAS(g_err, 0, code);
        *s_abort = 1;
        return false;
      }
    }
  }
}

// Bounded wait.  Returns false if the CTA should give up.  mbarrier.try_wait itself blocks for a while before it
// reports failure, so a short inline run of attempts covers every hand-over of a healthy pipeline; only a wait that
// outlasts it pays for the out-of-line call and its timer reads.
template <int BACKOFF_NS = 0, int ROLE = 0>
__device__ __forceinline__ bool bounded_wait(uint32_t bar, uint32_t parity, const WaitEnv& env, int code) {
#pragma unroll 1
  for (int i = 0; i < 16; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
  }
  return bounded_wait_slow<BACKOFF_NS, ROLE>(bar, parity, env.g_err, env.s_abort, env.limit_ns, code);
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one_lane() {
  uint32_t pred;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "elect.sync _|p, 0xffffffff;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(pred));
  return pred != 0;
}

// Position in a ring of N mbarrier pairs: slot index and the parity of the phase a consumer waits
// for (a producer waits for parity ^ 1).  Advanced incrementally: no division in the hot loops.
template <int N>
struct Ring {
  uint32_t slot = 0, parity = 0;
  __device__ __forceinline__ void advance() {
    if (++slot == N) {
      slot = 0;
      parity ^= 1u;
    }
  }
};

// Output activation of the layer (W4A4_ACT_*), applied in FP32 before the BF16 rounding.
// GELU, tanh form: 0.5 y (1 + tanh u) with u = sqrt(2/pi) (y + 0.044715 y^3) equals y * sigmoid(2 u) =
// y / (1 + exp(-2 u)); written that way it needs one ex2 and one reciprocal (both accurate to about 2^-22) instead
// of a full-precision tanh, and has no cancellation for negative y.
__device__ __forceinline__ float apply_activation(float y, int act) {
  if (act == 1) {
    const float y2 = y * y;
    // -2 u log2(e) = y (c1 + c3 y^2)
    const float t = y * fmaf(y2, -2.0f * 0.7978845608028654f * 0.044715f * 1.4426950408889634f,
                             -2.0f * 0.7978845608028654f * 1.4426950408889634f);
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(t));
    float rcp;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rcp) : "f"(1.0f + e));
    return y * rcp;
  }
  return y;
}

__device__ __forceinline__ uint32_t bf16x2_bits(float2 v) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(v.x, v.y);
  return *reinterpret_cast<const uint32_t*>(&b);
}

// acc + (a0 - b0)^2 + (a1 - b1)^2 for two pairs of BF16 values.
__device__ __forceinline__ float sq_diff_bf16x2(uint32_t a, uint32_t b, float acc) {
  const float d0 = __uint_as_float(a << 16) - __uint_as_float(b << 16);
  const float d1 = __uint_as_float(a & 0xffff0000u) - __uint_as_float(b & 0xffff0000u);
  return fmaf(d1, d1, fmaf(d0, d0, acc));
}

// n / divisor by one high multiplication and a shift, for n < 2^31 (round-up method: Granlund and Montgomery, "Division by
// invariant integers using multiplication", 1994).  A plain division cost the epilogue's tile change ~300 clocks each.
struct FastDiv {
  uint32_t divisor = 1, mul = 0, shift = 0;
  FastDiv() = default;
  explicit FastDiv(uint32_t d) : divisor(d) {
    while ((1ull << shift) < d) ++shift;
    mul = static_cast<uint32_t>((((1ull << shift) - d) << 32) / d + 1);
  }
  __device__ uint32_t quotient(uint32_t n) const { return (__umulhi(n, mul) + n) >> shift; }
};

// Order of the INT4 GEMM's output tiles: super-columns of `width` column tiles, all row blocks of one before the next;
// width == number of column tiles: plain row-major order.
struct TileOrder {
  FastDiv per_sc, width, last_width;   // tiles of a full super-column; its width; the width of what is left (if anything)
  uint32_t full = 0;                   // full super-columns
  TileOrder() = default;
  TileOrder(int tiles_m, int tiles_n, int sc)
      : per_sc(static_cast<uint32_t>(tiles_m) * sc), width(sc), last_width(tiles_n % sc ? tiles_n % sc : sc), full(tiles_n / sc) {}
};

struct GemmParams {
  const float* bias;    // [N] or nullptr
  uint16_t* Y;          // [M, N] BF16
  int M, N, K, r;
  int tiles_m, tiles_n;
  TileOrder order;
  int splits;           // CTAs of a cluster that share a tile's K (1: K is not split)
  int* err;
  uint64_t wait_limit_ns;
  int32_t* dbg_P;       // debug tap: [kBM, G, kBN] or nullptr
  int dbg_m0, dbg_n0;
  int dbg_stall_stage;  // test hook of the tap instantiation: every CTA's producer skips its stage of this number (-1: none)
  int dbg_late_warp;    // the same: issuing warp that waits dbg_late_ns in front of every tile (-1: none)
  uint64_t dbg_late_ns;
  // Clip-ratio search (Eq. 10): when yref is set, Y is not stored; the squared distance between the layer's
  // BF16 output and yref is accumulated into *sq_err instead.
  const uint16_t* yref; // [M, N] BF16 or nullptr
  double* sq_err;
  int act;              // output activation: 0 none, 1 GELU (tanh form)
};

// The end every GEMM kernel of this library shares after its role loops: if a wait gave up, copies that may
// still be in flight get time to land before the CTA's shared memory is released.
__device__ __forceinline__ void drain_after_abort(volatile int* s_abort) {
  if (*s_abort) {
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) __nanosleep(1000);
    __syncthreads();
  }
}

// Has any CTA of the cluster given up?  By whole warps, after a cluster barrier behind the role loops (no flag changes any more);
// `ctas` <= 32.
__device__ __forceinline__ bool cluster_gave_up(volatile int* s_abort, int ctas) {
  const int lane = threadIdx.x & 31;
  const uint32_t word = smem_u32(const_cast<int*>(s_abort));
  return __any_sync(0xffffffffu, lane < ctas && ld_cluster_u32(map_to_cta(word, lane)) != 0u);
}

constexpr int kMaxGemmSplits = 8;   // CTAs that share a tile's K at most: the portable cluster size

// Exercises the give-up path of bounded_wait without any pipeline around it: one warp waits for a phase of an
// mbarrier that nobody ever completes.  No copy, tensor-core operation or TMEM allocation is involved, so there is
// nothing to drain: after limit_ns the wait records kErrProbeWait in *err and the kernel returns normally.
static __global__ void wait_probe_kernel(int* err, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int s_abort;
  if (threadIdx.x == 0) {
    s_abort = 0;
    mbar_init(smem_u32(&bar), 1);
    mbar_fence_init();
  }
  __syncthreads();
  const WaitEnv env{err, &s_abort, limit_ns};
  bounded_wait<0, 9>(smem_u32(&bar), 0, env, kErrProbeWait);
}

}  // namespace w4a4
