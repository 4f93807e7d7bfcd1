// Kernel 1: fused smoothing + per-(token, 64-channel group) 4-bit quantization + code output
// + low-rank down-projection, one streaming pass over the BF16 activations (HBM bound by design).
//
//   Eq. 5      xh = f32(x) * (1/lambda)                      one FP32 multiply per element
//   Eq. 8      a  = max |xh| over the 64-channel group       shuffles among the eight lanes of a row
//   Eq. 9 / 4  s  = (rho * a) / 7 ,  is = 1 / s              correctly rounded, once per (row, group)
//   Eq. 3      q  = clip(rint(xh * is), -8, 7)               ties to even, by an addition that leaves no fraction bits
//   Eq. 7      T  = bf16(xh) L1                              tcgen05.mma kind::f16, accumulated in TMEM over all of K
//
// Work split.  A CTA of up to eight element-wise warps owns 4 STEPS rows per warp and walks the K groups; a lane holds 8
// consecutive channels (16 bytes) of one row per step, eight lanes a group.  The activations come by cp.async into a ring of
// shared memory in which every lane reads back only what it copied itself.  bf16(xh) goes into a K-major 128-byte-swizzled
// tile, from which one more warp issues four tcgen05.mma per group (M = 128, N = r, K = 16 each; the rows past the CTA's own
// read whatever lies behind the tile and only touch accumulator rows that nobody reads) against the group's r x 64 tile
// of L1, which it fetches by TMA into a ring of its own.
// The bound is instruction issue and latency: 93 (MXFP4) to 127 warp instructions per 8 values and lane at r = 32 take 60 to
// 68 % of the issue slots of two CTAs per SM; DRAM traffic is 60 % of what a copy reaches.  So the loop's addresses are kept in
// registers (derived anew in every pass they cost 15 of those instructions: 127 -> 94 us at 32760 x 5120 MXFP4) and the rare cases
// of the scale arithmetic have a branch of their own.  The predecessor held 16 rows of a warp in mma.sync fragments, with r
// accumulators per row in registers.  Eight launches replayed from one graph, 32760 x 5120, INT4 | MXFP4: r = 0 120 -> 99 | 93 ->
// 78 us, r = 32 148 -> 114 | 121 -> 90, r = 64 191 -> 117 | 158 -> 95, r = 96 278 -> 125 (INT4); 32760 x 13824, r = 32 390 -> 300 |
// 320 -> 236.  (335 MB in and 168 | 89 MB out take 76 | 64 us.)
//
// K split (gridDim.y > 1): with few token rows there are too few row blocks to fill the machine, so the K groups are divided
// among gridDim.y CTAs per row block, which form one thread-block cluster when there is a low-rank branch.  Codes and scales
// of different groups are independent; of T every CTA adds up a share of the rows, for which the others push their partial
// sums into its shared memory (st.async on an mbarrier there) and which it adds in split order.  Pulled over distributed
// shared memory between two cluster barriers instead, the end of the kernel took 5000 clocks, pushed about 2000.
// 100 x 5120, r = 32 12.9 -> 5.4 us INT4, 9.0 -> 5.1 MXFP4; 700 x 8192, r = 64 23.2 -> 13.2 | 16.5 -> 10.8.
//
// Weight expansion (ExpandJob): the CTAs past the row blocks turn the layer's 4-bit weights into the byte image the
// INT4 GEMM reads.  It is independent of the activations, so it shares their launch instead of being a kernel between
// two dependent ones; at the large sizes its traffic hides behind the activation CTAs.
//
// Code output, three formats (template parameter FORMAT):
//   kCodesE4M3    one E4M3 byte per code, row-major [M, K]: the tensor-core operand of kernel 2 as it is
//                 (fp8_codes.cuh), fetched by TMA straight into the swizzled operand tile;
//   kCodesInt8    one two's complement byte per code, row-major [M, K], and scales [M, K/64], for callers of
//                 w4a4_quantize_noalloc;
//   kCodesMxfp4   the MXFP4 variant of the layer (OCP MX v1.0: E2M1 elements, one E8M0 scale per 32 channels,
//                 shared exponent floor(log2(rho * block maximum)) - 2): two codes per byte, row-major
//                 [M, K/2], and the scale bytes in the 512-byte atoms the block-scaled tensor-core
//                 instruction wants in TMEM (see mx_gemm_kernel.cuh).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "fp8_codes.cuh"
#include "pipeline.cuh"
#include "ptx.cuh"
#include "quantize_plan.h"

namespace w4a4 {

constexpr int kCodesInt8 = 0, kCodesE4M3 = 1, kCodesMxfp4 = 2;
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// 16 bytes global -> shared, past L1; one commit group per activation stage.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Smooth 8 BF16 values (one 16-byte load) with 8 reciprocals.
__device__ __forceinline__ void smooth8(const uint4& raw, const float4& r0, const float4& r1, float* xh) {
  const float2 a = __fmul2_rn(make_float2(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u)), make_float2(r0.x, r0.y));
  const float2 b = __fmul2_rn(make_float2(__uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u)), make_float2(r0.z, r0.w));
  const float2 c = __fmul2_rn(make_float2(__uint_as_float(raw.z << 16), __uint_as_float(raw.z & 0xffff0000u)), make_float2(r1.x, r1.y));
  const float2 d = __fmul2_rn(make_float2(__uint_as_float(raw.w << 16), __uint_as_float(raw.w & 0xffff0000u)), make_float2(r1.z, r1.w));
  xh[0] = a.x; xh[1] = a.y; xh[2] = b.x; xh[3] = b.y; xh[4] = c.x; xh[5] = c.y; xh[6] = d.x; xh[7] = d.y;
}

// max |v| over a lane's 8 values, with three-input maxima.  PROPAGATE: NaN if any of them is NaN (else NaNs are ignored).
template <bool PROPAGATE>
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
  float d;
  if constexpr (PROPAGATE) asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  else asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
template <bool PROPAGATE>
__device__ __forceinline__ float absmax8(const float* xh) {
  const float a = max3_abs<PROPAGATE>(xh[0], xh[1], xh[2]), b = max3_abs<PROPAGATE>(xh[3], xh[4], xh[5]);
  return max3_abs<PROPAGATE>(max3_abs<PROPAGATE>(a, xh[6], xh[7]), b, b);
}
// ... and over the 2^n neighbouring lanes below LANES.
template <int LANES, bool PROPAGATE>
__device__ __forceinline__ float absmax_lanes(float a) {
#pragma unroll
  for (int o = 1; o < LANES; o *= 2) {
    const float b = __shfl_xor_sync(0xffffffffu, a, o);
    if constexpr (PROPAGATE) asm("max.NaN.f32 %0, %1, %2;" : "=f"(a) : "f"(a), "f"(b));
    else a = fmaxf(a, b);
  }
  return a;
}

// Eq. 8-9 / Eq. 4: s = x / 7 with x = rho * a, and is = 1 / s, both correctly rounded (IEEE); a == 0 -> 0, 0.  A threshold that
// vanishes although the group does not (underflow) has is = inf: the codes are the ends of the range.
__device__ __forceinline__ void group_scale(float rho, float a, float& s, float& is) {
  s = a > 0.0f ? __fdiv_rn(__fmul_rn(rho, a), 7.0f) : 0.0f;
  is = a > 0.0f ? __frcp_rn(s) : 0.0f;
}
// The same for kOrdinaryMin <= x <= kOrdinaryMax, where nothing under- or overflows: an approximation corrected by its exact
// remainder (Markstein, IBM J. Res. Dev. 34, 1990) is the correctly rounded quotient; the tests compare both results with
// group_scale's for every x of the range.  9 instructions instead of 27.
constexpr float kOrdinaryMin = 1e-30f, kOrdinaryMax = 1e30f;
__device__ __forceinline__ void group_scale_ordinary(float x, float& s, float& is) {
  const float seventh = 0.142857142857142857f;
  const float q = __fmul_rn(x, seventh);
  s = __fmaf_rn(__fmaf_rn(-7.0f, q, x), seventh, q);
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s));
  is = __fmaf_rn(__fmaf_rn(-s, y, 1.0f), y, y);
}

// Eq. 3 for a lane's 8 smoothed values: z = xh * is rounded to FP32, then to the nearest integer with ties to even, then
// clamped to [-8, 7].  The result is the code + 8, two to a word.
__device__ __forceinline__ void quantize8(const float* xh, float is, uint32_t* u) {
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    const int a = min(max(__float2int_rn(__fmul_rn(xh[e], is)), -8), 7) + 8, b = min(max(__float2int_rn(__fmul_rn(xh[e + 1], is)), -8), 7) + 8;
    u[e >> 1] = static_cast<uint32_t>(a | (b << 16));
  }
}
// The same where |z| < 2^15 and z is a number (ordinary scale, rho >= kRhoOrdinary: |z| <= 7 / rho): adding 1.5 * 2^23 rounds to the
// nearest even integer and leaves it in the low half-word, and one 16x2 add-min-relu clamps two of them.  16 instructions for
// 8 values, none of them on the conversion unit, whose 8 conversions to integer would take 64 cycles.  `one` is 1 and unknown to
// the compiler: a packed product and a packed sum, even in PTX with .rn, became one FMA that skips the first rounding.
constexpr float kRhoOrdinary = 0x1p-10f;
__device__ __forceinline__ void quantize8_ordinary(const float* xh, float is, float one, uint32_t* u) {
#pragma unroll
  for (int e = 0; e < 8; e += 2) {
    const float2 z = __fmul2_rn(make_float2(xh[e], xh[e + 1]), make_float2(is, is));
    const float2 m = __ffma2_rn(z, make_float2(one, one), make_float2(12582912.0f, 12582912.0f));
    u[e >> 1] = __viaddmin_s16x2_relu(__byte_perm(__float_as_uint(m.x), __float_as_uint(m.y), 0x5410), 0x00080008u, 0x000f000fu);
  }
}
// Test hook: the two short forms above against the general ones, for every threshold whose bit pattern is in [first, first +
// count).  Codes at, next to and far outside every rounding boundary.  *differ: thresholds with a difference.
static __global__ void scale_arithmetic_kernel(uint32_t first, uint32_t count, float one, unsigned long long* differ) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float x = __uint_as_float(first + i);
    if (!(x >= kOrdinaryMin && x <= kOrdinaryMax)) continue;
    float s, is, s_general, is_general;
    group_scale_ordinary(x, s, is);
    group_scale(1.0f, x, s_general, is_general);
    bool bad = __float_as_uint(s) != __float_as_uint(s_general) || __float_as_uint(is) != __float_as_uint(is_general);
    for (int b = 0; b < 64; b += 8) {
      float xh[8];
      uint32_t u[4], u_general[4];
#pragma unroll
      for (int e = 0; e < 8; ++e) {   // boundary (b + e) / 3 and its neighbours below and above
        const int n = (b + e) / 3;
        const float z = n < 17 ? n - 8.5f : (n & 1 ? 7.0f : -7.0f) / (n < 19 ? kRhoOrdinary : 0.25f);
        xh[e] = __uint_as_float(__float_as_uint(__fmul_rn(s, z)) + (b + e) % 3 - 1);
      }
      quantize8_ordinary(xh, is, one, u);
      quantize8(xh, is, u_general);
#pragma unroll
      for (int w = 0; w < 4; ++w) bad = bad || u[w] != u_general[w];
    }
    if (bad) atomicAdd(differ, 1ull);
  }
}

// Codes + 8, two to a word -> E4M3 bytes.  A half-word 0 .. 15 read as FP16 is u 2^-24: two exact FP16 steps make it u - 8,
// and the conversion is exact too.
__device__ __forceinline__ uint2 e4m3_of_codes(const uint32_t* u) {
  uint16_t b[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t h;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(h) : "r"(u[i]), "r"(0x78007800u), "r"(0xa400a400u));   // u 2^-24 2^15 - 2^-6
    asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(h) : "r"(h), "r"(0x60006000u));                           // * 2^9
    asm("cvt.rn.satfinite.e4m3x2.f16x2 %0, %1;" : "=h"(b[i]) : "r"(h));
  }
  uint2 w;
  asm("mov.b32 %0, {%1, %2};" : "=r"(w.x) : "h"(b[0]), "h"(b[1]));
  asm("mov.b32 %0, {%1, %2};" : "=r"(w.y) : "h"(b[2]), "h"(b[3]));
  return w;
}
// ... -> two's complement bytes.
__device__ __forceinline__ uint2 int8_of_codes(const uint32_t* u) {
  uint2 w;
  w.x = ((__byte_perm(u[0], u[1], 0x6420) | 0x80808080u) - 0x08080808u) ^ 0x80808080u;
  w.y = ((__byte_perm(u[2], u[3], 0x6420) | 0x80808080u) - 0x08080808u) ^ 0x80808080u;
  return w;
}

// Where channel c of a group stands in the K order of T's operands: an MMA step of 16 takes four channels from each of four
// runs of 8.  Any order gives a dot product; with this one T keeps the bits that its mma.sync predecessor gave it, and with
// them the 4-bit codes of the fused FFN's hidden activations (another order moved its outputs by 4.5e-4 instead of 1.8e-5).
__host__ __device__ constexpr uint32_t xh_position(uint32_t c) {
  return (c >> 4 & 1) * 32 + (c >> 2 & 1) * 16 + (c >> 5) * 8 + (c >> 3 & 1) * 4 + (c & 3);
}

// Keeps an address that the loop needs from being derived again in every pass.
__device__ __forceinline__ void keep_in_register(uint32_t& v) { asm volatile("" : "+r"(v)); }

// Two entries of T as BF16 high parts and the BF16 rounding of the remainders.
__device__ __forceinline__ uint2 split_t_pair(float t0, float t1) {
  const __nv_bfloat16 h0 = __float2bfloat16_rn(t0), h1 = __float2bfloat16_rn(t1);
  return make_uint2(pack_bf16x2(__bfloat162float(h0), __bfloat162float(h1)), pack_bf16x2(t0 - __bfloat162float(h0), t1 - __bfloat162float(h1)));
}
// Four neighbouring entries of a row of T: high parts to columns c .. c + 3, remainders to R + c .. R + c + 3.
__device__ __forceinline__ void store_t4(uint16_t* row, int R, int c, const float4& t) {
  const uint2 a = split_t_pair(t.x, t.y), b = split_t_pair(t.z, t.w);
  *reinterpret_cast<uint2*>(row + c) = make_uint2(a.x, b.x);
  *reinterpret_cast<uint2*>(row + R + c) = make_uint2(a.y, b.y);
}
// Eight, 16 bytes each.  A lane stores a row of its own, so that every access touches as many sectors as there are rows: in 4-byte
// pieces 20000 x 256, r = 96 INT4 took 21.1 us instead of 10.0, 32760 x 5120 138 instead of 124.
__device__ __forceinline__ void store_t8(uint16_t* row, int R, int c, const uint32_t* t) {
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint2 p = split_t_pair(__uint_as_float(t[2 * i]), __uint_as_float(t[2 * i + 1]));
    hi[i] = p.x, lo[i] = p.y;
  }
  *reinterpret_cast<uint4*>(row + c) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  *reinterpret_cast<uint4*>(row + R + c) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

// Eight FP32 values -> eight E2M1 codes (round to nearest even, saturating at +-6), element 0 in the lowest nibble.
__device__ __forceinline__ uint32_t e2m1x8(const float* v) {
  uint32_t r;
  asm("{\n"
      ".reg .b8 t0, t1, t2, t3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t0, %2, %1;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t1, %4, %3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t2, %6, %5;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t3, %8, %7;\n"
      "mov.b32 %0, {t0, t1, t2, t3};\n"
      "}"
      : "=r"(r)
      : "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]));
  return r;
}

// The token side of the GEMM's scale MMA for one (row, group): the scale as two BF16 pieces, s = h + m up to 2^-16
// relative, laid out [h, h, m, m] against the channel side's [w1, w2, w1, w2].
__device__ __forceinline__ uint2 sop_slots_activation(float s) {
  const uint32_t h = pack_bf16x2(s, s);   // the packed conversion stays off the conversion unit
  const float m = s - __uint_as_float(h << 16);
  return make_uint2(h, pack_bf16x2(m, m));
}

// Weight codes at rest -> the E4M3 byte image the INT4 GEMM reads: [N, K/2] packed as code + 8 (byte j of a row holds
// K offsets 2 j in its low nibble and 2 j + 1 in its high nibble) -> [N, K] bytes.  One step turns 32 codes (16 bytes)
// into 32 bytes; each half-word of an input word is one byte-permute selector.
struct ExpandJob {
  const uint4* packed = nullptr;
  uint4* out = nullptr;
  uint32_t chunks = 0;      // of 32 codes
  uint32_t first_cta = 0;   // blockIdx.x from which CTAs do this instead of quantizing (gridDim.x: none)
};
__device__ __forceinline__ void expand_chunk(const uint4& w, uint4* out) {
  out[0] = make_uint4(e4m3_of_offset_nibbles4(w.x), e4m3_of_offset_nibbles4(w.x >> 16), e4m3_of_offset_nibbles4(w.y),
                      e4m3_of_offset_nibbles4(w.y >> 16));
  out[1] = make_uint4(e4m3_of_offset_nibbles4(w.z), e4m3_of_offset_nibbles4(w.z >> 16), e4m3_of_offset_nibbles4(w.w),
                      e4m3_of_offset_nibbles4(w.w >> 16));
}
constexpr int kExpandUnroll = 4;   // 16-byte loads a thread keeps in flight, in batches: the next one is on its way while one is turned
// `index` / `count`: this thread among all threads that share the job.
__device__ __forceinline__ void expand_weights(const ExpandJob& job, uint32_t index, uint32_t count) {
  uint4 w[kExpandUnroll];
  auto load = [&](uint32_t i) {
#pragma unroll
    for (int j = 0; j < kExpandUnroll; ++j)
      if (i + j * count < job.chunks) w[j] = __ldg(job.packed + i + j * count);
  };
  load(index);
  for (uint32_t i = index; i < job.chunks; i += kExpandUnroll * count) {
    uint4 now[kExpandUnroll];
#pragma unroll
    for (int j = 0; j < kExpandUnroll; ++j) now[j] = w[j];
    load(i + kExpandUnroll * count);
#pragma unroll
    for (int j = 0; j < kExpandUnroll; ++j)
      if (i + j * count < job.chunks) expand_chunk(now[j], job.out + 2 * static_cast<size_t>(i + j * count));
  }
}
// CTAs for a job: up to four batches each where that still leaves two CTAs per SM.
inline int expand_ctas(uint32_t chunks, int threads, int sms) {
  const uint32_t batches = (chunks + kExpandUnroll * threads - 1) / (kExpandUnroll * threads);
  const uint32_t each = batches / (2 * sms);
  return static_cast<int>(each <= 1 ? batches : (batches + (each < 4 ? each : 4) - 1) / (each < 4 ? each : 4));
}
// The same as a kernel of its own, for the GEMM without an activation pass in front of it.
static __global__ void expand_weight_kernel(const ExpandJob job) {
  expand_weights(job, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

struct QuantizeParams {
  const uint16_t* X;        // [M, K] BF16
  int M, K;
  const float* rlam;        // [K] reciprocal smoothing factors
  const float* clip_table;
  int clip_index;
  uint8_t* codes;
  float* scales;            // kCodesE4M3: FP32 [K/64, scales_ld] or nullptr; kCodesInt8: [M, K/64]; kCodesMxfp4: scale atoms
  int scales_ld;            // kCodesE4M3: pitch; kCodesMxfp4: atoms per row block
  uint16_t* t_hilo;         // [M, 2R]
  uint2* a_sop;             // kCodesE4M3: token-side scale operands of the GEMM
  ExpandJob expand;
  int* err;                 // error word of the bounded waits (R > 0)
  int row_warps;            // element-wise warps that a CTA has rows for; a launch may have spare ones, for the expansion
  float one = 1.0f;         // see quantize8_ordinary
  int dbg_stall_group;      // STALL: the group (of the first CTA of a cluster) whose part of L1 is never loaded
  uint64_t dbg_wait_limit_ns;
};

// Two CTAs per SM.  STALL: test hook, one load is withheld, so that the waits for it run into their limit.
template <int R, int FORMAT, int STEPS, bool STALL = false>
__global__ void __launch_bounds__(quantize_threads(R), 2)
quantize_kernel(const __grid_constant__ CUtensorMap tmL1, const QuantizeParams p) {
  const int warps = p.row_warps, cta_rows = quantize_rows(STEPS, warps);
  const int tensor_warp = static_cast<int>(blockDim.x >> 5) - 1;   // R > 0: the last one
  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (blockIdx.x >= p.expand.first_cta) {   // whole clusters: the cluster spans gridDim.y, never blockIdx.x
    grid_dependency_wait();
    grid_dependency_launch();
    const uint32_t cta = (blockIdx.x - p.expand.first_cta) * gridDim.y + blockIdx.y;
    expand_weights(p.expand, cta * blockDim.x + threadIdx.x, (gridDim.x - p.expand.first_cta) * gridDim.y * blockDim.x);
    return;
  }
  // This CTA's share of the groups (all of them unless the launch splits K).
  const int G = p.K >> 6;
  const int g_per_split = (G + gridDim.y - 1) / gridDim.y;
  const int g_begin = min(G, static_cast<int>(blockIdx.y) * g_per_split), g_end = min(G, g_begin + g_per_split);
  const int row0 = blockIdx.x * cta_rows;

  extern __shared__ uint8_t quant_smem[];
  __shared__ __align__(8) uint64_t s_bars[kL1Stages + 2 * kXhBuffers + 2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort_word;
  constexpr uint32_t kTmemCols = R <= 32 ? 32 : (R <= 64 ? 64 : 128);
  const uint32_t ring = R > 0 ? (smem_u32(quant_smem) + 1023u) & ~1023u : smem_u32(quant_smem);
  const uint32_t xh0 = ring + kL1Stages * R * 128, xh_tile = xh_tile_bytes(STEPS, warps);
  const uint32_t x_ring = R > 0 ? xh0 + kXhBuffers * xh_tile : ring;
  const uint32_t bar_l1 = smem_u32(s_bars), bar_xh_full = bar_l1 + 8 * kL1Stages, bar_xh_empty = bar_xh_full + 8 * kXhBuffers,
                 bar_t = bar_xh_empty + 8 * kXhBuffers, bar_push = bar_t + 8;
  // K split: CTA c of the cluster adds up rows [c rows_each, (c + 1) rows_each) of the tile; the others push their partial
  // sums of those rows into its shared memory.
  const uint32_t pushed = x_ring + x_ring_bytes(R, STEPS, warps);
  const int rows = min(cta_rows, p.M - row0), rows_each = (rows + gridDim.y - 1) / gridDim.y;
  const int rows_mine = max(0, min(rows_each, rows - static_cast<int>(blockIdx.y) * rows_each));
  const int active = (rows + 4 * STEPS - 1) / (4 * STEPS);   // element-wise warps that have rows; the others skip the groups
  uint32_t tmem = 0;
  const WaitEnv env{p.err, &s_abort_word, STALL ? p.dbg_wait_limit_ns : kWaitLimitNs};
  auto load_l1 = [&](int it) {   // by one lane
    if (STALL && it == p.dbg_stall_group && blockIdx.y == 0) return;
    const uint32_t bar = bar_l1 + 8 * (it % kL1Stages);
    mbar_arrive_expect_tx(bar, R * 128);
    tma_load_2d(ring + (it % kL1Stages) * (R * 128), &tmL1, bar, 64 * (g_begin + it), 0);
  };
  auto join_setup = [&] {   // barriers and TMEM are there; a cluster's CTAs have all started (the wait comes before the pushes)
    if constexpr (R > 0) {
      __syncthreads();
      tc_fence_after_sync();
      tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
      if (gridDim.y > 1) cluster_arrive();
    }
  };

  if (R > 0 && warp == tensor_warp) {
    // ------------------------------------------------------------------ L1 producer and MMA issuer (one lane issues)
    constexpr uint32_t idesc = umma_idesc(1, 1, 128, R > 0 ? R : 16);
    const bool issuer = elect_one_lane();
    const int n = g_end - g_begin;
    bool ok = true;
    if (issuer) {
      for (int i = 0; i < kL1Stages; ++i) mbar_init(bar_l1 + 8 * i, 1);
      for (int i = 0; i < kXhBuffers; ++i) {
        mbar_init(bar_xh_full + 8 * i, active);
        mbar_init(bar_xh_empty + 8 * i, 1);
      }
      mbar_init(bar_t, 1);
      mbar_init(bar_push, 1);
      mbar_fence_init();
      fence_proxy_async_smem();
      s_abort_word = 0;
      // constants of the layer: no need to wait for the kernel before this one
      for (int it = 0; it < kL1Stages - 1 && it < n; ++it) load_l1(it);
      if (gridDim.y > 1 && rows_mine > 0) mbar_arrive_expect_tx(bar_push, gridDim.y * rows_mine * (R * 4));
    }
    __syncwarp();
    tmem_alloc(smem_u32(&s_tmem), kTmemCols);
    tmem_relinquish();
    tc_fence_before_sync();
    join_setup();
    grid_dependency_wait();
    for (int it = 0; ok && it < n; ++it) {
      const int b = it % kXhBuffers;
      // the tile of the group after next goes where the previous group's was, once its MMAs are done
      if (it > 0)
        ok = __all_sync(0xffffffffu, bounded_wait<0, 5>(bar_xh_empty + 8 * ((it - 1) % kXhBuffers), ((it - 1) / kXhBuffers) & 1u, env, kErrMmaWait));
      if (!ok) break;
      if (issuer && it + kL1Stages - 1 < n) load_l1(it + kL1Stages - 1);
      ok = __all_sync(0xffffffffu, bounded_wait<0, 5>(bar_l1 + 8 * (it % kL1Stages), (it / kL1Stages) & 1u, env, kErrMmaWait)) &&
           __all_sync(0xffffffffu, bounded_wait<0, 5>(bar_xh_full + 8 * b, (it / kXhBuffers) & 1u, env, kErrMmaWait));
      if (!ok) break;
      tc_fence_after_sync();
      if (issuer) {
        const uint32_t a = xh0 + b * xh_tile, l1 = ring + (it % kL1Stages) * (R * 128);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          umma_f16(tmem, umma_desc_k_sw128(a, 32 * kk), umma_desc_k_sw128(l1, 32 * kk), idesc, it > 0 || kk > 0 ? 1u : 0u);
        umma_commit(bar_xh_empty + 8 * b);
        if (it + 1 == n) umma_commit(bar_t);
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------------ element-wise warps
    grid_dependency_wait();
    const int j = lane & 7;                                     // this lane's channels: 8 j .. 8 j + 7 of the group
    const int tile_row = warp * (4 * STEPS) + (lane >> 4) + 2 * (lane >> 3 & 1);   // and rows: + 4 per step
    const float rho = __ldg(p.clip_table + p.clip_index);
    const float x_min = rho >= kRhoOrdinary ? kOrdinaryMin : kOrdinaryMax * 2.0f;   // below it the general path is taken
    // 32-bit byte offsets from the CTA's first row (at most 128 rows of 16384 channels and a margin): half the address
    // arithmetic of 64-bit pointers.
    const uint8_t* const x_base = reinterpret_cast<const uint8_t*>(p.X + static_cast<size_t>(row0) * p.K);
    const uint8_t* const rl_base = reinterpret_cast<const uint8_t*>(p.rlam);
    constexpr uint32_t kCodeBits = FORMAT == kCodesMxfp4 ? 4 : 8;
    uint8_t* const code_base = p.codes + static_cast<size_t>(row0) * (p.K / 8 * kCodeBits);
    uint32_t x_off[STEPS], code_off[STEPS], xh_off[STEPS], scale_off[STEPS];
    bool row_ok[STEPS];
    // Where the scales of row0's 128-row block and of the next one begin: operand images, or atoms.
    const uint32_t block_pitch = FORMAT == kCodesMxfp4 ? p.scales_ld * 512u : ((G + 1) >> 1) * 2048u;
    uint8_t* const scale_base = reinterpret_cast<uint8_t*>(FORMAT == kCodesMxfp4 ? reinterpret_cast<void*>(p.scales) : p.a_sop) +
                                static_cast<size_t>(row0 >> 7) * block_pitch;
#pragma unroll
    for (int s = 0; s < STEPS; ++s) {   // rows past M read the last one and store nothing
      const int r = tile_row + 4 * s;
      row_ok[s] = r < rows;
      x_off[s] = static_cast<uint32_t>(min(r, rows - 1)) * p.K * 2 + 16 * j;
      code_off[s] = static_cast<uint32_t>(r) * (p.K / 8 * kCodeBits) + kCodeBits * j;
      xh_off[s] = xh0 + 128 * r + (xh_position(8 * j) * 2u ^ 16u * (r & 7));
      if constexpr (FORMAT == kCodesMxfp4) {
        // per 128-row block and per 4 scale blocks (128 channels) one 512-byte atom,
        // byte (row % 32) * 16 + (row % 128 / 32) * 4 + (scale block % 4)
        const int row = row0 + r;
        scale_off[s] = ((row >> 7) - (row0 >> 7)) * block_pitch + (row & 31) * 16 + ((row & 127) >> 5) * 4 + (j >> 2);
      } else {
        // The scale as four BF16 slots of the operand from which the GEMM's tensor core forms sx * sw: 2 KiB shared-memory
        // images per (128 rows, 2 groups), [8-row group][8 rows][group parity][8 bytes].  One lane per two steps (below).
        const int row = row0 + r + (STEPS > 1 ? 4 * (j & 1) : 0);
        scale_off[s] = ((row >> 7) - (row0 >> 7)) * block_pitch + ((row & 127) >> 3) * 128 + (row & 7) * 16;
      }
      keep_in_register(x_off[s]), keep_in_register(code_off[s]), keep_in_register(xh_off[s]), keep_in_register(scale_off[s]);
    }
    // A lane copies what it reads itself, and one lane in two 16 bytes of its warp's reciprocals, so a stage needs no
    // barrier beyond its own commit group and a __syncwarp.
    constexpr int kStages = kXStages(R, STEPS);
    const uint32_t stage_bytes = x_stage_bytes(STEPS, warps);
    const uint32_t my_x = x_ring + warp * (STEPS * 512u) + 16u * lane, my_rl = x_ring + warps * (STEPS * 512u) + 256u * warp;
    auto load = [&](int g, uint32_t slot) {
      if (g < g_end) {
#pragma unroll
        for (int s = 0; s < STEPS; ++s) cp_async16(my_x + slot + 512 * s, x_base + (x_off[s] + 128u * g));
        if (lane < 16) cp_async16(my_rl + slot + 16 * lane, rl_base + (256u * g + 16u * lane));
      }
      cp_async_commit();
    };
    // Warps without rows neither load nor walk the groups.  (A branch around the loop: bounds of their own made the loop 3 % longer.)
#pragma unroll
    for (int i = 0; i < kStages - 1; ++i)
      if (warp < active) load(g_begin + i, stage_bytes * i);
    join_setup();   // its microsecond passes beside the first loads
    // The MXFP4 GEMM's CTAs may come in now: every CTA of this grid has started by the time the last one passes here.  They come to SMs
    // that this grid leaves free or is done with, since their shared memory leaves no room beside a CTA that has TMEM (asserted in
    // w4a4_mx_api.cuh): a GEMM's CTA, which takes all of an SM's TMEM and keeps it until this grid has ended, never stands in front of
    // one that this grid waits for.  After the loop instead of here, 1 x 5120 -> 1024 took 8.1 us, 7.5 now.  The INT4 GEMM's CTAs come
    // after the loop.  From here it makes no difference where the launch expands much (forwards replayed from one graph, after the loop
    // | from here: 1 x 5120 -> 5120 26.8 | 26.7 us, 100 x 5120 -> 5120 24.4 | 24.4, 448 x 5120 -> 13824 80.6 | 80.7); of small layers 64 x 512 ->
    // 512, r = 0, gains (7.1 | 6.8) and 256 x 512 -> 512, r = 16, does not (9.2 | 9.2; called one by one 9.40 | 9.57).  (The GEMM itself
    // lets nobody in before its end: the next forward's activation CTAs then sat beside it, 78 -> 84 us at 1560 x 5120 -> 13824 MXFP4.)
    if constexpr (FORMAT == kCodesMxfp4) grid_dependency_launch();
    uint32_t slot = 0, slot_before = stage_bytes * (kStages - 1);   // this group's and the previous group's
    bool ok = true;
    if (warp < active) for (int g = g_begin; g < g_end; ++g) {
      float xh[STEPS][8];
      cp_async_wait<kStages - 2>();
      __syncwarp();
      load(g + kStages - 1, slot_before);
      {
        const float4 rl0 = lds_f32x4(my_rl + slot + 32 * j), rl1 = lds_f32x4(my_rl + slot + 32 * j + 16);
#pragma unroll
        for (int s = 0; s < STEPS; ++s) smooth8(lds_u32x4(my_x + slot + 512 * s), rl0, rl1, xh[s]);
      }
      slot_before = slot;
      slot = slot + stage_bytes == kStages * stage_bytes ? 0u : slot + stage_bytes;
      if constexpr (R > 0) {
        const int it = g - g_begin, b = it % kXhBuffers;
        ok = __all_sync(0xffffffffu, bounded_wait<0, 6>(bar_xh_empty + 8 * b, ((it / kXhBuffers) & 1u) ^ 1u, env, kErrEpilogueWait));
        if (!ok) break;
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
          uint4 v;
          v.x = pack_bf16x2(xh[s][0], xh[s][1]), v.y = pack_bf16x2(xh[s][2], xh[s][3]);
          v.z = pack_bf16x2(xh[s][4], xh[s][5]), v.w = pack_bf16x2(xh[s][6], xh[s][7]);
          sts_u32x2(xh_off[s] + b * xh_tile, v.x, v.y);
          sts_u32x2((xh_off[s] ^ 32u) + b * xh_tile, v.z, v.w);
        }
      }
      // After the scale chain, so that the fence finds its stores done.
      auto publish_xh = [&] {
        if constexpr (R > 0) {
          fence_proxy_async_smem();
          __syncwarp();
          mbar_arrive_if(lane == 0 ? 1u : 0u, bar_xh_full + 8 * ((g - g_begin) % kXhBuffers));
        }
      };
      if constexpr (FORMAT == kCodesMxfp4) {
        float a[STEPS];
#pragma unroll
        for (int s = 0; s < STEPS; ++s) a[s] = absmax_lanes<4, false>(absmax8<false>(xh[s]));
        publish_xh();
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
          const uint32_t field = (__float_as_uint(__fmul_rn(rho, a[s])) >> 23) & 0xffu;   // exponent of the clip threshold (Eq. 8)
          const uint32_t ex = field > 2u ? field - 2u : 0u;                            // minus the exponent of E2M1's top binade
          const float inv = __uint_as_float((254u - ex) << 23);                        // 2^(127 - ex): exact scaling
          float v[8];
#pragma unroll
          for (int e = 0; e < 8; e += 2) {
            const float2 z = __fmul2_rn(make_float2(xh[s][e], xh[s][e + 1]), make_float2(inv, inv));
            v[e] = z.x;
            v[e + 1] = z.y;
          }
          const uint32_t w = e2m1x8(v);
          if (row_ok[s]) {
            *reinterpret_cast<uint32_t*>(code_base + (code_off[s] + 32u * g)) = w;
            if ((j & 3) == 0) scale_base[scale_off[s] + ((g >> 1) * 512u + (g & 1) * 2u)] = static_cast<uint8_t>(ex);
          }
        }
      } else {
        // Two steps share the scale arithmetic: even lanes derive the first row's, odd lanes the second's.
        float s_mine[STEPS], is_mine[STEPS], is[STEPS];
        bool ordinary = true;
        uint32_t u[STEPS][4];
        {
          float a[STEPS];
#pragma unroll
          for (int s = 0; s < STEPS; ++s) a[s] = absmax_lanes<8, true>(absmax8<true>(xh[s]));
#pragma unroll
          for (int s = 0; s < STEPS; s += 2) {
            const float x = __fmul_rn(rho, STEPS > 1 && (j & 1) ? a[s + 1 < STEPS ? s + 1 : s] : a[s]);
            ordinary = ordinary && x >= x_min && x <= kOrdinaryMax;
            group_scale_ordinary(x, s_mine[s], is_mine[s]);
          }
        }
        publish_xh();
        auto share = [&] {
#pragma unroll
          for (int s = 0; s < STEPS; s += 2) {
            is[s] = is_mine[s];
            if constexpr (STEPS > 1) {
              const float is_other = __shfl_xor_sync(0xffffffffu, is_mine[s], 1);
              is[s] = (j & 1) ? is_other : is_mine[s];
              is[s + 1] = (j & 1) ? is_mine[s] : is_other;
            }
          }
        };
        if (__all_sync(0xffffffffu, ordinary)) {
          share();
#pragma unroll
          for (int s = 0; s < STEPS; ++s) quantize8_ordinary(xh[s], is[s], p.one, u[s]);
        } else {   // an empty group, or magnitudes at the ends of FP32's range, or no numbers at all
          float a[STEPS];
#pragma unroll
          for (int s = 0; s < STEPS; ++s) a[s] = absmax_lanes<8, false>(absmax8<false>(xh[s]));
#pragma unroll
          for (int s = 0; s < STEPS; s += 2)
            group_scale(rho, STEPS > 1 && (j & 1) ? a[s + 1 < STEPS ? s + 1 : s] : a[s], s_mine[s], is_mine[s]);
          share();
#pragma unroll
          for (int s = 0; s < STEPS; ++s) quantize8(xh[s], is[s], u[s]);
        }
#pragma unroll
        for (int s = 0; s < STEPS; ++s) {
          const uint2 w = FORMAT == kCodesE4M3 ? e4m3_of_codes(u[s]) : int8_of_codes(u[s]);
          uint8_t* const dst = code_base + (code_off[s] + 64u * g);
          if (FORMAT == kCodesInt8 && (reinterpret_cast<uintptr_t>(p.codes) & 7) != 0) {   // a caller's buffer on any boundary
#pragma unroll
            for (int e = 0; e < 8; ++e)
              if (row_ok[s]) dst[e] = static_cast<uint8_t>((e < 4 ? w.x : w.y) >> (8 * (e & 3)));
          } else if (row_ok[s]) {
            *reinterpret_cast<uint2*>(dst) = w;
          }
        }
#pragma unroll
        for (int s = 0; s < STEPS; s += 2) {
          if (j < (STEPS > 1 ? 2 : 1) && (STEPS > 1 && j == 1 ? row_ok[s + 1 < STEPS ? s + 1 : s] : row_ok[s])) {
            const float sc = s_mine[s];
            const size_t row = row0 + tile_row + 4 * s + (STEPS > 1 ? 4 * j : 0);
            if constexpr (FORMAT == kCodesInt8) {
              p.scales[row * G + g] = sc;
            } else {
              *reinterpret_cast<uint2*>(scale_base + (scale_off[s] + ((g >> 1) * 2048u + (g & 1) * 8u))) = sop_slots_activation(sc);
              if (p.scales != nullptr) p.scales[static_cast<size_t>(g) * p.scales_ld + row] = sc;   // for the parity tap
            }
          }
        }
      }
    }
    cp_async_wait<0>();
    if constexpr (FORMAT != kCodesMxfp4) grid_dependency_launch();
    if constexpr (R > 0) {
      // T: TMEM lane = row of the tile; warp w reads lanes 32 w .. 32 w + 31.
      if (32 * warp < cta_rows && warp < 4) {
        const bool any = g_begin < g_end;
        if (gridDim.y > 1) cluster_wait();
        if (ok && any) ok = __all_sync(0xffffffffu, bounded_wait<0, 6>(bar_t, 0u, env, kErrEpilogueWait));
        tc_fence_after_sync();
        const int r = 32 * warp + lane, row = row0 + r;
#pragma unroll
        for (int c = 0; c < R; c += 16) {
          uint32_t v[16];
          if (any) {
            tmem_ld_32x32b_x16(tmem + (static_cast<uint32_t>(32 * warp) << 16) + c, v);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = 0u;
          }
          if (gridDim.y == 1) {
            if (ok && r < rows) {
#pragma unroll
              for (int e = 0; e < 16; e += 8) store_t8(p.t_hilo + static_cast<size_t>(row) * (2 * R), R, c + e, v + e);
            }
          } else if (ok && r < rows) {
            const uint32_t owner = r / rows_each, at = pushed + ((blockIdx.y * rows_each + r - owner * rows_each) * R + c) * 4;
            const uint32_t to = map_to_cta(at, owner), bar = map_to_cta(bar_push, owner);
#pragma unroll
            for (int e = 0; e < 16; e += 4) st_async_u32x4(to + 4 * e, make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]), bar);
          }
        }
        tc_fence_before_sync();
      }
    }
  }
  if constexpr (R > 0) {
    if (gridDim.y > 1) {
      if (!(warp < 4 && 32 * warp < cta_rows)) cluster_wait();
      cluster_arrive();
      if (warp < warps && rows_mine > 0 &&
          __all_sync(0xffffffffu, bounded_wait<0, 6>(bar_push, 0u, env, kErrEpilogueWait))) {
        // the partial sums in split order, four columns per thread
        for (int i = threadIdx.x; i < rows_mine * (R / 4); i += 32 * warps) {
          const int r = i / (R / 4), q = i - r * (R / 4);
          const uint32_t at = pushed + 16 * i, pitch = rows_each * (R * 4);
          float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 4
          for (uint32_t c = 0; c < gridDim.y; ++c) {
            const float4 v = lds_f32x4(at + c * pitch);
            t.x += v.x, t.y += v.y, t.z += v.z, t.w += v.w;
          }
          uint16_t* dst = p.t_hilo + static_cast<size_t>(row0 + blockIdx.y * rows_each + r) * (2 * R);
          store_t4(dst, R, 4 * q, t);
        }
      }
      cluster_wait();   // nobody leaves while its shared memory may still be written
    }
    tc_fence_before_sync();
    __syncthreads();
    drain_after_abort(&s_abort_word);
    if (warp == tensor_warp) {
      tc_fence_after_sync();
      tmem_dealloc(tmem, kTmemCols);
    }
  }
}

// T in FP32 [M, r] -> the BF16 high | low pair kernel 2 reads (the fused producer of the MXFP4 variant accumulates T
// in FP32).
static __global__ void t_split_kernel(const float* __restrict__ t32, int M, int r, uint16_t* __restrict__ t_hilo) {
  const size_t idx = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= static_cast<size_t>(M) * r) return;
  const float t = t32[idx];
  const size_t row = idx / r;
  const int c = static_cast<int>(idx % r);
  const __nv_bfloat16 hi = __float2bfloat16_rn(t);
  const __nv_bfloat16 lo = __float2bfloat16_rn(t - __bfloat162float(hi));
  t_hilo[row * 2 * r + c] = *reinterpret_cast<const uint16_t*>(&hi);
  t_hilo[row * 2 * r + r + c] = *reinterpret_cast<const uint16_t*>(&lo);
}

}  // namespace w4a4
