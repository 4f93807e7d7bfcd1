// Kernel 2: fused W4A4 GEMM + per-group rescale + low-rank up-projection + bias + BF16 store.
//
//   Eq. 7 / 11    Y[m,n] = sum_g  P_g[m,n] * sx[m,g] * sw[g,n]  +  sum_j T[m,j] L2[j,n]  +  b[n]
//                 P_g[m,n] = sum_{k in group g} q[m,k] qw[k,n]            (exact: integers in FP32)
//
// Code products.  The 4-bit codes go through the tensor core as E4M3 bytes (fp8_codes.cuh): tcgen05.mma
// kind::f8f6f4 runs at the 8-bit rate and leaves every group's partial sums in TMEM as exact integers already in
// FP32 (|P| <= 4096).  The activation codes come straight from kernel 1, the weight codes from
// the expansion in kernel 1's launch (ExpandJob), which turns the layer's nibble-packed weights (their
// format at rest) into an N x K byte image that stays in L2 for the duration of the GEMM.
//
// Scale products.  The factor S_g = sx[:, g] (x) sw[g, :] is an outer product, i.e. a K = 16 BF16 MMA on operands
// that hold each scale as two BF16 pieces (s = h + m up to 2^-16 relative):
//     token row,   four slots per group:  [h,  h,  m,  m ]
//     channel row, four slots per group:  [w1, w2, w1, w2]      ->  h w1 + h w2 + m w1 + m w2 = sx sw (1 + O(2^-16))
// One 16-byte K chunk of a token row carries the slots of the two groups of a stage; the channel side has one
// chunk per group with zeros in the other group's slots, and every descriptor's second K chunk points at a tile of
// zeros.  The epilogue then needs one fused multiply-add per partial sum, acc += P_g * S_g, on two TMEM fragments
// and reads no scales from shared memory.  Operand tiles of the scale MMA live in global memory as ready-made
// shared-memory images (no-swizzle K-major canonical layout: [8-row group][8 rows][16 bytes]); kernel 1 writes the
// token side, the channel side is built once at pack time.  The low-rank product T L2 goes
// through the same path as one more "group" that opens a tile: its P is the BF16 product [T_hi | T_lo] [L2 | L2]^T,
// which the epilogue takes as the accumulators' first value.
//
// Persistent, one CTA (640 threads) per SM, 128 x 128 tiles, column tile fastest (the CTAs running at any moment
// share a few row blocks of A and a super-column of B through L2).  TMEM: two slots of 256 columns, one per group in flight:
// columns 0..127 P_g, columns 128..255 S_g.  Warp roles:
//   warp 0      producer: per stage of 128 K-codes (two groups) TMA loads of the A and B code tiles (16 KiB each,
//               128-byte swizzle) and of the two scale-operand images, all onto the stage's mbarrier;
//   warps 1, 2  code-MMA issuers, one per TMEM slot (CodeSlotWalk): per group two tcgen05.mma kind::f8f6f4 (K = 32) into the
//               slot's P columns, then a commit onto tmem_full[slot]; the low-rank entry is its slot's warp's;
//   warp 3      scale-MMA issuer: per group one tcgen05.mma kind::f16 (K = 16) into the slot's S columns and a commit
//               onto the same barrier (it counts two arrivals).  The issue of a tcgen05.mma waits for room in the tensor
//               pipe's queue and the loop around it costs as much again, so that one thread with everything to issue is
//               late for every slot: with one code-MMA warp a group takes 330 clocks, with two 321 (a fourth issuing warp for the
//               scale MMAs gained nothing, both products of a group from one warp lost 4 %);
//   warp 2      also TMEM allocation;
//   warps 4-19  epilogue: a thread owns one token row and 32 output channels.  Per group two round trips of two
//               tcgen05.ld.32x32b.x16 (P and S of 16 columns) with the eight packed multiply-adds of the first half
//               in between; the slot goes back to the issuing warps (tmem_empty[slot], 16 arrivals) as soon as the
//               second half is in registers.  Measured alternatives (all four loads in one round trip; the second
//               half's loads issued ahead of the first half's arithmetic; warps of a scheduler skewed against one
//               another) were slower.
// What bounds the kernel is the round trip of a TMEM slot, of which there are two: release, issue, MMAs, commit, wait, loads.
// 321 clocks per group and 2.7 thousand per tile beside its groups (sm__cycles_active at 4736 rows -> 5120, K = 2560 and 10240).
// Without any operand loads it took as long, with an epilogue that loads 16 columns and adds nothing 0.80 of that, with one MMA
// instead of three beside that 0.71 (measured with one code-MMA warp).
// Epilogue warps that form the scale products themselves leave room for three or four slots, but their broadcast reads of the
// channel scales made a group take 1.6 times as long (two CTAs per SM) or twice (16 warps with 8 of 32 channels' products from
// the tensor core).  A lone warp's dependent instructions
// cost 10-15 cycles each and a branch on a fresh mbarrier result ~70, so the hops are written as single instruction
// sequences without branches: wait_issue_* (try_wait, then fence, MMAs and commit predicated on its answer),
// wait_then_ld16 (try_wait, a vote, then fence and first TMEM load predicated on it), descriptors computed before the wait, and
// predicated instead of branched single-lane instructions (umma_*_if, mbar_arrive_if).  A wait that outlasts the
// try_wait falls back to the bounded wait of pipeline.cuh and the same instructions issued from C++.  The slots' addresses are
// toggled, not derived from a counter (342 clocks per group -> 318, before the vote in wait_then_ld16, which costs three).
// The tile's end: outputs in BF16 through a swizzled tile in shared memory and out by one TMA store per warp, which the next
// tile does not wait for.  16-byte stores from registers held the warps for 1150 of the tile change's 2600 clocks.
// Tile order: column tiles are walked in super-columns (GemmParams::order, all row blocks of a
// super-column before the next) sized so that the weight bytes a wave of CTAs touches stay in L2; with the plain
// row-major order the 71 MB weight image of the FFN shapes streamed from DRAM once per 1.4 row blocks.
// Split K (SPLIT instantiation): where the tiles alone leave most SMs idle, the CTAs of a thread-block cluster share one
// tile, each over its part of the operand stages (the first one with the low-rank product).  Their FP32 partial tiles meet
// in shared memory (the operand ring's, idle by then), and every CTA adds its share of them over distributed shared
// memory in split order, so results do not depend on timing; none does once a member has given up on a wait.  One tile per
// CTA, no loop.
// Every role loops warp-uniformly (waits are voted, only the TMA / tcgen05 instructions are predicated on one elected
// lane), which keeps ring positions, addresses and descriptors in uniform registers.  All waits are bounded
// (pipeline.cuh).  Finally + bias -> optional GELU -> BF16, or the squared error against a reference (clip search).
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "pipeline.cuh"
#include "ptx.cuh"
#include "tmem_slots.h"

namespace w4a4 {

constexpr int kGemmStages = 5;
constexpr uint32_t kOpATile = kBM * kBK;              // 16 KiB: 128 token rows x 128 codes
constexpr uint32_t kOpBTile = kBN * kBK;              // 16 KiB: 128 weight rows x 128 codes
constexpr uint32_t kSopATile = kBM * 16;              // 2 KiB: 128 token rows x one 16-byte chunk (two groups)
constexpr uint32_t kSopBTile = 2 * kBN * 16;          // 4 KiB: per group 128 channel rows x one 16-byte chunk
constexpr uint32_t kStageBytes = kOpATile + kOpBTile + kSopATile + kSopBTile;   // 38 KiB
constexpr uint32_t kLrStageBytes = kOpATile + kOpBTile;   // a low-rank stage: T tile and L2 rows
constexpr uint32_t kZeroTile = 2048;                  // tile of zeros: 128 rows x 16 bytes
constexpr uint32_t kOutTile = 32 * 2 * kEpiCols;      // an epilogue warp's 32 x 32 outputs in BF16
constexpr uint32_t kGemmNumBarriers = 2 * kGemmStages + 2 * kTmemSlots;
constexpr uint32_t kGemmSmemBytes = 1024 + kGemmStages * kStageBytes + kZeroTile + kEpiWarps * kOutTile + kGemmNumBarriers * 8 + 16;
static_assert(kGemmSmemBytes <= 232448, "shared memory budget of one CTA");
static_assert(kStageBytes % 1024 == 0, "operand tiles must stay 1024-byte aligned");

// Register budgets.  640 threads are launched with 96 registers each; the control warpgroup gives most of its share to the
// epilogue's four.  What the compiler makes of the epilogue's loop decides the kernel (clocks per 128 x 128 tile at K = 5120, before
// TMA stores and a second code-MMA warp: 96 registers 31314, 112 30529; 28.4 thousand now).
constexpr int kGemmRegs = 96, kControlRegs = 32, kEpilogueRegs = 112;
static_assert((kGemmThreads - 32 * kEpiWarps) * kControlRegs + 32 * kEpiWarps * kEpilogueRegs <= kGemmThreads * kGemmRegs,
              "a larger sum would wait forever for registers that the launch does not have");

// The epilogue's position in the two TMEM slots: the current slot's column address and full barrier, and its phase.
struct SlotUse {
  uint32_t t, full, phase = 0;
  static_assert(kTmemSlots == 2, "the slots differ in one bit of each address");
  __device__ __forceinline__ SlotUse(uint32_t t0, uint32_t full0) : t(t0), full(full0) {}
  __device__ __forceinline__ uint32_t empty() const { return full + 8 * kTmemSlots; }
  __device__ __forceinline__ void next() { t ^= 2 * kBN, full ^= 8u, phase ^= (~full >> 3) & 1u; }
};

// Wait for a TMEM slot and issue its MMAs in one branch-free instruction sequence: one try_wait (it blocks in hardware
// for a while before it gives up), then the fence, the MMAs and the commit predicated on its answer.  A branch on the
// fresh answer would hold the warp ~70 cycles; a second try_wait predicated on the first one's failure costs its
// latency even when it is skipped (both measured slower).  Returns 0 if the barrier did not complete (the caller then
// takes the bounded wait and issues from C++).
__device__ __forceinline__ uint32_t wait_issue_f8x2(uint32_t go, uint32_t bar, uint32_t parity, uint32_t d_tmem, uint64_t a0, uint64_t b0,
                                                    uint64_t a1, uint64_t b1, uint32_t idesc, uint32_t full_bar) {
  uint32_t done;
  asm volatile(
      "{\n"
      ".reg .pred p, q, pq;\n"
      "setp.ne.b32 q, %6, 0;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "and.pred pq, p, q;\n"
      "@p tcgen05.fence::after_thread_sync;\n"
      "@pq tcgen05.mma.cta_group::1.kind::f8f6f4 [%3], %4, %5, %7, 0;\n"
      "@pq tcgen05.mma.cta_group::1.kind::f8f6f4 [%3], %8, %9, %7, 1;\n"
      "@pq tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%10];\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity), "r"(d_tmem), "l"(a0), "l"(b0), "r"(go), "r"(idesc), "l"(a1), "l"(b1), "r"(full_bar)
      : "memory");
  return done;
}
__device__ __forceinline__ uint32_t wait_issue_f16(uint32_t go, uint32_t bar, uint32_t parity, uint32_t d_tmem, uint64_t a0, uint64_t b0,
                                                   uint32_t idesc, uint32_t full_bar) {
  uint32_t done;
  asm volatile(
      "{\n"
      ".reg .pred p, q, pq;\n"
      "setp.ne.b32 q, %6, 0;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "and.pred pq, p, q;\n"
      "@p tcgen05.fence::after_thread_sync;\n"
      "@pq tcgen05.mma.cta_group::1.kind::f16 [%3], %4, %5, %7, 0;\n"
      "@pq tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%8];\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity), "r"(d_tmem), "l"(a0), "l"(b0), "r"(go), "r"(idesc), "r"(full_bar)
      : "memory");
  return done;
}

// Wait for a full TMEM slot and start its first load in one branch-free instruction sequence.  The load is the whole warp's
// (.sync.aligned, undefined where the lanes' predicates differ), and a barrier that completes during a try_wait may answer the lanes
// differently: hence the vote in front of it, which behind the load would be hidden (32760 x 5120 -> 13824 3954 -> 3980 us).
// Returns 0, to all lanes, if the barrier did not complete within the try_wait of every lane (nothing was loaded then).
__device__ __forceinline__ uint32_t wait_then_ld16(uint32_t bar, uint32_t parity, uint32_t taddr, uint32_t (&v)[16]) {
  uint32_t done;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%17], %18;\n"
      "vote.sync.all.pred p, p, 0xffffffff;\n"
      "@p tcgen05.fence::after_thread_sync;\n"
      "@p tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%19];\n"
      "selp.u32 %16, 1, 0, p;\n"
      "}\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(done)
      : "r"(bar), "r"(parity), "r"(taddr)
      : "memory");
  return done;
}

// Tile raster: column tiles are walked in super-columns of `sc` tiles (all row blocks of one super-column before the
// next), so that the weight bytes a wave of CTAs touches stay in L2.  sc == tiles_n: plain row-major order.
__device__ __forceinline__ void tile_coords(uint32_t tile, const TileOrder& o, int& tm, int& tn) {
  const uint32_t s_idx = o.per_sc.quotient(tile);        // full super-columns before this tile, or all of them
  const uint32_t rem = tile - s_idx * o.per_sc.divisor;
  const bool last = s_idx >= o.full;                      // the narrower super-column that may end the order
  const uint32_t row = last ? o.last_width.quotient(rem) : o.width.quotient(rem);
  tm = static_cast<int>(row);
  tn = static_cast<int>(s_idx * o.width.divisor + rem - row * (last ? o.last_width.divisor : o.width.divisor));
}

// Ties a fragment to the tcgen05.wait::ld in front of it: the registers count as written there, so nothing that
// reads them can be scheduled above the wait (an asm statement takes at most 30 operands, hence one statement per
// fragment; volatile statements keep their order).
__device__ __forceinline__ void tie_fragment(uint32_t (&a)[16]) {
  asm volatile(""
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]), "+r"(a[8]),
                 "+r"(a[9]), "+r"(a[10]), "+r"(a[11]), "+r"(a[12]), "+r"(a[13]), "+r"(a[14]), "+r"(a[15])
               :
               : "memory");
}

// acc[j] += P * S for the fragment's eight column pairs.
template <bool DEBUG>
__device__ __forceinline__ void fma_fragment(const uint32_t (&pv)[16], const uint32_t (&sv)[16], float2* acc, int32_t* dbg_row) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float2 p2 = make_float2(__uint_as_float(pv[2 * j]), __uint_as_float(pv[2 * j + 1]));
    const float2 s2 = make_float2(__uint_as_float(sv[2 * j]), __uint_as_float(sv[2 * j + 1]));
    acc[j] = __ffma2_rn(p2, s2, acc[j]);
    if (DEBUG) {
      if (dbg_row != nullptr) {
        dbg_row[2 * j] = static_cast<int32_t>(p2.x);
        dbg_row[2 * j + 1] = static_cast<int32_t>(p2.y);
      }
    }
  }
}

// One scale as two BF16 pieces: s = h + m up to 2^-16 relative.
__device__ __forceinline__ uint32_t scale_pieces(float s) {
  const __nv_bfloat16 h = __float2bfloat16_rn(s);
  const __nv_bfloat16 m = __float2bfloat16_rn(s - __bfloat162float(h));
  return static_cast<uint32_t>(__bfloat16_as_ushort(h)) | (static_cast<uint32_t>(__bfloat16_as_ushort(m)) << 16);
}

// Weight-side scale operands of one expert (run once per layer): wscale [G, N] FP32 -> per (128 channels, stage) one
// 4 KiB image [group of the stage][8-row group][8 rows][16 bytes]; the chunk of group parity v holds
// [w1, w2, w1, w2] in slots 4 v .. 4 v + 3 and zeros in the other group's slots.  `out` is zero-filled beforehand.
__global__ void sop_weight_kernel(const float* __restrict__ wscale, uint4* __restrict__ out, int G, int N) {
  const size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<size_t>(G) * N) return;
  const int g = static_cast<int>(i / N), n = static_cast<int>(i % N);
  const uint32_t w = scale_pieces(wscale[i]);
  const int stages = (G + 1) >> 1;
  const size_t image = static_cast<size_t>(n >> 7) * stages + (g >> 1);
  out[image * 256 + (g & 1) * 128 + ((n & 127) >> 3) * 8 + (n & 7)] = (g & 1) ? make_uint4(0u, 0u, w, w) : make_uint4(w, w, 0u, 0u);
}

// Test hook of the tap instantiation: one issuing warp comes late to every tile.
__device__ __forceinline__ void late_start(const GemmParams& p, int warp) {
  if (warp != p.dbg_late_warp) return;
  const uint64_t t0 = global_timer_ns();
  while (global_timer_ns() - t0 < p.dbg_late_ns) __nanosleep(200);
}

template <bool DEBUG, bool SPLIT>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_w4a4_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmL2,
                 const __grid_constant__ CUtensorMap tmSopA, const __grid_constant__ CUtensorMap tmSopB,
                 const __grid_constant__ CUtensorMap tmY, const GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  // Above every operand tile so that the descriptors' chunk distances are positive.
  const uint32_t zero_base = smem_base + kGemmStages * kStageBytes;   // second K chunk of every scale MMA
  const uint32_t out_base = zero_base + kZeroTile;                    // the epilogue warps' output tiles (512-byte aligned: 64-byte swizzle)
  const uint32_t bar_base = out_base + kEpiWarps * kOutTile;
  const uint32_t bar_op_full = bar_base;   // 16-byte aligned; so is bar_tmem_full, behind an even number of barriers
  const uint32_t bar_op_empty = bar_op_full + 8 * kGemmStages;
  const uint32_t bar_tmem_full = bar_op_empty + 8 * kGemmStages;
  const uint32_t bar_tmem_empty = bar_tmem_full + 8 * kTmemSlots;
  const uint32_t misc_off = (bar_tmem_empty + 8 * kTmemSlots) - smem_base;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + misc_off);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + misc_off + 4);

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;  // provably warp-uniform
  const int G = p.K >> 6;
  const int n_int_stages = (G + 1) >> 1;
  const int n_lr_stages = p.r > 0 && (!SPLIT || cluster_ctarank() == 0) ? (2 * p.r + 63) / 64 : 0;
  const int num_tiles = p.tiles_m * p.tiles_n;
  // This CTA's tiles and operand stages (all of them unless K is split).
  const int split = SPLIT ? static_cast<int>(cluster_ctarank()) : 0;
  const int first_tile = SPLIT ? blockIdx.x / p.splits : blockIdx.x, tile_step = SPLIT ? num_tiles : gridDim.x;
  const int st_begin = SPLIT ? n_int_stages * split / p.splits : 0;
  const int st_end = SPLIT ? n_int_stages * (split + 1) / p.splits : n_int_stages;
  const int g_begin = SPLIT ? 2 * st_begin : 0, g_end = SPLIT ? min(G, 2 * st_end) : G;
  const WaitEnv env{p.err, s_abort, p.wait_limit_ns};

  if (threadIdx.x == 0) {
    for (int i = 0; i < kGemmStages; ++i) {
      mbar_init(bar_op_full + 8 * i, 1);
      mbar_init(bar_op_empty + 8 * i, 3);    // the code-MMA warps and the scale-MMA warp
    }
    for (int i = 0; i < kTmemSlots; ++i) {
      mbar_init(bar_tmem_full + 8 * i, 2);   // a code-MMA warp and the scale-MMA warp
      mbar_init(bar_tmem_empty + 8 * i, kEpiWarps);
    }
    mbar_fence_init();
    fence_proxy_async_smem();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    tma_prefetch_desc(&tmSopA);
    tma_prefetch_desc(&tmSopB);
    if (!SPLIT && p.yref == nullptr) tma_prefetch_desc(&tmY);
    if (p.r > 0) {
      tma_prefetch_desc(&tmT);
      tma_prefetch_desc(&tmL2);
    }
  }
  for (uint32_t i = threadIdx.x; i < kZeroTile / 16; i += blockDim.x)
    reinterpret_cast<uint4*>(smem + (zero_base - smem_base))[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();   // the tensor core reads the tile through the async proxy
  if (warp == 2) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
    tc_fence_before_sync();
  }
  // Everything above overlaps the end of the kernel before this one; its results are needed from here on.
  grid_dependency_wait();
  if (threadIdx.x == 0) *s_abort = (*reinterpret_cast<volatile int*>(p.err) != 0) ? 1 : 0;
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const bool live = __all_sync(0xffffffffu, *s_abort == 0);

  // Shared-memory stage: A codes | B codes | token scale operand (two groups) | channel scale operand (two groups).
  // Per tile the scale-MMA warp and the epilogue walk the same list of TMEM slot uses: [the low-rank entry, if r > 0]
  // followed by one entry per group.  The code-MMA warps take the list's uses of one slot each.
  if (warp < kEpiWarp0) {
    setmaxnreg_dec<kControlRegs>();
    if (live && warp == 0) {
      // ------------------------------------------------------------------ TMA producer (all lanes loop, one issues)
      const bool issuer = elect_one_lane();
      Ring<kGemmStages> op;
      bool ok = true;
      int stage_no = 0;
      for (int tile = first_tile; ok && tile < num_tiles; tile += tile_step) {
        int tm, tn;
        tile_coords(tile, p.order, tm, tn);
        const int m0 = tm * kBM, n0 = tn * kBN;
        for (int st = 0; st < n_lr_stages + st_end - st_begin; ++st) {
          ok = __all_sync(0xffffffffu, bounded_wait<64>(bar_op_empty + 8 * op.slot, op.parity ^ 1u, env, kErrProducerWait));
          if (!ok) break;
          if (DEBUG) {
            // Test hook: one stage is never loaded (of a cluster that shares K: by its first CTA), so its consumers' waits
            // run into their limit and every role of the CTA leaves through the common tail (error word, drain, TMEM release).
            if (stage_no++ == p.dbg_stall_stage && split == 0) {
              op.advance();
              continue;
            }
          }
          const uint32_t full = bar_op_full + 8 * op.slot;
          const uint32_t dst = smem_base + op.slot * kStageBytes;
          if (st < n_lr_stages) {
            if (issuer) {
              mbar_arrive_expect_tx(full, kLrStageBytes);
              tma_load_2d(dst, &tmT, full, st * 64, m0);
              tma_load_2d(dst + kOpATile, &tmL2, full, st * 64, n0);
            }
          } else if (issuer) {
            const int ks = st - n_lr_stages + st_begin;
            const uint32_t sop = dst + kOpATile + kOpBTile;
            mbar_arrive_expect_tx(full, kStageBytes);
            tma_load_2d(dst, &tmA, full, ks * kBK, m0);
            tma_load_2d(dst + kOpATile, &tmB, full, ks * kBK, n0);
            // scale operand images as rows of 32-bit words, 256 words (1 KiB) per box
            tma_load_2d(sop, &tmSopA, full, ks * 512, tm);
            tma_load_2d(sop + 1024, &tmSopA, full, ks * 512 + 256, tm);
#pragma unroll
            for (int c = 0; c < 4; ++c) tma_load_2d(sop + kSopATile + 1024 * c, &tmSopB, full, ks * 1024 + 256 * c, tn);
          }
          op.advance();
        }
      }
    } else if (live && (warp == 1 || warp == 2)) {
      // ------------------------------------------------------------------ code-MMA issuer (all lanes loop, one issues)
      constexpr uint32_t idesc_f8 = umma_idesc(1, 0, kBM, kBN);
      constexpr uint32_t idesc_bf16 = umma_idesc(1, 1, kBM, kBN);
      const bool issuer = elect_one_lane();
      const uint32_t go = issuer ? 1u : 0u;
      const int issue_lane = __ffs(__ballot_sync(0xffffffffu, issuer)) - 1;   // the decision below is the issuing lane's
      CodeSlotWalk walk(warp - 1);
      const uint32_t d = tmem_base + walk.own * 2 * kBN, full_bar = bar_tmem_full + 8 * walk.own, empty_bar = bar_tmem_empty + 8 * walk.own;
      Ring<kGemmStages> op;
      bool ok = true;
      for (int tile = first_tile; ok && tile < num_tiles; tile += tile_step) {
        if (DEBUG) late_start(p, warp);
        if (n_lr_stages > 0) {
          const bool mine = walk.owns_next();
          if (mine) {
            ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(empty_bar, walk.free_parity(), env, kErrMmaWait));
            if (!ok) break;
            tc_fence_after_sync();
          }
          for (int l = 0; ok && l < n_lr_stages; ++l) {
            ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(bar_op_full + 8 * op.slot, op.parity, env, kErrMmaWait));
            if (!ok) break;
            const uint32_t a = smem_base + op.slot * kStageBytes, b = a + kOpATile;
            if (issuer && mine) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                umma_f16(d, umma_desc_k_sw128(a, 32 * kk), umma_desc_k_sw128(b, 32 * kk), idesc_bf16, (l > 0 || kk > 0) ? 1u : 0u);
              umma_commit(bar_op_empty + 8 * op.slot);
            } else if (issuer) {
              mbar_arrive(bar_op_empty + 8 * op.slot);
            }
            op.advance();
          }
          if (!ok) break;
          if (mine) {
            if (issuer) umma_commit(full_bar);
            walk.issued();
          }
          walk.pass(1);
        }
        const int v = walk.group();   // the same one in all of the tile's stages
        for (int st = st_begin; ok && st < st_end; ++st) {
          ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(bar_op_full + 8 * op.slot, op.parity, env, kErrMmaWait));
          if (!ok) break;
          const uint32_t a = smem_base + op.slot * kStageBytes, b = a + kOpATile;
          const int groups = (2 * st + 1 < G) ? 2 : 1;
          if (v < groups) {
            // everything the issue needs is ready before the wait that sits on the slot's round trip
            const uint64_t da0 = umma_desc_k_sw128(a, 64 * v), db0 = umma_desc_k_sw128(b, 64 * v);
            const uint64_t da1 = umma_desc_k_sw128(a, 64 * v + 32), db1 = umma_desc_k_sw128(b, 64 * v + 32);
            if (__shfl_sync(0xffffffffu, wait_issue_f8x2(go, empty_bar, walk.free_parity(), d, da0, db0, da1, db1, idesc_f8, full_bar), issue_lane) == 0) {
              ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(empty_bar, walk.free_parity(), env, kErrMmaWait));
              if (!ok) break;
              tc_fence_after_sync();
              umma_f8_if(go, d, da0, db0, idesc_f8, 0u);
              umma_f8_if(go, d, da1, db1, idesc_f8, 1u);
              umma_commit_if(go, full_bar);
            }
            walk.issued();
          }
          umma_commit_if(go, bar_op_empty + 8 * op.slot);
          op.advance();
        }
        walk.pass(g_end - g_begin);
      }
    } else if (live && warp == 3) {
      // ------------------------------------------------------------------ scale-MMA issuer
      // Walks the slot uses of both code-MMA warps.
      constexpr uint32_t idesc_bf16 = umma_idesc(1, 1, kBM, kBN);
      const bool issuer = elect_one_lane();
      const uint32_t go = issuer ? 1u : 0u;
      const int issue_lane = __ffs(__ballot_sync(0xffffffffu, issuer)) - 1;   // the decision below is the issuing lane's
      Ring<kGemmStages> op;
      Ring<kTmemSlots> tm;
      bool ok = true;
      for (int tile = first_tile; ok && tile < num_tiles; tile += tile_step) {
        if (DEBUG) late_start(p, warp);
        if (n_lr_stages > 0) {
          ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(bar_tmem_empty + 8 * tm.slot, tm.parity ^ 1u, env, kErrMmaWait));
          if (!ok) break;
          tc_fence_after_sync();
          if (issuer) mbar_arrive(bar_tmem_full + 8 * tm.slot);   // the entry has no scale products, nor its stages anything for this warp
          tm.advance();
          for (int l = 0; ok && l < n_lr_stages; ++l) {
            ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(bar_op_full + 8 * op.slot, op.parity, env, kErrMmaWait));
            if (!ok) break;
            if (issuer) mbar_arrive(bar_op_empty + 8 * op.slot);
            op.advance();
          }
          if (!ok) break;
        }
        for (int st = st_begin; ok && st < st_end; ++st) {
          ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(bar_op_full + 8 * op.slot, op.parity, env, kErrMmaWait));
          if (!ok) break;
          const uint32_t sa = smem_base + op.slot * kStageBytes + kOpATile + kOpBTile, sb = sa + kSopATile;
          const int groups = (2 * st + 1 < G) ? 2 : 1;
          for (int v = 0; v < groups; ++v) {
            const uint32_t d = tmem_base + tm.slot * 2 * kBN + kBN;
            const uint32_t full_bar = bar_tmem_full + 8 * tm.slot;
            const uint32_t cb = sb + (kSopBTile / 2) * v;   // the channel side's chunk of this group
            const uint64_t dsa = umma_desc_k_plain(sa, zero_base - sa, 128), dsb = umma_desc_k_plain(cb, zero_base - cb, 128);
            if (__shfl_sync(0xffffffffu, wait_issue_f16(go, bar_tmem_empty + 8 * tm.slot, tm.parity ^ 1u, d, dsa, dsb, idesc_bf16, full_bar), issue_lane) == 0) {
              ok = __all_sync(0xffffffffu, bounded_wait<0, 1>(bar_tmem_empty + 8 * tm.slot, tm.parity ^ 1u, env, kErrMmaWait));
              if (!ok) break;
              tc_fence_after_sync();
              umma_f16_if(go, d, dsa, dsb, idesc_bf16, 0u);
              umma_commit_if(go, full_bar);
            }
            tm.advance();
          }
          if (!ok) break;
          umma_commit_if(go, bar_op_empty + 8 * op.slot);
          op.advance();
        }
      }
    }
  } else {
    setmaxnreg_inc<kEpilogueRegs>();
    if (live) {
      // ------------------------------------------------------------------ epilogue warps
      // Warp ew owns TMEM lanes 32 * (ew % 4) .. +31 (token rows) and the 32-column block ew / 4; a thread owns one
      // row and the block's 32 output channels.
      const int ew = warp - kEpiWarp0;
      const int quarter = ew & 3, colblk = ew >> 2;
      const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(32 * quarter) << 16) + kEpiCols * colblk;
      const uint32_t out_tile = out_base + kOutTile * ew;
      SlotUse use(t_lane, bar_tmem_full);
      bool ok = true;
      for (int tile = first_tile; ok && tile < num_tiles; tile += tile_step) {
        int tm_e, tn_e;
        tile_coords(tile, p.order, tm_e, tn_e);
        const int m0 = tm_e * kBM, n0 = tn_e * kBN;
        const bool dbg_tile = DEBUG && p.dbg_P != nullptr && m0 == p.dbg_m0 && n0 == p.dbg_n0;
        // Lane l holds the bias of the block's channel l; it reaches the other lanes through shared memory at the end.
        const float bias_lane = p.bias ? __ldg(p.bias + n0 + kEpiCols * colblk + lane) : 0.0f;
        float2 acc[16];  // pair k: channels ch0 + 2 k, ch0 + 2 k + 1
        if (n_lr_stages > 0) {   // the low-rank entry opens the tile: the accumulators start as T L2
          const uint32_t t = use.t;
          uint32_t pv[16], qv[16];
          ok = __all_sync(0xffffffffu, bounded_wait(use.full, use.phase, env, kErrEpilogueWait));
          if (!ok) break;
          tc_fence_after_sync();
          tmem_ld_32x32b_x16(t, pv);
          tmem_ld_32x32b_x16(t + 16, qv);
          tmem_wait_ld();
          tie_fragment(pv);
          tie_fragment(qv);
          tc_fence_before_sync();
          mbar_arrive_if(lane == 0 ? 1u : 0u, use.empty());
          use.next();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            acc[j] = make_float2(__uint_as_float(pv[2 * j]), __uint_as_float(pv[2 * j + 1]));
            acc[8 + j] = make_float2(__uint_as_float(qv[2 * j]), __uint_as_float(qv[2 * j + 1]));
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[j] = make_float2(0.0f, 0.0f);
        }
        for (int g = g_begin; g < g_end; ++g) {
          const uint32_t t = use.t;
          uint32_t pv[16], sv[16];
          if (wait_then_ld16(use.full, use.phase, t, pv) == 0) {
            ok = __all_sync(0xffffffffu, bounded_wait(use.full, use.phase, env, kErrEpilogueWait));
            if (!ok) break;
            tc_fence_after_sync();
            tmem_ld_32x32b_x16(t, pv);
          }
          int32_t* d0 = nullptr;
          if (DEBUG) {
            if (dbg_tile) d0 = p.dbg_P + (static_cast<size_t>(32 * quarter + lane) * G + g) * kBN + kEpiCols * colblk;
          }
          tmem_ld_32x32b_x16(t + kBN, sv);
          tmem_wait_ld();
          tie_fragment(pv);
          tie_fragment(sv);
          fma_fragment<DEBUG>(pv, sv, acc, d0);
          tmem_ld_32x32b_x16(t + 16, pv);
          tmem_ld_32x32b_x16(t + kBN + 16, sv);
          tmem_wait_ld();
          tie_fragment(pv);
          tie_fragment(sv);
          // The whole slot is in registers (loads and waits are warp-wide): hand it back to the MMA warps.
          tc_fence_before_sync();
          mbar_arrive_if(lane == 0 ? 1u : 0u, use.empty());
          use.next();
          fma_fragment<DEBUG>(pv, sv, acc + 8, DEBUG && d0 ? d0 + 16 : nullptr);
        }
        if (!ok) break;
        if constexpr (SPLIT) {
          // Partial tile: 512-byte rows of FP32, 16-byte chunk c at c ^ (row % 8): conflict free for both sides.
          const int row = 32 * quarter + lane;
#pragma unroll
          for (int c = 0; c < 8; ++c)
            sts_u32x4(smem_base + 512 * row + 16 * ((8 * colblk + c) ^ (row & 7)),
                      make_uint4(__float_as_uint(acc[2 * c].x), __float_as_uint(acc[2 * c].y), __float_as_uint(acc[2 * c + 1].x),
                                 __float_as_uint(acc[2 * c + 1].y)));
          break;
        }
        // The tile's end: bias, activation, BF16, then a swizzled tile in shared memory: the source of the TMA store to Y, and where the
        // clip search reads outputs beside the reference so that a warp's 16-byte reads of that cover eight rows x 64 bytes.
        if (!SPLIT && lane == 0) bulk_store_wait_read();   // the previous tile has left the staging tile
        __syncwarp();
        sts_f32(out_tile + 4 * lane, bias_lane);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kEpiCols / 4; ++i) {
          const float4 b = lds_f32x4(out_tile + 16 * i);
          acc[2 * i].x += b.x, acc[2 * i].y += b.y, acc[2 * i + 1].x += b.z, acc[2 * i + 1].y += b.w;
        }
        if (p.act != 0) {  // uniform over the grid
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[j] = make_float2(apply_activation(acc[j].x, p.act), apply_activation(acc[j].y, p.act));
        }
        __syncwarp();
        // Output tile: 64-byte rows, 16-byte chunk c at c ^ (row / 2 % 4): conflict free for both sides.
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint4 o;
          o.x = bf16x2_bits(acc[4 * c]), o.y = bf16x2_bits(acc[4 * c + 1]), o.z = bf16x2_bits(acc[4 * c + 2]), o.w = bf16x2_bits(acc[4 * c + 3]);
          sts_u32x4(out_tile + 64 * lane + 16 * (c ^ ((lane >> 1) & 3)), o);
        }
        __syncwarp();
        if (p.yref == nullptr) {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0 && m0 + 32 * quarter < p.M) {
            tma_store_2d(&tmY, out_tile, n0 + kEpiCols * colblk, m0 + 32 * quarter);
            bulk_store_commit();
          }
        } else {
          // Eq. 10's objective: || Y_ref - Y_hat ||^2 over the tile, with Y_hat rounded to BF16 exactly as the
          // forward would store it.  FP32 within the thread and the warp, FP64 across warps and tiles.
          __syncwarp();
          const int row = m0 + 32 * quarter + (lane >> 2);   // and rows + 8, + 16, + 24
          const size_t step = 8 * static_cast<size_t>(p.N);
          const uint16_t* rp = p.yref + static_cast<size_t>(row) * p.N + n0 + kEpiCols * colblk + 8 * (lane & 3);
          float sq = 0.0f;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (row + 8 * j < p.M) {
              const uint4 y = lds_u32x4(out_tile + 512 * j + 64 * (lane >> 2) + 16 * ((lane ^ (lane >> 3)) & 3));
              const uint4 ref = __ldg(reinterpret_cast<const uint4*>(rp + j * step));
              sq = sq_diff_bf16x2(ref.x, y.x, sq);
              sq = sq_diff_bf16x2(ref.y, y.y, sq);
              sq = sq_diff_bf16x2(ref.z, y.z, sq);
              sq = sq_diff_bf16x2(ref.w, y.w, sq);
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
          if (lane == 0) atomicAdd(p.sq_err, static_cast<double>(sq));
        }
      }
      tmem_wait_ld();   // a role that gave up may still have loads in flight
      if (!SPLIT && lane == 0) bulk_store_wait_read();   // stores still read the staging tile
    }
  }

  if constexpr (SPLIT) {
    cluster_sync_all();   // all partial tiles are written
    if (live && warp >= kEpiWarp0 && !cluster_gave_up(s_abort, p.splits)) {
      int tm_e, tn_e;
      tile_coords(first_tile, p.order, tm_e, tn_e);
      float sq = 0.0f;
      // A warp takes one row at a time, a lane four channels.
      for (int row = 16 * split + warp - kEpiWarp0; row < kBM; row += 16 * p.splits) {
        if (tm_e * kBM + row >= p.M) break;
        const uint32_t at = smem_base + 512 * row + 16 * (lane ^ (row & 7));
        // One remote load after the other: with all of them on their way first, as in the MXFP4 GEMM, this kernel's 96 registers
        // spill (100 x 5120 -> 5120 21.7 us and 28.0 so, 300 x 1024 -> 1024 14.3 and 23.1).
        float4 y = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        for (int i = 0; i < p.splits; ++i) {
          const float4 v = ld_cluster_f32x4(map_to_cta(at, i));
          y.x += v.x, y.y += v.y, y.z += v.z, y.w += v.w;
        }
        const int ch = tn_e * kBN + 4 * lane;
        const float4 b = p.bias ? __ldg(reinterpret_cast<const float4*>(p.bias + ch)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        y.x += b.x, y.y += b.y, y.z += b.z, y.w += b.w;
        if (p.act != 0)
          y = make_float4(apply_activation(y.x, p.act), apply_activation(y.y, p.act), apply_activation(y.z, p.act), apply_activation(y.w, p.act));
        const uint2 o = make_uint2(bf16x2_bits(make_float2(y.x, y.y)), bf16x2_bits(make_float2(y.z, y.w)));
        const size_t dst = static_cast<size_t>(tm_e * kBM + row) * p.N + ch;
        if (p.yref == nullptr) {
          *reinterpret_cast<uint2*>(p.Y + dst) = o;
        } else {
          const uint2 ref = __ldg(reinterpret_cast<const uint2*>(p.yref + dst));
          sq = sq_diff_bf16x2(ref.x, o.x, sq);
          sq = sq_diff_bf16x2(ref.y, o.y, sq);
        }
      }
      if (p.yref != nullptr) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0) atomicAdd(p.sq_err, static_cast<double>(sq));
      }
    }
    cluster_sync_all();   // nobody leaves while its shared memory is still being read
  }
  // ---------------------------------------------------------------------- common tail
  tc_fence_before_sync();
  __syncthreads();
  drain_after_abort(s_abort);
  if (warp == 2) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace w4a4
