// w4a4_gptq_quantize: GPTQ on the residual branch (Sec. III-B), entirely on the device in FP64.
//
// The published algorithm (Frantar et al., 2023, Algorithm 1 with the Cholesky reformulation of Sec. 4) quantizes
// the input channels of R [K, N] in order and spreads each channel's error, scaled by a row of
// U = chol(H^-1, upper), over the channels still to come, H = X_hat^T X_hat being the second-order statistic of the
// layer's calibration inputs.  Here:
//
//   1. H (upper triangle) = X_hat^T X_hat by a tiled FP64 GEMM; dead channels and damping on the diagonal.
//   2. H = V V^T with V UPPER triangular: a Cholesky factorization taken from the last channel to the first, blocked by 64.
//      U = V^-1 is the factor the algorithm asks for (H^-1 = V^-T V^-1), but neither H^-1 nor U is formed: with e_k the
//      algorithm's scaled errors and z = U^T e, i.e. V^T z = e, forward substitution gives the compensated weight of
//      channel j as
//          w_j = W_j - sum_{k<j} U_kj e_k = W_j + sum_{k<j} (V_kj / V_jj) z_k ,      z_k = W_k - q_k ,
//      the difference between the ORIGINAL weight and the value its code stands for (the form of the same procedure
//      published as LDLQ: Chee et al., "QuIP", 2023, Sec. 3).  So the sweep needs L = V with its columns divided by the
//      diagonal, and K^3 / 3 multiply-adds of a triangular inverse are not there.  A group's scale is taken from its weights
//      as compensated for the channels before the group only; with t_j = sum_{k before the group} L_kj z_k these are
//      W_g + L_gg^-T t_g, which needs the inverse of L's 64 x 64 diagonal blocks.
//   3. The sweep, 256 channels (a lazy batch) per launch, and one product for the channels after the batch.
//
// One stream, and nothing here waits on another block: every dependency is a kernel boundary.  (Large products beside the
// serial steps on a second stream gave nothing: sharing the FP64 pipe stretches the serial chains by as much as is hidden.)
#include "../../include/w4a4.h"

#include <cuda_runtime.h>

#include <cstdint>

namespace {

constexpr int kNb = 64;     // block of the factorization = quantization group
constexpr int kBand = 512;  // columns per band of the factorization
constexpr int kLazy = 256;  // input channels per lazy batch of the sweep

// ---------------------------------------------------------------------------------------------------------
// C = beta C + alpha A B in FP64, C row-major.  Each operand is stored with one of its two indices contiguous: k (AK,
// BK) or the output index (A(m, k) at A[k lda + m], B(k, n) at B[k ldb + n]).  M and N are multiples of 64, Kd of 16,
// leading dimensions and offsets multiples of two elements.
//
// BM x 64 tile per block, eight warps, each a (BM / 4) x 32 corner as 8 x 8 x 4 FP64 tensor-core steps; 16-deep slices in a
// ring of four, filled by 16-byte asynchronous copies three slices ahead, one barrier per slice.  The FP64 tensor path
// is the bound (37.0 TFLOP/s measured for every instruction shape): a slice of a 128 x 64 tile takes it ~2000 clocks and
// brings in 24 KiB, far below what shared memory and L2 deliver.
//
// With `upper_out`, blocks whose tile lies entirely below the diagonal (column index + diag_shift) return at once (only the
// upper triangle of C is wanted).
// ---------------------------------------------------------------------------------------------------------
constexpr int kBN = 64, kBK = 16, kGemmRing = 4;

struct GemmArgs {
  int M, N, Kd;
  const double* A;
  long lda;
  const double* B;
  long ldb;
  double* C;
  long ldc;
  double alpha, beta;   // +1 or -1; 0 or 1
  bool upper_out = false;
  int diag_shift = 0;
};

// 16-byte asynchronous copy global -> shared; with `valid` false nothing is read and zeros are written.
__device__ __forceinline__ void async_copy16(double* smem_dst, const double* gmem_src, bool valid) {
  const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  const int src_bytes = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(gmem_src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory"); }

// D (8 x 8) += A (8 x 4) B (4 x 8) on the FP64 tensor core; per lane one element of A and B, two of D.
__device__ __forceinline__ void dmma_8x8x4(double (&d)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
               : "+d"(d[0]), "+d"(d[1])
               : "d"(a), "d"(b));
}

// Place of element (k, x) in a slice of X output indices.  A fragment load of a half warp touches four k and four x:
// the swap of groups of four (by k where x is contiguous, by x where k is) spreads them over all banks and keeps the pairs
// of a 16-byte copy together.
template <int X, bool KFAST>
__device__ __forceinline__ int slice_at(int k, int x) {
  return KFAST ? x * kBK + ((((k >> 2) ^ (x & 3)) << 2) | (k & 3)) : k * X + (x ^ ((k & 3) << 2));
}

// One operand's share of a slice: X * 16 elements by 256 threads, two per copy.  `src` points at this thread's first pair
// of the slice.
template <int X, bool KFAST>
__device__ __forceinline__ void fetch_operand(double* dst, const double* src, long ld, int x_valid) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int i = 0; i < X / 32; ++i) {
    if (KFAST) {
      const int x = (tid >> 3) + 32 * i, k = 2 * (tid & 7);
      async_copy16(dst + slice_at<X, true>(k, x), src + 32 * i * ld, x < x_valid);
    } else {
      constexpr int kPerPass = 512 / X;   // k rows covered by one pass of the 256 threads
      const int x = 2 * (tid % (X / 2)), k = tid / (X / 2) + kPerPass * i;
      async_copy16(dst + slice_at<X, false>(k, x), src + static_cast<long>(kPerPass * i) * ld, x < x_valid);
    }
  }
}
template <int X, bool KFAST>
__device__ __forceinline__ const double* operand_start(const double* p, long ld, int x0, int k0) {
  const int tid = threadIdx.x;
  return KFAST ? p + static_cast<long>(x0 + (tid >> 3)) * ld + k0 + 2 * (tid & 7)
               : p + static_cast<long>(k0 + tid / (X / 2)) * ld + x0 + 2 * (tid % (X / 2));
}

constexpr size_t dgemm_smem_bytes(int BM) { return static_cast<size_t>(kGemmRing) * (BM + kBN) * kBK * sizeof(double); }

template <int BM, bool AK, bool BK>
__global__ void __launch_bounds__(256, 2) dgemm_kernel(const GemmArgs g) {
  constexpr int MT = BM / 32;  // 8 x 8 tensor-core tiles per warp along M (four along N)
  extern __shared__ __align__(16) double slices[];
  double* const As = slices;
  double* const Bs = slices + kGemmRing * BM * kBK;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * kBN;
  if (g.upper_out && m0 >= n0 + g.diag_shift + kBN) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = (warp & 3) * (8 * MT), wn = (warp >> 2) * 32;  // the warp's corner inside the block's tile
  const int fr = lane >> 2, fk = lane & 3;                      // fragment row (or column) and k index of this lane
  const int n_slices = g.Kd / kBK;
  const double* a_src = operand_start<BM, AK>(g.A, g.lda, m0, 0);
  const double* b_src = operand_start<kBN, BK>(g.B, g.ldb, n0, 0);
  const long a_step = AK ? kBK : kBK * g.lda, b_step = BK ? kBK : kBK * g.ldb;
  const int m_valid = g.M - m0;
  auto fetch_slice = [&](int slice) {
    const int buf = slice % kGemmRing;
    fetch_operand<BM, AK>(As + buf * (BM * kBK), a_src + slice * a_step, g.lda, m_valid);
    fetch_operand<kBN, BK>(Bs + buf * (kBN * kBK), b_src + slice * b_step, g.ldb, kBN);
  };
#pragma unroll
  for (int i = 0; i < kGemmRing - 1; ++i) {
    if (i < n_slices) fetch_slice(i);
    async_commit();
  }
  // Accumulator layout: rows fr, columns 2 fk and 2 fk + 1 of each 8 x 8 tile.  C = alpha (A B + (beta / alpha) C), alpha =
  // +-1: the accumulators start from C, whose loads run under the first slices' copies.
  const bool rows_valid = m0 + wm < g.M;   // M is a multiple of 64: a warp's rows lie on one side of it
  double* const C = g.C + static_cast<long>(m0 + wm + fr) * g.ldc + n0 + wn + 2 * fk;
  const bool pairs = (reinterpret_cast<uintptr_t>(g.C) & 15) == 0;   // a caller's statistic may be 8-byte aligned only
  double acc[MT][4][2];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double* c = C + static_cast<long>(8 * i) * g.ldc + 8 * j;
      double2 v = make_double2(0.0, 0.0);
      if (g.beta != 0.0 && rows_valid) v = pairs ? *reinterpret_cast<const double2*>(c) : make_double2(c[0], c[1]);
      acc[i][j][0] = g.alpha * v.x;   // beta is 0 or 1, alpha is its own inverse
      acc[i][j][1] = g.alpha * v.y;
    }
  for (int s = 0; s < n_slices; ++s) {
    async_wait<kGemmRing - 2>();
    __syncthreads();   // slice s is complete, and everyone is done with the slice whose place the next one takes
    if (s + kGemmRing - 1 < n_slices) fetch_slice(s + kGemmRing - 1);
    async_commit();
    const double* as = As + (s % kGemmRing) * (BM * kBK);
    const double* bs = Bs + (s % kGemmRing) * (kBN * kBK);
#pragma unroll
    for (int k = 0; k < kBK; k += 4) {
      // FP64 tensor-core step (8 x 8 x 4): this lane holds A[row fr][k fk] and B[k fk][column fr] of each tile
      double a[MT], b[4];
#pragma unroll
      for (int i = 0; i < MT; ++i) a[i] = as[slice_at<BM, AK>(k + fk, wm + 8 * i + fr)];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = bs[slice_at<kBN, BK>(k + fk, wn + 8 * j + fr)];
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) dmma_8x8x4(acc[i][j], a[i], b[j]);
    }
  }
  if (!rows_valid) return;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      double* c = C + static_cast<long>(8 * i) * g.ldc + 8 * j;
      const double c0 = g.alpha * acc[i][j][0], c1 = g.alpha * acc[i][j][1];
      if (pairs) {
        *reinterpret_cast<double2*>(c) = make_double2(c0, c1);
      } else {
        c[0] = c0;
        c[1] = c1;
      }
    }
}

// BF16 -> FP64, two values per thread; values from `n` on (the rows that pad a batch of tokens to a whole slice) are zeros.
__global__ void bf16_to_f64_kernel(const uint16_t* __restrict__ in, double2* __restrict__ out, long n, long n_padded) {
  const long i = 2 * ((long)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n_padded) return;
  const uint32_t lo = i < n ? in[i] : 0u, hi = i + 1 < n ? in[i + 1] : 0u;
  out[i >> 1] = make_double2((double)__uint_as_float(lo << 16), (double)__uint_as_float(hi << 16));
}

// Dead input channels (H_kk = 0) count as H_kk = 1; percdamp times the mean of the diagonal after that fix goes to *damp.
// One block; the sum runs in a fixed order (thread-strided partial sums, then a tree), so it is deterministic.
__global__ void gptq_diag_kernel(const double* __restrict__ H, int K, double percdamp, unsigned char* __restrict__ dead,
                                 double* __restrict__ damp) {
  __shared__ double part[1024];
  double s = 0.0;
  for (int k = threadIdx.x; k < K; k += 1024) {
    const double d = H[(long)k * K + k];
    dead[k] = d == 0.0 ? 1 : 0;
    s += d == 0.0 ? 1.0 : d;
  }
  part[threadIdx.x] = s;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *damp = percdamp * (part[0] / (double)K);
}

// ---------------------------------------------------------------------------------------------------------
// H = V V^T, V upper triangular, from the last block to the first (A holds H's upper triangle and ends as V).
// ---------------------------------------------------------------------------------------------------------

// One 64-column step: the diagonal block at j0, whose trailing updates are already applied, is factored, and the 64-row
// strip of the panel above it that belongs to this block of threads becomes the solution of x D^T = row (D the factored
// block), both in one elimination from the last column to the first: the strip's rows take the same column operations as
// the diagonal block's.  Every block factors the diagonal block for itself: that adds nothing to the chain of steps, which
// is what this kernel is bound by.  The strips of V stay in A for the factorization's own products; L gets block and strips
// with every column divided by its diagonal element, which is what the sweep reads.  The diagonal (dead channels, damping)
// is completed on the way in.  Entries below the diagonal are never used for a result (H_in's lower triangle is not
// defined).
// Eight columns at a time: each of 128 threads factors the 8 x 8 corner for itself in registers (a chain of eight reciprocal
// square roots) and solves its own row against it; then the columns still to come take the eight as 8 x 8 x 4 FP64
// tensor-core steps, warp w on the row tiles w of block and strip.  Two barriers per eight columns, and a loop body small
// enough for the instruction cache: column by column, 64 steps unrolled took 24 us per launch, rolled with predicates 55,
// in shared memory 39 + 16 in two kernels; this 18.6 (K = 5120).
constexpr int kCholThreads = 256, kCholSub = 8;
constexpr int kCholPitch = kNb + 2, kCholFPitch = 12;
constexpr size_t kCholSmemBytes = 2 * kNb * (kCholPitch + kCholFPitch) * sizeof(double);
__global__ void __launch_bounds__(kCholThreads) chol_step_kernel(double* __restrict__ A, double* __restrict__ L, long ld,
                                                                 int j0, const unsigned char* __restrict__ dead,
                                                                 const double* __restrict__ damp, int* not_pd) {
  extern __shared__ __align__(16) double chol_smem[];
  double(*S)[kCholPitch] = reinterpret_cast<double(*)[kCholPitch]>(chol_smem);   // rows 0..63 diagonal block, 64..127 strip
  double(*F)[kCholFPitch] = reinterpret_cast<double(*)[kCholFPitch]>(chol_smem + 2 * kNb * kCholPitch);   // eight finished columns
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int fr = lane >> 2, fk = lane & 3;
  const long strip0 = (long)blockIdx.x * kNb;
  const bool has_strip = strip0 < j0;                       // the one block of the last step (j0 = 0) has none
  for (int i = t >> 5; i < kNb; i += kCholThreads / 32) {
    async_copy16(&S[i][2 * lane], A + (long)(j0 + i) * ld + j0 + 2 * lane, true);
    async_copy16(&S[kNb + i][2 * lane], has_strip ? A + (strip0 + i) * ld + j0 + 2 * lane : A, has_strip);
  }
  async_commit();
  const double on_diagonal = t < kNb ? *damp + (dead[j0 + t] ? 1.0 : 0.0) : 0.0;
  async_wait<0>();
  __syncthreads();
  if (t < kNb) S[t][t] += on_diagonal;
  __syncthreads();
#pragma unroll 1
  for (int kb = kNb / kCholSub - 1; kb >= 0; --kb) {
    const int c0 = kCholSub * kb;
    if (t < 2 * kNb) {
      double a[kCholSub][kCholSub], inv[kCholSub];   // upper triangle of the corner
#pragma unroll
      for (int i = 0; i < kCholSub; ++i)
#pragma unroll
        for (int j = i & ~1; j < kCholSub; j += 2) {
          const double2 v = *reinterpret_cast<const double2*>(&S[c0 + i][c0 + j]);
          a[i][j] = v.x;   // (an entry below the diagonal in the first pair of an odd row: not used)
          a[i][j + 1] = v.y;
        }
#pragma unroll
      for (int j = kCholSub - 1; j >= 0; --j) {
        if (t == 0 && !(a[j][j] > 0.0)) *not_pd = 1;
        inv[j] = rsqrt(a[j][j]);
#pragma unroll
        for (int i = 0; i < j; ++i) a[i][j] *= inv[j];
#pragma unroll
        for (int i = 0; i < j; ++i)
#pragma unroll
          for (int m = i; m < j; ++m) a[i][m] = fma(-a[i][j], a[m][j], a[i][m]);
      }
      double x[kCholSub];
#pragma unroll
      for (int j = 0; j < kCholSub; j += 2) {
        const double2 v = *reinterpret_cast<const double2*>(&S[t][c0 + j]);
        x[j] = v.x;
        x[j + 1] = v.y;
      }
#pragma unroll
      for (int j = kCholSub - 1; j >= 0; --j) {
        x[j] *= inv[j];
#pragma unroll
        for (int m = 0; m < j; ++m) x[m] = fma(-x[j], a[m][j], x[m]);
      }
#pragma unroll
      for (int j = 0; j < kCholSub; j += 2) {
        const double2 v = make_double2(x[j], x[j + 1]);
        *reinterpret_cast<double2*>(&F[t][j]) = v;
        const double2 l = make_double2(x[j] * inv[j], x[j + 1] * inv[j + 1]);
        if (t < kNb ? blockIdx.x == 0 : has_strip)
          *reinterpret_cast<double2*>(L + (t < kNb ? j0 + t : strip0 + t - kNb) * ld + j0 + c0 + j) = l;
      }
    }
    __syncthreads();
    if (t < 2 * kNb) {   // after the barrier: the rows of the corner were still being read
#pragma unroll
      for (int j = 0; j < kCholSub; j += 2)
        *reinterpret_cast<double2*>(&S[t][c0 + j]) = *reinterpret_cast<const double2*>(&F[t][j]);
    }
#pragma unroll
    for (int part = 0; part < 2; ++part) {   // strip, diagonal block (its tiles on and above the diagonal)
      const int row = 8 * warp + (part == 0 ? kNb : 0) + fr;
      double f[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) f[h] = -F[row][4 * h + fk];
#pragma unroll 1
      for (int ct = part == 0 ? 0 : warp; ct < kb; ++ct) {
        double2* at = reinterpret_cast<double2*>(&S[row][8 * ct + 2 * fk]);
        double c[2] = {at->x, at->y};
#pragma unroll
        for (int h = 0; h < 2; ++h) dmma_8x8x4(c, f[h], F[8 * ct + fr][4 * h + fk]);
        *at = make_double2(c[0], c[1]);
      }
    }
    __syncthreads();
  }
  if (has_strip)
    for (int i = t >> 5; i < kNb; i += kCholThreads / 32)
      *reinterpret_cast<double2*>(A + (strip0 + i) * ld + j0 + 2 * lane) = *reinterpret_cast<const double2*>(&S[kNb + i][2 * lane]);
}

// Inverses of L's 64 x 64 diagonal blocks (unit upper triangular; nothing but the entries above the diagonal is read), one
// block of threads each: G [K / 64][64][64].  Thread c solves L x = e_c.
__global__ void __launch_bounds__(kNb) unit_inverse_kernel(const double* __restrict__ L, double* __restrict__ G, long ld) {
  __shared__ double D[kNb][kNb + 1];
  const int t = threadIdx.x, i0 = blockIdx.x * kNb;
  for (int r = 0; r < kNb; ++r) D[r][t] = L[(long)(i0 + r) * ld + i0 + t];
  __syncthreads();
  double b[kNb];
#pragma unroll
  for (int r = 0; r < kNb; ++r) b[r] = (r == t) ? 1.0 : 0.0;
#pragma unroll
  for (int k = kNb - 1; k >= 0; --k)
#pragma unroll
    for (int r = 0; r < k; ++r) b[r] = fma(-D[r][k], b[k], b[r]);
#pragma unroll
  for (int r = 0; r < kNb; ++r) G[(long)(i0 + r) * kNb + t] = b[r];
}

// ---------------------------------------------------------------------------------------------------------
// The sweep over one lazy batch of up to 256 input channels starting at b0 (Algorithm 1's inner loops), for 32 output
// channels per block; output channels are independent of one another.
// scale = FP32(max |w| / 7) over a group of 64 input channels as it stands when the sweep enters it; per channel code =
// clamp(round-half-even(w / scale), -8, 7) (0 for an all-zero group), z = original weight - code * scale, later channels +=
// z * L_kj with L = V with its columns divided by the diagonal.  Z [256, ldw] keeps the z for the update of the channels after
// the batch; T holds what the batches before have added to this one's channels (nothing in the first batch).
// MX: the same on the MXFP4 grid of the MX variant (OCP MX v1.0): one E8M0 exponent per 32 input channels,
// floor(log2 max|w|) - 2 over the block as it stands when the sweep enters it, and E2M1 elements {0, 0.5, 1, 1.5, 2,
// 3, 4, 6} * 2^e, nearest with ties to the even code, saturating at 6, sign bit from the compensated weight.
//
// What has been added to the batch's weights stays in shared memory (64 KiB of FP64), and the channels are taken eight channels at a time.  Warp 0 holds the
// eight of its 32 output channels (one per lane) in registers and walks them one after the other -- the chain that
// bounds the sweep -- after applying the previous eight's z to them itself; meanwhile the other warps apply the
// previous z to the channels further on, as 8 x 8 x 4 FP64 tensor-core steps.  One barrier per eight channels; where
// a group begins, everyone finishes the update first and all warps take part in the product with G and the maxima.  88 us
// per 256 channels at N = 5120; one launch per 64 channels with the weights in registers and a rank-64 product after it
// took 38 + 15 us per 64.
// ---------------------------------------------------------------------------------------------------------
constexpr int kSweepCols = 32, kSub = 8, kSweepThreads = 256;
struct SweepSmem {
  double t[kLazy * kSweepCols];          // sum of L_kj z_k over the channels k done so far; element (r, c) at r * 32 + (c ^ 8 (r & 1))
  double u[2][kSub][kLazy];              // eight rows of L over the batch's columns, column c at c ^ 4 (row & 3)
  double ud[4][kSub][2 * kSub];          // eight rows of L, their own eight columns and the next eight
  double z[2][kSub][kSweepCols];         // column c at c ^ 4 (row & 3)
  double amax[kSweepThreads / 32][kSweepCols];
  unsigned char dead[kLazy];
};
__device__ __forceinline__ int sweep_t(int r, int c) { return r * kSweepCols + (c ^ ((r & 1) << 3)); }

// INT4: the code of w at scale s (inv = 1 / s, safe = s (1/2 - 1e-9)).  The product with the reciprocal decides the code
// wherever the remainder is clearly below half a step; elsewhere (ties, clipping, s == 0) the true division does.
__device__ __forceinline__ double quantize_int4(double w, double s, double inv, double safe) {
  const double t = w * inv;
  double q = (t + 6755399441055744.0) - 6755399441055744.0;   // 1.5 * 2^52: round half to even
  q = t > 7.0 ? 7.0 : (t < -8.0 ? -8.0 : q);
  if (!(fabs(fma(-q, s, w)) <= safe)) q = s > 0.0 ? fmin(fmax(rint(w / s), -8.0), 7.0) : 0.0;
  return q;
}

template <bool MX>
__global__ void __launch_bounds__(kSweepThreads, 2) gptq_sweep_kernel(const float* __restrict__ R,
                                                                      const unsigned char* __restrict__ dead,
                                                                      const double* __restrict__ T, int ldw, int N,
                                                                      const double* __restrict__ L, long ldl,
                                                                      const double* __restrict__ G, int b0,
                                                                      int channels, void* __restrict__ codes_out,
                                                                      void* __restrict__ scales_out,
                                                                      double* __restrict__ Z) {
  extern __shared__ __align__(16) unsigned char sweep_smem[];
  SweepSmem& sm = *reinterpret_cast<SweepSmem*>(sweep_smem);
  constexpr int kGroup = MX ? 32 : 64, kGroupSubs = kGroup / kSub;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n0 = blockIdx.x * kSweepCols, n = n0 + lane;
  const int fr = lane >> 2, fk = lane & 3;
  const int subs = channels / kSub;
  const double* const Lb = L + (long)b0 * ldl + b0;   // the batch's own corner of L

  // Eight rows of L from the block after their own on, by the `count` threads from `first` on.
  auto fetch_u = [&](int sub, int first, int count) {
    const int c0 = kSub * (sub + 1), pairs = (channels - c0) / 2;
    for (int i = tid - first; i < kSub * pairs; i += count) {
      const int k = i / pairs, c = c0 + 2 * (i - k * pairs);
      async_copy16(&sm.u[sub & 1][k][c ^ ((k & 3) << 2)], Lb + (long)(kSub * sub + k) * ldl + c, true);
    }
  };
  auto fetch_ud = [&](int sub) {   // by one warp
    if (sub >= subs) return;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int k = (lane >> 3) + 4 * i, c = 2 * (lane & 7);
      if (kSub * sub + c < channels) async_copy16(&sm.ud[sub & 3][k][c], Lb + (long)(kSub * sub + k) * ldl + kSub * sub + c, true);
    }
  };
  // The original weight of channel b0 + r in output channel c; live() afterwards makes a dead channel's 0.  (Two steps, so
  // that a load made ahead of its use does not wait for the flag.)
  auto original = [&](int r, int c) { return c < N ? __ldg(R + (long)(b0 + r) * N + c) : 0.0f; };
  auto live = [&](int r, float w) { return sm.dead[r] ? 0.0f : w; };
  for (int i = tid; i < channels * (kSweepCols / 2); i += kSweepThreads) {
    const int r = i / (kSweepCols / 2), c = 2 * (i % (kSweepCols / 2));
    async_copy16(&sm.t[sweep_t(r, c)], b0 > 0 ? T + (long)(b0 + r) * ldw + n0 + c : T, b0 > 0);   // zeros in the first batch
  }
  if (warp == 0) {
    fetch_ud(0);
    fetch_ud(1);
  }
  async_commit();
  if (tid < channels) sm.dead[tid] = dead[b0 + tid];
  async_wait<0>();
  __syncthreads();

  // Row blocks first, first + step, ... += L^T z of the eight channels `sub`.
  auto apply = [&](int sub, int first, int step) {
    double b[2][4];
    const double(*z)[kSweepCols] = sm.z[sub & 1];
    const double(*u)[kLazy] = sm.u[sub & 1];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) b[h][j] = z[4 * h + fk][(8 * j + fr) ^ (fk << 2)];
    for (int rb = first; rb < subs; rb += step) {
      double a[2], c[4][2];
#pragma unroll
      for (int h = 0; h < 2; ++h) a[h] = u[4 * h + fk][(kSub * rb + fr) ^ (fk << 2)];
      double2* at[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        at[j] = reinterpret_cast<double2*>(&sm.t[sweep_t(kSub * rb + fr, 8 * j + 2 * fk)]);
        c[j][0] = at[j]->x, c[j][1] = at[j]->y;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j) dmma_8x8x4(c[j], a[h], b[h][j]);
#pragma unroll
      for (int j = 0; j < 4; ++j) *at[j] = make_double2(c[j][0], c[j][1]);
    }
  };

  double s = 0.0, inv = 0.0, safe = 0.0;   // warp 0: the lane's running scale
  double z[kSub] = {};                     // warp 0: z of the previous eight channels
  float next_w0[kSub];                     // warp 0: original weights of the next eight, on their way
  if (warp == 0) {
#pragma unroll
    for (int i = 0; i < kSub; ++i) next_w0[i] = original(i, n);
  }
  for (int sub = 0; sub < subs; ++sub) {
    const bool entry = sub % kGroupSubs == 0;
    if (entry) {
      // The scale's weights: warp w forms eight rows of W + G^T t (G = inverse of the group's diagonal block of L).
      constexpr int kSteps = kGroup / 4;
      const int r0 = kSub * sub, in_block = r0 & (kNb - 1);
      const bool has_rows = warp < kGroupSubs;
      double g[kSteps];
      float w0[4][2];
      if (has_rows) {
#pragma unroll
        for (int k = 0; k < kSteps; ++k)
          g[k] = G[(long)(b0 + r0 + 4 * k + fk) * kNb + in_block + 8 * warp + fr];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int c = 0; c < 2; ++c) w0[j][c] = original(r0 + 8 * warp + fr, n0 + 8 * j + 2 * fk + c);
      }
      if (sub > 0) {
        apply(sub - 1, sub + warp, kSweepThreads / 32);
        __syncthreads();
      }
      if (has_rows) {
        double y[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j][0] = live(r0 + 8 * warp + fr, w0[j][0]), y[j][1] = live(r0 + 8 * warp + fr, w0[j][1]);
#pragma unroll
        for (int k = 0; k < kSteps; ++k)
          if (k < 2 * (warp + 1)) {   // G is upper triangular
#pragma unroll
            for (int j = 0; j < 4; ++j) dmma_8x8x4(y[j], g[k], sm.t[sweep_t(r0 + 4 * k + fk, 8 * j + fr)]);
          }
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            double m = fabs(y[j][c]);
#pragma unroll
            for (int o = 4; o < 32; o *= 2) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (fr == 0) sm.amax[warp][8 * j + 2 * fk + c] = m;
          }
      }
      __syncthreads();
    }
    if (warp == 0) {
      fetch_ud(sub + 2);
      async_commit();
      if (entry) {
        double m = sm.amax[0][lane];
#pragma unroll
        for (int i = 1; i < kGroupSubs; ++i) m = fmax(m, sm.amax[i][lane]);
        const long at = (long)((b0 + kSub * sub) / kGroup) * N + n;
        if constexpr (MX) {
          int x = m > 0.0 ? ilogb(m) - 2 : -127;
          x = max(-127, min(125, x));
          s = scalbn(1.0, x);
          inv = scalbn(1.0, -x);
          if (n < N) static_cast<uint8_t*>(scales_out)[at] = (uint8_t)(x + 127);
        } else {
          const float s32 = (float)(m / 7.0);  // FP64 quotient rounded once to FP32
          if (n < N) static_cast<float*>(scales_out)[at] = s32;
          s = (double)s32;
          inv = s > 0.0 ? 1.0 / s : 0.0;
          safe = s * (0.5 - 1e-9);
        }
      }
      double w[kSub];
      float w0[kSub];
#pragma unroll
      for (int i = 0; i < kSub; ++i) {
        w0[i] = live(kSub * sub + i, next_w0[i]);
        w[i] = (double)w0[i] + sm.t[sweep_t(kSub * sub + i, lane)];
      }
      if (sub + 1 < subs) {
#pragma unroll
        for (int i = 0; i < kSub; ++i) next_w0[i] = original(kSub * (sub + 1) + i, n);
      }
      if (!entry) {   // the previous eight's z, which the other warps apply further on
#pragma unroll
        for (int k = 0; k < kSub; ++k)
#pragma unroll
          for (int i = 0; i < kSub; ++i) w[i] = fma(z[k], sm.ud[(sub - 1) & 3][k][kSub + i], w[i]);
      }
      const double(*ud)[2 * kSub] = sm.ud[sub & 3];
#pragma unroll
      for (int k = 0; k < kSub; ++k) {
        int code;
        if constexpr (MX) {
          const double v = fmin(fabs(w[k]) * inv, 6.0);  // exact: the scale is a power of two
          // one comparison per midpoint between neighbouring magnitudes, strict where the lower neighbour is the even code
          const int idx = (v > 0.25) + (v >= 0.75) + (v > 1.25) + (v >= 1.75) + (v > 2.5) + (v >= 3.5) + (v > 5.0);
          const double twice = __hiloint2double(0x43300000, (0xC8643210u >> (4 * idx)) & 15u) - 4503599627370496.0;
          z[k] = fma(w[k] < 0.0 ? 0.5 * twice : -0.5 * twice, s, (double)w0[k]);
          code = idx + (w[k] < 0.0 ? 8 : 0);
        } else {
          const double q = quantize_int4(w[k], s, inv, safe);
          z[k] = fma(-q, s, (double)w0[k]);
          code = (int)q;
        }
#pragma unroll
        for (int i = k + 1; i < kSub; ++i) w[i] = fma(z[k], ud[k][i], w[i]);
        const int row = b0 + kSub * sub + k;
        if (n < N) {
          if constexpr (MX) static_cast<uint8_t*>(codes_out)[(long)row * N + n] = (uint8_t)code;
          else static_cast<int8_t*>(codes_out)[(long)row * N + n] = (int8_t)code;
        }
        sm.z[sub & 1][k][lane ^ ((k & 3) << 2)] = z[k];
        Z[(long)(kSub * sub + k) * ldw + n] = z[k];
      }
      async_wait<0>();
    } else {
      fetch_u(sub, 32, kSweepThreads - 32);
      async_commit();
      if (!entry) apply(sub - 1, sub + warp, kSweepThreads / 32 - 1);
      async_wait<0>();
    }
    __syncthreads();
  }
}

// The temporaries of one call, carved out of one workspace (256-byte aligned pieces).
struct Workspace {
  double *H, *L, *G, *Xd, *T, *Z, *damp;
  unsigned char* dead;
  int* not_pd;
  int ldw;
  size_t bytes;
  static size_t padded_tokens(int M_cal) { return ((size_t)M_cal + kBK - 1) / kBK * kBK; }   // whole slices of the product
  Workspace(unsigned char* base, int K, int N, int M_cal) {
    size_t off = 0;
    auto take = [&](size_t n) {
      unsigned char* p = reinterpret_cast<unsigned char*>(reinterpret_cast<uintptr_t>(base) + off);
      off += (n + 255) & ~static_cast<size_t>(255);
      return p;
    };
    const size_t kk = (size_t)K * K * sizeof(double);
    G = reinterpret_cast<double*>(take((size_t)K * kNb * sizeof(double)));
    ldw = (N + kNb - 1) / kNb * kNb;   // rows of T and Z padded to whole tiles
    H = reinterpret_cast<double*>(take(kk));
    L = reinterpret_cast<double*>(take(kk));
    T = reinterpret_cast<double*>(take((size_t)K * ldw * sizeof(double)));
    Z = reinterpret_cast<double*>(take((size_t)kLazy * ldw * sizeof(double)));
    Xd = reinterpret_cast<double*>(take(padded_tokens(M_cal) * K * sizeof(double)));
    damp = reinterpret_cast<double*>(take(sizeof(double)));
    dead = take((size_t)K);
    not_pd = reinterpret_cast<int*>(take(sizeof(int)));
    bytes = off;
  }
};

struct OwnedAllocation {
  void* p = nullptr;
  ~OwnedAllocation() { cudaFree(p); }
};

template <int BM, bool AK, bool BK>
void launch_dgemm(cudaStream_t st, const GemmArgs& g) {
  static_assert(dgemm_smem_bytes(BM) <= 113 * 1024, "two blocks per SM");
  const dim3 grid(g.N / kBN, (g.M + BM - 1) / BM);
  dgemm_kernel<BM, AK, BK><<<grid, 256, dgemm_smem_bytes(BM), st>>>(g);
}
// 128-row tiles where they fill the 148 SMs; 64-row tiles (twice the blocks, 4/3 of the operand traffic) where they would not.
template <bool AK, bool BK>
void dgemm(cudaStream_t st, const GemmArgs& g) {
  if (g.M <= 0 || g.N <= 0 || g.Kd <= 0) return;
  const long blocks = (long)(g.N / kBN) * ((g.M + 127) / 128);
  if (g.M > 64 && blocks >= 148) launch_dgemm<128, AK, BK>(st, g);
  else launch_dgemm<64, AK, BK>(st, g);
}
template <bool AK, bool BK>
bool prepare_dgemm() {
  return cudaFuncSetAttribute(dgemm_kernel<128, AK, BK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dgemm_smem_bytes(128)) == cudaSuccess &&
         cudaFuncSetAttribute(dgemm_kernel<64, AK, BK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dgemm_smem_bytes(64)) == cudaSuccess;
}
// Shared-memory limits of this file's kernels on the current device.
bool prepare_kernels() {
  return prepare_dgemm<false, false>() && prepare_dgemm<true, true>() &&
         cudaFuncSetAttribute(chol_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCholSmemBytes) == cudaSuccess &&
         cudaFuncSetAttribute(gptq_sweep_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SweepSmem)) == cudaSuccess &&
         cudaFuncSetAttribute(gptq_sweep_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SweepSmem)) == cudaSuccess;
}

bool gptq_shape_ok(int K, int N, int M_cal) {
  return K > 0 && N > 0 && K % kNb == 0 && K <= 16384 && N <= 65536 && M_cal >= 0 && M_cal <= (1 << 20);
}

}  // namespace

extern "C" size_t w4a4_gptq_workspace_bytes(int K, int N, int M_cal) {
  if (!gptq_shape_ok(K, N, M_cal)) return 0;
  return Workspace(nullptr, K, N, M_cal).bytes;
}

namespace {

// H (upper tiles) = beta H + X^T X, X [rows, K] in FP64, rows a multiple of kBK.
void statistic(cudaStream_t st, const double* X, int rows, int K, double* H, double beta) {
  GemmArgs g{K, K, rows, X, K, X, K, H, K, 1.0, beta};
  g.upper_out = true;
  dgemm<false, false>(st, g);
}

w4a4_status_t gptq_run(bool mx, int device, const float* R, const uint16_t* Xhat, int M_cal, const double* H_in, int K,
                       int N, double percdamp, void* codes, void* scales, void* workspace, size_t workspace_bytes,
                       void* stream) {
  if (R == nullptr || codes == nullptr || scales == nullptr) return W4A4_ERR_INVALID_ARG;
  if ((Xhat == nullptr) == (H_in == nullptr)) return W4A4_ERR_INVALID_ARG;  // exactly one source of H
  if (Xhat == nullptr) M_cal = 0;
  if (!gptq_shape_ok(K, N, M_cal)) return W4A4_ERR_SHAPE;
  if (Xhat != nullptr && M_cal <= 0) return W4A4_ERR_SHAPE;
  if (!(percdamp >= 0.0)) return W4A4_ERR_INVALID_ARG;
  const size_t need = Workspace(nullptr, K, N, M_cal).bytes;
  if (workspace != nullptr && (workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255) != 0))
    return W4A4_ERR_INVALID_ARG;
  if (cudaSetDevice(device) != cudaSuccess) return W4A4_ERR_CUDA;
  int major = 0;   // (one attribute: the whole property record takes the driver milliseconds)
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess) return W4A4_ERR_CUDA;
  if (major != 10) return W4A4_ERR_ARCH;
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  OwnedAllocation own;
  if (workspace == nullptr) {
    if (cudaMalloc(&own.p, need) != cudaSuccess) {
      cudaGetLastError();
      return W4A4_ERR_ALLOC;
    }
    workspace = own.p;
  }
  const Workspace d(static_cast<unsigned char*>(workspace), K, N, M_cal);
  if (!prepare_kernels()) {
    cudaGetLastError();
    return W4A4_ERR_CUDA;
  }
  const size_t kk = (size_t)K * K * sizeof(double);
  cudaMemsetAsync(d.not_pd, 0, sizeof(int), st);

  // 1. H, its dead channels and damping.
  if (Xhat != nullptr) {
    const long n = (long)M_cal * K, padded = (long)Workspace::padded_tokens(M_cal) * K;
    bf16_to_f64_kernel<<<(unsigned)((padded / 2 + 255) / 256), 256, 0, st>>>(Xhat, reinterpret_cast<double2*>(d.Xd), n, padded);
    statistic(st, d.Xd, (int)(padded / K), K, d.H, 0.0);
  } else {
    cudaMemcpyAsync(d.H, H_in, kk, cudaMemcpyDeviceToDevice, st);
  }
  gptq_diag_kernel<<<1, 1024, 0, st>>>(d.H, K, percdamp, d.dead, d.damp);

  // 2. H = V V^T, band by band from the last channels: inside a band of kBand columns every 64-column block is factored,
  // solved against all rows above it and applied to the band's columns still to come; the columns to the left of the band
  // then take the whole band's panels in one product that is kBand deep.
  for (int hi = K; hi > 0;) {
    const int lo = hi - kBand > 0 ? hi - kBand : 0;
    for (int j0 = hi - kNb; j0 >= lo; j0 -= kNb) {
      chol_step_kernel<<<j0 > 0 ? j0 / kNb : 1, kCholThreads, kCholSmemBytes, st>>>(d.H, d.L, K, j0, d.dead, d.damp, d.not_pd);
      // H[0:j0, lo:j0] -= P P[lo:j0]^T, P = the panel just solved
      GemmArgs g{j0, j0 - lo, kNb, d.H + j0, K, d.H + (long)lo * K + j0, K, d.H + lo, K, -1.0, 1.0};
      g.upper_out = true;
      g.diag_shift = lo;
      dgemm<true, true>(st, g);
    }
    // H[0:lo, 0:lo] -= P P^T over the band's panels
    GemmArgs far{lo, lo, hi - lo, d.H + lo, K, d.H + lo, K, d.H, K, -1.0, 1.0};
    far.upper_out = true;
    dgemm<true, true>(st, far);
    hi = lo;
  }

  // 3. The sweep, one lazy batch of kLazy input channels per launch, and after each T[later] += L[batch, later]^T Z.
  unit_inverse_kernel<<<K / kNb, kNb, 0, st>>>(d.L, d.G, K);
  const int ldw = d.ldw;
  for (int b0 = 0; b0 < K; b0 += kLazy) {
    const int b1 = b0 + kLazy < K ? b0 + kLazy : K;
    const unsigned blocks = (unsigned)(ldw / kSweepCols);
    if (mx) gptq_sweep_kernel<true><<<blocks, kSweepThreads, sizeof(SweepSmem), st>>>(R, d.dead, d.T, ldw, N, d.L, K, d.G, b0, b1 - b0, codes, scales, d.Z);
    else gptq_sweep_kernel<false><<<blocks, kSweepThreads, sizeof(SweepSmem), st>>>(R, d.dead, d.T, ldw, N, d.L, K, d.G, b0, b1 - b0, codes, scales, d.Z);
    dgemm<false, false>(st, {K - b1, ldw, b1 - b0, d.L + (long)b0 * K + b1, K, d.Z, ldw, d.T + (long)b1 * ldw, ldw, 1.0, b0 > 0 ? 1.0 : 0.0});
  }

  int not_pd = 0;
  if (cudaMemcpyAsync(&not_pd, d.not_pd, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess ||
      cudaGetLastError() != cudaSuccess)
    return W4A4_ERR_CUDA;
  return not_pd ? W4A4_ERR_INVALID_ARG : W4A4_OK;
}

}  // namespace

extern "C" w4a4_status_t w4a4_gptq_accumulate(int device, const uint16_t* Xhat, int M_cal, int K, double* H,
                                              void* stream) {
  if (Xhat == nullptr || H == nullptr) return W4A4_ERR_INVALID_ARG;
  if (!gptq_shape_ok(K, 1, M_cal) || M_cal <= 0) return W4A4_ERR_SHAPE;
  if (cudaSetDevice(device) != cudaSuccess) return W4A4_ERR_CUDA;
  int major = 0;   // (one attribute: the whole property record takes the driver milliseconds)
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess) return W4A4_ERR_CUDA;
  if (major != 10) return W4A4_ERR_ARCH;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  constexpr int kChunkRows = 4096;  // tokens converted to FP64 at a time
  const int chunk = M_cal < kChunkRows ? M_cal : kChunkRows;
  OwnedAllocation xd;
  if (cudaMalloc(&xd.p, Workspace::padded_tokens(chunk) * K * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    return W4A4_ERR_ALLOC;
  }
  if (!prepare_kernels()) return W4A4_ERR_CUDA;
  double* Xd = static_cast<double*>(xd.p);
  for (int m0 = 0; m0 < M_cal; m0 += chunk) {
    const int rows = M_cal - m0 < chunk ? M_cal - m0 : chunk;
    const long n = (long)rows * K, padded = (long)Workspace::padded_tokens(rows) * K;
    bf16_to_f64_kernel<<<(unsigned)((padded / 2 + 255) / 256), 256, 0, st>>>(Xhat + (size_t)m0 * K, reinterpret_cast<double2*>(Xd), n, padded);
    statistic(st, Xd, (int)(padded / K), K, H, 1.0);
  }
  if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) return W4A4_ERR_CUDA;
  return W4A4_OK;
}

extern "C" w4a4_status_t w4a4_gptq_quantize(int device, const float* R, const uint16_t* Xhat, int M_cal,
                                            const double* H_in, int K, int N, double percdamp, int8_t* codes,
                                            float* scales, void* workspace, size_t workspace_bytes, void* stream) {
  return gptq_run(false, device, R, Xhat, M_cal, H_in, K, N, percdamp, codes, scales, workspace, workspace_bytes, stream);
}

extern "C" w4a4_status_t w4a4_mx_gptq_quantize(int device, const float* R, const uint16_t* Xhat, int M_cal,
                                               const double* H_in, int K, int N, double percdamp, uint8_t* codes,
                                               uint8_t* exps, void* workspace, size_t workspace_bytes, void* stream) {
  return gptq_run(true, device, R, Xhat, M_cal, H_in, K, N, percdamp, codes, exps, workspace, workspace_bytes, stream);
}
