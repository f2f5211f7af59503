// mg_colour_tc.cuh -- colour quadratic form on the 5th-generation tensor cores.
//
// Step A5 (paper Sect. 3: the "colour algebra" step run at reduced precision)
// for the 128 helicities h of one event:
//     ME_h = sum_ij Re/Im J_i(h) KNUM_ij Re/Im J_j(h)       (C = KNUM / CDEN)
// is computed as D = A . KNUM with A = [128 helicities x K] (K = NCOL padded to
// a multiple of 16) on the tensor cores, then a per-thread row dot J . D.
//
//   * KNUM holds small integers (|KNUM| <= 4096): exact in FP16.
//   * A = s * J split into FP16 hi + lo (hi = fp16(sJ), lo = fp16(sJ - hi)),
//     s a per-row power of two putting max|J| in [1, 2): the pair carries
//     ~22 significant bits, and D = A_hi.KNUM + A_lo.KNUM accumulates in FP32.
//   * Re and Im parts use two accumulators of N columns each in TMEM
//     (cta_group::1, M = 128: row h of D lives in TMEM lane h).
//   * One elected thread issues tcgen05.mma; completion is signalled on an
//     mbarrier through tcgen05.commit; every wait is bounded.
//
// Shared-memory operand layout: K-major, no swizzle ("interleaved" core
// matrices of 8 rows x 16 bytes).  Element (row r, k) of a tile lives at
//     (r / 8) * SBO + (k / 8) * LBO + (r % 8) * 16 + (k % 8) * 2
// with LBO = 128 bytes (next 8 k) and SBO = (K / 8) * 128 bytes (next 8 rows).
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "mg_kernels.cuh"

namespace mg {
namespace tc {

__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
// D[tmem] (+)= A[smem] . B[smem]^T, kind::f16 (FP16 inputs, FP32 accumulate)
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// 16 consecutive 32-bit TMEM columns of this thread's lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// shared-memory matrix descriptor: no swizzle, K-major core matrices
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of the 5th-generation tensor cores
  // base offset 0, relative LBO mode, layout type 0 (no swizzle)
  return d;
}
// instruction descriptor, kind::f16: D FP32, A/B FP16, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
  return (1u << 4)                        // D format: FP32
         | (0u << 7) | (0u << 10)         // A, B format: FP16
         | ((uint32_t)(N >> 3) << 17)     // N / 8
         | ((uint32_t)(M >> 4) << 24);    // M / 16
}

constexpr uint32_t LBO = 128;

__host__ __device__ constexpr int pad16(int n) { return ((n + 15) / 16) * 16; }

// byte offset of element (row, k) in a K-major no-swizzle tile with K columns
__host__ __device__ constexpr uint32_t tile_off(int row, int k, int K) {
  return (uint32_t)((row / 8) * (K / 8) * 128 + (k / 8) * 128 + (row % 8) * 16 + (k % 8) * 2);
}

}  // namespace tc

// The colour form of 128 rows (TMEM lane = row), Re and Im one after the other
// through one pair of operand tiles.  (1) Each row's thread writes its part's
// flows, scaled by the row's power of two s, as FP16 hi + lo.
template <class P, int K>
__device__ __forceinline__ float colour_scale(const float (&fr)[P::NCOL], const float (&fi)[P::NCOL]) {
  float mx = 0.f;
#pragma unroll
  for (int k = 0; k < P::NCOL; k++) mx = fmaxf(mx, fmaxf(fabsf(fr[k]), fabsf(fi[k])));
  const int ex = mx > 0.f ? ((int)((__float_as_uint(mx) >> 23) & 0xff) - 127) : 0;
  return __uint_as_float((uint32_t)(127 - ex) << 23);  // 2^-ex: max |J| in [1, 2)
}
template <class P, int K>
__device__ __forceinline__ void colour_operands(unsigned char* atile, size_t a_tile, int row, float s,
                                                const float (&f)[P::NCOL]) {
#pragma unroll
  for (int j = 0; j < K / 8; j++) {
    __align__(16) __half hi[8], lo[8];
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int k = 8 * j + q;
      const float x = k < P::NCOL ? s * f[k < P::NCOL ? k : 0] : 0.f;
      hi[q] = __float2half_rn(x);
      lo[q] = __float2half_rn(x - __half2float(hi[q]));
    }
    const uint32_t off = tc::tile_off(row, 8 * j, K);
    *reinterpret_cast<uint4*>(atile + off) = *reinterpret_cast<const uint4*>(hi);
    *reinterpret_cast<uint4*>(atile + a_tile + off) = *reinterpret_cast<const uint4*>(lo);
  }
}

// (2) One elected thread: D = (A_hi + A_lo) . KNUM into the N columns at d;
// completion arrives on mma_bar.
template <int K, int N>
__device__ __forceinline__ void colour_mma(uint32_t d, uint32_t a_addr, uint32_t b_addr, size_t a_tile,
                                           uint64_t* mma_bar) {
  constexpr uint32_t idesc = tc::idesc_f16(128, N);
  constexpr uint32_t SBO = (K / 8) * 128;
  tc::fence_after_sync();
  for (int kk = 0; kk < K / 16; kk++) {
    const uint64_t bd = tc::smem_desc(b_addr + kk * 2 * tc::LBO, tc::LBO, SBO);
    const uint32_t at = a_addr + kk * 2 * tc::LBO;
    tc::mma_f16(d, tc::smem_desc(at, tc::LBO, SBO), bd, idesc, kk > 0 ? 1u : 0u);
    tc::mma_f16(d, tc::smem_desc(at + (uint32_t)a_tile, tc::LBO, SBO), bd, idesc, 1u);
  }
  tc::mma_commit(mma_bar);
}

// (3) Warp-collective: the row of D at TMEM address d contracted with the
// flows, sum_k J_k D_k (still scaled by s).
template <class P, int N>
__device__ __forceinline__ float colour_readback(uint32_t d, const float (&f)[P::NCOL]) {
  float sum = 0.f;
#pragma unroll
  for (int c = 0; c < N; c += 16) {
    float v[16];
    tc::tmem_ld16(d + c, v);
    tc::tmem_wait_ld();
#pragma unroll
    for (int q = 0; q < 16; q++)
      if (c + q < P::NCOL) sum = fmaf(f[c + q < P::NCOL ? c + q : 0], v[q], sum);
  }
  return sum;
}

// FP16 bit pattern of an integer, or -1 if it is not exactly representable.
inline int fp16_bits_of_int(int v) {
  if (v == 0) return 0;
  const int sgn = v < 0 ? 0x8000 : 0;
  unsigned a = (unsigned)(v < 0 ? -v : v);
  int e = 31 - __builtin_clz(a);           // a in [2^e, 2^(e+1))
  if (e > 15) return -1;
  if (e > 10 && (a & ((1u << (e - 10)) - 1u))) return -1;  // more than 11 significant bits
  const unsigned mant = e >= 10 ? (a >> (e - 10)) & 0x3FFu : (a << (10 - e)) & 0x3FFu;
  return sgn | ((e + 15) << 10) | (int)mant;
}

// FP16 image of the colour-matrix numerators in the B-operand layout.
// Returns false if a numerator is not exact in FP16.
inline bool colour_tile_host(const int* knum, int ncol, unsigned short* out /* [N*K] */) {
  const int K = tc::pad16(ncol), N = tc::pad16(ncol);
  for (int i = 0; i < N * K; i++) out[i] = 0;
  for (int n = 0; n < ncol; n++)
    for (int k = 0; k < ncol; k++) {
      const int b = fp16_bits_of_int(knum[n * ncol + k]);
      if (b < 0) return false;
      out[tc::tile_off(n, k, K) / 2] = (unsigned short)b;
    }
  return true;
}

// ---------------------------------------------------------------------------
// Two-phase mixed path for processes whose colour operands do not fit in
// shared memory beside the per-event state (120 flows): the FP32 flows of
// every (event, helicity) row go to a workspace in HBM; a second kernel
// contracts them with the colour matrix (mg_recursion_kernels.cuh).
// ---------------------------------------------------------------------------
template <class P>
struct LayoutRows {
  static constexpr int K = tc::pad16(P::NCOL);
  static constexpr int N = tc::pad16(P::NCOL);
  static constexpr size_t a_tile = size_t(128) * K * 2;  // FP16 [128][K]
  static constexpr size_t b_tile = size_t(N) * K * 2;    // FP16 [N][K]
  static constexpr size_t a_off = 128;                    // MMA bar, TMEM address
  static constexpr size_t b_off = a_off + 2 * a_tile;   // one part (Re or Im) at a time: hi, lo
  static constexpr size_t base_bytes = b_off + b_tile;
  static constexpr uint32_t tmem_cols = (2 * N <= 32) ? 32 : (2 * N <= 64) ? 64 : (2 * N <= 128) ? 128 : 256;
};

// The stream-ordered workspace of one call: at most ROWS_WORKSPACE bytes of
// flows (FP32 complex).  The flow kernel writes every helicity of an event,
// whatever the list, so the workspace is a number of events, the same for every
// list: the call's, padded to 128, or as many as fit (8704 of 120 flows and 128
// helicities); larger calls run slice by slice.  When it was shared out by the
// listed helicities, 256 events with 94 of 128 listed took two slices and 117
// us instead of 69, and from 1.1 M events on it grew past the bound.
constexpr size_t ROWS_WORKSPACE = size_t(1) << 30;

// events of one slice (nhel: all helicities of the process)
inline long long rows_slice(int ncol, int nhel, long long nevt) {
  const size_t per128 = 128 * size_t(ncol) * size_t(nhel) * sizeof(float2);
  const long long most = (long long)(ROWS_WORKSPACE / per128) * 128, all = (nevt + 127) / 128 * 128;
  return all < most ? all : most;
}
// bytes one two-phase launch takes from the stream-ordered allocator
inline size_t rows_workspace_bytes(int ncol, int nhel, long long nevt) {
  return nevt <= 0 ? 0 : size_t(rows_slice(ncol, nhel, nevt)) * size_t(ncol) * size_t(nhel) * sizeof(float2);
}

}  // namespace mg
