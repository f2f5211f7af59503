// mg_unweight.cu -- hit-or-miss unweighting on the device (mg_unweight in
// include/mg.h).
//
// The paper (Sect. 2) lists hit-or-miss unweighting among the serial steps
// that follow the matrix element in the event generator, and names it as a
// candidate to offload to the GPU.  Event i is kept when r_i * w_max < w_i
// (r_i uniform in [0, 1)); the kept indices are written in increasing order,
// so the result does not depend on the launch configuration.  Two launches:
// per tile of 4096 events, the accept bits (one warp ballot per 32 events,
// n/8 bytes in all) and their count; then a warp per tile ranks its kept events
// from its bits alone and writes their indices behind the kept events of the
// tiles before it, whose counts its block adds up for itself (past 16384 tiles
// a scan of the counts in between).  w and r are read once: 16 bytes per event,
// plus 8 per kept index; bound by HBM.
#include <cuda_runtime.h>

#include "mg.h"

// MG_UW_FP32_FIRST (default 1): the decision r_i * w_max < w_i is taken in
// FP32 where the FP32 values are far enough apart to make it certain, in FP64
// otherwise (the FP64 multiply-and-compare of every event made the count pass
// FP64-bound: 82 % of the FP64 pipe on GB300, where FP64 runs at 1/64 of
// FP32); the kept set is the same bit for bit.
#ifndef MG_UW_FP32_FIRST
#define MG_UW_FP32_FIRST 1
#endif

namespace {

// MG_UW_PER_THREAD: events per thread and tile, a multiple of 4 (A/B on GB300,
// 67 M events: 4 / 8 / 16 / 24 / 32 -> 0.40 / 0.33 / 0.29 / 0.40 / 0.41 ms)
#ifndef MG_UW_PER_THREAD
#define MG_UW_PER_THREAD 16
#endif
constexpr int UW_THREADS = 256;
constexpr int UW_PER_THREAD = MG_UW_PER_THREAD;
constexpr int UW_TILE = UW_THREADS * UW_PER_THREAD;  // events per tile
constexpr int UW_WARPS = UW_THREADS / 32;
constexpr int UW_WORDS = UW_PER_THREAD * UW_WARPS;  // accept-bit words per tile

// x truncated toward zero to a normal FP32 value, built from its bits with
// integer operations (no FP64 instruction); false where x is zero, subnormal
// in FP32, beyond the FP32 range, infinite or NaN.  |x - f| < 2^-23 |x|.
__device__ __forceinline__ bool f32_trunc(double x, float& f) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ffu);  // biased FP64 exponent
  if (e < 897 || e > 1150) return false;    // FP32 exponents 1..254
  f = __uint_as_float((unsigned)(b >> 32 & 0x80000000u) | ((unsigned)(e - 896) << 23) |
                      (unsigned)((b >> 29) & 0x7fffffu));
  return true;
}

// r * w_max < w, exactly as in FP64.  In FP32, p = rf * wmf carries a
// relative error below 3e-7 from the truncations and the product, and wf
// below 1.2e-7; a gap |p - wf| above 1e-6 |wf| (with p a normal FP32 value)
// therefore has the sign of r * w_max - w, which the FP64 product's rounding
// (1.1e-16) cannot change.  Closer cases, and anything outside the FP32
// normal range (zero, NaN, infinities included), take the FP64 comparison.
__device__ __forceinline__ bool kept_exact(double r, double w, double w_max, float wmf, bool wm_ok) {
#if MG_UW_FP32_FIRST
  float rf, wf;
  if (wm_ok && f32_trunc(r, rf) && f32_trunc(w, wf)) {
    const float p = rf * wmf;
    const float ap = fabsf(p);
    const float d = p - wf;
    if (ap >= 1.17549435e-38f && ap <= 3.40282347e38f && fabsf(d) > 1e-6f * fabsf(wf)) return d < 0.f;
  }
#endif
  return r * w_max < w;
}

// First pass.  Thread t of tile b takes events b*TILE + j*THREADS + t, j < PER_THREAD
// (coalesced); word j*WARPS + warp of the tile's bits holds the ballot of
// events b*TILE + j*THREADS + warp*32 + lane, so the words in order cover the
// tile in increasing index order.
__global__ void __launch_bounds__(UW_THREADS)
    tile_count_kernel(const double* __restrict__ w, const double* __restrict__ r, long long n, double w_max,
                      long long* __restrict__ counts, unsigned* __restrict__ bits) {
  __shared__ int warp_sum[UW_WARPS];
  const long long base = (long long)blockIdx.x * UW_TILE;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned* tb = bits + (long long)blockIdx.x * UW_WORDS;
  float wmf = 0.f;
  const bool wm_ok = f32_trunc(w_max, wmf);
  // every load of the tile issued before the first vote
  double wv[UW_PER_THREAD], rv[UW_PER_THREAD];
#pragma unroll
  for (int j = 0; j < UW_PER_THREAD; j++) {
    const long long i = base + j * UW_THREADS + threadIdx.x;
    wv[j] = i < n ? __ldcs(w + i) : 0.0;
    rv[j] = i < n ? __ldcs(r + i) : 1.0;
  }
  int c = 0;
#pragma unroll
  for (int j = 0; j < UW_PER_THREAD; j++) {
    const long long i = base + j * UW_THREADS + threadIdx.x;
    const unsigned m = __ballot_sync(0xffffffffu, i < n && kept_exact(rv[j], wv[j], w_max, wmf, wm_ok));
    if (lane == 0) tb[j * UW_WARPS + warp] = m;
    c += __popc(m);  // the same in every lane of the warp
  }
  if (lane == 0) warp_sum[warp] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    for (int k = 0; k < UW_WARPS; k++) t += warp_sum[k];
    counts[blockIdx.x] = t;
  }
}

// Many tiles: exclusive scan of the tile counts in place, by one block, in
// passes of SCAN_T * SCAN_V tiles: thread t of warp w holds the tiles
// base + j*SCAN_T + t (j < SCAN_V; coalesced loads and stores), so the
// (j, w, lane) order is the index order.  Warp scans of each j, one scan of
// the SCAN_V * 32 warp totals in order by the first warp, the pass's total
// carried to the next; the grand total into *n_acc.
constexpr int SCAN_T = 1024, SCAN_V = 16, SCAN_W = SCAN_T / 32;

__global__ void __launch_bounds__(SCAN_T) tile_scan_kernel(long long* __restrict__ counts, long long ntiles,
                                                           long long* __restrict__ n_acc) {
  __shared__ long long wt[SCAN_V * SCAN_W];  // warp totals, then their exclusive prefixes
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  long long carry = 0;  // kept by the first warp
  for (long long base = 0; base < ntiles; base += (long long)SCAN_T * SCAN_V) {
    // tile counts are at most TILE: a warp's partial sums fit in 32 bits
    int ex[SCAN_V];
#pragma unroll
    for (int j = 0; j < SCAN_V; j++) {
      const long long b = base + (long long)j * SCAN_T + t;
      ex[j] = b < ntiles ? (int)counts[b] : 0;
    }
#pragma unroll
    for (int j = 0; j < SCAN_V; j++) {
      int x = ex[j];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += a;
      }
      if (lane == 31) wt[j * SCAN_W + warp] = x;
      ex[j] = x - ex[j];  // exclusive within the warp
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll 1
      for (int q = 0; q < SCAN_V * SCAN_W / 32; q++) {
        const long long own = wt[q * 32 + lane];
        long long x = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const long long a = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += a;
        }
        wt[q * 32 + lane] = carry + x - own;
        carry += __shfl_sync(0xffffffffu, x, 31);
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < SCAN_V; j++) {
      const long long b = base + (long long)j * SCAN_T + t;
      if (b < ntiles) counts[b] = wt[j * SCAN_W + warp] + ex[j];
    }
    __syncthreads();  // wt is rewritten by the next pass
  }
  if (t == 0) *n_acc = carry;
}

// Last pass: a warp per tile, WRITE_TILES tiles per block.  The kept events
// before the block's first tile: SCANNED, from the scan; otherwise the block
// adds up the counts of all earlier tiles (ntiles^2 / 4 bytes of L2 reads over
// all blocks, 67 MB at SUM_TILES tiles).  A call with the sum / with the scan,
// us: 512 tiles 35.0 / 45.0, 4096 69.9 / 76.8, 8192 113 / 119, 16384 193 / 201,
// 24576 273 / 286, 32768 357 / 365, 65536 708 / 705; the reads grow with the
// square of the tiles, and the line stays a factor of two below the crossing.
// 33.6 M events, 2.7 % kept: count 78 + scan 8 + a
// block per tile 22 us before; count 78 + write 9 us now, 111.8 -> 92.4 us a
// call; 8 / 16 / 32 tiles per block 91.9 / 92.4 / 93.2 us; without the early
// launch 96.4 us.
// Lane l takes words l*WPL .. of the tile, consecutive events; a tile with few
// kept events writes them lane by lane, a fuller one word by word (coalesced).
// bits and counts are still being written while this kernel's first blocks wait:
// they are plain pointers, since const __restrict__ would promise that nothing
// writes them during the kernel and so allow loads (also through the
// non-coherent path) ahead of the wait.
constexpr int WRITE_TILES = 16;
constexpr long long SUM_TILES = 16384;

template <bool SCANNED>
__global__ void __launch_bounds__(UW_THREADS)
    tile_write_kernel(unsigned* bits, long long* counts, long long ntiles, long long* n_acc, long long* idx_out) {
  constexpr int WPL = UW_WORDS / 32;               // words per lane
  constexpr int PER_WARP = WRITE_TILES / UW_WARPS;  // tiles per warp
  static_assert(UW_WORDS % 32 == 0 && WRITE_TILES <= 32, "whole warps of words, at most one tile count per lane");
  __shared__ long long part[UW_WARPS], first[WRITE_TILES];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long t0 = (long long)blockIdx.x * WRITE_TILES;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // launched while the pass before it drains
  unsigned m[PER_WARP][WPL];
#pragma unroll
  for (int k = 0; k < PER_WARP; k++) {
    const long long t = t0 + warp * PER_WARP + k;
#pragma unroll
    for (int q = 0; q < WPL; q++) m[k][q] = t < ntiles ? bits[t * UW_WORDS + lane * WPL + q] : 0u;
  }
  if constexpr (SCANNED) {
    if (threadIdx.x < WRITE_TILES) first[threadIdx.x] = t0 + threadIdx.x < ntiles ? counts[t0 + threadIdx.x] : 0;
    __syncthreads();
  } else {
    long long before = 0;
#pragma unroll 8
    for (long long t = threadIdx.x; t < t0; t += UW_THREADS) before += counts[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (lane == 0) part[warp] = before;
    __syncthreads();
    if (warp == 0) {
      long long sum = 0;
#pragma unroll
      for (int k = 0; k < UW_WARPS; k++) sum += part[k];
      const long long own = lane < WRITE_TILES && t0 + lane < ntiles ? counts[t0 + lane] : 0;
      long long sc = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const long long a = __shfl_up_sync(0xffffffffu, sc, o);
        if (lane >= o) sc += a;
      }
      if (lane < WRITE_TILES) first[lane] = sum + sc - own;
      if (lane == 31 && t0 + WRITE_TILES >= ntiles) *n_acc = sum + sc;
    }
    __syncthreads();
  }
#pragma unroll 1
  for (int k = 0; k < PER_WARP; k++) {
    const long long t = t0 + warp * PER_WARP + k;
    if (t >= ntiles) break;
    int own = 0;
    unsigned w[WPL];
#pragma unroll
    for (int q = 0; q < WPL; q++) {
      w[q] = m[0][q];
#pragma unroll
      for (int kk = 1; kk < PER_WARP; kk++) w[q] = k == kk ? m[kk][q] : w[q];
      own += __popc(w[q]);
    }
    int sc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, sc, o);
      if (lane >= o) sc += a;
    }
    const int total = __shfl_sync(0xffffffffu, sc, 31);
    const long long base = t * UW_TILE;
    long long* out = idx_out + first[warp * PER_WARP + k];
    if (total <= UW_TILE / 8) {
      int at = sc - own;
#pragma unroll
      for (int q = 0; q < WPL; q++)
        for (unsigned b = w[q]; b; b &= b - 1) out[at++] = base + (lane * WPL + q) * 32 + __ffs(b) - 1;
    } else {
      for (int l = 0; l < 32; l++) {
        int at = __shfl_sync(0xffffffffu, sc - own, l);
#pragma unroll
        for (int q = 0; q < WPL; q++) {
          const unsigned b = __shfl_sync(0xffffffffu, w[q], l);
          if (b >> lane & 1u) out[at + __popc(b & ((1u << lane) - 1u))] = base + (l * WPL + q) * 32 + lane;
          at += __popc(b);
        }
      }
    }
  }
}

}  // namespace

extern "C" int mg_unweight(const double* w_dev, const double* r_dev, int64_t n, double w_max, int64_t* idx_out_dev,
                           int64_t* n_acc_dev, void* stream) {
  if (n < 0 || !(w_max > 0) || !n_acc_dev) return MG_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (n == 0) return cudaMemsetAsync(n_acc_dev, 0, sizeof(int64_t), s) == cudaSuccess ? MG_OK : MG_ERR_CUDA;
  if (!w_dev || !r_dev || !idx_out_dev) return MG_ERR_ARG;
  const long long ntiles = (n + UW_TILE - 1) / UW_TILE;
  if (ntiles > 0x7fffffffLL) return MG_ERR_ARG;
  // workspace: the tile counts (then offsets), then the accept bits
  long long* counts = nullptr;
  const size_t bytes = (size_t)ntiles * (sizeof(long long) + UW_WORDS * sizeof(unsigned));
  if (cudaMallocAsync(reinterpret_cast<void**>(&counts), bytes, s) != cudaSuccess) return MG_ERR_NOMEM;
  unsigned* bits = reinterpret_cast<unsigned*>(counts + ntiles);
  long long* acc = reinterpret_cast<long long*>(n_acc_dev);
  long long* idx = reinterpret_cast<long long*>(idx_out_dev);
  const unsigned blocks = (unsigned)((ntiles + WRITE_TILES - 1) / WRITE_TILES);
  tile_count_kernel<<<(unsigned)ntiles, UW_THREADS, 0, s>>>(w_dev, r_dev, n, w_max, counts, bits);
  if (ntiles > SUM_TILES) {
    tile_scan_kernel<<<1, SCAN_T, 0, s>>>(counts, ntiles, acc);
  }
  // the write pass may be set up while the pass before it drains (it waits for
  // that pass's memory before its first read)
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(UW_THREADS);
  cfg.stream = s;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  cudaError_t e1 = cudaLaunchKernelEx(&cfg, ntiles > SUM_TILES ? tile_write_kernel<true> : tile_write_kernel<false>,
                                      bits, counts, ntiles, acc, idx);
  const cudaError_t e3 = cudaGetLastError();
  if (e1 == cudaSuccess) e1 = e3;
  const cudaError_t e2 = cudaFreeAsync(counts, s);
  return (e1 == cudaSuccess && e2 == cudaSuccess) ? MG_OK : MG_ERR_CUDA;
}
