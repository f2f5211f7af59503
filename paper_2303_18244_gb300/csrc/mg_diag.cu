// mg_diag.cu -- FMA peak probe and per-kernel timing of a two-phase ME call
// (include/mg_diag.h).
#include <cuda_runtime.h>

#include <mutex>
#include <new>

#include "mg.h"
#include "mg_colour_tc.cuh"
#include "mg_diag.h"
#include "mg_runtime_internal.h"

namespace {

constexpr int CHAINS = 8;    // independent FMA chains per thread
constexpr int ITERS = 4096;  // loop trips per launch

template <typename R>
__global__ void __launch_bounds__(256) fma_probe(R* out, R a, R b) {
  R x[CHAINS];
  for (int c = 0; c < CHAINS; c++) x[c] = R(threadIdx.x + c);
#pragma unroll 4
  for (int i = 0; i < ITERS; i++)
#pragma unroll
    for (int c = 0; c < CHAINS; c++) x[c] = x[c] * a + b;
  R s = R(0);
  for (int c = 0; c < CHAINS; c++) s += x[c];
  if (s == R(-1.2345)) out[0] = s;  // keeps the loop alive, never taken
}

template <typename R>
int run(double* gflops) {
  int dev, sms;
  if (cudaGetDevice(&dev) != cudaSuccess) return MG_ERR_CUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return MG_ERR_CUDA;
  R* out = nullptr;
  cudaStream_t s;
  cudaEvent_t e0, e1;
  if (cudaMalloc(&out, sizeof(R)) != cudaSuccess) return MG_ERR_CUDA;
  cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int grid = 8 * sms, block = 256;
  const R a = R(0.999999), b = R(1e-7);
  fma_probe<R><<<grid, block, 0, s>>>(out, a, b);
  cudaEventRecord(e0, s);
  const int reps = sizeof(R) == 8 ? 1 : 10;
  for (int r = 0; r < reps; r++) fma_probe<R><<<grid, block, 0, s>>>(out, a, b);
  cudaEventRecord(e1, s);
  cudaError_t err = cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaStreamDestroy(s);
  cudaFree(out);
  if (err != cudaSuccess || ms <= 0.f) return MG_ERR_CUDA;
  const double fmas = double(reps) * grid * block * double(ITERS) * CHAINS;
  *gflops = 2.0 * fmas / (ms * 1e-3) / 1e9;
  return MG_OK;
}

// Tensor-core probe: one CTA per SM, one elected thread issues `iters`
// tcgen05.mma kind::f16 of M = 128, N = 128, K = 16 (FP16 operands in shared
// memory, one FP32 accumulator in TMEM) back to back, then commits; every
// thread waits (bounded) for the commit.  The large dynamic shared-memory
// request only keeps a second CTA off the SM.
constexpr int MMA_M = 128, MMA_N = 128, MMA_K = 16;
constexpr size_t MMA_PROBE_SMEM = 160 * 1024;

__global__ void __launch_bounds__(128) mma_probe(int iters, unsigned* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char dyn[];
  __shared__ __align__(128) unsigned char tiles[(MMA_M + MMA_N) * MMA_K * 2];  // A [M][K], B [N][K] FP16
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x;
  if (tid == 0) dyn[0] = 0;
  for (int i = tid; i < (int)(sizeof(tiles) / 4); i += 128)
    reinterpret_cast<uint32_t*>(tiles)[i] = 0x3c003c00u;  // FP16 1.0 in both halves
  if (tid == 0) {
    mg::mbar_init(&bar, 1);
    mg::fence_mbar_init();
  }
  if (tid < 32) {
    mg::tc::tmem_alloc(&tslot, MMA_N);
    mg::tc::tmem_relinquish();
  }
  mg::fence_proxy_async_smem();
  mg::tc::fence_before_sync();
  __syncthreads();
  mg::tc::fence_after_sync();
  const uint32_t tmem = tslot;
  if (tid == 0) {
    constexpr uint32_t idesc = mg::tc::idesc_f16(MMA_M, MMA_N);
    constexpr uint32_t SBO = (MMA_K / 8) * 128;  // 8-row groups of K-major core matrices
    const uint32_t a = mg::smem_u32(tiles), b = a + MMA_M * MMA_K * 2;
    const uint64_t ad = mg::tc::smem_desc(a, mg::tc::LBO, SBO), bd = mg::tc::smem_desc(b, mg::tc::LBO, SBO);
    for (int i = 0; i < iters; i++) mg::tc::mma_f16(tmem, ad, bd, idesc, i > 0 ? 1u : 0u);
    mg::tc::mma_commit(&bar);
  }
  if (!__syncthreads_and(mg::mbar_wait_bounded(&bar, 0, mg::WAIT_POLLS) ? 1 : 0)) {
    if (tid == 0) atomicOr(status, 1u);
    mg::mbar_wait_bounded(&bar, 0, mg::WAIT_POLLS);
  }
  mg::tc::fence_before_sync();
  __syncthreads();
  if (tid < 32) {
    mg::tc::fence_after_sync();
    mg::tc::tmem_dealloc(tmem, MMA_N);
  }
}

}  // namespace

extern "C" int mg_diag_mma_peak(double* tflops) {
  if (!tflops) return MG_ERR_ARG;
  int dev, sms;
  if (cudaGetDevice(&dev) != cudaSuccess) return MG_ERR_CUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return MG_ERR_CUDA;
  if (cudaFuncSetAttribute(mma_probe, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MMA_PROBE_SMEM) !=
      cudaSuccess)
    return MG_ERR_CUDA;
  unsigned* st = nullptr;
  if (cudaMalloc(&st, sizeof(unsigned)) != cudaSuccess) return MG_ERR_CUDA;
  cudaStream_t s;
  cudaEvent_t e0, e1;
  cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaMemsetAsync(st, 0, sizeof(unsigned), s);
  const int iters = 16384;
  mma_probe<<<sms, 128, MMA_PROBE_SMEM, s>>>(iters / 8, st);  // warm-up
  cudaEventRecord(e0, s);
  mma_probe<<<sms, 128, MMA_PROBE_SMEM, s>>>(iters, st);
  cudaEventRecord(e1, s);
  cudaError_t err = cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  unsigned flag = 0;
  if (err == cudaSuccess) err = cudaMemcpy(&flag, st, sizeof(unsigned), cudaMemcpyDeviceToHost);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaStreamDestroy(s);
  cudaFree(st);
  if (err != cudaSuccess || ms <= 0.f) return MG_ERR_CUDA;
  if (flag) return MG_ERR_TIMEOUT;
  *tflops = 2.0 * MMA_M * MMA_N * MMA_K * double(iters) * sms / (ms * 1e-3) / 1e12;
  return MG_OK;
}

extern "C" int mg_diag_fma_peak(int kind, double* gflops) {
  if (!gflops) return MG_ERR_ARG;
  if (kind == MG_DIAG_FP32) return run<float>(gflops);
  if (kind == MG_DIAG_FP64) return run<double>(gflops);
  return MG_ERR_ARG;
}

extern "C" int mg_diag_sigma_phases(mg_process* h, const double* momenta_dev, int64_t nevt, double* me_out_dev,
                                    void* stream, float* ms_first, float* ms_second, int* slices) {
  if (!h || nevt <= 0 || !momenta_dev || !me_out_dev) return MG_ERR_ARG;
  if (h->par.precision != MG_MIXED || !h->d->rows_mixed) return MG_ERR_ARG;
  if (reinterpret_cast<uintptr_t>(momenta_dev) & 15u) return MG_ERR_ARG;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != h->device) cudaSetDevice(h->device);
  // a mark before the first kernel and after every kernel of every slice
  const int64_t slice = mg::rows_slice(h->d->ncol, h->d->nhel, nevt), most = 1 + 2 * ((nevt + slice - 1) / slice);
  mg::PhaseMarks marks{most < (1 << 20) ? new (std::nothrow) cudaEvent_t[most] : nullptr, (int)most};
  int made = 0, rc = marks.ev ? MG_OK : MG_ERR_NOMEM;
  for (; marks.ev && made < marks.max; made++)
    if (cudaEventCreate(&marks.ev[made]) != cudaSuccess) {
      rc = MG_ERR_CUDA;
      break;
    }
  const cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (rc == MG_OK) {
    std::lock_guard<std::mutex> lk(h->lock);
    rc = mg_launch_sigma_locked(h, momenta_dev, nevt, me_out_dev, s, &marks);
  }
  if (rc == MG_OK && cudaStreamSynchronize(s) != cudaSuccess) rc = MG_ERR_CUDA;
  float t1 = 0.f, t2 = 0.f;
  if (rc == MG_OK) {
    for (int i = 0; i + 2 < marks.n; i += 2) {
      float a = 0.f, b = 0.f;
      if (cudaEventElapsedTime(&a, marks.ev[i], marks.ev[i + 1]) != cudaSuccess ||
          cudaEventElapsedTime(&b, marks.ev[i + 1], marks.ev[i + 2]) != cudaSuccess) {
        rc = MG_ERR_CUDA;
        break;
      }
      t1 += a;
      t2 += b;
    }
  }
  for (int i = 0; i < made; i++) cudaEventDestroy(marks.ev[i]);
  delete[] marks.ev;
  if (prev >= 0 && prev != h->device) cudaSetDevice(prev);
  if (rc != MG_OK) return rc;
  if (ms_first) *ms_first = t1;
  if (ms_second) *ms_second = t2;
  if (slices) *slices = (marks.n - 1) / 2;
  return MG_OK;
}

static_assert(MG_DIAG_WAIT_POLLS == mg::WAIT_POLLS, "default bound of the device waits");

extern "C" int mg_diag_set_wait_polls(mg_process* h, uint32_t polls) {
  if (!h) return MG_ERR_ARG;
  std::lock_guard<std::mutex> lk(h->lock);
  h->kp.polls = polls;
  return MG_OK;
}
