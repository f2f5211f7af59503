// mg_phasespace.cu -- flat phase-space momenta generated on the device
// (mg_rambo in include/mg.h).
//
// The paper (Sect. 2) identifies the host-side random-number -> momenta step
// of the event generator as the next serial part to move to the GPU once the
// matrix elements are fast.  This kernel produces the same event stream as
// the host input module: Philox4x64-10 (Salmon et al., SC'11) with key
// (seed, 0) and counter (event, final-state slot, 0, 0), uniforms
// ((w >> 11) + 0.5) 2^-53, then RAMBO (Kleiss, Stirling, Ellis 1986) at fixed
// sqrt(s): isotropic massless momenta, conformal map to the centre-of-mass
// frame, removal of the residual 3-momentum, and the common 3-momentum scale
// that puts every final state on its mass shell.  One event per thread.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "mg.h"
#include "mg_runtime_internal.h"

namespace {

__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
  const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
  const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int r = 0; r < 10; r++) {
    const uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
    const uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
    const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
    k0 += W0;
    k1 += W1;
  }
}

struct PSArgs {
  double sqrt_s;
  uint64_t seed;
  long long first_event, nevt;
  double unit;  // the power of two with sqrt_s / unit in [1, 2)
  double rs;    // sqrt_s / unit, exact
  double mass;  // of the first two final states / unit, exact
  double xi0;   // sqrt(1 - (sum of the masses / sqrt_s)^2): start of the scale
};

// One event per thread, everything in registers (NF final states, a template
// parameter).  The FP64 pipe bounds it (16 cycles per warp instruction and
// SM): about 530 FP64 instructions per event for NF = 4.  The map works on
// momenta in units of the generated mass M; their scale x onto the mass shells
// solves f(x) = sum_j sqrt(m_j^2 + x^2 |p_j|^2) - sqrt_s = 0:
//   - Newton in FP32 first, which leaves about 1e-7 (NF > 2; for two equal
//     masses the start is the solution up to the rounding of the map);
//   - then FP64 steps with the FP32 derivative, each of which gains those
//     seven digits again; a step below 1e-9 of x leaves less than the rounding
//     of f, so two steps are usual (at most 60).
// Masses, sqrt_s and x are in units of a power of two, so that nothing is
// rounded before sqrt_s and the masses cancel in f: in units of sqrt_s itself
// the gluons lost digits near threshold (energies off by 1e-8 at sqrt_s = 2 m_t
// (1 + 1e-9), 1e-5 at 1e-12; by 1e-10 and 1e-13 now, five final states).
// Against 113-bit values, mean error of a component over its energy at four
// final states: 9.0e-17 (9.1e-17 in units of sqrt_s, 11.9e-17 with Newton in
// FP64 alone, until a step fell below 1e-16 of x: as many iterations as the
// slowest lane of the warp needed to meet a bound below the rounding of f, up to
// all 60; 524288 events 5.66 ms).
template <int NF, bool ALIGNED>
__global__ void __launch_bounds__(128) rambo_kernel(PSArgs a, double* __restrict__ out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= a.nevt) return;
  const long long ev = a.first_event + i;
  double q[NF][4];
#pragma unroll
  for (int j = 0; j < NF; j++) {
    uint64_t c[4] = {(uint64_t)ev, (uint64_t)j, 0ull, 0ull};
    philox4x64_10(c, a.seed, 0ull);
    // u = v 2^-53 with v = (w >> 11) + 0.5; scaling by powers of two is exact
    const double v0 = (double)(c[0] >> 11) + 0.5, v1 = (double)(c[1] >> 11) + 0.5;
    const double v2 = (double)(c[2] >> 11) + 0.5, v3 = (double)(c[3] >> 11) + 0.5;
    const double ct = ::fma(v0, 0x1.0p-52, -1.0);  // 2 u0 - 1
    const double st = sqrt(fmax(0.0, ::fma(-ct, ct, 1.0)));
    double sn, cs;
    sincospi(v1 * 0x1.0p-52, &sn, &cs);  // azimuth 2 pi u1
    const double q0 = -log(v2 * v3 * 0x1.0p-106);
    const double qt = q0 * st;
    q[j][0] = q0;
    q[j][1] = qt * cs;
    q[j][2] = qt * sn;
    q[j][3] = q0 * ct;
  }
  double Q[4] = {0, 0, 0, 0};
#pragma unroll
  for (int j = 0; j < NF; j++)
#pragma unroll
    for (int mu = 0; mu < 4; mu++) Q[mu] += q[j][mu];
  const double M = sqrt(Q[0] * Q[0] - (Q[1] * Q[1] + Q[2] * Q[2] + Q[3] * Q[3]));
  const double im = 1.0 / M;
  const double b[3] = {-Q[1] * im, -Q[2] * im, -Q[3] * im};
  const double aa = 1.0 / ::fma(Q[0], im, 1.0);
  // 3-momenta in the centre-of-mass frame, in units of M
  double R3[3] = {0, 0, 0};
#pragma unroll
  for (int j = 0; j < NF; j++) {
    const double bq = b[0] * q[j][1] + b[1] * q[j][2] + b[2] * q[j][3];
    const double w = ::fma(aa, bq, q[j][0]);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      q[j][k + 1] = ::fma(b[k], w, q[j][k + 1]);
      R3[k] += q[j][k + 1];
    }
  }
  // the map's residual 3-momentum removed evenly
  double p2[NF], root[NF];
  float p2f[NF];
  double S = 0.0;  // sum of the massless |p|
#pragma unroll
  for (int j = 0; j < NF; j++) {
#pragma unroll
    for (int k = 0; k < 3; k++) q[j][k + 1] = ::fma(R3[k], -1.0 / NF, q[j][k + 1]);
    p2[j] = q[j][1] * q[j][1] + q[j][2] * q[j][2] + q[j][3] * q[j][3];
    p2f[j] = (float)p2[j];
    if (j >= 2) {
      root[j] = sqrt(p2[j]);
      S += root[j];
    }
  }
  // common scale onto the mass shells
  const double x0 = a.xi0 * im * a.rs, m2 = a.mass * a.mass;
  const float Sf = (float)S;
  double x = x0;
  if constexpr (NF > 2) {
    const float m2f = (float)m2, rsf = (float)a.rs;
    float xf = (float)x0, dinv = 0.f;
#pragma unroll 1
    for (int it = 0; it < 6; it++) {
      float f = fmaf(xf, Sf, -rsf), df = Sf;
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const float r = rsqrtf(fmaf(xf * xf, p2f[j], m2f));
        f = fmaf(fmaf(xf * xf, p2f[j], m2f), r, f);
        df = fmaf(xf * p2f[j], r, df);
      }
      dinv = 1.f / df;
      xf = fmaf(-f, dinv, xf);
    }
    // else FP32 did not converge
    if (xf > 0.f && xf < 1e30f && dinv > 0.f && dinv < 1e30f) x = (double)xf;
  }
#pragma unroll 1
  for (int it = 0; it < 60; it++) {
    double e[2], df;
    const double x2 = x * x;
    const float xf = (float)x;
    float dm = Sf;
#pragma unroll
    for (int j = 0; j < 2; j++) {
      e[j] = sqrt(::fma(x2, p2[j], m2));
      dm = fmaf(xf * p2f[j], 1.f / (float)e[j], dm);
    }
    const double f = ::fma(x, S, (e[0] - a.rs) + e[1]);
    df = (double)(1.f / dm);
    if (!(dm > 1e-30f) || !(dm < 1e30f)) {  // outside the FP32 range: the derivative in FP64
      df = S;
      for (int j = 0; j < 2; j++) df += x * p2[j] / sqrt(::fma(x2, p2[j], m2));
      df = 1.0 / df;
    }
    const double step = f * df;
    x -= step;
    if (fabs(step) <= 1e-9 * fabs(x)) break;
  }
  double* o = out + i * (long long)(NF + 2) * 4;
  auto put = [&](int slot, double e, double x, double y, double z) {
    double* t = o + 4 * slot;
    if constexpr (ALIGNED) {
      reinterpret_cast<double2*>(t)[0] = make_double2(e, x);
      reinterpret_cast<double2*>(t)[1] = make_double2(y, z);
    } else {
      t[0] = e;
      t[1] = x;
      t[2] = y;
      t[3] = z;
    }
  };
  const double E = 0.5 * a.sqrt_s, scale = x * a.unit;
  put(0, E, 0.0, 0.0, E);
  put(1, E, 0.0, 0.0, -E);
#pragma unroll
  for (int j = 0; j < NF; j++)
    // two equal masses: half of sqrt_s each
    put(2 + j, NF == 2 ? E : (j < 2 ? a.unit * sqrt(::fma(x * x, p2[j], m2)) : scale * root[j]), scale * q[j][1],
        scale * q[j][2], scale * q[j][3]);
}

template <int NF>
void launch_rambo(const PSArgs& a, double* out, cudaStream_t s) {
  const unsigned grid = (unsigned)((a.nevt + 127) / 128);
  if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0)
    rambo_kernel<NF, true><<<grid, 128, 0, s>>>(a, out);
  else
    rambo_kernel<NF, false><<<grid, 128, 0, s>>>(a, out);
}

}  // namespace

extern "C" int mg_rambo(const mg_process* h, double sqrt_s, uint64_t seed, int64_t first_event, int64_t nevt,
                        double* momenta_dev, void* stream) {
  if (!h || nevt < 0 || first_event < 0 || !(sqrt_s > 0)) return MG_ERR_ARG;
  if (nevt == 0) return MG_OK;
  if (!momenta_dev) return MG_ERR_ARG;
  PSArgs a{};
  a.sqrt_s = sqrt_s;
  a.seed = seed;
  a.first_event = first_event;
  a.nevt = nevt;
  const int nf = h->d->npar - 2;
  if (nf < 2 || nf > 5) return MG_ERR_ARG;
  // final-state masses: the top pair of g g -> t t~ (+ gluons); massless leptons
  const bool tops = std::strcmp(h->d->tag, "eemumu") != 0;
  const double mass = tops ? h->par.mt : 0.0;
  if (2.0 * mass >= sqrt_s) return MG_ERR_ARG;
  a.unit = std::ldexp(1.0, std::ilogb(sqrt_s));
  a.rs = sqrt_s / a.unit;
  a.mass = mass / a.unit;
  a.xi0 = std::sqrt(1.0 - (2.0 * mass / sqrt_s) * (2.0 * mass / sqrt_s));
  int prev = -1, dev = h->device;
  cudaGetDevice(&prev);
  if (prev != dev) cudaSetDevice(dev);
  const cudaStream_t cs = static_cast<cudaStream_t>(stream);
  if (nf == 2)
    launch_rambo<2>(a, momenta_dev, cs);
  else if (nf == 3)
    launch_rambo<3>(a, momenta_dev, cs);
  else if (nf == 4)
    launch_rambo<4>(a, momenta_dev, cs);
  else
    launch_rambo<5>(a, momenta_dev, cs);
  const cudaError_t e = cudaGetLastError();
  if (prev >= 0 && prev != dev) cudaSetDevice(prev);
  return e == cudaSuccess ? MG_OK : MG_ERR_CUDA;
}
