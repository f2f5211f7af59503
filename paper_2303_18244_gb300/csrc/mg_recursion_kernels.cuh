// mg_recursion_kernels.cuh -- |M|^2 kernels of the helicity-shared recursion.
//
// A group of T threads owns an event at a time and keeps its store in shared
// memory; a CTA runs up to EV groups side by side, stage by stage, over tiles
// of consecutive events (persistent grid; the next tile's momenta arrive by a
// bulk copy while the current tile is worked on).  The block barrier between
// the stages keeps all warps of an SM on the same stretch of code: the program
// is several times larger than the instruction caches close to the schedulers,
// and warps that run it at their own pace fetch it each for themselves.
#pragma once

#include "mg_colour_tc.cuh"
#include "mg_kernels.cuh"
#include "mg_recursion.cuh"

namespace mg {

// Threads per event and events per CTA (register and shared-memory limits).
template <class P, typename R>
struct RecShape {
  static constexpr bool f32 = sizeof(R) == 4;
  // Thread = gluon helicities x top spin, both antitop spins; or thread =
  // helicity: five gluons (registers), and four in FP64, where the flows of one
  // helicity leave room for 12 warps (six events, the late vectors over others)
  // instead of 4, and 12 keep the FP64 pipe busier: 32749 events 11.3 -> 9.97 ms
  // (8 / 10 warps 10.2 / 10.5), though 0.3 KB a thread are spilled.  In FP32 the
  // antitop spins share the loads of the rows: 4.76 ms for 524288 events against
  // 5.8 / 5.5 / 5.4 ms with a thread per helicity and 24 / 20 / 16 warps.  Three gluons, FP64, 65536 events: 2.88
  // against 2.92 .. 3.6 ms.
  static constexpr int T = P::N == 5 || (P::N == 4 && !f32) ? P::NHEL : 1 << (P::N + 1);
  // warps of a CTA, a multiple of the four schedulers.  Measured, 524288 events
  // of four gluons in FP32 (with every current computed, before half of them
  // came by conjugation): 5 / 8 / 10 / 12 warps 9.6 / 6.9 / 7.2 / 6.6 ms; 12
  // fill the shared memory.  Several smaller CTAs per SM, which could overlap
  // one's FP64 set-up with another's closings, give nothing: 1 x 12 / 2 x 6 /
  // 3 x 4 warps 4.89 / 4.97 / 5.03 ms.  Three gluons 8 / 12 warps 0.19 / 0.23 ms
  // per 65536.
  static constexpr int WARPS = P::N == 4 ? 12 : f32 ? 8 : 4;
  static constexpr int EV = WARPS * 32 / T;
  // Five gluons in FP64: one event fills the shared memory, and its 4 warps leave
  // the FP64 pipe idle for a quarter of the time.  As many helper threads share
  // the lists of currents and half of the colour form: 4096 events 18.4 -> 16.6 ms.
  static constexpr int HELP = P::N == 5 && !f32 ? T : 0;
  static constexpr int MAXT = T * EV + HELP;
};

template <class P, typename R>
struct RecLayout {
  using ST = rec::Store<R, P::N, P::template NVEC<R>>;
  static constexpr int T = RecShape<P, R>::T, EV = RecShape<P, R>::EV;
  static constexpr size_t r128(size_t b) { return (b + 127) / 128 * 128; }
  static constexpr size_t mom_bytes = size_t(P::NPAR) * 4 * sizeof(double);  // per event
  static constexpr size_t red_off = 16;                                       // after the mbarrier: partial sums
  static constexpr size_t mom_off = r128(red_off + RecShape<P, R>::MAXT / 32 * sizeof(double));
  static constexpr size_t store_off = mom_off + r128(EV * mom_bytes);
  static constexpr size_t store_bytes = ST::stride;
  static constexpr size_t base_bytes = store_off + EV * store_bytes;
};

// Sum over the T threads of the event's group, the same value in every thread
// (every thread of the CTA calls it; `red`: one slot per warp).
template <int T, typename A>
__device__ __forceinline__ A rec_group_sum(A v, A* red) {
#pragma unroll
  for (int o = (T < 32 ? T : 32) / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if constexpr (T > 32) {
    constexpr int NW = T / 32;
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) red[warp] = v;
    __syncthreads();
    v = A(0);
#pragma unroll
    for (int w = 0; w < NW; w++) v += red[warp / NW * NW + w];
    __syncthreads();
  }
  return v;
}

// reduce-scatter of N <= 32 values over a warp: lane k < N returns the sum
// over the lanes of their v[k] (31 additions instead of 5 per value)
template <int N>
__device__ __forceinline__ double warp_scatter_sum(const double (&v)[N]) {
  const int lane = threadIdx.x & 31;
  double x[32];
#pragma unroll
  for (int k = 0; k < 32; k++) x[k] = k < N ? v[k < N ? k : 0] : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < o; k++) {
      const double mine = up ? x[k + o] : x[k], other = up ? x[k] : x[k + o];
      x[k] = mine + __shfl_xor_sync(0xffffffffu, other, o);
    }
  }
  return x[0];
}

template <int N>
using Count = std::integral_constant<int, N>;

// The event loop; blockDim.x = T * (events per tile) + HELP.  body(store, e, valid)
// runs with the currents complete; groups past the last event repeat it.
template <class P, typename R, typename D, class BODY>
__device__ __forceinline__ void rec_events(unsigned char* smem, const double* __restrict__ mom, long long nevt,
                                           const KParams& kp, unsigned* status, const BODY& body) {
  using LY = RecLayout<P, R>;
  using ST = typename LY::ST;
  constexpr int T = LY::T;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
  constexpr bool help = RecShape<P, R>::HELP > 0;  // one event per tile
  const int tid = threadIdx.x, nt = blockDim.x, ge = help ? 0 : tid / T;
  const int per = help ? 1 : nt / T;
  const ST all(smem + LY::store_off), st = all.at(ge);
  const R kr[2] = {R(kp.v[0]), R(kp.v[1])};
  const long long step = (long long)gridDim.x * per;
  auto fetch = [&](long long e0) {
    const uint32_t bytes = (uint32_t)((nevt - e0 < per ? nevt - e0 : per) * LY::mom_bytes);
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, bytes);
    bulk_g2s(smem + LY::mom_off, mom + e0 * P::NPAR * 4, bytes, bar);
  };
  const long long first = (long long)blockIdx.x * per;
  if (first >= nevt) return;
  if (tid == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    fetch(first);
  }
  __syncthreads();
  uint32_t phase = 0;
  for (long long e0 = first; e0 < nevt; e0 += step) {
    // bounded wait, its outcome uniform across the CTA
    if (!__syncthreads_and(mbar_wait_bounded(bar, phase, kp.polls) ? 1 : 0)) {
      if (tid == 0) atomicOr(status, ST_TMA_TIMEOUT);
      mbar_wait_bounded(bar, phase, WAIT_POLLS);  // no copy is left in flight
      return;
    }
    phase ^= 1u;
    const bool valid = e0 + ge < nevt;
    const long long e = valid ? e0 + ge : nevt - 1;
    const double* tile = reinterpret_cast<const double*>(smem + LY::mom_off);
    const int last = (int)(nevt - e0 < per ? nevt - e0 : per) - 1;
    auto momenta = [&](int ev) { return tile + (ev < last ? ev : last) * P::NPAR * 4; };
    // the set-up's tasks of all events of the tile, like the lists of currents
    auto each = [&](auto count, const auto& task) {
      constexpr int n = decltype(count)::value;
      for (int t = tid; t < n * per; t += nt) task(t / n, t % n);
    };
    constexpr bool pairs = sizeof(R) == 4 && sizeof(D) == 8;
    each(Count<P::NPAR * 4>{}, [&](int ev, int t) { all.at(ev).momenta()[t] = rec::narrow<R>(momenta(ev)[t]); });
    if constexpr (pairs)
      each(Count<(P::N + 1) * (P::N + 2) / 2>{},
           [&](int ev, int t) { rec::setup_pair<P>(all.at(ev).pairs(), momenta(ev), kp.v, t); });
    __syncthreads();
    each(Count<ST::NSUB>{}, [&](int ev, int m) { rec::setup_momenta<P, R>(all.at(ev), all.at(ev).momenta(), m); });
    each(Count<P::N + 2>{}, [&](int ev, int l) { rec::setup_leg<P, R>(all.at(ev), all.at(ev).momenta(), kr, l); });
    if constexpr (pairs)
      each(Count<ST::NSUB>{}, [&](int ev, int m) { rec::setup_coef_pairs<P>(all.at(ev), all.at(ev).pairs(), kp.v, m); });
    else
      each(Count<2 * ST::NSUB>{},
           [&](int ev, int c) { rec::setup_coef<P, R, D>(all.at(ev), momenta(ev), kp.v, c); });
    __syncthreads();
    if (tid == 0 && e0 + step < nevt) fetch(e0 + step);  // the momenta are consumed
    P::template currents<R>(all, kr, tid, nt, [] { __syncthreads(); }, per);
    __syncthreads();
    body(st, e, valid);
    __syncthreads();  // the store is rewritten by the next tile
  }
}

// Bit b: the helicity of gluon bits hg, top spin s, antitop spin b is listed.
template <class P>
__device__ __forceinline__ unsigned rec_good_bits(const int* __restrict__ hels, int nhel, int hg, int s) {
  unsigned g = 0;
  const int h0 = P::helicity(hg, s, 0), h1 = P::helicity(hg, s, 1);
  for (int i = 0; i < nhel; i++) {
    const int h = __ldg(hels + i);
    g |= (h == h0 ? 1u : 0u) | (h == h1 ? 2u : 0u);
  }
  return g;
}

// The choice of select_kernel from the values mh[helicity] and the flow
// weights wk[flow] of one event (one thread each).
__device__ __forceinline__ int rec_choose_helicity(const double* mh, const int* __restrict__ hels, int nhel,
                                                   double th) {
  int sel = -1, last = 0;
  double cum = 0.0;
  for (int ih = 0; ih < nhel; ih++) {
    const double v = mh[__ldg(hels + ih)];
    if (v > 0.0) last = ih;
    cum += v;
    if (sel < 0 && cum > th && v > 0.0) sel = ih;
  }
  return __ldg(hels + (sel < 0 ? last : sel));
}
template <int NCOL>
__device__ __forceinline__ int rec_choose_flow(const double* wk, double r) {
  double wt = 0.0, cum = 0.0;
  for (int k = 0; k < NCOL; k++) wt += wk[k];
  const double tc = r * wt;
  int sel = -1, last = 0;
  for (int k = 0; k < NCOL; k++) {
    if (wk[k] > 0.0) last = k;
    cum += wk[k];
    if (sel < 0 && cum > tc && wk[k] > 0.0) sel = k;
  }
  return sel < 0 ? last : sel;
}

enum RecMode {
  REC_SIGMA,       // |M|^2
  REC_PAPER,       // the same, colour form in FP32 on FP64 flows
  REC_HELICITIES,  // |M_h|^2 / IDEN of every helicity
  REC_SELECT       // |M|^2 with the helicity and colour choice
};

// Up to four gluons: the flows of a helicity fit in registers.  A thread has a
// helicity of its own, or both antitop spins: at once in FP32 (they share every
// load that does not depend on the antitop), one after the other in FP64.
template <class P, typename R, typename D, typename A, RecMode MODE>
__global__ void __launch_bounds__(RecShape<P, R>::T* RecShape<P, R>::EV, 1) rec_kernel(LaunchArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  using LY = RecLayout<P, R>;
  constexpr int T = LY::T, NW = T > 32 ? T / 32 : 1;
  constexpr bool own = T == P::NHEL;  // a helicity of one's own
  constexpr int NB = sizeof(R) == 4 && !own ? 2 : 1;
  static_assert(own || NB == 2 || !P::LATE, "every helicity's first closings come before the late vectors");
  const int gt = threadIdx.x % T, ge = threadIdx.x / T;
  const int hg = gt & ((1 << P::N) - 1), s = gt >> P::N & 1;
  unsigned good = 0;
  if constexpr (MODE != REC_HELICITIES) good = rec_good_bits<P>(a.hels, a.nhel, hg, s);
  // choice: the helicities' values and the flow weights (of each warp) of each event
  double* mh = reinterpret_cast<double*>(smem + LY::base_bytes) + ge * (P::NHEL + NW * P::NCOL);
  double* wk = mh + P::NHEL;
  rec_events<P, R, D>(smem, a.mom, a.nevt, a.kp, a.status, [&](const auto& st, long long e, bool valid) {
    constexpr double norm = 1.0 / (P::IDEN * P::CDEN);
    A part = A(0);
    [[maybe_unused]] double w = 0.0;
    const auto close = [&](const int b0) {
      cx<R> f[NB][P::NCOL];
      P::template flows_open<R, NB>(st, hg, s, b0, f);
      if constexpr (P::LATE) {  // takes the space of the vectors just closed
        __syncthreads();
        P::template late<R>(st.at(-ge), threadIdx.x, blockDim.x, blockDim.x / T);
        __syncthreads();
      }
      P::template flows_block<R, NB>(st, hg, s, b0, f);
#pragma unroll
      for (int ib = 0; ib < NB; ib++) {
        R v;
        if constexpr (MODE == REC_PAPER)
          v = (R)P::colour_form_paper(f[ib]);
        else
          v = P::template colour_form<R>(f[ib]);
        const bool in = (good >> (b0 + ib) & 1) != 0;
        if constexpr (MODE == REC_HELICITIES) {
          if (valid) a.out[e * P::NHEL + P::helicity(hg, s, b0 + ib)] = (double)v * norm;
        } else if (in) {
          part += (A)v;
        }
        if constexpr (MODE == REC_SELECT) {
          static_assert(P::NCOL <= (T < 32 ? T : 32), "lane k of the group sums flow k");
          mh[P::helicity(hg, s, b0 + ib)] = (double)v;
          double sq[P::NCOL];
#pragma unroll
          for (int k = 0; k < P::NCOL; k++)
            sq[k] = in ? f[ib][k].re * f[ib][k].re + f[ib][k].im * f[ib][k].im : 0.0;
          if constexpr (T >= 32) {
            w += warp_scatter_sum(sq);
          } else {
#pragma unroll
            for (int k = 0; k < P::NCOL; k++) {
              const double t = rec_group_sum<T>(sq[k], static_cast<double*>(nullptr));
              if (gt == k) w += t;
            }
          }
        }
      }
    };
    if constexpr (own) {
      close(gt >> (P::N + 1));
    } else {
#pragma unroll 1
      for (int b0 = 0; b0 < 2; b0 += NB) close(b0);
    }
    if constexpr (MODE != REC_HELICITIES) {
      const A acc = rec_group_sum<T>(part, reinterpret_cast<A*>(smem + LY::red_off));
      if (gt == 0 && valid) a.out[e] = (double)(acc * A(norm));
      if constexpr (MODE == REC_SELECT) {
        const int lane = gt & 31;
        if (lane < P::NCOL) wk[(gt >> 5) * P::NCOL + lane] = w;
        __syncthreads();
        if (gt < P::NCOL) {
#pragma unroll
          for (int q = 1; q < NW; q++) w += wk[q * P::NCOL + gt];
          wk[gt] = w;
          if (a.colw_out && valid) a.colw_out[e * P::NCOL + gt] = w;
        }
        __syncwarp();
        if (gt == 0 && valid) a.hel_out[e] = rec_choose_helicity(mh, a.hels, a.nhel, a.rnd[2 * e] * (double)acc);
        if (gt == 1 && valid) a.col_out[e] = rec_choose_flow<P::NCOL>(wk, a.rnd[2 * e + 1]);
      }
    }
  });
}

// Five gluons: the flows of the thread's helicity through get(k) and
// put(k, value), in the emitted order.
template <class P, typename R, class ST, class GET, class PUT>
__device__ __forceinline__ void rec_cta_flows(const ST& st, const KParams& kp, const GET& get, const PUT& put) {
  constexpr bool help = RecShape<P, R>::HELP > 0;
  const int gt = threadIdx.x % P::NHEL, ge = help ? 0 : threadIdx.x / P::NHEL;
  const bool main = !help || threadIdx.x < P::NHEL;
  const int hg = gt & ((1 << P::N) - 1), s = gt >> P::N & 1, b = gt >> (P::N + 1);
  if (main) P::template closings<R, 1>(st, hg, s, b, [&](int, int k, cx<R> v) { put(k, v); });
  __syncthreads();
  const R kr[2] = {R(kp.v[0]), R(kp.v[1])};
  P::template late<R>(st.at(-ge), kr, threadIdx.x, blockDim.x, help ? 1 : blockDim.x / P::NHEL);
  __syncthreads();
  if (main)
    P::template all_flows<R, 1>(
        st, hg, s, b, [&](int, int k) { return get(k); }, [&](int, int k, cx<R> v) { put(k, v); });
}
template <class P>
__device__ __forceinline__ int rec_cta_helicity() {
  const int gt = threadIdx.x % P::NHEL;
  return P::helicity(gt & ((1 << P::N) - 1), gt >> P::N & 1, gt >> (P::N + 1));
}

// Five gluons, one kernel; the thread's flows wait in local memory for the
// colour form.
template <class P, typename R, typename D, typename A, RecMode MODE>
__global__ void __launch_bounds__(RecShape<P, R>::MAXT, 1) rec_cta_kernel(LaunchArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  using LY = RecLayout<P, R>;
  constexpr int T = LY::T, NW = T / 32;
  constexpr bool help = RecShape<P, R>::HELP > 0;
  const int gt = threadIdx.x % T, ge = help ? 0 : threadIdx.x / T, lane = threadIdx.x & 31, warp = gt >> 5;
  const bool main = !help || threadIdx.x < T;
  const int hel = rec_cta_helicity<P>();
  bool good = false;
  if constexpr (MODE != REC_HELICITIES)
    for (int i = 0; i < a.nhel; i++) good |= __ldg(a.hels + i) == hel;
  rec_events<P, R, D>(smem, a.mom, a.nevt, a.kp, a.status, [&](const auto& st, long long e, bool valid) {
    constexpr double norm = 1.0 / (P::IDEN * P::CDEN);
    cx<R> fl[P::NCOL];
    rec_cta_flows<P, R>(
        st, a.kp, [&](int k) { return fl[k]; }, [&](int k, cx<R> v) { fl[k] = v; });
    if constexpr (help && MODE == REC_SIGMA) {
      // two of the four colour blocks go to the helper of the helicity, through
      // the store's space once every thread has its flows
      constexpr int NQ = P::NBLOCK;
      static_assert(2 * NQ * T * sizeof(cx<R>) <= LY::store_bytes, "two blocks of every helicity");
      cx<R>* x = reinterpret_cast<cx<R>*>(smem + LY::store_off) + gt;
      cx<R> f[NQ];
      __syncthreads();
      if (main) {
        P::template colour_blocks<R>(fl);
        P::template colour_block<2, R>(fl, f);
#pragma unroll
        for (int q = 0; q < NQ; q++) x[q * T] = f[q];
        P::template colour_block<3, R>(fl, f);
#pragma unroll
        for (int q = 0; q < NQ; q++) x[(NQ + q) * T] = f[q];
      }
      __syncthreads();
      A v = A(0);
#pragma unroll 1
      for (int c = 0; c < 2; c++) {
        if (!main) {
#pragma unroll
          for (int q = 0; q < NQ; q++) f[q] = x[(c * NQ + q) * T];
        } else if (c == 0) {
          P::template colour_block<0, R>(fl, f);
        } else {
          P::template colour_block<1, R>(fl, f);
        }
        v += (A)P::template block_value<R>(main ? c : 2 + c, f);
      }
      const A acc = rec_group_sum<2 * T>(good ? v : A(0), reinterpret_cast<A*>(smem + LY::red_off));
      if (threadIdx.x == 0) a.out[e] = (double)(acc * A(norm));
      return;
    }
    // the choice's values take the store's space once every thread has its flows
    double* mh = reinterpret_cast<double*>(smem + LY::store_off + ge * LY::store_bytes);
    double* wp = mh + P::NHEL;       // [warp][flow]
    double* wl = wp + NW * P::NCOL;  // sums, flows in lexicographic order
    if constexpr (MODE == REC_SELECT) {  // flow weights: the colour form overwrites the flows
      __syncthreads();
      static_assert(P::NCOL % 24 == 0, "chunks of 24 flows");
      for (int k0 = 0; k0 < P::NCOL; k0 += 24) {
        double sq[24];
#pragma unroll
        for (int k = 0; k < 24; k++)
          sq[k] = good ? fl[k0 + k].re * fl[k0 + k].re + fl[k0 + k].im * fl[k0 + k].im : 0.0;
        const double w = warp_scatter_sum(sq);
        if (main && lane < 24) wp[warp * P::NCOL + k0 + lane] = w;
      }
    }
    A v = A(0);
    if (main) {
      if constexpr (MODE == REC_PAPER)
        v = (A)P::colour_form_paper(fl);
      else
        v = (A)P::template colour_form<R>(fl);
    }
    valid = valid && main;
    if constexpr (MODE == REC_HELICITIES) {
      if (valid) a.out[e * P::NHEL + hel] = (double)v * norm;
    } else {
      if constexpr (MODE == REC_SELECT)
        if (main) mh[hel] = (double)v;
      const A acc = rec_group_sum<T>(good ? v : A(0), reinterpret_cast<A*>(smem + LY::red_off));
      if (gt == 0 && valid) a.out[e] = (double)(acc * A(norm));
      if constexpr (MODE == REC_SELECT) {
        if (main && gt < P::NCOL) {
          double w = 0.0;
          for (int q = 0; q < NW; q++) w += wp[q * P::NCOL + gt];
          wl[P::lex_flow(gt)] = w;
          if (a.colw_out && valid) a.colw_out[e * P::NCOL + P::lex_flow(gt)] = w;
        }
        __syncthreads();
        if (gt == 0 && valid) a.hel_out[e] = rec_choose_helicity(mh, a.hels, a.nhel, a.rnd[2 * e] * (double)acc);
        if (gt == 32 && valid) a.col_out[e] = rec_choose_flow<P::NCOL>(wl, a.rnd[2 * e + 1]);
      }
    }
  });
}

// Phase 1 of the mixed path of five gluons: the FP32 flows of every helicity,
// J[event][flow][thread's helicity] (coalesced).
template <class P>
__global__ void __launch_bounds__(RecShape<P, float>::T* RecShape<P, float>::EV, 1)
    rec_flows_kernel(const double* __restrict__ mom, long long nevt, float2* __restrict__ J, KParams kp,
                     unsigned* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem[];
  rec_events<P, float, double>(smem, mom, nevt, kp, status, [&](const auto& st, long long e, bool valid) {
    // a group past the last event leaves that event's row to its own group
    float2* row = J + e * (long long)(P::NCOL * P::NHEL) + threadIdx.x % P::NHEL;
    rec_cta_flows<P, float>(
        st, kp,
        [&](int k) {
          const float2 v = valid ? row[k * P::NHEL] : make_float2(0.f, 0.f);
          return cx<float>{v.x, v.y};
        },
        [&](int k, cx<float> v) {
          if (valid) row[k * P::NHEL] = make_float2(v.re, v.im);
        });
  });
}

// Phase 2: one CTA per event at a time, TMEM lane = helicity: FP16 hi/lo
// operand tiles of the rows, D = A K for Re, then Im, sum_k J_k D_k per row with
// the FP32 flows, and the rows of the list summed in FP64.  The loads of an
// event (123 KB from HBM) bound it: one part at a time keeps two CTAs on an SM
// (97 KB of shared memory and half of the tensor memory each), so that one
// loads while the other converts and contracts.
template <class P>
__global__ void __launch_bounds__(128, 2)
    rec_colour_tc_kernel(const float2* __restrict__ J, long long nevt, double* __restrict__ me,
                         const int* __restrict__ hels, int nhel, const uint4* __restrict__ ctile,
                         unsigned* __restrict__ status, uint32_t polls) {
  using LY = LayoutRows<P>;
  constexpr int NT = 128, K = LY::K, N = LY::N;
  static_assert(P::NHEL == NT && 2 * N <= 256, "a row per helicity, two accumulators of N columns");
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* mma_bar = reinterpret_cast<uint64_t*>(smem);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + 16);
  double* red = reinterpret_cast<double*>(smem + 32);
  unsigned char* atile = smem + LY::a_off;
  unsigned char* btile = smem + LY::b_off;
  const int tid = threadIdx.x, warp = tid >> 5;
  for (int i = tid; i < (int)(LY::b_tile / 16); i += NT) reinterpret_cast<uint4*>(btile)[i] = __ldg(ctile + i);
  if (tid == 0) {
    mbar_init(mma_bar, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tc::tmem_alloc(tmem_slot, LY::tmem_cols);
    tc::tmem_relinquish();
  }
  const int hel = rec_cta_helicity<P>();
  bool good = false;
  for (int i = 0; i < nhel; i++) good |= __ldg(hels + i) == hel;
  fence_proxy_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
  const uint32_t a_addr = smem_u32(atile), b_addr = smem_u32(btile);
  uint32_t phase = 0;
  bool ok = true;
  for (long long e = blockIdx.x; e < nevt; e += gridDim.x) {
    const float2* row = J + e * (long long)(P::NCOL * NT) + tid;
    float fr[P::NCOL], fi[P::NCOL];
    // the CTA's next rows on their way to L2 while this event is worked on (8229
    // events 0.33 -> 0.285 ms)
    if (tid == 0 && e + gridDim.x < nevt)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row + (long long)gridDim.x * (P::NCOL * NT)),
                   "r"((uint32_t)(P::NCOL * NT * sizeof(float2)))
                   : "memory");
#pragma unroll
    for (int k = 0; k < P::NCOL; k++) {
      const float2 v = __ldcs(row + k * NT);
      fr[k] = v.x;
      fi[k] = v.y;
    }
    const float s = colour_scale<P, K>(fr, fi);
    float dsum = 0.f;
#pragma unroll
    for (int part = 0; part < 2; part++) {  // Re, then Im
      colour_operands<P, K>(atile, LY::a_tile, tid, s, part ? fi : fr);
      fence_proxy_async_smem();  // generic-proxy tile writes -> visible to the tensor core
      tc::fence_before_sync();
      __syncthreads();
      if (tid == 0) colour_mma<K, N>(tmem + part * N, a_addr, b_addr, LY::a_tile, mma_bar);
      if (part) dsum = colour_readback<P, N>(lane_base, fr);  // Re, while the tensor core works on Im
      // the outcome of the bounded wait is made uniform across the CTA, so that
      // no thread can skip the warp-collective TMEM loads or a barrier alone
      if (!__syncthreads_and(mbar_wait_bounded(mma_bar, phase, polls) ? 1 : 0)) {
        if (tid == 0) atomicOr(status, ST_MMA_TIMEOUT);
        ok = false;
        break;
      }
      phase ^= 1u;
      tc::fence_after_sync();
    }
    if (!ok) break;
    dsum += colour_readback<P, N>(lane_base + N, fi);
    const double part = rec_group_sum<32>(good ? (double)(dsum / s) : 0.0, static_cast<double*>(nullptr));
    if ((tid & 31) == 0) red[warp] = part;
    tc::fence_before_sync();
    __syncthreads();  // tiles and accumulators are reused by the next event
    if (tid == 0) {
      constexpr double norm = 1.0 / (P::IDEN * P::CDEN);
      me[e] = (red[0] + red[1] + red[2] + red[3]) * norm;
    }
  }
  if (!ok) mbar_wait_bounded(mma_bar, phase, WAIT_POLLS);
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, LY::tmem_cols);
  }
}

// ---------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------
inline int rec_sms() {
  int dev = 0, sms = 0;
  return cudaGetDevice(&dev) == cudaSuccess &&
                 cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess
             ? sms
             : 0;
}
// Resident CTAs of a kernel on the current device: the persistent grid.
template <class K>
inline int rec_resident(K kernel, int threads, size_t smem) {
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess)
    return 0;
  return sms * per;
}

// Grid and events per tile: full tiles when the events fill the resident CTAs,
// smaller ones (fewer threads per CTA) when they do not, so that a small batch
// spreads over the SMs.
struct RecGrid {
  unsigned grid;
  int per;
};
inline RecGrid rec_grid(long long nevt, int resident, int ev) {
  const long long share = (nevt + resident - 1) / resident;
  const int per = share < ev ? (int)share : ev;
  const long long tiles = (nevt + per - 1) / per;
  return {(unsigned)(tiles < resident ? tiles : resident), per};
}

template <class P, typename R, typename D, typename A, RecMode MODE = REC_SIGMA>
int launch_rec(const LaunchArgs& a) {
  using LY = RecLayout<P, R>;
  constexpr size_t smem =
      LY::base_bytes + (MODE == REC_SELECT && P::N <= 4
                            ? LY::EV * (P::NHEL + (LY::T > 32 ? LY::T / 32 : 1) * P::NCOL) * sizeof(double)
                            : 0);
  constexpr auto kernel = [] {
    if constexpr (P::N <= 4)
      return rec_kernel<P, R, D, A, MODE>;
    else
      return rec_cta_kernel<P, R, D, A, MODE>;
  }();
  static const cudaError_t attr = set_smem_attr(kernel, smem);
  if (attr != cudaSuccess) return -4;
  static const int resident = rec_resident(kernel, RecShape<P, R>::MAXT, smem);
  if (resident < 1) return -4;
  if (a.nevt <= 0) return 0;  // one-time set-up only
  const RecGrid g = rec_grid(a.nevt, resident, LY::EV);
  kernel<<<g.grid, LY::T * g.per + RecShape<P, R>::HELP, smem, a.stream>>>(a);
  return cudaGetLastError() == cudaSuccess ? 0 : -4;
}

// The two phases over slices of the events that fit the workspace (rows_slice).
template <class P>
int launch_rec_rows(const LaunchArgs& a) {
  using LY = RecLayout<P, float>;
  constexpr size_t smem1 = LY::base_bytes, smem2 = LayoutRows<P>::base_bytes;
  static const cudaError_t attr1 = set_smem_attr(rec_flows_kernel<P>, smem1);
  static const cudaError_t attr2 = set_smem_attr(rec_colour_tc_kernel<P>, smem2);
  if (attr1 != cudaSuccess || attr2 != cudaSuccess) return -4;
  static const int res1 = rec_resident(rec_flows_kernel<P>, LY::T * LY::EV, smem1);
  // two CTAs per SM (launch bounds, shared and tensor memory; the occupancy
  // query counts one for a kernel that allocates tensor memory)
  static const int res2 = 2 * rec_sms();
  if (res1 < 1 || res2 < 1) return -4;
  if (a.nevt <= 0 || a.nhel <= 0) return 0;
  const size_t bytes = rows_workspace_bytes(P::NCOL, P::NHEL, a.nevt);
  const long long slice = rows_slice(P::NCOL, P::NHEL, a.nevt);
  float2* J = nullptr;
  const cudaError_t e0 = a.pool ? cudaMallocFromPoolAsync(reinterpret_cast<void**>(&J), bytes, a.pool, a.stream)
                                : cudaMallocAsync(reinterpret_cast<void**>(&J), bytes, a.stream);
  if (e0 != cudaSuccess) return -4;
  if (a.marks) a.marks->mark(a.stream);
  for (long long i = 0; i < a.nevt; i += slice) {
    const long long ne = a.nevt - i < slice ? a.nevt - i : slice;
    const RecGrid g = rec_grid(ne, res1, LY::EV);
    rec_flows_kernel<P><<<g.grid, LY::T * g.per, smem1, a.stream>>>(a.mom + i * P::NPAR * 4, ne, J, a.kp, a.status);
    if (a.marks) a.marks->mark(a.stream);
    rec_colour_tc_kernel<P><<<(unsigned)(ne < res2 ? ne : res2), 128, smem2, a.stream>>>(
        J, ne, a.out + i, a.hels, a.nhel, static_cast<const uint4*>(a.ctile), a.status, a.kp.polls);
    if (a.marks) a.marks->mark(a.stream);
  }
  const cudaError_t e1 = cudaGetLastError();
  const cudaError_t e2 = cudaFreeAsync(J, a.stream);
  return (e1 == cudaSuccess && e2 == cudaSuccess) ? 0 : -4;
}

}  // namespace mg
