// mg_recursion.cuh -- tasks of the helicity-shared colour-ordered recursion.
//
// The currents of one event live in a store of 4-component complex vectors,
// one per (current, helicity combination of its own external legs), and are
// computed by independent tasks, a list per stage (generator/recursion.py
// writes the lists).  The threads that own the event take the tasks of a
// stage in turn; a group barrier separates the stages.  All helicities of the
// event share every current, and one task routine serves a whole stage, so
// the program is a few KB of code instead of one straight line per diagram.
//
// Everything is written against plain memory, so that the same code compiles
// for the host.
//
// Columns are stored as the row of their charge conjugate: with
// b = (b_L, b_R) the row is b~ = (b_L^T eps, -b_R^T eps), eps = i sigma_2,
// i.e. b~ = (-b1, b0, b3, -b2).  Then (Jslash b)~ = -b~ Jslash, and one
// routine propagates rows and columns:
//   row    R' = c  [sum r Jslash] (Qslash + m),  Q = p_t    - K
//   column C' = -c [sum c~ Jslash] (Qslash + m), Q = p_tbar - K.
#pragma once

#include "mg_vertices.cuh"

#ifndef MG_REC_TABLE
#ifdef __CUDACC__
#define MG_REC_TABLE static __device__ const  // read by each thread at its own place
#define MG_REC_CONST static __constant__      // read by all threads at one place
#else
#define MG_REC_TABLE static const
#define MG_REC_CONST static const
#endif
#endif

// task loops stay loops (their bodies are long; see the kernels on the
// instruction caches)
#ifdef __CUDACC__
#define MG_REC_UNROLL _Pragma("unroll")
#ifndef MG_REC_LOOP
#define MG_REC_LOOP _Pragma("unroll 1")
#endif
#else
#define MG_REC_UNROLL
#define MG_REC_LOOP
#endif
namespace mg {
namespace rec {

template <typename R>
__device__ __forceinline__ R fmad(R a, R b, R c) {
#ifdef __CUDA_ARCH__
  return ::fma(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}
// (float)x and (double)f with integer instructions: the conversions run on the
// FP64 pipe (16 cycles per warp instruction and SM), which bounds the set-up of
// the FP32 paths.  The same results bit for bit; values outside the FP32 normal
// range take the conversion itself.
__device__ __forceinline__ float round_f32(double x) {
#ifdef __CUDA_ARCH__
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), a = hi & 0x7fffffffu;
  uint32_t m = __funnelshift_l(lo, a, 3) - 0xC0000000u;     // exponent rebased by 896 << 23, modulo 2^32
  m += ((lo & 0x1fffffffu) + 0x0fffffffu + (m & 1u)) >> 29;  // to nearest, ties to even
  if (a - 0x38100000u < 0x0fd00000u) return __uint_as_float(m | (hi & 0x80000000u));  // exponents 897 .. 1149
  if ((a | lo) == 0u) return __uint_as_float(hi);
#endif
  return (float)x;
}
__device__ __forceinline__ double widen_f64(float f) {
#ifdef __CUDA_ARCH__
  const uint32_t u = __float_as_uint(f), a = u & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u || a == 0u)
    return __hiloint2double((int)((a ? (a >> 3) + 0x38000000u : 0u) | (u & 0x80000000u)), (int)(u << 29));
#endif
  return (double)f;
}

template <typename T>
__device__ __forceinline__ T narrow(double x) {
  if constexpr (sizeof(T) == 4)
    return round_f32(x);
  else
    return x;
}

// acc += a b, acc -= a b (complex): four fused multiply-adds
template <typename R>
__device__ __forceinline__ void cmac(cx<R>& acc, cx<R> a, cx<R> b) {
  acc.re = fmad(a.re, b.re, acc.re);
  acc.im = fmad(a.re, b.im, acc.im);
  acc.re = fmad(-a.im, b.im, acc.re);
  acc.im = fmad(a.im, b.re, acc.im);
}
template <typename R>
__device__ __forceinline__ void cmsc(cx<R>& acc, cx<R> a, cx<R> b) {
  cmac(acc, cx<R>{-a.re, -a.im}, b);
}
template <typename R>
__device__ __forceinline__ cx<R> cmul(cx<R> a, cx<R> b) {
  cx<R> r = {a.re * b.re, a.re * b.im};
  r.re = fmad(-a.im, b.im, r.re);
  r.im = fmad(a.im, b.re, r.im);
  return r;
}
// a.b (Minkowski)
template <typename R>
__device__ __forceinline__ cx<R> vdot(const V4<R>& a, const V4<R>& b) {
  cx<R> s = cmul(a.c[0], b.c[0]);
  cmsc(s, a.c[1], b.c[1]);
  cmsc(s, a.c[2], b.c[2]);
  cmsc(s, a.c[3], b.c[3]);
  return s;
}
template <typename R>
__device__ __forceinline__ cx<R> kdot(const M4<R>& k, const V4<R>& b) {
  cx<R> s = {k.v[0] * b.c[0].re, k.v[0] * b.c[0].im};
#pragma unroll
  for (int mu = 1; mu < 4; mu++) {
    s.re = fmad(-k.v[mu], b.c[mu].re, s.re);
    s.im = fmad(-k.v[mu], b.c[mu].im, s.im);
  }
  return s;
}
// acc += row . column, the column given as its conjugate row:
// a0 b~1 - a1 b~0 - a2 b~3 + a3 b~2
template <typename R>
__device__ __forceinline__ void close_rc(cx<R>& acc, const V4<R>& a, const V4<R>& b) {
  cmac(acc, a.c[0], b.c[1]);
  cmsc(acc, a.c[1], b.c[0]);
  cmsc(acc, a.c[2], b.c[3]);
  cmac(acc, a.c[3], b.c[2]);
}
// o += r Jslash = (r_R Y, r_L X)
template <typename R>
__device__ __forceinline__ void row_slash(V4<R>& o, const V4<R>& r, const V4<R>& J) {
  const cx<R> jp = J.c[0] + J.c[3], jm = J.c[0] - J.c[3];
  const cx<R> iJ2 = mul_i(J.c[2]);
  const cx<R> u = J.c[1] - iJ2, w = J.c[1] + iJ2;
  cmac(o.c[0], r.c[2], jp);
  cmac(o.c[0], r.c[3], w);
  cmac(o.c[1], r.c[2], u);
  cmac(o.c[1], r.c[3], jm);
  cmac(o.c[2], r.c[0], jm);
  cmsc(o.c[2], r.c[1], w);
  cmsc(o.c[3], r.c[0], u);
  cmac(o.c[3], r.c[1], jp);
}
// coef * (t (Qslash + m)), Q real
template <typename R>
__device__ __forceinline__ V4<R> row_prop(const V4<R>& t, const M4<R>& Q, R m, cx<R> coef) {
  const R qp = Q.v[0] + Q.v[3], qm = Q.v[0] - Q.v[3];
  const cx<R> u = {Q.v[1], -Q.v[2]}, w = {Q.v[1], Q.v[2]};
  V4<R> o;
#pragma unroll
  for (int i = 0; i < 4; i++) o.c[i] = {m * t.c[i].re, m * t.c[i].im};
  auto rmac = [](cx<R>& a, R x, cx<R> b) {
    a.re = fmad(x, b.re, a.re);
    a.im = fmad(x, b.im, a.im);
  };
  rmac(o.c[0], qp, t.c[2]);
  cmac(o.c[0], t.c[3], w);
  cmac(o.c[1], t.c[2], u);
  rmac(o.c[1], qm, t.c[3]);
  rmac(o.c[2], qm, t.c[0]);
  cmsc(o.c[2], t.c[1], w);
  cmsc(o.c[3], t.c[0], u);
  rmac(o.c[3], qp, t.c[1]);
#pragma unroll
  for (int i = 0; i < 4; i++) o.c[i] = cmul(coef, o.c[i]);
  return o;
}

// ---------------------------------------------------------------------------
// the event's store: NV vectors in planes of 16 bytes (the threads of a warp
// mostly touch consecutive vectors, so each 16-byte access of a warp falls on
// consecutive banks), then the scalars: sums of gluon momenta per subset,
// p_t, p_tbar, propagator coefficients per subset
// ---------------------------------------------------------------------------
template <typename R>
struct alignas(16) Pack {
  R x[16 / sizeof(R)];
};

template <typename R, int N, int NV>
struct Store {
  static constexpr int PER = 16 / sizeof(R);  // reals per plane entry
  static constexpr int NP = 8 / PER;          // planes
  static constexpr int NSUB = 1 << N;
  static constexpr int S_K = 0;                   // [NSUB][4]
  static constexpr int S_PT = 4 * NSUB;           // p_t, p_tbar
  static constexpr int S_CF = S_PT + 8;           // [NSUB] complex
  static constexpr int S_CG = S_CF + 2 * NSUB;    // [NSUB]
  static constexpr int NS = S_CG + NSUB;
  static constexpr size_t vec_bytes = size_t(NV) * 8 * sizeof(R);
  static constexpr size_t pair_off = vec_bytes + size_t(NS) * sizeof(R);  // setup_pair (FP32)
  static constexpr size_t mom_off = pair_off + (sizeof(R) == 4 ? size_t((N + 1) * (N + 2) / 2) * sizeof(double) : 0);
  static constexpr size_t bytes = mom_off + size_t(N + 2) * 4 * sizeof(R);  // the event's momenta in R
  static constexpr size_t stride = (bytes + 127) / 128 * 128;               // to the next event's store
  Pack<R>* p;
  R* sc;
  __device__ __forceinline__ explicit Store(void* mem)
      : p(reinterpret_cast<Pack<R>*>(mem)),
        sc(reinterpret_cast<R*>(reinterpret_cast<unsigned char*>(mem) + vec_bytes)) {}
  // the store e events on
  __device__ __forceinline__ Store at(int e) const {
    return Store(reinterpret_cast<unsigned char*>(p) + (ptrdiff_t)e * (ptrdiff_t)stride);
  }
  __device__ __forceinline__ double* pairs() const {
    return reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(p) + pair_off);
  }
  __device__ __forceinline__ R* momenta() const {
    return reinterpret_cast<R*>(reinterpret_cast<unsigned char*>(p) + mom_off);
  }
  __device__ __forceinline__ V4<R> ld(int v) const {
    V4<R> o;
#pragma unroll
    for (int q = 0; q < NP; q++) {
      const Pack<R> t = p[q * NV + v];
#pragma unroll
      for (int i = 0; i < PER / 2; i++) o.c[q * (PER / 2) + i] = {t.x[2 * i], t.x[2 * i + 1]};
    }
    return o;
  }
  __device__ __forceinline__ void st(int v, const V4<R>& o) const {
#pragma unroll
    for (int q = 0; q < NP; q++) {
      Pack<R> t;
#pragma unroll
      for (int i = 0; i < PER / 2; i++) {
        t.x[2 * i] = o.c[q * (PER / 2) + i].re;
        t.x[2 * i + 1] = o.c[q * (PER / 2) + i].im;
      }
      p[q * NV + v] = t;
    }
  }
  __device__ __forceinline__ M4<R> mom(int off) const {
    const Pack<R>* m = reinterpret_cast<const Pack<R>*>(sc + off);
    M4<R> k;
#pragma unroll
    for (int q = 0; q < 4 / PER; q++) {
      const Pack<R> t = m[q];
#pragma unroll
      for (int i = 0; i < PER; i++) k.v[q * PER + i] = t.x[i];
    }
    return k;
  }
  __device__ __forceinline__ M4<R> K(int mask) const { return mom(S_K + 4 * mask); }
  __device__ __forceinline__ cx<R> cf(int mask) const { return {sc[S_CF + 2 * mask], sc[S_CF + 2 * mask + 1]}; }
};

// ---------------------------------------------------------------------------
// set-up of one event from its momenta p[NPAR][4] (FP64): task t of
// setup_tasks() computes one subset's momentum sum and coefficients, or the
// external wavefunctions of one leg.  D: arithmetic of the propagator
// denominators; external states in FP32 where the amplitudes are FP32, as in
// the per-helicity program.
// ---------------------------------------------------------------------------
// (sum_n s_n v_n)^2 - m2 with s_n in {-1, 0, 1}: zero terms leave every
// partial result unchanged, so this is inv_mass2 of the terms present
template <typename R, typename D, int NT>
__device__ __forceinline__ D inv_mass2_masked(const double* p, const int (&slot)[NT], const D (&s)[NT], D m2) {
  if constexpr (sizeof(R) == 8 && sizeof(D) == 8) {
    D hi = -m2, lo = D(0);
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      D ch = s[0] * D(p[4 * slot[0] + mu]), cl = D(0);
#pragma unroll
      for (int k = 1; k < NT; k++) {
        D e;
        two_sum(ch, s[k] * D(p[4 * slot[k] + mu]), ch, e);
        cl += e;
      }
      const D sq = ch * ch;
      const D sq_lo = fmad(ch, ch, -sq) + D(2) * ch * cl;
      D e;
      if (mu == 0) {
        two_sum(hi, sq, hi, e);
        lo += e + sq_lo;
      } else {
        two_sum(hi, -sq, hi, e);
        lo += e - sq_lo;
      }
    }
    return hi + lo;
  } else {
    D c[4];
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      c[mu] = s[0] * D(p[4 * slot[0] + mu]);
#pragma unroll
      for (int k = 1; k < NT; k++) c[mu] = c[mu] + s[k] * D(p[4 * slot[k] + mu]);
    }
    return c[0] * c[0] - c[1] * c[1] - c[2] * c[2] - c[3] * c[3] - m2;
  }
}

// Tasks of the set-up, in lists that a thread group strides over, after the
// momenta have been brought to R (k[NPAR][4]): subset m in [0, 2^N): momentum
// sum; denominators of the propagators' subsets; leg l in [0, N + 2): external
// wavefunctions.  kr: g_s, m_t in R.  g is folded into the row of the outgoing
// top (one factor per amplitude).
template <class P, typename R, class ST>
__device__ __forceinline__ void setup_momenta(const ST& st, const R* k, int m) {
  constexpr int N = P::N;
  R t[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll
  for (int i = 0; i < N; i++) {
    const int slot = i < 2 ? i : i + 2;
    const R sg = !(m >> i & 1) ? R(0) : (i < 2 ? R(1) : R(-1));
#pragma unroll
    for (int mu = 0; mu < 4; mu++) t[mu] = fmad(sg, k[4 * slot + mu], t[mu]);
  }
#pragma unroll
  for (int mu = 0; mu < 4; mu++) st.sc[ST::S_K + 4 * m + mu] = t[mu];
  if (m < 2) {
#pragma unroll
    for (int mu = 0; mu < 4; mu++) st.sc[ST::S_PT + 4 * m + mu] = k[8 + 4 * m + mu];
  }
}
// c in [0, 2^(N+1)): bit N selects the fermion denominators
template <int N>
__device__ __forceinline__ bool is_propagator(int c) {
  const int m = c & ((1 << N) - 1);
  return c >> N ? (m != 0 && m != (1 << N) - 1) : (m & (m - 1)) != 0;
}
template <typename R, class ST>
__device__ __forceinline__ void store_coef(const ST& st, int m, bool f, R re, R im) {
  if (f) {
    st.sc[ST::S_CF + 2 * m] = re;
    st.sc[ST::S_CF + 2 * m + 1] = im;
  } else {
    st.sc[ST::S_CG + m] = re;
  }
}
template <class P, typename R, typename D, class ST>
__device__ __forceinline__ void setup_coef(const ST& st, const double* p, const double* kp, int c) {
  constexpr int N = P::N;
  if (!is_propagator<N>(c)) return;
  const bool f = (c >> N) != 0;
  const int m = c & (ST::NSUB - 1);
  const D g = D(kp[0]), mt = D(kp[1]), wt = D(kp[2]);
  int slot[N + 1];
  D s[N + 1];
  slot[0] = 2;
  s[0] = f ? D(1) : D(0);
#pragma unroll
  for (int i = 0; i < N; i++) {
    slot[i + 1] = i < 2 ? i : i + 2;
    const D sg = (i < 2) != f ? D(1) : D(-1);
    s[i + 1] = (m >> i & 1) ? sg : D(0);
  }
  const D v = inv_mass2_masked<R, D, N + 1>(p, slot, s, f ? mt * mt : D(0));
  const D dim = mt * wt;
  const D r = -g / (f ? v * v + dim * dim : v);
  store_coef<R>(st, m, f, f ? R(r * v) : R(r), R(-r * dim));
}

// The same for FP32 amplitudes with FP64 denominators, with a third of the
// FP64 instructions (GB300's FP64 pipe takes 16 cycles per warp instruction;
// the plain form kept it busy for a third of the four-gluon kernel): first
// the products p_t^2 - m^2, k_i^2 and twice those of every other pair of the
// momenta p_t, k_0 .. k_N-1 (incoming), then
//   K^2 = sum k_i^2 + sum 2 k_i.k_j,
//   (p_t - K)^2 - m^2 = (p_t^2 - m^2 - sum 2 p_t.k_i) + K^2,
// which rounds like the square of the sum (a few 1e-16 of the largest energy
// squared; masses and on-shell conditions are not assumed), and 1 / d from
// the FP32 reciprocal and one Newton step (1e-14, then rounded to FP32).
// pairs: scratch of (N + 1) (N + 2) / 2 doubles; entry j (j + 1) / 2 + i for i <= j,
// 0: p_t, 1 + i: k_i.  kp: g_s, m_t, width, m_t^2, m_t width, (m_t width)^2.
template <int N>
__host__ __device__ constexpr int pair_at(int i, int j) {
  return j * (j + 1) / 2 + i;
}
template <class P>
__device__ __forceinline__ void setup_pair(double* pairs, const double* p, const double* kp, int t) {
  constexpr int N = P::N;
  if (t >= (N + 1) * (N + 2) / 2) return;
  int j = 0;
  while ((j + 1) * (j + 2) / 2 <= t) j++;
  const int i = t - j * (j + 1) / 2;
  auto at = [](int q) { return q == 0 ? 2 : (q < 3 ? q - 1 : q + 1); };  // particle slot
  auto in = [](int q) { return q == 0 || q > 2; };                         // outgoing momentum
  const double* a = p + 4 * at(i);
  const double* b = p + 4 * at(j);
  double d = fmad(a[0], b[0], t == 0 ? -kp[3] : 0.0);
  d = fmad(-a[1], b[1], d);
  d = fmad(-a[2], b[2], d);
  d = fmad(-a[3], b[3], d);
  // k = -p for the outgoing gluons; p_t as it is
  const bool minus = (i > 0 && in(i)) != (j > 0 && in(j));
  d = minus ? -d : d;
  pairs[t] = i == j ? d : d + d;
}
__device__ __forceinline__ double quick_inverse(double d) {
  const float f = round_f32(d);
  const float y = 1.0f / f;
  if (!(y < 1e38f && y > -1e38f) || !(f < 1e38f && f > -1e38f)) return 1.0 / d;  // outside the FP32 range, or NaN
  const double w = widen_f64(y);
  return fmad(fmad(-d, w, 1.0), w, w);
}
// subset m: both of its denominators
template <class P, class ST>
__device__ __forceinline__ void setup_coef_pairs(const ST& st, const double* pairs, const double* kp, int m) {
  constexpr int N = P::N;
  const double g = kp[0];
  double v = 0.0, f = pairs[0];
#pragma unroll
  for (int j = 0; j < N; j++) {
    if (m >> j & 1) {
      v += pairs[pair_at<N>(j + 1, j + 1)];
      f -= pairs[pair_at<N>(0, j + 1)];
    }
#pragma unroll
    for (int i = 0; i < j; i++)
      if ((m >> i & 1) && (m >> j & 1)) v += pairs[pair_at<N>(i + 1, j + 1)];
  }
  if (is_propagator<N>(m)) store_coef<float>(st, m, false, round_f32(-g * quick_inverse(v)), 0.f);
  if (is_propagator<N>(m | 1 << N)) {
    f += v;
    const double r = -g * quick_inverse(fmad(f, f, kp[5]));
    store_coef<float>(st, m, true, round_f32(r * f), round_f32(-r * kp[4]));
  }
}

// external states of leg l (gluons, then t, t~) of momentum q
template <class P, typename R, typename E, class ST>
__device__ __forceinline__ void leg_states(const ST& st, const E (&q)[4], const R* kr, int l) {
  constexpr int N = P::N;
  if (l < N) {
    E b[6];
    vector_basis(q, b);
    const R e1[3] = {R(b[0]), R(b[1]), R(b[2])}, e2[3] = {R(b[3]), R(b[4]), R(b[5])};
    const int base = P::j1_base(l);
    st.st(base, ext_vector<R>(e1, e2, R(-1), l >= 2));
    st.st(base + 1, ext_vector<R>(e1, e2, R(1), l >= 2));
  } else {
    E f[5];
    fermion_ingredients(q, E(kr[1]), f);
    const FermIngr<R> fi = {R(f[0]), R(f[1]), R(f[2]), R(f[3]), R(f[4])};
    const R g = kr[0];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int lam = 2 * h - 1;
      if (l == N) {
        const Sp<R> u = ext_ubar<R>(fi, lam);
        V4<R> o;
        for (int i = 0; i < 4; i++) o.c[i] = g * u.c[i];
        st.st(P::R0 + h, o);
      } else {
        const Sp<R> v = ext_v<R>(fi, lam);
        V4<R> o;
        o.c[0] = -v.c[1];
        o.c[1] = v.c[0];
        o.c[2] = v.c[3];
        o.c[3] = -v.c[2];
        st.st(P::C0 + h, o);
      }
    }
  }
}
template <class P, typename R, class ST>
__device__ __forceinline__ void setup_leg(const ST& st, const R* k, const R* kr, int l) {
  constexpr int N = P::N;
  const int slot = l < 2 ? l : (l < N ? l + 2 : l - N + 2);
  const R q[4] = {k[4 * slot], k[4 * slot + 1], k[4 * slot + 2], k[4 * slot + 3]};
  leg_states<P, R, R>(st, q, kr, l);
}

// ---------------------------------------------------------------------------
// tasks; row: the task's line of the stage table; kr: g_s, m_t in R
// ---------------------------------------------------------------------------
template <int W>
struct alignas(16) Row {
  unsigned short v[W];
};

// J(w) of m ordered gluons, c = -g / P^2:
//   c { sum_i V3(J(w_1..i), J(w_i+1..m)) + sum_i<j Q(J(w_1..i), J(w_i+1..j), J(w_j+1..m)) }
//   V3(X, Y) = (X.Y)(kX - kY) + 2 (kY.X) Y - 2 (kX.Y) X   (currents are conserved: kX.X = 0)
//   Q(X, Y, Z) = -g [2 (X.Z) Y - (Y.Z) X - (X.Y) Z].
// The coefficient of each sub-current is collected first, so that every one
// is scaled and added once.  Table: the sub-currents [i, j) in (i, j) order,
// the two masks of every split, the destination and that of the current with
// every helicity flipped, (-1)^m J* (and for pairs the two destinations of
// J(w reversed) = -J(w)).
template <typename R>
__device__ __forceinline__ V4<R> flipped(const V4<R>& a, bool odd) {
  V4<R> o;
#pragma unroll
  for (int mu = 0; mu < 4; mu++) o.c[mu] = {odd ? -a.c[mu].re : a.c[mu].re, odd ? a.c[mu].im : -a.c[mu].im};
  return o;
}
template <int M, typename R, class ST, class RW>
__device__ __forceinline__ void j_task(const ST& st, const RW& row, const R* kr) {
  constexpr int NSUBW = M * (M + 1) / 2 - 1;
  // position of the sub-current [i, j) in the table
  auto at = [](int i, int j) constexpr {
    int q = 0;
    for (int a = 0; a < M; a++)
      for (int b = a + 1; b <= M; b++)
        if (b - a < M) {
          if (a == i && b == j) return q;
          q++;
        }
    return 0;
  };
  V4<R> J[NSUBW];
  cx<R> c[NSUBW];
#pragma unroll
  for (int q = 0; q < NSUBW; q++) {
    J[q] = st.ld(row.v[q]);
    c[q] = {R(0), R(0)};
  }
  V4<R> acc;
#pragma unroll
  for (int mu = 0; mu < 4; mu++) acc.c[mu] = {R(0), R(0)};
#pragma unroll
  for (int i = 1; i < M; i++) {
    const V4<R>&X = J[at(0, i)], &Y = J[at(i, M)];
    const M4<R> kx = st.K(row.v[NSUBW + 2 * (i - 1)]), ky = st.K(row.v[NSUBW + 2 * (i - 1) + 1]);
    const cx<R> xy = vdot(X, Y), yx = kdot(ky, X), xk = kdot(kx, Y);
    c[at(i, M)].re = fmad(R(2), yx.re, c[at(i, M)].re);
    c[at(i, M)].im = fmad(R(2), yx.im, c[at(i, M)].im);
    c[at(0, i)].re = fmad(R(-2), xk.re, c[at(0, i)].re);
    c[at(0, i)].im = fmad(R(-2), xk.im, c[at(0, i)].im);
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      const R d = kx.v[mu] - ky.v[mu];
      acc.c[mu].re = fmad(d, xy.re, acc.c[mu].re);
      acc.c[mu].im = fmad(d, xy.im, acc.c[mu].im);
    }
  }
  if constexpr (M > 2) {
    const R g = kr[0];
#pragma unroll
    for (int i = 1; i < M - 1; i++)
#pragma unroll
      for (int j = i + 1; j < M; j++) {
        const V4<R>&X = J[at(0, i)], &Y = J[at(i, j)], &Z = J[at(j, M)];
        const cx<R> xz = vdot(X, Z), yz = vdot(Y, Z), xy = vdot(X, Y);
        c[at(i, j)].re = fmad(R(-2) * g, xz.re, c[at(i, j)].re);
        c[at(i, j)].im = fmad(R(-2) * g, xz.im, c[at(i, j)].im);
        c[at(0, i)].re = fmad(g, yz.re, c[at(0, i)].re);
        c[at(0, i)].im = fmad(g, yz.im, c[at(0, i)].im);
        c[at(j, M)].re = fmad(g, xy.re, c[at(j, M)].re);
        c[at(j, M)].im = fmad(g, xy.im, c[at(j, M)].im);
      }
  }
#pragma unroll
  for (int q = 0; q < NSUBW; q++)
#pragma unroll
    for (int mu = 0; mu < 4; mu++) cmac(acc.c[mu], c[q], J[q].c[mu]);
  constexpr int DST = NSUBW + 2 * (M - 1);
  const R cg = st.sc[ST::S_CG + (row.v[NSUBW] | row.v[NSUBW + 1])];  // mask of w: of its first split
#pragma unroll
  for (int mu = 0; mu < 4; mu++) acc.c[mu] = {cg * acc.c[mu].re, cg * acc.c[mu].im};
  st.st(row.v[DST], acc);
  st.st(row.v[DST + 1], flipped(acc, M % 2 != 0));
  if constexpr (M == 2) {
#pragma unroll
    for (int mu = 0; mu < 4; mu++) acc.c[mu] = -acc.c[mu];
    st.st(row.v[DST + 2], acc);
    st.st(row.v[DST + 3], flipped(acc, false));
  }
}

// +- the sum of one to three vectors (Kleiss-Kuijf): x1, x2, x3, destination,
// number of terms, sign flag, destination with every helicity flipped, odd
// number of gluons
template <typename R, class ST, class RW>
__device__ __forceinline__ void comb_task(const ST& st, const RW& row) {
  V4<R> o = st.ld(row.v[0]);
#pragma unroll
  for (int q = 1; q < 3; q++)
    if (q < row.v[4]) {
      const V4<R> x = st.ld(row.v[q]);
      for (int mu = 0; mu < 4; mu++) o.c[mu] = o.c[mu] + x.c[mu];
    }
  const R sg = row.v[5] ? R(-1) : R(1);
  for (int mu = 0; mu < 4; mu++) o.c[mu] = {sg * o.c[mu].re, sg * o.c[mu].im};
  st.st(row.v[3], o);
  st.st(row.v[6], flipped(o, row.v[7] != 0));
}

// amputated line: sum over NT pairs (spinor, current); table: the pairs, destination
template <int NT, typename R, class ST, class RW>
__device__ __forceinline__ V4<R> line_sum(const ST& st, const RW& row) {
  V4<R> o;
#pragma unroll
  for (int i = 0; i < 4; i++) o.c[i] = {R(0), R(0)};
#pragma unroll
  for (int q = 0; q < NT; q++) row_slash(o, st.ld(row.v[2 * q]), st.ld(row.v[2 * q + 1]));
  return o;
}
template <int NT, typename R, class ST, class RW>
__device__ __forceinline__ void amp_task(const ST& st, const RW& row) {
  st.st(row.v[2 * NT], line_sum<NT, R>(st, row));
}
// full line; table: the pairs, destination, line (0 top, 1 antitop), mask of
// the momenta it absorbed, mask of the denominator
template <int NT, typename R, class ST, class RW>
__device__ __forceinline__ void line_task(const ST& st, const RW& row, const R* kr) {
  const V4<R> t = line_sum<NT, R>(st, row);
  const int line = row.v[2 * NT + 1];
  const M4<R> e = st.mom(ST::S_PT + 4 * line), k = st.K(row.v[2 * NT + 2]);
  cx<R> c = st.cf(row.v[2 * NT + 3]);
  const R sg = line ? R(-1) : R(1);
  c = {sg * c.re, sg * c.im};
  M4<R> Q;
#pragma unroll
  for (int mu = 0; mu < 4; mu++) Q.v[mu] = e.v[mu] - k.v[mu];
  st.st(row.v[2 * NT], row_prop(t, Q, kr[1], c));
}
// V with V.J = row Jslash column; table: row, column, destination
template <typename R, class ST, class RW>
__device__ __forceinline__ void vec_task(const ST& st, const RW& row) {
  const V4<R> a = st.ld(row.v[0]), t = st.ld(row.v[1]);
  // the column behind its conjugate row: b = (t1, -t0, -t3, t2)
  cx<R> p = cmul(a.c[0], t.c[3]), q = cmul(a.c[1], t.c[2]);  // -a0 b2, a1 b3
  cx<R> r = cmul(a.c[0], t.c[2]), s = cmul(a.c[1], t.c[3]);  // a0 b3, -a1 b2
  cx<R> P = cmul(a.c[2], t.c[1]), Q = cmul(a.c[3], t.c[0]);  // a2 b0, -a3 b1
  cx<R> S = cmul(a.c[2], t.c[0]), T = cmul(a.c[3], t.c[1]);  // -a2 b1, a3 b0
  V4<R> g;
  const cx<R> u02 = -p, u13 = q, u03 = r, u12 = -s, l20 = P, l31 = -Q, l21 = -S, l30 = T;
  g.c[0] = (u02 + u13) + (l20 + l31);
  g.c[1] = (u03 + u12) - (l21 + l30);
  g.c[2] = mul_i((u12 - u03) + (l21 - l30));
  g.c[3] = (u02 - u13) - (l20 - l31);
  st.st(row.v[2], g);
}

// ---------------------------------------------------------------------------
// one thread per event (two gluons): the store in registers -- every index is a
// constant once the task calls are inlined
// ---------------------------------------------------------------------------
template <typename R, int N, int NV>
struct RegStore {
  static constexpr int NSUB = 1 << N;
  static constexpr int S_K = 0, S_PT = 4 * NSUB, S_CF = S_PT + 8, S_CG = S_CF + 2 * NSUB, NS = S_CG + NSUB;
  mutable V4<R> v[NV];
  mutable R sc[NS];
  __device__ __forceinline__ V4<R> ld(int i) const { return v[i]; }
  __device__ __forceinline__ void st(int i, const V4<R>& o) const { v[i] = o; }
  __device__ __forceinline__ M4<R> mom(int off) const { return {{sc[off], sc[off + 1], sc[off + 2], sc[off + 3]}}; }
  __device__ __forceinline__ M4<R> K(int mask) const { return mom(S_K + 4 * mask); }
  __device__ __forceinline__ cx<R> cf(int mask) const { return {sc[S_CF + 2 * mask], sc[S_CF + 2 * mask + 1]}; }
};

// (p_t - K)^2 - m2 (f) or K^2 of the subset m; m and f are constants once
// inlined.  FP64 amplitudes: compensated like inv_mass2, term by term.
template <int N, typename R, typename D>
__device__ __forceinline__ D subset_mass2(const D (&q)[N + 2][4], bool f, int m, D m2) {
  constexpr bool comp = sizeof(R) == 8 && sizeof(D) == 8;
  D hi = -m2, lo = D(0);
#pragma unroll
  for (int mu = 0; mu < 4; mu++) {
    D ch = D(0), cl = D(0);
    bool first = true;
    if (f) {
      ch = q[N][mu];
      first = false;
    }
#pragma unroll
    for (int i = 0; i < N; i++)
      if (m >> i & 1) {
        const D x = (i < 2) != f ? q[i][mu] : -q[i][mu];  // q: physical momenta, incoming first
        if (first) {
          ch = x;
        } else if constexpr (comp) {
          D e;
          two_sum(ch, x, ch, e);
          cl += e;
        } else {
          ch += x;
        }
        first = false;
      }
    if constexpr (comp) {
      const D sq = ch * ch;
      const D sq_lo = fmad(ch, ch, -sq) + D(2) * ch * cl;
      D e;
      two_sum(hi, mu == 0 ? sq : -sq, hi, e);
      lo += mu == 0 ? e + sq_lo : e - sq_lo;
    } else {
      hi = fmad(mu == 0 ? ch : -ch, ch, hi);
    }
  }
  return comp ? hi + lo : hi;
}

// set-up of a RegStore from the event's momenta
template <class P, typename R, typename D, class ST>
__device__ __forceinline__ void setup_thread(const ST& st, const double* p, const double* kp, const R* kr) {
  constexpr int N = P::N;
  D q[N + 2][4];  // gluons, top, antitop
  R k[N + 2][4];
#pragma unroll
  for (int i = 0; i < N + 2; i++)
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      const double x = p[4 * (i < 2 ? i : (i < N ? i + 2 : i - N + 2)) + mu];
      q[i][mu] = narrow<D>(x);
      k[i][mu] = narrow<R>(x);
    }
#pragma unroll
  for (int m = 0; m < ST::NSUB; m++)
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
      R s = R(0);
      bool first = true;
#pragma unroll
      for (int i = 0; i < N; i++)
        if (m >> i & 1) {
          const R x = i < 2 ? k[i][mu] : -k[i][mu];
          s = first ? x : s + x;
          first = false;
        }
      st.sc[ST::S_K + 4 * m + mu] = s;
    }
#pragma unroll
  for (int mu = 0; mu < 4; mu++) {
    st.sc[ST::S_PT + mu] = k[N][mu];
    st.sc[ST::S_PT + 4 + mu] = k[N + 1][mu];
  }
  constexpr bool mixed = sizeof(R) == 4 && sizeof(D) == 8;
  const D g = D(kp[0]), mt = D(kp[1]);
  const D mt2 = mixed ? D(kp[3]) : mt * mt, dim = mixed ? D(kp[4]) : mt * D(kp[2]);
  const D dim2 = mixed ? D(kp[5]) : dim * dim;
#pragma unroll
  for (int c = 0; c < 2 * ST::NSUB; c++) {
    const bool f = (c >> N) != 0;
    const int m = c & (ST::NSUB - 1);
    if (!is_propagator<N>(c)) continue;
    const D v = subset_mass2<N, R, D>(q, f, m, f ? mt2 : D(0));
    const D den = f ? fmad(v, v, dim2) : v;
    D r;
    if constexpr (mixed)
      r = -g * quick_inverse(den);
    else
      r = -g / den;
    if constexpr (mixed)
      store_coef<float>(st, m, f, f ? round_f32(r * v) : round_f32(r), f ? round_f32(-r * dim) : 0.f);
    else
      store_coef<R>(st, m, f, f ? R(r * v) : R(r), R(-r * dim));
  }
  using E = typename std::conditional<sizeof(R) == 4, float, D>::type;
#pragma unroll
  for (int l = 0; l < N + 2; l++) {
    E e[4];
#pragma unroll
    for (int mu = 0; mu < 4; mu++) e[mu] = E(k[l][mu]);
    leg_states<P, R, E>(st, e, kr, l);
  }
}

// x of the subset bits of the gluon helicities hg: bit i of `mask` set ->
// bit i of hg, packed
template <int MASK, int N>
__device__ __forceinline__ int hel_bits(int hg) {
  int o = 0, q = 0;
#pragma unroll
  for (int i = 0; i < N; i++)
    if (MASK >> i & 1) o |= (hg >> i & 1) << q++;
  return o;
}

}  // namespace rec
}  // namespace mg
