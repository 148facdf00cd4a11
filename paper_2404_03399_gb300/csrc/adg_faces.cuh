// PE faces of the composed steps (upwind advection, a > 0): the loads of a face, the synchronous
// traces of its element's stage inputs and the stage differences, shared by the face kernels
// (adg_kernels.cu) and the fixed-point run kernel (adg_fixed_run.cu).
#pragma once

#include "adg_bfp.cuh"
#include "adg_device.cuh"

namespace adg {
namespace {

// What the PE-face correction of face j at step n reads besides the field: its delay k and
// order q' (delay_at), the AT coefficients, and the upwind traces of levels n-k-i (i < q')
// for the S stages from the ring [slot][stage][P] (zero when k = 0).
template <int S>
struct FaceLoads {
  double Rv[S][kMaxQ];
  double c[kMaxQ];
  int k, qe, nm;   // nm: the ring slot of step n
};

template <int S>
__device__ __forceinline__ void face_loads(const Inst &I, int j, int64_t n, FaceLoads<S> &f) {
  const DelayAt dl = delay_at(I, j, n);
  const int P = I.P, R = I.R;
  const int nm = mod_step(n, R);
  f.nm = nm;
  const double2 *col = I.ring + j;
  f.k = dl.k;
  f.qe = dl.qe;
#pragma unroll
  for (int i = 0; i < kMaxQ; ++i) {
    int sl = nm - (dl.k + i);
    if (sl < 0) sl += R;
    const bool use = dl.k > 0 && i < dl.qe;
    f.c[i] = i < dl.qe ? dl.c[i] : 0.0;
    const double2 *lv = col + (size_t)sl * (S * P);
#pragma unroll
    for (int st = 0; st < S; ++st) f.Rv[st][i] = use ? lv[st * P].x : 0.0;
  }
}

// The synchronous traces of element e-1's stage inputs at a PE face (e the face's element):
// T[0] = p^{e-1}, the right trace of u^{e-1}, and the channel scalars T[s] = Y_s^{e-1}_p =
// r_s . u^{e-1} + sum_{t<s} k_st Y_t^{e-2}_p, from elements e-S .. e-1 (w = 0 .. S-1).
template <int S>
struct FaceTraces {
  double T[S];
};

// The channel scalars Y_s^m_p of elements m = e-S+1 .. e-1 in FP64, from the elements
// e-S .. e-1 (U[w], w = 0 .. S-1): element e-S+w forms Y_1 .. Y_w from its values and the
// scalars of the element before it.
template <int NP, int S>
__device__ __forceinline__ FaceTraces<S> face_traces(const Inst &I, const double (*U)[NP]) {
  const StepConsts &C = I.st;
  double Yp[S];   // the channel scalars of the element one to the left (Yp[0] = its trace)
  Yp[0] = U[0][NP - 1];
#pragma unroll
  for (int w = 1; w < S; ++w) {
    const int ns = w;   // channels 1 .. w of element e-S+w
    double Y[S];
    Y[0] = U[w][NP - 1];
#pragma unroll
    for (int s = 1; s <= ns; ++s) {
      double a = C.r[s][0] * U[w][0];
#pragma unroll
      for (int i = 1; i < NP; ++i) a = fma(C.r[s][i], U[w][i], a);
#pragma unroll
      for (int t = 0; t < s; ++t) a = fma(C.k[s][t], Yp[t], a);
      Y[s] = a;
    }
#pragma unroll
    for (int s = 0; s <= ns; ++s) Yp[s] = Y[s];
  }
  FaceTraces<S> t;
#pragma unroll
  for (int s = 0; s < S; ++s) t.T[s] = Yp[s];
  return t;
}

// The right trace of an int64 element: its last value, or for block-basis coordinates the
// sum of the first coordinate of each block, w_0 + w_2 (exact).
template <int NP>
__device__ __forceinline__ long long fx_trace(const Inst &I, const long long *X) {
  if (!I.basis) return X[NP - 1];
  return NP > 2 ? X[0] + X[2] : X[0];
}

// The stage differences d_s = T_s - V_s at PE face j, step n, from the synchronous traces and
// the face's loads in FP64, and the ring write of T_s (the FP64 composed step). With zero delay
// V_s = T_s (the current traces), so d_s = 0.
template <int S>
__device__ __forceinline__ void face_diffs(const Inst &I, int j, const FaceLoads<S> &f,
                                           const FaceTraces<S> &tr, double *d) {
  const int P = I.P;
  const StepConsts &C = I.st;
  double2 *lv = I.ring + j + (size_t)f.nm * (S * P);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    double V = __dmul_rn(f.c[0], f.Rv[s][0]);
#pragma unroll
    for (int i = 1; i < kMaxQ; ++i)
      if (i < f.qe && f.c[i] != 0.0) V = __dadd_rn(V, __dmul_rn(f.c[i], f.Rv[s][i]));
    double T = tr.T[s];
#pragma unroll
    for (int t = 0; t < s; ++t) T = fma(C.rho[s][t], d[t], T);
    d[s] = f.k > 0 ? __dsub_rn(T, V) : 0.0;
    lv[s * P] = make_double2(T, 0.0);
  }
}

// The fixed-point step's PE faces: a group of kFaceLanes<S> consecutive lanes per face, lane r < S
// of it stage r of the differences and element e - S + r of the traces, lane r <= S element
// e - 1 + r of the correction's window. A face is a chain of some hundreds of dependent
// integer instructions and a warp or two per SM all there is, so its latency is the time:
// the stages' values side by side take a third of one thread's (a lane per face), and the
// integers about half of FP64's, whose instruction holds a sub-partition's pipe for 64
// clocks. Every function is called by all 32 lanes of a warp together, those without a face too
// (under a mask known only at run time the shuffles cost the run kernel a microsecond a step).
constexpr unsigned kFullWarp = 0xffffffffu;
template <int S>
constexpr int kFaceLanes = S <= 3 ? 4 : 8;

struct FaceGroup {
  unsigned bits;   // the group's lanes
  int base, r;     // its first lane, and the lane in it
};
template <int S>
__device__ __forceinline__ FaceGroup face_group() {
  constexpr int G = kFaceLanes<S>;
  const int lane = threadIdx.x & 31, base = lane & ~(G - 1);
  return {((1u << G) - 1u) << base, base, lane - base};
}

// Delay k <= n and order in use q' of a face at step n (as delay_at), from its table entry.
struct FaceDelay {
  int k, qe;
};
__device__ __forceinline__ FaceDelay face_delay(const Inst &I, int delay, int64_t n) {
  FaceDelay d;
  d.k = n < delay ? (int)n : delay;
  d.qe = n - d.k + 1 < I.q ? (int)(n - d.k + 1) : I.q;
  return d;
}

// Lane r's (stage r's) delayed value V = sum_i c_i T_i in integers from the ring's traces Rv
// (level n - k - i; 0 beyond the order or without a delay), at the face's scale: be (bf_from),
// from the largest of all stages' traces with three bits of room, 0 where it is left to FP64.
// The coefficients are integers, so the sum is exact (formed modulo 2^64, its high part apart
// to see that it fits).
template <int S>
__device__ __forceinline__ void face_ahead(const Inst &I, const FaceGroup &g, const double *Rv,
                                           const int *c, int qe, long long &V, int &be) {
  int hi = 0;
#pragma unroll
  for (int i = 0; i < kMaxQ; ++i) hi = max(hi, __double2hiint(Rv[i]) & 0x7fffffff);
#pragma unroll
  for (int o = 1; o < kFaceLanes<S>; o *= 2) hi = max(hi, __shfl_xor_sync(kFullWarp, hi, o));
  be = (hi >> 20) + 3;   // |x| < 2^(be - 1025): |X| < 2^54
  const bool range = be >= 103 && be <= 2000 && I.rho_fx;
  long long v = 0, vh = 0;
#pragma unroll
  for (int i = 0; i < kMaxQ; ++i)
    if (i < qe) {
      const long long x = bf_from(Rv[i], be);
      v += (long long)c[i] * x;
      vh += (long long)c[i] * (int)(x >> 32);
    }
  V = v;
  if (!(range && vh > -(1ll << 27) && vh < (1ll << 27))) be = 0;
}

// Lane r's synchronous trace T_r of element e-1's stage inputs from the int64 elements (X: lane
// r's, e - S + r, at 2^sig): the composed step's two-limb sums at a scale chosen from these S
// elements alone (|X'| < 2^(56 - fxh), so the result does not depend on any other face),
// rounded to FP64.
template <int NP, int S>
__device__ __forceinline__ double face_trace_fixed(const Inst &I, const FaceGroup &g, bool on,
                                                   const long long *X, int sig) {
  const StepFixed &F = I.sf;
  unsigned long long m = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i) m |= on ? fx_mag(X[i]) : 0ull;
#pragma unroll
  for (int o = 1; o < kFaceLanes<S>; o *= 2) m |= __shfl_xor_sync(kFullWarp, m, o);
  const int len = m ? 64 - __clzll((long long)m) : 0, cap = 55 - I.fxh;   // |X| < 2^(len + 1)
  const int down = len > cap ? len - cap : 0;
  FxAcc own[S - 1];
  long long Xs[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    Xs[i] = fx_rescale(X[i], down);
    int xh, xl;
    fx_split(Xs[i], xh, xl);
#pragma unroll
    for (int s = 1; s < S; ++s) fx_mac(own[s - 1], F.r[s][i], xh, xl);
  }
  const long long tr = fx_trace<NP>(I, Xs);
  // element e-S+w forms Y_1 .. Y_w from its own sums and the scalars of the element before it
  // (every lane alike)
  long long Yp[S];
  Yp[0] = __shfl_sync(kFullWarp, tr, g.base);
#pragma unroll
  for (int w = 1; w < S; ++w) {
    int ph[S], pl[S];
#pragma unroll
    for (int t = 0; t < w; ++t) fx_split(Yp[t], ph[t], pl[t]);
    long long Y[S];
    Y[0] = __shfl_sync(kFullWarp, tr, g.base + w);
#pragma unroll
    for (int s = 1; s <= w; ++s) {
      FxAcc a;
      a.a = __shfl_sync(kFullWarp, own[s - 1].a, g.base + w);
      a.b = __shfl_sync(kFullWarp, own[s - 1].b, g.base + w);
#pragma unroll
      for (int t = 0; t < s; ++t) fx_mac(a, F.k[s][t], ph[t], pl[t]);
      Y[s] = fx_round(a);
    }
#pragma unroll
    for (int s = 0; s <= w; ++s) Yp[s] = Y[s];
  }
  long long Yr = __shfl_sync(kFullWarp, fx_trace<NP>(I, X), g.base + S - 1);
#pragma unroll
  for (int s = 1; s < S; ++s)
    if (g.r == s) Yr = Yp[s];
  return on ? fx_to_double(Yr, g.r == 0 ? sig : sig + down) : 0.0;
}

// The same from FP64 elements (their bits in X; the first step of a run).
template <int NP, int S>
__device__ __forceinline__ double face_trace_fp64(const Inst &I, const FaceGroup &g, bool on,
                                                  const long long *X) {
  double U[S][NP];
#pragma unroll
  for (int w = 0; w < S; ++w)
#pragma unroll
    for (int i = 0; i < NP; ++i) U[w][i] = __longlong_as_double(__shfl_sync(kFullWarp, X[i], g.base + w));
  const FaceTraces<S> t = face_traces<NP, S>(I, U);
  double T = 0.0;
#pragma unroll
  for (int s = 0; s < S; ++s)
    if (on && g.r == s) T = t.T[s];
  return T;
}

// Lane r's difference d_r = T_r - V_r and its trace T_r with the responses rho to the earlier
// stages' differences, from the synchronous trace T0 and face_ahead's V and be, in integers;
// in FP64 where a value does not fit (rv(i, s): stage s's trace of level n - k - i). Without a
// delay T_r = T0 and d_r = 0.
template <int S, class Ring>
__device__ __forceinline__ void face_differences(const Inst &I, const FaceGroup &g, bool late,
                                                 double T0, long long V, int be, const int *c, int qe,
                                                 Ring &&rv, double &T, double &d) {
  bool ok = be != 0 && biased_exponent(T0) <= be;
  const long long t0 = ok ? bf_from(T0, be) : 0;
  int dh[S], dl[S];
  long long Tr = 0, Dr = 0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    long long t = __shfl_sync(kFullWarp, t0, g.base + s);
    if (s > 0) {
      FxAcc a;
      a.a = t;
#pragma unroll
      for (int q = 0; q < s; ++q) fx_mac(a, I.rhof[s][q], dh[q], dl[q]);
      t = fx_round(a);
    }
    const long long D = t - __shfl_sync(kFullWarp, V, g.base + s);
    ok = ok && fx_mag(D) < (1ull << 58);
    fx_split(D, dh[s], dl[s]);
    if (g.r == s) {
      Tr = t;
      Dr = D;
    }
  }
  // late: a stage's lane of a face with a delay
  const unsigned out = __ballot_sync(kFullWarp, !ok && late);
  ok = (out & g.bits) == 0;
  T = T0;
  d = 0.0;
  if (late) {
    T = bf_to(Tr, be - 1079);
    d = bf_to(Dr, be - 1079);
  }
  if (out) {   // warp-uniform
    double dd[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      double v = 0.0;
      for (int i = 0; i < kMaxQ; ++i) {
        const double x = rv(i, s);
        if (i == 0) v = __dmul_rn((double)c[0], x);
        else if (i < qe && c[i] != 0) v = __dadd_rn(v, __dmul_rn((double)c[i], x));
      }
      double Ts = __shfl_sync(kFullWarp, T0, g.base + s);
#pragma unroll
      for (int q = 0; q < s; ++q) Ts = fma(I.st.rho[s][q], dd[q], Ts);
      dd[s] = __dsub_rn(Ts, v);
      if (late && !ok && g.r == s) {
        T = Ts;
        d = dd[s];
      }
    }
  }
}

// d 2^-sigma rounded, into D; false (left to FP64) where it reaches 2^57.
__device__ __forceinline__ bool face_to_fixed(double d, int sigma, long long &D) {
  const int be = sigma + 1079;
  D = 0;
  if (!nonzero(d)) return true;
  if (be < 100 || biased_exponent(d) > be) return false;
  D = bf_from(d, be);
  return true;
}

// The group's differences in the step's units 2^sigma, as limbs in every lane: 0 nothing to add,
// 1 integer, 2 FP64 (a difference past the integer range).
template <int S>
__device__ __forceinline__ int face_limbs(const Inst &I, const FaceGroup &g, bool on, double d, int sigma,
                                          int *dh, int *dl) {
  long long D = 0;
  const bool fits = !on || face_to_fixed(d, sigma, D);
  const bool any = (__ballot_sync(kFullWarp, on && nonzero(d)) & g.bits) != 0;
  const bool all = (__ballot_sync(kFullWarp, !fits) & g.bits) == 0 && I.face_fx;
  int h, l;
  fx_split(D, h, l);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    dh[s] = __shfl_sync(kFullWarp, h, g.base + s);
    dl[s] = __shfl_sync(kFullWarp, l, g.base + s);
  }
  return any ? (all ? 1 : 2) : 0;
}

// What the correction sum_s R_s d_s adds to window element w in FP64, in the state's units
// (block-basis coordinates: the nodal correction times Tbi).
template <int NP, int S>
__device__ __forceinline__ void face_correction_fp64(const Inst &I, int w, const double *d, int sigma,
                                                     long long *add) {
  double c[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    c[i] = I.st.R[0][w][i] * d[0];
#pragma unroll
    for (int s = 1; s < S; ++s) c[i] = fma(I.st.R[s][w][i], d[s], c[i]);
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    double x = c[i];
    if (I.basis) {
      x = I.Tbi[i * NP] * c[0];
#pragma unroll
      for (int k = 1; k < NP; ++k) x = fma(I.Tbi[i * NP + k], c[k], x);
    }
    add[i] = llrint(pow2_scale(x, -sigma));
  }
}

// The same in integers.
template <int NP, int S>
__device__ __forceinline__ void face_correction(const Inst &I, int w, const int *dh, const int *dl,
                                                long long *add) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    FxAcc a;
#pragma unroll
    for (int s = 0; s < S; ++s) fx_mac(a, I.Rf[s][w][i], dh[s], dl[s]);
    add[i] = fx_round(a);
  }
}

}  // namespace
}  // namespace adg
