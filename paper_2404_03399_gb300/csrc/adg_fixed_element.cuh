// One element of the fixed-point composed step: its own channel sums, its left neighbour's
// channel scalars and its output rows (adg_fixed.cu, adg_fixed_run.cu).
#pragma once

#include "adg_fixed.cuh"

namespace adg {
namespace {

// Per element slot (S slots before the block's tile for the elements e0-S .. e0-1): the right
// trace p and the unrounded own parts (a, b) of its channel scalars r_s . u, s = 1 .. S-1.
template <int N, int S>
struct ChannelSlots {
  long long p[N + S];
  long long sa[S - 1][N + S], sb[S - 1][N + S];
};
template <int EPT, int S>
struct FixedShared : ChannelSlots<EPT * kTile, S> {
  FxScale sc;
};

// Working-scale value of node j of an element (FP64 input, or int64 input already brought
// to the working scale).
template <bool FIN>
__device__ __forceinline__ long long fx_in(double x, long long X, const FxScale &sc) {
  if (FIN) return X;
  return fx_from_double(x, sc.sigma + 1079);
}

// p = the element's right trace, own[s-1] = the own parts r_s . u of its channel scalars
// (unrounded sums, s = 1 .. S-1), and the limbs of its values for the output rows. BLK: the
// values are block-basis coordinates w (an FP64 input is transformed, w = Tbi u, in FP64
// before its conversion) and the right trace is the exact sum w_0 + w_2 (the first
// coordinate of each block).
template <int NP, bool FIN, int S, bool BLK>
__device__ __forceinline__ void fx_own(const StepFixed &F, const double *Tbi, const double *ud,
                                       const long long *uq, const FxScale &sc, long long &p,
                                       FxAcc *own, int *xh, int *xl) {
  double wd[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    if (BLK && !FIN) {
      double a = Tbi[i * NP] * ud[0];
#pragma unroll
      for (int k = 1; k < NP; ++k) a = fma(Tbi[i * NP + k], ud[k], a);
      wd[i] = a;
    } else {
      wd[i] = FIN ? 0.0 : ud[i];
    }
  }
  p = 0;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const long long X = fx_in<FIN>(wd[j], FIN ? uq[j] : 0ll, sc);
    fx_split(X, xh[j], xl[j]);
#pragma unroll
    for (int s = 1; s < S; ++s) fx_mac(own[s - 1], F.r[s][j], xh[j], xl[j]);
    if (BLK ? (j == 0 || j == 2) : (j == NP - 1)) p += X;
  }
}

template <int N, int S>
__device__ __forceinline__ void fx_publish(ChannelSlots<N, S> &sh, int sl, long long p,
                                           const FxAcc *own) {
  sh.p[sl] = p;
#pragma unroll
  for (int s = 0; s < S - 1; ++s) {
    sh.sa[s][sl] = own[s].a;
    sh.sb[s][sl] = own[s].b;
  }
}

// The channel scalars of element e-1 (P[s], split into limbs) from the published slots
// b .. b+S-1 of elements e-S .. e-1: element e-S+w forms Y_1 .. Y_w from its own parts and the
// scalars of the element before it, Y_s = r_s . u + sum_{t<s} k_st Y_t (each rounded once; every
// thread that needs one of them forms it from the same values, so all agree bit for bit).
template <int N, int S>
__device__ __forceinline__ void fx_left_channels(const StepFixed &F, const ChannelSlots<N, S> &sh,
                                                 int b, int (*P)[2]) {
  long long Yp[S];
  Yp[0] = sh.p[b];
#pragma unroll
  for (int w = 1; w < S; ++w) {
    int ph[S], pl[S];
#pragma unroll
    for (int t = 0; t < w; ++t) fx_split(Yp[t], ph[t], pl[t]);
    long long Y[S];
    Y[0] = sh.p[b + w];
#pragma unroll
    for (int s = 1; s <= w; ++s) {
      FxAcc c{sh.sa[s - 1][b + w], sh.sb[s - 1][b + w]};
#pragma unroll
      for (int t = 0; t < s; ++t) fx_mac(c, F.k[s][t], ph[t], pl[t]);
      Y[s] = fx_round(c);
    }
#pragma unroll
    for (int s = 0; s <= w; ++s) Yp[s] = Y[s];
  }
#pragma unroll
  for (int s = 0; s < S; ++s) fx_split(Yp[s], P[s][0], P[s][1]);
}

// u'^e = G u^e + sum_s h_s P_s for output row i. BLK: G's entries of row i's block only
// (blocks {0, 1} and {2, .., NP-1}); the first row of a 2 x 2 block (and of the 3 x 3 block
// where it was sheared) is (1, 2^-k), whose
// products, X_i and xh_{i+1} 2^(29-k) + xl_{i+1} 2^(29-k) 2^-29, are shifts (the same sums
// as the multiply-adds with the limbs {2^29, 0} and {2^(29-k), 0}).
template <int NP, int S, bool BLK>
__device__ __forceinline__ long long fx_row(const StepFixed &F, int i, const int *xh, const int *xl,
                                            const int (*P)[2]) {
  FxAcc acc;
  if (BLK) {
    const int j0 = i < 2 ? 0 : 2, j1 = i < 2 ? 2 : NP;   // the block [j0, j1)
    // a pair's first row, or the triple's (NP = 5) when its basis was sheared (gs[1] != 0):
    // (1, 2^-k) or (1, 2^-k, 0)
    if (i == j0 && (j1 - j0 == 2 || (j1 - j0 == 3 && F.gs[1] != 0))) {
      // 64-bit values from 32-bit funnel shifts of the limbs (sign words s0, s1)
      const unsigned sh = (unsigned)F.gs[i >> 1];
      const unsigned h0 = (unsigned)xh[i], s0 = (unsigned)(xh[i] >> 31);
      const unsigned h1 = (unsigned)xh[i + 1], s1 = (unsigned)(xh[i + 1] >> 31);
      const unsigned l1 = (unsigned)xl[i + 1];
      const long long x0 = fx_join(__funnelshift_l(0u, h0, 29) | (unsigned)xl[i],
                                   __funnelshift_l(h0, s0, 29));   // X_i
      const long long t1 = fx_join(__funnelshift_l(0u, h1, sh), __funnelshift_l(h1, s1, sh));
      const long long b1 = fx_join(__funnelshift_l(0u, l1, sh), __funnelshift_l(l1, 0u, sh));
      acc.a += x0 + t1;
      acc.b += b1;
    } else {
#pragma unroll
      for (int j = j0; j < j1; ++j) fx_mac(acc, F.G[i * NP + j], xh[j], xl[j]);
    }
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) fx_mac(acc, F.G[i * NP + j], xh[j], xl[j]);
  }
#pragma unroll
  for (int s = 0; s < S; ++s) fx_mac(acc, F.h[s][i], P[s][0], P[s][1]);
  return fx_round(acc);
}

}  // namespace
}  // namespace adg
