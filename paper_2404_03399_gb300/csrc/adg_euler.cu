// One-dimensional Euler equations (Section 6, Sod's shock tube): FP64 stage and limiter
// kernels for sm_103a.
//
// State U = (rho, m, E), E = rho u^2 / 2 + p / (gamma - 1), gamma = 1.4, three node-major
// planes per component (component c of a field at field + c K Np). One thread per element;
// in the stage kernel a warp takes 30 elements with their two neighbours in its edge lanes.
//   * k_euler_stage: one stage of SSP-RK in Shu and Osher's form,
//       out = alpha u + beta (v + dt L(v)),   dt L(v) = dt [ -QD f + qlL (f_0 - F_L) + qlR (f_p - F_R) ]
//     (the strong form of the nodal DG operator, QD = (2/dx) D, qlL = -(2/dx) M^{-1} e_0,
//     qlR = (2/dx) M^{-1} e_p), with the local Lax-Friedrichs flux at faces; at PE faces the
//     flux is the AT sum (Eq. at-flux-gen) of the stored Lax-Friedrichs fluxes of
//     the common delayed level, and the face owner stores the stage's flux.
//   * k_euler_limit: the TVB-minmod slope limiter on every component (cell average a0 and
//     P_1 coefficient a1; a1' = minmod(2 a1, d+, d-) / 2 unless |a1| <= M dx^2 / 2; an
//     element whose a1 changes becomes a0 + a1' xi). Its stencil ends at PE faces (one-sided
//     there), so it needs no exchange.
#include <algorithm>
#include <cmath>

#include "adg_device.cuh"

namespace adg {

namespace {

constexpr double kGamma = 1.4;

// Flux f(U) of a state (u = m / rho through one division 1/rho, as below).
__device__ __forceinline__ void euler_flux(const double U[3], double f[3]) {
  const double u = U[1] * (1.0 / U[0]);
  const double p = (kGamma - 1.0) * (U[2] - 0.5 * U[1] * u);
  f[0] = U[1];
  f[1] = fma(U[1], u, p);
  f[2] = (U[2] + p) * u;
}

// Flux f(U) and wave speed |u| + c of a state, with one division (1/rho) and one square root.
__device__ __forceinline__ void euler_flux_speed(const double U[3], double f[3], double &speed) {
  const double r = 1.0 / U[0];
  const double u = U[1] * r;
  const double p = (kGamma - 1.0) * (U[2] - 0.5 * U[1] * u);
  f[0] = U[1];
  f[1] = fma(U[1], u, p);
  f[2] = (U[2] + p) * u;
  speed = fabs(u) + sqrt(kGamma * p * r);
}

// Local Lax-Friedrichs flux from the traces' states, fluxes and wave speeds.
__device__ __forceinline__ void euler_llf_from(const double UL[3], const double UR[3],
                                               const double fl[3], const double fr[3], double sl,
                                               double sr, double F[3]) {
  const double lam = fmax(sl, sr);
#pragma unroll
  for (int c = 0; c < 3; ++c) F[c] = 0.5 * (fl[c] + fr[c]) - 0.5 * lam * (UR[c] - UL[c]);
}

// AT value of the flux at PE face j (delay d.k > 0), stage s of the step whose ring slot is nm,
// from the ring [R][ns][3][P] of the face's fluxes.
__device__ __forceinline__ void euler_pe_flux(const Inst &I, const DelayAt &d, int j, int nm, int s,
                                              double F[3]) {
  const int P = I.P;
  for (int i = 0; i < d.qe; ++i) {
    const double ci = d.c[i];
    if (i && ci == 0.0) continue;
    int slot = nm - d.k - i;
    if (slot < 0) slot += I.R;
    const double2 *col = I.ring + ((size_t)slot * I.ns + s) * 3 * P + j;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double x = __dmul_rn(ci, col[(size_t)c * P].x);
      F[c] = i ? __dadd_rn(F[c], x) : x;
    }
  }
}

// Elements per warp of k_euler_stage: lanes 1 .. 30 own elements, lanes 0 and 31 hold their
// left and right neighbours, so every face flux of the warp is formed by the lanes together.
constexpr int kEulerLanes = 30;

template <int NP, int STAGE, bool FACES>
__global__ void __launch_bounds__(kTile) k_euler_stage(const Inst I, int rel, double *__restrict__ dst) {
  const int K = I.K;
  const size_t nd = (size_t)K * NP;
  const int lane = threadIdx.x & 31;
  const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int eraw = gw * kEulerLanes - 1 + lane;   // -1 .. K + 30
  const int ec = (int)(((long long)eraw + K) % K);
  const bool own = lane >= 1 && lane <= kEulerLanes && eraw < K;
  const int e = own ? eraw : K;   // K: not this lane's to write
  const double *vin = STAGE == 0 ? I.u : (STAGE == 1 ? I.v1 : I.v2);
  const StageConsts &C = I.sc[STAGE];
  double V[3][NP];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double *q = vin + c * nd + ec;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      V[c][i] = __ldg(q);
      q += K;
    }
  }
  const unsigned full = 0xffffffffu;
  // node fluxes, and the wave speeds of the two end nodes
  double f[3][NP], s0 = 0.0, sp = 0.0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const double Ui[3] = {V[0][i], V[1][i], V[2][i]};
    double fi[3];
    if (i == 0 || i == NP - 1) {
      double si;
      euler_flux_speed(Ui, fi, si);
      if (i == 0) s0 = si;
      if (i == NP - 1) sp = si;
    } else {
      euler_flux(Ui, fi);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c][i] = fi[c];
  }
  // left face: U^- with its flux and speed from the left neighbour's last node (the lane
  // below), U^+ this element's first node; the right face's flux from the lane above
  double VLm[3], V0[3], Vp[3], fLm[3], f0[3], fp[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    V0[c] = V[c][0];
    Vp[c] = V[c][NP - 1];
    f0[c] = f[c][0];
    fp[c] = f[c][NP - 1];
    VLm[c] = __shfl_up_sync(full, Vp[c], 1);
    fLm[c] = __shfl_up_sync(full, fp[c], 1);
  }
  const double sLm = __shfl_up_sync(full, sp, 1);
  double FL[3], FR[3];
  euler_llf_from(VLm, V0, fLm, f0, sLm, s0, FL);
  if (FACES && lane > 0) {
    // the lane of the element right of a PE face takes its flux: the owner stores it in the
    // ring, and a delayed one replaces it (the left element's lane below takes it as its FR)
    const int j = ec / I.Kpe;
    if (ec == j * I.Kpe) {
      const int64_t n = I.meta[0] + rel;
      const int nm = (int)(n % I.R);
      const DelayAt d = delay_at(I, j, n);
      if (own) {
        double2 *col = I.ring + ((size_t)nm * I.ns + STAGE) * 3 * I.P + j;
#pragma unroll
        for (int c = 0; c < 3; ++c) col[(size_t)c * I.P] = make_double2(FL[c], 0.0);
      }
      if (d.k > 0) euler_pe_flux(I, d, j, nm, STAGE, FL);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) FR[c] = __shfl_down_sync(full, FL[c], 1);
  if (e >= K) return;
  const double dt = I.dt;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double jl = __dsub_rn(f[c][0], FL[c]);
    const double jr = __dsub_rn(f[c][NP - 1], FR[c]);
    double u[NP];
    if (STAGE > 0) {
      const double *q = I.u + c * nd + e;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        u[i] = *q;
        q += K;
      }
    }
    double *o = dst + c * nd + e;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      double r = -I.QD[i * NP] * f[c][0];
#pragma unroll
      for (int j = 1; j < NP; ++j) r = fma(-I.QD[i * NP + j], f[c][j], r);
      r = fma(I.qlL[i], jl, r);
      r = fma(I.qlR[i], jr, r);
      double out = C.beta * fma(dt, r, V[c][i]);
      if (STAGE > 0) out = fma(C.alpha, u[i], out);
      *o = out;
      o += K;
    }
  }
}

// Sign of a non-NaN double from its bit pattern (-0 and +0 give 0).
__device__ __forceinline__ int bit_sign(long long b) { return b > 0 ? 1 : ((b << 1) != 0 ? -1 : 0); }

// minmod of 2 a1 and the used differences, halved (0 where the signs disagree). Signs,
// magnitudes and minima are taken on the IEEE bit patterns (integer pipe): for non-negative
// doubles the patterns order like the values.
__device__ __forceinline__ double limited_slope(double a1, double dp, double dm, bool use_p,
                                                bool use_m) {
  const long long mask = 0x7fffffffffffffffLL;
  const long long bt = __double_as_longlong(2.0 * a1);
  const int st = bit_sign(bt);
  long long mag = bt & mask;
  bool ok = st != 0;
  if (use_p) {
    const long long b = __double_as_longlong(dp);
    ok = ok && bit_sign(b) == st;
    const long long m = b & mask;
    mag = m < mag ? m : mag;
  }
  if (use_m) {
    const long long b = __double_as_longlong(dm);
    ok = ok && bit_sign(b) == st;
    const long long m = b & mask;
    mag = m < mag ? m : mag;
  }
  const double r = 0.5 * __longlong_as_double(mag);
  return ok ? (st > 0 ? r : -r) : 0.0;
}

template <int NP>
__device__ __forceinline__ double cell_average(const Inst &I, const double *v) {
  double a = I.lim.avg[0] * v[0];
#pragma unroll
  for (int j = 1; j < NP; ++j) a = fma(I.lim.avg[j], v[j], a);
  return a;
}

template <int NP>
__device__ __forceinline__ double first_moment(const Inst &I, const double *v) {
  double a = I.lim.p1[0] * v[0];
#pragma unroll
  for (int j = 1; j < NP; ++j) a = fma(I.lim.p1[j], v[j], a);
  return a;
}

// The limited element of values v (average a0, slope a1) between the neighbours' averages.
template <int NP>
__device__ __forceinline__ void limit_element(const Inst &I, const double *v, double a0, double a1,
                                              double dp, double dm, bool use_p, bool use_m,
                                              double keep, double *out) {
  double a1n = limited_slope(a1, dp, dm, use_p, use_m);
  if ((__double_as_longlong(a1) & 0x7fffffffffffffffLL) <= __double_as_longlong(keep)) a1n = a1;
  const bool change = a1n != a1;
#pragma unroll
  for (int i = 0; i < NP; ++i) out[i] = change ? fma(a1n, I.lim.xi[i], a0) : v[i];
}

template <int NP, bool PES>
__global__ void __launch_bounds__(kTile) k_euler_limit(const Inst I, const double *__restrict__ src,
                                                       double *__restrict__ dst) {
  const int K = I.K;
  const size_t nd = (size_t)K * NP;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const int ec = e < K ? e : K - 1;
  const bool edge = (lane == 31) || (ec + 1 >= K);
  const int fR = ec + 1 >= K ? 0 : ec + 1;
  const int fL = ec == 0 ? K - 1 : ec - 1;
  const bool use_m = !(PES && ec % I.Kpe == 0);
  const bool use_p = !(PES && (ec + 1) % I.Kpe == 0);
  const double keep = I.tvb_m * (I.dx * I.dx) * 0.5;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double v[NP], w[NP];
    const double *q = src + c * nd + ec;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      v[i] = __ldg(q);
      q += K;
    }
    const double a0 = cell_average<NP>(I, v);
    const double a1 = first_moment<NP>(I, v);
    double aL = __shfl_up_sync(0xffffffffu, a0, 1);
    double aR = __shfl_down_sync(0xffffffffu, a0, 1);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < NP; ++i) w[i] = __ldg(src + c * nd + (size_t)i * K + fL);
      aL = cell_average<NP>(I, w);
    }
    if (edge) {
#pragma unroll
      for (int i = 0; i < NP; ++i) w[i] = __ldg(src + c * nd + (size_t)i * K + fR);
      aR = cell_average<NP>(I, w);
    }
    if (e >= K) continue;
    limit_element<NP>(I, v, a0, a1, aR - a0, a0 - aL, use_p, use_m, keep, w);
    double *o = dst + c * nd + e;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      *o = w[i];
      o += K;
    }
  }
}

constexpr int kEulerThreads = 128;

// m steps of a small mesh in one launch. Four threads per element (eight at p = 4): node by
// node for the fluxes and wave speeds, then component by component for the face fluxes, the
// rows and the limiter, exchanged through shared memory. A warp's FP64 instruction holds its
// sub-partition's FP64 pipe for 64 clocks however many lanes are active, so at a warp or
// two per SM a step takes as long as one thread's FP64 instructions: about 57 a stage at p = 1
// in this form, about 155 with a whole element per thread (14.7 us a step below). A block
// owns EB - 2 H of its EB elements and forms the H on either side again (one per stage for the
// faces, one more for the limiter), so blocks need nothing from one another. Every element's
// arithmetic is that of k_euler_stage and k_euler_limit, so the results are theirs bit for bit,
// whatever the block or the split of a run into launches. A PE face's fluxes are kept in shared
// memory, the ring's levels before the launch (loaded at its start) and then the launch's own;
// the ring has kEulerSteps - 1 spare slots, so that no block overwrites a level that another
// still reads. Sod's problem on 1024 elements, ADG-AT2-RK2: 42 us a step as two stage and
// two limiter kernels (whose PE lanes recomputed the fluxes of delayed traces), 8.0 us so.
template <int NP, bool FACES, bool PES, bool LIM>
__global__ void __launch_bounds__(kEulerThreads)
    k_euler_steps(const __grid_constant__ Inst I, const double *__restrict__ uin,
                  double *__restrict__ uout, int rel, int m, int H) {
  constexpr int LPE = NP <= 4 ? 4 : 8, EB = kEulerThreads / LPE;
  __shared__ double Vs[3][NP][EB], fs[3][NP][EB], s0[EB], sp[EB], Fs[3][EB], as[3][EB];
  __shared__ unsigned char delay[FACES ? kEulerSteps : 1][EB];
  extern __shared__ double hist[];   // [levels][ns][3][EB], then the AT coefficients
  const int K = I.K, S = I.ns;
  const size_t nd = (size_t)K * NP;
  const int el = threadIdx.x / LPE, r = threadIdx.x - el * LPE;
  const int c = r;                    // component (r < 3)
  const int OWN = EB - 2 * H;
  const int eraw = (int)blockIdx.x * OWN - H + el;
  const bool own = el >= H && el < H + OWN && eraw < K;
  int e = eraw;
  if ((unsigned)e >= (unsigned)K) {
    e %= K;
    if (e < 0) e += K;
  }
  const int elL = el ? el - 1 : 0, elR = el + 1 < EB ? el + 1 : el;
  double V[NP], u[NP];
  if (r < 3) {
    load_elem<NP>(uin + c * nd, K, e, u);
#pragma unroll
    for (int i = 0; i < NP; ++i) Vs[c][i][el] = u[i];
  }
  const int j = e / I.Kpe;
  const bool face = FACES && r < 3 && e == j * I.Kpe;
  const bool use_m = !(PES && e == j * I.Kpe), use_p = !(PES && e + 1 == (j + 1) * I.Kpe);
  const double keep = I.tvb_m * (I.dx * I.dx) * 0.5;
  const double dt = I.dt;
  const int back = I.L - 1 + I.q - 1;   // levels before the current step that it can reach
  const int64_t n0 = FACES ? I.meta[0] + rel : 0;
  auto at = [&](int level, int s) -> double & {   // level: relative to n0
    return hist[(((level + back) * S + s) * 3 + c) * EB + el];
  };
  double *coef = hist + (back + m) * S * 3 * EB;
  if (FACES)
    for (int k = threadIdx.x; k < I.L * I.q * I.q; k += kEulerThreads) coef[k] = __ldg(I.coef + k);
  if (face) {
    const uint8_t *row = I.table + (n0 - I.meta[1]) * I.P + j;
    for (int t = c; t < m; t += 3) delay[t][el] = row[(size_t)t * I.P];
    for (int b = 1; b <= back && b <= n0; ++b) {
      const int slot = mod_step(n0 - b, I.R);
      for (int s = 0; s < S; ++s) at(-b, s) = I.ring[(((size_t)slot * S + s) * 3 + c) * I.P + j].x;
    }
  }
  __syncthreads();
  for (int t = 0; t < m; ++t) {
    // as delay_at: k <= n, order q' = min(q, n - k + 1)
    int dk = 0, qe = 0, nm = 0;
    const double *cf = nullptr;
    if (face) {
      const int64_t n = n0 + t;
      dk = (int)min((int64_t)delay[t][el], n);
      qe = (int)min((int64_t)I.q, n - dk + 1);
      cf = coef + (dk * I.q + qe - 1) * I.q;
      nm = mod_step(n, I.R);
    }
    if (r < 3) {
#pragma unroll
      for (int i = 0; i < NP; ++i) V[i] = u[i];
    }
    for (int s = 0; s < S; ++s) {
      const StageConsts &C = I.sc[s];
      if (r < NP) {   // node r
        const double Ui[3] = {Vs[0][r][el], Vs[1][r][el], Vs[2][r][el]};
        double fi[3], si;
        euler_flux_speed(Ui, fi, si);
#pragma unroll
        for (int k = 0; k < 3; ++k) fs[k][r][el] = fi[k];
        if (r == 0) s0[el] = si;
        if (r == NP - 1) sp[el] = si;
      }
      __syncthreads();
      if (r < 3) {
        const double lam = fmax(sp[elL], s0[el]);
        double F = 0.5 * (fs[c][NP - 1][elL] + fs[c][0][el]) -
                   0.5 * lam * (Vs[c][0][el] - Vs[c][NP - 1][elL]);
        if (face) {
          at(t, s) = F;
          if (own) I.ring[(((size_t)nm * S + s) * 3 + c) * I.P + j] = make_double2(F, 0.0);
          if (dk > 0) {
            F = __dmul_rn(cf[0], at(t - dk, s));
            for (int k = 1; k < qe; ++k)
              if (cf[k] != 0.0) F = __dadd_rn(F, __dmul_rn(cf[k], at(t - dk - k, s)));
          }
        }
        Fs[c][el] = F;
      }
      __syncthreads();
      double o[NP], a0 = 0.0, a1 = 0.0;
      if (r < 3) {
        double f[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) f[i] = fs[c][i][el];
        const double jl = __dsub_rn(f[0], Fs[c][el]);
        const double jr = __dsub_rn(f[NP - 1], Fs[c][elR]);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          double x = -I.QD[i * NP] * f[0];
#pragma unroll
          for (int k = 1; k < NP; ++k) x = fma(-I.QD[i * NP + k], f[k], x);
          x = fma(I.qlL[i], jl, x);
          x = fma(I.qlR[i], jr, x);
          o[i] = C.beta * fma(dt, x, V[i]);
          if (s > 0) o[i] = fma(C.alpha, u[i], o[i]);
        }
        if (LIM) {
          a0 = cell_average<NP>(I, o);
          a1 = first_moment<NP>(I, o);
          as[c][el] = a0;
        }
      }
      if (LIM) __syncthreads();
      if (r < 3) {
        if (LIM) {
          limit_element<NP>(I, o, a0, a1, as[c][elR] - a0, a0 - as[c][elL], use_p, use_m, keep, V);
        } else {
#pragma unroll
          for (int i = 0; i < NP; ++i) V[i] = o[i];
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) Vs[c][i][el] = V[i];
      }
      __syncthreads();
    }
    if (r < 3) {
#pragma unroll
      for (int i = 0; i < NP; ++i) u[i] = V[i];
    }
  }
  if (own && r < 3) {
#pragma unroll
    for (int i = 0; i < NP; ++i) uout[c * nd + (size_t)i * K + e] = u[i];
  }
}

template <int NP, int STAGE>
cudaError_t euler_stage_np(const Inst &I, int rel, double *dst, cudaStream_t s) {
  const int bs = stage_block(I.K);
  const long long threads = (long long)((I.K + kEulerLanes - 1) / kEulerLanes) * 32;
  const unsigned grid = (unsigned)((threads + bs - 1) / bs);
  if (I.async) k_euler_stage<NP, STAGE, true><<<grid, bs, 0, s>>>(I, rel, dst);
  else k_euler_stage<NP, STAGE, false><<<grid, bs, 0, s>>>(I, rel, dst);
  return cudaGetLastError();
}

template <int NP>
cudaError_t euler_stage(const Inst &I, int stage, int rel, double *dst, cudaStream_t s) {
  switch (stage) {
    case 0: return euler_stage_np<NP, 0>(I, rel, dst, s);
    case 1: return euler_stage_np<NP, 1>(I, rel, dst, s);
    default: return euler_stage_np<NP, 2>(I, rel, dst, s);
  }
}

template <int NP>
cudaError_t euler_limit(const Inst &I, const double *src, double *dst, cudaStream_t s) {
  const int bs = stage_block(I.K);
  const unsigned grid = (unsigned)((I.K + bs - 1) / bs);
  if (I.P > 1) k_euler_limit<NP, true><<<grid, bs, 0, s>>>(I, src, dst);
  else k_euler_limit<NP, false><<<grid, bs, 0, s>>>(I, src, dst);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_euler_stage(const Inst &I, int stage, int rel, double *dst, cudaStream_t s) {
  if (stage < 0 || stage >= I.ns || stage > 2) return cudaErrorInvalidValue;
  switch (I.Np) {
    case 2: return euler_stage<2>(I, stage, rel, dst, s);
    case 3: return euler_stage<3>(I, stage, rel, dst, s);
    case 4: return euler_stage<4>(I, stage, rel, dst, s);
    case 5: return euler_stage<5>(I, stage, rel, dst, s);
    default: return cudaErrorInvalidValue;
  }
}

namespace {
constexpr int euler_block(int Np) { return kEulerThreads / (Np <= 4 ? 4 : 8); }

// Halo of m steps of k_euler_steps and its dynamic shared memory.
int euler_halo(const Inst &I, int m) { return m * I.ns * (I.limiter ? 2 : 1); }
size_t euler_hist(const Inst &I, int m) {
  return I.async ? ((size_t)(I.L + I.q - 2 + m) * I.ns * 3 * euler_block(I.Np) + I.L * I.q * I.q) *
                       sizeof(double)
                 : 0;
}

template <int NP>
cudaError_t euler_steps(const Inst &I, const double *uin, double *uout, int rel, int m,
                        cudaStream_t s) {
  const int H = euler_halo(I, m), own = euler_block(NP) - 2 * H;
  const unsigned g = (unsigned)((I.K + own - 1) / own);
  auto go = [&](auto kernel) {
    kernel<<<g, kEulerThreads, euler_hist(I, m), s>>>(I, uin, uout, rel, m, H);
    return cudaGetLastError();
  };
  if (I.async)
    return I.limiter ? go(k_euler_steps<NP, true, true, true>) : go(k_euler_steps<NP, true, true, false>);
  if (I.P > 1 && I.limiter) return go(k_euler_steps<NP, false, true, true>);
  return I.limiter ? go(k_euler_steps<NP, false, false, true>) : go(k_euler_steps<NP, false, false, false>);
}
}  // namespace

// A launch costs about 2.5 us; a block's stage holds its SM's FP64 pipes (one warp each) for 64
// clocks per instruction of a thread, an element's stage and limiter in the two kernels of a
// stage its warp's pipe for as many of a whole element. The number of steps with the least
// estimated time; 0: the stage and limiter kernels.
int euler_steps_per_launch(const Inst &I) {
  const double sms = sm_count(), clk = 64 / 1900.0 * I.ns;
  const int NP = I.Np, lim = I.limiter ? 2 * NP + 5 : 0;
  const double thread = clk * (35 + NP * (NP + 4) + lim);
  const double element = clk * (30 * NP + 3 * (5 + NP * (NP + 4) + lim));
  double best = 2.5 * I.ns * (I.limiter ? 2 : 1) + element * std::max(1.0, I.K / 30.0 / (4 * sms));
  int pick = 0;
  for (int m = 1; m <= kEulerSteps; ++m) {
    const int own = euler_block(NP) - 2 * euler_halo(I, m);
    if (own < 1 || euler_hist(I, m) > 32 * 1024) break;
    const double us = 2.5 / m + thread * std::max(1.0, std::ceil((double)I.K / own) / sms);
    if (us < best) {
      best = us;
      pick = m;
    }
  }
  return pick;
}

cudaError_t launch_euler_steps(const Inst &I, const double *uin, double *uout, int rel, int m,
                               cudaStream_t s) {
  if (uin == uout || m < 1 || m > kEulerSteps ||
      euler_block(I.Np) - 2 * euler_halo(I, m) < 1)
    return cudaErrorInvalidValue;
  switch (I.Np) {
    case 2: return euler_steps<2>(I, uin, uout, rel, m, s);
    case 3: return euler_steps<3>(I, uin, uout, rel, m, s);
    case 4: return euler_steps<4>(I, uin, uout, rel, m, s);
    case 5: return euler_steps<5>(I, uin, uout, rel, m, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_euler_limit(const Inst &I, const double *src, double *dst, cudaStream_t s) {
  if (src == dst) return cudaErrorInvalidValue;
  switch (I.Np) {
    case 2: return euler_limit<2>(I, src, dst, s);
    case 3: return euler_limit<3>(I, src, dst, s);
    case 4: return euler_limit<4>(I, src, dst, s);
    case 5: return euler_limit<5>(I, src, dst, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace adg
