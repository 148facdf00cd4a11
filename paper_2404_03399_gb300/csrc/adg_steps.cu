// Staged SSP-RK3 advection on small meshes: several steps per launch.
#include <algorithm>
#include <cmath>

#include "adg_device.cuh"

namespace adg {
namespace {

constexpr int kAdvThreads = 128;

// m SSP-RK3 steps of advection in one launch, for the meshes whose staged steps are launches
// and little else. One thread per node: a warp's FP64 instruction holds its sub-partition's
// FP64 pipe for 64 clocks however many lanes are active, so with a warp or two per SM the time
// of a stage is the number of FP64 instructions of one thread, Np + 1 for a node's row
// instead of Np (Np + 2) for an element's (that form took 4.5 us a step below).
// A block owns EB - 1 - 3 m of its EB = 128 / Np elements and forms 3 m on the upwind side
// again (one per stage) and, for the value at the last PE face, one on the other side, so
// blocks need nothing from one another; the stages exchange values through shared memory. The
// arithmetic of a node is that of stage_body_halo, in FP64, so the results are the staged
// kernels' bit for bit, whatever the block or the split of a run into launches. A face's
// traces are kept in shared memory: the ring's levels before the launch, loaded at its start, then the launch's own; the
// ring has spare slots (kAdvSteps - 1), so that no block overwrites a level that another still
// reads. K = 64, p = 2, ADG-AT3: 10.3 us a step as three launches, 2.6 us with m = 8.
template <int NP, int DIR, bool FACES>
__global__ void __launch_bounds__(kAdvThreads) k_adv_steps(const __grid_constant__ Inst I,
                                                           const double *__restrict__ uin,
                                                           double *__restrict__ uout, int rel,
                                                           int m) {
  constexpr int EB = kAdvThreads / NP;
  __shared__ double vs[2][EB][NP];
  __shared__ double V[kStages][EB];        // delayed values of the elements' left faces
  __shared__ unsigned char late[EB + 1];   // a PE face with a delay at this step
  __shared__ unsigned char delay[FACES ? kAdvSteps : 1][EB];
  extern __shared__ double hist[];         // [levels][3][EB], then the AT coefficients
  const int K = I.K;
  const int el = threadIdx.x / NP, i = threadIdx.x - el * NP;   // element of the block, node
  const bool in = el < EB;
  const int OWN = EB - 1 - 3 * m;
  const int first = DIR > 0 ? 3 * m : 0;   // the first owned element
  const int eraw = (int)blockIdx.x * OWN - first + el;
  const bool own = in && el >= first && el < first + OWN && eraw < K;
  int e = eraw;
  if ((unsigned)e >= (unsigned)K) {
    e %= K;
    if (e < 0) e += K;
  }
  const int j = e / I.Kpe;
  const bool face = FACES && in && e == j * I.Kpe;
  const bool faceR = FACES && el + 1 < EB && (e + 1 == (j + 1) * I.Kpe);
  const int back = I.L - 1 + I.q - 1;   // levels before the current step that it can reach
  const int64_t n0 = FACES ? I.meta[0] + rel : 0;
  auto at = [&](int level, int s) -> double & {   // level: relative to n0
    return hist[((level + back) * kStages + s) * EB + el];
  };
  double A[kStages][NP], lL[kStages], lR[kStages];
#pragma unroll
  for (int s = 0; s < kStages; ++s) {
#pragma unroll
    for (int k = 0; k < NP; ++k) A[s][k] = I.sc[s].A[i * NP + k];
    lL[s] = I.sc[s].lL[i];
    lR[s] = I.sc[s].lR[i];
  }
  double u = in ? __ldg(uin + (size_t)i * K + e) : 0.0;
  if (in) vs[0][el][i] = u;
  const int nc = I.L * I.q * I.q;
  double *coef = hist + (back + m) * kStages * EB;
  if (FACES)
    for (int k = threadIdx.x; k < nc; k += kAdvThreads) coef[k] = __ldg(I.coef + k);
  if (face) {   // node i loads the steps' delays and the levels i + 1, i + 1 + NP, ..
    const uint8_t *row = I.table + (n0 - I.meta[1]) * I.P + j;
    for (int t = i; t < m; t += NP) delay[t][el] = row[(size_t)t * I.P];
    for (int b = 1 + i; b <= back && b <= n0; b += NP) {
      const double2 *col = I.ring + (size_t)mod_step(n0 - b, I.R) * kStages * I.P + j;
#pragma unroll
      for (int s = 0; s < kStages; ++s) at(-b, s) = DIR > 0 ? col[s * I.P].x : col[s * I.P].y;
    }
  }
  if (FACES && in && i == 0) late[el] = 0;
  __syncthreads();
  int buf = 0;
  for (int t = 0; t < m; ++t) {
    int slot = 0;
    if (FACES) {
      if (face) {   // node i forms the values of stages i, i + NP, ..
        // as delay_at: k <= n, order q' = min(q, n - k + 1)
        const int64_t n = n0 + t;
        const int dk = (int)min((int64_t)delay[t][el], n);
        const int qe = (int)min((int64_t)I.q, n - dk + 1);
        const double *c = coef + (dk * I.q + qe - 1) * I.q;
        slot = mod_step(n, I.R);
        if (i == 0) late[el] = dk > 0;
        if (dk > 0) {
          for (int s = i; s < kStages; s += NP) {
            double x = __dmul_rn(c[0], at(t - dk, s));
            for (int k = 1; k < qe; ++k)
              if (c[k] != 0.0) x = __dadd_rn(x, __dmul_rn(c[k], at(t - dk - k, s)));
            V[s][el] = x;
          }
        }
      }
      __syncthreads();
    }
    const bool lateL = FACES && face && late[el], lateR = FACES && faceR && late[el + 1];
#pragma unroll
    for (int s = 0; s < kStages; ++s) {
      const double alpha = I.sc[s].alpha;
      if (in) {
        double v[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k) v[k] = vs[buf][el][k];
        // the neighbour's trace on the upwind side (out of the block: not owned, any value)
        const double nb = DIR > 0 ? vs[buf][el ? el - 1 : 0][NP - 1]
                                  : vs[buf][el + 1 < EB ? el + 1 : el][0];
        double acc = s == 0 ? A[s][0] * v[0] : fma(A[s][0], v[0], alpha * u);
#pragma unroll
        for (int k = 1; k < NP; ++k) acc = fma(A[s][k], v[k], acc);
        acc = DIR > 0 ? fma(lL[s], v[0] - nb, acc) : fma(lR[s], v[NP - 1] - nb, acc);
        // synchronous minus delayed values of the two faces
        if (lateL) acc = fma(lL[s], (DIR > 0 ? nb : v[0]) - V[s][el], acc);
        if (lateR) acc = fma(lR[s], (DIR > 0 ? v[NP - 1] : nb) - V[s][el + 1], acc);
        if (face && i == 0) {   // this level's trace
          const double T = DIR > 0 ? nb : v[0];
          at(t, s) = T;
          if (own)
            I.ring[((size_t)slot * kStages + s) * I.P + j] =
                DIR > 0 ? make_double2(T, 0.0) : make_double2(0.0, T);
        }
        vs[buf ^ 1][el][i] = acc;
        if (s == kStages - 1) u = acc;
      }
      buf ^= 1;
      __syncthreads();
    }
  }
  if (own) uout[(size_t)i * K + e] = u;
}

size_t adv_hist(const Inst &I, int m) {
  return I.async ? ((size_t)(I.L + I.q - 2 + m) * kStages * (kAdvThreads / I.Np) + I.L * I.q * I.q) *
                       sizeof(double)
                 : 0;
}

template <int NP>
cudaError_t adv_steps(const Inst &I, const double *uin, double *uout, int rel, int m,
                      cudaStream_t s) {
  const int own = kAdvThreads / NP - 1 - 3 * m;
  const unsigned g = (unsigned)((I.K + own - 1) / own);
  auto go = [&](auto kernel) {
    kernel<<<g, kAdvThreads, adv_hist(I, m), s>>>(I, uin, uout, rel, m);
    return cudaGetLastError();
  };
  if (I.a >= 0.0) return I.async ? go(k_adv_steps<NP, 1, true>) : go(k_adv_steps<NP, 1, false>);
  return I.async ? go(k_adv_steps<NP, -1, true>) : go(k_adv_steps<NP, -1, false>);
}

}  // namespace

// A launch costs about 2.5 us; a block's step holds its SM's FP64 pipes (one warp each) for 64
// clocks per instruction of a thread (3 (Np + 2) and some 10 of the faces). The number of steps
// with the least estimated time, against three launches a step with 30 of 32 lanes, whose
// threads take whole elements.
int adv_steps_per_launch(const Inst &I) {
  const double sms = sm_count(), clk = 64 / 1900.0;
  double best = 7.5 + 3 * I.Np * (I.Np + 2) * clk * std::max(1.0, I.K / 30.0 / (4 * sms));
  int pick = 0;
  for (int m = 1; m <= kAdvSteps; ++m) {
    const int own = kAdvThreads / I.Np - 1 - 3 * m;
    if (own < 1 || adv_hist(I, m) > 40 * 1024) break;
    const double us = 2.5 / m + (3 * (I.Np + 2) + (I.async ? 10 : 0)) * clk *
                                    std::max(1.0, std::ceil((double)I.K / own) / sms);
    if (us < best) {
      best = us;
      pick = m;
    }
  }
  return pick;
}

cudaError_t launch_adv_steps(const Inst &I, const double *uin, double *uout, int rel, int m,
                             cudaStream_t s) {
  if (uin == uout || m < 1 || m > kAdvSteps || kAdvThreads / I.Np - 1 - 3 * m < 1) return cudaErrorInvalidValue;
  switch (I.Np) {
    case 2: return adv_steps<2>(I, uin, uout, rel, m, s);
    case 3: return adv_steps<3>(I, uin, uout, rel, m, s);
    case 4: return adv_steps<4>(I, uin, uout, rel, m, s);
    case 5: return adv_steps<5>(I, uin, uout, rel, m, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace adg
