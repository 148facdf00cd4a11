// Inviscid Burgers, SSP-RK3: one kernel per step, the three stages in registers.
#include "adg_bfp.cuh"
#include "adg_device.cuh"

namespace adg {
namespace {

constexpr int kHalo = 3;   // elements a step's stages read on either side (one per stage)

// A warp's 32 consecutive elements: the first and last kHalo are the neighbours' (periodic),
// formed again so that warps need nothing from one another. own: written by this warp.
constexpr int kOwn = 32 - 2 * kHalo;

__device__ __forceinline__ int warp_element(int K, int warp, int lane, bool &own) {
  int e = warp * kOwn - kHalo + lane;
  own = lane >= kHalo && lane < kHalo + kOwn && e < K;
  if ((unsigned)e >= (unsigned)K) {
    e %= K;
    if (e < 0) e += K;
  }
  return e;
}

// The delayed / AT flux of PE face j at stage s of step n (k = d.k > 0) from the ring, whose
// entries hold the face's flux of each level.
__device__ __forceinline__ double ring_flux(const Inst &I, const DelayAt &d, int j, int nm, int s) {
  double V = 0.0;
  for (int i = 0; i < d.qe; ++i) {
    int sl = nm - d.k - i;
    if (sl < 0) sl += I.R;
    const double x = __dmul_rn(d.c[i], I.ring[((size_t)sl * kStages + s) * I.P + j].x);
    V = i ? __dadd_rn(V, x) : x;
  }
  return V;
}

// The step in FP64 (warps that the integer path does not take): the stages of the staged
// kernels, with the delayed fluxes sV[stage][lane] at PE faces (pe: the element's left face is
// one; late: its flux is a delayed one).
template <int NP, bool FACES, bool REC>
__device__ __noinline__ void burgers_step_fp64(const Inst &I, int warp, const double *uin,
                                               double *uout, double *r1, double *r2, int nm,
                                               const double (*sV)[32], bool pe, bool late) {
  const int K = I.K;
  const int lane = threadIdx.x & 31;
  bool own;
  const int e = warp_element(K, warp, lane, own);
  const unsigned full = 0xffffffffu;
  double u[NP], v[NP];
  load_elem<NP>(uin, K, e, u);
#pragma unroll
  for (int i = 0; i < NP; ++i) v[i] = u[i];
#pragma unroll
  for (int s = 0; s < kStages; ++s) {
    const StageConsts &C = I.sc[s];
    double FL = num_flux<1>(0.0, __shfl_up_sync(full, v[NP - 1], 1), v[0]);
    if (FACES && pe) {
      if (own) I.ring[((size_t)nm * kStages + s) * I.P + e / I.Kpe] = make_double2(FL, 0.0);
      if (late) FL = sV[s][lane];
    }
    const double FR = __shfl_down_sync(full, FL, 1);
    const double jL = __dsub_rn(phys_flux<1>(0.0, v[0]), FL);
    const double jR = __dsub_rn(phys_flux<1>(0.0, v[NP - 1]), FR);
    double g[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) g[i] = v[i] * v[i];
    double *o = s == 2 ? uout : (REC ? (s == 0 ? r1 : r2) : nullptr);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      double acc = s == 0 ? v[i] : fma(C.beta, v[i], C.alpha * u[i]);
#pragma unroll
      for (int k = 0; k < NP; ++k) acc = fma(C.A[i * NP + k], g[k], acc);
      v[i] = fma(C.lR[i], jR, fma(C.lL[i], jL, acc));
      if (o && own) o[(size_t)i * K + e] = v[i];
    }
  }
}

// One SSP-RK3 step of inviscid Burgers. Warp w owns 26 elements and forms three more on
// either side, so the three stages run in registers with shuffles for the face values and no
// barrier, and u is read and written once per step (three launches and eight field passes
// before). The stage operator
//   dt L(v)_i = sum_j W_ij v_j^2 + a_i F_L + b_i F_R
// (W = c2/2 (D + M^-1 e_0 e_0^T - M^-1 e_p e_p^T), a = -c2 M^-1 e_0, b = c2 M^-1 e_p) maps the
// even part of (v^2, faces) to the odd part and back, since the nodes are symmetric, so it is
// applied to sums and differences of mirrored nodes: 17 products instead of 35 at p = 4
// (BurgersFixed). REC also writes the stage inputs v1, v2 (recorded sweeps of the gradient).
// Bound by instruction issue (integer). K = 2^20, p = 4, ADG-AT2: 0.50 ms a step as three FP64
// stage kernels (80% of the FP64 pipe), 0.078 ms so; K = 10125, p = 2: 14.5 -> 5.3 us, where
// the launch and the dependent loads of the delays and ring levels are what is left. Two
// elements per thread (58 of 64 owned, 128 registers) took 0.089 ms and 7.0 us.
template <int NP, bool FACES, bool REC>
__global__ void __launch_bounds__(128) k_burgers_step(const __grid_constant__ Inst I,
                                                      const double *__restrict__ uin,
                                                      double *__restrict__ uout,
                                                      double *__restrict__ r1,
                                                      double *__restrict__ r2, int rel) {
  constexpr int HP = NP / 2, MID = NP % 2;   // mirrored pairs, middle node
  __shared__ double sV_[FACES ? 4 * kStages : 1][32];
  pdl_wait();
  pdl_trigger();
  const int K = I.K;
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if ((int64_t)warp * kOwn >= K) return;
  const unsigned full = 0xffffffffu;
  bool own;
  const int e = warp_element(K, warp, lane, own);
  double ud[NP];
  load_elem<NP>(uin, K, e, ud);

  // a PE face on the left of this lane's element, and its delayed fluxes
  bool pe = false, late = false;
  int nm = 0;
  double (*sV)[32] = sV_ + (FACES ? (threadIdx.x >> 5) * kStages : 0);
  int vmax = 0;   // largest high word of a delayed flux
  if (FACES) {
    const int j = e / I.Kpe;
    const int64_t n = I.meta[0] + rel;
    nm = (int)(n % I.R);
    pe = e == j * I.Kpe;
    if (pe) {
      const DelayAt d = delay_at(I, j, n);
      late = d.k > 0;
      if (late) {
#pragma unroll
        for (int s = 0; s < kStages; ++s) {
          const double V = ring_flux(I, d, j, nm, s);
          sV[s][lane] = V;
          vmax = max(vmax, __double2hiint(V) & 0x7fffffff);
        }
      }
    }
  }

  // the warp's scale, and whether the integer path takes it
  int hi = 0;
  unsigned lo = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    hi = max(hi, __double2hiint(ud[i]) & 0x7fffffff);
    lo |= (unsigned)__double2loint(ud[i]);
  }
  const int be = __reduce_max_sync(full, hi) >> 20;
  const int E = be - 1022;              // |u| < 2^E
  const int d0 = -(I.bf.sc + E + 1);    // operator sums -> value units
  bool bad = be < kBfMinE || be > kBfMaxE || d0 < -2 || !I.bf.ok;
  bad = bad || (hi ? (hi >> 20) < be - kBfSpan : lo != 0);
  if (FACES) bad = bad || (vmax >> 20) > 2 * E + 1023;   // a delayed flux of 2^(2E + 1) or more

  if (!__any_sync(full, bad)) {
    const BurgersFixed &B = I.bf;
    const int sg = 2 * E - 56;   // unit of the squares and fluxes
    long long u[NP], v[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) v[i] = u[i] = bf_from(ud[i], be);
    unsigned long long mag = 0;
#pragma unroll
    for (int s = 0; s < kStages; ++s) {
      // shift of the operator's sums: stage 1 takes a quarter of them, stage 2 (inside the
      // sum divided by 3) twice
      int d = s == 0 ? d0 : (s == 1 ? d0 + 2 : d0 - 1);
      d = d > 60 ? 60 : d;
      const long long half = d > 0 ? 1ll << (d - 1) : 0;
      long long G[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        int xh, xl;
        fx_split(v[i], xh, xl);
        G[i] = bf_square(xh, xl);
      }
      const long long vl = __shfl_up_sync(full, v[NP - 1], 1);
      const long long gl = __shfl_up_sync(full, G[NP - 1], 1);
      long long FL = bf_llf(vl, v[0], gl, G[0]);
      if (FACES && pe) {
        if (own)
          I.ring[((size_t)nm * kStages + s) * I.P + e / I.Kpe] = make_double2(bf_to(FL, sg), 0.0);
        if (late) FL = bf_from(sV[s][lane], 2 * E + 1023);
      }
      const long long FR = __shfl_down_sync(full, FL, 1);
      // sums and differences of mirrored nodes, and of the faces
      int dh[HP + 1], dl[HP + 1], sh[HP + MID + 1], sl[HP + MID + 1];
#pragma unroll
      for (int j = 0; j < HP; ++j) {
        fx_split(G[j] - G[NP - 1 - j], dh[j], dl[j]);
        fx_split(G[j] + G[NP - 1 - j], sh[j], sl[j]);
      }
      if (MID) fx_split(G[HP], sh[HP], sl[HP]);
      fx_split(FL - FR, dh[HP], dl[HP]);
      fx_split(FL + FR, sh[HP + MID], sl[HP + MID]);
#pragma unroll
      for (int i = 0; i < HP + MID; ++i) {
        FxAcc a;
        a.a = half;
#pragma unroll
        for (int j = 0; j <= HP; ++j) fx_mac(a, B.S[i][j], dh[j], dl[j]);
        const long long odd = fx_round(a);
        long long even = 0;
        if (i < HP) {
          FxAcc b;
#pragma unroll
          for (int j = 0; j <= HP + MID; ++j) fx_mac(b, B.D[i][j], sh[j], sl[j]);
          even = fx_round(b);
        }
#pragma unroll
        for (int m = 0; m < (i < HP ? 2 : 1); ++m) {
          const int k = m ? NP - 1 - i : i;
          const long long r = m ? odd - even : odd + even;
          if (d < 0 && (fx_mag(r) >> (kBfTop + d))) mag |= 1ull << kBfTop;
          const long long x = bf_shift(r, d);
          if (s == 0) {
            v[k] += x;
          } else if (s == 1) {
            v[k] = ((3 * u[k] + v[k] + 2) >> 2) + x;
          } else {
            const long long T = u[k] + 2 * v[k] + x;
            mag |= fx_mag(T) >> 2;   // below 2^60: its high limb fits 32 bits
            int th, tl;
            fx_split(T, th, tl);
            FxAcc c;
            fx_mac(c, make_int2(kThirdHi, kThirdLo), th, tl);
            v[k] = fx_round(c);
          }
          mag |= fx_mag(v[k]);
        }
      }
      if (REC && s < 2 && own) {
        double *o = s == 0 ? r1 : r2;
#pragma unroll
        for (int i = 0; i < NP; ++i) o[(size_t)i * K + e] = bf_to(v[i], E - 57);
      }
    }
    if (!__any_sync(full, (mag >> kBfTop) != 0)) {
      if (own) {
#pragma unroll
        for (int i = 0; i < NP; ++i) uout[(size_t)i * K + e] = bf_to(v[i], E - 57);
      }
      return;
    }
  }
  burgers_step_fp64<NP, FACES, REC>(I, warp, uin, uout, r1, r2, nm, sV, pe, late);
}

// One-warp blocks while the mesh gives fewer than 16 warps per SM (they spread evenly).
template <int NP>
cudaError_t burgers_np(const Inst &I, const double *uin, double *uout, double *r1, double *r2,
                       int rel, cudaStream_t s, bool pdl) {
  const int64_t warps = ((int64_t)I.K + kOwn - 1) / kOwn;
  const int bs = warps < 16 * sm_count() ? 32 : 128;
  const dim3 g((unsigned)((warps * 32 + bs - 1) / bs)), b(bs);
  auto go = [&](auto kernel) { return launch_maybe_pdl(kernel, g, b, s, pdl, I, uin, uout, r1, r2, rel); };
  if (r1) return I.async ? go(k_burgers_step<NP, true, true>) : go(k_burgers_step<NP, false, true>);
  return I.async ? go(k_burgers_step<NP, true, false>) : go(k_burgers_step<NP, false, false>);
}

}  // namespace

cudaError_t launch_burgers_step(const Inst &I, const double *uin, double *uout, double *r1,
                                double *r2, int rel, cudaStream_t s, bool pdl) {
  if (uin == uout) return cudaErrorInvalidValue;
  switch (I.Np) {
    case 2: return burgers_np<2>(I, uin, uout, r1, r2, rel, s, pdl);
    case 3: return burgers_np<3>(I, uin, uout, r1, r2, rel, s, pdl);
    case 4: return burgers_np<4>(I, uin, uout, r1, r2, rel, s, pdl);
    case 5: return burgers_np<5>(I, uin, uout, r1, r2, rel, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace adg
