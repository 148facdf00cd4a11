// Burgers: one kernel per step (every RK scheme, inviscid or viscous) and one per step of the
// discrete adjoint (inviscid, SSP-RK3), the stages in registers.
#include "adg_bfp.cuh"
#include "adg_device.cuh"

namespace adg {
namespace {

constexpr int kHalo = kStages;   // elements an SSP-RK3 step's stages read on either side
constexpr int kOwn = 32 - 2 * kHalo;

// A warp's 32 consecutive elements: the first H and the last HR are the neighbours' (periodic),
// formed again so that warps need nothing from one another: one on either side per stage (and
// one more on the right for a delayed uhat at the last element's right face, viscous Burgers).
// own: written by this warp.
__device__ __forceinline__ int warp_element(int K, int warp, int lane, int H, int HR, bool &own) {
  int e = warp * (32 - H - HR) - H + lane;
  own = lane >= H && lane < 32 - HR && e < K;
  if ((unsigned)e >= (unsigned)K) {
    e %= K;
    if (e < 0) e += K;
  }
  return e;
}

// Face quantities of a stage with a delayed / AT value at PE faces: the flux, and for viscous
// Burgers uhat = u^- and qhat = q^+ (kept as y = -2 nu q^+).
template <bool VISC>
constexpr int kFaceVals = VISC ? 3 : 1;

// The delay of PE face j at step n and its AT coefficients, from the step and the first row of
// the delay table as the host knows them (one load ahead of the coefficients and the ring).
__device__ __forceinline__ DelayAt step_delay(const Inst &I, int j, int64_t n, int64_t tbase) {
  int64_t k = I.table[(n - tbase) * I.P + j];
  if (k > n) k = n;
  const int64_t qe = n - k + 1 < I.q ? n - k + 1 : I.q;
  return {(int)k, (int)qe, I.coef + ((size_t)k * I.q + (qe - 1)) * I.q};
}

// The delayed / AT values of PE face j (d.k > 0) at stages s0 .. s0 + NS - 1, NV of them each (the
// flux, u^-, y), into V[value * S + stage][lane]; every level's load is issued before any is
// used.
template <int NV, int NS>
__device__ __forceinline__ void ring_sums(const Inst &I, const DelayAt &d, int j, int nm, int S, int s0,
                                          double (*V)[32], int &fmax, int &umax) {
  const int lane = threadIdx.x & 31;
  double c[kMaxQ], x[NS][NV][kMaxQ];
#pragma unroll
  for (int i = 0; i < kMaxQ; ++i) {
    int sl = nm - d.k - i;
    if (sl < 0) sl += I.R;
    const bool use = i < d.qe;
    c[i] = use ? d.c[i] : 0.0;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const size_t at = ((size_t)sl * I.ns + s0 + s) * I.P + j;
      x[s][0][i] = use ? I.ring[at].x : 0.0;
      if constexpr (NV == 3) {
        x[s][1][i] = use ? I.ring[at].y : 0.0;
        x[s][2][i] = use ? I.ringq[at] : 0.0;
      }
    }
  }
#pragma unroll
  for (int s = 0; s < NS; ++s)
#pragma unroll
    for (int w = 0; w < NV; ++w) {
      double v = __dmul_rn(c[0], x[s][w][0]);
#pragma unroll
      for (int i = 1; i < kMaxQ; ++i)
        if (i < d.qe) v = __dadd_rn(v, __dmul_rn(c[i], x[s][w][i]));
      V[w * S + s0 + s][lane] = v;
      const int h = __double2hiint(v) & 0x7fffffff;
      if (w == 0) fmax = max(fmax, h);
      if (w == 1) umax = max(umax, h);
    }
}

// Fields of a step and what it writes besides.
struct StepArgs {
  const double *uin;
  double *uout;
  double *r1, *r2;   // REC: the inputs of stages 1 and 2
  int64_t n, tbase;   // the step, and the first step of the delay table
  int H, HR;
};

// The step in FP64 (warps that the integer path does not take): stage by stage in the staged
// kernels' arithmetic, with the delayed values sV[value * ns + stage][lane] at PE faces (pe:
// the element's left face is one; late: its values are delayed ones).
template <int NP, bool FACES, bool REC, bool VISC, bool LS>
__device__ __noinline__ void burgers_step_fp64(const Inst &I, const StepArgs &A, int warp, int nm,
                                               const double (*sV)[32], bool pe, bool late) {
  const int K = I.K, S = LS ? I.ns : kStages;
  const int lane = threadIdx.x & 31;
  bool own;
  const int e = warp_element(K, warp, lane, A.H, A.HR, own);
  const unsigned full = 0xffffffffu;
  double u[NP], v[NP];   // u: u^n, or dU of a 2N scheme
  load_elem<NP>(A.uin, K, e, v);
#pragma unroll
  for (int i = 0; i < NP; ++i) u[i] = LS ? 0.0 : v[i];
  for (int s = 0; s < S; ++s) {
    const StageConsts &C = I.sc[LS ? 0 : s];
    const double vl = __shfl_up_sync(full, v[NP - 1], 1);
    double FL = llf_flux(vl, v[0]);
    const size_t at = FACES && pe ? ((size_t)nm * I.ns + s) * I.P + e / I.Kpe : 0;
    if (FACES && pe) {
      if (own) I.ring[at] = make_double2(FL, vl);
      if (late) FL = sV[s][lane];
    }
    double q[NP], jqL = 0.0, jqR = 0.0;
    if (VISC) {
      const double uL = FACES && late ? sV[S + s][lane] : vl;
      const double uN = __shfl_down_sync(full, uL, 1);
      const double uR = FACES && lane < 31 ? uN : v[NP - 1];   // v_p but at delayed faces
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        double acc = I.QD[i * NP] * v[0];
#pragma unroll
        for (int k = 1; k < NP; ++k) acc = fma(I.QD[i * NP + k], v[k], acc);
        acc = fma(I.qlL[i], uL - v[0], acc);
        q[i] = fma(I.qlR[i], uR - v[NP - 1], acc);
      }
      double qL = q[0];
      if (FACES && pe) {
        if (own) I.ringq[at] = -2.0 * I.nu * q[0];
        if (late) qL = sV[2 * S + s][lane] / (-2.0 * I.nu);
      }
      jqL = qL - q[0];
      jqR = __shfl_down_sync(full, qL, 1) - q[NP - 1];
    }
    const double FR = __shfl_down_sync(full, FL, 1);
    const double jL = __dsub_rn(burgers_flux(v[0]), FL);
    const double jR = __dsub_rn(burgers_flux(v[NP - 1]), FR);
    double g[NP], out[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) g[i] = v[i] * v[i];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      double acc = LS ? I.lsA[s] * u[i] : (s == 0 ? v[i] : fma(C.beta, v[i], C.alpha * u[i]));
#pragma unroll
      for (int k = 0; k < NP; ++k) acc = fma(C.A[i * NP + k], g[k], acc);
      acc = fma(C.lR[i], jR, fma(C.lL[i], jL, acc));
      if (VISC) {
        double vq = C.A[i * NP] * q[0];
#pragma unroll
        for (int k = 1; k < NP; ++k) vq = fma(C.A[i * NP + k], q[k], vq);
        acc = fma(I.nu, fma(C.lL[i], jqL, fma(C.lR[i], jqR, -2.0 * vq)), acc);
      }
      out[i] = acc;
    }
    double *o = s == S - 1 ? A.uout : (REC ? (s == 0 ? A.r1 : A.r2) : nullptr);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (LS) {
        u[i] = out[i];
        v[i] = fma(I.lsB[s], out[i], v[i]);
      } else {
        v[i] = out[i];
      }
      if (o && own) o[(size_t)i * K + e] = v[i];
    }
  }
}

// The operator on mirrored nodes (BurgersFixed): sums of the rows i and p - i, odd[i] + even[i]
// and odd[i] - even[i], of node values g (|g| < 2^59) and face values FL, FR (|.| < 2^59),
// with `half` added to each (a rounding constant of the shift that follows).
template <int NP>
__device__ __forceinline__ void burgers_operator(const BurgersFixed &B, const long long *g,
                                                 long long FL, long long FR, long long half,
                                                 long long *out) {
  constexpr int HP = NP / 2, MID = NP % 2;   // mirrored pairs, middle node
  int dh[HP + 1], dl[HP + 1], sh[HP + MID + 1], sl[HP + MID + 1];
#pragma unroll
  for (int j = 0; j < HP; ++j) {
    fx_split(g[j] - g[NP - 1 - j], dh[j], dl[j]);
    fx_split(g[j] + g[NP - 1 - j], sh[j], sl[j]);
  }
  if (MID) fx_split(g[HP], sh[HP], sl[HP]);
  fx_split(FL - FR, dh[HP], dl[HP]);
  fx_split(FL + FR, sh[HP + MID], sl[HP + MID]);
#pragma unroll
  for (int i = 0; i < HP + MID; ++i) {
    FxAcc a{half, B.rS[i]};
#pragma unroll
    for (int j = 0; j <= HP; ++j) fx_mac(a, B.S[i][j], dh[j], dl[j]);
    const long long odd = fx_round(a);
    if (i < HP) {
      FxAcc b{0, B.rD[i]};
#pragma unroll
      for (int j = 0; j <= HP + MID; ++j) fx_mac(b, B.D[i][j], sh[j], sl[j]);
      const long long even = fx_round(b);
      out[i] = odd + even;
      out[NP - 1 - i] = odd - even;
    } else {
      out[i] = odd;
    }
  }
}

// One step of Burgers (SSP-RK3, or with LS a 2N low-storage scheme; with VISC the viscous term
// of the local DG method). Warp w owns 32 - H - HR elements and forms H = ns more on the left
// and HR on the right (warp_element), so the stages run in registers with shuffles for the face
// values and no barrier, and u is read and written once per step. The operator
//   dt L(v)_i = sum_j W_ij g_j + a_i F_L + b_i F_R,   g = v^2
// (W = c2/2 (D + M^-1 e_0 e_0^T - M^-1 e_p e_p^T), a = -c2 M^-1 e_0, b = c2 M^-1 e_p) maps the
// even part of (g, faces) to the odd part and back, since the nodes are symmetric, so it is
// applied to sums and differences of mirrored nodes: 17 products instead of 35 at p = 4
// (BurgersFixed). REC also writes the stage inputs v1, v2 (recorded sweeps of the gradient).
// VISC: with (g, F) = (2 v, uhat) the same operator gives Z = -dt q of the local DG method
// (uhat = u^-), and (g, F) = (v^2 - 2 nu q, F - nu qhat) (qhat = q^+) the whole dt L; Z is
// brought to 58 bits by its largest value in the element, since smooth fields leave it far
// below its bound.
// Bound by instruction issue (integer). K = 2^20, p = 4, ADG-AT2, SSP-RK3: 0.50 ms a step as
// three FP64 stage kernels (80% of the FP64 pipe, eight field passes), 0.075 ms so (0.0815 with
// 64-bit headroom checks and the face flux's magnitudes); viscous, K = 2^18, p = 2, RK2: 0.127 ->
// 0.022 ms; K = 10125, p = 2: 14.5 -> 5.0 us, where the launch and the dependent loads of the
// delays and ring levels are what is left. Two elements per thread (58 of 64 owned, 128
// registers) took 0.089 ms and 7.0 us when one per thread took 0.078 and 5.3.
template <int NP, bool FACES, bool REC, bool VISC, bool LS>
__global__ void __launch_bounds__(128) k_burgers_step(const __grid_constant__ Inst I,
                                                      const __grid_constant__ StepArgs A) {
  constexpr int NV = kFaceVals<VISC>, MS = LS ? kMaxStages : kStages;
  __shared__ double sV_[FACES ? 4 * NV * MS : 1][32];
  pdl_wait();
  pdl_trigger();
  const int K = I.K, S = LS ? I.ns : kStages;
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if ((int64_t)warp * (32 - A.H - A.HR) >= K) return;
  const unsigned full = 0xffffffffu;
  bool own;
  const int e = warp_element(K, warp, lane, A.H, A.HR, own);
  double ud[NP];
  load_elem<NP>(A.uin, K, e, ud);

  // a PE face on the left of this lane's element, and its delayed values
  bool pe = false, late = false;
  int nm = 0;
  double (*sV)[32] = sV_ + (FACES ? (threadIdx.x >> 5) * NV * MS : 0);
  int fmax = 0, umax = 0;   // largest high words of the delayed fluxes and traces
  if (FACES) {
    const int j = e / I.Kpe;
    nm = mod_step(A.n, I.R);
    pe = e == j * I.Kpe;
    if (pe) {
      const DelayAt d = step_delay(I, j, A.n, A.tbase);
      late = d.k > 0;
      if (late) {
if constexpr (!LS && !VISC) {
          ring_sums<1, kStages>(I, d, j, nm, S, 0, sV, fmax, umax);
        } else {
          for (int s = 0; s < S; ++s) ring_sums<NV, 1>(I, d, j, nm, S, s, sV, fmax, umax);
        }
      }
    }
  }

  // the element's scale, and whether the integer path takes the warp
  int hi = 0;
  unsigned lo = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    hi = max(hi, __double2hiint(ud[i]) & 0x7fffffff);
    lo |= (unsigned)__double2loint(ud[i]);
  }
  const int be = bf_window_max(hi >> 20, 1);
  const int E = be - 1022;              // |u| < 2^E
  const BurgersFixed &B = I.bf;
  const int d0 = -(B.sc + E + 1);       // operator sums -> value units (inviscid)
  bool bad = be < kBfMinE || be > kBfMaxE || d0 < -2 || !B.ok;
  bad = bad || (hi ? (hi >> 20) < be - kBfSpan<LS> : lo != 0);
  // a delayed flux of 2^(2E + 1) or more, a delayed trace of 2^(E + 1) or more
  if (FACES) bad = bad || (fmax >> 20) > 2 * E + 1023;
  if (FACES && VISC) bad = bad || (umax >> 20) > be + 1;

  if (!__any_sync(full, bad)) {
    const int sg = 2 * E - 56;   // unit of the squares and fluxes
    // scales of the neighbours below this lane's
    const int dEL = E - __shfl_up_sync(full, E, 1), dER = E - __shfl_down_sync(full, E, 1);
    long long u[NP], v[NP];      // u: u^n, or dU of a 2N scheme
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      v[i] = bf_from(ud[i], be);
      u[i] = LS ? 0 : v[i];
    }
    unsigned mag = 0;
    auto stage = [&](int s) {
      long long G[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        int xh, xl;
        fx_split(v[i], xh, xl);
        G[i] = bf_square(xh, xl);
      }
      long long vl = __shfl_up_sync(full, v[NP - 1], 1);
      long long gl = __shfl_up_sync(full, G[NP - 1], 1);
      if (dEL != 0) {   // rarely: most neighbours have one scale
        vl = bf_bring(vl, dEL, mag);
        int xh, xl;
        fx_split(vl, xh, xl);
        gl = bf_square(xh, xl);
      }
      long long FL = bf_llf<LS>(vl, v[0], gl, G[0]);
      const size_t at = FACES && pe ? ((size_t)nm * I.ns + s) * I.P + e / I.Kpe : 0;
      if (FACES && pe) {
        if (own) I.ring[at] = make_double2(bf_to(FL, sg), VISC ? bf_to(vl, E - 57) : 0.0);
        if (late) FL = bf_from(sV[s][lane], 2 * E + 1023);
      }
      int d = d0, uf = sg;   // unit of the nodes' and faces' fluxes
      if (VISC) {
        long long uL = vl;
        if (FACES && late) uL = bf_from(sV[S + s][lane], be + 1) << 1;
        const long long uN = bf_bring(__shfl_down_sync(full, uL, 1), dER, mag);
        const bool lateR = FACES && __shfl_down_sync(full, late ? 1 : 0, 1) != 0 && lane < 31;
        const long long uR = lateR ? uN : v[NP - 1];   // v_p but at delayed faces
        long long g2[NP], Z[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) g2[i] = 2 * v[i];
        burgers_operator<NP>(B, g2, uL, uR, 0, Z);
        // Z 2^nz below 2^58
        unsigned zh = 0;
#pragma unroll
        for (int i = 0; i < NP; ++i) zh = max(zh, (unsigned)(fx_mag(Z[i]) >> 32));
        const int nz = __clz((int)zh) - 6;   // bit length of |Z| at most 64 - clz(zh)
        // y = -2 nu q = (2 nu / dt) Z: limbs of (2 nu / dt) 2^-sn, in units of 2^uq
        const int uq = B.sc + E - 57 - nz + B.sn;
        uf = max(uq, sg);
        const int sq = min(uf - uq, 60), sf = min(uf - sg, 60);
        const long long hq = sq > 0 ? 1ll << (sq - 1) : 0, hf = sf > 0 ? 1ll << (sf - 1) : 0;
        long long y0 = 0;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          int zh2, zl2;
          fx_split(bf_shift(Z[i], -nz), zh2, zl2);
          const long long y = (fx_scaled(B.vn, zh2, zl2) + hq) >> sq;
          G[i] = ((G[i] + hf) >> sf) + y;
          if (i == 0) y0 = y;
        }
        FL = (FL + hf) >> sf;
        if (FACES && pe) {
          if (own) I.ringq[at] = bf_to(y0, uf);
          if (late) {
            const double y = sV[2 * S + s][lane];
            // |y| < 2^(uf + 58)
            if (((__double2hiint(y) & 0x7fffffff) >> 20) > uf + 1080) mag |= kBfOver;
            else y0 = bf_from(y, uf + 1080) << 1;
          }
        }
        FL += (y0 + 1) >> 1;
        d = -(B.sc + uf - E + 57);
        if (d < -2) {
          mag |= kBfOver;
          d = -2;
        }
      }
      const int dF = VISC ? uf - __shfl_down_sync(full, uf, 1) : 2 * dER;
      long long FR = __shfl_down_sync(full, FL, 1);
      if (dF != 0) FR = bf_bring<kBfTop + 1>(FR, dF, mag);   // faces below 2^59 (burgers_operator)
      // shift of the operator's sums: in SSP-RK3 stage 1 takes a quarter of them, stage 2
      // (inside the sum divided by 3) twice
      if (!LS) d = s == 0 ? d : (s == 1 ? d + 2 : d - 1);
      d = d > 60 ? 60 : d;
      long long r[NP];
      // (2N: halves of the shift go up or down by a square's last bit)
      burgers_operator<NP>(B, G, FL, FR, d > 0 ? (1ll << (d - 1)) - (LS ? G[0] & 1 : 0) : 0, r);
      if (__any_sync(full, d < 0)) {   // large Courant numbers
#pragma unroll
        for (int k = 0; k < NP; ++k) {
          if (d < 0 && (fx_mag(r[k]) >> (kBfTop + d))) mag |= kBfOver;
          r[k] = bf_shift(r[k], d);
        }
      } else {
#pragma unroll
        for (int k = 0; k < NP; ++k) r[k] >>= d;
      }
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        const long long x = r[k];
        if (LS) {
          if (s > 0) {
            int h, l;
            fx_split(u[k], h, l);
            u[k] = fx_scaled(B.lsA[s], h, l) + x;
          } else {
            u[k] = x;
          }
          mag |= bf_mag(u[k]);
          int h, l;
          fx_split(u[k], h, l);
          // halves (the two-stage scheme's B = 1/2) up or down by v's last bit: always up, they
          // moved the field by a quarter unit a step
          FxAcc c;
          c.b += (B.lsB[s].y >> 1) - (int)(v[k] & 1);
          fx_mac(c, B.lsB[s], h, l);
          v[k] += fx_round(c);
        } else if (s == 0) {
          v[k] += x;
        } else if (s == 1) {
          v[k] = ((3 * u[k] + v[k] + 2) >> 2) + x;
        } else {
          const long long T = u[k] + 2 * v[k] + x;
          mag |= bf_mag(T) >> 2;   // below 2^60: its high limb fits 32 bits
          int th, tl;
          fx_split(T, th, tl);
          v[k] = fx_scaled(make_int2(kThirdHi, kThirdLo), th, tl);
        }
        mag |= bf_mag(v[k]);
      }
      if (REC && s < 2 && own) {
        double *o = s == 0 ? A.r1 : A.r2;
#pragma unroll
        for (int i = 0; i < NP; ++i) o[(size_t)i * K + e] = bf_to(v[i], E - 57);
      }
    };
    if (LS) {
      for (int s = 0; s < S; ++s) stage(s);
    } else {
#pragma unroll
      for (int s = 0; s < kStages; ++s) stage(s);
    }
    if (!__any_sync(full, mag >= kBfOver)) {
      if (own) {
#pragma unroll
        for (int i = 0; i < NP; ++i) A.uout[(size_t)i * K + e] = bf_to(v[i], E - 57);
      }
      return;
    }
  }
  burgers_step_fp64<NP, FACES, REC, VISC, LS>(I, A, warp, nm, sV, pe, late);
}

// What the reverse step reads: the recorded stage inputs u, v1, v2 (y, one field of nd values
// after another), the adjoint of u^{n+1} (w), the adjoint ring; it writes the adjoint of u^n.
struct AdjArgs {
  const double *y;
  const double *w;
  double *out;
  double *lring;
  int64_t n, tbase;
};

// Partial derivatives of the local Lax-Friedrichs flux (adg_adjoint.cu), doubled and in
// integers: lambda from a where |a| >= |b|, d|x|/dx = 1 for x >= 0.
__device__ __forceinline__ void bf_llf_partials2(long long a, long long b, long long &dl,
                                                 long long &dr) {
  const long long ma = a < 0 ? -a : a, mb = b < 0 ? -b : b;
  if (ma >= mb) {
    dl = a >= 0 ? 3 * a - b : b - a;
    dr = b - ma;
  } else {
    dl = a + mb;
    dr = b >= 0 ? a - b : 3 * b - a;
  }
}

// The same in FP64.
__device__ __forceinline__ void llf_partials_fp64(double a, double b, double &dl, double &dr) {
  const bool left = abs_bits(a) >= abs_bits(b);
  const double lam = left ? fabs(a) : fabs(b), jump = b - a;
  const double gl = left ? (nonneg(a) ? 1.0 : -1.0) : 0.0;
  const double gr = left ? 0.0 : (nonneg(b) ? 1.0 : -1.0);
  dl = 0.5 * a + 0.5 * lam - 0.5 * gl * jump;
  dr = 0.5 * b - 0.5 * lam - 0.5 * gr * jump;
}

// A PE face in the reverse sweep: the flux adjoint mu of the stage is posted, times the AT
// coefficients, to the delayed levels' ring entries (its owner only; one addition per entry in
// a step, so the atomic's order does not matter and its latency is not waited for).
__device__ __forceinline__ void post_levels(const Inst &I, double *lring, int j, int nm, int s,
                                            int k, int qe, const double *c, double mu) {
  for (int i = 0; i < qe; ++i) {
    if (k + i < 1 || c[i] == 0.0) continue;
    int sl = nm - k - i;
    if (sl < 0) sl += I.R;
    atomicAdd(lring + ((size_t)sl * kStages + s) * I.P + j, c[i] * mu);
  }
}

// The reverse step in FP64 (warps that the integer path does not take); face: pe as in
// burgers_step_fp64, sR[stage][lane] the ring entries of this step.
template <int NP, bool FACES>
__device__ __noinline__ void burgers_adj_fp64(const Inst &I, const AdjArgs &A, int warp, int nm,
                                              const double (*sR)[32], bool pe, int k, int qe,
                                              const double *c) {
  const int K = I.K;
  const size_t nd = (size_t)K * NP;
  const int lane = threadIdx.x & 31;
  bool own;
  const int e = warp_element(K, warp, lane, kHalo, kHalo, own);
  const unsigned full = 0xffffffffu;
  double w[NP], acc[NP];
  load_elem<NP>(A.w, K, e, w);
#pragma unroll
  for (int i = 0; i < NP; ++i) acc[i] = 0.0;
#pragma unroll
  for (int s = kStages - 1; s >= 0; --s) {
    const StageConsts &C = I.sc[s];
    double v[NP], lv[NP];
    load_elem<NP>(A.y + s * nd, K, e, v);
    double sL = 0.0, sRt = 0.0;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      sL = fma(C.lL[i], w[i], sL);
      sRt = fma(C.lR[i], w[i], sRt);
    }
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      double a = C.A[j] * w[0];
#pragma unroll
      for (int i = 1; i < NP; ++i) a = fma(C.A[i * NP + j], w[i], a);
      lv[j] = fma(C.beta, w[j], 2.0 * v[j] * a);
    }
    lv[0] = fma(v[0], sL, lv[0]);
    lv[NP - 1] = fma(v[NP - 1], sRt, lv[NP - 1]);
    double mu = -sL - __shfl_up_sync(full, sRt, 1);
    double dl, dr;
    llf_partials_fp64(__shfl_up_sync(full, v[NP - 1], 1), v[0], dl, dr);
    if (FACES && pe) {
      const double r = sR[s][lane];
      if (own) post_levels(I, A.lring, e / I.Kpe, nm, s, k, qe, c, mu);
      mu = k > 0 ? r : mu + r;
    }
    lv[0] = fma(mu, dr, lv[0]);
    lv[NP - 1] += __shfl_down_sync(full, mu * dl, 1);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (s == 2) acc[i] = C.alpha * w[i];
      if (s == 1) acc[i] = fma(C.alpha, w[i], acc[i]);
      w[i] = lv[i];
    }
  }
  if (own) {
#pragma unroll
    for (int i = 0; i < NP; ++i) A.out[(size_t)i * K + e] = acc[i] + w[i];
  }
}

// The adjoint of one SSP-RK3 step of inviscid Burgers, from the recorded stage inputs: the
// layout and the integer arithmetic of k_burgers_step, with a second scale for the adjoint
// (|w| < 2^Ew near the element). For the adjoint w of a stage's output the adjoint of its
// input v is beta (w + Z),
//   Z_j = 2 v_j (W^T w)_j + (mu_L dF_L/du^+ at j = 0) + (mu_R dF_R/du^- at j = p),
// mu the flux adjoints a . w^e + b . w^{e-1}; W^T, a and b act on sums and differences of
// mirrored nodes with the coefficients of the forward step (transposed). A PE face posts
// c_i mu to the delayed levels of the adjoint ring and takes the ring entry of its own step
// and stage for (delay > 0) or beside (delay 0) mu; its owner clears the entries of step
// n + 1, which the kernel before this one read. The gradient on 65536 elements (p = 3, 100
// steps) with this kernel: 6.3 -> 3.9 ms, against three FP64 stage kernels of 14 us each, bound
// by the FP64 pipe (11.3 -> 2.9 ms with the forward's step and without recomputation). Bound by
// the latency of a warp's chain: 65536 elements are 17 warps per SM, and the 5 million warp
// instructions of a launch some 4 of its 12 us. The compiler's own choices are 64 to 80
// registers, with spills at p = 1 and 2 (and 3, 2.92 ms); the 96 of five blocks hold every degree
// but p = 4, which takes 128, without them (p = 3 2.75 ms; p = 2 on 65536 elements 2.157 -> 2.139
// ms, p = 1 1.879 -> 1.866).
template <int NP, bool FACES>
__global__ void __launch_bounds__(128, NP <= 4 ? 5 : 0) k_burgers_adj(const __grid_constant__ Inst I,
                                                     const __grid_constant__ AdjArgs A) {
  constexpr int HP = NP / 2, MID = NP % 2;
  __shared__ double sR_[FACES ? 4 * kStages : 1][32];
  pdl_wait();
  pdl_trigger();
  const int K = I.K;
  const size_t nd = (size_t)K * NP;
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if ((int64_t)warp * kOwn >= K) return;
  const unsigned full = 0xffffffffu;
  bool own;
  const int e = warp_element(K, warp, lane, kHalo, kHalo, own);
  double wd[NP], yd[kStages][NP];
  load_elem<NP>(A.w, K, e, wd);
#pragma unroll
  for (int s = 0; s < kStages; ++s) load_elem<NP>(A.y + s * nd, K, e, yd[s]);

  bool pe = false;
  int nm = 0, k = 0, qe = 0;
  const double *c = nullptr;
  double (*sR)[32] = sR_ + (FACES ? (threadIdx.x >> 5) * kStages : 0);
  int rmax = 0;
  if (FACES) {
    const int j = e / I.Kpe;
    nm = mod_step(A.n, I.R);
    pe = e == j * I.Kpe;
    if (pe) {
      const DelayAt d = step_delay(I, j, A.n, A.tbase);
      k = d.k;
      qe = d.qe;
      c = d.c;
      const int nx = nm + 1 == I.R ? 0 : nm + 1;
#pragma unroll
      for (int s = 0; s < kStages; ++s) {
        const double r = A.lring[((size_t)nm * kStages + s) * I.P + j];
        sR[s][lane] = r;
        rmax = max(rmax, __double2hiint(r) & 0x7fffffff);
        if (own && I.R > 1) A.lring[((size_t)nx * kStages + s) * I.P + j] = 0.0;
      }
    }
  }

  // the scales: of the adjoint (as the forward step's), and of the stage inputs of the element
  // and its neighbours (2^E, which enter as factors of w)
  int hw = 0, hv = 0;
  unsigned lo = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    hw = max(hw, __double2hiint(wd[i]) & 0x7fffffff);
    lo |= (unsigned)__double2loint(wd[i]);
#pragma unroll
    for (int s = 0; s < kStages; ++s) hv = max(hv, __double2hiint(yd[s][i]) & 0x7fffffff);
  }
  const int bw = bf_window_max(hw >> 20, 1), bv = bf_window_max(hv >> 20, 1);
  const int Ew = bw - 1022, E = bv - 1022;
  const int d0 = -(I.bf.sc + E + 1);   // products (below) -> units of w
  bool bad = bw < kBfMinE || bw > kBfMaxE || bv < kBfMinE || bv > kBfMaxE || d0 < -1 || !I.bf.ok;
  bad = bad || (hw ? (hw >> 20) < bw - kBfSpan<false> : lo != 0);
  // ring entries below 2^60 in units of mu
  if (FACES) bad = bad || (rmax >> 20) > I.bf.sc + Ew + 1025;

  if (!__any_sync(full, bad)) {
    const BurgersFixed &B = I.bf;
    const int smu = I.bf.sc + Ew - 57;   // unit of the flux adjoints
    // scales of the neighbours below this lane's
    const int dWL = Ew - __shfl_up_sync(full, Ew, 1), dWR = Ew - __shfl_down_sync(full, Ew, 1);
    const int dVL = E - __shfl_up_sync(full, E, 1);
    const int d = d0 > 60 ? 60 : d0;
    const long long half = d > 0 ? 1ll << (d - 1) : 0;
    const bool up = __any_sync(full, d < 0);   // large Courant numbers
    // z 2^-d
    auto scale = [&](long long z, unsigned &over) -> long long {
      if (!up) return z >> d;
      if (d < 0 && (fx_mag(z) >> (kBfTop + d))) over |= kBfOver;
      return bf_shift(z, d);
    };
    long long w[NP], acc[NP];
    double post[kStages];   // beta mu of a PE face's stages (FP64), posted once the step holds
#pragma unroll
    for (int i = 0; i < NP; ++i) w[i] = bf_from(wd[i], bw);
    unsigned mag = 0;
    // x / 3 for |x| < 2^60
    auto third = [](long long x) {
      int h, l;
      fx_split(x, h, l);
      return fx_scaled(make_int2(kThirdHi, kThirdLo), h, l);
    };
    // x y 2^(k - 58) rounded for |x|, |y| < 2^60, from the limbs of both
    auto mul = [](int xh, int xl, int yh, int yl, int k) {
      const long long c = fx_mul(xh, yl) + fx_mul(xl, yh) +
                          (long long)__umulhi((unsigned)xl << 3, (unsigned)yl);
      return (fx_mul(xh, yh) << k) + ((c + (1 << (28 - k))) >> (29 - k));
    };
    // x / 4, halves to even
    auto quarter = [](long long x) { return (x + 1 + ((x >> 2) & 1)) >> 2; };
#pragma unroll
    for (int s = kStages - 1; s >= 0; --s) {
      long long v[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) v[i] = bf_from(yd[s][i], bv);
      int th[HP ? HP : 1], tl[HP ? HP : 1], sh[HP + MID], sl[HP + MID];
#pragma unroll
      for (int i = 0; i < HP; ++i) {
        fx_split(w[i] - w[NP - 1 - i], th[i], tl[i]);
        fx_split(w[i] + w[NP - 1 - i], sh[i], sl[i]);
      }
      if (MID) fx_split(w[HP], sh[HP], sl[HP]);
      // a . w = ev + od, b . w = od - ev
      FxAcc ae{0, B.rSt[HP]}, ao{0, B.rDt[HP + MID]};
#pragma unroll
      for (int i = 0; i < HP + MID; ++i) fx_mac(ae, B.S[i][HP], sh[i], sl[i]);
#pragma unroll
      for (int i = 0; i < HP; ++i) fx_mac(ao, B.D[i][HP + MID], th[i], tl[i]);
      const long long ev = fx_round(ae), od = fx_round(ao);
      // (|ev|, |od| < 2^61)
      const long long bl = bf_bring<kBfTop + 4>(__shfl_up_sync(full, od - ev, 1), dWL, mag);
      long long mu = ev + od + bl;
      long long dl, dr;
      bf_llf_partials2(bf_bring(__shfl_up_sync(full, v[NP - 1], 1), dVL, mag), v[0], dl, dr);
      if (FACES && pe) {
        const long long r = bf_from(sR[s][lane], B.sc + Ew + 1025) << 3;
        mag |= bf_mag(mu) >> 3;   // below 2^61
        const double m = bf_to(mu, smu);
        post[s] = s == 2 ? m * (2.0 / 3.0) : (s == 1 ? 0.25 * m : m);
        // the ring holds adjoints of the flux with beta: divided by it here
        const long long rb = s == 2 ? r + (r >> 1) : (s == 1 ? 4 * r : r);
        mu = k > 0 ? rb : mu + rb;
      }
      mag |= bf_mag(mu) >> 3;   // below 2^61
      // products in quarters of the unit of mu times that of the stage inputs
      int mh, ml, xh, xl;
      fx_split((mu + ((mu >> 1) & 1)) >> 1, mh, ml);
      fx_split(dl, xh, xl);
      const long long pl = mul(mh, ml, xh, xl, 0);
      fx_split(dr, xh, xl);
      const long long pr = mul(mh, ml, xh, xl, 0);
      // the left element's part, in units of this lane's w, from the lane above
      const long long pR = bf_bring<kBfTop + 2>(__shfl_down_sync(full, scale(pl + half, mag), 1), dWR, mag);
#pragma unroll
      for (int j = 0; j < HP + MID; ++j) {
        // half the sum and half the difference of (W^T w)_j and (W^T w)_{p-j}
        FxAcc a{0, B.rDt[j]}, b{0, j < HP ? B.rSt[j] : 0};
#pragma unroll
        for (int i = 0; i < HP; ++i) fx_mac(a, B.D[i][j], th[i], tl[i]);
        const long long sum = fx_round(a);
        long long dif = 0;
        if (j < HP) {
#pragma unroll
          for (int i = 0; i < HP + MID; ++i) fx_mac(b, B.S[i][j], sh[i], sl[i]);
          dif = fx_round(b);
        }
#pragma unroll
        for (int m = 0; m < (j < HP ? 2 : 1); ++m) {
          const int q = m ? NP - 1 - j : j;
          int rh, rl, vh, vl;
          const long long r = m ? sum - dif : sum + dif;
          mag |= bf_mag(r) >> 2;   // below 2^60
          fx_split(r, rh, rl);
          fx_split(v[q], vh, vl);
          long long z = mul(rh, rl, vh, vl, 1) + half;
          if (q == 0) z += pr;
          const long long x = w[q] + scale(z, mag) + (q == NP - 1 ? pR : 0);
          mag |= bf_mag(x);
          if (s == 2) {
            acc[q] = third(w[q]);
            w[q] = third(2 * x);
          } else if (s == 1) {
            acc[q] += quarter(3 * w[q]);
            w[q] = quarter(x);
          } else {
            w[q] = x + acc[q];
            mag |= bf_mag(w[q]);
          }
        }
      }
    }
    if (!__any_sync(full, mag >= kBfOver)) {
      if (own) {
#pragma unroll
        for (int i = 0; i < NP; ++i) A.out[(size_t)i * K + e] = bf_to(w[i], Ew - 57);
        if (FACES && pe) {
#pragma unroll
          for (int s = 0; s < kStages; ++s)
            post_levels(I, A.lring, e / I.Kpe, nm, s, k, qe, c, post[s]);
        }
      }
      return;
    }
  }
  burgers_adj_fp64<NP, FACES>(I, A, warp, nm, sR, pe, k, qe, c);
}

// One-warp blocks while the mesh gives fewer than 32 warps per SM: they spread evenly, and all
// are resident at once. Larger meshes run several waves of four-warp blocks; so do viscous ones
// from 16 warps per SM, whose blocks' shared memory (fixed, four warps' worth) leaves no room for
// 32 on an SM.
constexpr size_t kSmemSM = 228 * 1024;   // of an SM; a block takes 1 KB besides its own
int burgers_block(int64_t warps, size_t fixed) {
  const int per = fixed + 1024 <= kSmemSM / 32 ? 32 : 16;
  return warps < per * sm_count() ? 32 : 128;
}

// Dynamic shared memory (never read) that lets an SM hold only its even share of the blocks, for
// grids of 16 to 32 one-warp blocks per SM. A step's blocks become resident while the step before
// still runs, so without it the SMs that drain first take too many of them and the others too
// few: 50 steps on 65536 elements, p = 3: 591 us in four-warp blocks, 512 with those held to
// their share, 490 in one-warp blocks so; p = 1: 515 -> 413; the gradient of 50 steps 1.50 ->
// 1.30 ms. Below 16 warps per SM the next step's blocks all wait beside the present ones and
// hide their launch (16384 elements: 299 us, 302 with their share only). Not where another stream's
// steps run beside these (the gradient's recomputation beside its reverse sweep), whose blocks
// the room is for: 2000 steps in segments of 50 on 65536 elements 65.5 ms with it, 60.4 without.
size_t burgers_smem(int64_t grid, int bs, size_t fixed) {
  const int64_t per = (grid + sm_count() - 1) / sm_count();
  if (bs != 32 || per < 16) return 0;
  const size_t block = kSmemSM / (per + 1) + 128;
  return block > fixed + 1024 ? block - fixed - 1024 : 0;
}

template <int NP, bool FACES>
cudaError_t burgers_np(const Inst &I, const StepArgs &A, cudaStream_t s, bool pdl, bool alone) {
  const int own = 32 - A.H - A.HR;
  const int64_t warps = ((int64_t)I.K + own - 1) / own;
  const size_t fixed = FACES ? sizeof(double) * 32 * 4 * (I.visc ? kFaceVals<true> : kFaceVals<false>) *
                                   (I.ls ? kMaxStages : kStages) : 0;   // sV_
  const int bs = burgers_block(warps, fixed);
  const dim3 g((unsigned)((warps * 32 + bs - 1) / bs)), b(bs);
  const size_t smem = alone ? burgers_smem(g.x, bs, fixed) : 0;
  auto go = [&](auto kernel) { return launch_smem_pdl(kernel, g, b, smem, s, pdl, I, A); };
  if (A.r1) return go(k_burgers_step<NP, FACES, true, false, false>);
  if (I.ls)
    return I.visc ? go(k_burgers_step<NP, FACES, false, true, true>)
                  : go(k_burgers_step<NP, FACES, false, false, true>);
  return I.visc ? go(k_burgers_step<NP, FACES, false, true, false>)
                : go(k_burgers_step<NP, FACES, false, false, false>);
}

template <int NP>
cudaError_t burgers_adj_np(const Inst &I, const AdjArgs &A, cudaStream_t s, bool pdl, bool alone) {
  const int64_t warps = ((int64_t)I.K + kOwn - 1) / kOwn;
  const size_t fixed = I.async ? sizeof(double) * 32 * 4 * kStages : 0;   // sR_
  const int bs = burgers_block(warps, fixed);
  const dim3 g((unsigned)((warps * 32 + bs - 1) / bs)), b(bs);
  const size_t smem = alone ? burgers_smem(g.x, bs, fixed) : 0;
  return I.async ? launch_smem_pdl(k_burgers_adj<NP, true>, g, b, smem, s, pdl, I, A)
                 : launch_smem_pdl(k_burgers_adj<NP, false>, g, b, smem, s, pdl, I, A);
}

}  // namespace

cudaError_t launch_burgers_adj(const Inst &I, const double *y, const double *w, double *out,
                               double *lring, int64_t n, int64_t tbase, cudaStream_t s, bool pdl,
                               bool alone) {
  if (w == out) return cudaErrorInvalidValue;
  const AdjArgs A{y, w, out, lring, n, tbase};
  switch (I.Np) {
    case 2: return burgers_adj_np<2>(I, A, s, pdl, alone);
    case 3: return burgers_adj_np<3>(I, A, s, pdl, alone);
    case 4: return burgers_adj_np<4>(I, A, s, pdl, alone);
    case 5: return burgers_adj_np<5>(I, A, s, pdl, alone);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_burgers_step(const Inst &I, const double *uin, double *uout, double *r1,
                                double *r2, int64_t n, int64_t tbase, cudaStream_t s, bool pdl,
                                bool alone) {
  if (uin == uout || (r1 && (I.ls || I.visc))) return cudaErrorInvalidValue;
  const StepArgs A{uin, uout, r1, r2, n, tbase, I.ns, I.ns + (I.visc ? 1 : 0)};
  switch (I.Np) {
    case 2:
      return I.async ? burgers_np<2, true>(I, A, s, pdl, alone)
                     : burgers_np<2, false>(I, A, s, pdl, alone);
    case 3:
      return I.async ? burgers_np<3, true>(I, A, s, pdl, alone)
                     : burgers_np<3, false>(I, A, s, pdl, alone);
    case 4:
      return I.async ? burgers_np<4, true>(I, A, s, pdl, alone)
                     : burgers_np<4, false>(I, A, s, pdl, alone);
    case 5:
      return I.async ? burgers_np<5, true>(I, A, s, pdl, alone)
                     : burgers_np<5, false>(I, A, s, pdl, alone);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace adg
