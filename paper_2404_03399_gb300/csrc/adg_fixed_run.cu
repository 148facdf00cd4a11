// The fixed-point composed step on meshes that fit on the chip: a run of steps in one launch.
#include <algorithm>
#include <type_traits>

#include "adg_faces.cuh"
#include "adg_fixed_element.cuh"

namespace adg {
namespace {

// Where the AT coefficients lie in a block's shared memory: behind the fixed part, the rings of
// nf faces and the delays of a launch's steps.
__host__ __device__ inline size_t run_coef_at(size_t fixed, int nf, int R, int S) {
  return fixed + ((size_t)nf * R * S * sizeof(double) + (size_t)nf * kRunSteps + 7) / 8 * 8;
}

constexpr int kRunThreads = 448;               // element threads of a block, two elements each
constexpr int kRunTile = 2 * kRunThreads;
constexpr int kRunFaces = 32;                  // PE faces of a block's tile
constexpr int kRunFaceWarps = 3;               // at most, in a block of at most 512 threads
constexpr int kRunBlock = 512;                 // (128 registers)

// Shared memory of a block; behind it the tile's faces' ring [faces][R][S], their delays
// [nsteps][faces] and the AT coefficients.
template <int NP, int S>
struct RunShared {
  ChannelSlots<kRunTile, S> ch;
  long long fx[kRunFaces][S][NP];   // the elements e-S .. e-1 of each face, at the stored scale
  int Dh[kRunFaces][S], Dl[kRunFaces][S];   // the differences in the step's units, limbs
  double d[kRunFaces][S];
  int how[kRunFaces];               // correction: 0 none, 1 integer, 2 FP64
  long long V[kRunFaces][S];        // delayed values (run_ahead), and their exponents
  int be[kRunFaces][S];
  unsigned long long mag;           // OR of |y| over the block
  int bits, stop;                   // bit length of the field's OR; the barrier's wait ran out
};

// The grid barrier's words, one pair per step of the launch (zeroed before it): blocks arrived
// (bits 0-15), those whose OR has the length of the step before (16-31) and a larger one
// (32-47); and the largest length, read only where the first word leaves it open.
struct RunWords {
  unsigned long long arrived[kRunSteps];
  unsigned top[kRunSteps];
};

// Arrival of a block whose OR has bit length top (bits: the field's length of the step before),
// and the wait for all nb: the field's new length, or -1 when the wait ran out.
__device__ __forceinline__ int run_barrier(RunWords *w, int t, int nb, int top, int bits, long long most) {
  unsigned long long *a = &w->arrived[t];
  if (top != bits)
    asm volatile("red.relaxed.gpu.global.max.u32 [%0], %1;" ::"l"(&w->top[t]), "r"(top) : "memory");
  __threadfence();   // the block's exchange slot and ring entries (and top) before its arrival
  const unsigned long long add =
      1ull | (top == bits ? 1ull << 16 : 0ull) | (top > bits ? 1ull << 32 : 0ull);
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(a), "l"(add) : "memory");
  unsigned long long v = 0;
  for (long long polls = 0; polls < most; ++polls) {
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
    if ((int)(v & 0xffffu) == nb) break;
  }
  __threadfence();
  if ((int)(v & 0xffffu) != nb) return -1;
  if ((v >> 32) == 0 && ((v >> 16) & 0xffffu) != 0) return bits;
  unsigned m;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(m) : "l"(&w->top[t]) : "memory");
  return (v >> 32) == 0 && ((v >> 16) & 0xffffu) != 0 ? bits : (int)m;
}

// What a lane knows of its face group's face.
struct RunFace {
  int l;       // the face of the tile
  int j;       // ... and of the mesh
  bool own;    // this block writes its ring
  bool on;     // the lane is one of the group's stages
};

// The delayed values of a face at the step of ring slot nm (face_ahead), kept for run_face. They
// do not depend on the step's input: formed while the grid's barrier is waited for.
template <int NP, int S>
__device__ __forceinline__ void run_ahead(const Inst &I, RunShared<NP, S> &sh, const RunFace &f,
                                          const double *hist, const int *c, const FaceDelay &dl, int nm) {
  const FaceGroup g = face_group<S>();
  double Rv[kMaxQ];
#pragma unroll
  for (int i = 0; i < kMaxQ; ++i) {
    int sl = nm - (dl.k + i);
    if (sl < 0) sl += I.R;
    Rv[i] = f.on && dl.k > 0 && i < dl.qe ? hist[sl * S + g.r] : 0.0;
  }
  long long V;
  int be;
  face_ahead<S>(I, g, Rv, c, dl.k > 0 ? dl.qe : 0, V, be);
  if (f.on) {
    sh.V[f.l][g.r] = V;
    sh.be[f.l][g.r] = be;
  }
}

// The differences of one face by its group, with the ring's levels in hist [R][S], and the limbs
// of the correction.
template <int NP, int S>
__device__ __forceinline__ void run_face(const Inst &I, RunShared<NP, S> &sh, const RunFace &f,
                                         double *hist, const int *c, const FaceDelay &dl, int nm, int sig,
                                         int sigw, bool bad) {
  const FaceGroup g = face_group<S>();
  const int r = g.r;
  const bool late = f.on && dl.k > 0;
  long long X[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) X[i] = f.on ? sh.fx[f.l][r][i] : 0;
  const long long V = f.on ? sh.V[f.l][r] : 0;
  const int be = f.on ? sh.be[f.l][r] : 0;
  const double T0 = face_trace_fixed<NP, S>(I, g, f.on, X, sig);
  double T, d;
  face_differences<S>(I, g, late, T0, V, be, c, dl.qe,
                      [&](int i, int s) {
                        int sl = nm - (dl.k + i);
                        if (sl < 0) sl += I.R;
                        return dl.k > 0 && i < dl.qe ? hist[sl * S + s] : 0.0;
                      },
                      T, d);
  int dh[S], dlo[S];
  const int how = face_limbs<S>(I, g, f.on, d, sigw, dh, dlo);
  if (f.on) {
    sh.d[f.l][r] = d;
    if (r == 0) {
#pragma unroll
      for (int s = 0; s < S; ++s) {
        sh.Dh[f.l][s] = dh[s];
        sh.Dl[f.l][s] = dlo[s];
      }
      sh.how[f.l] = bad ? 0 : how;
    }
    hist[nm * S + r] = T;
    if (f.own) I.ring[((size_t)nm * S + r) * I.P + f.j] = make_double2(T, 0.0);
  }
}

// nsteps steps of the fixed-point composed step, int64 -> int64 (block-basis coordinates), in
// one cooperative launch: block b keeps the elements [b K / nb, (b+1) K / nb) in registers, two
// consecutive ones per thread, for the whole run. A step is what k_step_fixed and k_face_step
// do in two launches, with the same arithmetic (bit for bit):
//   * element threads publish their channel sums in shared memory while one more warp does the
//     same for the S elements left of the tile (from the left block's exchange slot);
//   * element threads form the composed step while the face warp forms the stage differences
//     d_s of the tile's PE faces, S of a group's lanes per face (a face near a tile boundary
//     in both blocks, from the same values; its ring levels, delays and AT coefficients are
//     kept in shared memory);
//   * the corrections sum_s R_s d_s of the elements around each face are added;
//   * the block's last 2S-1 elements go to its exchange slot, and the block arrives at the
//     grid's barrier, whose word also carries the reduction of the next step's scale. The wait
//     is bounded: after `polls` polls a block sets *err and returns.
// Bound by latency: the chain through a tile's elements, the faces' differences and the barrier.
// K = 65536, p = 3, ADG-AT3 (256 PEs): 8.9 us a step as two kernels in a graph, 5.0 us so
// with the read of the state (sync steps alone 3.9 -> 3.0 us). (Every block
// polling a flag of every other took 1.5-2.9 us a step for the barrier alone, which is 1.0 us; a
// face per lane with its ring in global memory 3.4 us for the faces.)
template <int NP, int S, bool FACES>
__global__ void __launch_bounds__(kRunBlock, 1)
    k_fixed_run(const __grid_constant__ Inst I, const long long *__restrict__ in,
                long long *__restrict__ out, int rel, int nsteps, int elems, RunWords *words,
                long long *exch, int *err, long long polls) {
  constexpr int HL = 2 * S - 1;   // elements left of the tile that the faces' traces reach
  constexpr int G = kFaceLanes<S>;
  extern __shared__ __align__(16) unsigned char smem_[];
  RunShared<NP, S> &sh = *reinterpret_cast<RunShared<NP, S> *>(smem_);
  const StepFixed &F = I.sf;
  const int K = I.K, P = I.P, nb = gridDim.x, b = blockIdx.x;
  const int e0 = (int)((int64_t)b * K / nb), cnt = (int)((int64_t)(b + 1) * K / nb) - e0;
  // elems element threads, a warp for the elements left of the tile, and the face warps
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool halo_warp = warp == elems / 32, face_warp = FACES && warp > elems / 32;
  const int faces0 = (warp - elems / 32 - 1) * (32 / G);   // a face warp's first face,
  const int faces_by = ((int)(blockDim.x - elems) / 32 - 1) * (32 / G);   // and its stride
  const int left = b == 0 ? nb - 1 : b - 1;
  const int64_t n0 = I.meta[0] + rel;

  // the tile's faces: face l at position pos (of its element e) relative to e0
  const int first = FACES ? (max(e0 - (S - 1), 0) + I.Kpe - 1) / I.Kpe : 0;
  auto face_pos = [&](int l) { return (first + l) * I.Kpe - e0; };
  const int nf = FACES && cnt >= face_pos(0) ? (cnt - face_pos(0)) / I.Kpe + 1 : 0;
  // the face whose window [pos - S, pos + S - 1] holds the element at position x, if any (and r =
  // x - pos)
  auto face_of = [&](int x, int &r) -> int {
    if (!FACES || nf == 0) return -1;
    const int y = x + S - face_pos(0);
    if (y < 0) return -1;
    const int l = min(y / I.Kpe, nf - 1);
    r = x - face_pos(l);
    return r <= S - 1 ? l : -1;
  };
  double *hist = reinterpret_cast<double *>(&sh + 1);
  unsigned char *delays = reinterpret_cast<unsigned char *>(hist + nf * I.R * S);
  int *coefi = reinterpret_cast<int *>(smem_ + run_coef_at(sizeof(RunShared<NP, S>), nf, I.R, S));
  if (FACES) {
    for (int x = threadIdx.x; x < nf * I.R * S; x += blockDim.x) {
      const int l = x / (I.R * S), y = x - l * (I.R * S);   // y = slot S + stage
      hist[x] = __ldcg(&I.ring[(size_t)y * P + (first + l) % P].x);
    }
    for (int x = threadIdx.x; x < nf * nsteps; x += blockDim.x) {
      const int t = x / nf, l = x - t * nf;
      delays[x] = I.table[(n0 + t - I.meta[1]) * P + (first + l) % P];
    }
    for (int x = threadIdx.x; x < I.L * I.q * I.q; x += blockDim.x) coefi[x] = __ldg(I.coefi + x);
  }

  long long X[2][NP], hX[NP];
  int fl[2] = {-1, -1}, fr[2] = {0, 0}, hf = -1, hr = 0;
  const int x0 = 2 * (int)threadIdx.x;
  const bool elem = threadIdx.x < elems;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool ok = elem && x0 + h < cnt;
#pragma unroll
    for (int i = 0; i < NP; ++i) X[h][i] = ok ? in[(size_t)i * K + e0 + x0 + h] : 0;
    if (ok) fl[h] = face_of(x0 + h, fr[h]);
    if (fl[h] >= 0 && fr[h] < 0) {
#pragma unroll
      for (int i = 0; i < NP; ++i) sh.fx[fl[h]][fr[h] + S][i] = X[h][i];
    }
  }
  const bool halo = halo_warp && lane < HL;
  if (halo) hf = face_of(lane - HL, hr);
  const int slot0 = mod_step(n0, 3);
  int sig = I.fx[slot0].sigma;
  const bool bad = I.fx[slot0].E >= 2047;
  const unsigned long long M0 = I.fx[slot0].mag;
  int bits = M0 ? 64 - __clzll((long long)M0) : 0;
  int nm = FACES ? mod_step(n0, I.R) : 0;   // the ring slot of the step
  auto face_at = [&](int l0) {
    const int l = l0 + lane / G;
    const bool active = l < nf;
    const int pos = face_pos(active ? l : 0);
    return RunFace{active ? l : 0, (first + l) % P, pos >= 0 && pos < cnt, active && lane % G < S};
  };
  auto ahead = [&](int t) {
    for (int l0 = faces0; l0 < nf; l0 += faces_by) {
      const RunFace f = face_at(l0);
      const FaceDelay dl = face_delay(I, delays[t * nf + f.l], n0 + t);
      run_ahead<NP, S>(I, sh, f, hist + f.l * I.R * S, coefi + (dl.k * I.q + dl.qe - 1) * I.q, dl, nm);
    }
  };
  if (FACES) {
    __syncthreads();
    if (face_warp) ahead(0);
  }

  for (int t = 0; t < nsteps; ++t) {
    // working scale (fx_scale of an int64 input)
    const int shift = bits ? bits - 56 + I.fxh : 0;
    const int sigw = sig + shift;
    if (halo) {
      int e = e0 - HL + lane;
      if (e < 0) e += K;
      const long long *q = t == 0 ? in + e : exch + (((size_t)((t - 1) & 1) * nb + left) * HL + lane) * NP;
      const size_t stride = t == 0 ? (size_t)K : 1;
#pragma unroll
      for (int i = 0; i < NP; ++i) hX[i] = __ldcg(q + i * stride);
      if (hf >= 0 && hr < 0) {
#pragma unroll
        for (int i = 0; i < NP; ++i) sh.fx[hf][hr + S][i] = hX[i];
      }
      if (lane >= S - 1) {   // elements e0-S .. e0-1
        const FxScale sc{};
        long long p;
        FxAcc own[S - 1];
        int xh[NP], xl[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) hX[i] = fx_rescale(hX[i], shift);
        fx_own<NP, true, S, true>(F, nullptr, nullptr, hX, sc, p, own, xh, xl);
        fx_publish(sh.ch, lane - (S - 1), p, own);
      }
      if (lane == 0) sh.mag = 0;
    }
    int xh[2][NP], xl[2][NP];
    long long pE = 0;
    FxAcc ownE[S - 1];
    if (elem) {
      const FxScale sc{};
      long long pO;
      FxAcc ownO[S - 1];
      if (shift) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < NP; ++i) X[h][i] = fx_rescale(X[h][i], shift);
      }
      fx_own<NP, true, S, true>(F, nullptr, nullptr, X[0], sc, pE, ownE, xh[0], xl[0]);
      fx_own<NP, true, S, true>(F, nullptr, nullptr, X[1], sc, pO, ownO, xh[1], xl[1]);
      fx_publish(sh.ch, x0 + S, pE, ownE);
      fx_publish(sh.ch, x0 + S + 1, pO, ownO);
    }
    __syncthreads();
    if (face_warp) {
      for (int l0 = faces0; l0 < nf; l0 += faces_by) {
        const RunFace f = face_at(l0);
        const FaceDelay dl = face_delay(I, delays[t * nf + f.l], n0 + t);
        run_face<NP, S>(I, sh, f, hist + f.l * I.R * S, coefi + (dl.k * I.q + dl.qe - 1) * I.q, dl, nm, sig,
                        sigw, bad);
      }
    }
    unsigned long long mag = 0;
    if (elem) {
      int Pc[2][S][2];
      fx_left_channels(F, sh.ch, x0, Pc[0]);
      fx_split(pE, Pc[1][0][0], Pc[1][0][1]);
#pragma unroll
      for (int s = 1; s < S; ++s) {
        FxAcc c = ownE[s - 1];
#pragma unroll
        for (int q = 0; q < s; ++q) fx_mac(c, F.k[s][q], Pc[0][q][0], Pc[0][q][1]);
        fx_split(fx_round(c), Pc[1][s][0], Pc[1][s][1]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          X[h][i] = fx_row<NP, S, true>(F, i, xh[h], xl[h], Pc[h]);
          if (x0 + h < cnt) mag |= fx_mag(X[h][i]);
        }
      }
    }
    if (FACES) {
      __syncthreads();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int l = fl[h], w = fr[h] + 1;
        if (l < 0) continue;
        const int how = w >= 0 ? sh.how[l] : 0;
        if (how) {
          long long add[NP];
          if (how == 1) face_correction<NP, S>(I, w, sh.Dh[l], sh.Dl[l], add);
          else face_correction_fp64<NP, S>(I, w, sh.d[l], sigw, add);
#pragma unroll
          for (int i = 0; i < NP; ++i) X[h][i] += add[i];
        }
        if (how) {
#pragma unroll
          for (int i = 0; i < NP; ++i) mag |= fx_mag(X[h][i]);
        }
        if (fr[h] < 0) {
#pragma unroll
          for (int i = 0; i < NP; ++i) sh.fx[l][fr[h] + S][i] = X[h][i];
        }
      }
    }
    sig = sigw;
    if (FACES) nm = nm + 1 == I.R ? 0 : nm + 1;
    // the block's OR of |y| and its exchange slot, then the barrier
    if (elem) {
      const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)mag);
      const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(mag >> 32));
      if (lane == 0) atomicOr(&sh.mag, ((unsigned long long)hi << 32) | lo);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = x0 + h - (cnt - HL);
        if (k >= 0 && x0 + h < cnt) {
          long long *q = exch + (((size_t)(t & 1) * nb + b) * HL + k) * NP;
#pragma unroll
          for (int i = 0; i < NP; ++i) __stcg(q + i, X[h][i]);
        }
      }
    }
    __syncthreads();
    if (face_warp && t + 1 < nsteps) ahead(t + 1);
    if (halo_warp && lane == 0) {
      const unsigned long long m = sh.mag;
      int top = m ? 64 - __clzll((long long)m) : 0;
      if (nb > 1) top = run_barrier(words, t, nb, top, bits, polls);
      sh.stop = top < 0;
      sh.bits = top;
    }
    __syncthreads();
    bits = sh.bits;
    if (sh.stop) {
      if (threadIdx.x == 0) *(volatile int *)err = 1;
      return;
    }
  }
  if (elem) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (x0 + h < cnt) {
#pragma unroll
        for (int i = 0; i < NP; ++i) out[(size_t)i * K + e0 + x0 + h] = X[h][i];
      }
  }
  if (b == 0 && threadIdx.x == 0) {
    const int s = mod_step(n0 + nsteps, 3);
    I.fx[s].mag = bits ? 1ull << (bits - 1) : 0;
    I.fx[s].E = bad ? 2047 : 0;
    I.fx[s].sigma = sig;
    const FxSlot none{};
    I.fx[fx_next(s)] = none;
    I.fx[fx_clear(s)] = none;
  }
}

// The most PE faces a tile of `most` elements (and the S - 1 before it) can hold.
int run_faces(const Inst &I, int most) { return (most + I.ns) / I.Kpe + 2; }

// Blocks and element threads of an instance's runs: a tile of about K / SMs elements, at least
// 64 (one warp; up to kRunTile elements one block, without the grid barrier: 1.6 us a sync step at
// 512 elements against 2.5 us with it).
bool run_shape(const Inst &I, int &nb, int &elems) {
  if (I.fused != 2 || !I.basis || I.K < 32 || (I.ns != 3 && I.ns != kMaxCS)) return false;
  const int sms = sm_count();
  const int tile = I.K <= kRunTile ? I.K : std::max(64, (I.K + sms - 1) / sms);
  nb = (I.K + tile - 1) / tile;
  const int most = (I.K + nb - 1) / nb;   // of the balanced tiles
  elems = ((most + 1) / 2 + 31) / 32 * 32;
  if (elems > kRunThreads || I.K / nb < 2 * kMaxCS) return false;
  return !I.async || run_faces(I, most) <= kRunFaces;
}

// The most dynamic shared memory of a block that an instance's run may take: the kernels' limit,
// set to this whatever the instance, since it belongs to the kernel and other open instances
// launch it with their own sizes.
constexpr size_t kRunSmem = 200 * 1024;

// Dynamic shared memory of a block.
size_t run_smem(const Inst &I, size_t fixed) {
  int nb, elems;
  if (!I.async || !run_shape(I, nb, elems)) return fixed;
  const int nf = run_faces(I, (I.K + nb - 1) / nb);
  return run_coef_at(fixed, nf, I.R, I.ns) + (size_t)I.L * I.q * I.q * sizeof(int);
}

template <int NP, int S, bool FACES>
cudaError_t run_prepare(const Inst &I) {
  int dev = 0, coop = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (e == cudaSuccess && !coop) return cudaErrorNotSupported;
  const size_t smem = run_smem(I, sizeof(RunShared<NP, S>));
  if (smem > kRunSmem) return cudaErrorNotSupported;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_fixed_run<NP, S, FACES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kRunSmem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fixed_run<NP, S, FACES>,
                                                      kRunBlock, smem);
  return e == cudaSuccess && per_sm < 1 ? cudaErrorNotSupported : e;
}

template <int NP, int S, bool FACES>
cudaError_t run_launch(const Inst &I, int nb, int elems, const long long *in, long long *out, int rel,
                       int nsteps, const FixedRun &R, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(R.words, 0, sizeof(RunWords), s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nb);
  // one face warp per 32 / G faces of a tile
  const int per = 32 / kFaceLanes<S>, nf = FACES ? run_faces(I, (I.K + nb - 1) / nb) : 0;
  const int most = std::min(kRunFaceWarps, (kRunBlock - 32 - elems) / 32);
  cfg.blockDim = dim3(elems + 32 + 32 * std::min(most, (nf + per - 1) / per));
  cfg.dynamicSmemBytes = run_smem(I, sizeof(RunShared<NP, S>));
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_fixed_run<NP, S, FACES>, I, in, out, rel, nsteps, elems,
                            static_cast<RunWords *>(R.words), R.exch, R.err, R.polls);
}

template <class F>
cudaError_t run_dispatch(const Inst &I, F &&f) {
  auto np = [&](auto n) -> cudaError_t {
    constexpr int NP = decltype(n)::value;
    if (I.ns == 3)
      return I.async ? f.template operator()<NP, 3, true>() : f.template operator()<NP, 3, false>();
    return I.async ? f.template operator()<NP, kMaxCS, true>() : f.template operator()<NP, kMaxCS, false>();
  };
  switch (I.Np) {
    case 2: return np(std::integral_constant<int, 2>());
    case 3: return np(std::integral_constant<int, 3>());
    case 4: return np(std::integral_constant<int, 4>());
    case 5: return np(std::integral_constant<int, 5>());
    default: return cudaErrorInvalidValue;
  }
}

struct Prepare {
  const Inst &I;
  template <int NP, int S, bool FACES>
  cudaError_t operator()() const { return run_prepare<NP, S, FACES>(I); }
};
struct Launch {
  const Inst &I;
  int nb, elems;
  const long long *in;
  long long *out;
  int rel, nsteps;
  const FixedRun &R;
  cudaStream_t s;
  template <int NP, int S, bool FACES>
  cudaError_t operator()() const {
    return run_launch<NP, S, FACES>(I, nb, elems, in, out, rel, nsteps, R, s);
  }
};

}  // namespace

size_t fixed_run_bytes(const Inst &I) {
  int nb, elems;
  if (!run_shape(I, nb, elems)) return 0;
  if (run_dispatch(I, Prepare{I}) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return sizeof(RunWords) + 2 * (size_t)nb * (2 * I.ns - 1) * I.Np * sizeof(long long);
}

FixedRun fixed_run(void *buf, int *err, long long polls) {
  return {buf, reinterpret_cast<long long *>(static_cast<char *>(buf) + sizeof(RunWords)), err, polls};
}

cudaError_t launch_fixed_run(const Inst &I, const FixedRun &R, const void *in, void *out, int rel,
                             int nsteps, cudaStream_t s) {
  int nb, elems;
  if (!R.words || nsteps < 1 || nsteps > kRunSteps || !run_shape(I, nb, elems))
    return cudaErrorInvalidValue;
  return run_dispatch(I, Launch{I, nb, elems, static_cast<const long long *>(in),
                                static_cast<long long *>(out), rel, nsteps, R, s});
}

}  // namespace adg
