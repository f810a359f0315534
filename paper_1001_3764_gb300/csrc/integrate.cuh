// integrate.cuh -- the velocity-Verlet update of one atom and the sums over a
// replica's atoms that the thermostats need, shared by the integrator
// (k_integrate.cu) and the fused step kernel (k_step.cu).
#pragma once
#include <type_traits>

#include "md_kernels.cuh"

namespace mdg {

__device__ __forceinline__ bool past_box(double x, double L) { return __double_as_longlong(x) >= __double_as_longlong(L); }
__device__ __forceinline__ bool past_box(float x, float L) { return __float_as_int(x) >= __float_as_int(L); }
__device__ __forceinline__ bool negative(double x) { return __double_as_longlong(x) < 0; }
__device__ __forceinline__ bool negative(float x) { return __float_as_int(x) < 0; }

__device__ __forceinline__ void report_move(const MoveReport& m, int j, unsigned* flags) {
  if (!m.ctl) {
    atomicOr(flags, kFlagDisplacement);
  } else if (atomicMin(m.ctl, j) == kNoMove) {
    cudaGraphSetConditional(m.handle, 1u);
    *m.events += 1ull;
  }
}

// One atom through a step's update.  MODE KKD: close the previous step's
// second half kick, open this one's first, drift; KD: the opening alone; K:
// the closing alone.  F is the force (fixed-point units in the mixed form:
// 2^-32 is folded into dt / 2m), xi and vi the state, img the image counters.
// The drift leaves the FP32 cell-unit position in loc and reports
// displacement (moved) and non-finite values (bad).  KE: the v^2 (and with
// Nose-Hoover, TH = 2, the v) that the thermostat asks for, weighted by the
// atom's mass over mass[0]: chain ends alone pay a multiplication on the
// narrow FP64 pipe, and the sums are scaled once.
struct AtomOut {
  float loc[3];
  bool moved, bad;
  double ke, mom[3];
};
template <int TH, class T>
__device__ __forceinline__ void kinetic_terms(const T (&vi)[3], int type, const ForceParams& fp, AtomOut& o) {
  const double u[3] = {(double)vi[0], (double)vi[1], (double)vi[2]};
  o.ke = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  if (TH == 2)
#pragma unroll
    for (int a = 0; a < 3; ++a) o.mom[a] = u[a];
  if (type) {
    o.ke *= fp.mass_ratio;
    if (TH == 2)
#pragma unroll
      for (int a = 0; a < 3; ++a) o.mom[a] *= fp.mass_ratio;
  }
}

// Nose-Hoover factor k of a replica in the state's type
template <class T>
__device__ __forceinline__ T nh_factor(const double* __restrict__ lam, int rep, int k) {
  const double* nh = lam + (size_t)kNhDoubles * rep;
  if constexpr (sizeof(T) == 8) return nh[k];
  else return reinterpret_cast<const float*>(nh + 12)[k];
}

template <bool MIXED, int MODE, bool KE, int TH, class T>
__device__ __forceinline__ void integrate_atom(const T (&F)[3], T (&xi)[3], T (&vi)[3], int* __restrict__ img, int i,
                                               int N, int type, int cc, float4 r0, const RepDev& R, int rep,
                                               const ForceParams& fp, const double* __restrict__ lam, AtomOut& o) {
  T hdt_m;
  if constexpr (MIXED) hdt_m = fp.hdt_m_fix[type]; else hdt_m = fp.hdt_m_f[type];
  o.ke = 0.0;
  o.mom[0] = o.mom[1] = o.mom[2] = 0.0;
  o.moved = o.bad = false;
  // Without a kinetic-energy read-out the two half kicks of KKD are one
  // kick of dt F/m (the full-step velocity is never needed in between).
  constexpr bool kMerged = MODE == kKickKickDrift && !KE;
  // Nose-Hoover in the mixed form takes KKD's two kicks in one (below)
  constexpr bool kOneKick = MIXED && TH == 2 && MODE == kKickKickDrift;
  if constexpr ((MODE == kKickKickDrift && KE && !kOneKick) || MODE == kKickOnly) {
    if constexpr (TH == 2) {
      const T fc = nh_factor<T>(lam, rep, 2);
#pragma unroll
      for (int a = 0; a < 3; ++a) vi[a] = (vi[a] - nh_factor<T>(lam, rep, 3 + a) + hdt_m * F[a]) * fc;   // v_k
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) vi[a] += hdt_m * F[a];   // v(t): close the previous step
    }
  }
  if constexpr (KE && TH != 2) kinetic_terms<TH>(vi, type, fp, o);
  if constexpr (MODE == kKickDrift || MODE == kKickKickDrift) {
    if (TH == 1) {
      const T l = (T)lam[rep];
#pragma unroll
      for (int a = 0; a < 3; ++a) vi[a] *= l;
    }
    T dt, L;
    if constexpr (MIXED) { dt = fp.dt; L = R.L; } else { dt = fp.dt_f; L = R.Lf; }
    const float r0a[3] = {r0.x, r0.y, r0.z};
    const float halfM = 0.5f * R.Mf;
    float d2 = 0.f;
    bool bad = false;
    // Nose-Hoover: v_{k+1/2} = fo v_k + dt F / 2m; kOneKick puts in v_k =
    // (v_{k-1/2} - V_com + dt F / 2m) fc: A v - A V_com + (1 + A) dt F / 2m,
    // two FMAs per component of the narrow FP64 pipe instead of five operations
    T va = (T)1, fb = (T)1;
    if constexpr (TH == 2) {
      va = nh_factor<T>(lam, rep, kOneKick ? 6 : 1);
      fb = kOneKick ? hdt_m * nh_factor<T>(lam, rep, 7) : hdt_m;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if constexpr (kOneKick) vi[a] = fma(va, vi[a], fma(fb, F[a], -nh_factor<T>(lam, rep, 8 + a)));
      else if constexpr (TH == 2) vi[a] = vi[a] * va + fb * F[a];
      else vi[a] = kMerged ? vi[a] + (hdt_m + hdt_m) * F[a] : vi[a] + hdt_m * F[a];
      T xa = xi[a] + dt * vi[a];
      // wrap into [0, L): for non-negative IEEE numbers the bit patterns
      // order like the values, so the tests run on the integer pipe
      if (past_box(xa, L)) { xa -= L; img[a * N + i] += 1; }
      else if (negative(xa)) { xa += L; img[a * N + i] -= 1; if (past_box(xa, L)) xa = (T)0; }
      xi[a] = xa;
      // cell units in the frame of the rebin cell; an atom that crossed a
      // face since the rebin is moved back by one box (M cell units)
      const int c = (cc >> (10 * a)) & 1023;
      float ua;
      if constexpr (MIXED) ua = cell_unit_t(xa, c, R); else ua = cell_unit(xa, c, 0, R);
      const float du = ua - r0a[a];
      if (du > halfM || du < -halfM) {
        if constexpr (MIXED) ua = cell_unit_tw(xa, c, du > halfM ? -1 : 1, R);
        else ua = cell_unit(xa, c, du > halfM ? -1 : 1, R);
      }
      o.loc[a] = ua;
      const float d = ua - r0a[a];
      d2 += d * d;
      bad |= !isfinite(ua);          // a non-finite x or v reaches u
    }
    o.moved = d2 > R.hs2u;
    o.bad = bad;
    if constexpr (TH == 2) kinetic_terms<TH>(vi, type, fp, o);
  }
}

// Sums over the block's threads of NV values each, val[a][thread], left in
// val[a][0] on return (a barrier included): every stage adds four values per
// thread, so 256 values take 4 stages of 3 dependent additions, and the adds
// of all NV values fill whole warps.  This GPU's FP64 pipe is narrow: a
// shuffle tree would issue five adds on every lane, and one thread per 32
// values (the former form) is a chain of 40.  The order depends on the block
// size alone.
template <int NV, int NT>
__device__ __forceinline__ void block_sums(double (&val)[NV][NT]) {
  int m = blockDim.x;
  __syncthreads();
  while (m > 1) {
    const int q = (m + 3) >> 2;
    for (int u = threadIdx.x; u < NV * q; u += blockDim.x) {
      const int a = u / q, j = u - a * q;
      double s = val[a][j];
#pragma unroll
      for (int k = 1; k < 4; ++k)
        if (j + k * q < m) s += val[a][j + k * q];
      val[a][j] = s;
    }
    m = q;
    __syncthreads();
  }
}

// Kinetic energy (and with Nose-Hoover the momentum) of a replica: every
// block leaves the sums of its tile, and the last block of the replica to
// finish (a ticket per replica; no waiting) adds the replica's tiles, in an
// order that depends only on their number, and sets the thermostat factors of
// the next step.  One ticket per replica lets the replicas finish side by
// side: with one for the whole launch, a single block went through 64
// replicas one after another (100 us of a 152 us launch).
template <int TH, int NT>
__device__ __forceinline__ void replica_kinetic(const AtomOut& o, int rep, int tile, int first_tile, int n_tiles,
                                                const RepDev* __restrict__ reps, const ForceParams& fp,
                                                double* __restrict__ kepart, unsigned* __restrict__ done,
                                                double* __restrict__ ke_out, double* __restrict__ lam, double tau) {
  constexpr int NV = TH == 2 ? 4 : 1;
  __shared__ double vals[NV][NT];
  __shared__ bool last;
  const int tid = threadIdx.x;
  vals[0][tid] = o.ke;
  if constexpr (TH == 2) {
#pragma unroll
    for (int a = 0; a < 3; ++a) vals[1 + a][tid] = o.mom[a];
  }
  block_sums<NV, NT>(vals);
  if (tid < NV) kepart[(size_t)NV * tile + tid] = vals[tid][0];
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(done + rep, 1u) == (unsigned)n_tiles - 1u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  double P[NV];
#pragma unroll
  for (int a = 0; a < NV; ++a) P[a] = 0.0;
#pragma unroll 4
  for (int q = tid; q < n_tiles; q += blockDim.x)
#pragma unroll
    for (int a = 0; a < NV; ++a) P[a] += __ldcg(kepart + (size_t)NV * (first_tile + q) + a);
#pragma unroll
  for (int a = 0; a < NV; ++a) vals[a][tid] = P[a];
  block_sums<NV, NT>(vals);
  if (tid != 0) return;
  done[rep] = 0u;
  const RepDev& Q = reps[rep];
  const double sum = 0.5 * fp.mass[0] * vals[0][0];
  ke_out[rep] = sum;
  if (TH == 1) {
    const double T_inst = 2.0 * sum / (Q.dof * 0.0083144626);
    lam[rep] = sqrt(1.0 + fp.dt / tau * (Q.T0 / T_inst - 1.0));
  }
  if constexpr (TH == 2) {
    const double T_half = 2.0 * sum / (Q.dof * 0.0083144626);
    const double Qm = tau * tau * Q.T0 / (4.0 * 3.14159265358979323846 * 3.14159265358979323846);
    double* nh = lam + (size_t)kNhDoubles * rep;
    const double xi = nh[0] + fp.dt * (T_half - Q.T0) / Qm;
    const double c = 0.5 * fp.dt * xi;
    const double s = fp.mass[0] / ((double)Q.n_chains * fp.mol_mass);
    nh[0] = xi; nh[1] = 1.0 - c; nh[2] = 1.0 / (1.0 + c);
    const double A = nh[1] * nh[2];
    nh[6] = A; nh[7] = 1.0 + A;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      nh[3 + a] = s * vals[1 + a][0];
      nh[8 + a] = A * nh[3 + a];
    }
    float* nf = reinterpret_cast<float*>(nh + 12);
    for (int k = 0; k < 11; ++k) nf[k] = (float)nh[k];
  }
}

}  // namespace mdg
