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
  const double u[3] = {f2d_int(vi[0]), f2d_int(vi[1]), f2d_int(vi[2])};
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

// Sums over n threads' values, NV rows of val (stride `stride`), left in
// place 0 of each row on return (a barrier included): every stage adds four
// values per thread, so 256 values take 4 stages of 3 dependent additions, and
// the adds of all NV values fill whole warps.  This GPU's FP64 pipe is narrow:
// a shuffle tree would issue five adds on every lane, and one thread per 32
// values (the former form) is a chain of 40.  The order depends on n alone.
template <int NV>
__device__ __forceinline__ void block_sums(double* val, int stride, int n) {
  int m = n;
  __syncthreads();
  while (m > 1) {
    const int q = (m + 3) >> 2;
    for (int u = threadIdx.x; u < NV * q; u += blockDim.x) {
      const int a = u / q, j = u - a * q;
      double* row = val + a * stride;
      double s = row[j];
#pragma unroll
      for (int k = 1; k < 4; ++k)
        if (j + k * q < m) s += row[j + k * q];
      row[j] = s;
    }
    m = q;
    __syncthreads();
  }
}

// Kinetic energy (and with Nose-Hoover the momentum) of a tile, left in kepart
template <int TH, int NT>
__device__ __forceinline__ void tile_kinetic(const AtomOut& o, int tile, double* __restrict__ kepart) {
  constexpr int NV = TH == 2 ? 4 : 1;
  __shared__ double vals[NV][NT];
  vals[0][threadIdx.x] = o.ke;
  if constexpr (TH == 2) {
#pragma unroll
    for (int a = 0; a < 3; ++a) vals[1 + a][threadIdx.x] = o.mom[a];
  }
  block_sums<NV>(&vals[0][0], NT, blockDim.x);
  if (threadIdx.x < NV) kepart[(size_t)NV * tile + threadIdx.x] = vals[threadIdx.x][0];
}

// A replica's sums over its tiles, in an order that depends only on their
// number: sum of value a at val[a * blockDim.x] (a barrier included).  val
// holds NV rows of blockDim.x doubles.
template <int NV>
__device__ __forceinline__ void replica_sums(const double* __restrict__ kepart, int first_tile, int n_tiles,
                                             double* val) {
  double P[NV];
#pragma unroll
  for (int a = 0; a < NV; ++a) P[a] = 0.0;
#pragma unroll 4
  for (int q = threadIdx.x; q < n_tiles; q += blockDim.x)
#pragma unroll
    for (int a = 0; a < NV; ++a) P[a] += __ldcg(kepart + (size_t)NV * (first_tile + q) + a);
#pragma unroll
  for (int a = 0; a < NV; ++a) val[a * blockDim.x + threadIdx.x] = P[a];
  block_sums<NV>(val, blockDim.x, blockDim.x);
}

// The thermostat factors of the next drift, by a block of the LJ launch that
// follows a drift: the sums wait for no one there, where a last block of the
// drift's launch added a ticket, a fence and a lone block's 5 us to it (150k
// plain: 18.4 -> 11.4 us per update; 35k Nose-Hoover 14.4 -> 8.9).
__device__ __forceinline__ void replica_thermostat(const ThermoArgs& ta, const RepDev& Q, int rep, double* val) {
  const int first = ta.chain ? Q.ctile_off : Q.tile_off, n = ta.chain ? Q.n_ctiles : Q.n_tiles;
  if (ta.th == 1) {
    replica_sums<1>(ta.kepart, first, n, val);
    if (threadIdx.x != 0) return;
    const double sum = val[0];
    ta.lam[rep] = sqrt(ta.one_minus_rate + Q.vr_num / sum);
    return;
  }
  replica_sums<4>(ta.kepart, first, n, val);
  if (threadIdx.x != 0) return;
  double* nh = ta.lam + (size_t)kNhDoubles * rep;
  const double xi = nh[0] + Q.nh_rate * (Q.t_scale * val[0] - Q.T0);
  const double c = 0.5 * ta.dt * xi;
  nh[0] = xi; nh[1] = 1.0 - c; nh[2] = 1.0 / (1.0 + c);
  const double A = nh[1] * nh[2];
  nh[6] = A; nh[7] = 1.0 + A;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    nh[3 + a] = Q.com_scale * val[(1 + a) * blockDim.x];
    nh[8 + a] = A * nh[3 + a];
  }
  float* nf = reinterpret_cast<float*>(nh + 12);
  for (int k = 0; k < 11; ++k) nf[k] = (float)nh[k];
}

}  // namespace mdg
