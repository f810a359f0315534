// k_integrate.cu -- velocity-Verlet update (Sec. 3.4), kinetic energy and
// weak-coupling thermostat, energy reductions.
//
// Velocity Verlet gives the positions of the paper's Leap-Frog scheme.  A
// step is split as: [complete the previous step's second half-kick, kinetic
// energy, thermostat scale] + [first half-kick, drift] in one kernel (mode
// KKD); a call's first step skips the completion (KD) and its last step is
// closed by a kick-only pass (K), so the state at every API boundary is
// (x(t), v(t), F(t)).
//
// The paper's Nose-Hoover coupling needs the whole-system kinetic energy,
// which it sums through a per-atom array and a tree reduction (Sec. 3.4).
// Here each block writes one FP64 partial, and a block per replica of the LJ
// launch that follows sums the replica's partials in a fixed order and
// computes its rescaling factor.
// The factor computed at step k is applied at step k+1 (one-step lag).
//
// Nose-Hoover (TH = 2; the paper's NVT ensemble with Leap-Frog, Sec. 2 and
// 3.4): per replica xi_k, 1 - c_k, 1/(1 + c_k), V_com (kNhDoubles in
// md_kernels.cuh), c_k = dt xi_k / 2.  A step closes v_k = (v_{k-1/2} - V_com + dt F/(2m)) /
// (1 + c_k), opens v_{k+1/2} = (1 - c_k) v_k + dt F/(2m) and drifts; the
// replica's block of the LJ launch takes T_{k+1/2} and the momentum of v_{k+1/2} and leaves
// xi_{k+1} = xi_k + dt (T_{k+1/2} - T0)/Q, Q = tau^2 T0/(4 pi^2), and the
// centre-of-mass velocity that the next step subtracts.  This is the
// leap-frog update v_{k+1/2} = [v_{k-1/2}(1 - c_k) + dt F/m]/(1 + c_k).
//
// The drift also refreshes the FP32 cell-unit positions in sorted order for
// the force kernels, wraps positions into [0, L) with image counters, and
// flags atoms that moved more than skin/2 since the last rebin.
//
// The update of an atom and the thermostats' sums are in integrate.cuh,
// shared with the fused step kernels (k_step.cu), which do every inner and
// closing update of a block of steps; this kernel opens a block and reads out
// the kinetic energy.
#include <type_traits>

#include "integrate.cuh"

namespace mdg {

constexpr int kIntBlock = 256;

template <bool MIXED, int MODE, bool KE, int TH>
__global__ void __launch_bounds__(kIntBlock) k_integrate(void* __restrict__ xv, void* __restrict__ vv,
                                                         int* __restrict__ img, const void* __restrict__ Fv,
                                                         const uint16_t* __restrict__ site,
                                                         const int* __restrict__ cellc,
                                                         const int* __restrict__ inv_perm,
                                                         const float4* __restrict__ ref, float4* __restrict__ pos,
                                                         long long* __restrict__ flj_next, int Npad, int N,
                                                         const Tile* __restrict__ tiles,
                                                         const RepDev* __restrict__ reps, const ForceParams fp,
                                                         double* __restrict__ kepart, const double* __restrict__ lam,
                                                         unsigned* __restrict__ flags, const StepGate gate, const MoveReport mr) {
  using T = typename std::conditional<MIXED, double, float>::type;
  T* x = reinterpret_cast<T*>(xv);
  T* v = reinterpret_cast<T*>(vv);
  wait_for_predecessor();
  const Tile t = tiles[blockIdx.x];
  const RepDev& R = reps[t.rep];
  const int i = t.start + threadIdx.x;
  if (!drift_runs(gate)) return;
  AtomOut o;
  o.ke = 0.0;
  o.mom[0] = o.mom[1] = o.mom[2] = 0.0;
  if ((int)threadIdx.x < t.len) {
    const int type = atom_type(site[i], fp);
    T F[3] = {(T)0, (T)0, (T)0}, xi[3] = {(T)0, (T)0, (T)0}, vi[3] = {v[i], v[N + i], v[2 * N + i]};
    if (MODE == kKineticOnly) {
    } else if (MIXED) {
      const F4i f = reinterpret_cast<const F4i*>(Fv)[i];
      F[0] = fix_to_double_i(f.x); F[1] = fix_to_double_i(f.y); F[2] = fix_to_double_i(f.z);   // integer pipe
    } else {
      const float4 f = reinterpret_cast<const float4*>(Fv)[i];
      F[0] = f.x; F[1] = f.y; F[2] = f.z;
    }
    int cc = 0;
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    constexpr bool kDrift = MODE == kKickDrift;
    if (kDrift) {
      cc = cellc[i];
      r0 = ref[i];
#pragma unroll
      for (int a = 0; a < 3; ++a) xi[a] = x[a * N + i];
    }
    integrate_atom<MIXED, MODE, KE, TH>(F, xi, vi, img, i, N, type, cc, r0, R, t.rep, fp, lam, o);
    if (kDrift) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        v[a * N + i] = vi[a];
        x[a * N + i] = xi[a];
        flj_next[(size_t)a * Npad + i] = 0ll;
      }
      if (o.moved) report_move(mr, gate.j, flags);
      if (o.bad) atomicOr(flags, kFlagNaN);
      pos[inv_perm[i]] = make_float4(o.loc[0], o.loc[1], o.loc[2], (float)type);   // w: LJ type, as the sort writes it
    }
  }
  if constexpr (KE) tile_kinetic<TH, kIntBlock>(o, blockIdx.x, kepart);
}

template <bool MIXED>
static void launch_int_t(IntegMode mode, int th, const StepArgs& a, const ForceParams& fp,
                         const StepGate& gate, const MoveReport& mr, cudaStream_t st) {
#define MDG_INT(MODE, KE, TH)                                                                                        \
  launch_dependent(gate.dep, k_integrate<MIXED, MODE, KE, TH>, a.n_tiles, kIntBlock, 0, st, a.x, a.v, a.img, a.F, a.site,      \
                   a.cellc, a.inv_perm, a.ref, a.pos, a.flj_next, a.Npad, a.N, a.tiles, a.reps, fp, a.kepart, a.lam, \
                   a.flags, gate, mr)
  // With the weak-coupling thermostat (th = 1), every step that starts (KD,
  // KKD) takes the temperature of the unscaled v(t_k), scales v(t_k) by the
  // factor of the previous step and leaves the factor of step k for the next
  // one.  With Nose-Hoover (th = 2) every KD and KKD sums the kinetic energy
  // and momentum of v_{k+1/2} for xi_{k+1} and the centre-of-mass velocity.
  // The closing kick (K) only completes v; the next call's KD picks up from
  // there.
  if (mode == kKickDrift) {
    if (th == 2) MDG_INT(kKickDrift, true, 2);
    else if (th == 1) MDG_INT(kKickDrift, true, 1);
    else MDG_INT(kKickDrift, false, 0);
  } else {
    MDG_INT(kKineticOnly, true, 0);
  }
#undef MDG_INT
}

void launch_integrate(bool mixed, IntegMode mode, int thermostat, const StepArgs& a, const ForceParams& fp,
                      const StepGate& gate, const MoveReport& mr, cudaStream_t st) {
  if (a.n_tiles <= 0) return;
  if (mixed) launch_int_t<true>(mode, thermostat, a, fp, gate, mr, st);
  else launch_int_t<false>(mode, thermostat, a, fp, gate, mr, st);
}

// kinetic energies of the replicas from the tiles' sums (a read-out)
constexpr int kKineticThreads = 256;
__global__ void __launch_bounds__(kKineticThreads) k_kinetic(const double* __restrict__ kepart,
                                                             const RepDev* __restrict__ reps, double half_m0,
                                                             double* __restrict__ ke_out) {
  __shared__ double val[kKineticThreads];
  const RepDev& Q = reps[blockIdx.x];
  replica_sums<1>(kepart, Q.tile_off, Q.n_tiles, val);
  if (threadIdx.x == 0) ke_out[blockIdx.x] = half_m0 * val[0];
}

void launch_kinetic(const double* kepart, const RepDev* reps, int n_reps, const ForceParams& fp, double* ke_out,
                    cudaStream_t st) {
  if (n_reps > 0) k_kinetic<<<n_reps, kKineticThreads, 0, st>>>(kepart, reps, 0.5 * fp.mass[0], ke_out);
}

// ---------------------------------------------------------------- early rebin
__global__ void __launch_bounds__(32) k_resume(cudaGraphConditionalHandle h, int* __restrict__ ctl) {
  if (threadIdx.x != 0) return;
  ctl[1] = ctl[0];
  ctl[0] = kNoMove;
  cudaGraphSetConditional(h, 0u);
}

void launch_resume(cudaGraphConditionalHandle h, int* ctl, cudaStream_t st) { k_resume<<<1, 32, 0, st>>>(h, ctl); }

// ---------------------------------------------------------------- energy reduction
// LJ partials are per cell (replica r owns cells [cell_base, cell_base + M^3)),
// bonded partials per integrator tile.  Fixed summation order.
// out[r*16 + k]: k = 0 lj, 1 lj_shifted, 2 bond, 3 angle, 4 dihedral, 5..10 virial
// Two passes, spread over the GPU (FP64 adds are slow on one SM):
//  1. slice j of replica r covers its cells [j*1024, (j+1)*1024) and the same
//     share of its bonded tiles; thread t adds every 256th entry in order,
//     then a fixed tree over the block (warp shuffles, then the warps in
//     order) gives the slice's 11 sums;
//  2. one warp per replica adds its slices in slice order.
// The slices of a replica depend only on its own size, so a replica gets the
// same bits alone or batched with others.
constexpr int kRedThreads = 256;

__host__ __device__ inline int energy_slices(int n_cells) { return (n_cells + kEnergySliceCells - 1) / kEnergySliceCells; }

__global__ void __launch_bounds__(kRedThreads) k_energy_slices(const double* __restrict__ lj_part,
                                                               const double* __restrict__ b_part,
                                                               const RepDev* __restrict__ reps, int max_slices,
                                                               double* __restrict__ slices) {
  __shared__ double sh[11][kRedThreads / 32];
  const int r = blockIdx.x / max_slices, j = blockIdx.x % max_slices;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const RepDev& R = reps[r];
  const int nc = R.M * R.M * R.M, ns = energy_slices(nc);
  if (j >= ns) return;
  const int lt = (R.n_tiles + ns - 1) / ns;
  double acc[11] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  const int c0 = R.cell_base + j * kEnergySliceCells, c1 = R.cell_base + min(nc, (j + 1) * kEnergySliceCells);
  for (int c = c0 + tid; c < c1; c += kRedThreads) {
    const double* p = lj_part + (size_t)c * 8;
    acc[0] += p[0]; acc[1] += p[1];
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[5 + k] += p[2 + k];
  }
  const int q0 = R.tile_off + j * lt, q1 = R.tile_off + min(R.n_tiles, (j + 1) * lt);
  for (int q = q0 + tid; q < q1; q += kRedThreads) {
    const double* p = b_part + (size_t)q * 9;
    acc[2] += p[0]; acc[3] += p[1]; acc[4] += p[2];
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[5 + k] += p[3 + k];
  }
#pragma unroll
  for (int k = 0; k < 11; ++k) {
    double v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[k][w] = v;
  }
  __syncthreads();
  if (tid < 11) {
    double v = 0.0;
    for (int q = 0; q < kRedThreads / 32; ++q) v += sh[tid][q];
    slices[(size_t)blockIdx.x * 11 + tid] = v;
  }
}

__global__ void __launch_bounds__(32) k_energy_reduce(const double* __restrict__ slices, const RepDev* __restrict__ reps,
                                                      int max_slices, double* __restrict__ out) {
  const int r = blockIdx.x, k = threadIdx.x;
  if (k >= 11) return;
  const int ns = energy_slices(reps[r].M * reps[r].M * reps[r].M);
  double v = 0.0;
  for (int j = 0; j < ns; ++j) v += slices[((size_t)r * max_slices + j) * 11 + k];
  out[r * 16 + k] = v;
}

int energy_slice_count(int n_cells) { return energy_slices(n_cells); }

void launch_energy_reduce(const double* lj_part, const double* b_part, const RepDev* reps, int n_reps, int max_slices,
                          double* slices, double* out, cudaStream_t st) {
  if (n_reps <= 0) return;
  k_energy_slices<<<n_reps * max_slices, kRedThreads, 0, st>>>(lj_part, b_part, reps, max_slices, slices);
  k_energy_reduce<<<n_reps, 32, 0, st>>>(slices, reps, max_slices, out);
}

// ------------------------------------------------------------ chain observables
// One warp per chain (the structural observables of the paper's Sec. 5):
// the chain is made continuous by minimum-image bonds, R_ee = x_last -
// x_first (Fig. 8), R_g^2 = sum m |x - x_cm|^2 / sum m (mass-weighted, from
// sums relative to site 0), and the number of backbone dihedrals in the trans
// state, |phi| > 120 deg, i.e. cos(phi) = n1.n2 / (|n1||n2|) < -1/2 with n1 =
// b1 x b2, n2 = b2 x b3 (IUPAC, trans at 180 deg).  The trans counts of a
// replica are added as integers.
// Lane l of a warp takes sites l, l + 32, ...: a thread per chain walked 150
// sites alone, with 1,000 threads on the GPU and loads 1,200 bytes apart.
// A site's whole-box shift is the number of face crossings up to it, counted
// by ballots, so the continuous position is one FMA and no serial sum.
// 150k sites: 383 -> 27 us.
constexpr int kObsWarps = 4;

template <class T>
__global__ void __launch_bounds__(32 * kObsWarps) k_chain_observables(const T* __restrict__ x, int N,
                                                                      const RepDev* __restrict__ reps, int n_reps,
                                                                      const ForceParams fp, int n_chains_total,
                                                                      double* __restrict__ ree,
                                                                      double* __restrict__ rg2,
                                                                      unsigned long long* __restrict__ trans) {
  const int c = blockIdx.x * kObsWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= n_chains_total) return;   // the whole warp leaves together
  int lo = 0, hi = n_reps - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (reps[mid].chain_off <= c) lo = mid; else hi = mid - 1;
  }
  const int r = lo;
  const RepDev& R = reps[r];
  const int S = fp.sites;
  const int o = R.atom_off + (c - R.chain_off) * S;
  const double L = R.L, hL = R.half_L;
  const double x0[3] = {(double)x[o], (double)x[N + o], (double)x[2 * N + o]};
  const unsigned le = 0xffffffffu >> (31 - lane);   // this lane and those before it
  int shift[3] = {0, 0, 0};                         // whole boxes up to the previous chunk's last site
  double px[3] = {x0[0], x0[1], x0[2]};             // that site's position
  double pb[3] = {0.0, 0.0, 0.0}, pn[3] = {0.0, 0.0, 0.0};   // its bond and normal (used from site 3 on)
  double m_sum = 0.0, s1[3] = {0.0, 0.0, 0.0}, s2 = 0.0, end[3] = {0.0, 0.0, 0.0};
  int nt = 0;
  for (int k0 = 0; k0 < S; k0 += 32) {
    const int k = k0 + lane;
    const bool on = k < S;
    double b[3], p[3], xk[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      xk[a] = on ? (double)x[a * N + o + k] : px[a];
      double prev = __shfl_up_sync(0xffffffffu, xk[a], 1);
      if (lane == 0) prev = px[a];
      double e = xk[a] - prev;
      const bool dn = e > hL, up = e < -hL;         // crossed the lower / upper face
      if (dn) e -= L; else if (up) e += L;
      b[a] = e;
      const unsigned bu = __ballot_sync(0xffffffffu, up && on), bd = __ballot_sync(0xffffffffu, dn && on);
      const int sh = shift[a] + __popc(bu & le) - __popc(bd & le);
      shift[a] += __popc(bu) - __popc(bd);
      p[a] = fma((double)sh, L, xk[a]) - x0[a];
      px[a] = __shfl_sync(0xffffffffu, xk[a], 31);
    }
    double q[3], n[3], nq[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      q[a] = __shfl_up_sync(0xffffffffu, b[a], 1);
      if (lane == 0) q[a] = pb[a];
      pb[a] = __shfl_sync(0xffffffffu, b[a], 31);
    }
    n[0] = q[1] * b[2] - q[2] * b[1];
    n[1] = q[2] * b[0] - q[0] * b[2];
    n[2] = q[0] * b[1] - q[1] * b[0];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      nq[a] = __shfl_up_sync(0xffffffffu, n[a], 1);
      if (lane == 0) nq[a] = pn[a];
      pn[a] = __shfl_sync(0xffffffffu, n[a], 31);
    }
    const double dn = nq[0] * n[0] + nq[1] * n[1] + nq[2] * n[2];
    const double l2 = n[0] * n[0] + n[1] * n[1] + n[2] * n[2];
    const double l1 = nq[0] * nq[0] + nq[1] * nq[1] + nq[2] * nq[2];
    // cos(phi) < -1/2  <=>  n1.n2 < 0 and (n1.n2)^2 > |n1|^2 |n2|^2 / 4
    const bool tr = on && k >= 3 && dn < 0.0 && 4.0 * dn * dn > l1 * l2;
    nt += __popc(__ballot_sync(0xffffffffu, tr));
    if (on) {
      const double m = fp.mass[(k == 0 || k == S - 1) ? 1 : 0];
      m_sum += m;
#pragma unroll
      for (int a = 0; a < 3; ++a) s1[a] += m * p[a];
      s2 += m * (p[0] * p[0] + p[1] * p[1] + p[2] * p[2]);
      if (k == S - 1)
#pragma unroll
        for (int a = 0; a < 3; ++a) end[a] = p[a];
    }
  }
  const int last = (S - 1) & 31;
#pragma unroll
  for (int a = 0; a < 3; ++a) end[a] = __shfl_sync(0xffffffffu, end[a], last);
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    m_sum += __shfl_xor_sync(0xffffffffu, m_sum, m);
    s2 += __shfl_xor_sync(0xffffffffu, s2, m);
#pragma unroll
    for (int a = 0; a < 3; ++a) s1[a] += __shfl_xor_sync(0xffffffffu, s1[a], m);
  }
  if (lane != 0) return;
#pragma unroll
  for (int a = 0; a < 3; ++a) ree[3 * c + a] = end[a];
  const double cx = s1[0] / m_sum, cy = s1[1] / m_sum, cz = s1[2] / m_sum;
  rg2[c] = s2 / m_sum - (cx * cx + cy * cy + cz * cz);
  if (nt) atomicAdd(trans + r, (unsigned long long)nt);
}

void launch_chain_observables(bool mixed, const void* x, int N, const RepDev* reps, int n_reps,
                              const ForceParams& fp, int n_chains_total, double* ree, double* rg2,
                              unsigned long long* trans, cudaStream_t st) {
  const int blocks = (n_chains_total + kObsWarps - 1) / kObsWarps;
  if (blocks == 0) return;
  if (mixed)
    k_chain_observables<double><<<blocks, 32 * kObsWarps, 0, st>>>((const double*)x, N, reps, n_reps, fp,
                                                                   n_chains_total, ree, rg2, trans);
  else
    k_chain_observables<float><<<blocks, 32 * kObsWarps, 0, st>>>((const float*)x, N, reps, n_reps, fp,
                                                                  n_chains_total, ree, rg2, trans);
}

// ------------------------------------------------------------------ output state
// SoA state -> AoS FP64 positions, velocities and image counters (null: not
// wanted).  One element of the AoS arrays per thread: whole lines are written (the reads, a
// third of a line per row, meet in L1).  With an atom per thread the writes were
// 24 bytes apart (1.5M sites: 38.6 -> 34.9 us).
template <bool MIXED>
__global__ void __launch_bounds__(256) k_egress_state(const void* __restrict__ xv, const void* __restrict__ vv,
                                                      const int* __restrict__ img, int N, double* __restrict__ pos,
                                                      double* __restrict__ vel, int* __restrict__ im) {
  using T = typename std::conditional<MIXED, double, float>::type;
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;   // 3 N < 2^28
  if (e >= 3u * (unsigned)N) return;
  const unsigned i = e / 3u, q = (e - 3u * i) * (unsigned)N + i;
  if (pos) pos[e] = (double)reinterpret_cast<const T*>(xv)[q];
  if (vel) vel[e] = (double)reinterpret_cast<const T*>(vv)[q];
  if (im) im[e] = img[q];
}

// total force (int64 fixed point or FP32) -> AoS FP64 kJ/mol/nm
template <bool MIXED>
__global__ void __launch_bounds__(256) k_egress_forces(const void* __restrict__ Fv, int N, double scale,
                                                       double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  if constexpr (MIXED) {
    const F4i f = reinterpret_cast<const F4i*>(Fv)[i];
    out[3 * (size_t)i] = fix_to_double_i(f.x) * scale;
    out[3 * (size_t)i + 1] = fix_to_double_i(f.y) * scale;
    out[3 * (size_t)i + 2] = fix_to_double_i(f.z) * scale;
  } else {
    const float4 f = reinterpret_cast<const float4*>(Fv)[i];
    out[3 * (size_t)i] = f.x; out[3 * (size_t)i + 1] = f.y; out[3 * (size_t)i + 2] = f.z;
  }
}

void launch_egress_state(bool mixed, const void* x, const void* v, const int* img, int N, double* pos, double* vel,
                         int* im, cudaStream_t st) {
  if (N <= 0) return;
  if (mixed) k_egress_state<true><<<(3 * N + 255) / 256, 256, 0, st>>>(x, v, img, N, pos, vel, im);
  else k_egress_state<false><<<(3 * N + 255) / 256, 256, 0, st>>>(x, v, img, N, pos, vel, im);
}

void launch_egress_forces(bool mixed, const void* F, int N, double scale, double* out, cudaStream_t st) {
  if (N <= 0) return;
  if (mixed) k_egress_forces<true><<<(N + 255) / 256, 256, 0, st>>>(F, N, scale, out);
  else k_egress_forces<false><<<(N + 255) / 256, 256, 0, st>>>(F, N, scale, out);
}

// ------------------------------------------------------------------ input state
template <bool MIXED>
__global__ void __launch_bounds__(kIntBlock) k_ingest(const double* __restrict__ pos, const double* __restrict__ vel, int N,
                                                      const Tile* __restrict__ tiles, const RepDev* __restrict__ reps,
                                                      void* __restrict__ xv, void* __restrict__ vv,
                                                      int* __restrict__ img, unsigned* __restrict__ flags) {
  using T = typename std::conditional<MIXED, double, float>::type;
  const Tile t = tiles[blockIdx.x];
  if ((int)threadIdx.x >= t.len) return;
  const RepDev& R = reps[t.rep];
  const int i = t.start + threadIdx.x;
  T* x = reinterpret_cast<T*>(xv);
  T* v = reinterpret_cast<T*>(vv);
  bool bad = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double xa = pos[3 * (size_t)i + a];
    const double va = vel[3 * (size_t)i + a];
    bad |= !isfinite(xa) || !isfinite(va);
    xa -= R.L * floor(xa / R.L);
    if (!(xa < R.L) || xa < 0.0) xa = 0.0;
    if (!MIXED && (float)xa >= R.Lf) xa = 0.0;
    x[a * N + i] = (T)xa;
    v[a * N + i] = (T)va;
    img[a * N + i] = 0;
  }
  if (bad) atomicOr(flags, kFlagBadInput);
}

void launch_ingest(bool mixed, const double* pos, const double* vel, int N, const Tile* tiles, int n_tiles, const RepDev* reps,
                   void* x, void* v, int* img, unsigned* flags, cudaStream_t st) {
  if (n_tiles <= 0) return;
  if (mixed) k_ingest<true><<<n_tiles, kIntBlock, 0, st>>>(pos, vel, N, tiles, reps, x, v, img, flags);
  else k_ingest<false><<<n_tiles, kIntBlock, 0, st>>>(pos, vel, N, tiles, reps, x, v, img, flags);
}

}  // namespace mdg
