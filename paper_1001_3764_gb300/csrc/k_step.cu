// k_step.cu -- bonded forces (Eqs. 4-6, Sec. 3.3) and the velocity-Verlet
// update (Sec. 3.4) of linear chains in one kernel: everything of a step but
// the LJ force.
//
// A block owns whole chains (as many as fit 256 threads, at least one), a
// thread per site, so no bond, angle or dihedral crosses blocks and the
// positions can be updated in place: every position a block reads is its own,
// and it writes them after a barrier.  The bond vectors and the terms' forces
// pass between threads through shared memory as in k_bonded (k_force.cu),
// with the same term functions, so the force has the same bits.
//
// Bound: DRAM traffic of the state at large sizes (243 B per atom mixed: x and v
// read and written, the LJ force read and the other buffer cleared, the rebin
// reference, the sorted positions written), latency below.  As two kernels the force went through memory
// in between (96 B per atom written and read) and the positions were read
// twice; the clearing of the LJ force was a memset of its own.
#include <algorithm>
#include <type_traits>

#include "bonded.cuh"
#include "integrate.cuh"

namespace mdg {

// The update of atom i once its force F is known, and the stores of it
template <bool MIXED, int MODE, bool KE, int TH, class T>
__device__ __forceinline__ void update_atom(const T (&F)[3], T (&xi)[3], T (&vi)[3], int i, int N, int type, int cc,
                                            float4 r0, int slot, T* x, T* v, int* img, float4* pos,
                                            long long* flj_next, int Npad, const RepDev& R, int rep,
                                            const ForceParams& fp, const double* lam, unsigned* flags,
                                            const StepGate& gate, const MoveReport& mr, AtomOut& o) {
  integrate_atom<MIXED, MODE, KE, TH>(F, xi, vi, img, i, N, type, cc, r0, R, rep, fp, lam, o);
#pragma unroll
  for (int a = 0; a < 3; ++a) v[a * N + i] = vi[a];
  if (MODE != kKickOnly) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      x[a * N + i] = xi[a];
      flj_next[(size_t)a * Npad + i] = 0ll;   // the buffer the next step's LJ adds to
    }
    if (o.moved) report_move(mr, gate.j, flags);
    if (o.bad) atomicOr(flags, kFlagNaN);
    pos[slot] = make_float4(o.loc[0], o.loc[1], o.loc[2], (float)type);   // w: LJ type, as the sort writes it
  }
}

// A launch that is off passes its wait and leaves (the gate is read together with the tile)
template <int MODE>
__device__ __forceinline__ bool step_off(const StepGate& gate, const Tile& t) {
  const bool off = MODE == kKickOnly ? !lj_runs(gate) : !drift_runs(gate);
  asm volatile("" ::"r"(t.start));
  if (off) wait_for_predecessor();
  return off;
}

template <bool MIXED, int MODE, bool KE, int TH, int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 4 : NT == 512 ? 2 : 1)
    k_step(void* __restrict__ xv, void* __restrict__ vv, int* __restrict__ img, void* __restrict__ Fv,
           const uint16_t* __restrict__ site, const int* __restrict__ cellc, const int* __restrict__ inv_perm,
           const float4* __restrict__ ref, float4* __restrict__ pos, const long long* __restrict__ flj,
           long long* __restrict__ flj_next, int Npad, int N, const Tile* __restrict__ tiles,
           const RepDev* __restrict__ reps, const ForceParams fp, double* __restrict__ kepart,
           const double* __restrict__ lam, unsigned* __restrict__ flags, const StepGate gate, const MoveReport mr) {
  using T = typename std::conditional<MIXED, double, float>::type;
  T* x = reinterpret_cast<T*>(xv);
  T* v = reinterpret_cast<T*>(vv);
  // bond vectors, the terms' forces (three places of zeros before the first
  // site) and r^2 - b0^2 of the bonds, in arrays of the block's size
  extern __shared__ float step_smem[];
  const int W3 = blockDim.x + 3;
  f3* bv = reinterpret_cast<f3*>(step_smem);
  f3 *fbd = bv + W3, *fan_a = fbd + W3, *fan_c = fan_a + W3, *fdi1 = fan_c + W3, *fdi2 = fdi1 + W3, *fdi3 = fdi2 + W3;
  float* bD = reinterpret_cast<float*>(fdi3 + W3);
  const Tile t = tiles[blockIdx.x];
  const RepDev& R = reps[t.rep];
  const int tid = threadIdx.x, i = t.start + tid, S = fp.sites;
  const bool on = tid < t.len;
  if (step_off<MODE>(gate, t)) return;
  int sm = 0, slot = 0;
  T xi[3];
  if (on) {
    sm = site[i];
    slot = inv_perm[i];
#pragma unroll
    for (int a = 0; a < 3; ++a) xi[a] = x[a * N + i];
    // bond vector to the next site of the chain
    f3 b = mk(0.f, 0.f, 0.f);
    float D = 0.f;
    if (sm < S - 1) {
      const T xn[3] = {x[i + 1], x[N + i + 1], x[2 * N + i + 1]};
      bond_vector<MIXED>(xi, xn, R, fp, b, D);
    }
    bv[tid] = b;
    bD[tid] = D;
  }
  if (tid < 3) fbd[tid] = fan_a[tid] = fan_c[tid] = fdi1[tid] = fdi2[tid] = fdi3[tid] = mk(0.f, 0.f, 0.f);
  __syncthreads();
  {
    const f3 z = mk(0.f, 0.f, 0.f);
    f3 fb = z, fa = z, fc = z, f1 = z, f2 = z, f3v = z;
    float Eb = 0.f, Ea = 0.f, Ed = 0.f, W[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (on) chain_terms<false>(fp, sm, S, bv, bD, tid, false, fb, fa, fc, f1, f2, f3v, Eb, Ea, Ed, W);
    fbd[tid + 3] = fb; fan_a[tid + 3] = fa; fan_c[tid + 3] = fc;
    fdi1[tid + 3] = f1; fdi2[tid + 3] = f2; fdi3[tid + 3] = f3v;
  }
  // all before this line reads what the update before the LJ launch left: it
  // runs while the last LJ blocks finish
  wait_for_predecessor();
  __syncthreads();
  AtomOut o;
  o.ke = 0.0;
  o.mom[0] = o.mom[1] = o.mom[2] = 0.0;
  if (on) {
    // loaded here, and 64 registers: held across the terms these values and
    // the registers they cost leave five blocks an SM instead of six (1.5M
    // mixed: 114 us with 78 registers, 97 held in 64, 91 loaded here)
    T vi[3];
    long long l[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) { l[a] = __ldg(flj + (size_t)a * Npad + slot); vi[a] = v[a * N + i]; }
    int cc = 0;
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MODE != kKickOnly) { cc = cellc[i]; r0 = ref[i]; }
    const f3 fb = chain_force(fbd, fan_a, fan_c, fdi1, fdi2, fdi3, tid + 3);
    T F[3];
    if constexpr (MIXED) {
      F4i f;
      f.x = l[0] + to_fix(fb.x, flags);
      f.y = l[1] + to_fix(fb.y, flags);
      f.z = l[2] + to_fix(fb.z, flags);
      f.w = 0;
      if (MODE == kKickOnly) reinterpret_cast<F4i*>(Fv)[i] = f;   // the force at the call's end
      F[0] = fix_to_double_i(f.x); F[1] = fix_to_double_i(f.y); F[2] = fix_to_double_i(f.z);
    } else {
      const float4 f = make_float4(fix_to_float(l[0]) + fb.x, fix_to_float(l[1]) + fb.y, fix_to_float(l[2]) + fb.z, 0.f);
      if (MODE == kKickOnly) reinterpret_cast<float4*>(Fv)[i] = f;
      F[0] = f.x; F[1] = f.y; F[2] = f.z;
    }
    const int type = (sm == 0 || sm == S - 1) ? 1 : 0;
    update_atom<MIXED, MODE, KE, TH>(F, xi, vi, i, N, type, cc, r0, slot, x, v, img, pos, flj_next, Npad, R, t.rep, fp,
                                     lam, flags, gate, mr, o);
  }
  if constexpr (KE) tile_kinetic<TH, NT>(o, blockIdx.x, kepart);
}

// The same step for general molecules (mixed form): a block owns whole
// molecules, a thread evaluates every blockDim-th term of their bond graph and
// adds its forces in shared memory, then every thread updates its atom.  A
// force is an int64 fixed-point sum kept as two words: a 32-bit shared atomic
// on each, the carry out of the low word added to the high one, so the sum is
// the same in any order and wraps like an int64.
//
// Bound: the latency of a term's chain of FP64 differences and divisions (35k
// atoms in 12-atom molecules: 43 terms a molecule).  So the terms are dealt out
// one per thread from one table (per atom, as they are listed, an atom had
// between none and 9) and blocks are of 128 threads (35k atoms are 292 of them on 152
// SMs).  As three kernels (LJ force into F, terms with global int64 atomics,
// integrator) a step took 62 us with the LJ force, now 39 (10 steps: 621 -> 389 us).
__device__ __forceinline__ void sum_add(unsigned* lo, unsigned* hi, long long f) {
  const unsigned l = (unsigned)f;
  unsigned h = (unsigned)((unsigned long long)f >> 32);
  const unsigned old = atomicAdd(lo, l);
  h += old + l < old ? 1u : 0u;
  if (h) atomicAdd(hi, h);
}

template <int MODE, bool KE, int TH, int NT>
__global__ void __launch_bounds__(NT) k_step_molecules(double* __restrict__ x, double* __restrict__ v,
                                                       int* __restrict__ img, F4i* __restrict__ F_out,
                                                       const uint16_t* __restrict__ site,
                                                       const int* __restrict__ cellc, const int* __restrict__ inv_perm,
                                                       const float4* __restrict__ ref, float4* __restrict__ pos,
                                                       const long long* __restrict__ flj,
                                                       long long* __restrict__ flj_next, int Npad, int N,
                                                       const Tile* __restrict__ tiles, const RepDev* __restrict__ reps,
                                                       const ForceParams fp, const TopoDev tp,
                                                       double* __restrict__ kepart, const double* __restrict__ lam,
                                                       unsigned* __restrict__ flags, const StepGate gate,
                                                       const MoveReport mr) {
  extern __shared__ __align__(16) double mol_smem[];
  const int W = blockDim.x;
  double* xs = mol_smem;                                       // 3 rows of positions
  unsigned* lo = reinterpret_cast<unsigned*>(xs + 3 * W);      // 3 rows of force sums, low and high words
  unsigned* hi = lo + 3 * W;
  const Tile t = tiles[blockIdx.x];
  const RepDev& R = reps[t.rep];
  const int tid = threadIdx.x, i = t.start + tid;
  const bool on = tid < t.len;
  if (step_off<MODE>(gate, t)) return;
  int type = 0, slot = 0;
  if (on) {
    type = atom_type(site[i], fp);
    slot = inv_perm[i];
#pragma unroll
    for (int a = 0; a < 3; ++a) xs[a * W + tid] = x[a * N + i];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) lo[a * W + tid] = hi[a * W + tid] = 0u;
  __syncthreads();
  {
    const auto add = [&](int k, f3 f) {
      sum_add(lo + k, hi + k, to_fix(f.x, flags));
      sum_add(lo + W + k, hi + W + k, to_fix(f.y, flags));
      sum_add(lo + 2 * W + k, hi + 2 * W + k, to_fix(f.z, flags));
    };
    float E = 0.f, Wv[6];   // not summed in the steps
    const int mols = t.len / tp.naom, nb = mols * tp.n_bonds, na = mols * tp.n_angles, nd = mols * tp.n_dihedrals;
    for (int q = tid; q < nb + na + nd; q += W) {
      if (q < nb) {
        const int m = q / tp.n_bonds, o = m * tp.naom;
        const ushort4 e = tp.terms[q - m * tp.n_bonds];
        bond_term<false>(xs, W, o + e.x, o + e.y, R, fp, add, E, Wv);
      } else if (q < nb + na) {
        const int m = (q - nb) / tp.n_angles, o = m * tp.naom;
        const ushort4 e = tp.terms[tp.n_bonds + q - nb - m * tp.n_angles];
        angle_term<false>(xs, W, o + e.x, o + e.y, o + e.z, R, fp, add, E, Wv);
      } else {
        const int m = (q - nb - na) / tp.n_dihedrals, o = m * tp.naom;
        const ushort4 e = tp.terms[tp.n_bonds + tp.n_angles + q - nb - na - m * tp.n_dihedrals];
        dihedral_term<false>(xs, W, o + e.x, o + e.y, o + e.z, o + e.w, R, fp, add, E, Wv);
      }
    }
  }
  // all before this line reads what the update before the LJ launch left (k_step)
  wait_for_predecessor();
  __syncthreads();
  AtomOut o;
  o.ke = 0.0;
  o.mom[0] = o.mom[1] = o.mom[2] = 0.0;
  if (on) {
    double vi[3], xi[3], F[3];
    long long f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      f[a] = __ldg(flj + (size_t)a * Npad + slot) +
             (long long)(((unsigned long long)hi[a * W + tid] << 32) | lo[a * W + tid]);
      vi[a] = v[a * N + i];
      xi[a] = xs[a * W + tid];
      F[a] = fix_to_double_i(f[a]);
    }
    int cc = 0;
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MODE != kKickOnly) { cc = cellc[i]; r0 = ref[i]; }
    if (MODE == kKickOnly) {   // the force at the call's end
      F4i w;
      w.x = f[0]; w.y = f[1]; w.z = f[2]; w.w = 0;
      F_out[i] = w;
    }
    update_atom<true, MODE, KE, TH>(F, xi, vi, i, N, type, cc, r0, slot, x, v, img, pos, flj_next, Npad, R, t.rep, fp,
                                    lam, flags, gate, mr, o);
  }
  if constexpr (KE) tile_kinetic<TH, NT>(o, blockIdx.x, kepart);
}

static size_t step_smem_bytes(int threads) { return (size_t)(threads + 3) * (7 * sizeof(f3) + sizeof(float)); }

static size_t molecules_smem_bytes(int threads) { return (size_t)threads * (3 * sizeof(double) + 6 * sizeof(unsigned)); }

int step_chains_per_block(int sites, bool generic) { return std::max(1, (generic ? 128 : 256) / sites); }

template <bool MIXED, int NT>
static void launch_step_t(IntegMode mode, int th, int threads, const StepArgs& a, const ForceParams& fp,
                          const StepGate& gate, const MoveReport& mr, cudaStream_t st) {
#define MDG_STEP(MODE, KE, TH)                                                                                       \
  launch_dependent(gate.dep, k_step<MIXED, MODE, KE, TH, NT>, a.n_tiles, threads, step_smem_bytes(threads), st,     \
                   a.x, a.v, a.img, a.F, a.site, a.cellc, a.inv_perm, a.ref, a.pos, a.flj, a.flj_next, a.Npad, a.N, a.tiles, a.reps,  \
                   fp, a.kepart, a.lam, a.flags, gate, mr)
  if (mode == kKickKickDrift) {
    if (th == 2) MDG_STEP(kKickKickDrift, true, 2);
    else if (th == 1) MDG_STEP(kKickKickDrift, true, 1);
    else MDG_STEP(kKickKickDrift, false, 0);
  } else {
    if (th == 2) MDG_STEP(kKickOnly, false, 2);
    else MDG_STEP(kKickOnly, false, 0);
  }
#undef MDG_STEP
}

template <int NT>
static void launch_molecules_t(IntegMode mode, int th, int threads, const StepArgs& a, const ForceParams& fp,
                               const TopoDev& tp, const StepGate& gate, const MoveReport& mr, cudaStream_t st) {
#define MDG_STEP(MODE, KE, TH)                                                                                        \
  launch_dependent(gate.dep, k_step_molecules<MODE, KE, TH, NT>, a.n_tiles, threads, molecules_smem_bytes(threads),   \
                   st, (double*)a.x, (double*)a.v, a.img, (F4i*)a.F, a.site, a.cellc, a.inv_perm, a.ref, a.pos, a.flj, \
                   a.flj_next, a.Npad, a.N, a.tiles, a.reps, fp, tp, a.kepart, a.lam, a.flags, gate, mr)
  if (mode == kKickKickDrift) {
    if (th == 2) MDG_STEP(kKickKickDrift, true, 2);
    else if (th == 1) MDG_STEP(kKickKickDrift, true, 1);
    else MDG_STEP(kKickKickDrift, false, 0);
  } else {
    if (th == 2) MDG_STEP(kKickOnly, false, 2);
    else MDG_STEP(kKickOnly, false, 0);
  }
#undef MDG_STEP
}

// Dynamic shared memory of a form: beside the static array of the kinetic sums
// (tile_kinetic: up to 16 KB for 512 threads, 32 KB for 1,024) it can exceed the
// 48 KB that need no opt-in from 353 sites a chain on, so every form opts in to
// the most that its block size asks for (once per device)
cudaError_t step_kernels_init() {
  cudaError_t e = cudaSuccess;
  auto allow = [&](const void* kernel, size_t bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
#define MDG_STEP_ATTR(MIXED, MODE, KE, TH)                                     \
  allow((const void*)k_step<MIXED, MODE, KE, TH, 256>, step_smem_bytes(256));  \
  allow((const void*)k_step<MIXED, MODE, KE, TH, 512>, step_smem_bytes(512));  \
  allow((const void*)k_step<MIXED, MODE, KE, TH, 1024>, step_smem_bytes(1024))
#define MDG_STEP_ATTRS(MIXED)                     \
  MDG_STEP_ATTR(MIXED, kKickKickDrift, true, 2);  \
  MDG_STEP_ATTR(MIXED, kKickKickDrift, true, 1);  \
  MDG_STEP_ATTR(MIXED, kKickKickDrift, false, 0); \
  MDG_STEP_ATTR(MIXED, kKickOnly, false, 2);      \
  MDG_STEP_ATTR(MIXED, kKickOnly, false, 0)
  MDG_STEP_ATTRS(true);
  MDG_STEP_ATTRS(false);
#undef MDG_STEP_ATTRS
#undef MDG_STEP_ATTR
#define MDG_STEP_ATTR(MODE, KE, TH)                                                            \
  allow((const void*)k_step_molecules<MODE, KE, TH, 128>, molecules_smem_bytes(128));          \
  allow((const void*)k_step_molecules<MODE, KE, TH, 1024>, molecules_smem_bytes(1024))
  MDG_STEP_ATTR(kKickKickDrift, true, 2);
  MDG_STEP_ATTR(kKickKickDrift, true, 1);
  MDG_STEP_ATTR(kKickKickDrift, false, 0);
  MDG_STEP_ATTR(kKickOnly, false, 2);
  MDG_STEP_ATTR(kKickOnly, false, 0);
#undef MDG_STEP_ATTR
  return e;
}

void launch_step(bool mixed, IntegMode mode, int th, int sites, const StepArgs& a, const ForceParams& fp,
                 const TopoDev* topo, const StepGate& gate, const MoveReport& mr, cudaStream_t st) {
  if (a.n_tiles <= 0) return;
  const int threads = (step_chains_per_block(sites, topo != nullptr) * sites + 31) / 32 * 32;
  if (topo) {
    if (threads <= 128) launch_molecules_t<128>(mode, th, threads, a, fp, *topo, gate, mr, st);
    else launch_molecules_t<1024>(mode, th, threads, a, fp, *topo, gate, mr, st);
  } else if (threads <= 256) {
    if (mixed) launch_step_t<true, 256>(mode, th, threads, a, fp, gate, mr, st);
    else launch_step_t<false, 256>(mode, th, threads, a, fp, gate, mr, st);
  } else if (threads <= 512) {
    if (mixed) launch_step_t<true, 512>(mode, th, threads, a, fp, gate, mr, st);
    else launch_step_t<false, 512>(mode, th, threads, a, fp, gate, mr, st);
  } else {
    if (mixed) launch_step_t<true, 1024>(mode, th, threads, a, fp, gate, mr, st);
    else launch_step_t<false, 1024>(mode, th, threads, a, fp, gate, mr, st);
  }
}

}  // namespace mdg
