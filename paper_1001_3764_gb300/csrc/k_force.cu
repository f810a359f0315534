// k_force.cu -- Dreiding II bonded forces (Eqs. 4-6, Sec. 3.3) on sm_103a for
// the read-outs: the total force at the present positions, and the bonded
// energies and virial.  The steps' form is in k_step.cu, the terms in bonded.cuh.
// The Lennard-Jones force (Eq. 2) is in k_lj.cu.
//
// Each thread block owns a contiguous range of atoms (whole or partial
// chains) plus a 3-atom halo.  Bond vectors are formed once per bond (FP64
// differences of the master positions in the mixed form, exact FP32
// differences in the plain form), every bond/angle/dihedral term is evaluated
// once by the thread of its first atom, and each home atom then sums the
// contributions of the (at most 2+3+4) terms that contain it in a fixed
// order.  This removes the paper's 2x/3x/4x redundant per-home-atom flops
// (Sec. 3.3) without atomics.  The kernel also adds the LJ force of the atom
// (read from cell-sorted order through inv_perm).  Energies and the virial are block sums: FP32 warp trees,
// then FP64 across warps, in a fixed order.
#include <type_traits>

#include "bonded.cuh"

namespace mdg {

// Block reduction of NV FP32 per-thread values into out[NV] (FP64; thread 0
// holds the result): each warp adds its 32 lanes in FP32 by a fixed shuffle
// tree (an FP64 tree per lane would load this GPU's narrow FP64 pipe), lane 0
// converts the warp sum to FP64 and the warps are added in FP64 in order.
// Fixed shape, so the summation order is the same on every run.
template <int NV, int NT>
__device__ __forceinline__ void block_sum(const float (&v)[NV], double* out) {
  __shared__ double red[NV][NT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    float s = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) red[k][w] = (double)s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double s = 0.0;
      for (int q = 0; q < NT / 32; ++q) s += red[k][q];
      out[k] = s;
    }
  }
}

// ======================================================================= bonded
constexpr int kBondedBlock = 256;
constexpr int kHalo = 3;
constexpr int kBondedVals = 9;   // bond, angle, dihedral, vxx, vyy, vzz, vxy, vxz, vyz

template <bool MIXED, bool ENERGY>
__global__ void __launch_bounds__(kBondedBlock) k_bonded(const void* __restrict__ xv, const uint16_t* __restrict__ site,
                                                         const int* __restrict__ inv_perm, const long long* __restrict__ flj,
                                                         int Npad, int N, const Tile* __restrict__ tiles,
                                                         const RepDev* __restrict__ reps, const ForceParams fp,
                                                         void* __restrict__ Fout, double* __restrict__ epart,
                                                         unsigned* __restrict__ flags) {
  using T = typename std::conditional<MIXED, double, float>::type;
  const T* x = reinterpret_cast<const T*>(xv);
  __shared__ f3 bv[kBondedBlock + 2 * kHalo];
  __shared__ float bD[kBondedBlock + 2 * kHalo];   // r^2 - b0^2 of each bond, free of cancellation
  __shared__ f3 fbd[kBondedBlock], fan_a[kBondedBlock], fan_c[kBondedBlock];
  __shared__ f3 fdi1[kBondedBlock], fdi2[kBondedBlock], fdi3[kBondedBlock];
  const Tile t = tiles[blockIdx.x];
  const RepDev& R = reps[t.rep];
  const int lo = R.atom_off, hi = R.atom_off + R.n_atoms;
  const int S = fp.sites;
  const int base = t.start - kHalo;
  // 1. bond vectors b_m = x_{m+1} - x_m for m in [start-3, start+len+3)
  for (int q = threadIdx.x; q < t.len + 2 * kHalo; q += blockDim.x) {
    const int m = base + q;
    f3 b = mk(0.f, 0.f, 0.f);
    float D = 0.f;
    if (m >= lo && m + 1 < hi && site[m] < S - 1) {
      const T xa[3] = {x[m], x[N + m], x[2 * N + m]}, xb[3] = {x[m + 1], x[N + m + 1], x[2 * N + m + 1]};
      bond_vector<MIXED>(xa, xb, R, fp, b, D);
    }
    bv[q] = b;
    bD[q] = D;
  }
  __syncthreads();
  // 2. terms starting at atom m = base + q
  float Eb = 0.f, Ea = 0.f, Ed = 0.f;
  float W[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  {
    const int q = threadIdx.x;
    const int m = base + q;
    f3 z = mk(0.f, 0.f, 0.f);
    f3 fb = z, fa = z, fc = z, f1 = z, f2 = z, f3v = z;
    if (q < t.len + kHalo && m >= lo && m < hi) {
      const int sm = site[m];
      const bool own = m >= t.start;   // energy/virial counted once, by the owning tile
      chain_terms<ENERGY>(fp, sm, S, bv, bD, q, own, fb, fa, fc, f1, f2, f3v, Eb, Ea, Ed, W);
    }
    if (q < kBondedBlock) {
      fbd[q] = fb; fan_a[q] = fa; fan_c[q] = fc; fdi1[q] = f1; fdi2[q] = f2; fdi3[q] = f3v;
    }
  }
  __syncthreads();
  // 3. sum the contributions on each home atom in a fixed order.  An energy
  // read-out passes no Fout; in the mixed form it still converts the forces, so
  // that one beyond the fixed-point range, or not a number, is reported.
  if ((MIXED || Fout) && (int)threadIdx.x < t.len) {
    const int q = threadIdx.x + kHalo;
    const int i = t.start + threadIdx.x;
    const f3 F = chain_force(fbd, fan_a, fan_c, fdi1, fdi2, fdi3, q);
    F4i o;
    if (MIXED) {
      o.x = to_fix(F.x, flags);
      o.y = to_fix(F.y, flags);
      o.z = to_fix(F.z, flags);
      o.w = 0;
    }
    if (Fout) {
      // the LJ force of the atom (sorted slot s)
      const int s = inv_perm[i];
      const long long lx = __ldg(flj + s), ly = __ldg(flj + Npad + s), lz = __ldg(flj + 2 * (size_t)Npad + s);
      if (MIXED) {
        o.x += lx;
        o.y += ly;
        o.z += lz;
        reinterpret_cast<F4i*>(Fout)[i] = o;
      } else {
        reinterpret_cast<float4*>(Fout)[i] =
            make_float4(fix_to_float(lx) + F.x, fix_to_float(ly) + F.y, fix_to_float(lz) + F.z, 0.f);
      }
    }
  }
  if (ENERGY) {
    const float v[kBondedVals] = {Eb, Ea, Ed, W[0], W[1], W[2], W[3], W[4], W[5]};
    block_sum<kBondedVals, kBondedBlock>(v, epart + (size_t)blockIdx.x * kBondedVals);
  }
}

// ======================================================================= bonded, general molecules
// A general molecule type (Sec. 3.3, t_bonds / t_angles / dihedral lists) in
// the read-outs (forces at the present positions, energies; the steps' form is
// in k_step.cu): one thread per atom of an integrator tile evaluates the terms
// listed under that atom (each term once, under its first atom) and adds their
// forces to every atom of the term with int64 atomics (integer sums:
// order-free, so deterministic).  k_bonded_init first writes the LJ force of
// every atom into F.

__device__ __forceinline__ void fix_add(F4i* F, int i, f3 f, unsigned* flags) {
  atomicAdd(reinterpret_cast<unsigned long long*>(&F[i].x), (unsigned long long)to_fix(f.x, flags));
  atomicAdd(reinterpret_cast<unsigned long long*>(&F[i].y), (unsigned long long)to_fix(f.y, flags));
  atomicAdd(reinterpret_cast<unsigned long long*>(&F[i].z), (unsigned long long)to_fix(f.z, flags));
}

__global__ void __launch_bounds__(256) k_bonded_init(const int* __restrict__ inv_perm, const long long* __restrict__ flj,
                                                     int Npad, int N, F4i* __restrict__ F) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int s = inv_perm[i];
  F4i o;
  o.x = __ldg(flj + s); o.y = __ldg(flj + Npad + s); o.z = __ldg(flj + 2 * (size_t)Npad + s); o.w = 0;
  F[i] = o;
}

template <bool ENERGY>
__global__ void __launch_bounds__(kBondedBlock) k_bonded_generic(const double* __restrict__ x, int N,
                                                                 const Tile* __restrict__ tiles,
                                                                 const RepDev* __restrict__ reps, const ForceParams fp,
                                                                 const TopoDev tp, F4i* __restrict__ F,
                                                                 double* __restrict__ epart,
                                                                 unsigned* __restrict__ flags) {
  const Tile t = tiles[blockIdx.x];
  const RepDev& R = reps[t.rep];
  float Eb = 0.f, Ea = 0.f, Ed = 0.f;
  float W[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if ((int)threadIdx.x < t.len) {
    const int i = t.start + threadIdx.x;
    const int a = (i - R.atom_off) % tp.naom, m0 = i - a;
    const auto add = [&](int k, f3 f) { fix_add(F, k, f, flags); };
    for (int q = tp.b_off[a]; q < tp.b_off[a + 1]; ++q)
      bond_term<ENERGY>(x, N, i, m0 + tp.b_at[q], R, fp, add, Eb, W);
    for (int q = tp.a_off[a]; q < tp.a_off[a + 1]; ++q)
      angle_term<ENERGY>(x, N, i, m0 + tp.a_at[2 * q], m0 + tp.a_at[2 * q + 1], R, fp, add, Ea, W);
    for (int q = tp.d_off[a]; q < tp.d_off[a + 1]; ++q)
      dihedral_term<ENERGY>(x, N, i, m0 + tp.d_at[3 * q], m0 + tp.d_at[3 * q + 1], m0 + tp.d_at[3 * q + 2], R, fp, add,
                            Ed, W);
  }
  if (ENERGY) {
    const float v[kBondedVals] = {Eb, Ea, Ed, W[0], W[1], W[2], W[3], W[4], W[5]};
    block_sum<kBondedVals, kBondedBlock>(v, epart + (size_t)blockIdx.x * kBondedVals);
  }
}

void launch_bonded_generic(bool energy, const double* x, const int* inv_perm, const long long* flj, int Npad, int N,
                           const Tile* tiles, int n_tiles, const RepDev* reps, const ForceParams& fp,
                           const TopoDev& topo, void* F, double* epart, unsigned* flags, cudaStream_t st) {
  if (N <= 0) return;
  k_bonded_init<<<(N + 255) / 256, 256, 0, st>>>(inv_perm, flj, Npad, N, reinterpret_cast<F4i*>(F));
  if (energy)
    k_bonded_generic<true><<<n_tiles, kBondedBlock, 0, st>>>(x, N, tiles, reps, fp, topo, reinterpret_cast<F4i*>(F),
                                                             epart, flags);
  else
    k_bonded_generic<false><<<n_tiles, kBondedBlock, 0, st>>>(x, N, tiles, reps, fp, topo, reinterpret_cast<F4i*>(F),
                                                              epart, flags);
}

void launch_bonded(bool mixed, bool energy, const void* x, const uint16_t* site, const int* inv_perm,
                   const long long* flj, int Npad, int N, const Tile* tiles, int n_tiles, const RepDev* reps,
                   const ForceParams& fp, void* F, double* epart, unsigned* flags, cudaStream_t st) {
#define MDG_BONDED(M, E) \
  k_bonded<M, E><<<n_tiles, kBondedBlock, 0, st>>>(x, site, inv_perm, flj, Npad, N, tiles, reps, fp, F, epart, flags)
  if (mixed) {
    if (energy) MDG_BONDED(true, true); else MDG_BONDED(true, false);
  } else {
    if (energy) MDG_BONDED(false, true); else MDG_BONDED(false, false);
  }
#undef MDG_BONDED
}

}  // namespace mdg
