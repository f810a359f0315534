// md_adjoint.cu -- gradients of trajectory means with respect to the
// force-field parameters, by a hand-written adjoint of the FP64
// velocity-Verlet run.
//
// The run is the NVE integrator of the hot path (Sec. 3 / 3.4) in FP64 on the
// GPU: x_{k+1} = x_k + dt v_{k+1/2}, v_{k+1/2} = v_{k-1/2} + dt a(x_k), with
// half kicks at both ends.  Observables J = 1/(K+1) sum_k O(x_k) with
// O = w0 U + w1 R_ee^2; U = shifted LJ (Eq. 2) + bond (Eq. 4) + angle (Eq. 5)
// + dihedral (Eq. 6), R_ee^2 the mean over chains of the squared end-to-end
// distance (the end-to-end vector of Sec. 4, Fig. 8) from unwrapped positions.
//
// Reverse pass (adjoint of the leapfrog form, newest step first), with
// alpha = dJ/dx_k and beta = dJ/dv_{k+1/2}, c_k = dt (dt/2 at k = 0, 0 at K):
//   u      = c_k M^-1 beta
//   alpha  = w_k grad O(x_k) + alpha - H(x_k) u
//   g     += w_k w0 dU/dtheta(x_k) - d/dtheta [grad U(x_k) . u]
//   beta  += dt alpha                                  (k >= 1)
// H u and d/dtheta[grad U . u] come from one forward-mode (dual-number)
// evaluation of the gradient formulas along u.  U is linear in the pair
// coefficients c12_t = 4 eps_t sigma_t^12, c6_t = 4 eps_t sigma_t^6 of the
// three pair types t and in k_phi, so the parameter derivatives are sums of
// per-pair (per-term) scalars, mapped to (eps, sigma) of the two site types
// through the geometric-mean mixing rule on the host.
//
// Positions are recomputed from (x, v) checkpoints every C steps; a segment
// store holds the C + 1 positions of the segment being reversed.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <new>
#include <type_traits>

#include "../../include/md.h"
#include "cell_order.cuh"

void md_set_global_error(const char* msg);   // md_api.cu: message for md_last_error(NULL)

namespace mdg {
namespace adj {

// ------------------------------------------------------------------ dual numbers
// value and derivative along one direction of configuration space
struct Dual {
  double v, t;
};
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return {a.v + b.v, a.t + b.t}; }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return {a.v - b.v, a.t - b.t}; }
__device__ __forceinline__ Dual operator-(Dual a) { return {-a.v, -a.t}; }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) { return {a.v * b.v, a.v * b.t + a.t * b.v}; }
__device__ __forceinline__ Dual operator*(double s, Dual a) { return {s * a.v, s * a.t}; }
__device__ __forceinline__ Dual operator*(Dual a, double s) { return {s * a.v, s * a.t}; }
__device__ __forceinline__ Dual operator+(Dual a, double s) { return {a.v + s, a.t}; }
__device__ __forceinline__ Dual operator+(double s, Dual a) { return {a.v + s, a.t}; }
__device__ __forceinline__ Dual operator-(Dual a, double s) { return {a.v - s, a.t}; }
__device__ __forceinline__ Dual operator-(double s, Dual a) { return {s - a.v, -a.t}; }
__device__ __forceinline__ Dual operator/(Dual a, Dual b) {
  const double q = a.v / b.v;
  return {q, (a.t - q * b.t) / b.v};
}
__device__ __forceinline__ Dual operator/(double s, Dual b) {
  const double q = s / b.v;
  return {q, -q * b.t / b.v};
}
__device__ __forceinline__ Dual& operator+=(Dual& a, Dual b) { a = a + b; return a; }

__device__ __forceinline__ double gsqrt(double a) { return sqrt(a); }
__device__ __forceinline__ Dual gsqrt(Dual a) {
  const double r = sqrt(a.v);
  return {r, 0.5 * a.t / r};
}
__device__ __forceinline__ double gatan2(double y, double x) { return atan2(y, x); }
__device__ __forceinline__ Dual gatan2(Dual y, Dual x) {
  return {atan2(y.v, x.v), (x.v * y.t - y.v * x.t) / (x.v * x.v + y.v * y.v)};
}
__device__ __forceinline__ double gcos(double a) { return cos(a); }
__device__ __forceinline__ double gsin(double a) { return sin(a); }
__device__ __forceinline__ Dual gcos(Dual a) {
  double s, c;
  sincos(a.v, &s, &c);
  return {c, -s * a.t};
}
__device__ __forceinline__ Dual gsin(Dual a) {
  double s, c;
  sincos(a.v, &s, &c);
  return {s, c * a.t};
}
__device__ __forceinline__ double value(double a) { return a; }
__device__ __forceinline__ double value(Dual a) { return a.v; }
__device__ __forceinline__ double tangent(double) { return 0.0; }
__device__ __forceinline__ double tangent(Dual a) { return a.t; }

// FP32 dual numbers for the reverse pass's Hessian-vector products (the
// optional FP32 HVP): separations still come from FP64 positions and the pair
// set from an FP64 cutoff test; only the term arithmetic runs in FP32, and its
// per-atom results are added into the FP64 records.  FP64 constants are
// rounded to FP32 where they meet an FP32 dual.
struct DualF {
  float v, t;
};
__device__ __forceinline__ DualF operator+(DualF a, DualF b) { return {a.v + b.v, a.t + b.t}; }
__device__ __forceinline__ DualF operator-(DualF a, DualF b) { return {a.v - b.v, a.t - b.t}; }
__device__ __forceinline__ DualF operator-(DualF a) { return {-a.v, -a.t}; }
__device__ __forceinline__ DualF operator*(DualF a, DualF b) { return {a.v * b.v, a.v * b.t + a.t * b.v}; }
__device__ __forceinline__ DualF operator*(double s, DualF a) { const float f = (float)s; return {f * a.v, f * a.t}; }
__device__ __forceinline__ DualF operator*(DualF a, double s) { const float f = (float)s; return {f * a.v, f * a.t}; }
__device__ __forceinline__ DualF operator+(DualF a, double s) { return {a.v + (float)s, a.t}; }
__device__ __forceinline__ DualF operator+(double s, DualF a) { return {a.v + (float)s, a.t}; }
__device__ __forceinline__ DualF operator-(DualF a, double s) { return {a.v - (float)s, a.t}; }
__device__ __forceinline__ DualF operator-(double s, DualF a) { return {(float)s - a.v, -a.t}; }
__device__ __forceinline__ DualF operator/(DualF a, DualF b) {
  const float q = a.v / b.v;
  return {q, (a.t - q * b.t) / b.v};
}
__device__ __forceinline__ DualF operator/(double s, DualF b) {
  const float q = (float)s / b.v;
  return {q, -q * b.t / b.v};
}
__device__ __forceinline__ DualF& operator+=(DualF& a, DualF b) { a = a + b; return a; }
__device__ __forceinline__ DualF gsqrt(DualF a) {
  const float r = sqrtf(a.v);
  return {r, 0.5f * a.t / r};
}
__device__ __forceinline__ DualF gatan2(DualF y, DualF x) {
  return {atan2f(y.v, x.v), (x.v * y.t - y.v * x.t) / (x.v * x.v + y.v * y.v)};
}
__device__ __forceinline__ DualF gcos(DualF a) {
  float s, c;
  sincosf(a.v, &s, &c);
  return {c, -s * a.t};
}
__device__ __forceinline__ DualF gsin(DualF a) {
  float s, c;
  sincosf(a.v, &s, &c);
  return {s, c * a.t};
}
__device__ __forceinline__ double value(DualF a) { return (double)a.v; }
__device__ __forceinline__ double tangent(DualF a) { return (double)a.t; }

template <class T>
struct V3 {
  T x, y, z;
};
template <class T>
__device__ __forceinline__ V3<T> operator+(V3<T> a, V3<T> b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
template <class T>
__device__ __forceinline__ V3<T> operator-(V3<T> a, V3<T> b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
template <class T, class S>
__device__ __forceinline__ V3<T> scale(S s, V3<T> a) { return {s * a.x, s * a.y, s * a.z}; }
template <class T>
__device__ __forceinline__ T dot(V3<T> a, V3<T> b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
template <class T>
__device__ __forceinline__ V3<T> cross(V3<T> a, V3<T> b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// ------------------------------------------------------------------ parameters
struct AdjDev {
  double L, inv_L, inv_h;     // box, 1/L, cells per nm
  int M, n_off;               // cells per side (1 when L < 3 r_c), neighbour cells visited (27 or 1)
  int sites, n_chains, N;
  double rc, rc2, irc6, irc12;   // cutoff and the shift terms (1/r_c)^6, (1/r_c)^12
  double irc7, irc13;            // force-shifted variant: (1/r_c)^7, (1/r_c)^13
  int sf;                        // 1 = force-shifted variant (not the paper's potential)
  float pre2;                    // FP32 prefilter: (r_c + margin)^2; a candidate beyond it is out in FP64 too
  double c6[3], c12[3];       // pair types 0 = C32-C32, 1 = C32-C33, 2 = C33-C33
  double kb, b0, ka, theta0, kphi, phis;
  int n_mult;
  double inv_mass[2];
};

__device__ __forceinline__ int site_type(int site, int sites) { return (site == 0 || site == sites - 1) ? 1 : 0; }

__device__ __forceinline__ double min_image(double d, const AdjDev& P) { return d - P.L * rint(d * P.inv_L); }

// separation x_b - x_a (minimum image, FP64 value) with the tangent
// u_b - u_a, u_k = cu * beta_k / m_k the direction of atom k, in the scalar
// type T of the evaluation
template <class T>
__device__ __forceinline__ V3<T> make_sep(double dx, double dy, double dz, const double* beta, double cu, int a,
                                          int b, const AdjDev& P);
template <>
__device__ __forceinline__ V3<double> make_sep<double>(double dx, double dy, double dz, const double*, double, int,
                                                       int, const AdjDev&) {
  return {dx, dy, dz};
}
template <>
__device__ __forceinline__ V3<Dual> make_sep<Dual>(double dx, double dy, double dz, const double* beta, double cu,
                                                   int a, int b, const AdjDev& P) {
  const double sa = cu * P.inv_mass[site_type(a % P.sites, P.sites)];
  const double sb = cu * P.inv_mass[site_type(b % P.sites, P.sites)];
  return {{dx, sb * beta[3 * b] - sa * beta[3 * a]}, {dy, sb * beta[3 * b + 1] - sa * beta[3 * a + 1]},
          {dz, sb * beta[3 * b + 2] - sa * beta[3 * a + 2]}};
}
template <>
__device__ __forceinline__ V3<DualF> make_sep<DualF>(double dx, double dy, double dz, const double* beta, double cu,
                                                     int a, int b, const AdjDev& P) {
  const double sa = cu * P.inv_mass[site_type(a % P.sites, P.sites)];
  const double sb = cu * P.inv_mass[site_type(b % P.sites, P.sites)];
  return {{(float)dx, (float)(sb * beta[3 * b] - sa * beta[3 * a])},
          {(float)dy, (float)(sb * beta[3 * b + 1] - sa * beta[3 * a + 1])},
          {(float)dz, (float)(sb * beta[3 * b + 2] - sa * beta[3 * a + 2])}};
}
template <class T>
__device__ __forceinline__ V3<T> sep(const double* x, const double* beta, double cu, int a, int b, const AdjDev& P) {
  return make_sep<T>(min_image(x[3 * b] - x[3 * a], P), min_image(x[3 * b + 1] - x[3 * a + 1], P),
                     min_image(x[3 * b + 2] - x[3 * a + 2], P), beta, cu, a, b, P);
}

__device__ __forceinline__ int cell_coord(double xv, const AdjDev& P) {
  const double s = xv - P.L * floor(xv * P.inv_L);
  int c = (int)floor(s * P.inv_h);
  return c < 0 ? 0 : (c > P.M - 1 ? P.M - 1 : c);
}

// ------------------------------------------------------------------ per-atom record
// fields of rec[kRec * i + f]
constexpr int kRec = 20;
constexpr int kA = 0;        // 4 per pair type t: A.v, A.t, B.v, B.t with A = sum (1/r^12 - 1/rc^12), B = sum (1/r^6 - 1/rc^6)
constexpr int kD = 12;       // D.v, D.t with D = sum (1 + cos(n phi - phi_s))
constexpr int kElj = 14;     // shifted LJ energy (half per pair)
constexpr int kEb = 15, kEa = 16, kEd = 17;
constexpr int kR2 = 18;      // |x_last - x_first|^2 on each chain's first atom
constexpr int kFields = 19;

// ------------------------------------------------------------------ binning (stable counting sort)
// wrapped coordinate in [0, L) (FP64), as the cell test takes it
__device__ __forceinline__ double wrapped(double xv, const AdjDev& P) { return xv - P.L * floor(xv * P.inv_L); }

// cell of every atom, counted
__global__ void __launch_bounds__(256) k_adj_count(const double* __restrict__ x, AdjDev P, int* __restrict__ cell_of,
                                                   const OrderBuf b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = 0;
  if (i < P.N)
    c = (cell_coord(x[3 * i + 2], P) * P.M + cell_coord(x[3 * i + 1], P)) * P.M + cell_coord(x[3 * i], P);
  if (i < P.N) cell_of[i] = c;
  order_count(i < P.N, c, blockIdx.x * 256, b);
}

// Atoms in cell order for the pair kernel, written by the last pass of the
// ordering: wrapped positions (FP64), the FP32 copy with the atom's index in w
// (bit 31: chain end, C_33), and for a tangent evaluation u = cu M^-1 beta.  The
// pair loop's two dependent gathers per candidate (perm, then the position)
// become one contiguous read.
struct EmitSorted {
  const double *x, *beta;
  double cu;
  AdjDev P;
  double *xs, *us;
  float4* s32;
  __device__ __forceinline__ void operator()(int s, int i) const {
    const int ty = site_type(i % P.sites, P.sites);
    float f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double w = wrapped(x[3 * i + a], P);
      xs[(size_t)a * P.N + s] = w;
      f[a] = (float)w;
      if (beta) us[(size_t)a * P.N + s] = cu * P.inv_mass[ty] * beta[3 * i + a];
    }
    s32[s] = make_float4(f[0], f[1], f[2], __uint_as_float((unsigned)i | ((unsigned)ty << 31)));
  }
};

// ------------------------------------------------------------------ LJ, Eq. (2): one warp per atom
// Bound: the FP64 pipe (about 2 operations per clock and SM).  A warp scans
// the 27 cells around its atom (945 candidates at 7,500 sites) with an FP32
// test, and queues those within r_c + 1e-4 nm in shared memory; the FP64
// arithmetic runs on 32 queued pairs at a time.  An FP64 warp instruction
// costs the same whether 4 or 32 lanes take part, and before the queue
// nearly every 32 candidates held a pair: 30 rounds of FP64 per atom where
// the ~138 pairs fill 5.  Periodic images come from the cells (the warp adds
// the cell's whole box to its own atom once), not from FP64 roundings per
// pair, and the lanes' sums are combined by a reduce-scatter (16 FP64 adds
// for 15 fields; a butterfly takes 75).  The cutoff is tested on the integer pipe and
// constants are taken out of the loop.  At 7,500 sites: values 376 -> 71 us,
// dual numbers 791 -> 150 us.
// Every operation of the gradient's value is written with its rounding, so
// the evaluations with and without energies give the same bits (the replay
// from a checkpoint reproduces the forward run).
constexpr int kLjWarps = 4;
constexpr int kAdjSlotBits = 22;   // a cell-order slot (N <= 2^22) in a queue entry

__device__ __forceinline__ double mul_r(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_r(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_r(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_r(float a, float b) { return __fadd_rn(a, b); }

// Sums of NF (a power of two) fields over the warp, by a fixed tree: after
// the first log2(NF) exchanges a lane holds one field, which the remaining
// ones complete.  Returns the sum of field (lane >> (5 - log2 NF)).
template <int NF, class R>
__device__ __forceinline__ R reduce_scatter(R (&f)[NF], int lane) {
  int n = NF;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int j = 0; j < NF / 2; ++j)
        if (j < n) {
          const R keep = up ? f[n + j] : f[j], send = up ? f[j] : f[n + j];
          f[j] = add_r(keep, __shfl_xor_sync(0xffffffffu, send, o));
        }
    } else {
      f[0] = add_r(f[0], __shfl_xor_sync(0xffffffffu, f[0], o));
    }
  }
  return f[0];
}

// R: scalar of the term arithmetic (double, or float for FP32 Hessian-vector
// products); TAN: with the derivative along u (and the parameter sums)
template <class R, bool TAN>
__global__ void __launch_bounds__(32 * kLjWarps) k_adj_lj(const double* __restrict__ xs, const double* __restrict__ us,
                                                          const float4* __restrict__ s32,
                                                          const int* __restrict__ cell_start,
                                                          const int* __restrict__ cell_of, AdjDev P, int energy,
                                                          double* __restrict__ gv, double* __restrict__ gt,
                                                          double* __restrict__ rec) {
  __shared__ int s_beg[kLjWarps][27];
  __shared__ int s_pre[kLjWarps][28];
  __shared__ float4 s_sh[kLjWarps][27];     // the atom moved to the cell's image (FP32); w: the image's code
  __shared__ unsigned s_q[kLjWarps][64];    // slot | image code << 22 | chain end << 28
  __shared__ double s_im[kLjWarps][9];      // the atom's coordinates (rows of 3) in images -1, 0, +1
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = blockIdx.x * kLjWarps + w;
  if (s >= P.N) return;   // the whole warp leaves together
  const size_t N = (size_t)P.N;
  const float4 xf = s32[s];
  const int i = (int)(__float_as_uint(xf.w) & 0x7fffffffu), ti = (int)(__float_as_uint(xf.w) >> 31);
  const int si = i % P.sites;
  const bool cells = P.n_off == 27;
  const float Lf = (float)P.L, iLf = (float)P.inv_L;
  if (lane < 9) {
    const double xa = xs[(size_t)(lane / 3) * N + s];
    s_im[w][lane] = lane % 3 == 1 ? xa : add_r(xa, lane % 3 == 0 ? P.L : -P.L);
  }
  // the neighbour cells: where their atoms start, how many, and the image
  // (-1, 0, +1 boxes per axis; code = sum of (n_a + 1) 4^a) they are met in
  int len = 0;
  if (lane < P.n_off) {
    int cell = 0, code = 21;                // 21: no shift on any axis
    float4 sh = xf;
    if (cells) {
      const int c = cell_of[i], M = P.M;
      int cx = c % M + lane % 3 - 1, cy = (c / M) % M + (lane / 3) % 3 - 1, cz = c / (M * M) + lane / 9 - 1;
      const int nx = cx < 0 ? -1 : (cx >= M ? 1 : 0), ny = cy < 0 ? -1 : (cy >= M ? 1 : 0),
                nz = cz < 0 ? -1 : (cz >= M ? 1 : 0);
      cx -= nx * M; cy -= ny * M; cz -= nz * M;
      cell = (cz * M + cy) * M + cx;
      code = (nx + 1) | ((ny + 1) << 2) | ((nz + 1) << 4);
      sh.x = xf.x - (float)nx * Lf; sh.y = xf.y - (float)ny * Lf; sh.z = xf.z - (float)nz * Lf;
    }
    sh.w = __int_as_float(code);
    s_sh[w][lane] = sh;
    s_beg[w][lane] = cell_start[cell];
    len = cell_start[cell + 1] - cell_start[cell];
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, len, o);
    if (lane >= o) len += v;
  }
  if (lane == 0) s_pre[w][0] = 0;
  if (lane < P.n_off) s_pre[w][lane + 1] = len;
  __syncwarp();
  const int total = s_pre[w][P.n_off];
  R gx = 0, gy = 0, gz = 0, hx = 0, hy = 0, hz = 0;         // gradient and its tangent
  R S12[2] = {0, 0}, S6[2] = {0, 0}, Sr[2] = {0, 0};        // sums over partners of type 0 / 1 of r^-12, r^-6, r
  R T12[2] = {0, 0}, T6[2] = {0, 0}, Tr[2] = {0, 0};        // r^-12 q/r^2, r^-6 q/r^2 (q = d(r^2)), dr
  R ev = 0;                                                 // value form: shifted energy (both halves of a pair)
  int cnt[2] = {0, 0};
  double du0 = 0, du1 = 0, du2 = 0;
  if (TAN) { du0 = us[s]; du1 = us[N + s]; du2 = us[2 * N + s]; }
  const long long rc2_bits = __double_as_longlong(P.rc2);
  // pair constants of the atom with a partner of type 0 / 1
  const R k6[2] = {(R)P.c6[ti], (R)P.c6[ti + 1]}, k12[2] = {(R)P.c12[ti], (R)P.c12[ti + 1]};
  const R k6x6[2] = {mul_r((R)6, k6[0]), mul_r((R)6, k6[1])}, nk24[2] = {(R)-24 * k6[0], (R)-24 * k6[1]};
  const R esh[2] = {k12[0] * (R)P.irc12 - k6[0] * (R)P.irc6, k12[1] * (R)P.irc12 - k6[1] * (R)P.irc6};

  auto pair = [&](unsigned ent) {
    const int t = (int)(ent & ((1u << kAdjSlotBits) - 1u)), code = (int)(ent >> kAdjSlotBits) & 63, tj = (int)(ent >> 28);
    double d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double xj = xs[a * N + t];
      if (cells) {
        d[a] = add_r(s_im[w][3 * a + ((code >> (2 * a)) & 3)], -xj);
      } else {
        d[a] = min_image(add_r(s_im[w][3 * a + 1], -xj), P);
      }
    }
    const double r2v = fma(d[2], d[2], fma(d[1], d[1], mul_r(d[0], d[0])));
    // the cutoff test on FP64 values, as the definition reads (r2v >= rc2 on
    // the integer pipe: non-negative numbers order like their bits, NaN stays in)
    const long long rb = __double_as_longlong(r2v);
    if (rb >= rc2_bits && rb <= 0x7ff0000000000000ll) return;
    const R dx = (R)d[0], dy = (R)d[1], dz = (R)d[2];
    const R r2 = std::is_same<R, double>::value ? (R)r2v : fma(dz, dz, fma(dy, dy, mul_r(dx, dx)));
    const R c6 = tj ? k6[1] : k6[0], c12 = tj ? k12[1] : k12[0], c6x6 = tj ? k6x6[1] : k6x6[0];
    const R i2 = (R)1 / r2;
    const R i6 = mul_r(mul_r(i2, i2), i2), i8 = mul_r(i6, i2);
    const R a = mul_r(c12, i6);
    // (1/r) dphi/dr = r^-8 (6 C6 - 12 C12 r^-6)
    R f = mul_r(fma((R)-12, a, c6x6), i8);
    R rr = 0, ir = 0, ksf = 0;
    if (P.sf) {
      // E_sf = E - E(r_c) - (r - r_c) E'(r_c): the same linear form in c12, c6
      rr = sqrt(r2);
      ir = (R)1 / rr;
      ksf = fma(c6x6, (R)P.irc7, -mul_r(mul_r((R)12, c12), (R)P.irc13));
      f = fma(-ksf, ir, f);
    }
    gx = fma(f, dx, gx); gy = fma(f, dy, gy); gz = fma(f, dz, gz);
    if (TAN) {
      const R vx = (R)(du0 - us[t]), vy = (R)(du1 - us[N + t]), vz = (R)(du2 - us[2 * N + t]);
      const R q = (R)2 * fma(dz, vz, fma(dy, vy, dx * vx));
      // df/d(r^2) = r^-10 (84 C12 r^-6 - 24 C6)
      R df = fma((R)84, a, tj ? nk24[1] : nk24[0]) * (i8 * i2);
      if (P.sf) df = fma((R)0.5 * ksf * ir, i2, df);
      const R ft = df * q;
      hx = fma(ft, dx, fma(f, vx, hx));
      hy = fma(ft, dy, fma(f, vy, hy));
      hz = fma(ft, dz, fma(f, vz, hz));
      const R i12 = i6 * i6, wq = i2 * q;
      const R rt = P.sf ? (R)0.5 * q * ir : (R)0;
      if (tj) {
        S12[1] += i12; S6[1] += i6; T12[1] = fma(i12, wq, T12[1]); T6[1] = fma(i6, wq, T6[1]);
        if (P.sf) { Sr[1] += rr; Tr[1] += rt; }
        ++cnt[1];
      } else {
        S12[0] += i12; S6[0] += i6; T12[0] = fma(i12, wq, T12[0]); T6[0] = fma(i6, wq, T6[0]);
        if (P.sf) { Sr[0] += rr; Tr[0] += rt; }
        ++cnt[0];
      }
    } else if (energy) {
      R e = fma(a - c6, i6, -(tj ? esh[1] : esh[0]));
      if (P.sf) e = fma(-ksf, rr - (R)P.rc, e);   // - (r - r_c) E'(r_c)
      ev += e;
    }
  };

  int qn = 0, o = 0;
  const unsigned lt = (1u << lane) - 1u;
  for (int base = 0; base < total; base += 32) {
    const int q = base + lane;
    bool pass = false;
    unsigned ent = 0u;
    if (q < total) {
      while (q >= s_pre[w][o + 1]) ++o;
      const int t = s_beg[w][o] + (q - s_pre[w][o]);
      const float4 c = s32[t], sh = s_sh[w][o];
      const unsigned cb = __float_as_uint(c.w);
      const int dj = (int)(cb & 0x7fffffffu) - i;
      // itself and its 1-2 and 1-3 neighbours (Sec. 3.1): |i - j| <= 2 on one chain
      const bool excl = (unsigned)(dj + 2) <= 4u && (unsigned)(si + dj) < (unsigned)P.sites;
      // FP32 prefilter on the wrapped copies (error ~1e-6 nm in a melt's box against a margin of 1e-4)
      float ex = sh.x - c.x, ey = sh.y - c.y, ez = sh.z - c.z;
      if (!cells) {
        ex -= Lf * rintf(ex * iLf); ey -= Lf * rintf(ey * iLf); ez -= Lf * rintf(ez * iLf);
      }
      pass = !excl && ex * ex + ey * ey + ez * ez <= P.pre2;
      ent = (unsigned)t | ((unsigned)__float_as_int(sh.w) << kAdjSlotBits) | ((cb >> 31) << 28);
    }
    const unsigned b = __ballot_sync(0xffffffffu, pass);
    if (pass) s_q[w][qn + __popc(b & lt)] = ent;
    qn += __popc(b);
    __syncwarp();
    if (qn >= 32) {
      pair(s_q[w][lane]);
      __syncwarp();
      const unsigned rest = s_q[w][32 + lane];
      __syncwarp();
      s_q[w][lane] = rest;
      __syncwarp();
      qn -= 32;
    }
  }
  if (lane < qn) pair(s_q[w][lane]);
  __syncwarp();

  if (!TAN) {
    R f[4] = {gx, gy, gz, (R)0.5 * ev};
    const double v = (double)reduce_scatter<4, R>(f, lane);
    if ((lane & 7) == 0) {
      const int k = lane >> 3;
      if (k < 3) gv[3 * i + k] = v;
      else if (energy) rec[(size_t)kRec * i + kElj] = v;
    }
  } else {
    // half of each pair: A = 1/2 sum (r^-12 - r_c^-12), B likewise (with the
    // force-shift terms), and their tangents
    R A[2], B[2], At[2], Bt[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const R n = (R)cnt[k];
      A[k] = (R)0.5 * (S12[k] - n * (R)P.irc12);
      B[k] = (R)0.5 * (S6[k] - n * (R)P.irc6);
      At[k] = (R)-3 * T12[k];
      Bt[k] = (R)-1.5 * T6[k];
      if (P.sf) {
        A[k] += (R)6 * (R)P.irc13 * (Sr[k] - n * (R)P.rc);
        B[k] += (R)3 * (R)P.irc7 * (Sr[k] - n * (R)P.rc);
        At[k] += (R)6 * (R)P.irc13 * Tr[k];
        Bt[k] += (R)3 * (R)P.irc7 * Tr[k];
      }
    }
    const R e = (k12[0] * A[0] - k6[0] * B[0]) + (k12[1] * A[1] - k6[1] * B[1]);
    R f[16] = {gx, gy, gz, hx, hy, hz, A[0], At[0], B[0], Bt[0], A[1], At[1], B[1], Bt[1], e, (R)0};
    const double v = (double)reduce_scatter<16, R>(f, lane);
    if ((lane & 1) == 0) {
      const int k = lane >> 1;
      double* rc = rec + (size_t)kRec * i;
      // partner type 0 -> pair type ti, partner type 1 -> pair type ti + 1;
      // the atom takes no part in the third type
      if (k < 3) gv[3 * i + k] = v;
      else if (k < 6) gt[3 * i + k - 3] = v;
      else if (k < 14) rc[kA + 4 * ti + k - 6] = v;
      else if (k == 14) rc[kElj] = v;
      else
        for (int z = 0; z < 4; ++z) rc[kA + 4 * (ti ? 0 : 2) + z] = 0.0;
    }
  }
}

// ------------------------------------------------------------------ bonded, Eqs. (4)-(6)
// gradient of each term's energy with respect to its atoms (not the force)
// d = x_b - x_a (minimum image)
template <class T>
__device__ __forceinline__ T bond_grad(V3<T> d, const AdjDev& P, V3<T>* g) {
  const T r = gsqrt(dot(d, d));
  const T dr = r - P.b0;
  const T s = P.kb * dr / r;
  g[0] = scale(-s, d);
  g[1] = scale(s, d);
  return 0.5 * P.kb * dr * dr;
}

// theta = angle(u, w), u = x_a - x_b, w = x_c - x_b:
// dtheta/du = ((u.w / u.u) u - w) / |u x w|, likewise for w
template <class T>
__device__ __forceinline__ T angle_grad(V3<T> u, V3<T> w, const AdjDev& P, V3<T>* g) {
  const T c = dot(u, w);
  const T s = gsqrt(dot(cross(u, w), cross(u, w)));
  const T th = gatan2(s, c);
  const T k = P.ka * (th - P.theta0) / s;
  g[0] = scale(k, scale(c / dot(u, u), u) - w);
  g[2] = scale(k, scale(c / dot(w, w), w) - u);
  g[1] = V3<T>{-(g[0].x + g[2].x), -(g[0].y + g[2].y), -(g[0].z + g[2].z)};
  return 0.5 * P.ka * (th - P.theta0) * (th - P.theta0);
}

// IUPAC dihedral of b1 = x_b - x_a, b2 = x_c - x_b, b3 = x_d - x_c with
// m = b1 x b2, n = b2 x b3, phi = atan2(|b2| b1.n, m.n).  Gradient of phi:
// G_a = -|b2|/|m|^2 m, G_d = |b2|/|n|^2 n, G_b = -(1+p) G_a + q G_d,
// G_c = p G_a - (1+q) G_d, p = b1.b2/|b2|^2, q = b3.b2/|b2|^2.
// Returns D = 1 + cos(n phi - phi_s); the energy is k_phi D (Eq. 6).
template <class T>
__device__ __forceinline__ T dihedral_grad(V3<T> b1, V3<T> b2, V3<T> b3, const AdjDev& P, V3<T>* g) {
  const V3<T> m = cross(b1, b2), n = cross(b2, b3);
  const T bb = dot(b2, b2);
  const T lb2 = gsqrt(bb);
  const T phi = gatan2(lb2 * dot(b1, n), dot(m, n));
  const T arg = (double)P.n_mult * phi - P.phis;
  const T dEdphi = (-P.kphi * (double)P.n_mult) * gsin(arg);
  const V3<T> Ga = scale(-(lb2 / dot(m, m)), m);
  const V3<T> Gd = scale(lb2 / dot(n, n), n);
  const T p = dot(b1, b2) / bb, q = dot(b3, b2) / bb;
  const V3<T> Gb = scale(q, Gd) - scale(1.0 + p, Ga);
  const V3<T> Gc = scale(p, Ga) - scale(1.0 + q, Gd);
  g[0] = scale(dEdphi, Ga);
  g[1] = scale(dEdphi, Gb);
  g[2] = scale(dEdphi, Gc);
  g[3] = scale(dEdphi, Gd);
  return 1.0 + gcos(arg);
}

// A block owns kBondTile consecutive atoms and evaluates every term that
// touches them once: warps 0-1 the dihedrals, 2-3 the angles, 4-5 the bonds
// starting at the atoms from 3 before the tile to its end (a halo of three
// terms is evaluated twice, by neighbouring blocks).  The bond vectors are
// formed once in shared memory; the terms leave their gradients there and
// each atom adds those of its terms in a fixed order.  Before, a thread per
// atom evaluated all nine terms the atom is in: four times the FP64
// operations that bound the kernel (44 -> 11 us, dual numbers 86 -> 22 us,
// at 7,500 sites).  rec == nullptr: the gradient alone.
constexpr int kBondTerms = 64;
constexpr int kBondTile = kBondTerms - 3;

template <class T>
__global__ void __launch_bounds__(3 * kBondTerms) k_adj_bonded(const double* __restrict__ x,
                                                               const double* __restrict__ beta, double cu, AdjDev P,
                                                               double* __restrict__ gv, double* __restrict__ gt,
                                                               double* __restrict__ rec) {
  __shared__ V3<T> bv[kBondTerms + 2];      // x_{m+1} - x_m of the term atoms' bonds
  __shared__ V3<T> gb[kBondTerms], ga[3][kBondTerms], gd[4][kBondTerms];
  __shared__ double eb[kBondTerms], ea[kBondTerms], dv[kBondTerms], dt[kBondTerms];
  const int start = blockIdx.x * kBondTile - 3;   // atom of term 0 (the first three: halo)
  const int tid = threadIdx.x, role = tid / kBondTerms, q = tid % kBondTerms;
  for (int k = tid; k < kBondTerms + 2; k += 3 * kBondTerms) {
    const int m = start + k;
    if (m >= 0 && m + 1 < P.N && m % P.sites + 1 < P.sites) bv[k] = sep<T>(x, beta, cu, m, m + 1, P);
  }
  __syncthreads();
  const int m = start + q;
  const int sm = m >= 0 && m < P.N ? m % P.sites : P.sites;   // P.sites: no term starts here
  if (role == 0) {
    V3<T> g[4] = {V3<T>{}, V3<T>{}, V3<T>{}, V3<T>{}};
    T D = T{};
    if (sm + 3 < P.sites) D = dihedral_grad<T>(bv[q], bv[q + 1], bv[q + 2], P, g);
#pragma unroll
    for (int k = 0; k < 4; ++k) gd[k][q] = g[k];
    dv[q] = value(D);
    dt[q] = tangent(D);
  } else if (role == 1) {
    V3<T> g[3] = {V3<T>{}, V3<T>{}, V3<T>{}};
    T e = T{};
    if (sm + 2 < P.sites) {
      const V3<T> u = V3<T>{-bv[q].x, -bv[q].y, -bv[q].z};
      e = angle_grad<T>(u, bv[q + 1], P, g);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) ga[k][q] = g[k];
    ea[q] = value(e);
  } else {
    V3<T> g[2] = {V3<T>{}, V3<T>{}};
    T e = T{};
    if (sm + 1 < P.sites) e = bond_grad<T>(bv[q], P, g);
    gb[q] = g[1];   // g[0] = -g[1]
    eb[q] = value(e);
  }
  __syncthreads();
  if (tid >= kBondTile) return;
  const int i = start + 3 + tid, k = tid + 3;
  if (i >= P.N) return;
  const int si = i % P.sites, o = i - si;
  V3<T> g = {T{}, T{}, T{}};
  if (si >= 1) g = g + gb[k - 1];
  if (si + 1 < P.sites) g = g - gb[k];
#pragma unroll
  for (int t = 2; t >= 0; --t)
    if (si >= t && si - t + 2 < P.sites) g = g + ga[t][k - t];
#pragma unroll
  for (int t = 3; t >= 0; --t)
    if (si >= t && si - t + 3 < P.sites) g = g + gd[t][k - t];
  gv[3 * i] += value(g.x); gv[3 * i + 1] += value(g.y); gv[3 * i + 2] += value(g.z);
  if (gt) { gt[3 * i] += tangent(g.x); gt[3 * i + 1] += tangent(g.y); gt[3 * i + 2] += tangent(g.z); }
  if (!rec) return;
  double* R = rec + (size_t)kRec * i;
  R[kD] = dv[k];
  R[kD + 1] = dt[k];
  R[kEb] = eb[k];
  R[kEa] = ea[k];
  R[kEd] = P.kphi * dv[k];
  double r2 = 0.0;
  if (si == 0) {
    const int l = o + P.sites - 1;
    const double ex = x[3 * l] - x[3 * o], ey = x[3 * l + 1] - x[3 * o + 1], ez = x[3 * l + 2] - x[3 * o + 2];
    r2 = ex * ex + ey * ey + ez * ez;
  }
  R[kR2] = r2;
}

// ------------------------------------------------------------------ reductions (fixed order)
// Fields F0 .. F0 + NF - 1 of the records in one launch: thread (group g,
// field f) of a block adds atoms g, g + G, ... of the block's range (the
// block reads its records as one contiguous run), the groups are added in a
// fixed order, and the last block to finish (a ticket; no waiting) adds the
// blocks' sums in block order.  Before, a block summed the fields one after
// another with two barriers each, and a second kernel added 64 partials on
// one thread per field: 18.4 + 5.0 -> 7.4 us (5.8 for the five fields of a forward step) at 7,500 sites.
constexpr int kRedBlocks = 128, kRedThreads = 320;

constexpr int kOrderPad = 16;   // ints ahead of the ordering's counters (the first is the reduction's ticket)

// accumulator layout
constexpr int kAccU = 0, kAccR2 = 1;      // forward sums of U_k and R_ee^2_k
constexpr int kAccC12 = 2, kAccC6 = 5;    // dJ/dc12_t, dJ/dc6_t (t = 0, 1, 2)
constexpr int kAccKphi = 8;               // dJ/dk_phi
constexpr int kAccN = 16;

// sum of sh[g][f] over the G groups, for thread f < NF (others: 0)
template <int NF, int G>
__device__ __forceinline__ double group_sum(double (*sh)[NF], double (*sh2)[NF]) {
  constexpr int P = 8;
  static_assert(G % P == 0 && NF * P <= kRedThreads, "group layout");
  __syncthreads();
  if ((int)threadIdx.x < NF * P) {
    const int f = threadIdx.x % NF, p = threadIdx.x / NF;
    double s = 0.0;
#pragma unroll
    for (int g = 0; g < G / P; ++g) s += sh[p * (G / P) + g][f];
    sh2[p][f] = s;
  }
  __syncthreads();
  double s = 0.0;
  if ((int)threadIdx.x < NF) {
#pragma unroll
    for (int p = 0; p < P; ++p) s += sh2[p][threadIdx.x];
  }
  return s;
}

// mode 0: forward sums, 1: reverse step (wu = w_k w0, the weight of U at this
// step), 2: totals only
template <int F0, int NF>
__global__ void __launch_bounds__(kRedThreads) k_adj_reduce(const double* __restrict__ rec, int N, int n_chains,
                                                            int mode, double wu, double* __restrict__ part,
                                                            int* __restrict__ ticket, double* __restrict__ totals,
                                                            double* __restrict__ acc) {
  constexpr int G = kRedThreads / NF / 8 * 8;
  __shared__ double sh[G][NF], sh2[8][NF];
  __shared__ bool last;
  const int f = threadIdx.x % NF, g = threadIdx.x / NF;
  const int per = (N + gridDim.x - 1) / gridDim.x;
  const int b = blockIdx.x * per, e = min(b + per, N);
  if (g < G) {
    double s = 0.0;
    for (int i = b + g; i < e; i += G) s += rec[(size_t)kRec * i + F0 + f];
    sh[g][f] = s;
  }
  double t = group_sum<NF, G>(sh, sh2);
  if ((int)threadIdx.x < NF) part[blockIdx.x * kRec + threadIdx.x] = t;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (g < G) {
    double s = 0.0;
    for (int k = g; k < (int)gridDim.x; k += G) s += __ldcg(part + k * kRec + f);
    sh[g][f] = s;
  }
  t = group_sum<NF, G>(sh, sh2);
  __shared__ double tot[kRec];
  if ((int)threadIdx.x < NF) totals[F0 + threadIdx.x] = tot[F0 + threadIdx.x] = t;
  __syncthreads();
  if (threadIdx.x != 0) return;
  *ticket = 0;
  if (mode == 0) {
    acc[kAccU] += tot[kElj] + tot[kEb] + tot[kEa] + tot[kEd];
    acc[kAccR2] += tot[kR2] / (double)n_chains;
  } else if (mode == 1) {
    for (int t3 = 0; t3 < 3; ++t3) {
      // U = sum_t (c12_t A_t - c6_t B_t) + bonded; the mixed term is the
      // tangent of the same sums along u
      acc[kAccC12 + t3] += wu * tot[kA + 4 * t3 + 0] - tot[kA + 4 * t3 + 1];
      acc[kAccC6 + t3] += -wu * tot[kA + 4 * t3 + 2] + tot[kA + 4 * t3 + 3];
    }
    acc[kAccKphi] += wu * tot[kD] - tot[kD + 1];
  }
}

// ------------------------------------------------------------------ integrator and adjoint updates
// Make every chain continuous (one thread per chain, x,y,z per atom): site k
// is moved by whole box lengths, L s_k, where s_k accumulates -rint(d / L)
// over the bonds d = x_k - x_{k-1} of the positions as given, so each bond
// becomes its minimum image.  A site with s_k = 0 keeps its bits.
__global__ void __launch_bounds__(128) k_adj_unwrap(double* __restrict__ x, AdjDev P) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= P.n_chains) return;
  double* xc = x + 3 * (size_t)c * P.sites;
  double prev[3] = {xc[0], xc[1], xc[2]};
  double s[3] = {0.0, 0.0, 0.0};
  for (int k = 1; k < P.sites; ++k) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double cur = xc[3 * k + a];
      s[a] -= rint((cur - prev[a]) * P.inv_L);
      prev[a] = cur;
      if (s[a] != 0.0) xc[3 * k + a] = cur + P.L * s[a];
    }
  }
}

__global__ void __launch_bounds__(256) k_adj_kick_drift(double* __restrict__ x, double* __restrict__ v,
                                                        const double* __restrict__ gv, AdjDev P, double dt,
                                                        double* __restrict__ x_store) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  const double hm = 0.5 * dt * P.inv_mass[site_type(i % P.sites, P.sites)];
  for (int q = 0; q < 3; ++q) {
    const double vh = v[3 * i + q] - hm * gv[3 * i + q];
    v[3 * i + q] = vh;
    x[3 * i + q] += dt * vh;
    if (x_store) x_store[3 * i + q] = x[3 * i + q];
  }
}

__global__ void __launch_bounds__(256) k_adj_kick(double* __restrict__ v, const double* __restrict__ gv, AdjDev P,
                                                  double dt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  const double hm = 0.5 * dt * P.inv_mass[site_type(i % P.sites, P.sites)];
  for (int q = 0; q < 3; ++q) v[3 * i + q] -= hm * gv[3 * i + q];
}

// alpha = wu grad U + wr grad R_ee^2 + alpha - H u;  beta += dt alpha (if update_beta)
__global__ void __launch_bounds__(256) k_adj_update(const double* __restrict__ x, const double* __restrict__ gv,
                                                    const double* __restrict__ gt, AdjDev P, double wu, double wr,
                                                    double dt, int update_beta, double* __restrict__ alpha,
                                                    double* __restrict__ beta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  const int si = i % P.sites, o = i - si, l = o + P.sites - 1;
  double gr[3] = {0.0, 0.0, 0.0};
  if (si == 0 || si == P.sites - 1) {
    const double sgn = (si == 0 ? -2.0 : 2.0) / (double)P.n_chains;
    for (int q = 0; q < 3; ++q) gr[q] = sgn * (x[3 * l + q] - x[3 * o + q]);
  }
  for (int q = 0; q < 3; ++q) {
    const double a = wu * gv[3 * i + q] + wr * gr[q] + alpha[3 * i + q] - gt[3 * i + q];
    alpha[3 * i + q] = a;
    if (update_beta) beta[3 * i + q] += dt * a;
  }
}

}  // namespace adj
}  // namespace mdg

using namespace mdg;
using namespace mdg::adj;

// ------------------------------------------------------------------ handle
struct md_adj {
  AdjDev P;
  double theta[5];
  double dt;
  int K, C, S;                 // steps, checkpoint interval, segments
  cudaStream_t st;
  bool own_stream;
  int C_cells;
  bool hvp32;                  // Hessian-vector products in FP32 (md_adj_desc.hvp_precision = 1)
  // device buffers (one allocation)
  void* mem;
  double *x, *v, *gv, *gt, *alpha, *beta, *rec, *part, *acc, *totals, *ckx, *ckv, *seg, *xk, *xs, *us;
  float4* x32;                 // cell order: FP32 wrapped position, atom index and type
  int *count, *cell_start, *cell_of, *tmp, *perm, *seg_scan, *ticket;
  bool have_forward;
  double obs[2];
};

namespace {

int adj_fail(int code, const char* msg) {
  md_set_global_error(msg);
  if (code == MD_ECUDA || code == MD_ENOMEM) cudaGetLastError();   // reported: not left to the next call
  return code;
}

void set_pair_coefficients(md_adj* a) {
  const double eps[2] = {a->theta[0], a->theta[1]}, sig[2] = {a->theta[2], a->theta[3]};
  const int ta[3] = {0, 0, 1}, tb[3] = {0, 1, 1};
  for (int t = 0; t < 3; ++t) {
    const double e = std::sqrt(eps[ta[t]] * eps[tb[t]]), s = std::sqrt(sig[ta[t]] * sig[tb[t]]);
    const double s6 = s * s * s * s * s * s;
    a->P.c6[t] = 4.0 * e * s6;
    a->P.c12[t] = 4.0 * e * s6 * s6;
  }
  a->P.kphi = a->theta[4];
}

// one evaluation at positions xp: gradient (and, with beta, its tangent
// along cu M^-1 beta) plus the per-atom record, then the reductions (mode as
// in k_adj_reduce; without beta, mode 2 is the gradient alone)
int evaluate(md_adj* a, const double* xp, const double* beta, double cu, int mode, double wu) {
  const AdjDev& P = a->P;
  cudaStream_t st = a->st;
  const int N = P.N;
  const OrderBuf ob = order_buffers(a->count, N, a->C_cells);
  // the reduction's ticket and the ordering's counters in one run
  if (cudaMemsetAsync(a->ticket, 0, sizeof(int) * (kOrderPad + order_clear_ints(ob, a->C_cells)), st) != cudaSuccess)
    return MD_ECUDA;
  k_adj_count<<<(N + 255) / 256, 256, 0, st>>>(xp, P, a->cell_of, ob);
  launch_cell_order(a->cell_of, N, a->C_cells, ob, a->cell_start, a->seg_scan, a->tmp, a->perm,
                    EmitSorted{xp, beta, cu, P, a->xs, a->us, a->x32}, false, st);
  const int lj_blocks = (N + kLjWarps - 1) / kLjWarps, b_blocks = (N + kBondTile - 1) / kBondTile;
  if (beta && a->hvp32) {
    k_adj_lj<float, true><<<lj_blocks, 32 * kLjWarps, 0, st>>>(a->xs, a->us, a->x32, a->cell_start, a->cell_of, P, 1,
                                                                 a->gv, a->gt, a->rec);
    k_adj_bonded<DualF><<<b_blocks, 3 * kBondTerms, 0, st>>>(xp, beta, cu, P, a->gv, a->gt, a->rec);
  } else if (beta) {
    k_adj_lj<double, true><<<lj_blocks, 32 * kLjWarps, 0, st>>>(a->xs, a->us, a->x32, a->cell_start, a->cell_of, P, 1,
                                                                  a->gv, a->gt, a->rec);
    k_adj_bonded<Dual><<<b_blocks, 3 * kBondTerms, 0, st>>>(xp, beta, cu, P, a->gv, a->gt, a->rec);
  } else {
    k_adj_lj<double, false><<<lj_blocks, 32 * kLjWarps, 0, st>>>(a->xs, a->us, a->x32, a->cell_start, a->cell_of, P,
                                                                   mode != 2, a->gv, nullptr, a->rec);
    k_adj_bonded<double><<<b_blocks, 3 * kBondTerms, 0, st>>>(xp, nullptr, 0.0, P, a->gv, nullptr,
                                                              mode != 2 ? a->rec : nullptr);
    if (mode == 2) return cudaPeekAtLastError() == cudaSuccess ? MD_OK : MD_ECUDA;   // the gradient alone
  }
  const int nb = N < kRedBlocks ? 1 : kRedBlocks;
  // without a tangent only the energies and R_ee^2 are asked for
  if (beta)
    k_adj_reduce<0, kFields><<<nb, kRedThreads, 0, st>>>(a->rec, N, P.n_chains, mode, wu, a->part, a->ticket,
                                                         a->totals, a->acc);
  else
    k_adj_reduce<kElj, kFields - kElj><<<nb, kRedThreads, 0, st>>>(a->rec, N, P.n_chains, mode, wu, a->part,
                                                                   a->ticket, a->totals, a->acc);
  return cudaPeekAtLastError() == cudaSuccess ? MD_OK : MD_ECUDA;
}

// (dJ/dc12_t, dJ/dc6_t, dJ/dk_phi) -> (eps_C32, eps_C33, sigma_C32, sigma_C33, k_phi)
void chain_rule(const md_adj* a, const double* acc, double* grad) {
  const double eps[2] = {a->theta[0], a->theta[1]}, sig[2] = {a->theta[2], a->theta[3]};
  const int ta[3] = {0, 0, 1}, tb[3] = {0, 1, 1};
  for (int k = 0; k < 4; ++k) grad[k] = 0.0;
  for (int t = 0; t < 3; ++t) {
    const double e = std::sqrt(eps[ta[t]] * eps[tb[t]]), s = std::sqrt(sig[ta[t]] * sig[tb[t]]);
    const double c6 = a->P.c6[t], c12 = a->P.c12[t];
    const double dJ_de = (acc[kAccC12 + t] * c12 + acc[kAccC6 + t] * c6) / e;
    const double dJ_ds = (12.0 * acc[kAccC12 + t] * c12 + 6.0 * acc[kAccC6 + t] * c6) / s;
    // d eps_t / d eps_a = eps_t / (2 eps_a) per appearance of a in the pair
    for (int side = 0; side < 2; ++side) {
      const int ty = side == 0 ? ta[t] : tb[t];
      grad[ty] += dJ_de * e / (2.0 * eps[ty]);
      grad[2 + ty] += dJ_ds * s / (2.0 * sig[ty]);
    }
  }
  grad[4] = acc[kAccKphi];
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Record the launches `body` enqueues on the adjoint's stream as one CUDA
// graph (the per-step launch sequence is replayed instead of re-launched).
template <class F>
bool capture(md_adj* a, cudaGraphExec_t* exec, F&& body) {
  *exec = nullptr;
  cudaGraph_t g = nullptr;
  if (cudaStreamBeginCapture(a->st, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return false;
  const int rc = body();
  const cudaError_t refused = cudaGetLastError();
  const cudaError_t e = cudaStreamEndCapture(a->st, &g);
  if (rc != MD_OK || refused != cudaSuccess || e != cudaSuccess || !g) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return false;
  }
  const cudaError_t ie = cudaGraphInstantiate(exec, g, 0);
  cudaGraphDestroy(g);
  if (ie != cudaSuccess) {
    *exec = nullptr;
    cudaGetLastError();
    return false;
  }
  return true;
}

}  // namespace

extern "C" int md_adj_create(const md_adj_desc* d, md_adj** out) {
  if (!d || !out) return adj_fail(MD_EINVAL, "null argument");
  *out = nullptr;
  if (d->n_chains < 1 || d->sites_per_chain < 2 || d->sites_per_chain > 4096)
    return adj_fail(MD_EINVAL, "n_chains must be >= 1 and sites_per_chain 2 .. 4096");
  const long long N = (long long)d->n_chains * d->sites_per_chain;
  if (N > (1 << 22)) return adj_fail(MD_EINVAL, "more than 4,194,304 atoms");
  if (!(d->box > 0) || !std::isfinite(d->box) || !(d->rc > 0) || !(d->dt > 0))
    return adj_fail(MD_EINVAL, "box, rc and dt must be positive");
  if (d->n_steps < 0 || d->n_steps > 10000000 || d->checkpoint_every < 1)
    return adj_fail(MD_EINVAL, "n_steps must be 0 .. 1e7 and checkpoint_every >= 1");
  const md_params& p = d->params;
  if (!(p.mass[0] > 0) || !(p.mass[1] > 0) || !(p.eps[0] > 0) || !(p.eps[1] > 0) || !(p.sigma[0] > 0) ||
      !(p.sigma[1] > 0))
    return adj_fail(MD_EINVAL, "masses, eps and sigma must be positive");
  md_adj* a = new (std::nothrow) md_adj();
  if (!a) return adj_fail(MD_ENOMEM, "host allocation failed");
  AdjDev& P = a->P;
  P.L = d->box;
  P.inv_L = 1.0 / d->box;
  int M = (int)std::floor(d->box / d->rc);
  if (M > 256) M = 256;
  if (M < 3) M = 1;
  P.M = M;
  P.n_off = M >= 3 ? 27 : 1;
  P.inv_h = (double)M / d->box;
  P.sites = d->sites_per_chain;
  P.n_chains = d->n_chains;
  P.N = (int)N;
  P.rc2 = d->rc * d->rc;
  const double irc2 = 1.0 / P.rc2;
  P.irc6 = irc2 * irc2 * irc2;
  P.irc12 = P.irc6 * P.irc6;
  P.rc = d->rc;
  P.irc7 = P.irc6 / d->rc;
  P.irc13 = P.irc12 / d->rc;
  if (d->lj_form != 0 && d->lj_form != 1) {
    delete a;
    return adj_fail(MD_EINVAL, "lj_form must be 0 or 1");
  }
  P.sf = d->lj_form;
  if (d->hvp_precision != 0 && d->hvp_precision != 1) {
    delete a;
    return adj_fail(MD_EINVAL, "hvp_precision must be 0 (FP64) or 1 (FP32)");
  }
  a->hvp32 = d->hvp_precision == 1;
  // margin over the FP32 roundings of two wrapped coordinates, L and the image's
  // sum: 2.5 spacings of L per axis, 5.2e-7 L in r (1e-4 nm up to 166 nm)
  const double margin = std::max(1e-4, 6e-7 * d->box);
  P.pre2 = (float)((d->rc + margin) * (d->rc + margin));
  P.kb = p.kb; P.b0 = p.b0; P.ka = p.ka; P.theta0 = p.theta0; P.phis = p.phis; P.n_mult = p.n_mult;
  P.inv_mass[0] = 1.0 / p.mass[0];
  P.inv_mass[1] = 1.0 / p.mass[1];
  a->theta[0] = p.eps[0]; a->theta[1] = p.eps[1]; a->theta[2] = p.sigma[0]; a->theta[3] = p.sigma[1];
  a->theta[4] = p.kphi;
  set_pair_coefficients(a);
  a->dt = d->dt;
  a->K = d->n_steps;
  a->C = d->checkpoint_every < d->n_steps ? d->checkpoint_every : (d->n_steps > 0 ? d->n_steps : 1);
  a->S = d->n_steps == 0 ? 1 : (d->n_steps + a->C - 1) / a->C;
  a->C_cells = M * M * M;
  a->st = (cudaStream_t)d->cuda_stream;
  a->own_stream = false;
  if (!a->st) {
    if (cudaStreamCreateWithFlags(&a->st, cudaStreamNonBlocking) != cudaSuccess) {
      delete a;
      return adj_fail(MD_ECUDA, "stream creation failed");
    }
    a->own_stream = true;
  }
  const size_t n3 = sizeof(double) * 3 * (size_t)N;
  const size_t sizes[] = {n3, n3, n3, n3, n3, n3, sizeof(double) * kRec * (size_t)N,
                          sizeof(double) * kRec * kRedBlocks, sizeof(double) * kAccN, sizeof(double) * kRec,
                          n3 * a->S, n3 * a->S, n3 * (size_t)(a->C + 1), sizeof(int) * (kOrderPad + order_ints((int)N, a->C_cells)),
                          sizeof(int) * (a->C_cells + 1), sizeof(int) * (size_t)N,
                          sizeof(int) * scan_seg_ints(a->C_cells), sizeof(int) * (size_t)N, sizeof(int) * (size_t)N, n3,
                          sizeof(float4) * (size_t)N, n3, n3};
  const int nbuf = sizeof(sizes) / sizeof(sizes[0]);
  size_t total = 0;
  for (int k = 0; k < nbuf; ++k) total += align256(sizes[k]);
  if (cudaMalloc(&a->mem, total) != cudaSuccess) {
    cudaGetLastError();
    if (a->own_stream) cudaStreamDestroy(a->st);
    delete a;
    return adj_fail(MD_ENOMEM, "device allocation for the adjoint failed");
  }
  char* m = (char*)a->mem;
  void* ptrs[nbuf];
  for (int k = 0; k < nbuf; ++k) { ptrs[k] = m; m += align256(sizes[k]); }
  a->x = (double*)ptrs[0]; a->v = (double*)ptrs[1]; a->gv = (double*)ptrs[2]; a->gt = (double*)ptrs[3];
  a->alpha = (double*)ptrs[4]; a->beta = (double*)ptrs[5]; a->rec = (double*)ptrs[6]; a->part = (double*)ptrs[7];
  a->acc = (double*)ptrs[8]; a->totals = (double*)ptrs[9]; a->ckx = (double*)ptrs[10]; a->ckv = (double*)ptrs[11];
  a->seg = (double*)ptrs[12]; a->ticket = (int*)ptrs[13]; a->count = a->ticket + kOrderPad; a->cell_start = (int*)ptrs[14];
  a->cell_of = (int*)ptrs[15]; a->seg_scan = (int*)ptrs[16]; a->tmp = (int*)ptrs[17]; a->perm = (int*)ptrs[18];
  a->xk = (double*)ptrs[19];
  a->x32 = (float4*)ptrs[20];
  a->xs = (double*)ptrs[21]; a->us = (double*)ptrs[22];
  a->have_forward = false;
  *out = a;
  return MD_OK;
}

extern "C" int md_adj_set_theta(md_adj* a, const double theta[5]) {
  if (!a || !theta) return adj_fail(MD_EINVAL, "null argument");
  for (int k = 0; k < 5; ++k)
    if (!std::isfinite(theta[k]) || (k < 4 && !(theta[k] > 0))) return adj_fail(MD_EINVAL, "eps and sigma must be positive");
  std::memcpy(a->theta, theta, sizeof(a->theta));
  set_pair_coefficients(a);
  a->have_forward = false;
  return MD_OK;
}

extern "C" int md_adj_forward(md_adj* a, const double* pos, const double* vel, double obs[2]) {
  if (!a || !pos || !vel) return adj_fail(MD_EINVAL, "null argument");
  const size_t n3 = sizeof(double) * 3 * (size_t)a->P.N;
  cudaStream_t st = a->st;
  if (cudaMemcpyAsync(a->x, pos, n3, cudaMemcpyDefault, st) != cudaSuccess ||
      cudaMemcpyAsync(a->v, vel, n3, cudaMemcpyDefault, st) != cudaSuccess ||
      cudaMemsetAsync(a->acc, 0, sizeof(double) * kAccN, st) != cudaSuccess)
    return adj_fail(MD_ECUDA, "upload of the initial state failed");
  k_adj_unwrap<<<(a->P.n_chains + 127) / 128, 128, 0, st>>>(a->x, a->P);
  const int nb = (a->P.N + 255) / 256;
  if (evaluate(a, a->x, nullptr, 0.0, 0, 0.0) != MD_OK) return adj_fail(MD_ECUDA, "force evaluation failed");
  // one velocity-Verlet step (kick-drift, forces and sums, kick) as a graph
  cudaGraphExec_t step = nullptr;
  if (a->K > 0 && !capture(a, &step, [&]() {
        k_adj_kick_drift<<<nb, 256, 0, st>>>(a->x, a->v, a->gv, a->P, a->dt, nullptr);
        const int rc = evaluate(a, a->x, nullptr, 0.0, 0, 0.0);
        k_adj_kick<<<nb, 256, 0, st>>>(a->v, a->gv, a->P, a->dt);
        return rc;
      }))
    return adj_fail(MD_ECUDA, "capturing the forward step failed");
  int grc = MD_OK;
  for (int k = 0; k < a->K && grc == MD_OK; ++k) {
    if (k % a->C == 0) {
      const size_t s = (size_t)(k / a->C);
      cudaMemcpyAsync(a->ckx + s * 3 * a->P.N, a->x, n3, cudaMemcpyDeviceToDevice, st);
      cudaMemcpyAsync(a->ckv + s * 3 * a->P.N, a->v, n3, cudaMemcpyDeviceToDevice, st);
    }
    if (cudaGraphLaunch(step, st) != cudaSuccess) grc = MD_ECUDA;
  }
  if (step) cudaGraphExecDestroy(step);
  if (grc != MD_OK) return adj_fail(MD_ECUDA, "forward step launch failed");
  if (a->K == 0) {
    cudaMemcpyAsync(a->ckx, a->x, n3, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(a->ckv, a->v, n3, cudaMemcpyDeviceToDevice, st);
  }
  double acc[2];
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(acc, a->acc, sizeof(acc), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return adj_fail(MD_ECUDA, "forward run failed");
  a->obs[0] = acc[0] / (double)(a->K + 1);
  a->obs[1] = acc[1] / (double)(a->K + 1);
  if (!std::isfinite(a->obs[0]) || !std::isfinite(a->obs[1])) return adj_fail(MD_EUNSTABLE, "non-finite observable");
  a->have_forward = true;
  if (obs) { obs[0] = a->obs[0]; obs[1] = a->obs[1]; }
  return MD_OK;
}

extern "C" int md_adj_backward(md_adj* a, const double weight[2], double grad[5]) {
  if (!a || !weight || !grad) return adj_fail(MD_EINVAL, "null argument");
  if (!a->have_forward) return adj_fail(MD_EINVAL, "md_adj_backward needs md_adj_forward at the current parameters");
  const AdjDev& P = a->P;
  const size_t n3 = sizeof(double) * 3 * (size_t)P.N;
  const size_t stride = 3 * (size_t)P.N;
  cudaStream_t st = a->st;
  const int nb = (P.N + 255) / 256;
  const double w = 1.0 / (double)(a->K + 1);
  const double wu = w * weight[0], wr = w * weight[1];
  if (cudaMemsetAsync(a->alpha, 0, n3, st) != cudaSuccess || cudaMemsetAsync(a->beta, 0, n3, st) != cudaSuccess ||
      cudaMemsetAsync(a->acc, 0, sizeof(double) * kAccN, st) != cudaSuccess)
    return adj_fail(MD_ECUDA, "clearing the adjoint state failed");
  // graphs: a recomputed forward step, and a reverse step with c_k = dt at
  // positions copied to xk (the steps k = K and k = 0 are launched directly)
  cudaGraphExec_t rec_step = nullptr, rev_step = nullptr;
  const bool have_graphs =
      capture(a, &rec_step, [&]() {
        k_adj_kick_drift<<<nb, 256, 0, st>>>(a->x, a->v, a->gv, P, a->dt, nullptr);
        const int rc = evaluate(a, a->x, nullptr, 0.0, 2, 0.0);
        k_adj_kick<<<nb, 256, 0, st>>>(a->v, a->gv, P, a->dt);
        return rc;
      }) &&
      capture(a, &rev_step, [&]() {
        const int rc = evaluate(a, a->xk, a->beta, a->dt, 1, wu);
        k_adj_update<<<nb, 256, 0, st>>>(a->xk, a->gv, a->gt, P, wu, wr, a->dt, 1, a->alpha, a->beta);
        return rc;
      });
  if (!have_graphs) {
    if (rec_step) cudaGraphExecDestroy(rec_step);
    if (rev_step) cudaGraphExecDestroy(rev_step);
    return adj_fail(MD_ECUDA, "capturing the adjoint steps failed");
  }
  struct GraphGuard {
    cudaGraphExec_t a, b;
    ~GraphGuard() { cudaGraphExecDestroy(a); cudaGraphExecDestroy(b); }
  } guard{rec_step, rev_step};
  for (int s = a->S - 1; s >= 0; --s) {
    const int k0 = s * a->C, k1 = (k0 + a->C < a->K) ? k0 + a->C : a->K;
    // recompute the segment's positions from its checkpoint
    cudaMemcpyAsync(a->x, a->ckx + s * stride, n3, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(a->v, a->ckv + s * stride, n3, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(a->seg, a->x, n3, cudaMemcpyDeviceToDevice, st);
    if (k1 > k0 && evaluate(a, a->x, nullptr, 0.0, 2, 0.0) != MD_OK)
      return adj_fail(MD_ECUDA, "force evaluation failed");
    for (int k = k0; k < k1; ++k) {
      if (k + 1 < k1) {
        if (cudaGraphLaunch(rec_step, st) != cudaSuccess) return adj_fail(MD_ECUDA, "recompute step launch failed");
        cudaMemcpyAsync(a->seg + (size_t)(k - k0 + 1) * stride, a->x, n3, cudaMemcpyDeviceToDevice, st);
      } else {
        k_adj_kick_drift<<<nb, 256, 0, st>>>(a->x, a->v, a->gv, P, a->dt, a->seg + (size_t)(k - k0 + 1) * stride);
      }
    }
    // reverse steps k1 .. k0 + 1 (and 0 in the first segment)
    const int k_lo = s == 0 ? 0 : k0 + 1;
    for (int k = k1; k >= k_lo; --k) {
      const double* xk = a->seg + (size_t)(k - k0) * stride;
      if (k != a->K && k != 0) {
        cudaMemcpyAsync(a->xk, xk, n3, cudaMemcpyDeviceToDevice, st);
        if (cudaGraphLaunch(rev_step, st) != cudaSuccess) return adj_fail(MD_ECUDA, "reverse step launch failed");
        continue;
      }
      const double ck = k == a->K ? 0.0 : 0.5 * a->dt;
      if (evaluate(a, xk, a->beta, ck, 1, wu) != MD_OK) return adj_fail(MD_ECUDA, "tangent evaluation failed");
      k_adj_update<<<nb, 256, 0, st>>>(xk, a->gv, a->gt, P, wu, wr, a->dt, k >= 1 ? 1 : 0, a->alpha, a->beta);
    }
  }
  double acc[kAccN];
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(acc, a->acc, sizeof(acc), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return adj_fail(MD_ECUDA, "reverse run failed");
  chain_rule(a, acc, grad);
  for (int k = 0; k < 5; ++k)
    if (!std::isfinite(grad[k])) return adj_fail(MD_EUNSTABLE, "non-finite gradient");
  return MD_OK;
}

extern "C" int md_adj_tangent(md_adj* a, const double* pos, const double* dir, double* grad_u, double* hvp,
                              double dtheta[10]) {
  if (!a || !pos || !dir) return adj_fail(MD_EINVAL, "null argument");
  const AdjDev& P = a->P;
  const size_t n3 = sizeof(double) * 3 * (size_t)P.N;
  cudaStream_t st = a->st;
  // the direction enters as cu M^-1 beta; store beta = M dir so that u = dir
  double* hb = (double*)std::malloc(n3);
  if (!hb) return adj_fail(MD_ENOMEM, "host allocation failed");
  for (int i = 0; i < P.N; ++i) {
    const int si = i % P.sites;
    const double m = 1.0 / P.inv_mass[(si == 0 || si == P.sites - 1) ? 1 : 0];
    for (int q = 0; q < 3; ++q) hb[3 * i + q] = m * dir[3 * i + q];
  }
  int rc = MD_OK;
  if (cudaMemcpyAsync(a->x, pos, n3, cudaMemcpyDefault, st) != cudaSuccess ||
      cudaMemcpyAsync(a->beta, hb, n3, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemsetAsync(a->acc, 0, sizeof(double) * kAccN, st) != cudaSuccess)
    rc = MD_ECUDA;
  // mode 1 with weight 1 gives dU/dtheta - d(grad U . u)/dtheta; mode 2 the totals alone
  if (rc == MD_OK) rc = evaluate(a, a->x, a->beta, 1.0, 2, 0.0);
  double tot[kRec];
  if (rc == MD_OK) {
    if ((grad_u && cudaMemcpyAsync(grad_u, a->gv, n3, cudaMemcpyDefault, st) != cudaSuccess) ||
        (hvp && cudaMemcpyAsync(hvp, a->gt, n3, cudaMemcpyDefault, st) != cudaSuccess) ||
        cudaMemcpyAsync(tot, a->totals, sizeof(tot), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      rc = MD_ECUDA;
  }
  std::free(hb);
  if (rc != MD_OK) return adj_fail(rc, "tangent evaluation failed");
  if (dtheta) {
    double acc[kAccN] = {0};
    // value part: dU/dtheta
    for (int t = 0; t < 3; ++t) { acc[kAccC12 + t] = tot[kA + 4 * t]; acc[kAccC6 + t] = -tot[kA + 4 * t + 2]; }
    acc[kAccKphi] = tot[kD];
    chain_rule(a, acc, dtheta);
    // tangent part: d(grad U . u)/dtheta
    for (int t = 0; t < 3; ++t) { acc[kAccC12 + t] = tot[kA + 4 * t + 1]; acc[kAccC6 + t] = -tot[kA + 4 * t + 3]; }
    acc[kAccKphi] = tot[kD + 1];
    chain_rule(a, acc, dtheta + 5);
  }
  return MD_OK;
}

extern "C" int md_adj_energy(md_adj* a, double out[6]) {
  // totals of the last evaluation: shifted LJ, bond, angle, dihedral, sum over chains of R_ee^2, U
  if (!a || !out) return adj_fail(MD_EINVAL, "null argument");
  double tot[kRec];
  if (cudaMemcpyAsync(tot, a->totals, sizeof(tot), cudaMemcpyDeviceToHost, a->st) != cudaSuccess ||
      cudaStreamSynchronize(a->st) != cudaSuccess)
    return adj_fail(MD_ECUDA, "copy of the totals failed");
  out[0] = tot[kElj]; out[1] = tot[kEb]; out[2] = tot[kEa]; out[3] = tot[kEd]; out[4] = tot[kR2];
  out[5] = tot[kElj] + tot[kEb] + tot[kEa] + tot[kEd];
  return MD_OK;
}

extern "C" void md_adj_destroy(md_adj* a) {
  if (!a) return;
  cudaStreamSynchronize(a->st);
  cudaFree(a->mem);
  if (a->own_stream) cudaStreamDestroy(a->st);
  delete a;
}
