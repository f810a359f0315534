// bonded.cuh -- Dreiding II bonded terms of a linear chain (Eqs. 4-6,
// Sec. 3.3), shared by the force kernel (k_force.cu) and the fused step kernel
// (k_step.cu), so that both give the same force bits.
#pragma once
#include "md_kernels.cuh"

namespace mdg {

// FP32 force -> int64 fixed point (2^-32 kJ/mol/nm); each part below 2^18
__device__ __forceinline__ long long to_fix(float f, unsigned* flags) {
  if (!(fabsf(f) < 262144.0f)) { atomicOr(flags, kFlagFixOverflow); return 0; }
  return fix_round_int(f);   // = __float2ll_rn(f * 2^32), on the integer pipe
}

struct f3 { float x, y, z; };
__device__ __forceinline__ f3 mk(float x, float y, float z) { return {x, y, z}; }
__device__ __forceinline__ f3 operator+(f3 a, f3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ f3 operator-(f3 a, f3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ f3 operator-(f3 a) { return {-a.x, -a.y, -a.z}; }
__device__ __forceinline__ f3 operator*(float s, f3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ float dot(f3 a, f3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ f3 cross(f3 a, f3 b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// bond vector x_{m+1} - x_m under the minimum image (FP64 master); |d| > L/2
// is tested on the bit patterns (integer pipe), which order like the values
__device__ __forceinline__ double bond_diff(double a, double b, double L, double hL) {
  double d = b - a;
  const long long bd = __double_as_longlong(d);
  if ((bd & 0x7fffffffffffffffll) > __double_as_longlong(hL)) d = bd < 0 ? d + L : d - L;
  return d;
}

// |b|^2 - b0^2 for an exact FP32 vector b: each square is split into its
// rounded value and exact error (FMA), the rounded parts are summed with
// error-free two-sums, and b0^2 = c_hi + c_lo is subtracted from the
// leading part, where the two nearly cancel without rounding.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ float sq_minus(f3 b, float c_hi, float c_lo) {
  const float px = b.x * b.x, py = b.y * b.y, pz = b.z * b.z;
  const float ex = fmaf(b.x, b.x, -px), ey = fmaf(b.y, b.y, -py), ez = fmaf(b.z, b.z, -pz);
  float s1, e1, s2, e2;
  two_sum(px, py, s1, e1);
  two_sum(s1, pz, s2, e2);
  return (s2 - c_hi) + ((e1 + e2) + (ex + ey + ez) - c_lo);
}
// FP32 master: the difference of two nearby floats is exact; across a face the
// partner is first moved by L (exact when it lies near the face, L being an
// FP32 number), so the result is again the exact difference.
__device__ __forceinline__ float bond_comp(float a, float b, float L, float hL) {
  float d = b - a;
  if (d > hL) d = (b - L) - a; else if (d < -hL) d = b - (a - L);
  return d;
}

__device__ __forceinline__ void add_vir(float (&W)[6], f3 r, f3 f) {
  W[0] += r.x * f.x; W[1] += r.y * f.y; W[2] += r.z * f.z;
  W[3] += r.x * f.y; W[4] += r.x * f.z; W[5] += r.y * f.z;
}

// int64 fixed point (2^-32 kJ/mol/nm) -> FP32 on the 32-bit pipes: the high
// word (|hi| < 2^24, exact) plus the low word scaled by 2^-32
__device__ __forceinline__ float fix_to_float(long long q) {
  const int hi = (int)(q >> 32);
  const unsigned lo = (unsigned)q;
  return fmaf((float)lo, 2.3283064365386963e-10f, (float)hi);
}

// The terms that start at a chain's site sm (S sites), from the bond vectors
// bv[q], bv[q + 1], bv[q + 2] and r^2 - b0^2 of the first bond, bD[q]: the
// forces fb on the bond's first atom, fa and fc on the angle's ends, f1, f2
// and f3v on the dihedral's first three atoms.  ENERGY and own: also the
// energies and the virial.
template <bool ENERGY>
__device__ __forceinline__ void chain_terms(const ForceParams& fp, int sm, int S, const f3* __restrict__ bv,
                                            const float* __restrict__ bD, int q, bool own, f3& fb, f3& fa, f3& fc,
                                            f3& f1, f3& f2, f3& f3v, float& Eb, float& Ea, float& Ed,
                                            float (&W)[6]) {
  if (sm <= S - 2) {               // bond (m, m+1), Eq. (4)
    const f3 b = bv[q];
    const float r = sqrtf(dot(b, b));
    const float dr = bD[q] / (r + fp.b0);   // r - b0 without cancellation
    const float g = fp.kb * dr / r;
    fb = g * b;                    // force on atom m
    if (ENERGY && own) { Eb += 0.5f * fp.kb * dr * dr; add_vir(W, b, -fb); }
  }
  if (sm <= S - 3) {               // angle (m, m+1, m+2), vertex m+1, Eq. (5)
    const f3 u = -bv[q], w = bv[q + 1];
    const float lu = sqrtf(dot(u, u)), lw = sqrtf(dot(w, w));
    const f3 cr = cross(u, w);
    const float sn = sqrtf(dot(cr, cr)), cs = dot(u, w);
    const float th = atan2f(sn, cs);
    const float dth = th - fp.theta0;
    const float inv = 1.0f / (lu * lw);
    const float sin_t = sn * inv, cos_t = cs * inv;
    if (sin_t > 1e-6f) {
      const float g = fp.ka * dth / sin_t;
      const f3 uh = (1.0f / lu) * u, wh = (1.0f / lw) * w;
      fa = (g / lu) * (wh - cos_t * uh);
      fc = (g / lw) * (uh - cos_t * wh);
    }
    if (ENERGY && own) { Ea += 0.5f * fp.ka * dth * dth; add_vir(W, u, fa); add_vir(W, w, fc); }
  }
  if (sm <= S - 4) {               // dihedral (m .. m+3), Eq. (6), IUPAC phi
    const f3 b1 = bv[q], b2 = bv[q + 1], b3 = bv[q + 2];
    const f3 mm = cross(b1, b2), nn = cross(b2, b3);
    const float lb2 = sqrtf(dot(b2, b2)), m2 = dot(mm, mm), n2 = dot(nn, nn);
    const float phi = atan2f(lb2 * dot(b1, nn), dot(mm, nn));
    const float arg = (float)fp.n_mult * phi - fp.phis;
    float sa, ca;
    sincosf(arg, &sa, &ca);
    if (m2 > 1e-24f && n2 > 1e-24f) {
      const float dEdphi = -fp.kphi * (float)fp.n_mult * sa;
      const float cam = -lb2 / m2, cdn = lb2 / n2;
      const float cbm = lb2 / m2 + dot(b1, b2) / (lb2 * m2), cbn = dot(b2, b3) / (lb2 * n2);
      const f3 ga = cam * mm, gd = cdn * nn, gb = cbm * mm + cbn * nn;
      const f3 gc = -(ga + gb + gd);
      f1 = -dEdphi * ga; f2 = -dEdphi * gb; f3v = -dEdphi * gc;
      if (ENERGY && own) {
        const f3 f4 = -(f1 + f2 + f3v);
        add_vir(W, b1, f2); add_vir(W, b1 + b2, f3v); add_vir(W, b1 + b2 + b3, f4);
      }
    }
    if (ENERGY && own) Ed += fp.kphi * (1.0f + ca);
  }
}

// The bonded force on an atom from the terms around it, in a fixed order
// (q: the atom's place in the term arrays; three places before it must hold
// its predecessors' terms or zeros).
__device__ __forceinline__ f3 chain_force(const f3* fbd, const f3* fan_a, const f3* fan_c, const f3* fdi1,
                                          const f3* fdi2, const f3* fdi3, int q) {
  f3 F = fbd[q] - fbd[q - 1];
  F = F + fan_a[q] - (fan_a[q - 1] + fan_c[q - 1]) + fan_c[q - 2];
  F = F + fdi1[q] + fdi2[q - 1] + fdi3[q - 2] - (fdi1[q - 3] + fdi2[q - 3] + fdi3[q - 3]);
  return F;
}

// bond vector x_{m+1} - x_m and r^2 - b0^2 of atom m of a chain
template <bool MIXED, class T>
__device__ __forceinline__ void bond_vector(const T (&a)[3], const T (&c)[3], const RepDev& R, const ForceParams& fp,
                                            f3& b, float& D) {
  if constexpr (MIXED) {
    const double dx = bond_diff(a[0], c[0], R.L, R.half_L);
    const double dy = bond_diff(a[1], c[1], R.L, R.half_L);
    const double dz = bond_diff(a[2], c[2], R.L, R.half_L);
    b = mk(d2f_rn_int(dx), d2f_rn_int(dy), d2f_rn_int(dz));
    D = d2f_rn_int(fma(dx, dx, fma(dy, dy, fma(dz, dz, -fp.b0sq))));
  } else {
    b.x = bond_comp(a[0], c[0], R.Lf, R.half_Lf);
    b.y = bond_comp(a[1], c[1], R.Lf, R.half_Lf);
    b.z = bond_comp(a[2], c[2], R.Lf, R.half_Lf);
    D = sq_minus(b, fp.b0sq_hi, fp.b0sq_lo);
  }
}

// ---------------------------------------------------------------- general molecules
// The terms of a bond-graph topology, shared by the fused step kernel
// (k_step.cu) and k_bonded_generic (k_force.cu).  x holds the FP64 positions as
// three rows of N; add(i, f) adds f to the force of atom i.  The separations are
// minimum-image differences rounded to FP32, as in the chain kernels.

// FP32 separation x_b - x_a
__device__ __forceinline__ f3 sep_ab(const double* x, int N, int a, int b, const RepDev& R) {
  const double dx = bond_diff(x[a], x[b], R.L, R.half_L);
  const double dy = bond_diff(x[N + a], x[N + b], R.L, R.half_L);
  const double dz = bond_diff(x[2 * N + a], x[2 * N + b], R.L, R.half_L);
  return mk(d2f_rn_int(dx), d2f_rn_int(dy), d2f_rn_int(dz));
}

// bond (i, j), Eq. (4); |x_j - x_i|^2 - b0^2 in FP64
template <bool ENERGY, class Add>
__device__ __forceinline__ void bond_term(const double* x, int N, int i, int j, const RepDev& R, const ForceParams& fp,
                                          Add add, float& Eb, float (&W)[6]) {
  const f3 b = sep_ab(x, N, i, j, R);
  const double dx = bond_diff(x[i], x[j], R.L, R.half_L), dy = bond_diff(x[N + i], x[N + j], R.L, R.half_L);
  const double dz = bond_diff(x[2 * N + i], x[2 * N + j], R.L, R.half_L);
  const float D = d2f_rn_int(fma(dx, dx, fma(dy, dy, fma(dz, dz, -fp.b0sq))));
  const float r = sqrtf(dot(b, b));
  const float dr = D / (r + fp.b0);   // r - b0 without cancellation
  const f3 fb = (fp.kb * dr / r) * b; // force on a
  add(i, fb);
  add(j, -fb);
  if (ENERGY) { Eb += 0.5f * fp.kb * dr * dr; add_vir(W, b, -fb); }
}

// angle (i, jb, jc), vertex jb, Eq. (5)
template <bool ENERGY, class Add>
__device__ __forceinline__ void angle_term(const double* x, int N, int i, int jb, int jc, const RepDev& R,
                                           const ForceParams& fp, Add add, float& Ea, float (&W)[6]) {
  const f3 u = sep_ab(x, N, jb, i, R), w = sep_ab(x, N, jb, jc, R);
  const float lu = sqrtf(dot(u, u)), lw = sqrtf(dot(w, w));
  const f3 cr = cross(u, w);
  const float sn = sqrtf(dot(cr, cr)), cs = dot(u, w);
  const float th = atan2f(sn, cs);
  const float dth = th - fp.theta0;
  const float inv = 1.0f / (lu * lw);
  const float sin_t = sn * inv, cos_t = cs * inv;
  f3 fa = mk(0.f, 0.f, 0.f), fc = fa;
  if (sin_t > 1e-6f) {
    const float g = fp.ka * dth / sin_t;
    const f3 uh = (1.0f / lu) * u, wh = (1.0f / lw) * w;
    fa = (g / lu) * (wh - cos_t * uh);
    fc = (g / lw) * (uh - cos_t * wh);
  }
  add(i, fa);
  add(jc, fc);
  add(jb, -(fa + fc));
  if (ENERGY) { Ea += 0.5f * fp.ka * dth * dth; add_vir(W, u, fa); add_vir(W, w, fc); }
}

// dihedral (i, jb, jc, jd), Eq. (6), IUPAC phi
template <bool ENERGY, class Add>
__device__ __forceinline__ void dihedral_term(const double* x, int N, int i, int jb, int jc, int jd, const RepDev& R,
                                              const ForceParams& fp, Add add, float& Ed, float (&W)[6]) {
  const f3 b1 = sep_ab(x, N, i, jb, R), b2 = sep_ab(x, N, jb, jc, R), b3 = sep_ab(x, N, jc, jd, R);
  const f3 mm = cross(b1, b2), nn = cross(b2, b3);
  const float lb2 = sqrtf(dot(b2, b2)), m2 = dot(mm, mm), n2 = dot(nn, nn);
  const float phi = atan2f(lb2 * dot(b1, nn), dot(mm, nn));
  const float arg = (float)fp.n_mult * phi - fp.phis;
  float sa, ca;
  sincosf(arg, &sa, &ca);
  if (m2 > 1e-24f && n2 > 1e-24f) {
    const float dEdphi = -fp.kphi * (float)fp.n_mult * sa;
    const float cam = -lb2 / m2, cdn = lb2 / n2;
    const float cbm = lb2 / m2 + dot(b1, b2) / (lb2 * m2), cbn = dot(b2, b3) / (lb2 * n2);
    const f3 ga = cam * mm, gd = cdn * nn, gb = cbm * mm + cbn * nn;
    const f3 gc = -(ga + gb + gd);
    const f3 f1 = -dEdphi * ga, f2 = -dEdphi * gb, f3v = -dEdphi * gc;
    const f3 f4 = -(f1 + f2 + f3v);
    add(i, f1);
    add(jb, f2);
    add(jc, f3v);
    add(jd, f4);
    if (ENERGY) { add_vir(W, b1, f2); add_vir(W, b1 + b2, f3v); add_vir(W, b1 + b2 + b3, f4); }
  }
  if (ENERGY) Ed += fp.kphi * (1.0f + ca);
}

}  // namespace mdg
