// k_observe.cu -- structural observables of Sec. 5 on the GPU: the radial
// distribution function of non-bonded site pairs and the end-to-end vector
// autocorrelation function (Fig. 8).
//
// RDF: a cell's atoms pair with the later atoms of the cell and with every
// atom of the 13 forward cells of a half shell, so each pair within one cell
// side is met once.  The distance is the plain definition in FP64 with every
// operation explicitly rounded (d = x_j - x_i, d -= L rint(d / L),
// r = sqrt(dx^2 + dy^2 + dz^2), summed left to right), and the bin is the k
// with edges[k] <= r < edges[k + 1] (the last bin closed), so the integer
// counts equal those of the FP64 definition on the same positions.  Counts
// are summed in shared memory and added to the per-replica histogram with
// integer atomics (order-free).
//
// ACF: samples of the chains' end-to-end vectors go to a ring of max_lag + 1
// slots; each new sample s adds, for every lag tau <= min(s, max_lag) and
// every replica, sum_c R_c(s) . R_c(s - tau) to acc[r][tau], one block per
// (replica, tau) with a fixed-order reduction over the replica's chains.
// After n samples acc[r][tau] = sum_{t < n - tau} sum_c R_c(t + tau) . R_c(t).
#include <cmath>
#include <type_traits>

#include "md_kernels.cuh"

namespace mdg {

// The FP64 pipe of this GPU issues about 2 operations per clock and SM, and
// the definition costs some 60 of them per candidate pair (three divisions,
// a square root).  So a pair's bin is taken from the FP32 cell-unit
// positions of the fresh bins wherever that cannot differ: the FP32 distance
// is within kRdfMargin cell sides of the FP64 one, and a pair whose FP32
// distance lies further than that inside a bin's edges (or beyond the last
// one) has that bin by the definition too.  The few others (0.1% of the
// pairs in range at 200 bins) are evaluated by the definition.
//
// A lane holds one atom j of the 14 cells, moved to the home cell's frame,
// and a warp walks the home atoms in shared memory, two at a time in packed
// FP32.  40% of the candidates lie too far from the home cell for any of its
// atoms and are left out before.  Of the rest 15% are in range, so nearly
// every round of 32 holds one: they are queued and binned 32 at a time.  A block takes a cell, or
// above 4 times the resident blocks a run of consecutive ones, so that a
// histogram is flushed once per run.  Bound: instruction issue.  150k sites,
// r_max 1.0 nm, 200 bins: 9,824 us (FP64 for every candidate) -> 251 (binned
// as met, runs of one or two cells) -> 175 (all candidates) -> 161.
constexpr int kRdfThreads = 128;
constexpr int kRdfStage = 128;       // home atoms staged at a time
constexpr int kRdfBlocks = kSMs * 16;
constexpr int kRdfQueue = 256;       // a ring: at most 31 + 64 pairs wait
constexpr int kRdfCand = 128;        // a ring: at most 31 + 32 candidates wait, and none is written over as it is read
constexpr int kRdfSlotBits = 26;     // atoms < 2^26; six bits of the home atom above, its seventh with r^2
// FP32 cell units: each position is rounded by at most 2^-25 (FP32 master:
// 2^-24.6), the offset and the difference add 2^-24 each, so a component is
// off by at most 1.9e-7 and r <= 1 by 3.3e-7; r^2, rsqrt.approx and the scaling by h add 5e-7
constexpr float kRdfMargin = 1.0e-6f;

__device__ __forceinline__ int rdf_find_rep(const RepDev* reps, int n_reps, int c) {
  int lo = 0, hi = n_reps - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (reps[mid].cell_base <= c) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// bin of the pair (i, j) by the FP64 definition, or -1
template <class T>
__device__ __noinline__ int rdf_exact_bin(const T* __restrict__ x, int N, int i, int j, double L,
                                          const double* __restrict__ edges, int n_bins, double norm) {
  double d2 = 0.0;
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    double d = __dsub_rn((double)x[ax * N + j], (double)x[ax * N + i]);
    d = __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
    d2 = ax == 0 ? __dmul_rn(d, d) : __dadd_rn(d2, __dmul_rn(d, d));
  }
  const double rr = __dsqrt_rn(d2);
  if (!(rr <= edges[n_bins]) || rr < edges[0]) return -1;
  int k = (int)((rr - edges[0]) * norm);
  k = k < 0 ? 0 : (k > n_bins - 1 ? n_bins - 1 : k);
  if (rr < edges[k]) --k;
  else if (k < n_bins - 1 && rr >= edges[k + 1]) ++k;
  return k;
}

template <class T>
__global__ void __launch_bounds__(kRdfThreads) k_rdf(const T* __restrict__ x, int N, const int* __restrict__ cell_start,
                                                     const int* __restrict__ perm, const float4* __restrict__ pos,
                                                     const int* __restrict__ tag, const RepDev* __restrict__ reps,
                                                     int n_reps, int C, const double* __restrict__ edges,
                                                     const float2* __restrict__ inner, int n_bins, double norm,
                                                     unsigned long long* __restrict__ counts) {
  extern __shared__ unsigned int hist[];
  __shared__ __align__(8) float hx[kRdfStage], hy[kRdfStage], hz[kRdfStage];   // home atoms: cell units
  __shared__ __align__(8) int ht[kRdfStage];                                   // and chain/site tags
  __shared__ uint2 queue[kRdfThreads / 32][kRdfQueue];
  __shared__ unsigned cand[kRdfThreads / 32][kRdfCand];
  __shared__ int s_start[14], s_pre[15];
  __shared__ float s_off[14][3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint2* qw = queue[warp];
  unsigned* cw = cand[warp];
  const unsigned lt = (1u << lane) - 1u;
  const int c0 = (int)((long long)C * blockIdx.x / gridDim.x), c1 = (int)((long long)C * (blockIdx.x + 1) / gridDim.x);
  if (c0 >= c1) return;
  for (int k = threadIdx.x; k < n_bins; k += kRdfThreads) hist[k] = 0u;
  int r = rdf_find_rep(reps, n_reps, c0);
  const float e0 = (float)edges[0], fnorm = (float)norm, r_top = (float)edges[n_bins];
  for (int c = c0; c < c1; ++c) {
    __syncthreads();   // the previous cell's tables are no longer read
    if (r + 1 < n_reps && reps[r + 1].cell_base <= c) {   // the next replica begins: its histogram is another
      for (int k = threadIdx.x; k < n_bins; k += kRdfThreads) {
        if (hist[k]) atomicAdd(counts + (size_t)r * n_bins + k, (unsigned long long)hist[k]);
        hist[k] = 0u;
      }
      ++r;
    }
    const RepDev& R = reps[r];
    const int M = R.M, b = cell_start[c], n = cell_start[c + 1] - b;
    if (warp == 0) {
      int len = 0;
      if (lane < 14) {   // the cell itself, then its 13 forward neighbours
        int ox = 0, oy = 0, oz = 0;
        if (lane > 0) {
          const int q = lane - 1;           // 9 cells of the z + 1 layer, 3 of y + 1, then x + 1
          if (q < 9) { oz = 1; oy = q / 3 - 1; ox = q % 3 - 1; }
          else if (q < 12) { oy = 1; ox = q - 10; }
          else { ox = 1; }
        }
        const int lc = c - R.cell_base;
        const int cx = lc % M, cy = (lc / M) % M, cz = lc / (M * M);
        const int nc = R.cell_base + (((cz + oz + M) % M) * M + ((cy + oy + M) % M)) * M + ((cx + ox + M) % M);
        s_start[lane] = cell_start[nc];
        len = cell_start[nc + 1] - cell_start[nc];
        s_off[lane][0] = (float)ox; s_off[lane][1] = (float)oy; s_off[lane][2] = (float)oz;
      }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, len, o);
        if (lane >= o) len += v;
      }
      if (lane == 0) s_pre[0] = 0;
      if (lane < 14) s_pre[lane + 1] = len;
    }
    const float hf = R.hf, Mf = R.Mf;
    // beyond this squared FP32 distance (cell units) a pair is out of range by the definition
    const float rt = r_top / hf + 2.f * kRdfMargin;
    const float far2 = rt * rt;
    const float low = e0 - 4.f * kRdfMargin * hf;   // below this one, out of range as well
    const bool fold = M == 3;   // two images of a pair can both be near a cell side away
    // half the home cell's side and the atoms' rounding; with folded images every candidate is near
    const float box = fold ? 4.f : 0.5f + kRdfMargin;
    for (int i0 = 0; i0 < n; i0 += kRdfStage) {
      const int ni = min(kRdfStage, n - i0);
      __syncthreads();
      for (int k = threadIdx.x; k < ni; k += kRdfThreads) {
        const float4 p = pos[b + i0 + k];
        hx[k] = p.x; hy[k] = p.y; hz[k] = p.z;
        ht[k] = tag[b + i0 + k] & (int)kTagMask;
      }
      __syncthreads();
      // bin of one queued pair
      auto take = [&](uint2 e) {
        const int k = (int)((e.x >> 31) << 6 | e.y >> kRdfSlotBits), sj = (int)(e.y & ((1u << kRdfSlotBits) - 1u));
        const float r2 = __uint_as_float(e.x & 0x7fffffffu);
        const float rr = r2 * rsqrtf(r2) * hf;
        if (rr < low) return;
        int g = (int)((rr - e0) * fnorm);
        g = g < 0 ? 0 : (g > n_bins - 1 ? n_bins - 1 : g);
        const float2 in = __ldg(inner + g);
        if (!(rr >= in.x && rr < in.y))
          g = rdf_exact_bin<T>(x, N, perm[b + i0 + k], perm[sj], R.L, edges, n_bins, norm);
        if (g >= 0) atomicAdd(hist + g, 1u);
      };
      int qn = 0, head = 0;   // waiting pairs: ring places head .. head + qn - 1
      // the home atoms against candidate e (tile slot | cell << kRdfSlotBits) of each lane
      auto walk = [&](unsigned e, bool on) {
        int sj = b, tj = 0, last = 0;   // home atoms i0 .. i0 + last - 1 pair with j
        float4 pj = make_float4(0.f, 0.f, 0.f, 0.f);
        if (on) {
          const int o = (int)(e >> kRdfSlotBits);
          sj = (int)(e & ((1u << kRdfSlotBits) - 1u));
          pj = pos[sj];
          pj.x += s_off[o][0]; pj.y += s_off[o][1]; pj.z += s_off[o][2];
          tj = tag[sj] & (int)kTagMask;
          last = o == 0 ? min(ni, sj - b - i0) : ni;   // the cell itself: each pair once, i before j
        }
        const float2 jx = make_float2(pj.x, pj.x), jy = make_float2(pj.y, pj.y), jz = make_float2(pj.z, pj.z);
        const float2 m1 = make_float2(-1.f, -1.f);
        for (int k = 0; k < ni; k += 2) {   // a place past the last home atom is not below `last`
          float2 dx = __ffma2_rn(*reinterpret_cast<const float2*>(hx + k), m1, jx),
                 dy = __ffma2_rn(*reinterpret_cast<const float2*>(hy + k), m1, jy),
                 dz = __ffma2_rn(*reinterpret_cast<const float2*>(hz + k), m1, jz);
          const int2 t = *reinterpret_cast<const int2*>(ht + k);
          if (fold) {
            dx.x -= Mf * rintf(dx.x / Mf); dy.x -= Mf * rintf(dy.x / Mf); dz.x -= Mf * rintf(dz.x / Mf);
            dx.y -= Mf * rintf(dx.y / Mf); dy.y -= Mf * rintf(dy.y / Mf); dz.y -= Mf * rintf(dz.y / Mf);
          }
          const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
          // |i - j| <= 2 within one chain: 1-2 and 1-3 neighbours (Sec. 3.1)
          const bool pass0 = k < last && r2.x <= far2 && (unsigned)(t.x - tj + 2) > 4u;
          const bool pass1 = k + 1 < last && r2.y <= far2 && (unsigned)(t.y - tj + 2) > 4u;
          const unsigned b0 = __ballot_sync(0xffffffffu, pass0), b1 = __ballot_sync(0xffffffffu, pass1);
          const int at = head + qn + __popc(b0 & lt) + __popc(b1 & lt);
          const unsigned hi = (unsigned)(k >> 6) << 31, lo = (unsigned)sj | (unsigned)(k & 63) << kRdfSlotBits;
          if (pass0) qw[at & (kRdfQueue - 1)] = make_uint2(__float_as_uint(r2.x) | hi, lo);
          if (pass1)
            qw[(at + (pass0 ? 1 : 0)) & (kRdfQueue - 1)] =
                make_uint2(__float_as_uint(r2.y) | hi, lo + (1u << kRdfSlotBits));   // k is even
          qn += __popc(b0) + __popc(b1);
          // one barrier a round: the 64 places that are taken lie before head,
          // and the next round writes at most 94 past it (256 in the ring)
          __syncwarp();
          while (qn >= 32) {
            take(qw[(head + lane) & (kRdfQueue - 1)]);
            head += 32;
            qn -= 32;
          }
        }
      };
      // candidates that no home atom can be in range of (further than that from
      // the cell) are left out: the others wait until 32 can be taken together
      const int total = s_pre[14];
      int o = 0, cn = 0, chead = 0;
      for (int q0 = 32 * warp;; q0 += kRdfThreads) {
        const bool more = q0 < total;
        if (more) {
          const int q = q0 + lane;
          bool near = false;
          unsigned e = 0u;
          if (q < total) {
            while (q >= s_pre[o + 1]) ++o;
            const int sj = s_start[o] + (q - s_pre[o]);
            const float4 pj = pos[sj];
            const float bx = fmaxf(fabsf(pj.x + s_off[o][0]) - box, 0.f), by = fmaxf(fabsf(pj.y + s_off[o][1]) - box, 0.f),
                        bz = fmaxf(fabsf(pj.z + s_off[o][2]) - box, 0.f);
            near = bx * bx + by * by + bz * bz <= far2;
            e = (unsigned)sj | (unsigned)o << kRdfSlotBits;
          }
          const unsigned m = __ballot_sync(0xffffffffu, near);
          if (near) cw[(chead + cn + __popc(m & lt)) & (kRdfCand - 1)] = e;
          cn += __popc(m);
          __syncwarp();
        }
        while (cn >= 32 || (!more && cn > 0)) {
          walk(cw[(chead + lane) & (kRdfCand - 1)], lane < cn);
          const int n = min(cn, 32);
          chead += n;
          cn -= n;
        }
        if (!more) break;
      }
      __syncwarp();
      if (lane < qn) take(qw[(head + lane) & (kRdfQueue - 1)]);
      __syncwarp();
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < n_bins; k += kRdfThreads)
    if (hist[k]) atomicAdd(counts + (size_t)r * n_bins + k, (unsigned long long)hist[k]);
}

// the part of each bin further than the FP32 distance's error from its edges
// (h_max: the largest cell side), edges rounded outward
void rdf_inner_edges(const double* edges, int n_bins, double h_max, float2* inner) {
  const double m = (double)kRdfMargin * h_max;
  for (int k = 0; k < n_bins; ++k)
    inner[k] = make_float2(std::nextafterf((float)(edges[k] + m), INFINITY),
                           std::nextafterf((float)(edges[k + 1] - m), -INFINITY));
}

void launch_rdf(bool mixed, const void* x, int N, const int* cell_start, const int* perm, const float4* pos,
                const int* tag, const RepDev* reps, int n_reps, int C, const double* edges, const float2* inner,
                int n_bins, double norm, unsigned long long* counts, cudaStream_t st) {
  if (C <= 0) return;
  const size_t sm = (size_t)n_bins * sizeof(unsigned int);
  const int grid = C < 4 * kRdfBlocks ? C : kRdfBlocks;
  // The histogram, queues and staged atoms may exceed 48 KB.  The opt-in is the
  // kernel's, not the launch's, so it is always the one for the most bins: a
  // smaller one would take it from another thread's call between that one's
  // opt-in and its launch.
  if (sm > 36000) {
    constexpr int most = kRdfMaxBins * (int)sizeof(unsigned int);
    cudaFuncSetAttribute(k_rdf<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    cudaFuncSetAttribute(k_rdf<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  }
  if (mixed)
    k_rdf<double><<<grid, kRdfThreads, sm, st>>>((const double*)x, N, cell_start, perm, pos, tag, reps, n_reps, C,
                                                 edges, inner, n_bins, norm, counts);
  else
    k_rdf<float><<<grid, kRdfThreads, sm, st>>>((const float*)x, N, cell_start, perm, pos, tag, reps, n_reps, C,
                                                edges, inner, n_bins, norm, counts);
}

// ------------------------------------------------------------------ ACF
constexpr int kAcfThreads = 256;

// acc[r * (max_lag + 1) + tau] += sum over replica r's chains of
// R(s) . R(s - tau); ring slot of sample t is t % (max_lag + 1).  Block
// (tau, r); thread k adds chains k, k + 256, ... in order, then a fixed tree.
__global__ void __launch_bounds__(kAcfThreads) k_acf_add(const double* __restrict__ ring, int n_chains_total,
                                                         const RepDev* __restrict__ reps, long long s, int max_lag,
                                                         double* __restrict__ acc) {
  const int tau = blockIdx.x, r = blockIdx.y;
  if (tau > s) return;
  const RepDev& R = reps[r];
  const int slots = max_lag + 1;
  const double* a = ring + (size_t)(s % slots) * 3 * n_chains_total;
  const double* b = ring + (size_t)((s - tau) % slots) * 3 * n_chains_total;
  double v = 0.0;
  for (int c = R.chain_off + threadIdx.x; c < R.chain_off + R.n_chains; c += kAcfThreads)
    v += a[3 * c] * b[3 * c] + a[3 * c + 1] * b[3 * c + 1] + a[3 * c + 2] * b[3 * c + 2];
  __shared__ double red[kAcfThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kAcfThreads / 32; ++w) t += red[w];
    acc[(size_t)r * slots + tau] += t;
  }
}

void launch_acf_add(const double* ring, int n_chains_total, const RepDev* reps, int n_reps, long long s, int max_lag,
                    double* acc, cudaStream_t st) {
  const int lags = (int)(s < max_lag ? s : max_lag) + 1;
  k_acf_add<<<dim3(lags, n_reps), kAcfThreads, 0, st>>>(ring, n_chains_total, reps, s, max_lag, acc);
}

}  // namespace mdg
