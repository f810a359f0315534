// cell_order.cuh -- a stable order of n atoms by cell (ascending atom index
// inside each cell) for the callers whose cells may hold any number of atoms
// (md_bin_static, the adjoint): a radix sort of the atoms by cell id, up to 9
// bits a pass.  Its work does not depend on how the atoms are spread: one pass up to
// 512 cells, two up to 262,144, three up to 2^27.
//
// The counting kernel of the caller (one thread per atom, 256-thread blocks)
// calls order_count; launch_cell_order does the rest.  Buffers are in one run
// of ints that the caller clears before counting (order_clear_ints of them):
// count[C], then for odd and even passes the digit totals and the digit
// counts of every tile of consecutive atoms.
#pragma once
#include <type_traits>

#include "md_kernels.cuh"

namespace mdg {

constexpr int kMaxDigitBits = 9, kMaxDigits = 1 << kMaxDigitBits;

struct OrderBuf {
  int* count;                 // atoms of each cell
  int *tot[2], *hist[2];      // digit totals; [tile][digit] counts, then places
  int tile, n_tiles, passes;
  int bits;                   // of a digit: the id's bits spread evenly over the passes
};

// layout of the buffers for n atoms in C cells from base on
inline OrderBuf order_buffers(int* base, int n, long long C) {
  OrderBuf b;
  // 256 threads' items, one to eight each: 30 tiles at 7,500 atoms, 512 at 2^20
  b.tile = n <= 8192 ? 256 : n <= (1 << 17) ? 1024 : 2048;
  b.n_tiles = (n + b.tile - 1) / b.tile;
  int id_bits = 5;   // at least 32 digits (a warp of them)
  while (((long long)1 << id_bits) < C) ++id_bits;
  b.passes = (id_bits + kMaxDigitBits - 1) / kMaxDigitBits;
  b.bits = (id_bits + b.passes - 1) / b.passes;
  const int kDigits = 1 << b.bits;
  b.count = base;
  int* p = base + C;
  for (int k = 0; k < 2; ++k) {
    b.tot[k] = p;
    b.hist[k] = p + kDigits;
    p += (size_t)kDigits * (1 + b.n_tiles);
  }
  return b;
}
inline size_t order_ints(int n, long long C) {   // ints of the buffers
  const OrderBuf b = order_buffers(nullptr, n, C);
  return (size_t)C + 2 * ((size_t)1 << b.bits) * (1 + b.n_tiles);
}
// leading ints to clear before counting (a second pass's part only where there is one)
inline size_t order_clear_ints(const OrderBuf& b, long long C) {
  return (size_t)C + (size_t)(b.passes > 1 ? 2 : 1) * ((size_t)1 << b.bits) * (1 + b.n_tiles);
}

// Count atom i (< n, or on = false) in cell c; every thread of a 256-thread
// block calls it, with the block's 256 consecutive atoms.
__device__ __forceinline__ void order_count(bool on, int c, int first_atom, const OrderBuf& b) {
  if (!on) return;
  atomicAdd(b.count + c, 1);
  atomicAdd(b.hist[0] + ((size_t)(first_atom / b.tile) << b.bits) + (c & ((1 << b.bits) - 1)), 1);
}

// totals of digits 32 q .. + 31 over the tiles, by a block of 1,024 threads
__device__ __forceinline__ void digit_totals(int q, int bits, const int* __restrict__ hist, int n_tiles,
                                             int* __restrict__ tot) {
  __shared__ int part[32][33];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  int s = 0;
#pragma unroll 8
  for (int t = g; t < n_tiles; t += 32) s += hist[((size_t)t << bits) + 32 * q + lane];
  part[g][lane] = s;
  __syncthreads();
  if (g == 0) {
    int v = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) v += part[k][lane];
    tot[32 * q + lane] = v;
  }
}

// Places of a pass: hist[tile][digit] becomes the first place of the tile's
// items of that digit.  Block q takes digits 32 q .. + 31 (a lane each); warp g
// takes a run of tiles.  Items of smaller digits: from the totals, or in the
// last pass from cell_start (the digit's first cell).
static __global__ void __launch_bounds__(1024) k_digit_places(const int* __restrict__ tot, const int* __restrict__ cell_start,
                                                       int C, int shift, int bits, int* __restrict__ hist,
                                                       int n_tiles) {
  __shared__ int part[32][33];
  __shared__ int before;
  wait_for_predecessor();
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, d = 32 * blockIdx.x + lane;
  const int per = (n_tiles + 31) / 32, t0 = min(g * per, n_tiles), t1 = min(t0 + per, n_tiles);
  int s = 0;
#pragma unroll 8
  for (int t = t0; t < t1; ++t) s += hist[((size_t)t << bits) + d];
  part[g][lane] = s;
  if (g == 0 && !cell_start) {
    int v = 0;
    for (int k = lane; k < 32 * (int)blockIdx.x; k += 32) v += tot[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) before = v;
  }
  __syncthreads();
  int run;
  if (cell_start) {
    run = cell_start[(int)min((long long)C, (long long)d << shift)];
  } else {
    const int own = tot[d];
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    run = before + incl - own;
  }
  for (int k = 0; k < g; ++k) run += part[k][lane];
#pragma unroll 4
  for (int t = t0; t < t1; ++t) {
    int* h = hist + ((size_t)t << bits) + d;
    const int v = *h;
    *h = run;
    run += v;
  }
}

static __global__ void __launch_bounds__(1024) k_digit_totals(int bits, const int* __restrict__ hist,
                                                              int n_tiles, int* __restrict__ tot) {
  digit_totals(blockIdx.x, bits, hist, n_tiles, tot);
}

struct EmitNothing {
  __device__ __forceinline__ void operator()(int, int) const {}
};

// One pass: a block moves a tile of items (ROUNDS per thread, in order) to the
// places of their digits.  A warp holds a contiguous run of the tile and ranks
// its items round by round with a match over the lanes, so equal digits keep
// their order.  OWN: the last pass of a sort of at most 32 tiles, whose blocks
// find their places from the raw counts (no k_digit_places).  next_hist: the digit
// counts of the next pass, by the place each item goes to.  emit(place, atom)
// is called for every item (the last pass: its cell-order slot).
template <int ROUNDS, bool OWN, class Emit>
__global__ void __launch_bounds__(256) k_digit_scatter(const int* __restrict__ cell_of, const int* __restrict__ in, int n,
                                                       const int* __restrict__ cell_start, int C, int shift,
                                                       int bits, const int* __restrict__ hist, int* __restrict__ out,
                                                       int* __restrict__ next_hist, const Emit emit) {
  __shared__ int cnt[8][kMaxDigits];
  const int kDigits = 1 << bits;
  wait_for_predecessor();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int kTile = 256 * ROUNDS;
  const int first = blockIdx.x * kTile + w * 32 * ROUNDS;
  int id[ROUNDS], key[ROUNDS], rank[ROUNDS];
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int p = first + 32 * r + lane;
    id[r] = p < n ? (in ? in[p] : p) : -1;
  }
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) key[r] = id[r] >= 0 ? cell_of[id[r]] : 0;
  for (int k = threadIdx.x; k < 8 * kDigits; k += 256) cnt[k >> bits][k & (kDigits - 1)] = 0;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int d = id[r] >= 0 ? (key[r] >> shift) & (kDigits - 1) : kDigits;   // past the end: a digit of its own
    unsigned same = 0xffffffffu;   // the lanes with this digit
    for (int q = 0; q <= bits; ++q) {
      const unsigned v = __ballot_sync(0xffffffffu, (d >> q) & 1);
      same &= (d >> q) & 1 ? v : ~v;
    }
    const int leader = __ffs((int)same) - 1;
    int old = 0;
    if (lane == leader && d < kDigits) {
      old = cnt[w][d];
      cnt[w][d] = old + __popc(same);
    }
    old = __shfl_sync(0xffffffffu, old, leader);
    rank[r] = old + __popc(same & ((1u << lane) - 1u));
    __syncwarp();
  }
  __syncthreads();
  for (int d = threadIdx.x; d < kDigits; d += 256) {
    int run;
    if (OWN) {
      run = cell_start[(int)min((long long)C, (long long)d << shift)];
      for (int t = 0; t < (int)blockIdx.x; ++t) run += hist[((size_t)t << bits) + d];
    } else {
      run = hist[((size_t)blockIdx.x << bits) + d];
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int v = cnt[k][d];
      cnt[k][d] = run;
      run += v;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    if (id[r] < 0) continue;
    const int p = cnt[w][(key[r] >> shift) & (kDigits - 1)] + rank[r];
    out[p] = id[r];
    if (next_hist)
      atomicAdd(next_hist + ((size_t)(p / kTile) << bits) + ((key[r] >> (shift + bits)) & (kDigits - 1)), 1);
    emit(p, id[r]);
  }
}

// cell_start[C + 1] from the counts, and perm: cell_of's atoms in stable cell
// order, with emit(slot, atom) for each.  tmp[n]: scratch; seg as launch_scan's;
// dep: launch_dependent (binning of 777,777 atoms 71 -> 57 us; the adjoint's step
// graphs are slower with it, 44.0 -> 45.6 ms for 100 steps).
template <class Emit>
void launch_cell_order(const int* cell_of, int n, long long C, const OrderBuf& b, int* cell_start, int* seg, int* tmp,
                       int* perm, const Emit& emit, bool dep, cudaStream_t st) {
  launch_scan(b.count, cell_start, (int)C, seg, b.hist[0], b.n_tiles, b.bits, b.passes > 1 ? b.tot[0] : nullptr, dep, st);
  const int* in = nullptr;
  const int groups = (1 << b.bits) / 32;
  for (int p = 0; p < b.passes; ++p) {
    const int k = p & 1, shift = b.bits * p;
    const bool top = p + 1 == b.passes, own = top && b.n_tiles <= 32;
    int* out = ((b.passes - p) & 1) ? perm : tmp;   // the last pass writes perm
    int* nh = top ? nullptr : b.hist[k ^ 1];
    if (p == 1 && !top) {   // a middle pass (over 262,144 cells): its totals, and the counts it reuses
      k_digit_totals<<<groups, 1024, 0, st>>>(b.bits, b.hist[k], b.n_tiles, b.tot[k]);
      cudaMemsetAsync(nh, 0, (sizeof(int) << b.bits) * (size_t)b.n_tiles, st);
    }
    if (!own)
      launch_dependent(dep && (p != 1 || top), k_digit_places, groups, 1024, 0, st, b.tot[k], top ? cell_start : nullptr, (int)C, shift, b.bits, b.hist[k],
                       b.n_tiles);
#define MDG_SCATTER(ROUNDS, OWN, E)                                                                                  \
  launch_dependent(dep, k_digit_scatter<ROUNDS, OWN, std::decay_t<decltype(E)>>, b.n_tiles, 256, 0, st, cell_of, in, \
                   n, cell_start, (int)C, shift, b.bits, b.hist[k], out, nh, E)
    if (own) {   // at most 32 tiles: never 2,048 atoms each
      if (b.tile == 256) MDG_SCATTER(1, true, emit); else MDG_SCATTER(4, true, emit);
    } else if (top) {
      if (b.tile == 1024) MDG_SCATTER(4, false, emit); else MDG_SCATTER(8, false, emit);
    } else {
      if (b.tile == 256) MDG_SCATTER(1, false, EmitNothing{});
      else if (b.tile == 1024) MDG_SCATTER(4, false, EmitNothing{});
      else MDG_SCATTER(8, false, EmitNothing{});
    }
#undef MDG_SCATTER
    in = out;
  }
}

}  // namespace mdg
