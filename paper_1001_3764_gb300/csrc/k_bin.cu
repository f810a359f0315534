// k_bin.cu -- on-GPU cell binning (Sec. 3.1).
//
// The paper's GBIN_NEW claims a slot per atom with atomicAdd into a
// fixed-capacity bin (Sec. 3.1, GBIN_NEW listing).  Here the same histogram
// feeds a counting sort: histogram -> exclusive scan -> scatter -> per-cell
// rank by atom index.  The result is a stable order (cell, atom index) that
// does not depend on the order in which atomics were served, and no bin has
// a capacity limit.  Cell indices are computed in FP64 from the master
// positions with explicitly rounded operations, so they equal the oracle's.
//
// Sorted positions are stored in units of the cell side relative to the
// centre of the atom's cell (|u| <= 1/2 at the rebin), so neighbour cells are
// offset by exact integers and an FP32 coordinate carries about 2^-25 h.
// The cluster lists are built in k_lj.cu.
#include "cell_order.cuh"

namespace mdg {

// --------------------------------------------------------------- helpers
__device__ __forceinline__ int find_rep_by_cell(const RepDev* reps, int n_reps, int c) {
  int lo = 0, hi = n_reps - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (reps[mid].cell_base <= c) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// cell coordinate along one axis: s = x - L floor(x/L); k = floor(s * M/L).
// The integrator keeps x in [0, L), where the wrap leaves x unchanged, so the
// FP64 division is only taken for positions outside the box.
__device__ __forceinline__ int cell_coord(double x, double L, double inv_h, int M) {
  double s = x;
  if (__double_as_longlong(x) < 0 || __double_as_longlong(x) >= __double_as_longlong(L))
    s = __dsub_rn(x, __dmul_rn(L, floor(__ddiv_rn(x, L))));
  return cell_floor(__dmul_rn(s, inv_h), M);
}

// --------------------------------------------------------------- histogram
template <typename T>
__global__ void __launch_bounds__(256) k_bin_count(const T* __restrict__ x, int N, const Tile* __restrict__ tiles,
                                                   const RepDev* __restrict__ reps, int* __restrict__ cell_of,
                                                   int* __restrict__ cellc, int* __restrict__ count,
                                                   int* __restrict__ slot) {
  const Tile t = tiles[blockIdx.x];
  if ((int)threadIdx.x >= t.len) return;
  const int i = t.start + threadIdx.x;
  const RepDev& R = reps[t.rep];
  const double L = R.L, ih = R.inv_h;
  const int M = R.M;
  int cx = cell_coord((double)x[i], L, ih, M);
  int cy = cell_coord((double)x[N + i], L, ih, M);
  int cz = cell_coord((double)x[2 * N + i], L, ih, M);
  int c = R.cell_base + (cz * M + cy) * M + cx;
  cell_of[i] = c;
  cellc[i] = cx | (cy << 10) | (cz << 20);
  slot[i] = atomicAdd(count + c, 1);
}

void launch_bin_count(bool mixed, const void* x, int N, const Tile* tiles, int n_tiles, const RepDev* reps,
                      int* cell_of, int* cellc, int* count, int* slot, cudaStream_t st) {
  if (mixed)
    k_bin_count<double><<<n_tiles, 256, 0, st>>>((const double*)x, N, tiles, reps, cell_of, cellc, count, slot);
  else
    k_bin_count<float><<<n_tiles, 256, 0, st>>>((const float*)x, N, tiles, reps, cell_of, cellc, count, slot);
}

// --------------------------------------------------------------- exclusive scans
// A block scans a segment of 4,096 cells (four per thread, one 16-byte load)
// and finds what lies before it itself: up to kScanDirect cells by adding
// their counts (a coalesced read of at most 512 KB, from L2), above by adding
// the segment sums that a first launch leaves.  No block waits for another,
// and all segments run side by side; the one block that scanned everything
// before took 83 us for 32,768 cells, this 6.6.  CL: also the scan of
// ceil(count / 4), the clusters.
constexpr int kScanSeg = 4096;
constexpr int kScanDirect = 1 << 17;

template <bool CL>
__device__ __forceinline__ void scan_add4(const int* __restrict__ count, int k, int C, int& s, int& sc) {
  if (k + 3 < C) {
    const int4 v = *reinterpret_cast<const int4*>(count + k);
    s += v.x + v.y + v.z + v.w;
    if (CL) sc += ((v.x + 3) >> 2) + ((v.y + 3) >> 2) + ((v.z + 3) >> 2) + ((v.w + 3) >> 2);
  } else {
    for (; k < C; ++k) { s += count[k]; if (CL) sc += (count[k] + 3) >> 2; }
  }
}

// sums over the block of two values per thread; valid on every thread
__device__ __forceinline__ int2 block_add2(int s, int sc, int2* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    sc += __shfl_xor_sync(0xffffffffu, sc, o);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[w] = make_int2(s, sc);
  __syncthreads();
  int2 v = sh[lane];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}

// segment sums (the first launch of a scan of many cells)
template <bool CL>
__global__ void __launch_bounds__(1024) k_scan_sums(const int* __restrict__ count, int C, int2* __restrict__ seg) {
  __shared__ int2 sh[32];
  int s = 0, sc = 0;
  scan_add4<CL>(count, blockIdx.x * kScanSeg + 4 * threadIdx.x, C, s, sc);
  const int2 v = block_add2(s, sc, sh);
  if (threadIdx.x == 0) seg[blockIdx.x] = v;
}

template <bool CL>
__global__ void __launch_bounds__(1024) k_scan_segments(const int* __restrict__ count, int* __restrict__ start,
                                                        int* __restrict__ cl_start, int C, int2* __restrict__ seg,
                                                        int segs, const int* __restrict__ hist, int n_tiles,
                                                        int bits, int* __restrict__ tot) {
  __shared__ int2 sh[32];
  wait_for_predecessor();
  if ((int)blockIdx.x >= segs) {   // blocks past the segments: 32 digit totals each (cell_order.cuh)
    digit_totals(blockIdx.x - segs, bits, hist, n_tiles, tot);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, b0 = blockIdx.x * kScanSeg;
  int s = 0, sc = 0;
  if (seg) {
    for (int k = tid; k < (int)blockIdx.x; k += 1024) { s += seg[k].x; sc += seg[k].y; }
  } else {
    for (int k = 4 * tid; k < b0; k += kScanSeg) scan_add4<CL>(count, k, b0, s, sc);
  }
  const int2 pre = block_add2(s, sc, sh);
  // the segment: four cells per thread
  const int k0 = b0 + 4 * tid;
  int n[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) n[q] = k0 + q < C ? count[k0 + q] : 0;
  const int ts = n[0] + n[1] + n[2] + n[3];
  const int tc = CL ? ((n[0] + 3) >> 2) + ((n[1] + 3) >> 2) + ((n[2] + 3) >> 2) + ((n[3] + 3) >> 2) : 0;
  int is = ts, ic = tc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, is, o), c = CL ? __shfl_up_sync(0xffffffffu, ic, o) : 0;
    if (lane >= o) { is += a; ic += c; }
  }
  __syncthreads();
  if (lane == 31) sh[w] = make_int2(is, ic);
  __syncthreads();
  if (w == 0) {
    int2 v = sh[lane];
    const int2 own = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int a = __shfl_up_sync(0xffffffffu, v.x, o), c = __shfl_up_sync(0xffffffffu, v.y, o);
      if (lane >= o) { v.x += a; v.y += c; }
    }
    sh[lane] = make_int2(v.x - own.x, v.y - own.y);
  }
  __syncthreads();
  int run = pre.x + sh[w].x + is - ts, runc = pre.y + sh[w].y + ic - tc;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (k0 + q < C) {
      start[k0 + q] = run;
      if (CL) cl_start[k0 + q] = runc;
      run += n[q];
      runc += (n[q] + 3) >> 2;
      if (k0 + q == C - 1) { start[C] = run; if (CL) cl_start[C] = runc; }
    }
  }
}

size_t scan_seg_ints(long long C) { return C <= kScanDirect ? 0 : 2 * (size_t)((C + kScanSeg - 1) / kScanSeg); }

template <bool CL>
static void launch_scan_t(const int* count, int* start, int* cl_start, int C, int* seg, const int* hist, int n_tiles,
                          int bits, int* tot, bool dep, cudaStream_t st) {
  const int segs = (C + kScanSeg - 1) / kScanSeg;
  int2* sg = C <= kScanDirect ? nullptr : reinterpret_cast<int2*>(seg);
  if (sg) k_scan_sums<CL><<<segs, 1024, 0, st>>>(count, C, sg);
  launch_dependent(dep, k_scan_segments<CL>, segs + (tot ? (1 << bits) / 32 : 0), 1024, 0, st, count, start, cl_start, C,
                   sg, segs, hist, n_tiles, bits, tot);
}

void launch_scan(const int* count, int* cell_start, int C, int* seg, const int* hist, int n_tiles, int bits,
                 int* tot, bool dep, cudaStream_t st) {
  launch_scan_t<false>(count, cell_start, nullptr, C, seg, hist, n_tiles, bits, tot, dep, st);
}

void launch_scan2(const int* count, int* cell_start, int* cl_start, int C, int* seg, bool dep, cudaStream_t st) {
  launch_scan_t<true>(count, cell_start, cl_start, C, seg, nullptr, 0, 0, nullptr, dep, st);
}

// --------------------------------------------------------------- scatter
__global__ void __launch_bounds__(256) k_bin_scatter(const int* __restrict__ cell_of, const int* __restrict__ slot,
                                                     const int* __restrict__ cell_start, int* __restrict__ tmp, int N) {
  wait_for_predecessor();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) tmp[cell_start[cell_of[i]] + slot[i]] = i;
}

void launch_bin_scatter(const int* cell_of, const int* slot, const int* cell_start, int* tmp, int N, bool dep,
                        cudaStream_t st) {
  if (N > 0) launch_dependent(dep, k_bin_scatter, (N + 255) / 256, 256, 0, st, cell_of, slot, cell_start, tmp, N);
}

// --------------------------------------------------------------- per-cell stable order + sorted arrays
// A block takes a cell, or where cells outnumber atoms and are many kSortCells
// of them, of which it orders those that hold atoms: a block per empty cell is
// its launch and its wait, 1.0 ns a cell over the GPU, which for kSortMany cells
// is the 30 us that a block may take for the atoms of its kSortCells.  12 chains in
// 36.5 / 60 / 150 nm (36k, 157k, 2.5M cells): 37 / 159 / 2,531 us, 7 / 9 / 80 now.
constexpr int kSortCap = 2048;
constexpr int kSortThreads = 128, kSortCells = 32, kSortMany = 1 << 15;

// stable order of the n atoms from place b on, cell c, by the whole block
template <typename T>
__device__ __forceinline__ void sort_cell(int c, int b, int n, int* __restrict__ ids, const T* __restrict__ x, int N,
                                          const int* __restrict__ tmp, const unsigned char* __restrict__ mtype,
                                          const int* __restrict__ cellc, const uint16_t* __restrict__ site,
                                          const RepDev* __restrict__ reps, int n_reps, int sites,
                                          int* __restrict__ perm, int* __restrict__ inv_perm,
                                          float4* __restrict__ pos, int* __restrict__ tag, float4* __restrict__ ref,
                                          unsigned* __restrict__ flags) {
  const RepDev& R = reps[find_rep_by_cell(reps, n_reps, c)];
  // A cell of more than kSortCap atoms (over 40 times a melt's ~46) cannot
  // be staged by the force kernels either: it is reported as a capacity
  // overflow, and its atoms keep their bucket order (bounded work).
  const bool in_smem = n <= kSortCap;
  if (!in_smem && threadIdx.x == 0) atomicOr(flags, kFlagNbrOverflow);
  if (in_smem)
    for (int k = threadIdx.x; k < n; k += blockDim.x) ids[k] = tmp[b + k];
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const int id = in_smem ? ids[k] : tmp[b + k];
    int rank = k;
    if (in_smem) {
      rank = 0;
      for (int q = 0; q < n; ++q) rank += ids[q] < id;
    }
    const int s = b + rank;
    perm[s] = id;
    inv_perm[id] = s;
    const int cc = cellc[id];
    float4 p;
    if constexpr (sizeof(T) == 8) {      // FP64 master: integer-pipe offset and rounding, same value
      p.x = cell_unit_t(x[id], cc & 1023, R);
      p.y = cell_unit_t(x[N + id], (cc >> 10) & 1023, R);
      p.z = cell_unit_t(x[2 * N + id], (cc >> 20) & 1023, R);
    } else {
      p.x = cell_unit(x[id], cc & 1023, 0, R);
      p.y = cell_unit(x[N + id], (cc >> 10) & 1023, 0, R);
      p.z = cell_unit(x[2 * N + id], (cc >> 20) & 1023, 0, R);
    }
    const int st = site[id];
    const int chain = R.chain_off + (id - R.atom_off) / sites;
    const int type = mtype ? (int)mtype[st] : ((st == 0 || st == sites - 1) ? 1 : 0);
    p.w = (float)type;   // LJ type: the tile kernels copy positions as they are
    pos[s] = p;
    ref[id] = p;
    tag[s] = (chain << kTagSiteBits) | st | (type << kTagTypeBit);
  }
}

template <typename T, bool MANY>
__global__ void __launch_bounds__(kSortThreads) k_cell_sort(const T* __restrict__ x, int N, const int* __restrict__ cell_start,
                                                            const int* __restrict__ tmp, const unsigned char* __restrict__ mtype,
                                                            const int* __restrict__ cellc,
                                                            const uint16_t* __restrict__ site, const RepDev* __restrict__ reps,
                                                            int n_reps, int C, int sites, int* __restrict__ perm,
                                                            int* __restrict__ inv_perm, float4* __restrict__ pos,
                                                            int* __restrict__ tag, float4* __restrict__ ref,
                                                            unsigned* __restrict__ flags) {
  __shared__ int ids[kSortCap];
  wait_for_predecessor();
  if constexpr (!MANY) {
    const int c = blockIdx.x, b = cell_start[c], n = cell_start[c + 1] - b;
    if (n == 0) return;
    sort_cell(c, b, n, ids, x, N, tmp, mtype, cellc, site, reps, n_reps, sites, perm, inv_perm, pos, tag, ref, flags);
  } else {
    __shared__ int3 found[kSortCells];   // cell, first place, atoms
    __shared__ int n_found;
    if (threadIdx.x == 0) n_found = 0;
    __syncthreads();
    const int c = blockIdx.x * kSortCells + threadIdx.x;
    if (threadIdx.x < kSortCells && c < C) {
      const int b = cell_start[c], n = cell_start[c + 1] - b;
      if (n > 0) found[atomicAdd(&n_found, 1)] = make_int3(c, b, n);
    }
    __syncthreads();
    for (int k = 0; k < n_found; ++k) {
      const int3 f = found[k];
      sort_cell(f.x, f.y, f.z, ids, x, N, tmp, mtype, cellc, site, reps, n_reps, sites, perm, inv_perm, pos, tag, ref, flags);
      __syncthreads();   // ids are no longer read
    }
  }
}

void launch_cell_sort(bool mixed, const void* x, int N, const int* cell_start, const int* tmp,
                      const unsigned char* mtype, const int* cellc,
                      const uint16_t* site, const RepDev* reps, int n_reps, int C, int sites, int* perm,
                      int* inv_perm, float4* pos, int* tag, float4* ref, unsigned* flags, bool dep,
                      cudaStream_t st) {
  const bool many = C > N && C >= kSortMany;
  const int grid = many ? (C + kSortCells - 1) / kSortCells : C;
#define MDG_SORT(T, MANY)                                                                                           \
  launch_dependent(dep, k_cell_sort<T, MANY>, grid, kSortThreads, 0, st, (const T*)x, N, cell_start, tmp, mtype, cellc, \
                   site, reps, n_reps, C, sites, perm, inv_perm, pos, tag, ref, flags)
  if (mixed) {
    if (many) MDG_SORT(double, true); else MDG_SORT(double, false);
  } else {
    if (many) MDG_SORT(float, true); else MDG_SORT(float, false);
  }
#undef MDG_SORT
}

}  // namespace mdg
