// md_static.cu -- cell binning that allocates no device memory, and the stable
// cell order it shares with the adjoint (cell_order.cuh).
//
// md_bin_static runs the same stable counting sort as md_rebin (cell id per
// atom, histogram, exclusive scan, order by atom index inside each cell) for
// one periodic box whose positions the caller already holds on the GPU.  Its
// scratch lives in g_bin_scratch below, a fixed-size array in the library's
// device image; the caller passes only inputs and outputs.  The order is a
// radix sort by cell id, whose work is the same whatever the positions.
// 777,777 atoms in 25^3 cells: 90 -> 55 us of kernels in 6 launches instead of
// 18 (bucket by atomics, ordered runs per cell, twelve merge passes of which
// the host cannot know that none is needed).
#include <cuda_runtime.h>

#include <cmath>

#include "../../include/md.h"
#include "cell_order.cuh"

namespace mdg {

constexpr int kStaticMaxAtoms = 1 << 20;   // 1,048,576 atoms
constexpr int kStaticMaxCells = 1 << 17;   // 131,072 cells (M <= 50)

// One copy per device that loads the library, kept until the process exits:
// per-cell counters, the digit counts of the order's passes and one per-atom
// array.  The size is 4 * (2^17 + 3 * 2^20 + 64) bytes = 13.1 MB.
constexpr size_t kScratchInts = (size_t)kStaticMaxCells + 3 * (size_t)kStaticMaxAtoms + 64;
static __device__ __align__(256) int g_bin_scratch[kScratchInts];

// same cell formula as the system path: s = x - L floor(x/L), k = floor(s M/L)
__device__ __forceinline__ int static_coord(double x, double L, double inv_h, int M) {
  double s = x;
  if (__double_as_longlong(x) < 0 || __double_as_longlong(x) >= __double_as_longlong(L))
    s = __dsub_rn(x, __dmul_rn(L, floor(__ddiv_rn(x, L))));
  return cell_floor(__dmul_rn(s, inv_h), M);
}

__global__ void __launch_bounds__(256) k_static_count(const double* __restrict__ x, int n, double L, double inv_h, int M,
                                                      int* __restrict__ cell_of, const OrderBuf b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = 0;
  if (i < n) {
    const int cx = static_coord(x[i], L, inv_h, M);
    const int cy = static_coord(x[n + i], L, inv_h, M);
    const int cz = static_coord(x[2 * n + i], L, inv_h, M);
    c = (cz * M + cy) * M + cx;
    cell_of[i] = c;
  }
  order_count(i < n, c, blockIdx.x * 256, b);
}

}  // namespace mdg

using namespace mdg;

void md_set_global_error(const char* msg);   // md_api.cu: message for md_last_error(NULL)

extern "C" int md_bin_static(const double* pos, int32_t n_atoms, double box, int32_t cells_per_side, int32_t* cell_of,
                             int32_t* cell_start, int32_t* perm, void* cuda_stream) {
  auto fail = [](int code, const char* msg) {
    md_set_global_error(msg);
    if (code == MD_ECUDA) cudaGetLastError();   // reported: not left to the next call
    return code;
  };
  if (!pos || !cell_of || !cell_start || !perm) return fail(MD_EINVAL, "null pointer argument");
  if (n_atoms < 1 || n_atoms > kStaticMaxAtoms) return fail(MD_EINVAL, "n_atoms must be 1 .. 1,048,576");
  if (cells_per_side < 1) return fail(MD_EINVAL, "cells_per_side must be >= 1");
  const long long C = (long long)cells_per_side * cells_per_side * cells_per_side;
  if (C > kStaticMaxCells) return fail(MD_EINVAL, "more than 131,072 cells (cells_per_side > 50)");
  if (!(box > 0) || !std::isfinite(box)) return fail(MD_EINVAL, "box must be positive");
  // The array's device address on the current device (host code may not use
  // the symbol itself).  Looked up on every call: it is cheap, and a cached
  // address would go stale if the device's context were reset and the module
  // loaded again elsewhere.
  void* sp = nullptr;
  const cudaError_t se = cudaGetSymbolAddress(&sp, g_bin_scratch);
  if (se != cudaSuccess || !sp) return fail(MD_ECUDA, "cudaGetSymbolAddress of the binning scratch failed");
  int* scratch = (int*)sp;
  // counters and digit counts (131,072 + 2 * 513 * 512 ints at most), then n ints
  const OrderBuf ob = order_buffers(scratch, n_atoms, C);
  int* tmp = scratch + (order_ints(n_atoms, C) + 63) / 64 * 64;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const double inv_h = (double)cells_per_side / box;
  if (cudaMemsetAsync(scratch, 0, sizeof(int) * order_clear_ints(ob, C), st) != cudaSuccess)
    return fail(MD_ECUDA, "clearing the cell counters failed");
  k_static_count<<<(n_atoms + 255) / 256, 256, 0, st>>>(pos, n_atoms, box, inv_h, cells_per_side, cell_of, ob);
  launch_cell_order(cell_of, n_atoms, C, ob, cell_start, nullptr, tmp, perm, EmitNothing{}, true, st);   // C <= 2^17: no seg
  if (cudaGetLastError() != cudaSuccess) return fail(MD_ECUDA, "a binning kernel failed to launch");
  return MD_OK;
}

extern "C" int md_wait_selftest(int32_t spins) {
  if (spins < 1 || spins > 100000) {
    md_set_global_error("spins must be 1 .. 100000");
    return MD_EINVAL;
  }
  unsigned* flag = nullptr;
  if (cudaMalloc(&flag, sizeof(unsigned)) != cudaSuccess) {
    cudaGetLastError();
    md_set_global_error("device allocation failed");
    return MD_ENOMEM;
  }
  unsigned f = 0;
  const bool ok = cudaMemset(flag, 0, sizeof(unsigned)) == cudaSuccess &&
                  (launch_wait_selftest((unsigned)spins, flag, 0), cudaGetLastError() == cudaSuccess) &&
                  cudaMemcpy(&f, flag, sizeof f, cudaMemcpyDeviceToHost) == cudaSuccess;
  cudaFree(flag);
  if (!ok) {
    md_set_global_error("the wait self-test failed to run");
    return MD_ECUDA;
  }
  if (f & kFlagTimeout) {
    md_set_global_error("a bounded device wait gave up (expected in this self-test)");
    return MD_ETIMEOUT;
  }
  return MD_OK;
}
