// FP64 mode sums on the tensor cores (modes_split.cu): host-side declarations.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "split_tables.h"

namespace pp {

// Fragment tables of one sine table (see split_table_kernel): uint4 values
inline int split_tiles(int n) { return (n + 7) / 8; }       // columns of 8
inline int split_steps(int k) { return (k + 15) / 16; }     // k steps of 16
// contraction over `rows` table rows into the slots (halves: the slots' two
// parity halves start a tile of their own)
inline int split_contract_tiles(int slots, bool halves) {
  return halves ? 2 * split_tiles(slots / 2) : split_tiles(slots);
}
inline size_t split_contract_size(int rows, int slots, bool halves) {
  return size_t(split_steps(rows)) * split_contract_tiles(slots, halves) * (kSplitDigits / 2) * 32;
}
// expansion of the slots into `rows` rows
inline int split_expand_steps(int slots, bool halves) { return halves ? 2 * split_steps(slots / 2) : split_steps(slots); }
inline size_t split_expand_size(int rows, int slots, bool halves) {
  return size_t(split_tiles(rows)) * split_expand_steps(slots, halves) * (kSplitDigits / 2) * 32;
}
// tab [rows][slots] and scale in device memory
cudaError_t build_split_table(const double* tab, const int* scale, int rows, int slots, bool halves, bool expand,
                              uint4* out, cudaStream_t st);

// One FP64 solve's stages: tables, mesh and the buffer of the half-transformed
// field [nx][myp][zs] (zs z values at a time, split_slab)
struct SplitArgs {
  const uint4 *cy, *cx;      // contraction tables of the y modes and the x modes
  const uint4 *ey, *ex;      // expansion tables
  RowScale ys, xs;           // the tables' row scales
  int cy_run, cx_run;        // contract_steps of cy, cx
  bool ey_small, ex_small;   // expand_sums_small of ey, ex
  int nx, ny, nz;
  int mx, mxp, myp;
  int fold;                  // 0: all rows, 1: mirror pairs (j, ny-1-j), 2: (j, ny-j) with row 0 on the wall
  double* half;
  int zs;
  int nan_tile;              // 1: a value that is not finite makes its 16 planes' outputs NaN (single stages), 0: its own plane's
};
// z values per slab: the half-transformed field of a slab is at most 32 MiB
// (it stays in L2 between the kernel that writes it and the one that reads it)
constexpr size_t kSplitHalfBytes = size_t(32) << 20;
inline int split_slab(int nx, int myp, int nz) {
  int zs = nz;
  while (zs > 16 && size_t(nx) * myp * zs * sizeof(double) > kSplitHalfBytes) zs /= 2;
  return zs;
}
inline size_t split_half_bytes(int nx, int myp, int nz) {
  return size_t(nx) * myp * split_slab(nx, myp, nz) * sizeof(double);
}
// rho -> part [mxp * myp][nz], psi [mxp * myp][nz] -> phi
cudaError_t launch_split_project(const SplitArgs& s, const double* rho, double* part, cudaStream_t st);
cudaError_t launch_split_back(const SplitArgs& s, const double* psi, double* phi, cudaStream_t st);

}  // namespace pp
