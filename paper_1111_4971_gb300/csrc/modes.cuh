// Host-side declarations of the mode-space solve (modes_impl.cuh).
#pragma once

#include <cuda_runtime.h>

namespace pp {

template <typename T>
struct ModeArgs;

// The mode form takes a mesh where these two are within 227 KB: a ring of field
// rows, the y-mode table and 32 z values of the mode columns.  A rule of the
// interface, kept from kernels laid out so; the present ones need less (FP32:
// modes_sums.cu reads a long y table through L1, FP64: modes_split.cu takes 64 KB).
template <typename T>
inline size_t mode_proj_smem(int ny, int mxp, int myp, bool fold) {
  constexpr int XB = sizeof(T) == 4 ? 16 : 8, ZC = 32;
  const int mpass = sizeof(T) == 4 ? mxp : (mxp + 3) / 4 * 2;          // FP64: the x modes in two rounds
  const size_t ring = size_t(3) * XB * (fold ? 8 : 4) * ZC, sums = size_t(XB + mpass) * myp * ZC;
  return sizeof(T) * ((ring > sums ? ring : sums) + size_t(fold ? ny / 2 : ny) * myp + size_t(XB) * mxp);
}
template <typename T>
inline size_t mode_back_smem(int ny, int mx, int mxp, int myp, bool fold) {
  constexpr int XB = sizeof(T) == 4 ? 16 : 8, ZC = 32;
  return sizeof(T) * (size_t(mx) * myp * ZC + size_t(fold ? ny / 2 : ny) * myp + size_t(XB) * mxp);
}

// y-mode slots of the tables (MYP, a multiple of 4 in {8, 12, 16, 20, 24, 32}):
// with the mirror fold, the odd modes 1, 3, .. and the even modes 2, 4, ..
// take MYP/2 slots each; without it, the modes 1..my in order
inline int mode_slots(int my, bool fold) {
  int need = fold ? 2 * ((my + 1) / 2) : my;
  need = (need + 3) / 4 * 4;
  if (need <= 8) return 8;
  if (need <= 24) return need;
  return need <= 32 ? 32 : -1;
}
// the y mode held by slot s of MYP slots
inline int mode_of_slot(int s, int myp, bool fold) {
  if (!fold) return s + 1;
  return s < myp / 2 ? 2 * s + 1 : 2 * (s - myp / 2) + 2;
}

// the largest divisor of n that is at most 4
inline int divisor_to_4(int n) {
  for (int d = 4; d > 1; --d)
    if (n % d == 0) return d;
  return 1;
}

// Shape of the FP32 projection and back-projection (modes_sums.cu): warps per
// CTA (of kModeRowsPerWarp x rows each), and of the projection the x blocks that
// a CTA takes one after the other (reps) and the groups of them, each writing
// one partial.
//   Warps: 8, or 4 where 8 leave fewer than 128 CTAs (64^2 x 256, 8 / 4 warps:
//   projection 7.2 / 7.3, back-projection 6.5 / 5.9 us; 128^2 x 1024, 8 / 4 / 16:
//   20.3 / 21.9 / 31.6 and 17.5 / 18.1 / 17.1).  One x row a warp: 25.8 and 23.7.
//   Groups: every x block its own while there are at most 16 (128^2 x 1024, 8 / 4
//   groups: 20.3 / 23.5 us; all with x-mode sums of one slot at a time), else a
//   divisor of 4 to 8: the partials (1.6 MB each at 400 columns of 1024) would
//   come near the field's own bytes.  Their memory is at most 48 MiB, or what one
//   partial per up to 4 blocks of 16 rows takes.
constexpr int kModeRowsPerWarp = 2;
struct ModeShape {
  int warps, reps, groups;
};
inline ModeShape mode_shape(int nx, int nz, int columns) {
  ModeShape s{};
  s.warps = nz / 32 * nx / (8 * kModeRowsPerWarp) < 128 ? 4 : 8;
  const int xblocks = nx / (s.warps * kModeRowsPerWarp), xb16 = nx / 16;
  const size_t partial = sizeof(float) * size_t(columns) * nz, most = size_t(48) << 20;
  const size_t old = size_t(xb16 / divisor_to_4(xb16) + 1) * partial, cap = old > most ? old : most;
  s.groups = xblocks;
  if (xblocks > 16) {
    int g = 8;
    while (g >= 4 && xblocks % g) --g;
    for (int k = 9; g < 4 && k <= xblocks; ++k)
      if (xblocks % k == 0) { g = k; break; }
    s.groups = g;
  }
  while (s.groups > 1 && (xblocks % s.groups || size_t(s.groups + 1) * partial > cap)) --s.groups;
  s.reps = xblocks / s.groups;
  return s;
}

// z recurrences (modes_z.cu): z values per thread, and the parameters of a
// mode column: beta, gamma, 1 - q, q, then q^{kModeZRun 2^i} for i < 8
constexpr int kModeZRun = 8;
constexpr int kModeZPar = 12;

// stage 1, part -> psi: the z convolution, or the banded operator's stencil
template <typename T>
cudaError_t launch_mode_z_stage(const ModeArgs<T>& a, cudaStream_t st);
// FP32 stage 0 (projection rho -> part) or 2 (back-projection psi -> phi) on
// any mesh (modes_sums.cu; FP64: modes_split.cuh)
cudaError_t launch_mode_sums(int stage, int myp, bool fold, const ModeArgs<float>& a, cudaStream_t st);

// A group of FP32 mode-form solves of one shape (nx, ny, nz, mode layout),
// run by one launch per stage (the batched call):
// args[s] (device memory) holds solve s's tables and scratch, rho / phi its
// field arrays (kernel parameters, so that a captured launch keeps them).
constexpr int kMaxModeGroup = 64;
struct ModeGroup {
  const ModeArgs<float>* args;
  const float* rho[kMaxModeGroup];
  float* phi[kMaxModeGroup];
  int n;
  int nz;
};

// the z convolution as two recurrences per mode column (modes_z.cu): nz a
// power of two in 32..1024, groups partial projections summed on load
template <typename T>
cudaError_t launch_mode_z(const ModeArgs<T>& a, int groups, cudaStream_t st);
// the same for a group (columns of solve s in the CTAs s * cps ..)
cudaError_t launch_mode_z_group(const ModeArgs<float>& a, int groups, const ModeGroup& g, cudaStream_t st);

// launch_mode_sums for a group (g->args[s] shaped like a)
cudaError_t launch_mode_sums_group(int stage, int myp, bool fold, const ModeArgs<float>& a, const ModeGroup& g,
                                   cudaStream_t st);

}  // namespace pp
