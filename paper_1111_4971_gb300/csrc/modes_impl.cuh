// Mode-space form of the pipe operator: the solve of Sec. 2 Eq. 10 with its
// transverse transforms pruned to the frequencies where the transformed Green
// function is not zero.
//
// Why this is the same operator.  The Green function is the truncated sine
// series of Eq. 7,
//     G = (8 pi / ab) sum_{m <= Mx, n <= My} kappa_mn^{-1} sin(m pi x/a) sin(m pi x'/a)
//                                          sin(n pi y/b) sin(n pi y'/b) f_mn(z - z'),
// f_mn = e^{-kappa |w|} (Eq. 9) or the longitudinal IGF g_z (Eq. 15-16), so
// the discrete sum of Eq. 4 factorises exactly into
//     rhot[m][n][k] = sum_{i,j} Sx[m][i] Sy[n][j] rho[i][j][k]          (projection)
//     psi[m][n][k]  = sum_{k'} K_mn(k - k') rhot[m][n][k']             (z convolution)
//     phi[i][j][k]  = sum_{m,n} Sx[m][i] Sy[n][j] psi[m][n][k]          (back-projection)
// with Sx[m][i] = sin(m pi x_i / a), Sy likewise, and
// K_mn(d) = hx hy hz (8 pi / ab) kappa_mn^{-1} f_mn(d hz).  On a mesh that
// spans the pipe the 2n-point transforms of Eq. 10 along x and y are, for a
// Green table built from these modes, nonzero only at |kx| <= Mx, |ky| <= My
// (the closed-form spectrum), and their products with the transformed density
// are exactly these mode sums; the projection is those transforms evaluated at
// the Mx x My frequencies that survive the product, and the back-projection
// the inverse transforms restricted to them.  The form holds on any mesh
// inside the pipe (windows included).  The z convolution is the zero-padded
// one of Appendix A (Eq. A.1-A.4); its kernel is a two-sided exponential in z
// apart from the centre tap, so it runs as two first-order recurrences
// (modes_z.cu).
//
// The operator is symmetric (G(r, r') = G(r', r)): the projection and the
// back-projection use the same tables and the z kernel is even, so the
// adjoint is the same computation.
//
// Kernels:
//   FP32 (modes_sums.cu): rho -> part[g][c][k] (c = m' * myp + n'; one partial
//        per group g of x blocks, which the z kernel sums), psi -> phi
//   FP64 (modes_split.cu): the same sums as exact integer products on the
//        tensor cores, one partial
//   modes_z.cu: part -> psi[c][k]; modes.cu: the banded operator's stencil
// Fold: where the mesh is symmetric about the pipe's mid-plane in y, or its
// first row lies on the wall, a row j and its mirror image have
// Sy[n][mirror] = (-1)^{n+1} Sy[n][j]; the tables then hold the odd n first and
// the even n after them (myp/2 slots each), and each sum over j runs over the
// pairs on rho(j) + rho(mirror) (odd n) and rho(j) - rho(mirror) (even n).
#pragma once

#include "zfft_impl.cuh"

namespace pp {

template <typename T>
struct ModeArgs {
  const T* rho;          // [nx][ny][nz]
  T* phi;                // [nx][ny][nz]
  T* part;               // [groups][mc][nz]
  T* psi;                // [mc][nz]
  const T* sx;           // [nx][mxp]
  const T* sy;           // [fold ? ny/2 : ny][myp]
  const T* zp;           // [mc][kModeZPar]: the z recurrences' parameters
  int nx, ny, nz;
  int mx;                // x modes
  int mxp;               // x modes padded to a multiple of 4 (columns of sx)
  int mc;                // mxp * MYP mode columns
  int groups;            // partial projections in part
  int mirror, wall;      // folded y rows: pair j is (j, mirror - j); wall != 0: pair 0 is (0, wall)
  const T* kb;           // banded operator: [mc][nb+1] real-space z kernel K_c(d), d = 0..nb
  int nb;                // neighbour planes of the banded operator (Eq. 18), -1: the full z convolution
};

}  // namespace pp
