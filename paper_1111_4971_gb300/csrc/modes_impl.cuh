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
// Kernels (one warp lane per z value of a 32-value z chunk, so that every
// global access is a run of 32 consecutive z):
//   mode_project_kernel  rho -> part[g][c][k]  (c = m' * MYP + n'; the
//                        projection of one group of x blocks, those of one
//                        thread-block cluster; the z kernel sums the groups)
//   mode_z_kernel        part -> psi[c][k]
//   mode_back_kernel     psi -> phi
// FY: the mesh is symmetric about the pipe's mid-plane in y
// (y_{ny-1-j} = b - y_j), so Sy[n][ny-1-j] = (-1)^{n+1} Sy[n][j]; the tables
// then hold the odd n first and the even n after them (MYP/2 slots each), and
// each sum over j runs over half the rows on rho(j) + rho(ny-1-j) (odd n) and
// rho(j) - rho(ny-1-j) (even n).
#pragma once

#include <cooperative_groups.h>

#include "zfft_impl.cuh"

namespace pp {

namespace mcg = cooperative_groups;

template <typename T>
struct ModeArgs {
  const T* rho;          // [nx][ny][nz]
  T* phi;                // [nx][ny][nz]
  T* part;               // [nx / (XB * cluster)][mc][nz]
  T* psi;                // [mc][nz]
  const T* sx;           // [nx][mxp]
  const T* sy;           // [FY ? ny/2 : ny][MYP]
  const T* zp;           // [mc][kModeZPar]: the z recurrences' parameters
  int nx, ny, nz;
  int mx;                // x modes
  int mxp;               // x modes padded to a multiple of 4 (columns of sx)
  int mc;                // mxp * MYP mode columns
  int groups;            // partial projections in part
  const T* kb;           // banded operator: [mc][nb+1] real-space z kernel K_c(d), d = 0..nb
  int nb;                // neighbour planes of the banded operator (Eq. 18), -1: the full z convolution
};

template <typename T, int MYP, bool FY>
struct ProjCfg {
  using S = ModeShape<T>;
  static constexpr int ROWS = FY ? 2 * S::YK : S::YK;
  static constexpr size_t STAGE = size_t(S::XB) * ROWS * S::ZC;     // elements
  static constexpr size_t ABUF = size_t(S::XB) * MYP * S::ZC;
  __host__ __device__ static size_t union_elems(int mxp) { return mode_proj_union<T>(mxp, MYP, FY); }
};

// four consecutive table values from shared memory (16-byte aligned)
template <typename T>
__device__ __forceinline__ void load4(const T* p, T (&s)[4]) {
  if constexpr (sizeof(T) == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
  } else {
    const double2 u = reinterpret_cast<const double2*>(p)[0], v = reinterpret_cast<const double2*>(p)[1];
    s[0] = u.x; s[1] = u.y; s[2] = v.x; s[3] = v.y;
  }
}

// Projection of one (z chunk, x block): grid (nz / ZC, nx / XB), launched in
// clusters of consecutive x blocks of one z chunk.  The rows of the block
// arrive YK at a time (with their mirror rows under FY) in a ring of STAGES
// buffers filled by cp.async; each thread accumulates, for its XPW x rows and
// its z, the MYP y-mode sums; these go through shared memory so that each
// warp then sums, over the block's XB rows, the x modes of its passes into
// the block's projection (shared memory).  The cluster's CTAs then add up
// their blocks' projections through distributed shared memory, each CTA a
// slice of the mode columns, in a fixed order (rank 0 first), and write one
// partial per cluster.
template <typename T, int MYP, bool FY>
__device__ __forceinline__ void mode_project(const ModeArgs<T>& a, unsigned char* smem_raw) {
  using S = ModeShape<T>;
  using Cfg = ProjCfg<T, MYP, FY>;
  static_assert(MYP % 4 == 0, "mode slots in fours");
  T* slab = reinterpret_cast<T*>(smem_raw);
  T* abuf = slab;                                   // once the slab is consumed
  T* red = abuf + Cfg::ABUF;                        // one round of the block's projection [.][ZC]
  T* sy = slab + Cfg::union_elems(a.mxp);
  T* sxs = sy + (FY ? a.ny / 2 : a.ny) * MYP;       // x-mode rows of the block [XB][mxp]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int z0 = int(blockIdx.x) * S::ZC;
  const int xb0 = int(blockIdx.y) * S::XB;
  const int nyk = FY ? a.ny / 2 : a.ny;
  const int nchunks = nyk / S::YK;
  constexpr int PPR = S::ZC * int(sizeof(T)) / 16;  // 16-byte pieces of a row's z chunk

  // stage c: rows yc .. yc+YK-1 and (FY) ny-yc-YK .. ny-yc-1, yc = c * YK
  auto issue = [&](int c) {
    T* dst = slab + size_t(c % S::STAGES) * Cfg::STAGE;
    const int yc = c * S::YK;
    for (int idx = threadIdx.x; idx < S::XB * Cfg::ROWS * PPR; idx += S::THREADS) {
      const int piece = idx % PPR;
      const int r = (idx / PPR) % Cfg::ROWS;
      const int xl = idx / (PPR * Cfg::ROWS);
      const int y = r < S::YK ? yc + r : a.ny - yc - S::YK + (r - S::YK);
      const T* src = a.rho + (size_t(xb0 + xl) * a.ny + y) * a.nz + z0;
      cp_async16(reinterpret_cast<unsigned char*>(dst + size_t(xl * Cfg::ROWS + r) * S::ZC) + 16 * piece,
                 reinterpret_cast<const unsigned char*>(src) + 16 * piece);
    }
    cp_async_commit();
  };
#pragma unroll
  for (int c = 0; c < S::STAGES - 1; ++c) {
    if (c < nchunks) issue(c);
    else cp_async_commit();
  }
  for (int i = threadIdx.x; i < nyk * MYP; i += S::THREADS) sy[i] = a.sy[i];
  for (int i = threadIdx.x; i < S::XB * a.mxp; i += S::THREADS) sxs[i] = a.sx[size_t(xb0) * a.mxp + i];

  T acc[S::XPW][MYP];
#pragma unroll
  for (int i = 0; i < S::XPW; ++i)
#pragma unroll
    for (int n = 0; n < MYP; ++n) acc[i][n] = T(0);

#pragma unroll 1
  for (int c = 0; c < nchunks; ++c) {
    cp_async_wait<S::STAGES - 2>();
    __syncthreads();               // stage c landed for every thread; stage c-1 is free
    if (c + S::STAGES - 1 < nchunks) issue(c + S::STAGES - 1);
    else cp_async_commit();
    const T* st = slab + size_t(c % S::STAGES) * Cfg::STAGE;
#pragma unroll
    for (int j = 0; j < S::YK; ++j) {
      T pa[S::XPW], qa[S::XPW];
#pragma unroll
      for (int i = 0; i < S::XPW; ++i) {
        const int xl = warp * S::XPW + i;
        const T u = st[(xl * Cfg::ROWS + j) * S::ZC + lane];
        if constexpr (FY) {
          const T v = st[(xl * Cfg::ROWS + 2 * S::YK - 1 - j) * S::ZC + lane];
          pa[i] = u + v;
          qa[i] = u - v;
        } else {
          pa[i] = u;
          qa[i] = u;
        }
      }
      const T* srow = sy + (c * S::YK + j) * MYP;
#pragma unroll
      for (int g = 0; g < MYP; g += 4) {
        T s4[4];
        load4(srow + g, s4);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const bool odd_slot = !FY || (g + k < MYP / 2);
#pragma unroll
          for (int i = 0; i < S::XPW; ++i) acc[i][g + k] = fma(s4[k], odd_slot ? pa[i] : qa[i], acc[i][g + k]);
        }
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();                 // the slab becomes the buffer of y-mode sums
#pragma unroll
  for (int i = 0; i < S::XPW; ++i)
#pragma unroll
    for (int n = 0; n < MYP; ++n) abuf[((warp * S::XPW + i) * MYP + n) * S::ZC + lane] = acc[i][n];
  __syncthreads();

  // x modes, in rounds of mode_round_modes: warp w takes the passes of MQ
  // modes q = w, w + WARPS, ... of the round; then the cluster's blocks are
  // summed for the round's columns: CTA `rank` takes a slice of them and
  // reads them from every CTA in rank order
  mcg::cluster_group cl = mcg::this_cluster();
  const int ncl = int(cl.num_blocks()), rank = int(cl.block_rank());
  T* out = a.part + size_t(blockIdx.y / ncl) * a.mc * a.nz + z0 + lane;
  const int mpr = mode_round_modes<T>(a.mxp);
#pragma unroll 1
  for (int m0 = 0; m0 < a.mxp; m0 += mpr) {
    const int m1 = m0 + mpr < a.mxp ? m0 + mpr : a.mxp;
#pragma unroll 1
    for (int q = m0 / S::MQ + warp; q * S::MQ < m1; q += S::WARPS) {
      T acc2[S::MQ][MYP];
#pragma unroll
      for (int k = 0; k < S::MQ; ++k)
#pragma unroll
        for (int n = 0; n < MYP; ++n) acc2[k][n] = T(0);
#pragma unroll 2
      for (int xl = 0; xl < S::XB; ++xl) {
        T s[S::MQ];
#pragma unroll
        for (int k = 0; k < S::MQ; ++k) s[k] = sxs[xl * a.mxp + q * S::MQ + k];
#pragma unroll
        for (int n = 0; n < MYP; ++n) {
          const T av = abuf[(xl * MYP + n) * S::ZC + lane];
#pragma unroll
          for (int k = 0; k < S::MQ; ++k) acc2[k][n] = fma(s[k], av, acc2[k][n]);
        }
      }
#pragma unroll
      for (int k = 0; k < S::MQ; ++k)
#pragma unroll
        for (int n = 0; n < MYP; ++n) red[((q * S::MQ + k - m0) * MYP + n) * S::ZC + lane] = acc2[k][n];
    }
    cl.sync();                     // every block's projection of the round is complete
    const int nc = (m1 - m0) * MYP;
    const int per = (nc + ncl - 1) / ncl;
    const int c0 = rank * per, c1 = c0 + per < nc ? c0 + per : nc;
#pragma unroll 1
    for (int c = c0 + warp; c < c1; c += S::WARPS) {
      T sum = T(0);
#pragma unroll 1
      for (int r = 0; r < ncl; ++r) sum += cl.map_shared_rank(red, r)[c * S::ZC + lane];
      out[size_t(m0 * MYP + c) * a.nz] = sum;
    }
    cl.sync();                     // no CTA overwrites (or leaves) while its projection is still read
  }
}

// Back-projection of one (z chunk, x block): each thread forms, for its XPW x
// rows and its z, the MYP sums over the x modes (psi read from L2), then
// walks the y rows (pairs of mirror rows under FY) with the y-mode table in
// shared memory, writing phi one row of 32 z values per warp store.
template <typename T, int MYP, bool FY>
__device__ __forceinline__ void mode_back(const ModeArgs<T>& a, unsigned char* smem_raw) {
  using S = ModeShape<T>;
  const int nyk = FY ? a.ny / 2 : a.ny;
  T* ps = reinterpret_cast<T*>(smem_raw);           // psi chunk [mx * MYP][ZC]
  T* sy = ps + size_t(a.mx) * MYP * S::ZC;
  T* sxs = sy + nyk * MYP;                          // x-mode rows of the block [XB][mxp]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int z0 = int(blockIdx.x) * S::ZC;
  const int xb0 = int(blockIdx.y) * S::XB;
  const int x0 = xb0 + warp * S::XPW;
  {
    constexpr int PPR = S::ZC * int(sizeof(T)) / 16;
    for (int idx = threadIdx.x; idx < a.mx * MYP * PPR; idx += S::THREADS) {
      const int c = idx / PPR, piece = idx % PPR;
      cp_async16(reinterpret_cast<unsigned char*>(ps + size_t(c) * S::ZC) + 16 * piece,
                 reinterpret_cast<const unsigned char*>(a.psi + size_t(c) * a.nz + z0) + 16 * piece);
    }
    cp_async_commit();
  }
  for (int i = threadIdx.x; i < nyk * MYP; i += S::THREADS) sy[i] = a.sy[i];
  for (int i = threadIdx.x; i < S::XB * a.mxp; i += S::THREADS) sxs[i] = a.sx[size_t(xb0) * a.mxp + i];
  cp_async_wait<0>();
  __syncthreads();                 // psi chunk and tables in shared memory

  T bv[S::XPW][MYP];
#pragma unroll
  for (int i = 0; i < S::XPW; ++i)
#pragma unroll
    for (int n = 0; n < MYP; ++n) bv[i][n] = T(0);
#pragma unroll 2
  for (int m = 0; m < a.mx; ++m) {
    T s[S::XPW];
#pragma unroll
    for (int i = 0; i < S::XPW; ++i) s[i] = sxs[(warp * S::XPW + i) * a.mxp + m];
#pragma unroll
    for (int n = 0; n < MYP; ++n) {
      const T p = ps[(m * MYP + n) * S::ZC + lane];
#pragma unroll
      for (int i = 0; i < S::XPW; ++i) bv[i][n] = fma(s[i], p, bv[i][n]);
    }
  }

#pragma unroll 1
  for (int yh = 0; yh < nyk; ++yh) {
    const T* srow = sy + yh * MYP;
    T o[S::XPW], e[S::XPW];
#pragma unroll
    for (int i = 0; i < S::XPW; ++i) o[i] = e[i] = T(0);
#pragma unroll
    for (int g = 0; g < MYP; g += 4) {
      T s4[4];
      load4(srow + g, s4);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const bool odd_slot = !FY || (g + k < MYP / 2);
#pragma unroll
        for (int i = 0; i < S::XPW; ++i) {
          if (odd_slot) o[i] = fma(s4[k], bv[i][g + k], o[i]);
          else e[i] = fma(s4[k], bv[i][g + k], e[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < S::XPW; ++i) {
      T* row = a.phi + (size_t(x0 + i) * a.ny + yh) * a.nz + z0 + lane;
      if constexpr (FY) {
        row[0] = o[i] + e[i];
        row[size_t(a.ny - 1 - 2 * yh) * a.nz] = o[i] - e[i];
      } else {
        row[0] = o[i];
      }
    }
  }
}

}  // namespace pp
