// z stage of the mode-space solve (the method is described in modes_impl.cuh):
// the banded operator's stencil, or the recurrences of modes_z.cu.
#include <type_traits>

#include "modes.cuh"
#include "modes_impl.cuh"

namespace pp {

// Banded z stage (Sec. 5, Eq. 17-18 in mode space): psi[c][k] =
// sum_{|d| <= nb, 0 <= k-d < nz} K_c(|d|) rhot[c][k-d], rhot the groups' partial
// projections summed.  One CTA per column: the column (zero-padded by nb on
// both sides) and its taps in shared memory, taps summed from d = -nb up.
constexpr int kBandThreads = 256;

template <typename T>
__global__ void __launch_bounds__(kBandThreads) mode_band_kernel(ModeArgs<T> a, int groups) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* win = reinterpret_cast<T*>(smem_raw);           // [nz + 2 nb]: win[nb + k] = rhot[k]
  T* taps = win + a.nz + 2 * a.nb;                   // [nb + 1]
  const int c = int(blockIdx.x);
  wait_stage();
  for (int i = int(threadIdx.x); i < a.nb; i += kBandThreads) win[i] = win[a.nb + a.nz + i] = T(0);
  // the column summed over the groups (in group order, from zero), 16 bytes a
  // load, every group's load of a piece in flight together (nz is a power of
  // two >= 32, so the pieces tile it and stay 16-byte aligned)
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  constexpr int EV = 16 / sizeof(T);
  for (int q = int(threadIdx.x); q < a.nz / EV; q += kBandThreads) {
    T v[EV];
#pragma unroll
    for (int e = 0; e < EV; ++e) v[e] = T(0);
#pragma unroll 4
    for (int s = 0; s < groups; ++s) {
      const V p = reinterpret_cast<const V*>(a.part + (size_t(s) * a.mc + c) * a.nz)[q];
      const T* pe = reinterpret_cast<const T*>(&p);
#pragma unroll
      for (int e = 0; e < EV; ++e) v[e] += pe[e];
    }
#pragma unroll
    for (int e = 0; e < EV; ++e) win[a.nb + q * EV + e] = v[e];
  }
  for (int d = int(threadIdx.x); d <= a.nb; d += kBandThreads) taps[d] = a.kb[size_t(c) * (a.nb + 1) + d];
  __syncthreads();
  for (int k = int(threadIdx.x); k < a.nz; k += kBandThreads) {
    const T* w = win + k + a.nb;                     // w[-d] = rhot[k - d]
    T acc = T(0);
    for (int d = -a.nb; d <= a.nb; ++d) acc += taps[d < 0 ? -d : d] * w[-d];
    a.psi[size_t(c) * a.nz + k] = acc;
  }
}

namespace {

template <typename T>
cudaError_t launch_band(const ModeArgs<T>& a, cudaStream_t st) {
  const size_t smem = sizeof(T) * (size_t(a.nz) + 3 * size_t(a.nb) + 1);
  void (*kern)(ModeArgs<T>, int) = mode_band_kernel<T>;
  if (smem > 48 * 1024) {
    if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
  }
  return launch_stage(kern, dim3(unsigned(a.mc)), kBandThreads, smem, st, a, a.groups);
}

}  // namespace

template <typename T>
cudaError_t launch_mode_z_stage(const ModeArgs<T>& a, cudaStream_t st) {
  if (a.nz < 32 || a.nz > 1024 || (a.nz & (a.nz - 1))) return cudaErrorInvalidValue;
  return a.nb >= 0 ? launch_band<T>(a, st) : launch_mode_z<T>(a, a.groups, st);
}
template cudaError_t launch_mode_z_stage<float>(const ModeArgs<float>&, cudaStream_t);
template cudaError_t launch_mode_z_stage<double>(const ModeArgs<double>&, cudaStream_t);

}  // namespace pp
