// z convolution of the mode-space solve, psi[c][k] = sum_k' K_c(k - k') rhot[c][k'],
// as a pair of first-order recurrences.
//
// The kernel of a mode is a two-sided exponential with its own centre tap:
// with q = e^{-kappa hz}, K_c(d) = gamma q^{d-1} for d >= 1 (Eq. 9, and the
// longitudinal IGF of Eq. 15-16 at |w| >= hz) and K_c(0) = beta.  So the
// zero-padded convolution of Appendix A is, exactly,
//     psi_k = beta rhot_k + gamma (F_{k-1} + B_{k+1}),
//     F_k = rhot_k + q F_{k-1},   B_k = rhot_k + q B_{k+1},   F_{-1} = B_{nz} = 0,
// 9 operations a value instead of two padded FFTs.  (It replaced a warp-level
// four-step FFT in FP32 and a Stockham FFT in FP64.  A 128^2 x 1024 solve, 400
// columns, back to back: FP32 53.5 -> 50.3 us, its error against 64 bits
// 3.3e-7 -> 2.4e-7; FP64 1076 -> 1005 us, 1.6e-15 -> 3.6e-16.)
//
// A thread takes kV consecutive z of a column and a column nz / kV threads:
// both recurrences over the thread's values from zero, an inclusive scan of
// the threads' totals by shuffles (multipliers q^{kV 2^i}), across the warps
// of a column through shared memory, then the recurrences again from the
// incoming states.  kV = 8 keeps a load two 16-byte pieces of a run and gives
// 4 warps a column at nz = 1024; the kernel is bound by latency (one round
// trip of loads, the scan) and, in FP64, by the FP64 pipe.
//
// Precision.  beta, gamma, 1 - q and the multipliers are tabulated in FP64.
// FP32 steps take F <- (F - (1 - q) F) + x: q itself, rounded, would be wrong
// by its last bit per step, a systematic error where kappa hz is small.  (FP64
// too was measured so: the same errors, 3 us more of the FP64 pipe.)
#include <type_traits>

#include "modes.cuh"
#include "modes_impl.cuh"

namespace pp {

namespace {

constexpr int kV = kModeZRun;                     // z values per thread
constexpr int kZThreads = 128;                    // threads per CTA

// one step of a recurrence: x + q s  (FP32: p = 1 - q, FP64: p = q)
__device__ __forceinline__ float zstep(float s, float x, float p) { return fmaf(-p, s, s) + x; }
__device__ __forceinline__ double zstep(double s, double x, double p) { return fma(p, s, x); }

// CTA `blk` of a solve: its columns blk * (1024 / NZ) ..
template <typename T, int NZ>
__device__ __forceinline__ void z_scan(const ModeArgs<T>& a, int groups, int blk) {
  constexpr int TC = NZ / kV;                     // threads per column
  constexpr int CPC = kZThreads / TC;             // columns per CTA
  constexpr int SEG = TC < 32 ? TC : 32;          // lanes of a warp on one column
  constexpr int NW = TC / SEG;                    // warps per column
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  constexpr int EV = 16 / int(sizeof(T));         // values per 16-byte piece
  __shared__ T tot[2][kZThreads / 32];
  const int cl = int(threadIdx.x) / TC, t = int(threadIdx.x) % TC;
  const int ls = t % SEG, wq = t / SEG;
  const int col = blk * CPC + cl;
  const bool valid = col < a.mc;
  const T* zp = a.zp + size_t(valid ? col : 0) * kModeZPar;
  T par[kModeZPar];
#pragma unroll
  for (int i = 0; i < kModeZPar / EV; ++i) *reinterpret_cast<V*>(par + EV * i) = __ldg(reinterpret_cast<const V*>(zp) + i);
  const T beta = par[0], gamma = par[1], p = sizeof(T) == 4 ? par[2] : par[3];
  const T* w = par + 4;                           // w[i] = q^{kV 2^i}

  wait_stage();
  // the column's values, the groups of partial projections summed with the
  // rounding errors of the additions carried along (Knuth's TwoSum): the partial
  // sums of a density that changes sign can cancel
  T x[kV], c[kV];
#pragma unroll
  for (int j = 0; j < kV; ++j) x[j] = c[j] = T(0);
  if (valid) {
#pragma unroll 8
    for (int s = 0; s < groups; ++s) {
      const V* src = reinterpret_cast<const V*>(a.part + (size_t(s) * a.mc + col) * NZ + t * kV);
      T g[kV];
#pragma unroll
      for (int i = 0; i < kV / EV; ++i) *reinterpret_cast<V*>(g + EV * i) = src[i];
#pragma unroll
      for (int j = 0; j < kV; ++j) {
        const T sum = x[j] + g[j], d = sum - x[j];
        if (sizeof(T) == 4) c[j] += (x[j] - (sum - d)) + (g[j] - d);      // FP64 writes one partial
        x[j] = sum;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < kV; ++j) x[j] += c[j];
  // totals of the thread's values, then of all threads up to this one
  T sf = x[0], sb = x[kV - 1];
#pragma unroll
  for (int j = 1; j < kV; ++j) {
    sf = zstep(sf, x[j], p);
    sb = zstep(sb, x[kV - 1 - j], p);
  }
#pragma unroll
  for (int i = 0; (1 << i) < SEG; ++i) {
    const int d = 1 << i;
    const T uf = __shfl_up_sync(0xffffffffu, sf, d, SEG), ub = __shfl_down_sync(0xffffffffu, sb, d, SEG);
    if (ls >= d) sf = fma(w[i], uf, sf);
    if (ls + d < SEG) sb = fma(w[i], ub, sb);
  }
  T F = __shfl_up_sync(0xffffffffu, sf, 1, SEG), B = __shfl_down_sync(0xffffffffu, sb, 1, SEG);
  if (ls == 0) F = T(0);
  if (ls == SEG - 1) B = T(0);
  if constexpr (NW > 1) {                         // the other warps of the column
    const int warp = int(threadIdx.x) / 32, w0 = warp - wq;
    if (ls == SEG - 1) tot[0][warp] = sf;
    if (ls == 0) tot[1][warp] = sb;
    __syncthreads();
    T cf = T(0), cb = T(0);
#pragma unroll
    for (int u = 0; u < NW - 1; ++u) {
      if (u < wq) cf = fma(w[5], cf, tot[0][w0 + u]);
      if (NW - 1 - u > wq) cb = fma(w[5], cb, tot[1][w0 + NW - 1 - u]);
    }
    T pf = T(1), pb = T(1);                       // q^{kV ls}, q^{kV (31 - ls)}
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      if (ls >> i & 1) pf *= w[i];
      else pb *= w[i];
    }
    F = fma(pf, cf, F);
    B = fma(pb, cb, B);
  }
  T f[kV];
#pragma unroll
  for (int j = 0; j < kV; ++j) {
    f[j] = F;
    F = zstep(F, x[j], p);
  }
#pragma unroll
  for (int j = kV - 1; j >= 0; --j) {
    f[j] = fma(gamma, f[j] + B, beta * x[j]);
    B = zstep(B, x[j], p);
  }
  if (valid) {
    V* dst = reinterpret_cast<V*>(a.psi + size_t(col) * NZ + t * kV);
#pragma unroll
    for (int i = 0; i < kV / EV; ++i) dst[i] = *reinterpret_cast<const V*>(f + EV * i);
  }
}

template <typename T, int NZ>
__global__ void __launch_bounds__(kZThreads) mode_z_kernel(ModeArgs<T> a, int groups) {
  z_scan<T, NZ>(a, groups, int(blockIdx.x));
}

// a group of solves of one shape: solve s takes the CTAs s * cps .. (s + 1) * cps - 1
template <int NZ>
__global__ void __launch_bounds__(kZThreads) mode_z_group_kernel(const __grid_constant__ ModeGroup g, int groups,
                                                                 int cps) {
  const ModeArgs<float> a = g.args[int(blockIdx.x) / cps];
  z_scan<float, NZ>(a, groups, int(blockIdx.x) % cps);
}

template <typename T, int NZ>
cudaError_t launch_z_nz(const ModeArgs<T>& a, int groups, const ModeGroup* g, cudaStream_t st) {
  constexpr int per = kZThreads * kV / NZ;        // columns per CTA
  const int cps = (a.mc + per - 1) / per;         // CTAs per solve
  if constexpr (sizeof(T) == 4) {
    if (g) {
      return launch_stage(mode_z_group_kernel<NZ>, dim3(unsigned(g->n * cps)), kZThreads, 0, st, *g, groups, cps);
    }
  }
  return launch_stage(mode_z_kernel<T, NZ>, dim3(unsigned(cps)), kZThreads, 0, st, a, groups);
}

template <typename T>
cudaError_t launch_z_any(const ModeArgs<T>& a, int groups, const ModeGroup* g, cudaStream_t st) {
  switch (a.nz) {
    case 32: return launch_z_nz<T, 32>(a, groups, g, st);
    case 64: return launch_z_nz<T, 64>(a, groups, g, st);
    case 128: return launch_z_nz<T, 128>(a, groups, g, st);
    case 256: return launch_z_nz<T, 256>(a, groups, g, st);
    case 512: return launch_z_nz<T, 512>(a, groups, g, st);
    case 1024: return launch_z_nz<T, 1024>(a, groups, g, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

template <typename T>
cudaError_t launch_mode_z(const ModeArgs<T>& a, int groups, cudaStream_t st) {
  return launch_z_any<T>(a, groups, nullptr, st);
}
template cudaError_t launch_mode_z<float>(const ModeArgs<float>&, int, cudaStream_t);
template cudaError_t launch_mode_z<double>(const ModeArgs<double>&, int, cudaStream_t);

cudaError_t launch_mode_z_group(const ModeArgs<float>& a, int groups, const ModeGroup& g, cudaStream_t st) {
  if (g.n < 1 || g.n > kMaxModeGroup) return cudaErrorInvalidValue;
  return launch_z_any<float>(a, groups, &g, st);
}

}  // namespace pp
