// FP32 projection and back-projection of the mode-space solve, for every mesh:
// y mirror pairs about the mid-plane (cell-centred), mirror pairs with the first
// row on the wall, or no symmetry.
//
// A CTA of 4 or 8 warps (mode_shape) covers two x rows a warp and 32 consecutive
// z (one per lane), so every warp load or store of the fields is a run of 32 z
// values.
//   projection:      A[x][n][z] = sum_j Sy[j][n] rho[x][j][z]: the warp's field
//                    rows staged through a cp.async ring, a pair (j, mirror of
//                    j) giving u + v for the odd n and u - v for the even; then
//                    the x-mode sums over the CTA's rows,
//                    P[m][n][z] = sum_x Sx[x][m] A[x][n][z], written as one
//                    partial per group of `reps` x blocks (the z kernel adds
//                    them).  No reduction between CTAs: the thread-block
//                    clusters that this replaces kept every CTA of a one-wave
//                    grid in two cluster barriers while HBM idled.
//   back-projection: B[x][n][z] = sum_m Sx[x][m] psi[m][n][z] (psi chunk in
//                    shared memory, the warp's own two x rows), then
//                    phi[x][j][z] = O + E and phi[x][mirror][z] = O - E with O, E
//                    the sums of Sy[j][n] B[x][n][z] over odd and even n.
// All sums are FP32 FMAs, two at a time (fma.rn.f32x2).  Folded, a pair of
// slots is one odd and one even n: the data pair (u + v, u - v) and the result
// pair (O, E) then need no copies or additions across a pair; the y-mode table
// lies in shared memory in that order, four values a load, each load serving
// the warp's two x rows (tables too long for it are read through L1).
//
// The back-projection sums from the highest mode down: the terms of a potential
// fall with the mode, so the partial sums stay small until the last few
// additions.  From the first mode up every addition rounds at the size of the
// result, independently from node to node, which differences of the potential
// then show.  Error against 64 bits, up -> down: the potential at 128^2 x 1024
// 1.6e-7 -> 9.4e-8, deposit + solve + field at 64^2 x 256 1.6e-6 -> 7.4e-7, the
// energy's particle gradient at 128^2 x 512 7.7e-6 -> 4.0e-6; no time (40.9 us
// both at 128^2 x 1024).
//
// The x-mode sums ran as 3xTF32 MMA (mma.sync) before: the MMA's accumulation
// cuts instead of rounding, which doubled the error of the generic FP32 FMA
// kernels that this file also replaces, and splitting the operands cost more
// instructions than the FMAs.
//
// Bounds, 20 x 20 modes, us per launch back to back (before: the cluster kernels
// on ny = 32 .. 256 folded, generic 4-warp kernels elsewhere):
//   128^2 x 1024   project 25.2 -> 17.9, back 17.8 -> 16.3  (67 MB each: 10 us);
//                  of the projection 3 to 4 are the x-mode sums and their
//                  partials, when every CTA of the one wave leaves the stream
//   512^2 x 1024   project 303 -> 201, back 206 -> 172      (1.07 GB: 158 us)
//   48 x 80 x 512  project 29.0 -> 7.1, back 12.8 -> 7.4    (window: latency)
//   64^2 x 256     project 10.1 -> 5.8, back 8.4 -> 5.4     (latency)
// Ring depths of 3 to 6 stages differ by under 2 %.
#include "modes.cuh"
#include "modes_impl.cuh"

namespace pp {

namespace {

constexpr int XR = kModeRowsPerWarp;      // x rows per warp
constexpr int kZC = 32;                   // z values per CTA
constexpr int kRows = 8;                  // field rows of one x per ring stage (4 mirror pairs)
constexpr int kStages = 4;

// d = a * b + c on both halves of a pair (the packed FP32 FMA of sm_100 and
// later: one instruction for two FMAs, each rounded as fmaf)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// slot pair k: slots (k, myp/2 + k) folded (an odd and an even n), else (2k, 2k + 1)
template <int MYP, bool FOLD>
__device__ __forceinline__ constexpr int slot_of(int k, int half) {
  return FOLD ? k + half * (MYP / 2) : 2 * k + half;
}

// the y-mode table [rows][MYP] into shared memory, rows of slot pairs
template <int MYP, bool FOLD>
__device__ __forceinline__ void stage_table(float* stab, const float* sy, int rows) {
  for (int i = threadIdx.x; i < rows * (MYP / 2); i += int(blockDim.x)) {
    const int j = i / (MYP / 2), k = i % (MYP / 2);
    reinterpret_cast<float2*>(stab)[i] =
        make_float2(__ldg(sy + j * MYP + slot_of<MYP, FOLD>(k, 0)), __ldg(sy + j * MYP + slot_of<MYP, FOLD>(k, 1)));
  }
}
// row j of the table as slot pairs (TS: staged, else the table itself)
template <int MYP, bool FOLD, bool TS>
__device__ __forceinline__ void table_row(const float* tab, int j, float2 (&s)[MYP / 2]) {
  const float4* p = reinterpret_cast<const float4*>(tab + size_t(j) * MYP);
  float v[MYP];
#pragma unroll
  for (int q = 0; q < MYP / 4; ++q) {
    const float4 f = TS ? p[q] : __ldg(p + q);
    v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
  }
#pragma unroll
  for (int k = 0; k < MYP / 2; ++k)
    s[k] = TS ? make_float2(v[2 * k], v[2 * k + 1]) : make_float2(v[slot_of<MYP, FOLD>(k, 0)], v[slot_of<MYP, FOLD>(k, 1)]);
}

// floats of a warp's x row of A[x][n][z], and of its slot, which first is its ring
template <int MYP> constexpr int row_a() { return MYP * kZC; }
template <int MYP>
constexpr int slot_a() {
  return kStages * kRows * kZC > row_a<MYP>() ? XR * kStages * kRows * kZC : XR * row_a<MYP>();
}

template <int MYP>
constexpr size_t project_smem(int warps, int mxp, int table) {
  return sizeof(float) * (size_t(warps) * slot_a<MYP>() + warps * XR * mxp + table);
}
template <int MYP>
constexpr size_t back_smem(int warps, int mx, int mxp, int table) {
  return sizeof(float) * (size_t(mx) * MYP * kZC + warps * XR * mxp + table);
}

// P[m][n][z] = sum_x Sx[x][m] A[x][n][z] of the CTA's x rows for the slots n =
// warp, warp + warps, .., NB at a time (the last one again where a slot is
// missing, not stored), at most MQ quads of x modes.  Bound by the issue of the
// broadcast loads of Sx, one per two packed FMAs of a slot: two slots at a time
// halve them.
template <int MYP, int MQ, int NB>
__device__ __forceinline__ void x_modes(const float* abuf, const float* sxs, float* out, int mxp, int mq, int warps,
                                        int rows, size_t nz, bool add) {
  constexpr int RA = row_a<MYP>(), SL = slot_a<MYP>();
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int n0 = int(threadIdx.x) >> 5; n0 < MYP; n0 += NB * warps) {
    float2 p[NB][MQ][2];
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int q = 0; q < MQ; ++q) p[b][q][0] = p[b][q][1] = make_float2(0.f, 0.f);
    const float* av = abuf + n0 * kZC + lane;
    int step[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) step[b] = n0 + b * warps < MYP ? b * warps * kZC : 0;
#pragma unroll 2
    for (int x = 0; x < rows; ++x) {
      float2 v[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const float f = av[(x / XR) * SL + (x % XR) * RA + step[b]];
        v[b] = make_float2(f, f);
      }
      const float4* sx = reinterpret_cast<const float4*>(sxs + x * mxp);
#pragma unroll
      for (int q = 0; q < MQ; ++q)
        if (q < mq) {
          const float4 w = sx[q];
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            p[b][q][0] = ffma2(make_float2(w.x, w.y), v[b], p[b][q][0]);
            p[b][q][1] = ffma2(make_float2(w.z, w.w), v[b], p[b][q][1]);
          }
        }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (n0 + b * warps >= MYP) continue;
#pragma unroll
      for (int q = 0; q < MQ; ++q)
        if (q < mq) {
          float* d = out + size_t(4 * q * MYP + n0 + b * warps) * nz;
          const size_t ms = MYP * nz;
          float4 f = make_float4(p[b][q][0].x, p[b][q][0].y, p[b][q][1].x, p[b][q][1].y);
          if (add) {                                   // the same thread's sums of the blocks before
            f.x += d[0]; f.y += d[ms]; f.z += d[2 * ms]; f.w += d[3 * ms];
          }
          d[0] = f.x; d[ms] = f.y; d[2 * ms] = f.z; d[3 * ms] = f.w;
        }
    }
  }
}

// z chunk zc, x blocks grp * reps ..
template <int MYP, bool FOLD, bool TS>
__device__ __forceinline__ void project(const ModeArgs<float>& a, int zc, int grp, int reps) {
  constexpr int RA = row_a<MYP>(), SL = slot_a<MYP>(), H = MYP / 2;
  constexpr int kStage = XR * kRows * kZC;                     // floats of a stage
  const int kW = int(blockDim.x) / 32, kX = kW * XR;           // warps, x rows of the CTA
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* abuf = reinterpret_cast<float*>(smem_raw);            // [kW][SL]: rings, then A[x][n][z]
  float* sxs = abuf + kW * SL;                                 // [kX][mxp]: the block's x-mode rows
  float* stab = sxs + kX * a.mxp;                              // TS: the y-mode table
  const float* tab = TS ? stab : a.sy;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int z0 = zc * kZC;
  const int ns = a.ny / kRows;                                 // ring stages of a row
  float* ring = abuf + warp * SL;
  const size_t nz = size_t(a.nz), xs = size_t(a.ny) * nz;
  wait_stage();
  const int r4 = lane >> 3, piece = lane & 7;                  // this lane's row of a run of 4, 16-byte piece
#pragma unroll 1
  for (int rep = 0; rep < reps; ++rep) {
    const int xb0 = (grp * reps + rep) * kX;
    const float* xrow = a.rho + size_t(xb0 + XR * warp) * xs + z0 + 4 * piece;
    // stage s, per x: 8 rows from 8 s, or the pairs 4 s .. 4 s + 3 (4 rows, then their mirror rows)
    const float* lo = xrow + size_t(r4) * nz;
    const float* hi = FOLD ? xrow + size_t(a.mirror - r4) * nz : lo + 4 * nz;
    auto issue = [&](int s) __attribute__((always_inline)) {
      float* buf = ring + (s % kStages) * kStage + 4 * lane;
      const float* h = FOLD && a.wall && s == 0 && r4 == 0 ? xrow + size_t(a.wall) * nz : hi;
#pragma unroll
      for (int i = 0; i < XR; ++i) {
        cp_async16(buf + i * kRows * kZC, lo + i * xs);
        cp_async16(buf + (i * kRows + 4) * kZC, h + i * xs);
      }
      cp_async_commit();
      lo += (FOLD ? 4 : 8) * nz;
      if (FOLD) hi -= 4 * nz;
      else hi += 8 * nz;
    };
    float2 acc[XR][H];
#pragma unroll
    for (int i = 0; i < XR; ++i)
#pragma unroll
      for (int n = 0; n < H; ++n) acc[i][n] = make_float2(0.f, 0.f);
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) {
      if (s < ns) issue(s);
      else cp_async_commit();
    }
    // behind the first copies: the block's x-mode rows, and once the table
    for (int i = threadIdx.x; i < kX * a.mxp; i += int(blockDim.x)) sxs[i] = __ldg(a.sx + size_t(xb0) * a.mxp + i);
    if (TS && rep == 0) {
      stage_table<MYP, FOLD>(stab, a.sy, FOLD ? a.ny / 2 : a.ny);
      __syncthreads();
    }
#pragma unroll 1
    for (int s = 0; s < ns; ++s) {
      cp_async_wait<kStages - 2>();
      __syncwarp();
      if (s + kStages - 1 < ns) issue(s + kStages - 1);        // the buffer read at stage s - 1
      else cp_async_commit();
      const float* buf = ring + (s % kStages) * kStage + lane;
      if constexpr (FOLD) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          float2 sy[H];
          table_row<MYP, FOLD, TS>(tab, 4 * s + r, sy);
#pragma unroll
          for (int i = 0; i < XR; ++i) {
            float u = buf[(i * kRows + r) * kZC];
            const float v = buf[(i * kRows + 4 + r) * kZC];
            if (r == 0 && a.wall && s == 0) u *= 0.f;          // (a value that is not finite stays so)
            const float2 pq = make_float2(u + v, u - v);
#pragma unroll
            for (int n = 0; n < H; ++n) acc[i][n] = ffma2(sy[n], pq, acc[i][n]);
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          float2 sy[H];
          table_row<MYP, FOLD, TS>(tab, kRows * s + r, sy);
#pragma unroll
          for (int i = 0; i < XR; ++i) {
            const float u = buf[(i * kRows + r) * kZC];
            const float2 uu = make_float2(u, u);
#pragma unroll
            for (int n = 0; n < H; ++n) acc[i][n] = ffma2(sy[n], uu, acc[i][n]);
          }
        }
      }
    }
    cp_async_wait<0>();
    __syncwarp();                                              // ring reads done before A overwrites it
#pragma unroll
    for (int i = 0; i < XR; ++i)
#pragma unroll
      for (int n = 0; n < H; ++n) {
        ring[i * RA + slot_of<MYP, FOLD>(n, 0) * kZC + lane] = acc[i][n].x;
        ring[i * RA + slot_of<MYP, FOLD>(n, 1) * kZC + lane] = acc[i][n].y;
      }
    __syncthreads();

    // P[m][n][z]: up to 20 x modes the slots two at a time, beyond, where the sums
    // of two take 64 registers, one by one.  Projection at 128^2 x 1024, 64^2 x
    // 256 and 48 x 80 x 512 with 20 x modes: two at a time 17.9 / 5.8 / 7.1 us,
    // one 18.6 / 6.1 / 7.8, three 18.6 / 7.0 / 8.4, the form of 32 x modes for
    // all 19.6 / 6.7 / 8.1
    float* out = a.part + size_t(grp) * a.mc * nz + z0 + lane;
    const int mq = a.mxp / 4;
    if (mq <= 5) x_modes<MYP, 5, 2>(abuf, sxs, out, a.mxp, mq, kW, kX, nz, rep > 0);
    else x_modes<MYP, 8, 1>(abuf, sxs, out, a.mxp, mq, kW, kX, nz, rep > 0);
    if (rep + 1 < reps) __syncthreads();               // A and the x rows read before they are refilled
  }
}

template <int MYP, bool FOLD, bool TS>
__device__ __forceinline__ void back(const ModeArgs<float>& a, int zc, int xb) {
  constexpr int H = MYP / 2;
  const int kX = int(blockDim.x) / 32 * XR;          // x rows of the CTA
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* ps = reinterpret_cast<float*>(smem_raw);    // psi chunk [m][n][z]
  float* sxs = ps + size_t(a.mx) * MYP * kZC;        // [kX][mxp]: the block's x-mode rows
  float* stab = sxs + kX * a.mxp;                    // TS: the y-mode table
  const float* tab = TS ? stab : a.sy;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int z0 = zc * kZC, xb0 = xb * kX;
  const int nyk = FOLD ? a.ny / 2 : a.ny;
  const size_t nz = size_t(a.nz), xs = size_t(a.ny) * nz;
  for (int i = threadIdx.x; i < kX * a.mxp; i += int(blockDim.x)) sxs[i] = __ldg(a.sx + size_t(xb0) * a.mxp + i);
  if (TS) stage_table<MYP, FOLD>(stab, a.sy, nyk);
  wait_stage();
  for (int idx = threadIdx.x; idx < a.mx * MYP * (kZC / 4); idx += int(blockDim.x))
    cp_async16(ps + 4 * idx, a.psi + size_t(idx / (kZC / 4)) * nz + z0 + 4 * (idx % (kZC / 4)));
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();

  const int x0 = XR * warp;
  float2 bv[XR][H];
#pragma unroll
  for (int i = 0; i < XR; ++i)
#pragma unroll
    for (int n = 0; n < H; ++n) bv[i][n] = make_float2(0.f, 0.f);
#pragma unroll 2
  for (int m = a.mx - 1; m >= 0; --m) {              // (the small terms first, see the top)
    float2 s[XR];
#pragma unroll
    for (int i = 0; i < XR; ++i) s[i] = make_float2(sxs[(x0 + i) * a.mxp + m], sxs[(x0 + i) * a.mxp + m]);
    const float* p = ps + m * MYP * kZC + lane;
#pragma unroll
    for (int n = 0; n < H; ++n) {
      const float2 v = make_float2(p[slot_of<MYP, FOLD>(n, 0) * kZC], p[slot_of<MYP, FOLD>(n, 1) * kZC]);
#pragma unroll
      for (int i = 0; i < XR; ++i) bv[i][n] = ffma2(s[i], v, bv[i][n]);
    }
  }

  float* lo[XR];
  float* hi[XR];
#pragma unroll
  for (int i = 0; i < XR; ++i) {
    lo[i] = a.phi + size_t(xb0 + x0 + i) * xs + z0 + lane;
    hi[i] = lo[i] + size_t(a.mirror) * nz;
  }
  // the pair sums (O, E), or halves of the sum, of row j for x row i
  auto sums = [&](const float2 (&sy)[H], int i) __attribute__((always_inline)) {
    float2 o = make_float2(sy[H - 1].x * bv[i][H - 1].x, sy[H - 1].y * bv[i][H - 1].y);
#pragma unroll
    for (int n = H - 2; n >= 0; --n) o = ffma2(sy[n], bv[i][n], o);
    return o;
  };
  int j = 0;
  if (FOLD && a.wall) {                              // pair 0: the wall row is zero, row `wall` its own mirror
    float2 sy[H];
    table_row<MYP, FOLD, TS>(tab, 0, sy);
#pragma unroll
    for (int i = 0; i < XR; ++i) {
      const float2 o = sums(sy, i);
      *lo[i] = 0.f * o.x;
      lo[i][size_t(a.wall) * nz] = o.x - o.y;
      lo[i] += nz;
      hi[i] -= nz;
    }
    j = 1;
  }
#pragma unroll 4
  for (; j < nyk; ++j) {
    float2 sy[H];
    table_row<MYP, FOLD, TS>(tab, j, sy);
#pragma unroll
    for (int i = 0; i < XR; ++i) {
      const float2 o = sums(sy, i);
      *lo[i] = o.x + o.y;
      lo[i] += nz;
      if (FOLD) {
        *hi[i] = o.x - o.y;
        hi[i] -= nz;
      }
    }
  }
}

// grid (n * nz / 32, groups) and (n * nz / 32, x blocks): one solve (g.n = 0, n =
// 1) with its arguments in `one`, or a group of solves of one shape, solve s
// taking the z chunks s * nz/32 ..; the same arithmetic per solve
__device__ __forceinline__ ModeArgs<float> solve_args(const ModeArgs<float>& one, const ModeGroup& g, int& zc) {
  zc = int(blockIdx.x);
  if (g.n == 0) return one;
  const int zpc = g.nz / kZC, s = zc / zpc;
  zc -= s * zpc;
  ModeArgs<float> a = g.args[s];
  a.rho = g.rho[s];
  a.phi = g.phi[s];
  return a;
}
template <int MYP, bool FOLD, bool TS>
__global__ void __launch_bounds__(256, 2) mode_project_kernel(const __grid_constant__ ModeArgs<float> one,
                                                              const __grid_constant__ ModeGroup g, int reps) {
  int zc;
  const ModeArgs<float> a = solve_args(one, g, zc);
  project<MYP, FOLD, TS>(a, zc, int(blockIdx.y), reps);
}
template <int MYP, bool FOLD, bool TS>
__global__ void __launch_bounds__(256, MYP <= 24 ? 3 : 2) mode_back_kernel(const __grid_constant__ ModeArgs<float> one,
                                                           const __grid_constant__ ModeGroup g) {
  int zc;
  const ModeArgs<float> a = solve_args(one, g, zc);
  back<MYP, FOLD, TS>(a, zc, int(blockIdx.y));
}

template <typename K>
cudaError_t big_smem(K kern, size_t smem) {
  if (smem > kMaxSmem) return cudaErrorInvalidConfiguration;
  if (smem <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
}

// The y-mode table goes to shared memory while two CTAs still fit in an SM's;
// beyond (unfolded rows and many modes: ny above about 600) it is read through L1.
constexpr size_t kTableSmem = 113 * 1024;

template <int MYP, bool FOLD, bool TS>
cudaError_t launch_sums(int stage, const ModeArgs<float>& a, const ModeGroup& g, const ModeShape& sh, cudaStream_t st) {
  const int table = TS ? (FOLD ? a.ny / 2 : a.ny) * MYP : 0;
  const unsigned gx = unsigned((g.n ? g.n : 1) * (a.nz / kZC));
  cudaError_t e;
  if (stage == 0) {
    const size_t smem = project_smem<MYP>(sh.warps, a.mxp, table);
    if ((e = big_smem(mode_project_kernel<MYP, FOLD, TS>, smem)) != cudaSuccess) return e;
    return launch_stage(mode_project_kernel<MYP, FOLD, TS>, dim3(gx, unsigned(sh.groups)), 32 * sh.warps, smem, st, a, g, sh.reps);
  }
  const size_t smem = back_smem<MYP>(sh.warps, a.mx, a.mxp, table);
  if ((e = big_smem(mode_back_kernel<MYP, FOLD, TS>, smem)) != cudaSuccess) return e;
  return launch_stage(mode_back_kernel<MYP, FOLD, TS>, dim3(gx, unsigned(a.nx / (sh.warps * XR))), 32 * sh.warps, smem,
                      st, a, g);
}

template <int MYP, bool FOLD>
cudaError_t launch_sums2(int stage, const ModeArgs<float>& a, const ModeGroup& g, cudaStream_t st) {
  const ModeShape sh = mode_shape(a.nx, a.nz, a.mc);
  const int table = (FOLD ? a.ny / 2 : a.ny) * MYP;
  const size_t smem = stage == 0 ? project_smem<MYP>(sh.warps, a.mxp, table) : back_smem<MYP>(sh.warps, a.mx, a.mxp, table);
  return smem <= kTableSmem ? launch_sums<MYP, FOLD, true>(stage, a, g, sh, st)
                            : launch_sums<MYP, FOLD, false>(stage, a, g, sh, st);
}

cudaError_t launch_sums_any(int stage, int myp, bool fold, const ModeArgs<float>& a, const ModeGroup& g,
                            cudaStream_t st) {
  switch (myp) {
    case 8: return fold ? launch_sums2<8, true>(stage, a, g, st) : launch_sums2<8, false>(stage, a, g, st);
    case 12: return fold ? launch_sums2<12, true>(stage, a, g, st) : launch_sums2<12, false>(stage, a, g, st);
    case 16: return fold ? launch_sums2<16, true>(stage, a, g, st) : launch_sums2<16, false>(stage, a, g, st);
    case 20: return fold ? launch_sums2<20, true>(stage, a, g, st) : launch_sums2<20, false>(stage, a, g, st);
    case 24: return fold ? launch_sums2<24, true>(stage, a, g, st) : launch_sums2<24, false>(stage, a, g, st);
    case 32: return fold ? launch_sums2<32, true>(stage, a, g, st) : launch_sums2<32, false>(stage, a, g, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_mode_sums(int stage, int myp, bool fold, const ModeArgs<float>& a, cudaStream_t st) {
  return launch_sums_any(stage, myp, fold, a, ModeGroup{}, st);
}

cudaError_t launch_mode_sums_group(int stage, int myp, bool fold, const ModeArgs<float>& a, const ModeGroup& g,
                                   cudaStream_t st) {
  if (g.n < 1 || g.n > kMaxModeGroup) return cudaErrorInvalidValue;
  return launch_sums_any(stage, myp, fold, a, g, st);
}

}  // namespace pp
