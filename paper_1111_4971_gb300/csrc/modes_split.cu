// FP64 projection and back-projection of the mode-space solve on the tensor
// cores, as exact integer products.
//
// GB300's FP64 pipe does 2 FMAs per clock and SM (1.1 TFLOP/s in all), so the
// FP64 mode sums were bound by it: 512 of 520 us of a 128^2 x 1024 projection.
// Here every FP64 factor is split into 6 signed digits of 9 bits (54 bits
// below the largest value it is summed with; the scheme of Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", 2012), each digit a small integer that
// FP16 holds exactly.  Digit products are summed by FP16 MMA with FP32
// accumulators.  The products d_i t_j with i + j <= 5 are kept, 21 of 36: each one
// dropped is below 2^-54 of the largest term, the rounding of one FP64 product.
// The sums of the weights i + j = 0 .. 4 are exact, at most 2^24: how many rows go
// into one set of accumulators, 64 unless a table's digits are all large, follows
// from the table (contract_steps; |d_i| <= 256, |d_0| <= 512 for a folded pair); the
// expansion has 16 terms (32 unfolded, 32 (1024 + 4 256) 256 <= 2^24).  Those of weight
// 5 may pass 2^24 and lose their last bit, 2^-61 of a largest term.  The six sums
// are put together in 64-bit integers and rounded to FP64 once; half of the
// outputs are converted on the FP64 pipe, which else adds once per 64 rows.
//
// Two kernels, used for y and for x in turn; one warp per (outer index, 16
// consecutive z), no barrier beyond the warp:
//   contract: out[r][z] = sum_k T[k][r] in[k][z]   (K rows or mirror pairs long)
//             projection: rho -> half[x][n][z] (k = y), half -> P[m][n][z] (k = x)
//   expand:   out[r][z] = sum_k T[r][k] in[k][z]   (k the modes, at most 32)
//             back-projection: psi -> half[x][n][z] (k = m), half -> phi (k = n)
// mma.m16n8k16: rows of A are 16 z (row g is z = 2g, row g + 8 is z = 2g + 1,
// so that a lane's values are one 16-byte piece of a run of 128), columns of B
// are 8 table columns.  The table's digits come as ready fragments (three
// 16-byte loads per lane, L1 hits shared by the CTA's warps).
//
// The scale is a power of two per z plane of a warp's tile, the exponent of the
// plane's largest value over the rows: planes are independent in both sums, so a
// plane's accuracy is its own, whatever the 15 beside it hold (one scale a tile
// left a plane 2^k below its tile 54 - k bits).  A lane holds two planes, as rows
// g and g + 8 of A and of the accumulators; their maxima go over the four lanes of
// equal g by shuffles.  The tile is read twice, first for the maxima, then for the
// digits.
// A table row has a power of two of its own too (table_scales): next to a wall
// every sine of a row is small, and digits of the sines themselves would cut them
// 2^-54 below 1, not below the row (100 u of the row's terms where its largest
// sine is 0.005).  The expansion takes it off its output's exponent, the
// contraction off the value's; a row that is zero, on the wall, takes no part in
// the maxima.  Both together against one scale a tile: projection and
// back-projection at 128^2 x 1024 90.5 + 70.9 -> 86.4 + 71.8 us, 256^2 x 512 on the
// wall 190 + 128 -> 180 + 130, 48 x 80 x 512 21.4 + 18.4 -> 20.9 + 19.0: branches on
// a plane's exponent go by a vote, and the warp's index is broadcast, so that what
// follows from them stays in uniform registers (without: 105 us for the first).
// Splitting costs some 45 integer instructions a value and putting an output
// together some 30.  No pipe is full (along y: ALU 51 and 53 % busy, issue 48 and
// 51 %, tensor 22 and 38 %, DRAM 25 and 22 %): what bounds the kernels is latency,
// with 11 warps an SM (the contraction's 96 accumulators) and 14.  128^2 x 1024, 20
// x 20 modes, ncu, against FP64 FMAs: projection 516 -> 70 + 24 us (y, x),
// back-projection 468 -> 21 + 54; the solve 1005 -> 162 us, and 256^2 x 512 with
// nodes on the wall (which folds too) 3230 -> 284.
// Error against 64 bits, relative L2: 4 to 5e-16 over such meshes, the FP64 FMA
// sums' 4 to 7e-16.  Relative to the first row alone, for a bunch at the mesh's
// centre, whose potential is small there: 3.2e-15 at 128 rows and 3.4e-15 at 512
// (without the rows' scales 1.6e-14 and 6.9e-14, FMAs 0.7e-15 and 0.8e-15): an
// entry far below its row's largest sine still has the row's cut.
//
// Values that are not finite give NaN in every output of their z plane (a stage
// run by itself, pipe_stage_modes: of their 16 planes).
#include <cuda_fp16.h>

#include <utility>

#include "modes_impl.cuh"
#include "modes_split.cuh"

namespace pp {

namespace {

constexpr int kD = kSplitDigits;
constexpr int kSplitWarps = 4;                       // warps per CTA
constexpr int kSeg = 64;                             // rows of a warp's tile

constexpr long long kBiasLow = kSplitBiasLow, kBias = kSplitBias;
// a contraction's values keep kGuard more bits until their digits are taken, and
// are rounded there: cut off, they would all move towards zero, an error that a
// sum does not average out
constexpr int kGuard = 4;
constexpr long long kGuardBias = (kBias << kGuard) + (1LL << (kGuard - 1));

__device__ __forceinline__ unsigned hi32(unsigned long long v) { return unsigned(v >> 32); }
__device__ __forceinline__ unsigned long long pack64(unsigned hi, unsigned lo) {
  return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// magnitude and sign (0 or -1) of x 2^(1075 + kGuard - e), cut to an integer
// below 2^(53 + kGuard); top = e 2^20; the exponent field of x is at most e, e >= 64
// (zeros and subnormal values are then shifted out)
struct Fixed {
  unsigned long long v;      // magnitude XOR sign
  int s;
};
__device__ __forceinline__ Fixed to_fixed(double x, unsigned top) {
  const int hi = __double2hiint(x);
  const unsigned sh = min((top - (unsigned(hi) & 0x7ff00000u)) >> 20, 63u);
  const unsigned long long m = (pack64((unsigned(hi) & 0xfffffu) | 0x100000u, unsigned(__double2loint(x))) << kGuard) >> sh;
  const int s = hi >> 31;
  return {m ^ static_cast<unsigned long long>(static_cast<long long>(s)), s};
}
// sum and difference of two such values, biased
// (the signs' part of the two's complements fits the bias's low word)
__device__ __forceinline__ unsigned long long bias_plus(int d) {
  return pack64(unsigned(kGuardBias >> 32), unsigned(kGuardBias & 0xffffffffLL) + unsigned(d));
}
__device__ __forceinline__ unsigned long long fixed_sum(const Fixed& a, const Fixed& b) {
  return a.v + b.v + bias_plus(-a.s - b.s);
}
__device__ __forceinline__ unsigned long long fixed_difference(const Fixed& a, const Fixed& b) {
  return a.v - b.v + bias_plus(b.s - a.s);
}
__device__ __forceinline__ unsigned long long fixed_value(const Fixed& a) { return a.v + bias_plus(-a.s); }

__device__ __forceinline__ unsigned hsub(unsigned u, unsigned off) {
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&u), *reinterpret_cast<const __half2*>(&off));
  return *reinterpret_cast<const unsigned*>(&h);
}
// digits of two biased values (a: low halves, b: high halves) as FP16 pairs.  A
// field (above G guard bits) at bit 0 of a half word is or-ed into FP16 1024 (1024 + field), one at
// bit 1 into FP16 512 (whose last place is 1/2: 512 + field).
template <int G>
__device__ __forceinline__ void digits(unsigned long long a, unsigned long long b, unsigned (&d)[kD]) {
  const unsigned a0 = unsigned(a >> G), b0 = unsigned(b >> G);                  // fields 5, 4 at 0, 9
  const unsigned a1 = unsigned(a >> (18 + G)), b1 = unsigned(b >> (18 + G));    // fields 3, 2
  const unsigned a2 = hi32(a) >> (4 + G), b2 = hi32(b) >> (4 + G);              // field 1
  auto even = [](unsigned x, unsigned y) { return hsub((__byte_perm(x, y, 0x5410) & 0x01ff01ffu) | 0x64006400u, 0x65006500u); };
  auto odd = [](unsigned x, unsigned y) { return hsub((__byte_perm(x, y, 0x6521) & 0x03fe03feu) | 0x60006000u, 0x62006200u); };
  d[5] = even(a0, b0);
  d[4] = odd(a0, b0);
  d[3] = even(a1, b1);
  d[2] = odd(a1, b1);
  d[1] = even(a2, b2);
  // the leading field is 0 .. 1024: added, not or-ed, to the FP16 pattern of 1024
  d[0] = hsub(__byte_perm(hi32(a) >> (13 + G), hi32(b) >> (13 + G), 0x5410) + 0x64006400u, 0x66006600u);
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_from(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1, float c) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c));
}

// acc[s] += sum_{i + j = s} A_i B_j for one k step; A digits [i][4], the table's
// fragments at tb (kD / 2 pieces, 32 apart).  The 21 products go in an order
// that keeps three others between two of one weight (a dependent MMA waits 22
// clocks, an independent one 8).  FIRST: the sums start from c.
constexpr int kProducts = kD * (kD + 1) / 2;
__host__ __device__ constexpr int product_weight(int p) {
  constexpr int w[kProducts] = {5, 4, 3, 5, 2, 4, 5, 3, 1, 4, 5, 2, 3, 5, 4, 0, 5, 3, 4, 1, 2};
  return w[p];
}
__host__ __device__ constexpr int product_digit(int p) {        // i: earlier products of its weight
  int n = 0;
  for (int q = 0; q < p; ++q) n += product_weight(q) == product_weight(p);
  return n;
}
template <bool FIRST, int P>
__device__ __forceinline__ void mma_product(float (&acc)[kD][4], const unsigned (&A)[kD][4], const uint4 (&b)[kD / 2], float c) {
  constexpr int s = product_weight(P), i = product_digit(P), j = s - i;
  const unsigned b0 = j & 1 ? b[j / 2].z : b[j / 2].x, b1 = j & 1 ? b[j / 2].w : b[j / 2].y;
  if constexpr (FIRST && i == 0) mma_f16_from(acc[s], A[i], b0, b1, c);
  else mma_f16(acc[s], A[i], b0, b1);
}
template <bool FIRST, int... P>
__device__ __forceinline__ void mma_products(float (&acc)[kD][4], const unsigned (&A)[kD][4], const uint4 (&b)[kD / 2], float c,
                                             std::integer_sequence<int, P...>) {
  (mma_product<FIRST, P>(acc, A, b, c), ...);
}
template <bool FIRST>
__device__ __forceinline__ void mma_split(float (&acc)[kD][4], const unsigned (&A)[kD][4], const uint4* tb, float c = 0.f) {
  uint4 b[kD / 2];
#pragma unroll
  for (int i = 0; i < kD / 2; ++i) b[i] = __ldg(tb + 32 * i);
  mma_products<FIRST>(acc, A, b, c, std::make_integer_sequence<int, kProducts>{});
}

// a b + c with a 64-bit product
__device__ __forceinline__ unsigned long long mad_wide(unsigned a, unsigned b, unsigned long long c) {
  unsigned long long r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ long long mad_wide_s(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// v 2^e rounded to nearest, |v| < 2^63 and -1000 < e < 900 (no result is then
// subnormal or overflows): by integer arithmetic (halves away from zero), or,
// CVT, by the conversion instruction, which runs at 2 lanes a clock and SM: a
// kernel gives half of its outputs to each.  Other exponents: Exponent's e,
// then a factor of 2^300 or 2^-300 (e may then still lose a table row's scale).
struct Exponent {
  int e20, extra;            // e 2^20; for values that are not finite, extra is kNan
  static constexpr int kNan = 1;
  __device__ __forceinline__ Exponent(int x, bool finite) : extra(0) {
    if (x <= kMaxRowScale - 1000) extra = -300;
    if (x >= 900) extra = finite ? 300 : kNan;
    e20 = (x - extra) * (1 << 20);
  }
};
// v 2^extra, or NaN (a call, so that it is branched around and not predicated: the
// FP64 pipe would be taken all the same)
__device__ __noinline__ double2 rescale(double2 v, int extra0, int extra1) {
  auto factor = [](int extra) {
    if (extra == Exponent::kNan) return __longlong_as_double(0x7ff8000000000000LL);
    return extra == 0 ? 1.0 : (extra < 0 ? 0x1p-300 : 0x1p300);
  };
  return make_double2(v.x * factor(extra0), v.y * factor(extra1));
}
template <bool CVT>
__device__ __forceinline__ double to_double(long long v, int e20) {
  if constexpr (CVT) {
    const double d = __ll2double_rn(v);
    const int h = __double2hiint(d);
    return __hiloint2double(h != 0 ? h + e20 : 0, __double2loint(d));
  } else {
    const int s = int(v >> 63);
    const unsigned long long u = static_cast<unsigned long long>((v ^ s) - s);
    const int lz = __clzll(static_cast<long long>(u));               // >= 1; 64 for zero
    const unsigned long long r = ((u << (lz - 1)) + 0x200u) >> 10;   // 53 bits, the first is the implicit one
    const unsigned h = (hi32(r) + unsigned(e20) + (unsigned(1085 - lz) << 20)) | (unsigned(s) & 0x80000000u);
    return __hiloint2double(lz == 64 ? 0 : int(h), int(unsigned(r)));
  }
}

// Per z plane of a lane (x: plane 2g, y: plane 2g + 1): the larger of m and the
// high words of v, signs off; and the larger (the union) over the four lanes
// that hold the plane
__device__ __forceinline__ uint2 absmax(uint2 m, double2 v) {
  return make_uint2(max(m.x, unsigned(__double2hiint(v.x)) & 0x7fffffffu),
                    max(m.y, unsigned(__double2hiint(v.y)) & 0x7fffffffu));
}
__device__ __forceinline__ uint2 plane_max(uint2 m) {
#pragma unroll
  for (int d = 1; d < 4; d *= 2)
    m = make_uint2(max(m.x, __shfl_xor_sync(0xffffffffu, m.x, d)), max(m.y, __shfl_xor_sync(0xffffffffu, m.y, d)));
  return m;
}
__device__ __forceinline__ uint2 plane_or(uint2 m) {
#pragma unroll
  for (int d = 1; d < 4; d *= 2) {
    m.x |= __shfl_xor_sync(0xffffffffu, m.x, d);
    m.y |= __shfl_xor_sync(0xffffffffu, m.y, d);
  }
  return m;
}

__device__ __forceinline__ double2 load2(const double* p, bool on) {
  return on ? *reinterpret_cast<const double2*>(p) : make_double2(0.0, 0.0);
}

// Planes whose largest value is below 2^-959 are read with a factor of 2^128, so
// that to_fixed holds for them too.
constexpr int kTiny = 64;
__device__ __forceinline__ double2 raise(double2 v, bool x, bool y) {
  return make_double2(x ? v.x * 0x1p128 : v.x, y ? v.y * 0x1p128 : v.y);
}
constexpr unsigned kNotFinite = 0x7ff00000u;
// the exponent field that a plane is scaled by (0x7ff: not finite); planes of zeros
// take any that needs no rescaling
__device__ __forceinline__ int exponent_of(unsigned m) { return m == 0 ? 1075 : max(int(m >> 20), kTiny); }

// Contraction.  NT column tiles (FOLD: the first NT / 2 take the sums of the
// mirror pairs, the others their differences).
struct ContractArgs {
  const double* in;          // value (o, k, z) at o * in_o + k * in_k + z
  double* out;               // value (o, r, z) at o * out_o + r * out_r + z
  const uint4* tab;
  RowScale scale;            // of the rows k
  size_t in_o, in_k, out_o, out_r;
  int outer, ztiles;         // units: outer x ztiles, 16 z each
  int K;                     // rows, or mirror pairs
  int run;                   // 16-row steps summed in one set of accumulators (contract_steps)
  int rows;                  // output rows (slots)
  int mirror;                // FOLD: row k's mirror is row mirror - k
  int wall;                  // FOLD: pair 0 is row 0 (on the wall, table zero) and row `wall`
  int nan_tile;              // a value that is not finite takes the 16 planes of its tile, not its own alone
};

// A warp's tile in shared memory: [k step of the run][row, mirror row][16 rows][16 z],
// 16-byte pieces of a 128-byte row permuted by the row (piece c of row r at
// c ^ (r & 7): a fragment's lanes then read 8 different pieces of a bank sweep)
constexpr int kRowBytes = 128, kStepBytes = 16 * kRowBytes;
template <bool FOLD>
constexpr int tile_bytes() { return (kSeg / 16) * (FOLD ? 2 : 1) * kStepBytes; }

// copies the rows of k step ks of `unit` into their place in the warp's tile
template <bool FOLD>
__device__ __forceinline__ void copy_step(const ContractArgs& a, int unit, int ks, unsigned char* tile, int lane) {
  const int cr = lane >> 3, cc = lane & 7, o = unit / a.ztiles;
  const double* src = a.in + size_t(o) * a.in_o + (unit - o * a.ztiles) * 16 + 2 * cc;
  unsigned char* dst = tile + (ks % (kSeg / 16)) * ((FOLD ? 2 : 1) * kStepBytes);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = cr + 4 * q, k = 16 * ks + r;
    const int at = r * kRowBytes + ((cc ^ (r & 7)) << 4);
    if (16 * ks + 8 * (q >> 1) < a.K) {                // K is a multiple of 8
      cp_async16(dst + at, src + size_t(k) * a.in_k);
      if (FOLD) cp_async16(dst + kStepBytes + at, src + size_t(a.wall && k == 0 ? a.wall : a.mirror - k) * a.in_k);
    }
  }
  cp_async_commit();
}

// Persistent: a warp takes the runs (unit, at most a.run steps) of the units
// w, w + warps, ..; a.run divides the tile's 4 steps, so that a step's place in the
// tile is never one that the run in progress has still to read; as soon as a k step's values are in registers, the same
// step of its next run is copied over them (cp.async), so that a run's loads
// from memory overlap the digits and products of the one before.
template <int NT, bool FOLD>
__global__ void __launch_bounds__(32 * kSplitWarps, 3) split_contract_kernel(const __grid_constant__ ContractArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x) >> 5, 0);     // (uniform registers for what follows from it)
  const int units = a.outer * a.ztiles, stride = int(gridDim.x) * kSplitWarps;
  unsigned char* tile = smem_raw + warp * tile_bytes<FOLD>();
  constexpr int SB = (FOLD ? 2 : 1) * kStepBytes;      // bytes of a k step
  const int steps = (a.K + 15) / 16;
  auto copy = [&](int u, int ks) __attribute__((always_inline)) { copy_step<FOLD>(a, u, ks, tile, lane); };
  // this lane's values of row i (0 .. 3) of a step: rows 2t, 2t + 1, 2t + 8, 2t + 9
  const int at0 = 2 * t * kRowBytes + ((g ^ (2 * t)) << 4);
  const int at1 = (2 * t + 1) * kRowBytes + ((g ^ (2 * t + 1)) << 4);
  auto slot = [&](int ks, int half, int i) __attribute__((always_inline)) {
    return reinterpret_cast<double2*>(tile + (ks % (kSeg / 16)) * SB + half * kStepBytes + (i >> 1) * 8 * kRowBytes +
                                      (i & 1 ? at1 : at0));
  };
  auto value = [&](int ks, int half, int i) __attribute__((always_inline)) {
    return 16 * ks + 8 * (i >> 1) < a.K ? *slot(ks, half, i) : make_double2(0.0, 0.0);
  };
  // the scales of this lane's rows of a step, none in plain steps
  auto plain = [&](int ks) __attribute__((always_inline)) { return ks >= a.scale.plain0 && ks < a.scale.plain1; };
  auto row_scales = [&](int ks) __attribute__((always_inline)) {
    return __ldg(reinterpret_cast<const int4*>(a.scale.rows + 16 * ks + 4 * t));
  };
  int unit = int(blockIdx.x) * kSplitWarps + warp, s0 = 0;
  wait_stage();
  if (unit < units)
    for (int ks = 0; ks < min(a.run, steps); ++ks) copy(unit, ks);
#pragma unroll 1
  while (unit < units) {
    const int s1 = min(s0 + a.run, steps);
    // the run after this one
    const int unit2 = s1 < steps ? unit : unit + stride, n0 = s1 < steps ? s1 : 0;
    const int n1 = unit2 < units ? min(n0 + a.run, steps) : n0;
    cp_async_wait<0>();
    __syncwarp();
    // per plane, the largest high word of the values, each less its row's scale (a
    // table row that is zero takes no part, nor does the row on the wall)
    uint2 raw0 = make_uint2(0, 0);
    if (FOLD && a.wall && s0 == 0 && t == 0) {
      raw0 = absmax(raw0, *slot(0, 0, 0));
      *slot(0, 0, 0) = make_double2(0.0, 0.0);
    }
    uint2 low;                                         // the low words of all values together
    auto largest = [&]() __attribute__((always_inline)) {
      uint2 m = make_uint2(0, 0), raw = raw0;
      low = make_uint2(0, 0);
#pragma unroll 1
      for (int ks = s0; ks < s1; ++ks) {
        if (plain(ks)) {
#pragma unroll
          for (int i = 0; i < (FOLD ? 8 : 4); ++i) {
            const double2 v = value(ks, i >> 2, i & 3);
            m = absmax(m, v);
            low = make_uint2(low.x | unsigned(__double2loint(v.x)), low.y | unsigned(__double2loint(v.y)));
          }
        } else {
          const int4 cs = row_scales(ks);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint2 h = make_uint2(0, 0);
#pragma unroll
            for (int half = 0; half < (FOLD ? 2 : 1); ++half) {
              const double2 v = value(ks, half, i);
              h = absmax(h, v);
              low = make_uint2(low.x | unsigned(__double2loint(v.x)), low.y | unsigned(__double2loint(v.y)));
            }
            const int c = i < 2 ? (i == 0 ? cs.x : cs.y) : (i == 2 ? cs.z : cs.w);
            raw = make_uint2(max(raw.x, h.x), max(raw.y, h.y));
            m = make_uint2(unsigned(max(int(m.x), int(h.x) - c)), unsigned(max(int(m.y), int(h.y) - c)));
          }
        }
      }
      low = make_uint2(low.x | raw.x, low.y | raw.y);
      return plane_max(make_uint2(raw.x >= kNotFinite ? raw.x : m.x, raw.y >= kNotFinite ? raw.y : m.y));
    };
    uint2 m = largest();
    if (a.nan_tile && __any_sync(0xffffffffu, max(m.x, m.y) >= kNotFinite)) m = make_uint2(kNotFinite, kNotFinite);
    bool tiny0 = false, tiny1 = false, zero = false;
    constexpr unsigned kLow = unsigned(kTiny) << 20;
    if (__any_sync(0xffffffffu, min(m.x, m.y) < kLow)) {
      // planes of zeros, common outside a bunch, or without a value of 2^-959 or more
      const uint2 any = plane_or(make_uint2(low.x | m.x, low.y | m.y));
      tiny0 = m.x < kLow && any.x != 0;
      tiny1 = m.y < kLow && any.y != 0;
      if (__any_sync(0xffffffffu, tiny0 || tiny1)) {
#pragma unroll 1
        for (int ks = s0; ks < s1; ++ks)
#pragma unroll 1
          for (int i = 0; i < (FOLD ? 8 : 4); ++i)
            if (16 * ks + 8 * ((i & 3) >> 1) < a.K)
              *slot(ks, i >> 2, i & 3) = raise(value(ks, i >> 2, i & 3), tiny0, tiny1);
        m = largest();
      }
      zero = !__any_sync(0xffffffffu, (m.x | m.y) != 0);
    }
    const int emax0 = exponent_of(m.x), emax1 = exponent_of(m.y);
    const unsigned top0 = unsigned(emax0) << 20, top1 = unsigned(emax1) << 20;
    float acc[NT][kD][4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int s = 0; s < kD; ++s)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[n][s][e] = 0.f;
#pragma unroll 1
    for (int ks = s0; ks < s1; ++ks) {
      if (zero) {
        if (n0 + ks - s0 < n1) copy(unit2, n0 + ks - s0);
        continue;
      }
      const uint4* tb = a.tab + size_t(ks) * NT * (kD / 2) * 32 + lane;
      unsigned A[kD][4];
      auto split = [&](const unsigned long long (&X)[4][2]) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int zz = 0; zz < 2; ++zz) {
            unsigned d[kD];
            digits<kGuard>(X[2 * h][zz], X[2 * h + 1][zz], d);
#pragma unroll
            for (int i = 0; i < kD; ++i) A[i][2 * h + zz] = d[i];
          }
      };
      unsigned long long P[4][2], Q[4][2];
      int4 cs = make_int4(0, 0, 0, 0);
      if (!plain(ks)) cs = row_scales(ks);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const unsigned c = unsigned(i < 2 ? (i == 0 ? cs.x : cs.y) : (i == 2 ? cs.z : cs.w));
        const double2 u = value(ks, 0, i);
        if constexpr (FOLD) {
          const double2 v = value(ks, 1, i);
          const Fixed u0 = to_fixed(u.x, top0 + c), v0 = to_fixed(v.x, top0 + c);
          const Fixed u1 = to_fixed(u.y, top1 + c), v1 = to_fixed(v.y, top1 + c);
          P[i][0] = fixed_sum(u0, v0); Q[i][0] = fixed_difference(u0, v0);
          P[i][1] = fixed_sum(u1, v1); Q[i][1] = fixed_difference(u1, v1);
        } else {
          P[i][0] = fixed_value(to_fixed(u.x, top0 + c));
          P[i][1] = fixed_value(to_fixed(u.y, top1 + c));
        }
      }
      __syncwarp();                                    // every lane has this step's values
      if (n0 + ks - s0 < n1) copy(unit2, n0 + ks - s0);
      split(P);
#pragma unroll
      for (int n = 0; n < (FOLD ? NT / 2 : NT); ++n) mma_split<false>(acc[n], A, tb + n * (kD / 2) * 32);
      if constexpr (FOLD) {
        split(Q);
#pragma unroll
        for (int n = NT / 2; n < NT; ++n) mma_split<false>(acc[n], A, tb + n * (kD / 2) * 32);
      }
    }
#pragma unroll 1
    for (int ks = n0 + s1 - s0; ks < n1; ++ks) copy(unit2, ks);     // a longer run follows
    // V 2^-8 = acc_0 2^37 + acc_1 2^28 + acc_2 2^19 + (acc_3 2^18 + acc_4 2^9 + acc_5) 2^-8
    const Exponent e0(emax0 - 1075 - (tiny0 ? 128 : 0), emax0 < 0x7ff), e1(emax1 - 1075 - (tiny1 ? 128 : 0), emax1 < 0x7ff);
    const bool rare = __any_sync(0xffffffffu, (e0.extra | e1.extra) != 0);    // (the same for the warp: no divergence)
    const int o = unit / a.ztiles;
    double* out = a.out + size_t(o) * a.out_o + (unit - o * a.ztiles) * 16 + 2 * g;
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      auto fixed = [&](int q) {
        auto I = [&](int s) { return __float2int_rn(acc[n][s][q]); };
        const long long lo = mad_wide_s(I(3), 1 << 18, mad_wide_s(I(4), 1 << 9, I(5) + 128)) >> 8;
        return mad_wide_s(I(0), 1 << 30, 0) * 128 + mad_wide_s(I(1), 1 << 28, mad_wide_s(I(2), 1 << 19, lo));
      };
      const int nt = FOLD && n >= NT / 2 ? n - NT / 2 : n;
      const int half = a.rows / 2;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int q = 8 * nt + 2 * t + c;
        const int r = FOLD ? (n >= NT / 2 ? half + q : q) : q;
        if (q < (FOLD ? half : a.rows)) {
          double2* p = reinterpret_cast<double2*>(out + size_t(r) * a.out_r);
          double2 w = make_double2(0.0, 0.0);
          if (!zero) w = make_double2(to_double<false>(fixed(c), e0.e20), to_double<true>(fixed(2 + c), e1.e20));
          if (rare) w = rescale(w, e0.extra, e1.extra);
          if (s0 > 0) {
            const double2 b = *p;
            w.x += b.x;
            w.y += b.y;
          }
          *p = w;
        }
      }
    }
    unit = unit2;
    s0 = n0;
  }
}

// Expansion.  KS k steps of 16 modes (FOLD: the first KS / 2 steps are the
// modes even about the mid-plane, the others the odd ones, and a table row
// stands for a mirror pair).  With few terms the values keep 2 more bits and
// are rounded, not cut: nothing averages their errors.  SMALL: every sum stays
// below 2^22 (expand_sums_small, checked on the table's digits), so sums start
// from 1.5 2^23 and are read as integers off the bits, without conversions.
struct ExpandArgs {
  const double* in;          // value (o, k, z) at o * in_o + k * in_k + z
  double* out;               // value (o, r, z) at o * out_o + r * out_r + z
  const uint4* tab;
  RowScale scale;            // of the output rows
  size_t in_o, in_k, out_o, out_r;
  int outer, ztiles;
  int K;                     // modes (FOLD: both halves)
  int tiles;                 // output rows / 8 (FOLD: pairs / 8)
  int mirror, wall;          // as ContractArgs
  int nan_tile;
};
constexpr int kExtra = 2;    // |values| < 2^(53 + kExtra), |d_0| <= 256 << kExtra

// x 2^(1075 + kExtra - emax) rounded, plus kBiasLow and 1024 2^45 for the leading digit
__device__ __forceinline__ unsigned long long to_fixed_round(double x, int emax) {
  constexpr int G = 6;       // guard bits
  const int hi = __double2hiint(x);
  const unsigned sh = min(unsigned(emax - int((unsigned(hi) >> 20) & 0x7ffu)), 63u);
  const unsigned long long m =
      (pack64((unsigned(hi) & 0xfffffu) | 0x100000u, unsigned(__double2loint(x))) << (kExtra + G)) >> sh;
  const long long s = hi >> 31;
  return (((m ^ s) - s) + ((kBiasLow + (1024LL << 45)) << G) + (1LL << (G - 1))) >> G;
}
__device__ __forceinline__ void digits_round(unsigned long long a, unsigned long long b, unsigned (&d)[kD]) {
  digits<0>(a, b, d);        // the five lower ones; the leading one here has 12 bits
  const __half2 h = __halves2half2(__int2half_rn(int(hi32(a) >> 13) - 1024), __int2half_rn(int(hi32(b) >> 13) - 1024));
  d[0] = *reinterpret_cast<const unsigned*>(&h);
}

template <int KS, bool FOLD, bool SMALL>
__global__ void __launch_bounds__(32 * kSplitWarps, FOLD ? 4 : (KS == 2 ? 5 : 7)) split_expand_kernel(const __grid_constant__ ExpandArgs a) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int unit = int(blockIdx.x) * kSplitWarps + (int(threadIdx.x) >> 5);
  if (unit >= a.outer * a.ztiles) return;
  const int o = unit / a.ztiles, z = (unit % a.ztiles) * 16 + 2 * g;
  const double* in = a.in + size_t(o) * a.in_o + z;
  double* out = a.out + size_t(o) * a.out_o + z;
  constexpr int KH = FOLD ? KS / 2 : KS;             // k steps of an accumulator
  const int kmax = FOLD ? a.K / 2 : a.K;
  wait_stage();
  double2 x[KS][4];
  auto largest = [&]() {
    uint2 m = make_uint2(0, 0);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int i = 0; i < 4; ++i) m = absmax(m, x[ks][i]);
    return plane_max(m);
  };
#pragma unroll
  for (int ks = 0; ks < KS; ++ks)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = 16 * (ks % KH) + 2 * t + (i & 1) + 8 * (i >> 1);
      x[ks][i] = load2(in + size_t((ks / KH) * kmax + k) * a.in_k, k < kmax);
    }
  uint2 top = largest();
  if (a.nan_tile && __any_sync(0xffffffffu, max(top.x, top.y) >= kNotFinite)) top = make_uint2(kNotFinite, kNotFinite);
  const bool tiny0 = top.x < unsigned(kTiny) << 20, tiny1 = top.y < unsigned(kTiny) << 20;
  if (__any_sync(0xffffffffu, tiny0 || tiny1)) {
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int i = 0; i < 4; ++i) x[ks][i] = raise(x[ks][i], tiny0, tiny1);
    top = largest();
  }
  const int emax0 = exponent_of(top.x), emax1 = exponent_of(top.y);
  unsigned A[KS][kD][4];
#pragma unroll
  for (int ks = 0; ks < KS; ++ks)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double2 u = x[ks][2 * h], v = x[ks][2 * h + 1];
      unsigned d[kD];
      digits_round(to_fixed_round(u.x, emax0), to_fixed_round(v.x, emax0), d);
#pragma unroll
      for (int i = 0; i < kD; ++i) A[ks][i][2 * h] = d[i];
      digits_round(to_fixed_round(u.y, emax1), to_fixed_round(v.y, emax1), d);
#pragma unroll
      for (int i = 0; i < kD; ++i) A[ks][i][2 * h + 1] = d[i];
    }
  const Exponent e0(emax0 - 1083 - kExtra + 6 - (tiny0 ? 128 : 0), emax0 < 0x7ff);
  const Exponent e1(emax1 - 1083 - kExtra + 6 - (tiny1 ? 128 : 0), emax1 < 0x7ff);
  const bool rare = __any_sync(0xffffffffu, (e0.extra | e1.extra) != 0);      // (the same for the warp: no divergence)
  // V 2^-6 = acc_0 2^39 + acc_1 2^30 + acc_2 2^21 + acc_3 2^12 + acc_4 2^3 + acc_5 2^-6,
  // without kOff where the sums are read off with their offset M
  constexpr unsigned M = 0x4B400000u;                // the bits of 1.5 2^23
  constexpr unsigned long long kOff =
      SMALL ? (static_cast<unsigned long long>(M) << 39) + (static_cast<unsigned long long>(M) << 30) +
                  (static_cast<unsigned long long>(M) << 21) + (static_cast<unsigned long long>(M) << 12)
            : 0;
  auto fixed = [&](const float (&acc)[kD][4], int q) {
    auto I = [&](int s) { return SMALL ? __float_as_uint(acc[s][q]) : unsigned(__float2int_rn(acc[s][q])); };
    // acc_4 2^3 + acc_5 2^-6: 32 bits, the offsets subtracted (M 2^3 wraps)
    const int low = SMALL ? int(I(4) * 8u + (I(5) >> 6) - (M * 8u + (M >> 6))) : int(I(4)) * 8 + (int(I(5)) >> 6);
    unsigned long long v = static_cast<unsigned long long>(static_cast<long long>(low));
    if constexpr (SMALL) {
      v = mad_wide(I(3), 1u << 12, v);
      v = mad_wide(I(2), 1u << 21, v);
      v = mad_wide(I(1), 1u << 30, v);
    } else {
      v = static_cast<unsigned long long>(mad_wide_s(int(I(3)), 1 << 12, static_cast<long long>(v)));
      v = static_cast<unsigned long long>(mad_wide_s(int(I(2)), 1 << 21, static_cast<long long>(v)));
      v = static_cast<unsigned long long>(mad_wide_s(int(I(1)), 1 << 30, static_cast<long long>(v)));
    }
    return v + (static_cast<unsigned long long>(I(0) << 7) << 32);
  };
#pragma unroll 1
  for (int tile = 0; tile < a.tiles; ++tile) {
    const uint4* tb = a.tab + size_t(tile) * KS * (kD / 2) * 32 + lane;
    float acc[FOLD ? 2 : 1][kD][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      if (ks % KH == 0) mma_split<true>(acc[ks / KH], A[ks], tb + ks * (kD / 2) * 32, SMALL ? 12582912.f : 0.f);
      else mma_split<false>(acc[ks / KH], A[ks], tb + ks * (kD / 2) * 32);
    }
    const int2 scale = __ldg(reinterpret_cast<const int2*>(a.scale.rows + 16 * (tile >> 1) + 4 * t + 2 * (tile & 1)));
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int r = 8 * tile + 2 * t + c;
      const unsigned sc = unsigned(c ? scale.y : scale.x);              // (wraps for a row of zeros, whose sums are 0)
      const int x0 = int(unsigned(e0.e20) - sc), x1 = int(unsigned(e1.e20) - sc);
      const unsigned long long o0 = fixed(acc[0], c), o1 = fixed(acc[0], 2 + c);
      if constexpr (FOLD) {
        const unsigned long long v0 = fixed(acc[1], c), v1 = fixed(acc[1], 2 + c);
        double2 lo = make_double2(to_double<false>(static_cast<long long>(o0 + v0 - 2 * kOff), x0),
                                  to_double<false>(static_cast<long long>(o1 + v1 - 2 * kOff), x1));
        double2 hi = make_double2(to_double<true>(static_cast<long long>(o0 - v0), x0),
                                  to_double<true>(static_cast<long long>(o1 - v1), x1));
        const bool on_wall = a.wall && r == 0;
        if (on_wall) lo = make_double2(0.0, 0.0);
        if (rare) {
          lo = rescale(lo, e0.extra, e1.extra);
          hi = rescale(hi, e0.extra, e1.extra);
        }
        *reinterpret_cast<double2*>(out + size_t(r) * a.out_r) = lo;
        *reinterpret_cast<double2*>(out + size_t(on_wall ? a.wall : a.mirror - r) * a.out_r) = hi;
      } else {
        double2 v = make_double2(to_double<false>(static_cast<long long>(o0 - kOff), x0),
                                 to_double<true>(static_cast<long long>(o1 - kOff), x1));
        if (rare) v = rescale(v, e0.extra, e1.extra);
        *reinterpret_cast<double2*>(out + size_t(r) * a.out_r) = v;
      }
    }
  }
}

// Fragments of a table tab[rows][slots] (|values| <= 1), digits of
// round(value 2^(53 + the row's scale)).  contract: [k step over rows][tile of 8 slots][digit
// pair][lane]; expand: [tile of 8 rows][k step over slots][digit pair][lane].
// A piece is (b0, b1) of digit 2i, then of digit 2i + 1; b0 holds k = 2t,
// 2t + 1 and b1 k = 2t + 8, 2t + 9 of column g.
__device__ __forceinline__ unsigned short table_digit(const double* tab, const int* scale, int rows, int slots, int row,
                                                      int slot, int digit) {
  if (row >= rows || slot < 0 || slot >= slots) return 0;
  const int s = min(scale[scale_index(row)] >> 20, kMaxRowScale);        // (kZeroRow: only zeros there)
  const long long X = __double2ll_rn(ldexp(tab[size_t(row) * slots + slot], 53 + s));
  return __half_as_ushort(__int2half_rn(split_digit(X, digit)));
}

__global__ void split_table_kernel(const double* tab, const int* scale, int rows, int slots, int halves, int expand, uint4* out,
                                   long total) {
  const long idx = long(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const int lane = int(idx % 32), g = lane >> 2, t = lane & 3;
  const int dp = int((idx / 32) % (kD / 2));
  const long q = idx / (32 * (kD / 2));
  const int half = slots / 2;
  int step, tile, base = 0, limit = slots;
  if (expand) {                                      // k: slots, columns: rows
    const int per = halves ? (half + 15) / 16 : (slots + 15) / 16, steps = halves ? 2 * per : per;
    step = int(q % steps);
    tile = int(q / steps);
    if (halves) { base = (step / per) * half; limit = base + half; step %= per; }
  } else {                                           // k: rows, columns: slots
    const int per = halves ? (half + 7) / 8 : (slots + 7) / 8, tiles = halves ? 2 * per : per;
    tile = int(q % tiles);
    step = int(q / tiles);
    if (halves) { base = (tile / per) * half; limit = base + half; tile %= per; }
  }
  unsigned r[4];
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    unsigned short h[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int k = 16 * step + 2 * t + 8 * (w & 1) + c, n = 8 * tile + g;
      const int row = expand ? n : k;
      int slot = base + (expand ? k : n);
      if (slot >= limit) slot = -1;
      h[c] = table_digit(tab, scale, rows, slots, row, slot, 2 * dp + (w >> 1));
    }
    r[w] = unsigned(h[0]) | unsigned(h[1]) << 16;
  }
  out[idx] = make_uint4(r[0], r[1], r[2], r[3]);
}

inline unsigned units_grid(int units) { return unsigned((units + kSplitWarps - 1) / kSplitWarps); }

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 152;
  return n;
}

template <int NT, bool FOLD>
cudaError_t go_contract(const ContractArgs& a, cudaStream_t st) {
  constexpr int smem = kSplitWarps * tile_bytes<FOLD>();
  const cudaError_t e = cudaFuncSetAttribute(split_contract_kernel<NT, FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const unsigned need = units_grid(a.outer * a.ztiles), most = unsigned(3 * sm_count());   // 3 CTAs per SM
  // (the first kernel of a solve, whose input others write, waits for it at once)
  return launch_stage(split_contract_kernel<NT, FOLD>, dim3(need < most ? need : most), 32 * kSplitWarps, smem, st, a);
}

cudaError_t contract(const ContractArgs& a, bool fold, cudaStream_t st) {
  if (fold) return a.rows / 2 <= 8 ? go_contract<2, true>(a, st) : go_contract<4, true>(a, st);
  switch (split_tiles(a.rows)) {
    case 1: return go_contract<1, false>(a, st);
    case 2: return go_contract<2, false>(a, st);
    case 3: return go_contract<3, false>(a, st);
    case 4: return go_contract<4, false>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

template <typename K>
cudaError_t go(K kern, const ExpandArgs& a, cudaStream_t st) {
  return launch_stage(kern, dim3(units_grid(a.outer * a.ztiles)), 32 * kSplitWarps, 0, st, a);
}

cudaError_t expand(const ExpandArgs& a, bool fold, bool small, cudaStream_t st) {
  if (fold) return small ? go(split_expand_kernel<2, true, true>, a, st) : go(split_expand_kernel<2, true, false>, a, st);
  if (a.K <= 16) return small ? go(split_expand_kernel<1, false, true>, a, st) : go(split_expand_kernel<1, false, false>, a, st);
  return go(split_expand_kernel<2, false, false>, a, st);
}

}  // namespace

cudaError_t build_split_table(const double* tab, const int* scale, int rows, int slots, bool halves, bool expand,
                              uint4* out, cudaStream_t st) {
  const long total = long(expand ? split_expand_size(rows, slots, halves) : split_contract_size(rows, slots, halves));
  split_table_kernel<<<unsigned((total + 127) / 128), 128, 0, st>>>(tab, scale, rows, slots, halves, expand, out, total);
  return cudaGetLastError();
}

cudaError_t launch_split_project(const SplitArgs& s, const double* rho, double* part, cudaStream_t st) {
  const bool fold = s.fold != 0;
  for (int z0 = 0; z0 < s.nz; z0 += s.zs) {
    ContractArgs y{};
    y.in = rho + z0;
    y.in_o = size_t(s.ny) * s.nz;
    y.in_k = size_t(s.nz);
    y.out = s.half;
    y.out_o = size_t(s.myp) * s.zs;
    y.out_r = size_t(s.zs);
    y.tab = s.cy;
    y.run = s.cy_run;
    y.scale = s.ys;
    y.outer = s.nx;
    y.ztiles = s.zs / 16;
    y.K = fold ? s.ny / 2 : s.ny;
    y.rows = s.myp;
    y.mirror = s.fold == 2 ? s.ny : s.ny - 1;
    y.wall = s.fold == 2 ? s.ny / 2 : 0;
    y.nan_tile = s.nan_tile;
    cudaError_t e = contract(y, fold, st);
    if (e != cudaSuccess) return e;
    ContractArgs x{};
    x.in = s.half;
    x.in_o = size_t(s.zs);
    x.in_k = size_t(s.myp) * s.zs;
    x.out = part + z0;
    x.out_o = size_t(s.nz);
    x.out_r = size_t(s.myp) * s.nz;
    x.tab = s.cx;
    x.run = s.cx_run;
    x.scale = s.xs;
    x.outer = s.myp;
    x.ztiles = s.zs / 16;
    x.K = s.nx;
    x.rows = s.mxp;
    x.nan_tile = s.nan_tile;
    if ((e = contract(x, false, st)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_split_back(const SplitArgs& s, const double* psi, double* phi, cudaStream_t st) {
  const bool fold = s.fold != 0;
  for (int z0 = 0; z0 < s.nz; z0 += s.zs) {
    ExpandArgs x{};
    x.in = psi + z0;
    x.in_o = size_t(s.nz);
    x.in_k = size_t(s.myp) * s.nz;
    x.out = s.half;
    x.out_o = size_t(s.zs);
    x.out_r = size_t(s.myp) * s.zs;
    x.tab = s.ex;
    x.scale = s.xs;
    x.outer = s.myp;
    x.ztiles = s.zs / 16;
    x.K = s.mxp;
    x.tiles = s.nx / 8;
    x.nan_tile = s.nan_tile;
    cudaError_t e = expand(x, false, s.ex_small, st);
    if (e != cudaSuccess) return e;
    ExpandArgs y{};
    y.in = s.half;
    y.in_o = size_t(s.myp) * s.zs;
    y.in_k = size_t(s.zs);
    y.out = phi + z0;
    y.out_o = size_t(s.ny) * s.nz;
    y.out_r = size_t(s.nz);
    y.tab = s.ey;
    y.scale = s.ys;
    y.outer = s.nx;
    y.ztiles = s.zs / 16;
    y.K = s.myp;
    y.tiles = (fold ? s.ny / 2 : s.ny) / 8;
    y.mirror = s.fold == 2 ? s.ny : s.ny - 1;
    y.wall = s.fold == 2 ? s.ny / 2 : 0;
    y.nan_tile = s.nan_tile;
    if ((e = expand(y, fold, s.ey_small, st)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pp
