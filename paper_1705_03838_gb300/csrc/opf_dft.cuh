// FP64 Fourier sums on the tensor cores by an exact splitting into digits.
//
// A GB300 SM passes two FP64 multiply-adds per clock and about a thousand
// 16-bit ones, so a short FP64 transform is cheaper as a product with its
// cosine and sine matrices in which both factors are cut into seven 8-bit
// digits: x = 2^(e-55) sum_i D_i 256^(6-i) with one exponent e per row of data
// and |D_i| <= 128, the matrix likewise with e = 0.  Products of digits are
// integers; the sums over i + j = l of one level stay below 2^22 (for every
// length up to 96), so FP32 accumulators that start at 1.5 2^23 hold them
// exactly and their bit patterns are the integers.  Levels 0..7 are kept: the
// first dropped one is 2^-63 of the largest term.  They are joined and rounded
// to FP64 in integers.  The idea of summing exact slice products is that of
// Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012).
//
// Against 80-bit sums the results are closer than those of the FP64 FFT on
// spectra of every slope, and within its error where one term outweighs the
// rest; whole steps are as far from 64-bit references as with it.  FP64
// kernels against these, per launch (z synthesis, theta product, z analysis):
// N = 48, 96 x 72: 33, 82, 26 -> 20, 39, 17 us; 64 x (N = 32, 48 x 48): 321,
// 956, 199 -> 142, 357, 86 us; N = 32, 48 x 48: 13, 25, 13 -> 10, 21, 11 us.
// What bounds them now is the latency of their phases at 16 warps per SM: the
// tensor pipe is a third to two thirds busy in the products, the integer
// units in the splitting and joining.  Lengths above 96 stay with the FFT: the
// kernels give each warp one digit tile of a row's at most 32 harmonics, and
// the bound on a level's sums has been worked out up to there.  (The work grows
// with the square of the length, the FFT's does not; at 96 these are 1.6 times
// as fast in z, and where the two cross has not been measured.)
// Symmetry halves the work: with c, s the cosine and sine sums over
// harmonics h (or points p), a result at p and its mirror n - p are c + s and
// c - s (up to factors i).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

#include "opf_step.cuh"

namespace opf {

constexpr int kDig = 7;         // digits of a factor
constexpr int kLev = 8;         // levels of digit products kept
constexpr int kDftMaxH = 32;    // harmonics per transform (length 3 H)
constexpr float kDftBias = 12582912.0f;  // 1.5 2^23

// Digit products over one k tile of 16 and one tile of 16 rows: seven uint4
// (A) and seven uint2 (B) per lane, in the fragment order of m16n8k16.
constexpr int kTileA = kDig * 32;  // uint4 per (row tile, k tile)
constexpr int kTileB = kDig * 32;  // uint2 per (column tile, k tile)

// Table of one matrix: [column tile][k tile][digit][lane] uint2.
__host__ __device__ constexpr int dft_tiles(int n, int w) { return (n + w - 1) / w; }
__host__ __device__ constexpr int dft_points(int n) { return n / 2 + 1; }  // p = 0 .. n/2
// Entries (uint2) of a synthesis (k = harmonics, columns = points) and of an
// analysis matrix (k = points, columns = harmonics).
__host__ __device__ constexpr long dft_synth_size(int H, int n) {
  return (long)dft_tiles(H, 16) * dft_tiles(dft_points(n), 8) * kTileB;
}
__host__ __device__ constexpr long dft_anal_size(int H, int n) {
  return (long)dft_tiles(dft_points(n), 16) * dft_tiles(H, 8) * kTileB;
}

// The digits of BITS bits, most significant first, of a fixed-point value
// |v| <= 2^(7 BITS - 1): integers d_0 = -h..h, d_1.. = -h..h-1, h = 2^(BITS-1).
template <int BITS>
__host__ __device__ constexpr unsigned long long digit_bias() {  // h in every digit
  unsigned long long b = 0;
  for (int i = 0; i < kDig; ++i) b = (b << BITS) | (1ull << (BITS - 1));
  return b;
}
template <int BITS>
__host__ __device__ inline int dft_digit(long long v, int i) {
  const unsigned long long y = ((unsigned long long)v + digit_bias<BITS>()) >> (BITS * (6 - i));
  return (int)(i == 0 ? y : y & ((1ull << BITS) - 1)) - (1 << (BITS - 1));
}

// The radial stencils' factors: 62 bits in seven 9-bit digits.
constexpr int kStBits = 9, kStFixed = 62;
struct StencilTable {
  const uint2* tab;  // [parity][tile][digit][lane]
  const int* ew;     // [parity][8 tiles]
  const double* d1;  // the weights, [parity][N][9]
  int N, tiles, off;  // row i sits at i + off of the tiles
};
StencilTable stencil_at(const void* p, const double* d1, int N);  // p as filled by stencil_host_table
__host__ __device__ constexpr int stencil_tiles(int N) { return (N + 7) / 8; }
__host__ __device__ constexpr long stencil_table_size(int N) { return 2L * stencil_tiles(N) * kTileB; }
// Mesh row of lane t's value q = 0..3 in a tile whose first row is i0.
__host__ __device__ constexpr int stencil_row(int i0, int t, int q) {
  return q < 2 ? i0 + 2 * t + q : (t < 2 ? i0 - 4 + 2 * t : i0 + 4 + 2 * t) + q - 2;
}
__host__ __device__ inline unsigned long long dft_bits(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}
// x in fixed point of F bits, rounded to nearest: units of 2^(emax - 1022 - F +
// half), emax the largest biased exponent among the values that share it (200
// at least), |result| <= 2^(F - half); half = 1 leaves room for the sum of two.
template <int F = 55>
__host__ __device__ inline long long dft_fixed(double x, int emax, int half) {
  const unsigned long long b = dft_bits(x);
  const unsigned h = (unsigned)(b >> 32);
  const int e = (h >> 20) & 0x7ff;
  const unsigned hm = e ? ((h & 0xfffffu) | 0x100000u) : 0u;
  const unsigned long long m = ((unsigned long long)hm << 32) | (e ? (unsigned)b : 0u);
  const int s0 = (emax < 200 ? 200 : emax) - e + half, sh = s0 < 63 ? s0 : 63;
  const unsigned long long r = (((m << (F - 52)) >> sh) + 1) >> 1;
  return (h & 0x80000000u) ? -(long long)r : (long long)r;
}
// Table entry of (parity's) stencils d1 = [N][9]: fixed point of the weight
// that output row i gives row j, and the biased exponent that the row's
// weights share, that of the sum of their magnitudes (which bounds a result by
// the largest datum).
__host__ __device__ inline int stencil_exponent(const double* d1, int i) {
  double s = 0.0;
  for (int q = 0; q < 9; ++q) s += fabs(d1[i * 9 + q]);
  return (int)(dft_bits(s) >> 52) & 0x7ff;
}
__host__ __device__ inline long long stencil_weight(const double* d1, int N, int i, int j) {
  const int lo = i - 4 < 0 ? 0 : (i - 4 > N - 9 ? N - 9 : i - 4);
  if (i < 0 || i >= N || j < 0 || j >= N || j < lo || j > lo + 8) return 0;
  return dft_fixed<kStFixed>(d1[i * 9 + j - lo], stencil_exponent(d1, i), 0);
}

// Entry (k, n) of a table in fixed point: v(k, n), zero outside K x N.
#pragma nv_exec_check_disable
template <int BITS = 8, class V>
__host__ __device__ inline void table_entry(long idx, int KT, V v, uint2* out) {
  // idx = (nt * KT + kt) * 32 + lane
  const int lane = (int)(idx % 32), kt = (int)(idx / 32 % KT), nt = (int)(idx / 32 / KT);
  const int t = lane & 3, n = nt * 8 + (lane >> 2), k0 = kt * 16 + 2 * t;
  const long long f[4] = {v(k0, n), v(k0 + 1, n), v(k0 + 8, n), v(k0 + 9, n)};
  for (int i = 0; i < kDig; ++i) {
    unsigned short h[4];
    for (int q = 0; q < 4; ++q) {  // a small integer as a half
      const int d = dft_digit<BITS>(f[q], i);
#ifdef __CUDA_ARCH__
      h[q] = __half_as_ushort(__int2half_rn(d));
#else
      const int a = d < 0 ? -d : d;
      int e = 0;
      while ((a >> e) > 1) ++e;
      h[q] = a ? (unsigned short)((d < 0 ? 0x8000 : 0) | ((15 + e) << 10) | ((a << (10 - e)) & 0x3ff)) : 0;
#endif
    }
    out[((long)nt * KT + kt) * kTileB + i * 32 + lane] =
        make_uint2(h[0] | (unsigned)h[1] << 16, h[2] | (unsigned)h[3] << 16);
  }
}

// Entry idx = (parity * tiles + tile) * 32 + lane of the stencil table.
__host__ __device__ inline void stencil_entry(long idx, const double* d1, int N, uint2* tab, int* ew) {
  const int NT = stencil_tiles(N), off = 8 * NT - N;
  const int nt = (int)(idx / 32 % NT), par = (int)(idx / 32 / NT);
  const double* w = d1 + (long)par * N * 9;
  // a table of one k tile and NT column tiles: k, n of the tile -> row, weight
  table_entry<kStBits>(idx % (32L * NT), 1, [=](int k, int n) -> long long {
    const int i0 = (n >> 3) * 8 - off, t = (k & 7) >> 1, q = (k & 1) + (k >> 3) * 2;
    return stencil_weight(w, N, i0 + (n & 7), stencil_row(i0, t, q));
  }, tab + (long)par * NT * kTileB);
  const int lane = (int)(idx % 32), i = nt * 8 + lane - off;
  if (lane < 8) ew[(par * NT + nt) * 8 + lane] = i < 0 ? 0 : stencil_exponent(w, i) - 1022;
}

#ifdef __CUDACC__
__device__ __forceinline__ void dft_mma(float (&c)[4], const uint4& a, const uint2& b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

// acc[l] (one 16 x 8 tile per level) = bias + sum over KT k tiles and digits
// i + j = l.  A in shared memory, B a table (read through L1), this lane's.
__device__ __forceinline__ void dft_gemm(float (&acc)[kLev][4], const uint4* A, const uint2* __restrict__ B, int KT) {
#pragma unroll
  for (int l = 0; l < kLev; ++l)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[l][q] = kDftBias;
#pragma unroll 1
  for (int kt = 0; kt < KT; ++kt) {
    uint4 a[kDig];
    uint2 b[kDig];
#pragma unroll
    for (int i = 0; i < kDig; ++i) b[i] = __ldg(B + (kt * kDig + i) * 32);
#pragma unroll
    for (int i = 0; i < kDig; ++i) a[i] = A[(kt * kDig + i) * 32];
#pragma unroll
    for (int j = 0; j < kDig; ++j)
#pragma unroll
      for (int i = 0; i < kDig; ++i)
        if (i + j < kLev) dft_mma(acc[i + j], a[i], b[j]);
  }
}

// Two levels at a time as integers: w[q][k] = A_2k 256 + A_2k+1 + kDftPair
// (mod 2^32), q the fragment's element.
constexpr unsigned kDftPair = 0x4B400000u * 257u;  // the bias' bits in both levels
__device__ __forceinline__ void dft_pairs(const float (&acc)[kLev][4], unsigned (&w)[4][kLev / 2]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int k = 0; k < kLev / 2; ++k)
      w[q][k] = (unsigned)__float_as_int(acc[2 * k][q]) * 256u + (unsigned)__float_as_int(acc[2 * k + 1][q]);
}

// A row whose largest value lies outside 2^-823 .. 2^877 (emax: its biased
// exponent; zeros and values that are not finite are no such row).  A block that
// holds one sets a flag in shared memory and, when all is done, replaces its
// results by plain FP64 sums; the flag costs the others under half a percent of
// a launch.  (Scaling such rows on the way in and out cost them up to 4 %.)
__device__ __forceinline__ bool dft_outside(int emax) {
  return (unsigned)(emax - 1) < 199u || (unsigned)(emax - 1900) < 147u;
}

// Scaling of one row's results, which count 2^(e - 54): the exponent field's
// offset and, for a row with a non-finite value, the bits that make every
// result NaN.
struct DftScale {
  int e;
  unsigned nan;
};
// emax: the largest biased exponent of the row's data; its fixed point is
// then 2^(emax - 1022 - 55), the results' twice that for each of shift.
__device__ __forceinline__ DftScale dft_scale(int emax, int shift) {
  return DftScale{max(emax, 200) - 1022 + shift + 1030, emax >= 1900 ? 0x7ff80000u : 0u};
}
// The FP64 value nearest to level pairs t (|t| < 2^31, free of their offsets),
// put together in integers: two FP64 multiply-adds per result would take three
// times as long, at two lanes per clock, as the ~25 integer instructions.
__device__ __forceinline__ double dft_join(unsigned t0, unsigned t1, unsigned t2, unsigned t3, const DftScale& s) {
  // in units of level 5, 2^(e-54): |v| < 2^61, rounded at the half unit
  const int low = (int)t2 + (((int)t3 + 0x8000) >> 16);
  const long long v = (long long)(int)t1 * 65536ll + low + ((long long)(int)t0 << 32);
  const unsigned long long a = v < 0 ? -v : v;
  const int z = __clzll((long long)a) - 1;
  const unsigned long long m = ((a << z) + 512) >> 10;  // 2^52 .. 2^53
  unsigned h = (unsigned)(m >> 32) + ((unsigned)(s.e - z) << 20);
  h = a ? h : 0u;
  return __hiloint2double((int)(h | ((unsigned)(v >> 32) & 0x80000000u) | s.nan), (int)(unsigned)m);
}
__device__ __forceinline__ double dft_plus(const unsigned (&a)[4], const unsigned (&b)[4], const DftScale& s) {
  constexpr unsigned k = 2u * kDftPair;
  return dft_join(a[0] + b[0] - k, a[1] + b[1] - k, a[2] + b[2] - k, a[3] + b[3] - k, s);
}
__device__ __forceinline__ double dft_minus(const unsigned (&a)[4], const unsigned (&b)[4], const DftScale& s) {
  return dft_join(a[0] - b[0], a[1] - b[1], a[2] - b[2], a[3] - b[3], s);
}
__device__ __forceinline__ double dft_value(const unsigned (&a)[4], const DftScale& s) {
  constexpr unsigned k = kDftPair;
  return dft_join(a[0] - k, a[1] - k, a[2] - k, a[3] - k, s);
}
__device__ __forceinline__ double dft_negative(const unsigned (&a)[4], const DftScale& s) {
  constexpr unsigned k = kDftPair;
  return dft_join(k - a[0], k - a[1], k - a[2], k - a[3], s);
}

__device__ __forceinline__ int dft_exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// One fragment register per digit from two neighbouring k (va at the even one):
// bytes of the offset values, made halves 1024 + byte and brought to -128..128.
__device__ __forceinline__ void dft_split(long long va, long long vb, unsigned (&out)[kDig]) {
  const unsigned long long bias = 0x0080808080808080ull;
  const unsigned long long a = (unsigned long long)va + bias, b = (unsigned long long)vb + bias;
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
  unsigned v[kDig] = {__byte_perm(ah, bh, 0x7632), __byte_perm(ah, bh, 0x0501), __byte_perm(ah, bh, 0x0400),
                      __byte_perm(al, bl, 0x0703), __byte_perm(al, bl, 0x0602), __byte_perm(al, bl, 0x0501),
                      __byte_perm(al, bl, 0x0400)};
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6480));  // 1152
#pragma unroll
  for (int i = 0; i < kDig; ++i) {
    const unsigned u = (i == 0 ? v[i] : (v[i] & 0x00ff00ffu)) | 0x64006400u;
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&u), off);
    out[i] = *reinterpret_cast<const unsigned*>(&d);
  }
}

// This lane's fragment of a 16 x 16 tile: x[0..3] = row g at k = 2t, 2t+1,
// 2t+8, 2t+9, y[0..3] = row g+8 (lane = 4 g + t); tile: [digit][lane].
__device__ __forceinline__ void dft_put(uint4* tile, int lane, const long long (&x)[4], const long long (&y)[4]) {
  unsigned r0[kDig], r1[kDig], r2[kDig], r3[kDig];
  dft_split(x[0], x[1], r0);
  dft_split(y[0], y[1], r1);
  dft_split(x[2], x[3], r2);
  dft_split(y[2], y[3], r3);
#pragma unroll
  for (int i = 0; i < kDig; ++i) tile[i * 32 + lane] = make_uint4(r0[i], r1[i], r2[i], r3[i]);
}

// ---------------------------------------------------------------- radial stencils
// The 9-point first derivative of eight complex columns at eight rows, by the
// same digit products: the rows of the 16 x 16 data tile are the columns' real
// (0-7) and imaginary (8-15) parts, its k the 16 rows that the eight outputs
// reach -- k = 0..7 the output rows themselves, 8..15 the four below and the
// four above, so that a lane's first two values are the points it gets the
// derivative of.  Rows are counted in tiles of eight back from the wall (the
// wall rows' shifted stencils then stay within the window); rows outside the
// mesh have weight zero.  One exponent per column and window, one per row of
// the stencil.
//
// Digits of nine bits (an output has nine weights that are not zero, so a
// level's sums stay below 63 2^16 < 2^22) hold 62 bits below the window's
// largest value: the error of a row is about 2^-60 of that value times the
// row's weights.  Multiply-adds have 2^-53 of the row's own terms, which near
// the axis (columns go as r^m~) and at the wall are far smaller than the
// window's largest value.  So a column takes multiply-adds in a window in
// which some row has neither neighbour within 2^8 of the largest value, or in
// which that value is out of the fixed point's range.  The choice is the
// column's and the window's alone: it does not depend on which columns or
// tiles share a warp.  In units of 2^-53 of a row's terms, over r^m~ (m~ =
// 0..40), boundary layers, waves and noise at N = 21, 41, 48 and 96: digits,
// where taken, 0.09-0.15 rms, 1.3 at most; multiply-adds in the same rows
// 0.26-0.31 rms, 2.5 at most.  (Eight-bit digits without the choice, at the
// wall 460, next to the axis 7e8 at m~ = 20.)
//
// After 30 steps a tenth (N = 128, 255 x 128 modes) to two fifths (N = 32, 31 x
// 16) of the columns' windows take multiply-adds, in a quarter to three fifths
// of the warps; the other rows' derivatives cost no FP64 instruction.  Per
// launch, digits alone -> with the choice: split curl, N = 128: 242 -> 267 us,
// N = 48, 63 x 24 modes 12.6 -> 15.9 us; solve 1545 -> 1559 and 42.8 -> 45.9 us.
struct StencilAt {      // one lane's share of a tile
  const uint2* tab;      // the tile's table plus lane
  const double* d1;      // the parity's weights, [N][9]
  int N, i0, ew0, ew1;   // mesh rows, the tile's first one, exponents of rows 2t, 2t+1
  int shift;             // times 2^shift, 0 or -1
};
// Tile nt of parity par, with tile `table`'s digits (a lane past the last tile: nt = tiles).
__device__ __forceinline__ StencilAt stencil_tile(const StencilTable& s, int par, int table, int nt, int lane,
                                                  int shift) {
  const int* ew = s.ew + (par * s.tiles + min(nt, s.tiles - 1)) * 8 + 2 * (lane & 3);
  return StencilAt{s.tab + (long)(par * s.tiles + table) * kTileB + lane, s.d1 + (long)par * s.N * 9, s.N,
                   nt * 8 - s.off, ew[0], ew[1], shift};
}

// x: this lane's column (lane = 4 g + t) at rows 2t, 2t+1 of the tile, then of
// its halo (stencil_row).  The largest exponents of the column's parts, low
// half real, high half imaginary.
struct StencilWindow {
  unsigned p0, p1, halo, top;  // of the lane's own rows, the halo row next to the tile (lanes t = 1, 2), the window
};
__device__ __forceinline__ StencilWindow stencil_window(const double2 (&x)[4]) {
  unsigned p[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    p[q] = (__byte_perm((unsigned)__double2hiint(x[q].x), (unsigned)__double2hiint(x[q].y), 0x7632) >> 4) & 0x07ff07ffu;
  unsigned top = __vmaxu2(__vmaxu2(p[0], p[1]), __vmaxu2(p[2], p[3]));
  top = __vmaxu2(top, __shfl_xor_sync(0xffffffffu, top, 1));
  top = __vmaxu2(top, __shfl_xor_sync(0xffffffffu, top, 2));
  return StencilWindow{p[0], p[1], (threadIdx.x & 3) == 1 ? p[3] : p[2], top};
}

// The columns that take multiply-adds, one bit per column g at 4 g, given how
// many bits a row's neighbours may lie below the window's largest value.
// SMALL: so do those whose values are all tiny (to FP32 these come out right
// without, or as zero).  *all: no other column has values.  row (set if the
// result is not 0): whether it is this lane's own rows 2t, 2t+1 that need them.
template <int BITS, bool SMALL>
__device__ __forceinline__ unsigned stencil_steep(const double2 (&x)[4], const StencilWindow& w, int i0, int N, bool* all,
                                                  bool (&row)[2]) {
  constexpr unsigned kGuard = 0x80008000u, kOnes = 0x00010001u;
  const int t = threadIdx.x & 3, i = i0 + 2 * t;
  unsigned below = __shfl_up_sync(0xffffffffu, w.p1, 1, 4), above = __shfl_down_sync(0xffffffffu, w.p0, 1, 4);
  const unsigned halo = __shfl_sync(0xffffffffu, w.halo, t == 0 ? 1 : 2, 4);
  below = __vmaxu2(t == 0 ? halo : below, w.p1);  // the neighbours of row 2t
  above = __vmaxu2(t == 3 ? halo : above, w.p0);  // ... of row 2t+1
  const unsigned large = ((1899u * kOnes) | kGuard) - w.top, small = SMALL ? (w.top | kGuard) - 300u * kOnes : kGuard;
  const unsigned near0 = (i >= 0 && i < N ? ((below + BITS * kOnes) | kGuard) - w.top : kGuard) & large;
  const unsigned near1 = (i + 1 >= 0 && i + 1 < N ? ((above + BITS * kOnes) | kGuard) - w.top : kGuard) & large;
  *all = false;
  if (!__any_sync(0xffffffffu, (near0 & near1 & small & kGuard) != kGuard)) return 0u;
  row[0] = (near0 & kGuard) != kGuard;
  row[1] = (near1 & kGuard) != kGuard;
  bool bad = row[0] || row[1];
  if (SMALL) {  // (a part of zeros alone is not small)
    unsigned re = 0, im = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      re |= (unsigned)__double2hiint(x[q].x) << 1 | (unsigned)__double2loint(x[q].x);
      im |= (unsigned)__double2hiint(x[q].y) << 1 | (unsigned)__double2loint(x[q].y);
    }
    bad = bad || (!(small & 0x8000u) && re) || (!(small & 0x80000000u) && im);
  }
  unsigned cols = __ballot_sync(0xffffffffu, bad);
  cols |= cols >> 1;
  cols = (cols | cols >> 2) & 0x11111111u;
  *all = cols && __all_sync(0xffffffffu, w.top == 0 || (cols >> (threadIdx.x & 28) & 1u));
  return cols;
}

// The derivative of these columns by multiply-adds, from the lowest row up, into
// out of the lanes whose column it is.  Two columns at a time, a lane per row
// and part: a warp's FP64 instruction takes its time whatever the lanes in use,
// and often few of the eight columns are steep (a lane doing its own two rows, for all columns of the warp: solve at N = 128
// 1682 us instead of 1564, curl 314 instead of 277; taking the steep rows alone,
// the digits for the rest: the same on the whole).
// at(row, g, part): column g's value.
template <typename At>
__device__ __forceinline__ void stencil_fma(unsigned cols, const StencilAt& s, At at, double2 (&out)[2]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, part = (lane >> 3) & 1;
#pragma unroll 1
  while (cols) {
    const int c0 = (__ffs(cols) - 1) >> 2;
    cols &= cols - 1;
    const int c1 = cols ? (__ffs(cols) - 1) >> 2 : c0;
    cols &= cols - 1;
    const int c = lane < 16 ? c0 : c1, i = __shfl_sync(0xffffffffu, s.i0, 4 * c) + (lane & 7);
    double sum = 0.0;
    if (i >= 0 && i < s.N) {
      const int lo = min(max(i - 4, 0), s.N - 9);
      double v[9], w[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const bool in = lo + k <= i + 4;  // (the axis rows' weights beyond are zero, and past the window)
        w[k] = in ? __ldg(s.d1 + i * 9 + k) : 0.0;
        v[k] = in ? at(lo + k, c, part) : 0.0;
      }
#pragma unroll
      for (int k = 0; k < 9; ++k) sum = fma(w[k], v[k], sum);
      if (s.shift) sum = halved(sum);
    }
    const int src = (g == c0 ? 0 : 16) + 2 * t;
    const double2 a = double2{__shfl_sync(0xffffffffu, sum, src), __shfl_sync(0xffffffffu, sum, src + 8)};
    const double2 b = double2{__shfl_sync(0xffffffffu, sum, src + 1), __shfl_sync(0xffffffffu, sum, src + 9)};
    if (g == c0 || g == c1) {
      out[0] = a;
      out[1] = b;
    }
  }
}

// One fragment register per digit from two neighbouring k (va at the even one),
// as in dft_split: halves 1024 + the offset digit, brought to -256..256.
template <int DIG>
__device__ __forceinline__ void stencil_split(long long va, long long vb, unsigned (&out)[DIG]) {
  constexpr unsigned long long bias = digit_bias<kStBits>();
  const unsigned long long a = (unsigned long long)va + bias, b = (unsigned long long)vb + bias;
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6500));  // 1280
#pragma unroll
  for (int i = 0; i < DIG; ++i) {
    const unsigned v = __byte_perm((unsigned)(a >> (kStBits * (6 - i))), (unsigned)(b >> (kStBits * (6 - i))), 0x5410);
    const unsigned u = (i == 0 ? v : (v & 0x01ff01ffu)) | 0x64006400u;
    const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&u), off);
    out[i] = *reinterpret_cast<const unsigned*>(&d);
  }
}
// The window's digits as a fragment, DIG of them.
template <int DIG>
__device__ __forceinline__ void stencil_digits(const double2 (&x)[4], unsigned top, uint4 (&a)[DIG]) {
  const int er = (int)(top & 0xffffu), ei = (int)(top >> 16);
  auto fixed = [](double v, int e) { return dft_fixed<kStFixed>(v, e, 0); };
  unsigned r[DIG];
  stencil_split(fixed(x[0].x, er), fixed(x[1].x, er), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].x = r[i];
  stencil_split(fixed(x[0].y, ei), fixed(x[1].y, ei), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].y = r[i];
  stencil_split(fixed(x[2].x, er), fixed(x[3].x, er), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].z = r[i];
  stencil_split(fixed(x[2].y, ei), fixed(x[3].y, ei), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].w = r[i];
}
template <int DIG, int LEV>
__device__ __forceinline__ void stencil_products(const uint4 (&a)[DIG], const uint2* __restrict__ tab,
                                                 float (&acc)[LEV][4]) {
#pragma unroll
  for (int l = 0; l < LEV; ++l)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[l][q] = kDftBias;
#pragma unroll
  for (int j = 0; j < DIG; ++j) {
    const uint2 b = __ldg(tab + j * 32);
#pragma unroll
    for (int i = 0; i < DIG; ++i)
      if (i + j < LEV) dft_mma(acc[i + j], a[i], b);
  }
}
// Two levels as one integer, free of their biases (|level| < 2^22).
__device__ __forceinline__ int stencil_levels(float hi, float lo) {
  return (int)((unsigned)__float_as_int(hi) * 512u + (unsigned)__float_as_int(lo) - 0x4B400000u * 513u);
}
// The FP64 value nearest to the levels' sum, in units of half of level 5,
// 2^-62 of the largest datum times the sum of weights: |v| <= 2^62.
__device__ __forceinline__ double stencil_value(const float (&acc)[kLev][4], int q, int e) {
  const int t0 = stencil_levels(acc[0][q], acc[1][q]), t1 = stencil_levels(acc[2][q], acc[3][q]);
  const int t2 = stencil_levels(acc[4][q], acc[5][q]), t3 = stencil_levels(acc[6][q], acc[7][q]);
  const long long v = (long long)((unsigned long long)(long long)t0 << 37) + (long long)t1 * 524288ll +
                      ((long long)t2 * 2ll + ((t3 + 0x10000) >> 17));
  const unsigned long long a = v < 0 ? -v : v;
  const int z = __clzll((long long)a) - 1;
  const unsigned long long m = ((a << z) + 512) >> 10;  // 2^52 .. 2^53
  unsigned h = (unsigned)(m >> 32) + ((unsigned)(e - z) << 20);
  h = a ? h : 0u;
  return __hiloint2double((int)(h | ((unsigned)(v >> 32) & 0x80000000u)), (int)(unsigned)m);
}
__device__ __forceinline__ void stencil_join(const float (&acc)[kLev][4], unsigned top, const StencilAt& s, double2 (&out)[2]) {
  const int er = (int)(top & 0xffffu) + s.shift, ei = (int)(top >> 16) + s.shift;
  out[0] = double2{stencil_value(acc, 0, er + s.ew0), stencil_value(acc, 2, ei + s.ew0)};
  out[1] = double2{stencil_value(acc, 1, er + s.ew1), stencil_value(acc, 3, ei + s.ew1)};
}

constexpr int kNearBits = 8, kNearBits32 = 14;

// The digits' part.  PAIR: four modes at two tiles, lanes g < 4 at the first
// (table s.tab), the others at the next (if two).  Every lane goes through both
// tables' products, which are the cheap part, and joins its own.
template <bool PAIR>
__device__ __forceinline__ void stencil_by_digits(const double2 (&x)[4], unsigned top, const StencilAt& s, bool two,
                                                  bool second, double2 (&out)[2]) {
  uint4 a[kDig];
  float acc[kLev][4];
  stencil_digits(x, top, a);
  stencil_products(a, s.tab, acc);
  if (PAIR && two) {
    float acc1[kLev][4];
    stencil_products(a, s.tab + kTileB, acc1);
#pragma unroll
    for (int l = 0; l < kLev; ++l)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[l][q] = second ? acc1[l][q] : acc[l][q];
  }
  stencil_join(acc, top, s, out);
}
// That as one copy of the code per kernel, for blocks that have an SM to
// themselves and go through it once per use: there fetching the instructions
// is most of its time.
struct StencilRows {
  double2 v[2];
};
static __device__ __noinline__ StencilRows stencil_call(double2 x0, double2 x1, double2 x2, double2 x3, unsigned top,
                                                        StencilAt s, bool two, bool second) {
  const double2 x[4] = {x0, x1, x2, x3};
  StencilRows out;
  stencil_by_digits<true>(x, top, s, two, second, out.v);
  return out;
}
// The derivative at this lane's rows; at: as for stencil_fma, after put(x).
template <bool PAIR, bool CALL, typename Put, typename At>
__device__ __forceinline__ void dft_stencil(const double2 (&x)[4], const StencilAt& s, bool two, bool second, Put put,
                                            At at, double2 (&out)[2]) {
  const StencilWindow w = stencil_window(x);
  bool all, row[2];
  const unsigned cols = stencil_steep<kNearBits, true>(x, w, s.i0, s.N, &all, row);
  out[0] = out[1] = double2{0.0, 0.0};
  if (!all) {
    if constexpr (CALL) {
      const StencilRows r = stencil_call(x[0], x[1], x[2], x[3], w.top, s, two, second);
      out[0] = r.v[0];
      out[1] = r.v[1];
    } else {
      stencil_by_digits<PAIR>(x, w.top, s, two, second, out);
    }
  }
  if (cols) {
    put(x);
    stencil_fma(cols, s, at, out);
  }
}
// The same to FP32: five digits and levels are about 2^-39 of the window's
// largest value, against FP32 multiply-adds' 2^-24 of a row's own terms, which
// only the rows that need them take.
template <typename Put, typename At>
__device__ __forceinline__ void dft_stencil32(const double2 (&x)[4], const StencilAt& s, Put put, At at,
                                              float2 (&out)[2]) {
  constexpr int kD = 5;
  const StencilWindow w = stencil_window(x);
  uint4 a[kD];
  float acc[kD][4];
  stencil_digits(x, w.top, a);
  stencil_products(a, s.tab, acc);
  auto value = [&](int q, unsigned emax, int ew) {  // in units of level 3
    const int hi = stencil_levels(acc[0][q], acc[1][q]), lo = stencil_levels(acc[2][q], acc[3][q]);
    const int low = lo + ((__float_as_int(acc[4][q]) - __float_as_int(kDftBias) + 256) >> 9);
    // a power of two in two factors, for results down to the least subnormal
    const int e = min(max((int)emax + ew + s.shift - 1022 - 43, -252), 254), e1 = e >> 1;
    return fmaf((float)hi, 262144.f, (float)low) * __int_as_float((127 + e1) << 23) * __int_as_float((127 + e - e1) << 23);
  };
  out[0] = float2{value(0, w.top & 0xffffu, s.ew0), value(2, w.top >> 16, s.ew0)};
  out[1] = float2{value(1, w.top & 0xffffu, s.ew1), value(3, w.top >> 16, s.ew1)};
  bool all, row[2];
  const unsigned cols = stencil_steep<kNearBits32, false>(x, w, s.i0, s.N, &all, row);
  if (cols) {
    double2 y[2] = {double2{0.0, 0.0}, double2{0.0, 0.0}};
    put(x);
    stencil_fma(cols, s, at, y);  // (in FP64: converting the data takes its unit longer)
    bool rare = false;
    float2 f[2] = {float2{to_float(y[0].x, &rare), to_float(y[0].y, &rare)},
                   float2{to_float(y[1].x, &rare), to_float(y[1].y, &rare)}};
    if (rare) {
      f[0] = float2{(float)y[0].x, (float)y[0].y};
      f[1] = float2{(float)y[1].x, (float)y[1].y};
    }
    if (row[0]) out[0] = f[0];
    if (row[1]) out[1] = f[1];
  }
}
#endif  // __CUDACC__

}  // namespace opf
