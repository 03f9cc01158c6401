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
// N = 48, 96 x 72: 33, 82, 26 -> 20, 40, 18 us; 64 x (N = 32, 48 x 48): 321,
// 956, 199 -> 184, 412, 106 us; N = 32, 48 x 48: 13, 25, 13 -> 10, 21, 11 us.
// What bounds them now is the latency of their phases at 16 warps per SM: the
// tensor pipe is a third to two thirds busy in the products, the integer
// units in the splitting and joining.  The work grows with the square of the
// length, the FFT's does not: lengths above 96 stay with it.
// Symmetry halves the work: with c, s the cosine and sine sums over
// harmonics h (or points p), a result at p and its mirror n - p are c + s and
// c - s (up to factors i).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>

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

// The digits, most significant first, of a fixed-point value |v| <= 2^55 as
// half bits' integers d_0 = -128..128, d_1.. = -128..127.
__host__ __device__ inline int dft_digit(long long v, int i) {
  const unsigned long long y = (unsigned long long)v + 0x0080808080808080ull;
  return (i == 0 ? (int)(y >> 48) : (int)((y >> (8 * (6 - i))) & 255)) - 128;
}

struct StencilTable {
  const uint2* tab;  // [parity][tile][digit][lane]
  const int* ew;     // [parity][8 tiles]
  int tiles, off;    // row i sits at i + off of the tiles
};
StencilTable stencil_at(const void* p, int N);  // p as filled by stencil_host_table
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
// x in fixed point, rounded to nearest: units of 2^(emax - 1022 - 55 + half),
// emax the largest biased exponent among the values that share it (200 at
// least), |result| <= 2^(55 - half); half = 1 leaves room for the sum of two.
__host__ __device__ inline long long dft_fixed(double x, int emax, int half) {
  const unsigned long long b = dft_bits(x);
  const unsigned h = (unsigned)(b >> 32);
  const int e = (h >> 20) & 0x7ff;
  const unsigned hm = e ? ((h & 0xfffffu) | 0x100000u) : 0u;
  const unsigned long long m = ((unsigned long long)hm << 32) | (e ? (unsigned)b : 0u);
  const int s0 = (emax < 200 ? 200 : emax) - e + half, sh = s0 < 63 ? s0 : 63;
  const unsigned long long r = (((m << 3) >> sh) + 1) >> 1;
  return (h & 0x80000000u) ? -(long long)r : (long long)r;
}
// Table entry of (parity's) stencils d1 = [N][9]: fixed point of the weight
// that output row i gives row j, and the largest biased exponent of row i.
__host__ __device__ inline int stencil_exponent(const double* d1, int i) {
  int e = 0;
  for (int q = 0; q < 9; ++q) {
    const int f = (int)(dft_bits(d1[i * 9 + q]) >> 52) & 0x7ff;
    e = f > e ? f : e;
  }
  return e;
}
__host__ __device__ inline long long stencil_weight(const double* d1, int N, int i, int j) {
  const int lo = i - 4 < 0 ? 0 : (i - 4 > N - 9 ? N - 9 : i - 4);
  if (i < 0 || i >= N || j < 0 || j >= N || j < lo || j > lo + 8) return 0;
  return dft_fixed(d1[i * 9 + j - lo], stencil_exponent(d1, i), 0);
}

// Entry (k, n) of a table in fixed point: v(k, n), zero outside K x N.
#pragma nv_exec_check_disable
template <class V>
__host__ __device__ inline void table_entry(long idx, int KT, V v, uint2* out) {
  // idx = (nt * KT + kt) * 32 + lane
  const int lane = (int)(idx % 32), kt = (int)(idx / 32 % KT), nt = (int)(idx / 32 / KT);
  const int t = lane & 3, n = nt * 8 + (lane >> 2), k0 = kt * 16 + 2 * t;
  const long long f[4] = {v(k0, n), v(k0 + 1, n), v(k0 + 8, n), v(k0 + 9, n)};
  for (int i = 0; i < kDig; ++i) {
    unsigned short h[4];
    for (int q = 0; q < 4; ++q) {  // a small integer as a half
      const int d = dft_digit(f[q], i);
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
  table_entry(idx % (32L * NT), 1, [=](int k, int n) -> long long {
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

// Scaling of one row's results, which count 2^(e - 54): the exponent field's
// offset and, for a row with a non-finite value (or one above 2^877), the bits
// that make every result NaN.
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
// the stencil.  Nine FP64 multiply-adds per point and part become none.
//
// x: this lane's column (lane = 4 g + t) at rows 2t, 2t+1 of the tile, then of
// its halo (stencil_row); tab: the tile's table plus lane; ew: the exponents
// of output rows 2t, 2t+1.
// The window's digits as a fragment, DIG of them; er, ei: the columns' exponents.
template <int DIG>
__device__ __forceinline__ void stencil_digits(const double2 (&x)[4], uint4 (&a)[DIG], int* er_out, int* ei_out) {
  int er = 0, ei = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    er = max(er, dft_exponent(x[q].x));
    ei = max(ei, dft_exponent(x[q].y));
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    er = max(er, __shfl_xor_sync(0xffffffffu, er, o));
    ei = max(ei, __shfl_xor_sync(0xffffffffu, ei, o));
  }
  unsigned r[kDig];
  dft_split(dft_fixed(x[0].x, er, 0), dft_fixed(x[1].x, er, 0), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].x = r[i];
  dft_split(dft_fixed(x[0].y, ei, 0), dft_fixed(x[1].y, ei, 0), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].y = r[i];
  dft_split(dft_fixed(x[2].x, er, 0), dft_fixed(x[3].x, er, 0), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].z = r[i];
  dft_split(dft_fixed(x[2].y, ei, 0), dft_fixed(x[3].y, ei, 0), r);
#pragma unroll
  for (int i = 0; i < DIG; ++i) a[i].w = r[i];
  *er_out = er;
  *ei_out = ei;
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
__device__ __forceinline__ void stencil_join(const float (&acc)[kLev][4], int er, int ei, int ew0, int ew1,
                                             double2 (&out)[2]) {
  unsigned w[4][kLev / 2];
  dft_pairs(acc, w);
  out[0] = double2{dft_value(w[0], dft_scale(er, ew0)), dft_value(w[2], dft_scale(ei, ew0))};
  out[1] = double2{dft_value(w[1], dft_scale(er, ew1)), dft_value(w[3], dft_scale(ei, ew1))};
}
__device__ __forceinline__ void dft_stencil(const double2 (&x)[4], const uint2* __restrict__ tab, int ew0, int ew1,
                                            double2 (&out)[2]) {
  uint4 a[kDig];
  float acc[kLev][4];
  int er, ei;
  stencil_digits<kDig>(x, a, &er, &ei);
  stencil_products<kDig, kLev>(a, tab, acc);
  stencil_join(acc, er, ei, ew0, ew1, out);
}
// Four modes at two tiles: lanes g < 4 at the first (table tab), the others at
// the next (if two).  Every lane goes through both tables' products, which are
// the cheap part, and joins its own.
__device__ __forceinline__ void dft_stencil_pair(const double2 (&x)[4], const uint2* __restrict__ tab, bool two,
                                                 bool second, int ew0, int ew1, double2 (&out)[2]) {
  uint4 a[kDig];
  float acc[kLev][4];
  int er, ei;
  stencil_digits<kDig>(x, a, &er, &ei);
  stencil_products<kDig, kLev>(a, tab, acc);
  if (two) {
    float acc1[kLev][4];
    stencil_products<kDig, kLev>(a, tab + kTileB, acc1);
#pragma unroll
    for (int l = 0; l < kLev; ++l)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[l][q] = second ? acc1[l][q] : acc[l][q];
  }
  stencil_join(acc, er, ei, ew0, ew1, out);
}
// That as one copy of the code per kernel, for blocks that have an SM to
// themselves and go through it once per use: there fetching the instructions
// is most of its time.
struct StencilPair {
  double2 v[2];
};
static __device__ __noinline__ StencilPair dft_stencil_call(double2 x0, double2 x1, double2 x2, double2 x3,
                                                            const uint2* __restrict__ tab, bool two, bool second,
                                                            int ew0, int ew1) {
  const double2 x[4] = {x0, x1, x2, x3};
  StencilPair out;
  dft_stencil_pair(x, tab, two, second, ew0, ew1, out.v);
  return out;
}
// The same to FP32: five digits and levels are 2^-39 of the largest term.
__device__ __forceinline__ void dft_stencil32(const double2 (&x)[4], const uint2* __restrict__ tab, int ew0, int ew1,
                                              float2 (&out)[2]) {
  constexpr int kD = 5;
  uint4 a[kD];
  float acc[kD][4];
  int er, ei;
  stencil_digits<kD>(x, a, &er, &ei);
  stencil_products<kD, kD>(a, tab, acc);
  auto value = [&](int q, int emax, int shift) {  // in units of level 3, 2^(e - 38)
    const unsigned hi = (unsigned)__float_as_int(acc[0][q]) * 256u + (unsigned)__float_as_int(acc[1][q]) - kDftPair;
    const unsigned lo = (unsigned)__float_as_int(acc[2][q]) * 256u + (unsigned)__float_as_int(acc[3][q]) - kDftPair;
    const int low = (int)lo + (__float_as_int(acc[4][q]) - __float_as_int(kDftBias) + 128 >> 8);
    const int e = max(emax, 200) - 1022 + shift - 38 + 127;
    const float s = emax >= 1900 ? __int_as_float(0x7fc00000) : e > 0 ? __int_as_float(min(e, 254) << 23) : 0.f;
    return fmaf((float)(int)hi, 65536.f, (float)low) * s;
  };
  out[0] = float2{value(0, er, ew0), value(2, ei, ew0)};
  out[1] = float2{value(1, er, ew1), value(3, ei, ew1)};
}
#endif  // __CUDACC__

}  // namespace opf
