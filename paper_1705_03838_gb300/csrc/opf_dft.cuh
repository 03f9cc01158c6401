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

#include <cstdint>

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

// x in fixed point, rounded to nearest: |result| <= 2^(55 - half), half = 1
// leaves room for the sum of two.  emax as in dft_scale (there shift = half).
__device__ __forceinline__ long long dft_fixed(double x, int emax, int half) {
  const unsigned h = (unsigned)__double2hiint(x);
  const int e = (h >> 20) & 0x7ff;
  const unsigned hm = e ? ((h & 0xfffffu) | 0x100000u) : 0u;
  const unsigned long long m = ((unsigned long long)hm << 32) | (e ? (unsigned)__double2loint(x) : 0u);
  const int sh = min(max(emax, 200) - e + half, 63);
  const unsigned long long r = (((m << 3) >> sh) + 1) >> 1;
  return (h & 0x80000000u) ? -(long long)r : (long long)r;
}

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
#endif  // __CUDACC__

}  // namespace opf
