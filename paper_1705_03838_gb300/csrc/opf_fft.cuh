// Batched mixed-radix FFTs in shared memory (Stockham autosort, radices
// 2, 3, 4, 5, 8 and composites of them in registers), used for the Eq. 1 transforms on the 3K x 3M grid.
//
// A block transforms `batch` sequences of length p.n stored at stride `ld`
// (complex elements) in buffer a, ping-ponging with buffer b; the returned
// pointer is whichever buffer holds the result.  sign = +1 synthesises
// (sum_k X_k e^{+2 pi i jk/n}), sign = -1 analyses; no scaling.
// tw[t] = e^{+2 pi i t/n}, t < n, in shared or global memory.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "opf_internal.h"

namespace opf {

template <typename V> struct Scalar;
template <> struct Scalar<double2> { using T = double; };
template <> struct Scalar<float2> { using T = float; };

template <typename V>
__device__ __forceinline__ V cadd(V a, V b) { return V{a.x + b.x, a.y + b.y}; }
template <typename V>
__device__ __forceinline__ V csub(V a, V b) { return V{a.x - b.x, a.y - b.y}; }
// Multiply-adds are written out wherever a product meets a sum, so that every
// kernel that inlines a transform rounds alike.
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }
template <typename V>
__device__ __forceinline__ V cmul(V a, V b) {
  return V{madd(a.x, b.x, -(a.y * b.y)), madd(a.x, b.y, a.y * b.x)};
}
template <typename V, typename T>
__device__ __forceinline__ V cmadd(T f, V a, V b) { return V{madd(f, a.x, b.x), madd(f, a.y, b.y)}; }
// multiply by s*i (s = +-1)
template <typename V>
__device__ __forceinline__ V cmul_si(V a, int s) { return s > 0 ? V{-a.y, a.x} : V{a.y, -a.x}; }

// In-place DFT of size R on v[0..R-1] with kernel e^{sign 2 pi i tq/R}.
// Radix 8 with v[3] = v[4] = 0 (the first stage of a synthesis whose middle
// third is the zero padding of the 3/2 rule): the same outputs as
// butterfly<8> without the additions of the two zero inputs.
template <typename V>
__device__ __forceinline__ void butterfly8_zm(V* v, int sign) {
  using T = typename Scalar<V>::T;
  // even points (v0, v2, 0, v6)
  const V ec = cadd(v[2], v[6]), ed = cmul_si(csub(v[2], v[6]), sign);
  V e[4] = {cadd(v[0], ec), cadd(v[0], ed), csub(v[0], ec), csub(v[0], ed)};
  // odd points (v1, 0, v5, v7)
  const V oa = cadd(v[1], v[5]), ob = csub(v[1], v[5]);
  const V od = cmul_si(V{-v[7].x, -v[7].y}, sign);
  V o[4] = {cadd(oa, v[7]), cadd(ob, od), csub(oa, v[7]), csub(ob, od)};
  const T h = (T)0.70710678118654752440;  // 1 / sqrt(2)
  const T s = (T)sign;
  const V o1 = csub(o[1], V{s * o[1].y, -s * o[1].x});  // (times h below)
  const V o2 = cmul_si(o[2], sign);
  const V o3 = csub(V{-s * o[3].y, s * o[3].x}, o[3]);
  v[0] = cadd(e[0], o[0]);
  v[4] = csub(e[0], o[0]);
  v[1] = cmadd(h, o1, e[1]);
  v[5] = cmadd(-h, o1, e[1]);
  v[2] = cadd(e[2], o2);
  v[6] = csub(e[2], o2);
  v[3] = cmadd(h, o3, e[3]);
  v[7] = cmadd(-h, o3, e[3]);
}

// cos and sin of 2 pi i / n for the compile-time twiddles below (the series; |x| <= pi).
__host__ __device__ constexpr double turn_cos(int i, int n) {
  const double x = 6.283185307179586476925 * (2 * i > n ? i - n : i) / n;
  double t = 1.0, s = 1.0;
  for (int k = 1; k < 20; ++k) {
    t *= -x * x / ((2 * k - 1) * (2 * k));
    s += t;
  }
  return s;
}
__host__ __device__ constexpr double turn_sin(int i, int n) {
  const double x = 6.283185307179586476925 * (2 * i > n ? i - n : i) / n;
  double t = x, s = x;
  for (int k = 1; k < 20; ++k) {
    t *= -x * x / ((2 * k) * (2 * k + 1));
    s += t;
  }
  return s;
}

template <int R, typename V>
__device__ __forceinline__ void butterfly(V* v, int sign);

// v times e^{sign 2 pi i E/R}
template <int R, int E, typename V>
__device__ __forceinline__ V cmul_root(V v, int sign) {
  using T = typename Scalar<V>::T;
  if constexpr (E % R == 0) {
    return v;
  } else if constexpr (4 * E % R == 0) {
    constexpr int quarter = 4 * E / R % 4;
    if constexpr (quarter == 2) return V{-v.x, -v.y};
    else return cmul_si(v, quarter == 1 ? sign : -sign);
  } else {
    constexpr T c = (T)turn_cos(E % R, R), s = (T)turn_sin(E % R, R);
    return cmul(v, V{c, sign > 0 ? s : -s});
  }
}

// Size P Q in registers: P-point transforms of every Q-th value, roots of
// unity, Q-point transforms.
template <int P, int Q, int QI, int KI, typename V>
__device__ __forceinline__ void butterfly_roots(V (&y)[P * Q], int sign) {  // y[q P + k]
  if constexpr (QI < Q) {
    y[QI * P + KI] = cmul_root<P * Q, QI * KI>(y[QI * P + KI], sign);
    if constexpr (KI + 1 < P) butterfly_roots<P, Q, QI, KI + 1>(y, sign);
    else butterfly_roots<P, Q, QI + 1, 0>(y, sign);
  }
}
template <int P, int Q, typename V>
__device__ __forceinline__ void butterfly_pq(V* v, int sign) {
  V y[P * Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
#pragma unroll
    for (int i = 0; i < P; ++i) y[q * P + i] = v[q + Q * i];
    butterfly<P>(y + q * P, sign);
  }
  butterfly_roots<P, Q, 0, 0>(y, sign);
#pragma unroll
  for (int k = 0; k < P; ++k) {
    V z[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) z[q] = y[q * P + k];
    butterfly<Q>(z, sign);
#pragma unroll
    for (int q = 0; q < Q; ++q) v[k + P * q] = z[q];
  }
}

template <int R, typename V>
__device__ __forceinline__ void butterfly(V* v, int sign) {
  using T = typename Scalar<V>::T;
  if constexpr (R == 6) butterfly_pq<2, 3>(v, sign);
  else if constexpr (R == 9) butterfly_pq<3, 3>(v, sign);
  else if constexpr (R == 12) butterfly_pq<4, 3>(v, sign);
  else if constexpr (R == 16) butterfly_pq<4, 4>(v, sign);
  else if constexpr (R == 24) butterfly_pq<8, 3>(v, sign);
  else if constexpr (R == 2) {
    const V a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  } else if constexpr (R == 4) {
    const V a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
    const V c = cadd(v[1], v[3]), d = cmul_si(csub(v[1], v[3]), sign);
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = cadd(b, d);
    v[3] = csub(b, d);
  } else if constexpr (R == 3) {
    const T h = (T)0.86602540378443864676;  // sin(2 pi / 3)
    const V t1 = cadd(v[1], v[2]), t2 = csub(v[1], v[2]);
    const V base = cmadd((T)-0.5, t1, v[0]);
    const V rot = cmul_si(t2, sign);
    v[0] = cadd(v[0], t1);
    v[1] = cmadd(h, rot, base);
    v[2] = cmadd(-h, rot, base);
  } else if constexpr (R == 8) {
    // two radix-4 transforms of the even and odd points, joined by the
    // eighth roots of unity w^q = e^{sign 2 pi i q/8}
    V e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    butterfly<4>(e, sign);
    butterfly<4>(o, sign);
    const T h = (T)0.70710678118654752440;  // 1 / sqrt(2)
    const T s = (T)sign;
    const V o1 = csub(o[1], V{s * o[1].y, -s * o[1].x});  // (times h below)
    const V o2 = cmul_si(o[2], sign);
    const V o3 = csub(V{-s * o[3].y, s * o[3].x}, o[3]);
    v[0] = cadd(e[0], o[0]);
    v[4] = csub(e[0], o[0]);
    v[1] = cmadd(h, o1, e[1]);
    v[5] = cmadd(-h, o1, e[1]);
    v[2] = cadd(e[2], o2);
    v[6] = csub(e[2], o2);
    v[3] = cmadd(h, o3, e[3]);
    v[7] = cmadd(-h, o3, e[3]);
  } else if constexpr (R == 5) {
    const T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;
    const T s1 = (T)0.95105651629515357212, s2 = (T)0.58778525229247312917;
    const V t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const V t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
    const V a1 = V{v[0].x + c1 * t1.x + c2 * t2.x, v[0].y + c1 * t1.y + c2 * t2.y};
    const V a2 = V{v[0].x + c2 * t1.x + c1 * t2.x, v[0].y + c2 * t1.y + c1 * t2.y};
    const V b1 = cmul_si(V{s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y}, sign);
    const V b2 = cmul_si(V{s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y}, sign);
    v[0] = cadd(v[0], cadd(t1, t2));
    v[1] = cadd(a1, b1);
    v[4] = csub(a1, b1);
    v[2] = cadd(a2, b2);
    v[3] = csub(a2, b2);
  }
}

template <int R, typename V>
__device__ __forceinline__ void fft_stage(const V* __restrict__ a, V* __restrict__ b, int n, int ld,
                                          int batch, int Ns, const V* __restrict__ tw, int sign) {
  const int nR = n / R;
  const int work = batch * nR;
  const int step = n / (Ns * R);
  for (int w = threadIdx.x; w < work; w += blockDim.x) {
    const int bt = w / nR;
    const int j = w - bt * nR;
    const int jm = j % Ns;
    const V* src = a + bt * ld;
    V* dst = b + bt * ld;
    V v[R];
    v[0] = src[j];
#pragma unroll
    for (int q = 1; q < R; ++q) {
      V t = tw[q * jm * step];
      if (sign < 0) t.y = -t.y;
      v[q] = cmul(src[j + q * nR], t);
    }
    butterfly<R>(v, sign);
    const int d0 = (j / Ns) * Ns * R + jm;
#pragma unroll
    for (int q = 0; q < R; ++q) dst[d0 + q * Ns] = v[q];
  }
}

template <typename V>
__device__ V* block_fft(V* a, V* b, int batch, int ld, const FftPlan& p, const V* tw, int sign) {
  int Ns = 1;
  for (int s = 0; s < p.nst; ++s) {
    const int R = p.rad[s];
    switch (R) {
      case 2: fft_stage<2>(a, b, p.n, ld, batch, Ns, tw, sign); break;
      case 3: fft_stage<3>(a, b, p.n, ld, batch, Ns, tw, sign); break;
      case 4: fft_stage<4>(a, b, p.n, ld, batch, Ns, tw, sign); break;
      default: fft_stage<5>(a, b, p.n, ld, batch, Ns, tw, sign); break;
    }
    __syncthreads();
    V* t = a;
    a = b;
    b = t;
    Ns *= R;
  }
  return a;
}

// ---------------------------------------------------------------------------
// The same Stockham transform for a length N known at compile time (the
// common grid lengths 3K, 3M): radices, strides and the twiddle stride are
// constants, so the index arithmetic folds into shifts and multiply-highs, the
// first stage (all twiddles 1) skips its multiplications, and radix 8 cuts the
// number of shared-memory passes.  Same conventions as block_fft.
//
// The buffers between two stages hold element i of a sequence at
// fft_swz(i) = i ^ ((i >> 3) & 7) (a permutation inside each group of eight;
// every compiled length is a multiple of 8): the first stage writes element
// j R + q for consecutive j, a stride of R complex values that would put a
// warp's stores on two or four of the 16 eight-byte bank pairs, and the
// permutation spreads them.  The caller's input and the result are in the
// plain layout; the arithmetic is unchanged.
__host__ __device__ constexpr int fft_swz(int i) { return i ^ ((i >> 3) & 7); }

template <int R, int N, int NS, int SIGN, bool SWR, bool SWW, bool ZM, typename V>
__device__ __forceinline__ void fft_stage_c(const V* __restrict__ a, V* __restrict__ b, int ld, int batch,
                                            const V* __restrict__ tw) {
  constexpr bool zm = ZM && NS == 1 && R == 8;  // inputs 3 and 4 lie in the zero middle third
  static_assert(N % 8 == 0, "the swizzle permutes groups of eight");
  constexpr int nR = N / R, step = N / (NS * R);
  const int work = batch * nR;
  for (int w = threadIdx.x; w < work; w += blockDim.x) {
    const int bt = w / nR;
    const int j = w - bt * nR;
    const int jm = j % NS;
    const V* src = a + bt * ld;
    V* dst = b + bt * ld;
    V v[R];
    v[0] = src[SWR ? fft_swz(j) : j];
#pragma unroll
    for (int q = 1; q < R; ++q) {
      const int ix = j + q * nR;
      if constexpr (zm) {
        if (q == 3 || q == 4) continue;
      }
      if constexpr (NS == 1) {
        v[q] = src[SWR ? fft_swz(ix) : ix];
      } else {
        V t = tw[q * jm * step];
        if constexpr (SIGN < 0) t.y = -t.y;
        v[q] = cmul(src[SWR ? fft_swz(ix) : ix], t);
      }
    }
    if constexpr (zm) {
      butterfly8_zm(v, SIGN);
    } else {
      butterfly<R>(v, SIGN);
    }
    const int d0 = (j / NS) * NS * R + jm;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int ox = d0 + q * NS;
      dst[SWW ? fft_swz(ox) : ox] = v[q];
    }
  }
}

template <int N, int NS, int SIGN, bool ZM, int R, int... Rest, typename V>
__device__ __forceinline__ V* fft_stages_c(V* a, V* b, int ld, int batch, const V* tw) {
  constexpr bool last = sizeof...(Rest) == 0;
  fft_stage_c<R, N, NS, SIGN, (NS > 1), !last, ZM>(a, b, ld, batch, tw);
  __syncthreads();
  if constexpr (last) {
    return b;
  } else {
    return fft_stages_c<N, NS * R, SIGN, ZM, Rest...>(b, a, ld, batch, tw);
  }
}

// Element e < count of a block-wide copy: v = load(e), then store(e, v), with
// U loads in flight per thread (thread t takes e = t, t + blockDim.x, ...,
// as a plain strided loop would, so coalescing is the same).
template <int U, typename V, typename Load, typename Store>
__device__ __forceinline__ void block_copy_batched(int count, Load load, Store store) {
  for (int b = threadIdx.x; b < count; b += U * blockDim.x) {
    V v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = b + u * blockDim.x;
      if (e < count) v[u] = load(e);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int e = b + u * blockDim.x;
      if (e < count) store(e, v[u]);
    }
  }
}

// Lengths with a compiled plan (others use block_fft).
__host__ __device__ constexpr bool fft_length_compiled(int n) {
  return n == 48 || n == 72 || n == 96 || n == 192 || n == 384;
}

// The two passes of an FP32 transform: a synthesis takes r1 then r2, an
// analysis r2 then r1, so that the points a thread gets from the last pass of
// one are those it needs for the first pass of the other (k_product).
struct FftRadices {
  int r1, r2;
};
__host__ __device__ constexpr FftRadices fft_radices32(int n) {
  return n == 48 ? FftRadices{8, 6} : n == 72 ? FftRadices{9, 8} : n == 96 ? FftRadices{12, 8}
       : n == 192 ? FftRadices{16, 12} : FftRadices{24, 16};
}
// Butterfly j of the first pass with inputs load(i), i = j + q N / R, into the
// sequence dst (swizzled); of the last pass (twiddles tw) from src into v, whose
// v[q] is output j + q N / R.  The arithmetic is fft_stage_c's.
template <int R, int N, int SIGN, bool ZM, typename V, typename Load>
__device__ __forceinline__ void fft_first(int j, V* __restrict__ dst, Load load) {
  constexpr bool zm = ZM && R == 8;
  V v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    if (zm && (q == 3 || q == 4)) continue;
    v[q] = load(j + q * (N / R));
  }
  if constexpr (zm) butterfly8_zm(v, SIGN);
  else butterfly<R>(v, SIGN);
#pragma unroll
  for (int q = 0; q < R; ++q) dst[fft_swz(j * R + q)] = v[q];
}
template <int R, int N, int SIGN, typename V>
__device__ __forceinline__ void fft_last(int j, const V* __restrict__ src, const V* __restrict__ tw, V (&v)[R]) {
  v[0] = src[fft_swz(j)];
#pragma unroll
  for (int q = 1; q < R; ++q) {
    V t = tw[q * j];
    if constexpr (SIGN < 0) t.y = -t.y;
    v[q] = cmul(src[fft_swz(j + q * (N / R))], t);
  }
  butterfly<R>(v, SIGN);
}

// ZERO_MID: the inputs in the middle third, positions (N/3, 2N/3), are zero
// (a synthesis of the 3/2 rule); the radix-8 first stages then skip them.
template <int N, int SIGN, bool ZERO_MID = false, typename V>
__device__ __forceinline__ V* block_fft_c(V* a, V* b, int batch, int ld, const V* tw) {
  static_assert(fft_length_compiled(N), "no compiled plan for this length");
  // FP32: two passes over shared memory, whose load and store pipe bounds the
  // transforms, with radices up to 24 in registers, where 3 or 4 passes (8 4 4 3
  // at 384) took 221 against 197 us in the z synthesis and 504 against 467 us in
  // the product at N = 128, 255 x 128 modes.  (Their kernels now take the same
  // passes without the buffers; this form serves the fused launch.)  FP64 has
  // no registers for it.
  if constexpr (sizeof(V) == sizeof(float2)) {
    constexpr FftRadices r = fft_radices32(N);
    if constexpr (SIGN > 0) return fft_stages_c<N, 1, SIGN, ZERO_MID, r.r1, r.r2>(a, b, ld, batch, tw);
    else return fft_stages_c<N, 1, SIGN, ZERO_MID, r.r2, r.r1>(a, b, ld, batch, tw);
  } else {  // (FP64 lengths up to 96 are digit products)
    static_assert(N == 192 || N == 384, "no compiled FP64 plan for this length");
    if constexpr (N == 192) return fft_stages_c<192, 1, SIGN, ZERO_MID, 8, 8, 3>(a, b, ld, batch, tw);
    else return fft_stages_c<384, 1, SIGN, ZERO_MID, 8, 4, 4, 3>(a, b, ld, batch, tw);
  }
}

// Calls f(std::integral_constant<int, n>) for a compiled length n, else
// f(std::integral_constant<int, 0>) (runtime plan).
template <class F>
inline void with_fft_length(int n, F&& f) {
  switch (n) {
    case 48: f(std::integral_constant<int, 48>{}); break;
    case 72: f(std::integral_constant<int, 72>{}); break;
    case 96: f(std::integral_constant<int, 96>{}); break;
    case 192: f(std::integral_constant<int, 192>{}); break;
    case 384: f(std::integral_constant<int, 384>{}); break;
    default: f(std::integral_constant<int, 0>{}); break;
  }
}

// The same for FP64, where lengths up to 96 are products with digit tables
// (opf_dft.cu) and only longer ones come here.
template <class F>
inline void with_long_fft_length(int n, F&& f) {
  switch (n) {
    case 192: f(std::integral_constant<int, 192>{}); break;
    case 384: f(std::integral_constant<int, 384>{}); break;
    default: f(std::integral_constant<int, 0>{}); break;
  }
}

}  // namespace opf
