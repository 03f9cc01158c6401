// FP64 transforms of the nonlinear term (section 2.2) for lengths up to 96 on
// the tensor cores (opf_dft.cuh): z synthesis, theta transforms with the
// product u x omega, z analysis.  Same inputs, outputs and layouts as the FFT
// kernels of opf_kernels.cu, which take the longer transforms.
#include <algorithm>
#include <cmath>
#include <vector>

#include "opf_dft.cuh"
#include "opf_internal.h"
#include "opf_step.cuh"

namespace opf {

namespace {
constexpr int kThreads = 256, kWarps = kThreads / 32;

// ------------------------------------------------------------------ tables
// The eight matrices of a handle, in the order of DftTables.
struct TableShape {
  int H, n, anal, sine;
  double scale;   // of every entry
  double scale0;  // of the entries of harmonic 0
};
void table_shapes(int K, int M, double inv_grid, TableShape (&s)[8], int* zshift) {
  int r;
  const double g = std::frexp(inv_grid, &r);  // in [0.5, 1)
  *zshift = r;
  for (int q = 0; q < 2; ++q) {
    s[q] = TableShape{K, 3 * K, 0, q, 1.0, 1.0};
    s[2 + q] = TableShape{M, 3 * M, 0, q, 1.0, 0.5};
    s[4 + q] = TableShape{M, 3 * M, 1, q, 1.0, 1.0};
    s[6 + q] = TableShape{K, 3 * K, 1, q, g, g};
  }
}
// (0: the length takes the FFT)
long table_size(const TableShape& s) {
  if (s.H > kDftMaxH) return 0;
  return s.anal ? dft_anal_size(s.H, s.n) : dft_synth_size(s.H, s.n);
}

struct TableJobs {
  TableShape s[8];
  uint2* out[8];
  const double2* tw[8];  // e^{2 pi i t / n}, t < n
};
// One table per grid row.
__global__ void k_dft_tables(TableJobs jobs) {
  const TableShape s = jobs.s[blockIdx.y];
  uint2* out = jobs.out[blockIdx.y];
  const double2* tw = jobs.tw[blockIdx.y];
  if (!out) return;
  const int KT = s.anal ? dft_tiles(dft_points(s.n), 16) : dft_tiles(s.H, 16);
  const long total = (s.anal ? dft_anal_size(s.H, s.n) : dft_synth_size(s.H, s.n)) / kDig;
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  table_entry(idx, KT, [&](int k, int n) -> long long {
    const int h = s.anal ? n : k, p = s.anal ? k : n;
    if (h >= s.H || p >= dft_points(s.n)) return 0;
    const double2 w = tw[h * p % s.n];
    return __double2ll_rn((s.sine ? w.y : w.x) * ((h ? s.scale : s.scale0) * 36028797018963968.0));  // 2^55
  }, out);
}
}  // namespace

size_t dft_table_bytes(int K, int M) {
  TableShape s[8];
  int z;
  table_shapes(K, M, 1.0, s, &z);
  long n = 0;
  for (const TableShape& t : s) n += table_size(t);
  return (size_t)n * sizeof(uint2);
}

static void dft_set_tables(DftTables* t, const TableShape (&s)[8], int zshift, void* dev) {
  const uint2* p = (const uint2*)dev;
  for (int q = 0; q < 8; ++q) {
    t->m[q] = table_size(s[q]) ? p : nullptr;
    p += table_size(s[q]);
  }
  t->zshift = zshift;
}

void dft_host_tables(int K, int M, double inv_grid, void* host, void* dev, DftTables* t) {
  TableShape s[8];
  int zshift;
  table_shapes(K, M, inv_grid, s, &zshift);
  uint2* out = (uint2*)host;
  for (const TableShape& q : s) {
    if (!table_size(q)) continue;
    const int KT = q.anal ? dft_tiles(dft_points(q.n), 16) : dft_tiles(q.H, 16);
    std::vector<long long> fixed(q.n), fixed0(q.n);  // by the phase h p mod n
    for (int i = 0; i < q.n; ++i) {
      const long double a = 2.0L * 3.14159265358979323846264338327950288L * i / q.n;
      const long double v = (q.sine ? sinl(a) : cosl(a)) * 36028797018963968.0L;  // 2^55
      fixed[i] = llrintl(v * q.scale);
      fixed0[i] = llrintl(v * q.scale0);
    }
    for (long idx = 0; idx < table_size(q) / kDig; ++idx)
      table_entry(idx, KT, [&](int k, int n) -> long long {
        const int h = q.anal ? n : k, p = q.anal ? k : n;
        if (h >= q.H || p >= dft_points(q.n)) return 0;
        return (h ? fixed : fixed0)[h * p % q.n];
      }, out);
    out += table_size(q);
  }
  dft_set_tables(t, s, zshift, dev);
}

void dft_device_tables(int K, int M, double inv_grid, const double2* twz, const double2* twth, void* dev,
                       DftTables* t, cudaStream_t st) {
  TableShape s[8];
  int zshift;
  table_shapes(K, M, inv_grid, s, &zshift);
  dft_set_tables(t, s, zshift, dev);
  TableJobs jobs;
  long most = 0;
  for (int q = 0; q < 8; ++q) {
    jobs.s[q] = s[q];
    jobs.out[q] = (uint2*)t->m[q];
    jobs.tw[q] = q >= 2 && q < 6 ? twth : twz;
    most = std::max(most, table_size(s[q]) / kDig);
  }
  if (most) k_dft_tables<<<dim3((unsigned)((most + 127) / 128), 8), 128, 0, st>>>(jobs);
}

size_t stencil_bytes(int N) {
  return (size_t)stencil_table_size(N) * sizeof(uint2) + (size_t)16 * stencil_tiles(N) * sizeof(int);
}
StencilTable stencil_at(const void* p, const double* d1, int N) {
  const uint2* tab = (const uint2*)p;
  return StencilTable{tab, (const int*)(tab + stencil_table_size(N)), d1, N, stencil_tiles(N), 8 * stencil_tiles(N) - N};
}
void stencil_host_table(const double* d1, int N, void* host) {
  uint2* tab = (uint2*)host;
  for (long idx = 0; idx < 64L * stencil_tiles(N); ++idx)
    stencil_entry(idx, d1, N, tab, (int*)(tab + stencil_table_size(N)));
}
// ------------------------------------------------------------------ z synthesis
// A row tile is eight m columns of one field and radial row: rows 0-7 their
// real parts, 8-15 the imaginary ones; the sums over harmonics of X_k + X_-k
// with cosines and of X_k - X_-k with sines give the points p and n - p.
// Block: R consecutive row tiles, whose R KT digit tiles take a warp each and
// whose R NT products are dealt out to the warps.
namespace {
struct SynthShape {
  int R, blocks;
};
// The tiles per block that take the fewest rounds of the eight warps over the
// waves of two blocks per SM: few on small grids, a digit tile for every warp
// on large ones.  (64 x (N = 32, 31 x 16 modes), whose rows are two tiles of one
// digit tile each: 184 us with a row per block, most of its warps waiting for
// the two that cut digits; 141 us with eight tiles.)
SynthShape synth_shape(const Dims& d) {
  const int KT = dft_tiles(d.K, 16), NT = dft_tiles(dft_points(d.nz), 8);
  const long tiles = 6L * d.N * ((d.M + 7) / 8), slots = 2L * device_sms();
  SynthShape best{1, 0};
  long cost = -1;
  for (int R = 1; R * KT <= kWarps; ++R) {
    const long blocks = (tiles + R - 1) / R;
    const long c = (blocks * d.B + slots - 1) / slots * (1 + (R * NT + kWarps - 1) / kWarps);
    if (cost < 0 || c < cost) {
      cost = c;
      best = SynthShape{R, (int)blocks};
    }
  }
  return best;
}
}  // namespace
size_t dft_zsynth_smem(const Dims& d) {
  return (size_t)synth_shape(d).R * 2 * dft_tiles(d.K, 16) * kTileA * sizeof(uint4);
}

// A block's results as plain sums (dft_outside), here and for the kernels
// below: functions of their own, which leave the code around them as it is.
static __device__ __noinline__ void zsynth_sums(int t0, int RT, int K, int M, int N, const double2* __restrict__ tw,
                                                const double2* __restrict__ W6, double2* Z6) {
  const int nz = 3 * K, nk = 2 * K - 1, MT = (M + 7) / 8;
  for (int e = threadIdx.x; e < RT * 8 * nz; e += blockDim.x) {
    const int p = e / 8 % nz, r = t0 + e / (8 * nz), fn = r / MT, f = fn / N, m = (r - fn * MT) * 8 + e % 8;
    if (m >= M) continue;
    const double2* x = W6 + ((long)(f * M + m) * N + fn - f * N) * nk + K - 1;
    double2 sum = double2{0.0, 0.0};
#pragma unroll 1
    for (int k = 1 - K; k < K; ++k) {
      const double2 w = tw[(k + nz) * p % nz];
      sum.x = fma(x[k].x, w.x, fma(-x[k].y, w.y, sum.x));
      sum.y = fma(x[k].x, w.y, fma(x[k].y, w.x, sum.y));
    }
    Z6[((long)fn * nz + p) * M + m] = sum;
  }
}

__global__ void __launch_bounds__(kThreads, 2)
    k_dft_zsynth(Dims d, int R, const uint2* __restrict__ Tc, const uint2* __restrict__ Ts,
                 const double2* __restrict__ tw, const double2* __restrict__ W6, double2* __restrict__ Z6) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int emx[kWarps][8], outside;
  const int K = d.K, M = d.M, N = d.N, nk = d.nk, nz = d.nz;
  const int MT = (M + 7) / 8, t0 = blockIdx.x * R, RT = min(R, 6 * N * MT - t0);
  const int KT = dft_tiles(K, 16), P = dft_points(nz), NT = dft_tiles(P, 8);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  uint4* A = (uint4*)smraw;  // [row tile][sum, difference][k tile] tiles
  W6 = bofs(W6, d.ss);
  Z6 = bofs(Z6, d.ss);
  grid_dep_trigger_at(d, 1);
  if (threadIdx.x < kWarps * 8) emx[threadIdx.x >> 3][threadIdx.x & 7] = 0;
  if (threadIdx.x == 0) outside = 0;
  double2 xp[4], xm[4];  // X_k, X_-k
  const int rt = warp / KT, kt = warp - rt * KT;  // KT <= 2: one item per warp
  const bool have = rt < RT;
  const int fn = (t0 + rt) / MT, f = fn / N, m = (t0 + rt - fn * MT) * 8 + g;  // fn = field * N + row
  const double2* src = W6 + (long)f * d.F + ((long)m * N + fn - f * N) * nk + K - 1;
  __syncthreads();
  grid_dep_wait();
  if (have) {
    int e = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = kt * 16 + 2 * t + (i & 1) + (i >> 1) * 8;
      xp[i] = xm[i] = double2{0.0, 0.0};
      if (m < M && k < K) {
        xp[i] = src[k];
        if (k > 0) xm[i] = src[-k];
      }
      e = max(e, max(max(dft_exponent(xp[i].x), dft_exponent(xp[i].y)), max(dft_exponent(xm[i].x), dft_exponent(xm[i].y))));
    }
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
    if (t == 0) atomicMax(&emx[rt][g], e);
  }
  __syncthreads();
  if (have) {
    const int e = emx[rt][g];
    if (dft_outside(e)) outside = 1;
    long long sr[4], si[4], dr[4], di[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const long long pr = dft_fixed(xp[i].x, e, 1), pi = dft_fixed(xp[i].y, e, 1);
      const long long mr = dft_fixed(xm[i].x, e, 1), mi = dft_fixed(xm[i].y, e, 1);
      sr[i] = pr + mr;
      si[i] = pi + mi;
      dr[i] = pr - mr;
      di[i] = pi - mi;
    }
    dft_put(A + ((rt * 2 + 0) * KT + kt) * kTileA, lane, sr, si);
    dft_put(A + ((rt * 2 + 1) * KT + kt) * kTileA, lane, dr, di);
  }
  __syncthreads();
  grid_dep_trigger_at(d, 2);
  for (int it = warp; it < RT * NT; it += kWarps) {
    __syncwarp();
    const int r = it % RT, nt = it / RT;
    float acc[kLev][4];
    unsigned c[4][4], s[4][4];
    dft_gemm(acc, A + (r * 2 + 0) * KT * kTileA + lane, Tc + (long)nt * KT * kTileB + lane, KT);
    dft_pairs(acc, c);
    dft_gemm(acc, A + (r * 2 + 1) * KT * kTileA + lane, Ts + (long)nt * KT * kTileB + lane, KT);
    dft_pairs(acc, s);
    const int fn = (t0 + r) / MT, m = (t0 + r - fn * MT) * 8 + g;
    const DftScale sc = dft_scale(emx[r][g], 1);
    double2* dst = Z6 + (long)fn * nz * M + m;
#pragma unroll
    for (int q = 0; q < 2; ++q) {  // e^{+i phi}: (c + i s) at p, (c - i s) at n - p
      const int p = nt * 8 + 2 * t + q;
      if (m >= M || p >= P) continue;
      dst[(long)p * M] = double2{dft_minus(c[q], s[2 + q], sc), dft_plus(c[2 + q], s[q], sc)};
      if (p > 0 && 2 * p != nz)
        dst[(long)(nz - p) * M] = double2{dft_plus(c[q], s[2 + q], sc), dft_minus(c[2 + q], s[q], sc)};
    }
  }
  if (outside) {
    __syncthreads();
    zsynth_sums(t0, RT, K, M, N, bofs(tw, d.ps), W6, Z6);
  }
}

// ------------------------------------------------------------------ theta transforms and product
// Block: 16 z rows of one radial plane, the six fields in two rounds of three.
// Row tile: the 16 rows; 2 Re and -2 Im of the coefficients against cosines
// and sines give the points q and n - q, kept in shared memory for u x omega;
// the three products go back through sums and differences of mirrored points.
namespace {
struct ProductShape {
  int ldq, KT, NT, KT2, NT2;
  int fields;  // per round
  size_t phys, a1, a2;  // bytes: one field's rows, a round's digits, the products' digits
  size_t smem;
};
__host__ __device__ inline ProductShape product_shape(int M, int nth, int fields) {
  ProductShape s;
  s.fields = fields;
  s.ldq = (nth + 7) / 16 * 16 + 8;
  s.KT = dft_tiles(M, 16);
  s.NT = dft_tiles(dft_points(nth), 8);
  s.KT2 = dft_tiles(dft_points(nth), 16);
  s.NT2 = dft_tiles(M, 8);
  s.phys = (size_t)16 * s.ldq * sizeof(double);
  s.a1 = (size_t)2 * s.fields * s.KT * kTileA * sizeof(uint4);
  s.a2 = (size_t)6 * s.KT2 * kTileA * sizeof(uint4);
  // the products' digits start where fields 3.. lay
  const size_t over = s.a2 > 3 * s.phys ? s.a2 - 3 * s.phys : 0;
  s.smem = 6 * s.phys + (s.a1 > over ? s.a1 : over);
  return s;
}
}  // namespace

static __device__ __noinline__ void theta_sums(int z0, int nz, int n, int N, int M, int nth, int ldq,
                                               const double2* __restrict__ tw, const double2* __restrict__ Z6,
                                               double* ph) {
  for (int e = threadIdx.x; e < 6 * 16 * nth; e += blockDim.x) {
    const int q = e % nth, r = e / nth, z = z0 + (r & 15);
    if (z >= nz) continue;
    const double2* x = Z6 + (((long)(r >> 4) * N + n) * nz + z) * M;
    double sum = 0.0;
#pragma unroll 1
    for (int m = 1; m < M; ++m) sum = fma(x[m].x, tw[m * q % nth].x, fma(-x[m].y, tw[m * q % nth].y, sum));
    ph[r * ldq + q] = fma(2.0, sum, x[0].x);
  }
}
static __device__ __noinline__ void theta_back_sums(int z0, int nz, int n, int N, int M, int nth, int ldq,
                                                    const double2* __restrict__ tw, const double* ph, double2* ZN) {
  for (int e = threadIdx.x; e < 3 * 16 * M; e += blockDim.x) {
    const int m = e % M, r = e / M, z = z0 + (r & 15);
    if (z >= nz) continue;
    double2 sum = double2{0.0, 0.0};
#pragma unroll 1
    for (int q = 0; q < nth; ++q) {
      const double f = ph[r * ldq + q];
      sum.x = fma(f, tw[m * q % nth].x, sum.x);
      sum.y = fma(-f, tw[m * q % nth].y, sum.y);
    }
    ZN[(((long)(r >> 4) * N + n) * nz + z) * M + m] = sum;
  }
}

// FIELDS per round.  16 warps and all six where there are no more blocks than
// SMs.  Else 8 warps, two blocks per SM: with one k tile per row (M <= 16) and
// its small footprint all six fields at once, 6 digit tiles and 24 products for
// the 8 warps where two rounds of 3 and 12 left warps waiting (64 x (N = 32,
// 31 x 16 modes) 409 -> 352 us; six warps in three blocks 379 us); else three
// (M = 30 and 32: 120 and 123 KB of shared memory, so that one block resides).
template <int WARPS, int FIELDS, int BLOCKS>
__global__ void __launch_bounds__(WARPS * 32, BLOCKS)
    k_dft_product(Dims d, const uint2* __restrict__ Sc, const uint2* __restrict__ Ss, const uint2* __restrict__ Ac,
                  const uint2* __restrict__ As, const double2* __restrict__ tw, const double2* __restrict__ Z6,
                  double2* __restrict__ ZN) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int kFields = FIELDS;
  __shared__ int emx[kFields][16], emn[3][16], outside[2];  // (of the six fields; of the products)
  const int M = d.M, N = d.N, nz = d.nz, nth = d.nth;
  const ProductShape ps = product_shape(M, nth, FIELDS);
  const int ldq = ps.ldq, KT = ps.KT, KT2 = ps.KT2, P = dft_points(nth);
  double* ph = (double*)smraw;  // [6][16][ldq]
  uint4* A1 = (uint4*)(smraw + 6 * ps.phys);
  uint4* A2 = (uint4*)(smraw + 3 * ps.phys);
  const int z0 = blockIdx.x * 16, n = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  tw = bofs(tw, d.ps);
  Z6 = bofs(Z6, d.ss);
  ZN = bofs(ZN, d.ss);
  const long fstride = (long)N * nz * M;
  grid_dep_trigger_at(d, 1);
  if (threadIdx.x < 2) outside[threadIdx.x] = 0;
  grid_dep_wait();
  for (int round = 0; round < 6 / kFields; ++round) {
    if (threadIdx.x < kFields * 16) emx[threadIdx.x >> 4][threadIdx.x & 15] = 0;
    __syncthreads();
    double2 x[4], y[4];  // rows g, g + 8
    const int fi = warp / KT, kt = warp - fi * KT;  // KT <= 2: one item per warp
    const bool have = fi < kFields;
    if (have) {
      const double2* src = Z6 + ((long)(round * kFields + fi) * N + n) * nz * M;
      int ex = 0, ey = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int m = kt * 16 + 2 * t + (i & 1) + (i >> 1) * 8;
        x[i] = y[i] = double2{0.0, 0.0};
        if (m < M && z0 + g < nz) x[i] = src[(long)(z0 + g) * M + m];
        if (m < M && z0 + g + 8 < nz) y[i] = src[(long)(z0 + g + 8) * M + m];
        if (m == 0) x[i].y = y[i].y = 0.0;
        ex = max(ex, max(dft_exponent(x[i].x), dft_exponent(x[i].y)));
        ey = max(ey, max(dft_exponent(y[i].x), dft_exponent(y[i].y)));
      }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
        ey = max(ey, __shfl_xor_sync(0xffffffffu, ey, o));
      }
      if (t == 0) {
        atomicMax(&emx[fi][g], ex);
        atomicMax(&emx[fi][g + 8], ey);
      }
    }
    __syncthreads();
    if (have) {
      const int ex = emx[fi][g], ey = emx[fi][g + 8];
      if (dft_outside(ex) || dft_outside(ey)) outside[0] = 1;
      long long xr[4], xi[4], yr[4], yi[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        xr[i] = dft_fixed(x[i].x, ex, 0);
        xi[i] = -dft_fixed(x[i].y, ex, 0);
        yr[i] = dft_fixed(y[i].x, ey, 0);
        yi[i] = -dft_fixed(y[i].y, ey, 0);
      }
      dft_put(A1 + ((fi * 2 + 0) * KT + kt) * kTileA, lane, xr, yr);
      dft_put(A1 + ((fi * 2 + 1) * KT + kt) * kTileA, lane, xi, yi);
    }
    __syncthreads();
    for (int it = warp; it < kFields * ps.NT; it += WARPS) {
      __syncwarp();
      const int fq = it % kFields, nt = it / kFields;
      float acc[kLev][4];
      unsigned c[4][4], s[4][4];
      dft_gemm(acc, A1 + (fq * 2 + 0) * KT * kTileA + lane, Sc + (long)nt * KT * kTileB + lane, KT);
      dft_pairs(acc, c);
      dft_gemm(acc, A1 + (fq * 2 + 1) * KT * kTileA + lane, Ss + (long)nt * KT * kTileB + lane, KT);
      dft_pairs(acc, s);
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // rows g, g + 8
        const DftScale sc = dft_scale(emx[fq][g + 8 * h], 1);  // twice the half sums
        double* row = ph + ((round * kFields + fq) * 16 + g + 8 * h) * ldq;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int p = nt * 8 + 2 * t + q;
          if (p >= P) continue;
          row[p] = dft_plus(c[2 * h + q], s[2 * h + q], sc);
          if (p > 0 && 2 * p != nth) row[nth - p] = dft_minus(c[2 * h + q], s[2 * h + q], sc);
        }
      }
    }
    __syncthreads();
  }
  if (outside[0]) {
    theta_sums(z0, nz, n, N, M, nth, ldq, tw, Z6, ph);
    __syncthreads();
  }
  // ---- u x omega (with the Coriolis force and the CFL number), one warp per row
  double* cfl = bofs(d.cfl, d.ss);
  double inv_dr = 0, inv_rdt = 0, inv_dz = 0;
  if (cfl) {
    const double* rinv = bofs(d.rinv_cfl, d.ps);
    const double rn = 1.0 / rinv[n];
    const double rm = n > 0 ? 1.0 / rinv[n - 1] : -rn;
    const double rp = n < N - 1 ? 1.0 / rinv[n + 1] : 1.0 + (1.0 - rm);
    inv_dr = 1.0 / fmin(rn - rm, rp - rn);
    inv_rdt = (double)(d.m_p * nth) / (6.283185307179586 * rn);
    inv_dz = d.alpha * (double)nz / 6.283185307179586;
  }
  // cos and sin of theta_q = 2 pi q / n: a transverse axis has m_p = 1
  const bool transverse = d.rot_x != 0.0 || d.rot_y != 0.0;
  double cmax = 0.0;
  for (int r = warp; r < 16; r += WARPS) {
    int e0 = 0, e1 = 0, e2 = 0;
    if (z0 + r < nz) {
      double* row = ph + r * ldq;
      const int fs = 16 * ldq;
      for (int q = lane; q < nth; q += 32) {
        const double ur = row[q], ut = row[fs + q], uz = row[2 * fs + q];
        const double wr = row[3 * fs + q], wt = row[4 * fs + q], wz = row[5 * fs + q];
        double nr = ut * wz - uz * wt, nt = uz * wr - ur * wz, nzv = ur * wt - ut * wr;
        if (d.rotate) {  // Coriolis -2 Omega x u, Omega in cylindrical components at theta_q
          const double2 w = transverse ? tw[q] : double2{0.0, 0.0};
          const double o_r = d.rot_x * w.x + d.rot_y * w.y, o_t = -d.rot_x * w.y + d.rot_y * w.x, o_z = d.rot_z;
          nr -= 2.0 * (o_t * uz - o_z * ut);
          nt -= 2.0 * (o_z * ur - o_r * uz);
          nzv -= 2.0 * (o_r * ut - o_t * ur);
        }
        row[q] = nr;
        row[fs + q] = nt;
        row[2 * fs + q] = nzv;
        e0 = max(e0, dft_exponent(nr));
        e1 = max(e1, dft_exponent(nt));
        e2 = max(e2, dft_exponent(nzv));
        if (cfl) cmax = fmax(cmax, fmax(fabs(ur) * inv_dr, fmax(fabs(ut) * inv_rdt, fabs(uz) * inv_dz)));
      }
    }
    e0 = __reduce_max_sync(0xffffffffu, e0);
    e1 = __reduce_max_sync(0xffffffffu, e1);
    e2 = __reduce_max_sync(0xffffffffu, e2);
    if (lane == 0) {
      emn[0][r] = e0;
      emn[1][r] = e1;
      emn[2][r] = e2;
    }
  }
  if (cfl) {  // warp max, then one atomic per warp (non-negative doubles order as integers)
    for (int o = 16; o > 0; o >>= 1) cmax = fmax(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    if (lane == 0 && cmax > 0.0)
      atomicMax((unsigned long long*)cfl, (unsigned long long)__double_as_longlong(cmax));
  }
  __syncthreads();
  // ---- digits of the mirrored sums and differences
  for (int it = warp; it < 3 * KT2; it += WARPS) {
    const int c = it / KT2, kt = it - c * KT2;
    long long s[2][4], df[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = g + 8 * h, e = emn[c][r];
      if (dft_outside(e)) outside[1] = 1;
      const double* row = ph + (c * 16 + r) * ldq;
      const bool in = z0 + r < nz;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int q = kt * 16 + 2 * t + (i & 1) + (i >> 1) * 8;
        long long a = 0, b = 0;
        if (in && q < P) {
          a = dft_fixed(row[q], e, 1);
          if (q > 0 && 2 * q != nth) b = dft_fixed(row[nth - q], e, 1);
        }
        s[h][i] = a + b;
        df[h][i] = a - b;
      }
    }
    dft_put(A2 + ((c * 2 + 0) * KT2 + kt) * kTileA, lane, s[0], s[1]);
    dft_put(A2 + ((c * 2 + 1) * KT2 + kt) * kTileA, lane, df[0], df[1]);
  }
  __syncthreads();
  grid_dep_trigger_at(d, 2);
  // ---- F(m) = sum f(q) e^{-i m theta}: real part the cosine sum, imaginary
  //      part minus the sine sum, an item each
  for (int it = warp; it < 6 * ps.NT2; it += WARPS) {
    __syncwarp();
    const int cc = it % 6, nt = it / 6, comp = cc >> 1, sine = cc & 1;
    float acc[kLev][4];
    unsigned w[4][4];
    dft_gemm(acc, A2 + cc * KT2 * kTileA + lane, (sine ? As : Ac) + (long)nt * KT2 * kTileB + lane, KT2);
    dft_pairs(acc, w);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int z = z0 + g + 8 * h;
      const DftScale sc = dft_scale(emn[comp][g + 8 * h], 1);
      double* dst = (double*)(ZN + comp * fstride + ((long)n * nz + z) * M) + sine;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int m = nt * 8 + 2 * t + q;
        const double v = sine ? dft_negative(w[2 * h + q], sc) : dft_value(w[2 * h + q], sc);
        if (z < nz && m < M) dst[2 * m] = v;
      }
    }
  }
  if (outside[1]) {  // (the products' rows lie below their digits)
    __syncthreads();
    theta_back_sums(z0, nz, n, N, M, nth, ldq, tw, ph, ZN);
  }
}

// ------------------------------------------------------------------ z analysis
// Block: eight m columns of one radial row, three components; row tile as in
// the synthesis.  The sums go through shared memory for the +- form and the
// addends, written along k.
size_t dft_zanalysis_smem(const Dims& d) {
  const size_t a = (size_t)6 * dft_tiles(dft_points(d.nz), 16) * kTileA * sizeof(uint4);
  return std::max(a, (size_t)24 * d.nk * sizeof(double2));
}

static __device__ __noinline__ void zanalysis_sums(int m0, int n, int K, int M, int N, double scale,
                                                   const double2* __restrict__ tw, const double2* __restrict__ ZN,
                                                   double2* R) {
  const int nz = 3 * K, nk = 2 * K - 1;
  for (int e = threadIdx.x; e < 24 * nk; e += blockDim.x) {
    const int r = e / nk, m = m0 + (r & 7), h = e - r * nk - (K - 1) + nz;  // harmonic k + nz
    if (m >= M) continue;
    const double2* x = ZN + ((long)(r >> 3) * N + n) * nz * M + m;
    double2 sum = double2{0.0, 0.0};
#pragma unroll 1
    for (int p = 0; p < nz; ++p) {
      const double2 v = x[(long)p * M], w = tw[h * p % nz];
      sum.x = fma(v.x, w.x, fma(v.y, w.y, sum.x));
      sum.y = fma(v.y, w.x, fma(-v.x, w.y, sum.y));
    }
    R[e] = double2{sum.x * scale, sum.y * scale};
  }
}

// WARPS: its 3, 6, 9 or 12 digit tiles and as many products or fewer take
// multiples of three; six, with a third block per SM where the digits fit, were
// 106 -> 86 us against eight on 64 x (N = 32, 31 x 16 modes), and twelve where
// there are no more blocks than SMs 18.3 -> 17.1 us at N = 48, 63 x 24 modes.
// There eight do for up to 8 tiles (twelve: 1 us more per launch at N = 20, 32).
template <int WARPS, int BLOCKS>
__global__ void __launch_bounds__(WARPS * 32, BLOCKS)
    k_dft_zanalysis(Dims d, int zshift, const uint2* __restrict__ Tc, const uint2* __restrict__ Ts,
                    const double2* __restrict__ tw, const double2* __restrict__ ZN, double2* __restrict__ Nout) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int emx[3][8], outside;
  const int K = d.K, M = d.M, N = d.N, nk = d.nk, nz = d.nz;
  const int KT = dft_tiles(dft_points(nz), 16), NT = dft_tiles(K, 8), P = dft_points(nz);
  const int m0 = blockIdx.x * 8, n = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  uint4* A = (uint4*)smraw;        // [3][sum, difference][k tile] tiles
  double2* R = (double2*)smraw;    // [3][8][nk], after the last product
  ZN = bofs(ZN, d.ss);
  Nout = bofs(Nout, d.ss);
  const double Re = bofs(d.prm, d.ps)[kPrmRe];
  const long fs = d.F, fstride = (long)N * nz * M;
  grid_dep_trigger_at(d, 1);
  if (threadIdx.x < 24) emx[threadIdx.x >> 3][threadIdx.x & 7] = 0;
  if (threadIdx.x == 0) outside = 0;
  __syncthreads();
  grid_dep_wait();
  constexpr int kItems = (12 + WARPS - 1) / WARPS;  // 3 KT <= 12 items
  double2 x[kItems][4], y[kItems][4];  // points p, n - p
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int it = warp + u * WARPS;
    if (it < 3 * KT) {
      const int f = it / KT, kt = it - f * KT, m = m0 + g;
      const double2* src = ZN + f * fstride + (long)n * nz * M + m;
      int e = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int p = kt * 16 + 2 * t + (i & 1) + (i >> 1) * 8;
        x[u][i] = y[u][i] = double2{0.0, 0.0};
        if (m < M && p < P) {
          x[u][i] = src[(long)p * M];
          if (p > 0 && 2 * p != nz) y[u][i] = src[(long)(nz - p) * M];
        }
        e = max(e, max(max(dft_exponent(x[u][i].x), dft_exponent(x[u][i].y)),
                       max(dft_exponent(y[u][i].x), dft_exponent(y[u][i].y))));
      }
      e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
      e = max(e, __shfl_xor_sync(0xffffffffu, e, 2));
      if (t == 0) atomicMax(&emx[f][g], e);
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int it = warp + u * WARPS;
    if (it < 3 * KT) {
      const int f = it / KT, kt = it - f * KT, e = emx[f][g];
      if (dft_outside(e)) outside = 1;
      long long sr[4], si[4], dr[4], di[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const long long pr = dft_fixed(x[u][i].x, e, 1), pi = dft_fixed(x[u][i].y, e, 1);
        const long long mr = dft_fixed(y[u][i].x, e, 1), mi = dft_fixed(y[u][i].y, e, 1);
        sr[i] = pr + mr;
        si[i] = pi + mi;
        dr[i] = pr - mr;
        di[i] = pi - mi;
      }
      dft_put(A + ((f * 2 + 0) * KT + kt) * kTileA, lane, sr, si);
      dft_put(A + ((f * 2 + 1) * KT + kt) * kTileA, lane, dr, di);
    }
  }
  __syncthreads();
  // 3 NT <= 12 products; results stay in registers until every
  // warp has read its digits
  double2 res[kItems][4];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int it = warp + u * WARPS;
    if (it < 3 * NT) {
      __syncwarp();
      const int f = it % 3, nt = it / 3;
      float acc[kLev][4];
      unsigned c[4][4], s[4][4];
      dft_gemm(acc, A + (f * 2 + 0) * KT * kTileA + lane, Tc + (long)nt * KT * kTileB + lane, KT);
      dft_pairs(acc, c);
      dft_gemm(acc, A + (f * 2 + 1) * KT * kTileA + lane, Ts + (long)nt * KT * kTileB + lane, KT);
      dft_pairs(acc, s);
      const DftScale sc = dft_scale(emx[f][g], 1 + zshift);
#pragma unroll
      for (int q = 0; q < 2; ++q) {  // e^{-i phi}: c - i s at k, c + i s at -k
        res[u][2 * q] = double2{dft_plus(c[q], s[2 + q], sc), dft_minus(c[2 + q], s[q], sc)};
        res[u][2 * q + 1] = double2{dft_minus(c[q], s[2 + q], sc), dft_plus(c[2 + q], s[q], sc)};
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int it = warp + u * WARPS;
    if (it < 3 * NT) {
      const int f = it % 3, nt = it / 3;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int k = nt * 8 + 2 * t + q;
        if (k >= K) continue;
        double2* dst = R + (f * 8 + g) * nk + K - 1;
        dst[k] = res[u][2 * q];
        if (k > 0) dst[-k] = res[u][2 * q + 1];
      }
    }
  }
  __syncthreads();
  if (outside) {
    zanalysis_sums(m0, n, K, M, N, d.inv_grid, bofs(tw, d.ps), ZN, R);
    __syncthreads();
  }
  grid_dep_trigger_at(d, 2);
  const int mcn = min(8, M - m0);
  for (int e = threadIdx.x; e < mcn * nk; e += WARPS * 32) {
    const int mc = e / nk, kk = e - mc * nk;
    const double2 r = R[mc * nk + kk], th = R[(8 + mc) * nk + kk];
    double2 z = R[(16 + mc) * nk + kk];
    double2 np = double2{r.x - th.y, r.y + th.x};  // N+ = N_r + i N_theta
    double2 nm = double2{r.x + th.y, r.y - th.x};  // N- = N_r - i N_theta
    if (kk == K - 1 && m0 + mc == 0) z.x += 4.0 / Re;  // base driving force (laminar balance)
    const long o = ((long)(m0 + mc) * N + n) * nk + kk;
    if (d.forcing) {  // constant body force (shared by the trajectories of a group)
      const double2 a = d.forcing[o], b = d.forcing[fs + o], c = d.forcing[2 * fs + o];
      np.x += a.x;
      np.y += a.y;
      nm.x += b.x;
      nm.y += b.y;
      z.x += c.x;
      z.y += c.y;
    }
    Nout[o] = np;
    Nout[fs + o] = nm;
    Nout[2 * fs + o] = z;
  }
}

// ------------------------------------------------------------------ launches
bool dft_prepare_attrs() {
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return false;
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int lim = optin - 1024;  // (static shared memory counts too)
  return cudaFuncSetAttribute(k_dft_zsynth, a, lim) == cudaSuccess &&
         cudaFuncSetAttribute(k_dft_product<8, 3, 2>, a, lim) == cudaSuccess &&
         cudaFuncSetAttribute(k_dft_product<8, 6, 2>, a, lim) == cudaSuccess &&
         cudaFuncSetAttribute(k_dft_product<16, 6, 1>, a, lim) == cudaSuccess &&
         cudaFuncSetAttribute(k_dft_zanalysis<6, 3>, a, lim) == cudaSuccess &&
         cudaFuncSetAttribute(k_dft_zanalysis<8, 1>, a, lim) == cudaSuccess &&
         cudaFuncSetAttribute(k_dft_zanalysis<12, 1>, a, lim) == cudaSuccess;
}

void launch_dft_zsynth(const Dims& d, const DevSetup& s, const double2* W6, double2* Z6, cudaStream_t st) {
  const SynthShape sh = synth_shape(d);
  launch_step_kernel(d, k_dft_zsynth, dim3(sh.blocks, 1, d.B), dim3(kThreads), dft_zsynth_smem(d), st, d, sh.R,
                     s.dft.m[0], s.dft.m[1], (const double2*)s.tw_z, W6, Z6);
}
void launch_dft_product(const Dims& d, const DevSetup& s, const double2* Z6, double2* ZN, cudaStream_t st) {
  const dim3 g((d.nz + 15) / 16, d.N, d.B);
  auto go = [&](auto kern, int warps, int fields) {
    launch_step_kernel(d, kern, g, dim3(warps * 32), product_shape(d.M, d.nth, fields).smem, st, d, s.dft.m[2],
                       s.dft.m[3], s.dft.m[4], s.dft.m[5], (const double2*)s.tw_th, Z6, ZN);
  };
  if ((long)g.x * g.y * g.z <= device_sms()) go(k_dft_product<16, 6, 1>, 16, 6);
  else if (d.M <= 16) go(k_dft_product<8, 6, 2>, 8, 6);
  else go(k_dft_product<8, 3, 2>, 8, 3);
}
void launch_dft_zanalysis(const Dims& d, const DevSetup& s, const double2* ZN, double2* Nout, cudaStream_t st) {
  const dim3 g((d.M + 7) / 8, d.N, d.B);
  auto go = [&](auto kern, int warps) {
    launch_step_kernel(d, kern, g, dim3(warps * 32), dft_zanalysis_smem(d), st, d, s.dft.zshift, s.dft.m[6],
                       s.dft.m[7], (const double2*)s.tw_z, ZN, Nout);
  };
  if ((long)g.x * g.y * g.z > device_sms()) go(k_dft_zanalysis<6, 3>, 6);
  else if (3 * dft_tiles(dft_points(d.nz), 16) > 8) go(k_dft_zanalysis<12, 1>, 12);
  else go(k_dft_zanalysis<8, 1>, 8);
}

}  // namespace opf
