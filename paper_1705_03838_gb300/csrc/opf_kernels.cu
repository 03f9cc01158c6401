// Device kernels of the pipe-flow time step (paper section 2).
//
// Nonlinear term (section 2.2, evaluated pseudo-spectrally):
//   k_curl      spectral u+-, u_z -> (u_r, u_theta, u_z, w_r, w_theta, w_z)
//   k_zsynth    inverse FFT in z (2K-1 modes zero-padded to 3K points)
//   k_product   per (r, z) row: C2R in theta (M modes -> 3M points), u x w,
//               R2C in theta keeping m < M
//   k_zanalysis forward FFT in z keeping |k| < K, 1/(3K 3M) scaling,
//               (N_r, N_theta) -> N+-, base forcing 4/Re on the (0,0) mode
// Linear part (section 2.2, banded LU per Fourier mode; section 2 influence
// matrix): k_solve, one block per tile of T modes at fixed m.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdio>

#include "opf_dft.cuh"
#include "opf_fft.cuh"
#include "opf_internal.h"
#include "opf_step.cuh"

namespace opf {

__device__ __forceinline__ int row_lo_d(int i, int N) { return min(max(i - 4, 0), N - 9); }

// ------------------------------------------------------------------ ABI <-> internal
// abi: [3][M][nk][N] (u_r, u_theta, u_z); internal: [3][M][N][nk] (u+, u-, u_z).
// flag (optional): a non-zero value there (set by the NaN check launched
// before) leaves U as it is; beta (optional) is reset to 0 otherwise.
// nan_out (optional): set to 1 if any coefficient read is not finite (every
// coefficient is read by the thread of its own (m, k, n)).
// herm (optional, zeroed by the caller): herm[0], herm[1] become the upper 32
// bits of max |A(k,0) - conj A(-k,0)| and of max |A(k,0)| over the m = 0
// coefficients (real and imaginary parts separately, all three components):
// the upper word of a non-negative double orders like the double, and keeps
// it to 2^-20 relative.
__global__ void k_abi_to_internal(Dims d, const double2* __restrict__ abi, double2* __restrict__ U,
                                  const int* __restrict__ flag, double* __restrict__ beta, int* nan_out,
                                  unsigned* herm) {
  if (flag && *flag) return;
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (beta && idx == 0) *beta = 0.0;
  if (idx >= d.F) return;
  const int n = idx % d.N;
  const long t = idx / d.N;
  const int kk = t % d.nk;
  const int m = t / d.nk;
  const long fs = d.F;
  auto ld = [&](int c, int kq) { return abi[c * fs + ((long)m * d.nk + kq) * d.N + n]; };
  double2 ur = ld(0, kk), ut = ld(1, kk), uz = ld(2, kk);
  if (nan_out && !(isfinite(ur.x) && isfinite(ur.y) && isfinite(ut.x) && isfinite(ut.y) && isfinite(uz.x) &&
                   isfinite(uz.y)))
    atomicOr(nan_out, 1);
  if (m == 0) {  // Hermitian projection A(-k,0) = conj A(k,0)
    const int kq = d.nk - 1 - kk;
    const double2 vr = ld(0, kq), vt = ld(1, kq), vz = ld(2, kq);
    if (herm) {
      const double asym = fmax(fmax(fmax(fabs(ur.x - vr.x), fabs(ur.y + vr.y)),
                                    fmax(fabs(ut.x - vt.x), fabs(ut.y + vt.y))),
                               fmax(fabs(uz.x - vz.x), fabs(uz.y + vz.y)));
      const double amp = fmax(fmax(fmax(fabs(ur.x), fabs(ur.y)), fmax(fabs(ut.x), fabs(ut.y))),
                              fmax(fabs(uz.x), fabs(uz.y)));
      const unsigned lanes = __activemask();
      const unsigned ha = __reduce_max_sync(lanes, (unsigned)(__double_as_longlong(asym) >> 32));
      const unsigned hm = __reduce_max_sync(lanes, (unsigned)(__double_as_longlong(amp) >> 32));
      if ((int)(threadIdx.x & 31) == __ffs(lanes) - 1) {
        atomicMax(herm, ha);
        atomicMax(herm + 1, hm);
      }
    }
    ur = double2{0.5 * (ur.x + vr.x), 0.5 * (ur.y - vr.y)};
    ut = double2{0.5 * (ut.x + vt.x), 0.5 * (ut.y - vt.y)};
    uz = double2{0.5 * (uz.x + vz.x), 0.5 * (uz.y - vz.y)};
  }
  const long o = ((long)m * d.N + n) * d.nk + kk;
  U[0 * fs + o] = double2{ur.x - ut.y, ur.y + ut.x};  // u+ = u_r + i u_theta
  U[1 * fs + o] = double2{ur.x + ut.y, ur.y - ut.x};  // u- = u_r - i u_theta
  U[2 * fs + o] = uz;
}

__global__ void k_internal_to_abi(Dims d, const double2* __restrict__ U, double2* __restrict__ abi) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= d.F) return;
  const int n = idx % d.N;
  const long t = idx / d.N;
  const int kk = t % d.nk;
  const int m = t / d.nk;
  const long fs = d.F;
  const long i = ((long)m * d.N + n) * d.nk + kk;
  const double2 a = U[i], b = U[fs + i];
  const long o = ((long)m * d.nk + kk) * d.N + n;
  abi[o] = double2{0.5 * (a.x + b.x), 0.5 * (a.y + b.y)};           // u_r
  abi[fs + o] = double2{0.5 * (a.y - b.y), -0.5 * (a.x - b.x)};      // u_theta
  abi[2 * fs + o] = U[2 * fs + i];
}

void launch_abi_to_internal(const Dims& d, const double2* abi, double2* U, cudaStream_t st, const int* flag,
                            double* beta, int* nan_out, unsigned* herm) {
  const int nb = (int)((d.F + 255) / 256);
  k_abi_to_internal<<<nb, 256, 0, st>>>(d, abi, U, flag, beta, nan_out, herm);
}

// dst = src (n double2) unless *flag is set; beta reset to 0 with it
__global__ void k_copy_unless(const double2* __restrict__ src, double2* __restrict__ dst, long n,
                              const int* __restrict__ flag, double* __restrict__ beta) {
  if (*flag) return;
  const long i0 = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (beta && i0 == 0) *beta = 0.0;
  for (long i = i0; i < n; i += (long)gridDim.x * blockDim.x) dst[i] = src[i];
}

void launch_copy_unless(const double2* src, double2* dst, long n, const int* flag, double* beta,
                        cudaStream_t st) {
  const int nb = (int)std::min<long>((n + 255) / 256, 4L * 152);
  k_copy_unless<<<nb, 256, 0, st>>>(src, dst, n, flag, beta);
}
void launch_internal_to_abi(const Dims& d, const double2* U, double2* abi, int, cudaStream_t st) {
  const int nb = (int)((d.F + 255) / 256);
  k_internal_to_abi<<<nb, 256, 0, st>>>(d, U, abi);
}

// ------------------------------------------------------------------ curl (A1)
// One warp per item of eight modes (consecutive k at one m) and eight radial
// rows: a lane holds a mode's u+-, u_z at two of the rows and at two of the
// halo's, the radial derivatives of u_z and u_theta are digit products on the
// tensor cores (dft_stencil; multiply-adds where a column is steep), and
// everything else is pointwise in the lane.  Warps are independent; the rows of
// neighbouring items come from L1 again.
//
// SPLIT (mixed precision): the laminar base flow U = (1 - r^2) z,
// Omega = 2r theta is removed in FP64 (W6 then holds u', w' in FP32), and the
// terms linear in the perturbation, U x w' + u' x Omega (+ U x Omega on
// (0,0)), are evaluated here per mode in FP64 -- they are diagonal in r -- and
// written to Nlin in +- form.  FP64 arithmetic is kept to what Nlin needs
// (w_r, w_theta); w_z goes to the FP32 product only and is put together in
// FP32.  The factor 1/2 of u_r = (u+ + u-)/2 and u_theta = (u+ - u-)/(2i) goes
// into the constants that multiply them (exact scalings by two).
//
// What bounds it: the FP64 unit, with ~27 FP64 instructions per point left of
// 57 where the columns are not steep, then the integer units.  Against stencils
// as FP64 multiply-adds on columns staged in shared memory (whose loads of data
// and weights took about as long), split curl per launch: N = 128, 255 x 128
// modes 440 -> 267 us, groups of 8 x (N = 32 .. 48) and 6 x (N = 64, 63 x 32)
// 57 -> 44 us, N = 48, 63 x 24 modes, less than two waves of warps of which
// some take multiply-adds as well, 14.8 -> 15.9 us.
constexpr int kCurlWarps = 4;

// The (0,0) mode of the split curl: the base flow is taken off u_z and w_theta.
__device__ __noinline__ void curl_mean(double Ub, double Ob, double2 uz, double wtx, double wty, long fs, long w,
                                       float2* W6, double2* Nlin) {
  const double uzx = uz.x - Ub;
  wtx -= Ob;
  const double2 nr = double2{-Ub * wtx - Ob * uzx - Ub * Ob, -Ub * wty - Ob * uz.y};  // (w_r is zero)
  Nlin[w] = nr;
  Nlin[fs + w] = nr;
  W6[2 * fs + w].x = (float)uzx;
  W6[4 * fs + w].x = (float)wtx;
}
// Coriolis force of the base flow on (k, m~) = (0, 1): N- gains -2 U (Omega_y + i Omega_x).
__device__ __noinline__ void curl_rotation(double Ub, double rot_x, double rot_y, double2* nminus) {
  const double2 n = *nminus;
  *nminus = double2{n.x - 2.0 * Ub * rot_y, n.y - 2.0 * Ub * rot_x};
}

template <typename V, bool SPLIT>
__global__ void __launch_bounds__(kCurlWarps * 32, 4)
    k_curl(Dims d, StencilTable st, double ah, const double* __restrict__ rr, const double* __restrict__ rinv,
           const double2* __restrict__ U, V* __restrict__ W6, double2* __restrict__ Nlin) {
  const int N = d.N, nk = d.nk, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int G = (nk + 7) / 8;
  long item = (long)blockIdx.x * kCurlWarps + (threadIdx.x >> 5);
  grid_dep_trigger_at(d, 1);
  if (item >= (long)d.M * G * st.tiles) return;
  const int nt = (int)(item % st.tiles);
  item /= st.tiles;
  const int kk = (int)(item % G) * 8 + g, m = (int)(item / G);
  const bool in = kk < nk;
  st.tab = bofs(st.tab, d.ps);
  st.ew = bofs(st.ew, d.ps);
  st.d1 = bofs(st.d1, d.ps);
  rr = bofs(rr, d.ps);
  rinv = bofs(rinv, d.ps);
  U = bofs(U, d.ss);
  W6 = bofs(W6, d.ss);
  Nlin = bofs(Nlin, d.ss);
  const long fs = d.F;
  const int i0 = nt * 8 - st.off, mt = d.m_p * m, ps = mt & 1, pv = ps ^ 1;
  const long col = (long)m * N * nk + kk;
  grid_dep_wait();
  double2 uz[4], ut[4], ur[2];  // u_z; 2 u_theta; 2 u_r
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = stencil_row(i0, t, q);
    uz[q] = ut[q] = double2{0.0, 0.0};
    if (q < 2) ur[q] = uz[q];
    if (in && i >= 0 && i < N) {
      const double2 a = U[col + (long)i * nk], b = U[fs + col + (long)i * nk];
      uz[q] = U[2 * fs + col + (long)i * nk];
      ut[q] = double2{a.y - b.y, b.x - a.x};
      if (q < 2) ur[q] = double2{a.x + b.x, a.y + b.y};
    }
  }
  double2 dz[2];  // d/dr of u_z and u_theta
  V dt[2];
  {
    // multiply-adds read the columns from shared memory, a row of the window's
    // 16 every 18 parts (no bank conflicts); written when some column takes them
    __shared__ __align__(16) double window[kCurlWarps][16 * 18];
    double* wn = window[threadIdx.x >> 5];
    auto put = [&](const double2 (&x)[4]) {
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 4; ++q) *(double2*)(wn + (stencil_row(4, t, q) * 18 + 2 * g)) = x[q];
      __syncwarp();
    };
    auto at = [&](int i, int c, int part) { return wn[(i - i0 + 4) * 18 + 2 * c + part]; };
    dft_stencil<false, false>(uz, stencil_tile(st, ps, nt, nt, lane, 0), false, false, put, at, dz);
    const StencilAt pt = stencil_tile(st, pv, nt, nt, lane, -1);
    if constexpr (SPLIT) dft_stencil32(ut, pt, put, at, dt);
    else dft_stencil<false, false>(ut, pt, false, false, put, at, dt);
  }
  grid_dep_trigger_at(d, 2);
  if (!in) return;
  const double akh = ah * (kk - (d.K - 1));  // alpha k / 2
  const double mtd = mt;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int i = i0 + 2 * t + q;
    if (i < 0) continue;
    const double ri = rinv[i], mri = mtd * ri;
    // w_r = i (m~ u_z / r - ak u_theta)
    const double xr = fma(mri, uz[q].x, -akh * ut[q].x), xi = fma(mri, uz[q].y, -akh * ut[q].y);
    // w_theta = i ak u_r - d_r u_z
    const double wtx = fma(-akh, ur[q].y, -dz[q].x), wty = fma(akh, ur[q].x, -dz[q].y);
    const long w = col + (long)i * nk;
    if constexpr (SPLIT) {
      const double r = rr[i], Ub = fma(-r, r, 1.0), Ob = __hiloint2double(__double2hiint(r) + 0x100000, __double2loint(r));
      // N_r = -U w'_t - Omega u'_z, N_t = U w'_r, N_z = Omega u'_r
      const double nrx = fma(-Ub, wtx, -Ob * uz[q].x), nry = fma(-Ub, wty, -Ob * uz[q].y);
      // N- = N_r - i N_t, N+ = N_r + i N_t, N_t = U (-xi + i xr)
      Nlin[w] = double2{fma(-Ub, xr, nrx), fma(-Ub, xi, nry)};
      Nlin[fs + w] = double2{fma(Ub, xr, nrx), fma(Ub, xi, nry)};
      Nlin[2 * fs + w] = double2{r * ur[q].x, r * ur[q].y};  // Omega u_r = r (2 u_r)
      const double v[11] = {ur[q].x, ur[q].y, ut[q].x, ut[q].y, uz[q].x, uz[q].y, xi, xr, wtx, wty, ri};
      float f[11];
      bool rare = false;
#pragma unroll
      for (int u = 0; u < 11; ++u) f[u] = to_float(v[u], &rare);
      if (rare) {
#pragma unroll
        for (int u = 0; u < 11; ++u) f[u] = (float)v[u];
      }
      // w_z = d_r u_theta + u_theta / r - i m~ u_r / r, in FP32
      const float mri32 = (float)mt * f[10];
#pragma unroll
      for (int u = 0; u < 4; ++u) f[u] *= 0.5f;
      W6[0 * fs + w] = float2{f[0], f[1]};
      W6[1 * fs + w] = float2{f[2], f[3]};
      W6[2 * fs + w] = float2{f[4], f[5]};
      W6[3 * fs + w] = float2{-f[6], f[7]};
      W6[4 * fs + w] = float2{f[8], f[9]};
      W6[5 * fs + w] = float2{fmaf(mri32, f[1], fmaf(f[10], f[2], dt[q].x)),
                              fmaf(-mri32, f[0], fmaf(f[10], f[3], dt[q].y))};
      // the few modes with a term of their own, kept out of the others' way
      if (kk == d.K - 1) {
        if (m == 0) curl_mean(Ub, Ob, uz[q], wtx, wty, fs, w, (float2*)W6, Nlin);
        if (d.rotate && mt == 1) curl_rotation(Ub, d.rot_x, d.rot_y, Nlin + fs + w);
      }
    } else {
      const double2 u = double2{halved(ur[q].x), halved(ur[q].y)}, v = double2{halved(ut[q].x), halved(ut[q].y)};
      W6[0 * fs + w] = u;
      W6[1 * fs + w] = v;
      W6[2 * fs + w] = uz[q];
      W6[3 * fs + w] = V{-xi, xr};
      W6[4 * fs + w] = V{wtx, wty};
      W6[5 * fs + w] = V{fma(mri, u.y, fma(ri, v.x, dt[q].x)), fma(-mri, u.x, fma(ri, v.y, dt[q].y))};
    }
  }
}

template <typename V, bool SPLIT>
static void launch_curl_as(const Dims& d, const DevSetup& s, const double2* U, V* W6, double2* Nlin, cudaStream_t st) {
  const StencilTable tab = stencil_at(s.stab, s.d1, d.N);
  const long items = (long)d.M * ((d.nk + 7) / 8) * tab.tiles;
  launch_step_kernel(d, k_curl<V, SPLIT>, dim3((unsigned)((items + kCurlWarps - 1) / kCurlWarps), 1, d.B),
                     dim3(kCurlWarps * 32), 0, st, d, tab, 0.5 * d.alpha, (const double*)s.r, (const double*)s.rinv, U, W6, Nlin);
}

void launch_curl(const Dims& d, const DevSetup& s, const double2* U, double2* W6, cudaStream_t st) {
  launch_curl_as<double2, false>(d, s, U, W6, nullptr, st);
}

void launch_curl_split32(const Dims& d, const DevSetup& s, const double2* U, float2* W6, double2* Nlin,
                         cudaStream_t st) {
  launch_curl_as<float2, true>(d, s, U, W6, Nlin, st);
}

// Threads per block of the transform kernels: 256 for grids of at most four
// blocks per SM (a single wave of few blocks: more threads per batch of
// sequences shorten each block's passes), 128 for larger grids, which
// measured as fast or faster in the smaller unit.  The arithmetic is the
// same either way.
static unsigned transform_threads(const dim3& g) {
  return (long)g.x * g.y * g.z <= 4L * device_sms() ? 256u : 128u;
}

// The FP32 kernels that stream (a compiled plan) do with fewer, at every
// length: their composite butterflies take up to 164 registers a thread, and
// what counts is how many small blocks reside.  z synthesis and product: 96
// threads, us per launch against 64, 128 and 192 (z synthesis | product): N =
// 128, 384 x 384 points 113, 121, 123, 172 | 354, 360, 415, 536; 4 x (N = 64, 192 x
// 192) 58, 62, 60, 70 | 153, 143, 157, 228; 16 x (N = 48, 96 x 96) 47, 45, 50, 64 |
// 96, 100, 105, 127; 16 x (N = 48, 72 x 72) 32, 31, 35, 44 | 62, 66, 70, 86; 64 x
// (N = 32, 48 x 48) 36, 32, 41, 49 | 72, 81, 80, 106; a single N = 48, 96 x 72
// 8.2 | 12.1, the others up to 0.1 and 1.1 more.
constexpr unsigned kStreamThreads = 96;
// z analysis, whose block takes three components and reads the addends: a
// thread for nine of its points, at least 128, at most 192.  Those grids at 128
// and 192: 226, 178; 101, 90; 80, 70; 47, 45; 49, 57 (8 columns of 48 points,
// 1152); 11.2, 11.2 us.
static unsigned zanalysis_threads(int nz, int mca) {
  return (unsigned)std::min(192, std::max(128, mca * nz / 3 / 32 * 32));
}

// ------------------------------------------------------------------ z synthesis (A2)

// NZ > 0: the z length 3K is the compile-time constant NZ (compiled plan).
// FP32 with a compiled plan: both passes work between registers, global memory
// and one exchange through shared memory, whose pipe was 88 % busy with the
// staging and every pass; half the footprint lets twice the blocks reside.
// 197 -> 114 us at N = 128, 255 x 128 modes (500 MB, 75 us at the copy rate),
// groups of 8 x (N = 32 .. 48) and 6 x (N = 64, 63 x 32) 28.7 -> 18.1 us.
template <typename V, int NZ>
__global__ void __launch_bounds__(256) k_zsynth(Dims d, FftPlan pz, const V* __restrict__ twz,
                                                const V* __restrict__ W6, V* __restrict__ Z6) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nz = NZ > 0 ? NZ : d.nz, ld = nz + 1, MC = d.mcz;
  constexpr bool kStream = NZ > 0 && sizeof(V) == sizeof(float2);
  V* A = (V*)smraw;
  V* B = A + MC * ld;
  V* tw = kStream ? B : B + MC * ld;
  const int m0 = blockIdx.x * MC, n = blockIdx.y / 6, f = blockIdx.y % 6;
  const int K = d.K;
  twz = bofs(twz, d.ps);
  W6 = bofs(W6, d.ss);
  Z6 = bofs(Z6, d.ss);
  grid_dep_trigger_at(d, 1);
  for (int e = threadIdx.x; e < nz; e += blockDim.x) tw[e] = twz[e];
  const long fs = d.F;
  grid_dep_wait();
  if constexpr (kStream) {  // global to registers, one exchange through shared memory, and back
    constexpr FftRadices r = fft_radices32(NZ > 0 ? NZ : 48);
    const int mcn = min(MC, d.M - m0);
    for (int w = threadIdx.x; w < mcn * (NZ / r.r1); w += blockDim.x) {
      const int mc = w / (NZ / r.r1), j = w - mc * (NZ / r.r1);
      const V* src = W6 + f * fs + ((long)(m0 + mc) * d.N + n) * d.nk + K - 1;
      fft_first<r.r1, NZ, +1, true>(j, A + mc * ld, [&](int z) {
        return z < K ? src[z] : z > NZ - K ? src[z - NZ] : V{0, 0};
      });
    }
    __syncthreads();
    grid_dep_trigger_at(d, 2);
    V* out = Z6 + ((long)f * d.N + n) * NZ * d.M + m0;
    for (int w = threadIdx.x; w < mcn * (NZ / r.r2); w += blockDim.x) {
      const int j = w / mcn, mc = w - j * mcn;
      V v[r.r2];
      fft_last<r.r2, NZ, +1>(j, A + mc * ld, tw, v);
#pragma unroll
      for (int q = 0; q < r.r2; ++q) out[(long)(j + q * (NZ / r.r2)) * d.M + mc] = v[q];
    }
    return;
  }
  block_copy_batched<8, V>(
      MC * nz,
      [&](int e) {
        const int z = e % nz, m = m0 + e / nz;
        const int k = z < K ? z : z - nz;
        V v = V{0, 0};
        if (m < d.M && (z < K || z > nz - K)) v = W6[f * fs + ((long)m * d.N + n) * d.nk + k + K - 1];
        return v;
      },
      [&](int e, V v) { A[(e / nz) * ld + e % nz] = v; });
  __syncthreads();
  const V* res;
  if constexpr (NZ > 0) res = block_fft_c<NZ, +1, true>(A, B, MC, ld, tw);
  else res = block_fft(A, B, MC, ld, pz, tw, +1);
  const int mcn = min(MC, d.M - m0);
  grid_dep_trigger_at(d, 2);
  for (int e = threadIdx.x; e < mcn * nz; e += blockDim.x) {
    const int mc = e % mcn, z = e / mcn;
    Z6[(((long)f * d.N + n) * nz + z) * d.M + m0 + mc] = res[mc * ld + z];
  }
}

size_t zsynth_smem(const Dims& d, int mc, size_t vb) { return (2 * (size_t)mc * (d.nz + 1) + d.nz) * vb; }

void launch_zsynth32(const Dims& d, const DevSetup& s, const FftPlan& pz, const float2* W6,
                     float2* Z6, cudaStream_t st) {
  dim3 g((d.M + d.mcz - 1) / d.mcz, d.N * 6, d.B);
  with_fft_length(d.nz, [&](auto n) {
    const size_t sm = decltype(n)::value ? (size_t)(d.mcz * (d.nz + 1) + d.nz) * sizeof(float2)
                                         : zsynth_smem(d, d.mcz, sizeof(float2));
    launch_step_kernel(d, k_zsynth<float2, decltype(n)::value>, g,
                       dim3(decltype(n)::value ? kStreamThreads : transform_threads(g)), sm, st, d, pz,
                       (const float2*)s.tw_z32, W6, Z6);
  });
}

void launch_zsynth(const Dims& d, const DevSetup& s, const FftPlan& pz, const double2* W6,
                   double2* Z6, cudaStream_t st) {
  if (s.dft.m[0]) return launch_dft_zsynth(d, s, W6, Z6, st);
  dim3 g((d.M + d.mcz - 1) / d.mcz, d.N * 6, d.B);
  const size_t sm = zsynth_smem(d, d.mcz, sizeof(double2));
  with_long_fft_length(d.nz, [&](auto n) {
    launch_step_kernel(d, k_zsynth<double2, decltype(n)::value>, g, dim3(transform_threads(g)), sm, st, d, pz,
                       (const double2*)s.tw_z, W6, Z6);
  });
}

// ------------------------------------------------------------------ product (A3)

__device__ __forceinline__ void sincos_pi(double x, double* s, double* c) { sincospi(x, s, c); }
__device__ __forceinline__ void sincos_pi(float x, float* s, float* c) { sincospif(x, s, c); }

// NTH > 0: the theta length 3M is the compile-time constant NTH.
// FP32 with a compiled plan (kStream): three exchanges through shared memory
// instead of five passes with staging either side -- global memory to the first
// pass of the syntheses; their last pass, the product and the first pass of the
// analyses on the same points in registers; the last pass to global memory.
// What bounds it: barriers between the phases and instruction fetch, at 12 warps
// per SM (length 384).  N = 128,
// 255 x 128 modes 467 -> 362 us; groups of 8 x (N = 32 .. 48) and 6 x (N = 64,
// 63 x 32) 44.6 -> 34.3 us; N = 48, 63 x 24 modes 13.2 -> 12.1 us.
template <typename V, int NTH>
__global__ void __launch_bounds__(256) k_product(Dims d, FftPlan pth, const V* __restrict__ twth,
                                                 const V* __restrict__ Z6, V* __restrict__ ZN) {
  using T = typename Scalar<V>::T;
  // FP64: the real N_z of two z rows go through one complex forward
  // transform (1.5 instead of 2 transforms per row on the FP64 pipe); the
  // FP32 path keeps one per row, the arithmetic of the fused launch
  constexpr bool kPackNz = sizeof(T) == 8;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nth = NTH > 0 ? NTH : d.nth, ld = nth, M = d.M;
  const int ZC = d.zc;
  constexpr bool kStream = NTH > 0 && sizeof(V) == sizeof(float2);
  V* A = (V*)smraw;            // 3 * ZC sequences
  V* B = A + 3 * ZC * ld;      // 3 * ZC sequences (kStream: none)
  V* tw = kStream ? B : B + 3 * ZC * ld;
  const int z0 = blockIdx.x * ZC, n = blockIdx.y, nz = d.nz;
  const int zc = min(ZC, nz - z0);
  twth = bofs(twth, d.ps);
  Z6 = bofs(Z6, d.ss);
  ZN = bofs(ZN, d.ss);
  grid_dep_trigger_at(d, 1);
  for (int e = threadIdx.x; e < nth; e += blockDim.x) tw[e] = twth[e];
  const long fstride = (long)d.N * nz * M;
  grid_dep_wait();
  // spectra of the pairs (u_r,u_t), (u_z,w_r), (w_t,w_z):  Z = A + i B
  auto spectrum = [&](int zr, int pr, int q) {
    const long rowa = ((long)(2 * pr) * d.N + n) * nz + z0 + zr;
    const bool low = q < M;
    const int m = low ? q : nth - q;
    V a = V{0, 0}, b = V{0, 0};
    if (low || q > nth - M) {
      a = Z6[rowa * M + m];
      b = Z6[(rowa + (long)d.N * nz) * M + m];
    }
    if (q == 0) a.y = b.y = 0;
    return low ? V{a.x - b.y, a.y + b.x} : V{a.x + b.y, b.x - a.y};  // (mirrored: conj(a) + i conj(b))
  };
  V* res = nullptr;
  constexpr FftRadices rx = fft_radices32(NTH > 0 ? NTH : 48);
  if constexpr (kStream) {
    for (int w = threadIdx.x; w < 3 * zc * (NTH / rx.r1); w += blockDim.x) {
      const int bt = w / (NTH / rx.r1), j = w - bt * (NTH / rx.r1), zr = bt / 3, pr = bt - 3 * zr;
      fft_first<rx.r1, NTH, +1, true>(j, A + bt * ld, [&](int q) { return spectrum(zr, pr, q); });
    }
    __syncthreads();
  } else {
    block_copy_batched<8, V>(
        zc * 3 * nth, [&](int e) { return spectrum(e / (3 * nth), (e / nth) % 3, e % nth); },
        [&](int e, V v) { A[(e / nth) * ld + e % nth] = v; });
    __syncthreads();
    if constexpr (NTH > 0) res = block_fft_c<NTH, +1, true>(A, B, 3 * zc, ld, tw);
    else res = block_fft(A, B, 3 * zc, ld, pth, tw, +1);
  }
  V* C = (res == A) ? B : A;
  // CFL number of this radial plane (optional): max over the grid of
  // |u_r|/dr, |u_t|/(r dtheta), |u_z|/dz for the TOTAL velocity (the FP32
  // path carries the perturbation only, so the laminar 1 - r^2 is added back)
  // (taken in the transform precision T)
  double* cfl = bofs(d.cfl, d.ss);
  T inv_dr = 0, inv_rdt = 0, inv_dz = 0, Ubase = 0;
  if (cfl) {
    const double* rinv = bofs(d.rinv_cfl, d.ps);
    const T one = 1, rn = one / (T)rinv[n];
    const T rm = n > 0 ? one / (T)rinv[n - 1] : -rn;
    const T rp = n < d.N - 1 ? one / (T)rinv[n + 1] : one + (one - rm);
    const T twopi = (T)6.283185307179586;
    inv_dr = one / fmin(rn - rm, rp - rn);
    inv_rdt = (T)(d.m_p * nth) / (twopi * rn);
    inv_dz = (T)d.alpha * (T)nz / twopi;
    if constexpr (sizeof(T) == 4) Ubase = one - rn * rn;
  }
  T cmax = 0;
  // u x w (with the Coriolis term) at point q from the three pairs
  auto product = [&](int q, V x0, V x1, V x2, V* nrt, T* nzp) {
    const T ur = x0.x, ut = x0.y, uz = x1.x, wr = x1.y, wt = x2.x, wz = x2.y;
    T nr = madd(ut, wz, -(uz * wt)), nt = madd(uz, wr, -(ur * wz)), nz = madd(ur, wt, -(ut * wr));
    if (d.rotate) {  // Coriolis -2 Omega x u, Omega in cylindrical components at theta_q
      T sn, cs;
      sincos_pi((T)(2 * q) / (T)(d.m_p * nth), &sn, &cs);
      const T rx = (T)d.rot_x, ry = (T)d.rot_y;
      const T o_r = madd(rx, cs, ry * sn), o_t = madd(ry, cs, -(rx * sn));
      const T o_z = (T)d.rot_z;
      nr = madd((T)-2, madd(o_t, uz, -(o_z * ut)), nr);
      nt = madd((T)-2, madd(o_z, ur, -(o_r * uz)), nt);
      nz = madd((T)-2, madd(o_r, ut, -(o_t * ur)), nz);
    }
    if (cfl) cmax = fmax(cmax, fmax(fabs(ur) * inv_dr, fmax(fabs(ut) * inv_rdt, fabs(uz + Ubase) * inv_dz)));
    *nrt = V{nr, nt};
    *nzp = nz;
  };
  if constexpr (kStream) {
    // one item per thread (product32_items, which the launch gives threads for
    // at every zc; a loop over rounds of rows took 0.55 ms longer per step at
    // N = 128, 255 x 128 modes): the last pass of the three syntheses, the
    // product, and the first pass of the two analyses, which takes the same
    // points; written back in place once all have read
    constexpr int L = NTH / rx.r2;
    const int zr = threadIdx.x / L, j = threadIdx.x - zr * L;
    const bool have = zr < zc;
    V x0[rx.r2], x1[rx.r2];
    // (a zero the compiler cannot fold, which would let it round otherwise than
    // the fused launch)
    T zero = 0;
    asm("" : "+f"(zero));
    if (have) {
      V x2[rx.r2];
      fft_last<rx.r2, NTH, +1>(j, A + (zr * 3 + 0) * ld, tw, x0);
      fft_last<rx.r2, NTH, +1>(j, A + (zr * 3 + 1) * ld, tw, x1);
      fft_last<rx.r2, NTH, +1>(j, A + (zr * 3 + 2) * ld, tw, x2);
#pragma unroll
      for (int q = 0; q < rx.r2; ++q) {
        V nrt;
        T nzv;
        product(j + q * L, x0[q], x1[q], x2[q], &nrt, &nzv);
        x0[q] = nrt;
        x1[q] = V{nzv, zero};
      }
      butterfly<rx.r2>(x0, -1);
      butterfly<rx.r2>(x1, -1);
    }
    __syncthreads();
    if (have) {
#pragma unroll
      for (int q = 0; q < rx.r2; ++q) {
        A[zr * ld + fft_swz(j * rx.r2 + q)] = x0[q];
        A[(zc + zr) * ld + fft_swz(j * rx.r2 + q)] = x1[q];
      }
    }
  } else
  for (int e = threadIdx.x; e < zc * nth; e += blockDim.x) {
    const int q = e % nth, zr = e / nth;
    V nrt;
    T nz;
    product(q, res[(zr * 3 + 0) * ld + q], res[(zr * 3 + 1) * ld + q], res[(zr * 3 + 2) * ld + q], &nrt, &nz);
    if constexpr (kPackNz) {  // rows zr, zr^1 share one sequence for N_z: re <- even row, im <- odd row
      C[zr * ld + q] = nrt;
      T* pz = (T*)&C[(zc + (zr >> 1)) * ld + q];
      pz[zr & 1] = nz;
      if ((zc & 1) && zr == zc - 1) pz[1] = (T)0;  // the last row of an odd count has no partner
    } else {
      C[(zr * 2 + 0) * ld + q] = nrt;
      C[(zr * 2 + 1) * ld + q] = V{nz, (T)0};
    }
  }
  if (cfl) {  // warp max, then one atomic per warp (non-negative doubles order as integers)
    for (int o = 16; o > 0; o >>= 1) cmax = fmax(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    const double cm = (double)cmax;
    if ((threadIdx.x & 31) == 0 && cm > 0.0)
      atomicMax((unsigned long long*)cfl, (unsigned long long)__double_as_longlong(cm));
  }
  __syncthreads();
  if constexpr (kStream) {
    // the last pass of the analyses: N_z goes out, N_r + i N_theta through the
    // third of A that the products left free
    constexpr int L = NTH / rx.r1;
    V* Y = A + 2 * zc * ld;
    for (int w = threadIdx.x; w < 2 * zc * L; w += blockDim.x) {
      const int bt = w / L, j = w - bt * L;
      V v[rx.r1];
      fft_last<rx.r1, NTH, -1>(j, A + bt * ld, tw, v);
      if (bt < zc) {
#pragma unroll
        for (int q = 0; q < rx.r1; ++q) Y[bt * ld + j + q * L] = v[q];
      } else {
        V* out = ZN + 2 * fstride + ((long)n * nz + z0 + bt - zc) * M;
#pragma unroll
        for (int q = 0; q < rx.r1; ++q)
          if (j + q * L < M) out[j + q * L] = v[q];
      }
    }
    __syncthreads();
    grid_dep_trigger_at(d, 2);
    for (int e = threadIdx.x; e < zc * M; e += blockDim.x) {
      const int m = e % M, zr = e / M;
      const V y = Y[zr * ld + m], yc = Y[zr * ld + (m == 0 ? 0 : nth - m)];
      const long row = ((long)n * nz + z0 + zr) * M + m;
      ZN[row] = V{(T)0.5 * (y.x + yc.x), (T)0.5 * (y.y - yc.y)};
      ZN[fstride + row] = V{(T)0.5 * (y.y + yc.y), (T)-0.5 * (y.x - yc.x)};
    }
    return;
  }
  V* D = (C == A) ? B : A;
  const V* out;
  const int nfwd = kPackNz ? zc + (zc + 1) / 2 : 2 * zc;
  if constexpr (NTH > 0) out = block_fft_c<NTH, -1>(C, D, nfwd, ld, tw);
  else out = block_fft(C, D, nfwd, ld, pth, tw, -1);
  grid_dep_trigger_at(d, 2);
  for (int e = threadIdx.x; e < zc * M; e += blockDim.x) {
    const int m = e % M, zr = e / M, mc = m == 0 ? 0 : nth - m;
    const int rp = kPackNz ? zr : zr * 2;  // the (N_r + i N_theta) sequence of row zr
    const V y = out[rp * ld + m];
    const V yc = out[rp * ld + mc];
    const V nr = V{(T)0.5 * (y.x + yc.x), (T)0.5 * (y.y - yc.y)};
    const V nt = V{(T)0.5 * (y.y + yc.y), (T)-0.5 * (y.x - yc.x)};
    const long row = ((long)n * nz + z0 + zr) * M + m;
    ZN[row] = nr;
    ZN[fstride + row] = nt;
    if constexpr (kPackNz) {  // Z = F(a) + i F(b): F(a) = (Z + conj Z(-m)) / 2, F(b) = (Z - conj Z(-m)) / 2i
      const V w = out[(zc + (zr >> 1)) * ld + m], wc = out[(zc + (zr >> 1)) * ld + mc];
      ZN[2 * fstride + row] = (zr & 1) ? V{(T)0.5 * (w.y + wc.y), (T)-0.5 * (w.x - wc.x)}
                                       : V{(T)0.5 * (w.x + wc.x), (T)0.5 * (w.y - wc.y)};
    } else {
      ZN[2 * fstride + row] = out[(zr * 2 + 1) * ld + m];
    }
  }
}

size_t product_smem(const Dims& d, int zc, size_t vb) { return (2 * 3 * (size_t)zc * d.nth + d.nth) * vb; }

// The streamed FP32 product's middle phase has one item per thread, this many
// of them with zc rows per block (0: the length has no compiled plan).
static int product32_items(const Dims& d, int zc) {
  return fft_length_compiled(d.nth) ? zc * (d.nth / fft_radices32(d.nth).r2) : 0;
}
// Whether a block may take zc rows: its shared memory, and a thread per item.
bool product_fits(const Dims& d, int zc, size_t vb, size_t smem) {
  return product_smem(d, zc, vb) <= smem && (vb != sizeof(float2) || product32_items(d, zc) <= 256);
}

void launch_product32(const Dims& d, const DevSetup& s, const FftPlan& pth, const float2* Z6,
                      float2* ZN, cudaStream_t st) {
  dim3 g((d.nz + d.zc - 1) / d.zc, d.N, d.B);
  with_fft_length(d.nth, [&](auto n) {
    const size_t sm = decltype(n)::value ? (size_t)(3 * d.zc + 1) * d.nth * sizeof(float2)
                                         : product_smem(d, d.zc, sizeof(float2));
    const unsigned items = ((unsigned)product32_items(d, d.zc) + 31) / 32 * 32;
    launch_step_kernel(d, k_product<float2, decltype(n)::value>, g,
                       dim3(decltype(n)::value ? std::max(items, kStreamThreads) : transform_threads(g)), sm, st, d, pth,
                       (const float2*)s.tw_th32, Z6, ZN);
  });
}

void launch_product(const Dims& d, const DevSetup& s, const FftPlan& pth, const double2* Z6,
                    double2* ZN, cudaStream_t st) {
  if (s.dft.m[2]) return launch_dft_product(d, s, Z6, ZN, st);
  dim3 g((d.nz + d.zc - 1) / d.zc, d.N, d.B);
  const size_t sm = product_smem(d, d.zc, sizeof(double2));
  with_long_fft_length(d.nth, [&](auto n) {
    launch_step_kernel(d, k_product<double2, decltype(n)::value>, g, dim3(transform_threads(g)), sm, st, d, pth,
                       (const double2*)s.tw_th, Z6, ZN);
  });
}

// ------------------------------------------------------------------ z analysis (A4)
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(float x) { return to_double(x); }

// FP32 with a compiled plan: the first pass reads global memory itself.  N = 128,
// 255 x 128 modes 256 -> 179 us (with the threads of its launch rule),
// groups of 8 x (N = 32 .. 48) and 6 x (N = 64, 63 x 32) 40.3 -> 29.2 us, N = 48,
// 63 x 24 modes 12.3 -> 11.3 us.
template <typename V, int NZ>
__global__ void __launch_bounds__(256) k_zanalysis(Dims d, FftPlan pz, const V* __restrict__ twz,
                                                   const V* __restrict__ ZN, const double2* __restrict__ Nlin,
                                                   double2* __restrict__ Nout) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nz = NZ > 0 ? NZ : d.nz, ld = nz + 1, M = d.M, K = d.K, nk = d.nk;
  const int MC = d.mca;
  V* A = (V*)smraw;
  V* B = A + 3 * MC * ld;
  V* tw = B + 3 * MC * ld;
  const int m0 = blockIdx.x * MC, n = blockIdx.y;
  const int mcn = min(MC, M - m0);
  twz = bofs(twz, d.ps);
  ZN = bofs(ZN, d.ss);
  Nlin = bofs(Nlin, d.ss);
  Nout = bofs(Nout, d.ss);
  const double Re = bofs(d.prm, d.ps)[kPrmRe];
  grid_dep_trigger_at(d, 1);
  for (int e = threadIdx.x; e < nz; e += blockDim.x) tw[e] = twz[e];
  const long fs = d.F;
  grid_dep_wait();
  // FP64 addends of an output point (linear terms, body force); a thread's
  // first point has them loaded before the transform, so that their latency
  // overlaps it
  auto addends = [&](long o, double2* ap, double2* am, double2* az) {
    *ap = *am = *az = double2{0.0, 0.0};
    if (d.forcing) {  // constant body force (shared by the trajectories of a group)
      *ap = d.forcing[o];
      *am = d.forcing[fs + o];
      *az = d.forcing[2 * fs + o];
    }
    if (Nlin) {  // terms linear in the perturbation, evaluated in FP64
      const double2 a = Nlin[o], b = Nlin[fs + o], c = Nlin[2 * fs + o];
      *ap = double2{ap->x + a.x, ap->y + a.y};
      *am = double2{am->x + b.x, am->y + b.y};
      *az = double2{az->x + c.x, az->y + c.y};
    }
  };
  auto out_index = [&](int e) {
    const int kk = e % nk, mc = e / nk;
    return ((long)(m0 + mc) * d.N + n) * nk + kk;
  };
  double2 pp, pm, pz0;
  const bool have0 = threadIdx.x < mcn * nk;
  if (have0 && (Nlin || d.forcing)) addends(out_index(threadIdx.x), &pp, &pm, &pz0);
  const long fstride = (long)d.N * nz * M;
  const V* res;
  if constexpr (NZ > 0 && sizeof(V) == sizeof(float2)) {  // the first pass from global memory
    constexpr FftRadices r = fft_radices32(NZ > 0 ? NZ : 48);
    for (int w = threadIdx.x; w < 3 * MC * (NZ / r.r2); w += blockDim.x) {
      const int mc = w % MC, j = w / MC % (NZ / r.r2), f = w / (MC * (NZ / r.r2));
      const V* src = ZN + f * fstride + (long)n * NZ * M + m0 + mc;
      fft_first<r.r2, NZ, -1, false>(j, A + (f * MC + mc) * ld,
                                     [&](int z) { return mc < mcn ? src[(long)z * M] : V{0, 0}; });
    }
    __syncthreads();
    for (int w = threadIdx.x; w < 3 * MC * (NZ / r.r1); w += blockDim.x) {
      const int bt = w / (NZ / r.r1), j = w - bt * (NZ / r.r1);
      V v[r.r1];
      fft_last<r.r1, NZ, -1>(j, A + bt * ld, tw, v);
#pragma unroll
      for (int q = 0; q < r.r1; ++q) B[bt * ld + j + q * (NZ / r.r1)] = v[q];
    }
    __syncthreads();
    res = B;
  } else {
    block_copy_batched<8, V>(
        3 * MC * nz,
        [&](int e) {
          const int mc = e % MC, z = (e / MC) % nz, f = e / (MC * nz);
          V v = V{0, 0};
          if (mc < mcn) v = ZN[f * fstride + ((long)n * nz + z) * M + m0 + mc];
          return v;
        },
        [&](int e, V v) {
          const int mc = e % MC, z = (e / MC) % nz, f = e / (MC * nz);
          A[(f * MC + mc) * ld + z] = v;
        });
    __syncthreads();
    if constexpr (NZ > 0) res = block_fft_c<NZ, -1>(A, B, 3 * MC, ld, tw);
    else res = block_fft(A, B, 3 * MC, ld, pz, tw, -1);
  }
  // scaling and the +- combination in the transform's precision, then FP64
  using T = typename Scalar<V>::T;
  const T sc = (T)d.inv_grid;
  grid_dep_trigger_at(d, 2);
  for (int e = threadIdx.x; e < mcn * nk; e += blockDim.x) {
    const int kk = e % nk, mc = e / nk, m = m0 + mc;
    const int k = kk - (K - 1);
    const int zp = k < 0 ? k + nz : k;
    const V r_ = res[(0 * MC + mc) * ld + zp], t_ = res[(1 * MC + mc) * ld + zp];
    const V z_ = res[(2 * MC + mc) * ld + zp];
    double2 np = double2{wide(sc * (r_.x - t_.y)), wide(sc * (r_.y + t_.x))};  // N+ = N_r + i N_theta
    double2 nm = double2{wide(sc * (r_.x + t_.y)), wide(sc * (r_.y - t_.x))};  // N- = N_r - i N_theta
    double2 nz2 = double2{wide(sc * z_.x), wide(sc * z_.y)};
    if (k == 0 && m == 0) nz2.x += 4.0 / Re;  // base driving force (laminar balance)
    const long o = ((long)m * d.N + n) * nk + kk;
    if (Nlin || d.forcing) {
      double2 ap, am, az;
      if (e == (int)threadIdx.x) {
        ap = pp;
        am = pm;
        az = pz0;
      } else {
        addends(o, &ap, &am, &az);
      }
      np.x += ap.x;
      np.y += ap.y;
      nm.x += am.x;
      nm.y += am.y;
      nz2.x += az.x;
      nz2.y += az.y;
    }
    Nout[o] = np;
    Nout[fs + o] = nm;
    Nout[2 * fs + o] = nz2;
  }
}

size_t zanalysis_smem(const Dims& d, int mc, size_t vb) {
  return (2 * 3 * (size_t)mc * (d.nz + 1) + d.nz) * vb;
}

void launch_zanalysis(const Dims& d, const DevSetup& s, const FftPlan& pz, const double2* ZN,
                      double2* Nout, cudaStream_t st) {
  if (s.dft.m[6]) return launch_dft_zanalysis(d, s, ZN, Nout, st);
  dim3 g((d.M + d.mca - 1) / d.mca, d.N, d.B);
  const size_t sm = zanalysis_smem(d, d.mca, sizeof(double2));
  with_long_fft_length(d.nz, [&](auto n) {
    launch_step_kernel(d, k_zanalysis<double2, decltype(n)::value>, g, dim3(transform_threads(g)), sm, st, d, pz,
                       (const double2*)s.tw_z, ZN, (const double2*)nullptr, Nout);
  });
}

void launch_zanalysis32(const Dims& d, const DevSetup& s, const FftPlan& pz, const float2* ZN,
                        const double2* Nlin, double2* Nout, cudaStream_t st) {
  dim3 g((d.M + d.mca - 1) / d.mca, d.N, d.B);
  const size_t sm = zanalysis_smem(d, d.mca, sizeof(float2));
  with_fft_length(d.nz, [&](auto n) {
    launch_step_kernel(d, k_zanalysis<float2, decltype(n)::value>, g,
                       dim3(decltype(n)::value ? zanalysis_threads(d.nz, d.mca) : transform_threads(g)), sm, st, d, pz,
                       (const float2*)s.tw_z32, ZN, Nlin, Nout);
  });
}

// ------------------------------------------------------------------ fused FP32 transforms (A2-A4)
// The mixed-precision nonlinear term after the curl, in one launch: a cluster
// of C blocks per (radial plane n, trajectory b) keeps the plane's
// half-physical fields in distributed shared memory instead of round trips
// through L2 between three kernels.
//   phase 1  block r takes m columns [r MC, (r+1) MC) of all six fields:
//            inverse z transforms (the z synthesis kernel's arithmetic);
//   phase 2  block r takes z rows [r ZR, (r+1) ZR): gathers those rows of
//            every m column from the blocks that own them, inverse theta
//            transforms, u x w (with the Coriolis term and the CFL maximum),
//            forward theta transforms (the product kernel's arithmetic);
//   phase 3  block r takes its m columns again: gathers them over all z rows,
//            forward z transforms, truncation, scaling, +- form and the FP64
//            addends (the z analysis kernel's arithmetic).
// Each transform runs the same block FFT on the same sequences as the
// three-kernel path, so the results are identical to it.
namespace cg = cooperative_groups;

__host__ __device__ inline int fused_mc(int M, int C) { return (M + C - 1) / C; }
__host__ __device__ inline int fused_zr(int nz, int C) { return (nz + C - 1) / C; }

size_t fused32_smem(const Dims& d, int C) {
  const int MC = fused_mc(d.M, C), ZR = fused_zr(d.nz, C);
  return (2 * 6 * (size_t)MC * (d.nz + 1) + 3 * (size_t)ZR * d.M + d.nz + d.nth) * sizeof(float2);
}

template <int NZ, int NTH>
__global__ void __launch_bounds__(256) k_nl_fused32(Dims d, int C, const float2* __restrict__ twz,
                                                    const float2* __restrict__ twth,
                                                    const float2* __restrict__ W6,
                                                    const double2* __restrict__ Nlin,
                                                    double2* __restrict__ Nout) {
  using V = float2;
  using T = float;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int LDZ = NZ + 1;
  const int M = d.M, K = d.K, nk = d.nk, N = d.N;
  const int MC = fused_mc(M, C), ZR = fused_zr(NZ, C);
  const int rank = (int)cl.block_rank();
  const int n = blockIdx.x / C;
  V* A = (V*)smraw;            // [6 MC][LDZ]  phase 1 (then phase 3)
  V* B = A + 6 * MC * LDZ;     // [6 MC][LDZ]  phase 1 ping-pong (then phase 2)
  V* ZNl = B + 6 * MC * LDZ;   // [3][ZR][M]   product spectra of this block's z rows
  V* tz = ZNl + 3 * ZR * M;    // [NZ]
  V* tth = tz + NZ;            // [NTH]
  twz = bofs(twz, d.ps);
  twth = bofs(twth, d.ps);
  W6 = bofs(W6, d.ss);
  Nlin = bofs(Nlin, d.ss);
  Nout = bofs(Nout, d.ss);
  const double Re = bofs(d.prm, d.ps)[kPrmRe];
  for (int e = threadIdx.x; e < NZ; e += blockDim.x) tz[e] = twz[e];
  for (int e = threadIdx.x; e < NTH; e += blockDim.x) tth[e] = twth[e];
  const long fs = d.F;
  const int m0 = rank * MC;
  const int mcn = max(0, min(MC, M - m0));

  // ---- phase 1: inverse z transforms of this block's m columns, six fields
  for (int e = threadIdx.x; e < 6 * MC * NZ; e += blockDim.x) {
    const int z = e % NZ, col = e / NZ, f = col / MC, mc = col % MC;
    const int k = z < K ? z : z - NZ;
    V v = V{0, 0};
    if (mc < mcn && (z < K || z > NZ - K)) v = W6[f * fs + ((long)(m0 + mc) * N + n) * nk + k + K - 1];
    A[col * LDZ + z] = v;
  }
  __syncthreads();
  V* res1 = block_fft_c<NZ, +1, true>(A, B, 6 * MC, LDZ, tz);
  V* free1 = (res1 == A) ? B : A;
  cl.sync();  // every block's half-physical columns are in place

  // ---- phase 2: this block's z rows: theta transforms and the product
  const int z0 = rank * ZR;
  const int zrn = max(0, min(ZR, NZ - z0));
  const int ZC = max(1, min(max(zrn, 1), (6 * MC * LDZ) / (6 * NTH)));
  V* P0 = free1;               // [3 ZC][NTH]
  V* P1 = free1 + 3 * ZC * NTH;  // [3 ZC][NTH]
  double* cfl = bofs(d.cfl, d.ss);
  T inv_dr = 0, inv_rdt = 0, inv_dz = 0, Ubase = 0;
  if (cfl) {
    const double* rinv = bofs(d.rinv_cfl, d.ps);
    const T one = 1, rn = one / (T)rinv[n];
    const T rm = n > 0 ? one / (T)rinv[n - 1] : -rn;
    const T rp = n < N - 1 ? one / (T)rinv[n + 1] : one + (one - rm);
    const T twopi = (T)6.283185307179586;
    inv_dr = one / fmin(rn - rm, rp - rn);
    inv_rdt = (T)(d.m_p * NTH) / (twopi * rn);
    inv_dz = (T)d.alpha * (T)NZ / twopi;
    Ubase = one - rn * rn;
  }
  T cmax = 0;
  for (int c0 = 0; c0 < zrn; c0 += ZC) {
    const int zc = min(ZC, zrn - c0);
    // spectra of the pairs (u_r,u_t), (u_z,w_r), (w_t,w_z):  Z = A + i B
    for (int e = threadIdx.x; e < zc * 3 * NTH; e += blockDim.x) {
      const int q = e % NTH, pr = (e / NTH) % 3, zr = e / (3 * NTH);
      const int z = z0 + c0 + zr;
      V v = V{0, 0};
      const int mq = q < M ? q : (q > NTH - M ? NTH - q : -1);
      if (mq >= 0) {
        const V* src = cl.map_shared_rank(res1, mq / MC);
        V a = src[((2 * pr) * MC + mq % MC) * LDZ + z], b = src[((2 * pr + 1) * MC + mq % MC) * LDZ + z];
        if (q < M) {
          if (q == 0) {
            a.y = 0;
            b.y = 0;
          }
          v = V{a.x - b.y, a.y + b.x};
        } else {
          v = V{a.x + b.y, -a.y + b.x};  // conj(a) + i conj(b)
        }
      }
      P0[(zr * 3 + pr) * NTH + q] = v;
    }
    __syncthreads();
    V* res = block_fft_c<NTH, +1, true>(P0, P1, 3 * zc, NTH, tth);
    V* Cb = (res == P0) ? P1 : P0;
    for (int e = threadIdx.x; e < zc * NTH; e += blockDim.x) {
      const int q = e % NTH, zr = e / NTH;
      const V x0 = res[(zr * 3 + 0) * NTH + q], x1 = res[(zr * 3 + 1) * NTH + q], x2 = res[(zr * 3 + 2) * NTH + q];
      const T ur = x0.x, ut = x0.y, uz = x1.x, wr = x1.y, wt = x2.x, wz = x2.y;
      T nr = madd(ut, wz, -(uz * wt)), nt = madd(uz, wr, -(ur * wz)), nz = madd(ur, wt, -(ut * wr));
      if (d.rotate) {  // Coriolis -2 Omega x u, Omega in cylindrical components at theta_q
        T sn, cs;
        sincos_pi((T)(2 * q) / (T)(d.m_p * NTH), &sn, &cs);
        const T rx = (T)d.rot_x, ry = (T)d.rot_y;
        const T o_r = madd(rx, cs, ry * sn), o_t = madd(ry, cs, -(rx * sn));
        const T o_z = (T)d.rot_z;
        nr = madd((T)-2, madd(o_t, uz, -(o_z * ut)), nr);
        nt = madd((T)-2, madd(o_z, ur, -(o_r * uz)), nt);
        nz = madd((T)-2, madd(o_r, ut, -(o_t * ur)), nz);
      }
      Cb[(zr * 2 + 0) * NTH + q] = V{nr, nt};
      Cb[(zr * 2 + 1) * NTH + q] = V{nz, (T)0};
      if (cfl) cmax = fmax(cmax, fmax(fabs(ur) * inv_dr, fmax(fabs(ut) * inv_rdt, fabs(uz + Ubase) * inv_dz)));
    }
    __syncthreads();
    V* Db = (Cb == P0) ? P1 : P0;
    const V* out = block_fft_c<NTH, -1>(Cb, Db, 2 * zc, NTH, tth);
    for (int e = threadIdx.x; e < zc * M; e += blockDim.x) {
      const int m = e % M, zr = e / M;
      const V y = out[(zr * 2 + 0) * NTH + m];
      const V yc = out[(zr * 2 + 0) * NTH + (m == 0 ? 0 : NTH - m)];
      const int row = c0 + zr;
      ZNl[(0 * ZR + row) * M + m] = V{(T)0.5 * (y.x + yc.x), (T)0.5 * (y.y - yc.y)};
      ZNl[(1 * ZR + row) * M + m] = V{(T)0.5 * (y.y + yc.y), (T)-0.5 * (y.x - yc.x)};
      ZNl[(2 * ZR + row) * M + m] = out[(zr * 2 + 1) * NTH + m];
    }
    __syncthreads();  // P0 / P1 are reused by the next chunk of rows
  }
  if (cfl) {  // warp max, then one atomic per warp (non-negative doubles order as integers)
    for (int o = 16; o > 0; o >>= 1) cmax = fmax(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    const double cm = (double)cmax;
    if ((threadIdx.x & 31) == 0 && cm > 0.0)
      atomicMax((unsigned long long*)cfl, (unsigned long long)__double_as_longlong(cm));
  }
  cl.sync();  // every block's product spectra are in place; nobody reads res1 any more

  // ---- phase 3: forward z transforms of this block's m columns, three fields
  V* A3 = A;
  V* B3 = A + 3 * MC * LDZ;
  for (int e = threadIdx.x; e < 3 * MC * NZ; e += blockDim.x) {
    const int z = e % NZ, col = e / NZ, f = col / MC, mc = col % MC;
    V v = V{0, 0};
    if (mc < mcn) {
      const V* src = cl.map_shared_rank(ZNl, z / ZR);
      v = src[(f * ZR + z % ZR) * M + m0 + mc];
    }
    A3[col * LDZ + z] = v;
  }
  cl.sync();  // every remote read is done before any block moves on or exits
  const V* res3 = block_fft_c<NZ, -1>(A3, B3, 3 * MC, LDZ, tz);
  const T sc = (T)d.inv_grid;
  for (int e = threadIdx.x; e < mcn * nk; e += blockDim.x) {
    const int kk = e % nk, mc = e / nk, m = m0 + mc;
    const int k = kk - (K - 1);
    const int zp = k < 0 ? k + NZ : k;
    const V r_ = res3[(0 * MC + mc) * LDZ + zp], t_ = res3[(1 * MC + mc) * LDZ + zp];
    const V z_ = res3[(2 * MC + mc) * LDZ + zp];
    double2 np = double2{wide(sc * (r_.x - t_.y)), wide(sc * (r_.y + t_.x))};  // N+ = N_r + i N_theta
    double2 nm = double2{wide(sc * (r_.x + t_.y)), wide(sc * (r_.y - t_.x))};  // N- = N_r - i N_theta
    double2 nz2 = double2{wide(sc * z_.x), wide(sc * z_.y)};
    if (k == 0 && m == 0) nz2.x += 4.0 / Re;  // base driving force (laminar balance)
    const long o = ((long)m * N + n) * nk + kk;
    double2 ap = double2{0.0, 0.0}, am = ap, az = ap;
    if (d.forcing) {  // constant body force (shared by the trajectories of a group)
      ap = d.forcing[o];
      am = d.forcing[fs + o];
      az = d.forcing[2 * fs + o];
    }
    if (Nlin) {  // terms linear in the perturbation, evaluated in FP64
      const double2 a = Nlin[o], b = Nlin[fs + o], c = Nlin[2 * fs + o];
      ap = double2{ap.x + a.x, ap.y + a.y};
      am = double2{am.x + b.x, am.y + b.y};
      az = double2{az.x + c.x, az.y + c.y};
    }
    if (Nlin || d.forcing) {
      np.x += ap.x;
      np.y += ap.y;
      nm.x += am.x;
      nm.y += am.y;
      nz2.x += az.x;
      nz2.y += az.y;
    }
    Nout[o] = np;
    Nout[fs + o] = nm;
    Nout[2 * fs + o] = nz2;
  }
}

// Cluster size for a fused launch of this shape (0: the shape takes the
// three-kernel path): transform lengths with a compiled plan up to 96;
// d.fused = 2, 4 or 8 forces the cluster size, 1 chooses it (eight blocks
// per plane when the grid would otherwise leave SMs idle, else four).
int fused32_cluster(const Dims& d) {
  auto ok = [](int n) { return n == 48 || n == 72 || n == 96; };
  if (!d.fused || !ok(d.nz) || !ok(d.nth)) return 0;
  int dev = 0, sms = 152, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int C = d.fused >= 2 ? d.fused : ((long)4 * d.N * d.B < 2L * sms ? 8 : 4);
  if (fused32_smem(d, C) > (size_t)optin) return 0;
  if ((long)fused_mc(d.M, C) * (d.nz + 1) < d.nth) return 0;  // phase 2 needs one row's buffers
  return C;
}

template <int NZ, int NTH>
void launch_fused_len(const Dims& d, const DevSetup& s, int C, const float2* W6, const double2* Nlin,
                      double2* Nout, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(C * d.N, 1, d.B);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = fused32_smem(d, C);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_nl_fused32<NZ, NTH>, d, C, (const float2*)s.tw_z32, (const float2*)s.tw_th32, W6,
                     Nlin, Nout);
}

template <class F>
void with_fused_lengths(int nz, int nth, F&& f) {
  auto inner = [&](auto z) {
    switch (nth) {
      case 48: f(z, std::integral_constant<int, 48>{}); break;
      case 72: f(z, std::integral_constant<int, 72>{}); break;
      default: f(z, std::integral_constant<int, 96>{}); break;
    }
  };
  switch (nz) {
    case 48: inner(std::integral_constant<int, 48>{}); break;
    case 72: inner(std::integral_constant<int, 72>{}); break;
    default: inner(std::integral_constant<int, 96>{}); break;
  }
}

bool launch_nl_fused32(const Dims& d, const DevSetup& s, const float2* W6, const double2* Nlin, double2* Nout,
                       cudaStream_t st) {
  const int C = fused32_cluster(d);
  if (!C) return false;
  with_fused_lengths(d.nz, d.nth, [&](auto z, auto t) {
    launch_fused_len<decltype(z)::value, decltype(t)::value>(d, s, C, W6, Nlin, Nout, st);
  });
  return true;
}

// ------------------------------------------------------------------ linear solve (A5-A7)
struct SolveDev {
  const double* d1;
  const double* rinv;
  const double* wq;
  const int* hop;
  const double* luH;
  const double* luP;
  const double* basis;
  const double2* ainv;
  const double* G;
  const double* prm;
  StencilTable st;  // digit table of the stencils
  int nJ;
  int stage;  // u_j and the influence responses staged in shared memory
  // split solve: both blocks' factors, spikes, interface inverses
  const double* luH2;
  const double* luP2;
  const double* spkH;
  const double* spkP;
  const double* rH;
  const double* rP;
};

// Bulk L2 prefetch by the TMA unit: p 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void prefetch_l2_bulk(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Asynchronous global -> shared copies (8 or 16 bytes, both addresses aligned
// to the size); completion by commit groups, visibility by a block barrier.
__device__ __forceinline__ void cp_async8(void* sm, const void* g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(sm)), "l"(g)
               : "memory");
}
__device__ __forceinline__ void cp_async16(void* sm, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(sm)), "l"(g)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int G>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(G) : "memory"); }

// Shared memory of a solve block: the working arrays, then (when they fit in
// ~100 KB, i.e. for moderate N) u_j and the influence responses of the tile,
// staged by asynchronous copies at the start so that the right-hand sides,
// the influence step and the write-out read them from shared memory.
// The host stages only where that costs no resident blocks (see
// launch_solve); the launch gives the staged size then, the base size else.
// sp: the split solve's interface values (6T chains x 8 doubles) after misc.
// Where the stencils are digit products only the wall divergence's weights are
// kept here.
constexpr int kSolveDigitRows = 64;
__host__ __device__ constexpr bool solve_by_digits(int N, bool sp) { return !sp && N >= kSolveDigitRows; }
__host__ __device__ constexpr int solve_weights(int N, bool sp) { return solve_by_digits(N, sp) ? 10 : 2 * N * 9; }
__host__ __device__ constexpr size_t solve_smem_base(int N, int T, bool sp = false) {
  return (size_t)(2 * N * T + T) * 16 + (size_t)6 * N * T * 8 +
         (size_t)(solve_weights(N, sp) + 3 * N + 2) * 8 + 16 + (sp ? (size_t)48 * T * 8 : 0);
}
__host__ __device__ constexpr size_t solve_smem_staged(int N, int T, bool sp = false) {
  return solve_smem_base(N, T, sp) + (size_t)48 * N * T + (size_t)8 * basis_ld(N) * T;
}
__host__ __device__ constexpr bool solve_stage_fits(int N, int T) { return solve_smem_staged(N, T) <= 100 * 1024; }

// Banded substitution on one real right-hand side held in shared memory at
// x[i * st], i < N, by a group of 4 consecutive lanes: rows are dealt round
// robin to the lanes, each lane keeps the partial sum of the one row it owns
// among the four behind the current column, and once row c is final its owner
// broadcasts it and every lane subtracts its row's multiple of it (the owner
// from the next row it takes up).  The factor is stored by columns (13 N
// values, see to_columns on the host): [N][4] L(c+1+t, c), [N][4] L(c+5+t, c),
// [N] 1/U_ii, [N][4] U(c-1-t, c) / U_ii, zeros outside the band, so the four
// lanes of a chain read one 32-byte run per column.  The columns are walked in
// blocks of four counted so that the nine wall columns start a block: owners
// and queue slots are then compile-time constants, a lane takes up its next
// row and stores its finished one once per block, and the chain per row is
// one broadcast and one FMA (a form that shifted the partial sums along the
// lanes took eight shuffles per row; the same sums in the same order).  What
// bounds it is that chain, ~110 cycles per row, on grids of a wave, and the
// FP64 unit (one FMA per row and eight right-hand sides) on larger ones.
// Per solve launch, shifting against this form: N=48 63 x 24 modes 59.3 ->
// 47.1 us, N=128 255 x 128 modes 2.30 -> 1.83 ms, N=32 64 x 31 x 16 modes
// 596 -> 535 us.  Factor entries are loaded kAhead columns ahead into
// registers, which keeps the L2 latency off the recursion.
// All 32 lanes of the warp must call this together (8 right-hand sides per
// warp).
__device__ __forceinline__ void band_solve4(const double* __restrict__ L, double* x, int st, int N) {
  const int t = threadIdx.x & 3;
  const unsigned full = 0xffffffffu;
  constexpr int kAhead = 16;
  const double* Lw = L + 4 * N;  // L(c+5+t, c)
  const double* Dg = L + 8 * N;  // 1/U_ii
  const double* Uc = L + 9 * N;  // U(c-1-t, c) / U_(c-1-t)
  double q[kAhead], qd[kAhead / 4];
  // forward: y = L^{-1} b, stored as y_i / U_ii (the U rows are scaled by
  // 1/U_ii, so the backward sweep has one FMA per row).  Columns v0 < 0 of the
  // first round do not exist and are skipped.
  {
    const int nw = N - 9;                                    // first wall column
    const int v0 = nw - (nw + kAhead - 1) / kAhead * kAhead;  // <= 0
    auto l_of = [&](int c, int j) { return c >= 0 && c < N ? __ldg(L + c * 4 + ((t - j - 1) & 3)) : 0.0; };
    auto d_of = [&](int i) { return i >= 0 && i < N ? __ldg(Dg + i) : 0.0; };
#pragma unroll
    for (int j = 0; j < kAhead; ++j) q[j] = l_of(v0 + j, j & 3);
#pragma unroll
    for (int b = 0; b < kAhead / 4; ++b) qd[b] = d_of(v0 + 4 * b + t);
    double s = x[((t + v0) & 3) * st];
    // the last four rows, whose lower band reaches eight: lane t's one of them,
    // and its entries in the wall columns more than four to the left
    const int rw = t ? N - 5 + t : N - 1;
    double w = x[rw * st], qw[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = rw - (nw + i) - 5;
      qw[i] = o >= 0 ? __ldg(Lw + (nw + i) * 4 + o) : 0.0;
    }
    for (int c0 = v0; c0 < nw; c0 += kAhead) {
#pragma unroll
      for (int b = 0; b < kAhead / 4; ++b) {
        const int cb = c0 + 4 * b;  // warp-uniform
        if (cb > -4) {
          const double next = cb + t >= 0 ? x[(cb + 4 + t) * st] : 0.0;
          double own = 0.0;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (cb + j >= 0) {
              const double y = __shfl_sync(full, s, j, 4);
              if (t == j) {
                own = s;
                s = next;
              }
              s = fma(-q[4 * b + j], y, s);
            }
          }
          if (cb + t >= 0) x[(cb + t) * st] = own * qd[b];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) q[4 * b + j] = l_of(cb + kAhead + j, j);
        qd[b] = d_of(cb + kAhead + t);
      }
    }
    const double next = t == 0 ? x[(N - 5) * st] : 0.0;
    double own = 0.0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const double y = __shfl_sync(full, s, i & 3, 4);
      if (t == (i & 3)) {
        own = s;
        s = i == 0 ? next : w;
      }
      s = fma(-q[i], y, s);
      if (i < 4) w = fma(-qw[i], y, w);
      if ((i & 3) == 3) x[(nw + (i & ~3) + t) * st] = own * qd[i >> 2];
    }
    if (t == 0) x[(N - 1) * st] = own * qd[2];
  }
  __syncwarp();
  // backward: x = U~^{-1} (y / diag U), counted from the wall
  {
    auto u_of = [&](int c, int j) { return c >= 0 ? __ldg(Uc + c * 4 + ((t - j - 1) & 3)) : 0.0; };
#pragma unroll
    for (int j = 0; j < kAhead; ++j) q[j] = u_of(N - 1 - j, j & 3);
    double s = x[(N - 1 - t) * st];
    for (int c0 = N - 1; c0 >= 0; c0 -= kAhead) {
#pragma unroll
      for (int b = 0; b < kAhead / 4; ++b) {
        const int cb = c0 - 4 * b;  // warp-uniform
        if (cb >= 0) {
          const double next = cb - 4 - t >= 0 ? x[(cb - 4 - t) * st] : 0.0;
          double own = 0.0;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const double y = __shfl_sync(full, s, j, 4);
            if (t == j) {
              own = s;
              s = next;
            }
            s = fma(-q[4 * b + j], y, s);
          }
          if (cb - t >= 0) x[(cb - t) * st] = own;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) q[4 * b + j] = u_of(cb - kAhead - j, j);
      }
    }
  }
}

// One block: T consecutive k at fixed m (24T threads).  Row-parallel phases
// use all threads over (chain, row); only the banded substitutions are
// sequential in r, with 4 lanes per real right-hand side (2T pressure chains,
// then 6T velocity chains = (u+, u-, u_z) x T modes x (re, im)).  While warp
// 0 solves the pressure system the other warps assemble the p-independent part
// of the velocity right-hand sides (and stage u_j and the influence
// responses); the last pass applies u_j, the influence correction and the
// flux correction on the way out to global memory, and with a.W6 the block
// then takes the curl of its new state for the next nonlinear evaluation.
//
// The radial derivatives (of N+ + N- and of p) are digit products on the tensor
// cores (dft_stencil), a warp per eight modes and rows, from N = 64 on; on
// coarser meshes, whose windows reach from the axis or the wall and of whose columns
// many are steep, and in the split solve (a block per SM), FP64 multiply-adds with
// the weights in shared memory are the faster.
// What bounds it: the chains of the substitutions and, on large grids, the
// FP64 unit, which the stencils took 36 of ~90 instructions per point of.  Per
// launch, multiply-adds against digits: N = 128, 255 x 128 modes 1734, 1558 us;
// 8 x (63 x 32 modes) at N = 96 660, 521 us, 80 486, 452, 64 385, 372, 48 300,
// 298 us; 63 x 24 modes at N = 96 82.8, 78.4 us, 64 55.2, 58.3, 56 50.1, 54.2; 64
// x (N = 32, 31 x 16) 410, 422 us; N = 41, 53 x 20 modes 35.7, 39 us; N = 20, 7 x
// 5 modes, which takes the curl as well (by digits either way, in one copy of
// the code, stencil_call, 2 us faster than one per use), 28.4, 30.5 us.
//
// Resident blocks per SM the register budget must allow (the shared-memory
// footprints of the tiles allow about as many at moderate N).
template <int T, bool SP>
constexpr int solve_min_blocks() {
  return SP ? 3 : (T == 4 ? 4 : (T == 8 ? 3 : 2));
}

// Interface and correction of the split solve for nch chains held in x
// (chain c's column at x + col(c), rows at stride st) after both halves were
// substituted: z = R (y_T[k-4:k], y_B[0:4]) per chain, then every row
// x_i -= S_i . z_B (top half) or S_i . z_T (bottom half), k = N/2.  spk: per
// operator N rows of 4; R: per operator 8 x 8.  Ends with a block barrier.
template <int NB, typename OpOf>
__device__ __forceinline__ void spike_fix(int tid, int N, int nch, int st, double* x, const double* __restrict__ spk,
                                          const double* __restrict__ R, double* Zs, OpOf op_of) {
  const int kh = N >> 1;
  for (int e = tid; e < nch * 8; e += NB) {
    const int c = e >> 3, q = e & 7;
    const double* Rc = R + (long)op_of(c) * 64 + q * 8;
    const double* xc = x + c;
    double z = 0.0;
#pragma unroll
    for (int b = 0; b < 4; ++b) z = fma(Rc[b], xc[(kh - 4 + b) * st], z);
#pragma unroll
    for (int b = 0; b < 4; ++b) z = fma(Rc[4 + b], xc[(kh + b) * st], z);
    Zs[e] = z;
  }
  __syncthreads();
  for (int e = tid; e < nch * N; e += NB) {
    const int c = e % nch, i = e / nch;
    const double* S = spk + ((long)op_of(c) * N + i) * 4;
    const double* z = Zs + c * 8 + (i < kh ? 4 : 0);
    double v = x[i * st + c];
#pragma unroll
    for (int q = 0; q < 4; ++q) v = fma(-S[q], z[q], v);
    x[i * st + c] = v;
  }
  __syncthreads();
}

// SP: the split (two-partition) solve for the latency-bound grids -- each
// chain's substitution runs on 8 lanes, the two halves of its rows at once
// (twice the threads; the other phases use them too).
// CURL: may take the curl of its new state (a.W6).
// DIG: the stencils by digit products (solve_by_digits).
template <int T, bool DIG, bool SP = false, bool CURL = SP>
__global__ void __launch_bounds__((SP ? 48 : 24) * T, solve_min_blocks<T, SP>())
    k_solve(Dims d, SolveDev s, SolveArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int N = d.N, nk = d.nk, M = d.M, K = d.K;
  constexpr int NT = 6 * T;                // velocity right-hand sides (chains)
  constexpr int NB = (SP ? 48 : 24) * T;   // threads: 4 (SP: 8) lanes per velocity chain
  constexpr int NP = (SP ? 16 : 8) * T;    // threads of the pressure substitution (2T chains)
  // X holds N_eff first (chain layout: field f, mode mi, re/im part), then
  // the velocity right-hand sides built on it in place, then the chains'
  // solutions; S is reused by the influence step.
  double2* S = (double2*)smraw;                // [N][T]     N+ + N- (later u_j near the wall)
  double2* P = S + N * T;                      // [N][T]     pressure (later u_theta)
  double2* coef = P + N * T;                   // [T]        influence coefficients
  double* X = (double*)(coef + T);             // [N][6T]    N_eff -> right-hand sides -> velocity chains
  double* W1 = X + N * NT;                     // [2][N][9]  first-derivative stencils (digits: the wall's row)
  double* RI = W1 + solve_weights(N, SP);      // [N]        1/r
  double* RIp = RI + N;                        // [N]        (1 + m~) / (2r)
  double* RIm = RIp + N;                       // [N]        (1 - m~) / (2r)
  double* misc = RIm + N;                      // [2]        flux correction
  const bool stage = s.stage;
  // u_j near the wall for the influence step, when not staged: in S (free
  // after the pressure right-hand side) if it holds [T][16], else from global
  double2* UW = S;
  const bool uw_in_s = !stage && N >= 16;
  double* Zs = misc + 2;                       // [6T][8]    split-solve interface values (SP)
  double2* UJ = (double2*)(((size_t)(Zs + (SP ? 48 * T : 0)) + 15) & ~(size_t)15);  // [3][N][T] u_j (stage)
  double* BS = (double*)(UJ + 3 * N * T);                             // [T][basis_ld] responses (stage)
  // N_eff of field f, row i, mode mi as a complex pair in X's chain layout
  auto ne_at = [&](int f, int i, int mi) -> double2& {
    return *(double2*)(X + (long)i * NT + ((f * T + mi) << 1));
  };
  const int m = blockIdx.y, kk0 = blockIdx.x * T, tid = threadIdx.x;
  const int mt = d.m_p * m, ps = mt & 1, pv = ps ^ 1;
  s.d1 = bofs(s.d1, d.ps);
  s.rinv = bofs(s.rinv, d.ps);
  s.wq = bofs(s.wq, d.ps);
  s.hop = bofs(s.hop, d.ps);
  s.luH = bofs(s.luH, d.ps);
  s.luP = bofs(s.luP, d.ps);
  s.basis = bofs(s.basis, d.ps);
  s.ainv = bofs(s.ainv, d.ps);
  s.G = bofs(s.G, d.ps);
  s.prm = bofs(s.prm, d.ps);
  s.st.tab = bofs(s.st.tab, d.ps);
  s.st.ew = bofs(s.st.ew, d.ps);
  s.st.d1 = s.d1;
  if constexpr (SP) {
    s.luH2 = bofs(s.luH2, d.ps);
    s.luP2 = bofs(s.luP2, d.ps);
    s.spkH = bofs(s.spkH, d.ps);
    s.spkP = bofs(s.spkP, d.ps);
    s.rH = bofs(s.rH, d.ps);
    s.rP = bofs(s.rP, d.ps);
  }
  a.Uj = bofs(a.Uj, d.ss);
  a.Na = bofs(a.Na, d.ss);
  a.Nb = bofs(a.Nb, d.ss);
  a.Uout = bofs(a.Uout, d.ss);
  a.beta_p = bofs(a.beta_p, d.ss);
  const double ci = s.prm[kPrmCi], cu = s.prm[kPrmCu];  // 1 / (c dt), (1 - c) / c
  const long fs = d.F;
  const long base = (long)m * N * nk;
  const double* wv = W1 + pv * N * 9;  // stencils of u_r, u_theta parity
  const double* ws = W1 + ps * N * 9;  // stencils of u_z, p parity
  const double* wall = DIG ? W1 : wv + (N - 1) * 9;  // wall row of wv
  // chain c -> (field f, mode mi, part); element (f, row i, mode mi) of a field
  auto uj = [&](int f, int i, int mi) {
    return a.Uj[f * fs + base + (long)i * nk + min(kk0 + mi, nk - 1)];
  };

  grid_dep_trigger_at(d, 1);
  // Pull this block's factor blocks (pressure, u+, u-, u_z per mode) and
  // basis blocks towards L2 with one bulk prefetch each, so they arrive while
  // the right-hand sides are assembled.  Factor blocks start on 16 bytes only
  // for even N (104 N bytes per operator); basis blocks always do.
  if (tid < 5 * T) {
    const int mi = tid % T, which = tid / T;
    const int ik = abs(min(kk0 + mi, nk - 1) - (K - 1));
    if (which == 4) {
      if (!stage) prefetch_l2_bulk(s.basis + (long)(ik * M + m) * basis_ld(N), 8u * basis_ld(N));
    } else if (!(N & 1)) {
      const long op = which == 0 ? ((ik == 0 && m == 0) ? K * M : ik * M + m) : ik * s.nJ + s.hop[3 * m + which - 1];
      prefetch_l2_bulk((which == 0 ? (SP ? s.luP2 : s.luP) : (SP ? s.luH2 : s.luH)) + op * N * kLuSlots,
                       (unsigned)N * kLuSlots * 8u);
    }
  }

  // The stencils by asynchronous copies, waited for at the first barrier.
  if constexpr (DIG) {
    if (tid < 9) cp_async8(W1 + tid, s.d1 + ((long)pv * N + N - 1) * 9 + tid);
  } else {
    for (int e = tid; e < 2 * N * 9; e += NB) cp_async8(W1 + e, s.d1 + e);
  }
  if (CURL && !SP && a.W6)  // a block per SM: the digit tables to the SM's cache while it waits for its input
    for (int e = tid; e < 2 * s.st.tiles * (kTileB / 16); e += NB)
      asm volatile("{\n.reg .b32 t;\nld.global.ca.b32 t, [%0];\n}" ::"l"(s.st.tab + 16 * e));
  cp_async_commit();

  // ---- N_eff = N_a (predictor) or (N_a + N_b) / 2 (corrector, c = 1/2), and
  //      N+ + N- for the divergence
  for (int e = tid; e < N; e += NB) {
    const double ri = s.rinv[e];
    RI[e] = ri;
    RIp[e] = 0.5 * (1 + mt) * ri;
    RIm[e] = 0.5 * (1 - mt) * ri;
  }
  grid_dep_wait();  // everything above read setup data only
#pragma unroll 4
  for (int e = tid; e < 3 * N * T; e += NB) {
    const int mi = e % T, i = (e / T) % N, f = e / (T * N);
    const long g = f * fs + base + (long)i * nk + min(kk0 + mi, nk - 1);
    double2 v = a.Na[g];
    if (a.Nb) {
      const double2 w = a.Nb[g];
      v = double2{halved(v.x + w.x), halved(v.y + w.y)};
    }
    ne_at(f, i, mi) = v;
  }
  cp_async_wait<0>();
  __syncthreads();
  for (int e = tid; e < N * T; e += NB) {
    const int mi = e % T, i = e / T;
    const double2 p = ne_at(0, i, mi), q = ne_at(1, i, mi);
    S[e] = double2{p.x + q.x, p.y + q.y};
  }
  __syncthreads();

  // Row-parallel phases over (mode, row) give each thread one fixed mode
  // mi_t = tid % T and the rows tid / T, tid / T + NB / T, ...
  const int mi_t = tid % T;
  const double ak_t = d.alpha * (min(kk0 + mi_t, nk - 1) - (K - 1));

  // The derivative (times 2^shift) of a field at(row, mode) of one parity at every
  // row and mode, out(row, mode, alpha k, derivative): a warp per eight modes and
  // eight rows, or per four modes and two such tiles (one if there are warps
  // enough).
  auto for_stencil_items = [&](auto at, int parity, int shift, auto out) {
    const int lane = tid & 31, g = lane >> 2, t = lane & 3;
    constexpr int kGroups = T >= 8 ? T / 8 : 1;  // of modes
    const int tiles = s.st.tiles, per = T >= 8 || tiles <= NB / 32 ? 1 : 2;  // tiles per item
    for (int it = tid >> 5; it < (tiles + per - 1) / per * kGroups; it += NB / 32) {
      __syncwarp();
      const int first = it / kGroups * per, nt = T >= 8 || g < 4 ? first : per == 2 ? first + 1 : tiles;
      const int mi = T >= 8 ? it % kGroups * 8 + g : g & 3, i0 = nt * 8 - s.st.off;
      double2 x[4];
      double2 d9[2];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = stencil_row(i0, t, q);
        x[q] = nt < tiles && i >= 0 && i < N ? at(i, mi) : double2{0.0, 0.0};
      }
      const StencilAt w = stencil_tile(s.st, parity, first, nt, lane, shift);
      dft_stencil<(T < 8), CURL>(x, w, per == 2 && first + 1 < tiles, g >= 4, [](const double2 (&)[4]) {}, [&](int i, int c, int part) {
        const double2 v = at(i, T >= 8 ? mi - g + c : c & 3);
        return part ? v.y : v.x;
      }, d9);
      const double ak = d.alpha * (min(kk0 + mi, nk - 1) - (K - 1));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i = i0 + 2 * t + q;
        if (i >= 0 && i < N) out(i, mi, ak, d9[q]);
      }
    }
  };

  // ---- pressure right-hand side: div N_eff (rows < N-1), 0 at the wall
  if constexpr (DIG) {
    for_stencil_items([&](int i, int mi) { return S[i * T + mi]; }, pv, -1, [&](int i, int mi, double ak, double2 dr) {  // dr: half the derivative
      const double2 np = ne_at(0, i, mi), nm = ne_at(1, i, mi), nz = ne_at(2, i, mi);
      const double bx = dr.x + fma(RIp[i], np.x, fma(RIm[i], nm.x, -ak * nz.y));
      const double by = dr.y + fma(RIp[i], np.y, fma(RIm[i], nm.y, ak * nz.x));
      P[i * T + mi] = i < N - 1 ? double2{bx, by} : double2{0.0, 0.0};
    });
  } else
  for (int i = tid / T; i < N; i += NB / T) {
    double2 b = double2{0.0, 0.0};
    if (i < N - 1) {
      const int lo = row_lo_d(i, N);
      double ax = 0.0, ay = 0.0;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const double2 sv = S[(lo + q) * T + mi_t];
        const double w = wv[i * 9 + q];
        ax = fma(w, sv.x, ax);
        ay = fma(w, sv.y, ay);
      }
      const double2 np = ne_at(0, i, mi_t), nm = ne_at(1, i, mi_t), nz = ne_at(2, i, mi_t);
      b.x = fma(0.5, ax, fma(RIp[i], np.x, fma(RIm[i], nm.x, -ak_t * nz.y)));
      b.y = fma(0.5, ay, fma(RIp[i], np.y, fma(RIm[i], nm.y, ak_t * nz.x)));
    }
    P[i * T + mi_t] = b;
  }
  __syncthreads();

  if (tid < NP) {
    // ---- pressure-Poisson solve (provisional dp/dr(1) = 0; (0,0): p(1) = 0)
    const int j = tid >> (SP ? 3 : 2), part = j & 1, mi = j >> 1;
    const int k = min(kk0 + mi, nk - 1) - (K - 1), ik = abs(k);
    const int op = (ik == 0 && m == 0) ? K * M : ik * M + m;
    if constexpr (SP) {  // lanes 0-3 of the chain's 8: top half, 4-7: bottom half
      const int h = (tid >> 2) & 1, kh = N >> 1;
      band_solve4(s.luP2 + ((long)op * N + h * kh) * kLuSlots, (double*)P + 2 * mi + part + h * kh * 2 * T, 2 * T,
                  kh);
    } else {
      band_solve4(s.luP + (long)op * N * kLuSlots, (double*)P + 2 * mi + part, 2 * T, N);
    }
  } else {
    // ---- meanwhile: the p-independent part of the velocity right-hand sides
    for (int e = tid - NP; e < N * NT; e += NB - NP) {
      const int c = e % NT, i = e / NT;
      const int part = c & 1, mi = (c >> 1) % T, f = (c >> 1) / T;
      const double2 u = uj(f, i, mi);
      if (stage && part == 0) UJ[(f * N + i) * T + mi] = u;
      const double w = part ? u.y : u.x;
      double b;
      if (i < N - 1) b = fma(ci, w, X[i * NT + c]);  // X held N_eff of this chain's element
      else b = m == 0 && kk0 + mi == K - 1 ? 0.0 : cu * w;
      X[i * NT + c] = b;
    }
    // u_j near the wall for the influence step (rows N-9..N-2 of u+, u-), or,
    // staged, the influence responses of the tile
    if (stage) {
      const int nch = basis_ld(N) / 2;  // 16-byte chunks per mode
      for (int e = tid - NP; e < nch * T; e += NB - NP) {
        const int mi = e / nch, ch = e - mi * nch;
        const int ik = abs(min(kk0 + mi, nk - 1) - (K - 1));
        cp_async16(BS + (long)mi * basis_ld(N) + 2 * ch, s.basis + (long)(ik * M + m) * basis_ld(N) + 2 * ch);
      }
      cp_async_commit();
      cp_async_wait<0>();
    }
    if (uw_in_s) {
      for (int e = tid - NP; e < 16 * T; e += NB - NP) {
        const int mi = e % T, w = e / T;
        UW[mi * 16 + w] = uj(w >> 3, N - 9 + (w & 7), mi);
      }
    }
  }
  __syncthreads();
  if constexpr (SP)  // the pressure chains' interface and correction
    spike_fix<NB>(tid, N, 2 * T, 2 * T, (double*)P, s.spkP, s.rP, Zs, [&](int c) {
      const int ik = abs(min(kk0 + (c >> 1), nk - 1) - (K - 1));
      return (ik == 0 && m == 0) ? K * M : ik * M + m;
    });

  // ---- d_r p per (mode, row), subtracted at once from the right-hand sides of
  //      the three fields (rows < N-1):
  //      (grad p)+- = d_r p -+ m~ p / r,  (grad p)_z = i ak p
  auto subtract_gradient = [&](int i, int mi, double ak, double2 dp) {
    const double2 pp = P[i * T + mi];
    const double mr = mt * RI[i];
    double* xr = X + i * NT;
    const int c0 = mi << 1, c1 = (T + mi) << 1, c2 = (2 * T + mi) << 1;
    xr[c0] = fma(mr, pp.x, xr[c0] - dp.x);
    xr[c0 + 1] = fma(mr, pp.y, xr[c0 + 1] - dp.y);
    xr[c1] = fma(-mr, pp.x, xr[c1] - dp.x);
    xr[c1 + 1] = fma(-mr, pp.y, xr[c1 + 1] - dp.y);
    xr[c2] = fma(ak, pp.y, xr[c2]);
    xr[c2 + 1] = fma(-ak, pp.x, xr[c2 + 1]);
  };
  if constexpr (DIG) {
    for_stencil_items([&](int i, int mi) { return P[i * T + mi]; }, ps, 0, [&](int i, int mi, double ak, double2 dp) {
      if (i < N - 1) subtract_gradient(i, mi, ak, dp);
    });
  } else
  for (int i = tid / T; i < N - 1; i += NB / T) {
    const int lo = row_lo_d(i, N);
    double ax = 0.0, ay = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const double2 pv2 = P[(lo + q) * T + mi_t];
      const double w = ws[i * 9 + q];
      ax = fma(w, pv2.x, ax);
      ay = fma(w, pv2.y, ay);
    }
    subtract_gradient(i, mi_t, ak_t, double2{ax, ay});
  }
  __syncthreads();

  // ---- implicit viscous solves (1/dt - cL) v = rhs, v(1) = ((1-c)/c) u_j(1)
  {  // 6T chains x 4 (SP: 8) lanes = all threads
    const int c = tid >> (SP ? 3 : 2);
    const int mi = (c >> 1) % T, f = (c >> 1) / T;
    const int k = min(kk0 + mi, nk - 1) - (K - 1), ik = abs(k);
    const int op = ik * s.nJ + s.hop[3 * m + f];
    if constexpr (SP) {
      const int h = (tid >> 2) & 1, kh = N >> 1;
      band_solve4(s.luH2 + ((long)op * N + h * kh) * kLuSlots, X + c + h * kh * NT, NT, kh);
    } else {
      band_solve4(s.luH + (long)op * N * kLuSlots, X + c, NT, N);
    }
  }
  __syncthreads();
  if constexpr (SP)  // the velocity chains' interface and correction
    spike_fix<NB>(tid, N, NT, NT, X, s.spkH, s.rH, Zs, [&](int c) {
      const int ik = abs(min(kk0 + ((c >> 1) % T), nk - 1) - (K - 1));
      return ik * s.nJ + s.hop[3 * m + (c >> 1) / T];
    });

  // ---- influence matrix on u = v - ((1-c)/c) u_j.  The wall value of v makes
  //      u(1) = 0 exactly, so of the boundary vector g = (u+(1), u-(1), u_z(1),
  //      div u(1)) only the divergence is left, and of the coefficients
  //      a = -A^{-1} g only the pressure response's (the unit wall responses
  //      have zero there).  Eight threads per mode, one per row of the wall
  //      stencil (its ninth row is the wall).
  if (tid < 8 * T) {  // whole warps (T >= 4)
    const int mj = tid >> 3, q = tid & 7, i = N - 9 + q;
    const double2 A = s.ainv[(long)m * nk + min(kk0 + mj, nk - 1)];
    auto uv = [&](int ff) {
      const int c = (ff * T + mj) << 1;
      const double2 w = stage     ? UJ[(ff * N + i) * T + mj]
                        : uw_in_s ? UW[mj * 16 + ff * 8 + q]
                                  : uj(ff, i, mj);
      return double2{X[i * NT + c] - cu * w.x, X[i * NT + c + 1] - cu * w.y};
    };
    const double2 p = uv(0), mm = uv(1);
    const double w = 0.5 * wall[q];
    double2 g = double2{w * (p.x + mm.x), w * (p.y + mm.y)};
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      g.x += __shfl_xor_sync(0xffffffffu, g.x, o, 8);
      g.y += __shfl_xor_sync(0xffffffffu, g.y, o, 8);
    }
    if (q == 0) coef[mj] = double2{fma(A.y, g.y, -A.x * g.x), -fma(A.x, g.y, A.y * g.x)};
  }
  __syncthreads();

  // final value of chain c at row i: v - ((1-c)/c) u_j + pressure response
  auto final_value = [&](int i, int c) {
    const int part = c & 1, mi = (c >> 1) % T, f = (c >> 1) / T;
    const int kk = min(kk0 + mi, nk - 1), k = kk - (K - 1);
    const double* Bv = s.basis + (long)(abs(k) * M + m) * basis_ld(N);
    const double2 a0 = coef[mi];
    // u_z responses carry i sign(k): coefficient sign(k) (a0.x, -a0.y) swapped
    const double az = part ? a0.x : -a0.y;
    const double c0 = f == 2 ? (k > 0 ? az : (k < 0 ? -az : 0.0)) : (part ? a0.y : a0.x);
    const double2 w = stage ? UJ[(f * N + i) * T + mi] : a.Uj[f * fs + base + (long)i * nk + kk];
    const double* B = stage ? BS + (long)mi * basis_ld(N) : Bv;
    return fma(c0, B[i * 3 + f], X[i * NT + c] - cu * (part ? w.y : w.x));
  };

  // ---- fixed flux on (0,0): beta' so that 2 pi int u_z r dr = pi/2
  const bool has_mean = (m == 0 && kk0 <= K - 1 && K - 1 < kk0 + T);
  const int cz = (2 * T + (K - 1 - kk0)) << 1;  // chain (u_z, mode k=0, re)
  if (has_mean) {
    if (tid < 32) {  // warp 0 (full: NB >= 96)
      double q = 0.0;
      for (int i = tid; i < N; i += 32) q += s.wq[i] * final_value(i, cz);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      if (tid == 0) {
        const double bp = (0.25 - q) / s.prm[kPrmSumWG];
        misc[0] = bp;
        *a.beta_p = bp;
      }
    }
    __syncthreads();
  }
  const double bp = has_mean ? misc[0] : 0.0;

  grid_dep_trigger_at(d, 2);
  // ---- write out (coalesced over k)
#pragma unroll 4
  for (int e = tid; e < N * NT; e += NB) {
    const int c = e % NT, i = e / NT;
    const int part = c & 1, mi = (c >> 1) % T, f = (c >> 1) / T;
    if (kk0 + mi >= nk) continue;
    double v = final_value(i, c);
    if (has_mean && c == cz) v += bp * s.G[i];
    double* out = (double*)(a.Uout + f * fs + base + (long)i * nk + kk0 + mi) + part;
    *out = v;
    if (CURL && a.W6) X[i * NT + c] = v;  // (only this element's own X is read above)
  }

  // ---- FP64 steps on grids of at most a block per SM: the curl (A1) of the
  //      new state for the next nonlinear evaluation from the block's radial
  //      columns.  There the time is latency: a curl launch of its own took
  //      3 us longer per pass at N = 32, 31 x 16 modes (on larger grids it is
  //      the faster form).  But for the split solve the values are k_curl's.
  if (CURL && a.W6) {
    a.W6 = bofs(a.W6, d.ss);
    __syncthreads();
    const int c0 = mi_t << 1, c1 = (T + mi_t) << 1, c2 = (2 * T + mi_t) << 1;
    for (int i = tid / T; i < N; i += NB / T) {  // u_theta
      const double* xr = X + i * NT;
      P[i * T + mi_t] = double2{0.5 * (xr[c0 + 1] - xr[c1 + 1]), -0.5 * (xr[c0] - xr[c1])};
    }
    __syncthreads();
    auto put = [&](int i, int mi, double ak, double2 dz, double2 dt) {  // dz, dt: d/dr of u_z, u_theta
      if (kk0 + mi >= nk) return;
      const double* xr = X + i * NT;
      const int b0 = mi << 1, b1 = (T + mi) << 1, b2 = (2 * T + mi) << 1;
      const double2 ur = double2{0.5 * (xr[b0] + xr[b1]), 0.5 * (xr[b0 + 1] + xr[b1 + 1])};
      const double2 ut = P[i * T + mi], uz = double2{xr[b2], xr[b2 + 1]};
      const double ri = RI[i], mri = mt * ri;
      double2* W = a.W6 + base + (long)i * nk + kk0 + mi;
      W[0] = ur;
      W[fs] = ut;
      W[2 * fs] = uz;
      W[3 * fs] = double2{-fma(mri, uz.y, -ak * ut.y), fma(mri, uz.x, -ak * ut.x)};  // (as k_curl rounds)
      W[4 * fs] = double2{fma(-ak, ur.y, -dz.x), fma(ak, ur.x, -dz.y)};
      W[5 * fs] = double2{fma(mri, ur.y, fma(ri, ut.x, dt.x)), fma(-mri, ur.x, fma(ri, ut.y, dt.y))};
    };
    if constexpr (!SP) {  // (a row and mode belong to the same lane in both passes)
      for_stencil_items([&](int i, int mi) { return P[i * T + mi]; }, pv, 0,
                        [&](int i, int mi, double, double2 dt) { S[i * T + mi] = dt; });
      for_stencil_items([&](int i, int mi) { return *(const double2*)(X + i * NT + ((2 * T + mi) << 1)); }, ps, 0,
                        [&](int i, int mi, double ak, double2 dz) { put(i, mi, ak, dz, S[i * T + mi]); });
    } else {
      for (int i = tid / T; i < N; i += NB / T) {
        const int lo = row_lo_d(i, N);
        double2 dz = double2{0.0, 0.0}, dt = dz;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          const double* xq = X + (lo + q) * NT + c2;
          const double2 tq = P[(lo + q) * T + mi_t];
          dz.x = fma(ws[i * 9 + q], xq[0], dz.x);
          dz.y = fma(ws[i * 9 + q], xq[1], dz.y);
          dt.x = fma(wv[i * 9 + q], tq.x, dt.x);
          dt.y = fma(wv[i * 9 + q], tq.y, dt.y);
        }
        put(i, mi_t, ak_t, dz, dt);
      }
    }
  }
}

static size_t solve_smem(int N, int T);

// Tile of T modes: 4 keeps every warp of the sequential phases full (8
// right-hand sides per warp) with the most blocks; 8 when there are many
// modes per SM and two blocks of the tile still fit on an SM (so that one
// block's sequential phases overlap another's).  Measured on the ensemble's
// groups, 16 was never faster than 8 (N=32: 827 vs 767 us per launch); the
// autotuner and option "tile" can still choose it.
static int solve_tile(const Dims& d) {
  if (d.tile == 4 || d.tile == 8 || d.tile == 16) return d.tile;
  const long modes = (long)d.nk * d.M * d.B;
  if (modes / 8 >= 4 * 152 && solve_smem(d.N, 8) <= 110 * 1024) return 8;
  return 4;
}

// What a resolution or tile has to fit in to be accepted: a block that keeps
// the stencils' weights as well, as the split solve's does (N <= 475 with the
// 4-mode tile), whichever form then runs.
size_t solve_smem_bytes(int N, int T) {
  return std::max(solve_smem(N, T), (size_t)(2 * N * T + 4 * T) * 16 + (size_t)48 * N * T + (size_t)(21 * N + 4) * 8);
}

bool solve_takes_curl(const Dims& d) {
  return solve_tile(d) == 4 && (long)((d.nk + 3) / 4) * d.M * d.B <= device_sms();
}

static size_t solve_smem(int N, int T) {
  return solve_stage_fits(N, T) ? solve_smem_staged(N, T) : solve_smem_base(N, T);
}

// Stage u_j and the responses when the staged block fits and the SM still
// holds as many blocks as the grid can use (so staging never costs occupancy).
static bool solve_use_stage(const Dims& d, int T, long blocks, bool sp = false) {
  if (!solve_stage_fits(d.N, T)) return false;
  struct SmInfo {
    int sms = 1, smem_sm = 0;
  };
  static const SmInfo info = [] {  // (thread-safe one-time initialisation)
    SmInfo i;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&i.sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&i.smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (i.sms <= 0) i.sms = 1;
    return i;
  }();
  const int sms = info.sms, smem_sm = info.smem_sm;
  const size_t reserve = 1024;  // per-block shared memory the system keeps
  const long with = (long)(smem_sm / (solve_smem_staged(d.N, T, sp) + reserve));
  const long without = (long)(smem_sm / (solve_smem_base(d.N, T, sp) + reserve));
  const long need = (blocks + sms - 1) / sms;
  return with >= std::min(need, without);
}

// Chunk sizes keep every transform block within ~96 KB of shared memory (two
// blocks per SM) and give each transform kernel at least two blocks per SM
// (smaller chunks, same arithmetic per column).
void choose_chunks(Dims* d) {
  const size_t budget = 96 * 1024, vb = sizeof(double2);
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long target = 2L * sms;
  auto blocks = [&](int extent, int chunk, long rest) { return (long)((extent + chunk - 1) / chunk) * rest; };
  d->mcz = 8;
  while (d->mcz > 1 && (zsynth_smem(*d, d->mcz, vb) > budget || blocks(d->M, d->mcz, 6L * d->N * d->B) < target))
    d->mcz /= 2;
  d->mca = 8;
  while (d->mca > 1 && (zanalysis_smem(*d, d->mca, vb) > budget || blocks(d->M, d->mca, (long)d->N * d->B) < target))
    d->mca /= 2;
  d->zc = 4;
  while (d->zc > 1 && (product_smem(*d, d->zc, vb) > budget || blocks(d->nz, d->zc, (long)d->N * d->B) < target))
    d->zc /= 2;
}

// The dynamic shared-memory limit is a per-kernel, process-wide attribute, so
// it is raised to the device's opt-in maximum (never lowered): handles of
// different sizes then never restrict one another.
bool prepare_kernel_attrs(const Dims& d) {
  const size_t vb = sizeof(double2);
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return false;
  const size_t lim = (size_t)optin;
  if (zsynth_smem(d, d.mcz, vb) > lim || zanalysis_smem(d, d.mca, vb) > lim ||
      product_smem(d, d.zc, vb) > lim || solve_smem_bytes(d.N, solve_tile(d)) > lim)
    return false;
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  bool ok = dft_prepare_attrs();
  with_long_fft_length(d.nz, [&](auto n) {
    constexpr int L = decltype(n)::value;
    ok = ok && cudaFuncSetAttribute(k_zsynth<double2, L>, a, optin) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_zanalysis<double2, L>, a, optin) == cudaSuccess;
  });
  with_fft_length(d.nz, [&](auto n) {
    constexpr int L = decltype(n)::value;
    ok = ok && cudaFuncSetAttribute(k_zsynth<float2, L>, a, optin) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_zanalysis<float2, L>, a, optin) == cudaSuccess;
  });
  with_long_fft_length(d.nth, [&](auto n) {
    ok = ok && cudaFuncSetAttribute(k_product<double2, decltype(n)::value>, a, optin) == cudaSuccess;
  });
  with_fft_length(d.nth, [&](auto n) {
    constexpr int L = decltype(n)::value;
    ok = ok && cudaFuncSetAttribute(k_product<float2, L>, a, optin) == cudaSuccess;
  });
  auto solves = [&](auto dig) {
    constexpr bool D = decltype(dig)::value;
    ok = ok && cudaFuncSetAttribute(k_solve<16, D>, a, optin) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_solve<8, D>, a, optin) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_solve<4, D>, a, optin) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_solve<4, D, false, true>, a, optin) == cudaSuccess;
  };
  if (solve_by_digits(d.N, false)) solves(std::true_type{});
  else solves(std::false_type{});
  ok = ok && cudaFuncSetAttribute(k_solve<4, false, true>, a, optin) == cudaSuccess;
  auto fusable = [](int n) { return n == 48 || n == 72 || n == 96; };
  if (fusable(d.nz) && fusable(d.nth))  // (the option or the autotuner may switch the fused launch on later)
    with_fused_lengths(d.nz, d.nth, [&](auto z, auto t) {
      ok = ok && cudaFuncSetAttribute(k_nl_fused32<decltype(z)::value, decltype(t)::value>, a, optin) == cudaSuccess;
    });
  return ok;
}

// Shared-memory limits of the FP64 nonlinear-term kernels only (z synthesis,
// theta product, z analysis) for the allocation-free entry point: checks their
// footprints, which do not depend on N, against the opt-in limit and raises
// their dynamic shared-memory limit to it.
bool prepare_nonlinear_attrs(const Dims& d) {
  const size_t vb = sizeof(double2);
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return false;
  const size_t lim = (size_t)optin;
  if (zsynth_smem(d, d.mcz, vb) > lim || zanalysis_smem(d, d.mca, vb) > lim || product_smem(d, d.zc, vb) > lim)
    return false;
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  bool ok = dft_prepare_attrs();
  with_long_fft_length(d.nz, [&](auto n) {
    constexpr int L = decltype(n)::value;
    ok = ok && cudaFuncSetAttribute(k_zsynth<double2, L>, a, optin) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(k_zanalysis<double2, L>, a, optin) == cudaSuccess;
  });
  with_long_fft_length(d.nth, [&](auto n) {
    constexpr int L = decltype(n)::value;
    ok = ok && cudaFuncSetAttribute(k_product<double2, L>, a, optin) == cudaSuccess;
  });
  return ok;
}

// The radial resolution that entry point accepts: that of a block which keeps
// up to four columns of the curl (N <= 968 with four), although k_curl itself
// needs no shared memory.
bool nonlinear_radial_fits(const Dims& d) {
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return false;
  const size_t cols = (size_t)d.M * d.nk, blocks = (cols + 3) / 4, kc = (cols + blocks - 1) / blocks;
  return (size_t)d.N * (56 * kc + 16) + 16 * kc <= (size_t)optin;
}

void launch_solve(const Dims& d, const DevSetup& s, const SolveArgs& a, int nJ, cudaStream_t st) {
  const int T = solve_tile(d);
  const bool sp = d.spike && T == 4 && s.luH2;  // the split solve (one-wave grids, factors built)
  dim3 g((d.nk + T - 1) / T, d.M, d.B);
  const bool stage = solve_use_stage(d, T, (long)g.x * g.y * g.z, sp);
  SolveDev sd{s.d1,  s.rinv, s.wq,   s.hop,  s.luH,  s.luP,  s.basis, s.ainv, s.G,  s.prm,
              stencil_at(s.stab, s.d1, d.N), nJ,    stage ? 1 : 0,  s.luH2, s.luP2, s.spkH,  s.spkP, s.rH, s.rP};
  const size_t sm = stage ? solve_smem_staged(d.N, T, sp) : solve_smem_base(d.N, T, sp);
  if (sp) return launch_step_kernel(d, k_solve<4, false, true>, g, dim3(48 * 4), sm, st, d, sd, a);
  auto go = [&](auto dig) {
    constexpr bool D = decltype(dig)::value;
    if (T == 16) launch_step_kernel(d, k_solve<16, D>, g, dim3(24 * 16), sm, st, d, sd, a);
    else if (T == 8) launch_step_kernel(d, k_solve<8, D>, g, dim3(24 * 8), sm, st, d, sd, a);
    else if (a.W6) launch_step_kernel(d, k_solve<4, D, false, true>, g, dim3(24 * 4), sm, st, d, sd, a);
    else launch_step_kernel(d, k_solve<4, D>, g, dim3(24 * 4), sm, st, d, sd, a);
  };
  if (solve_by_digits(d.N, false)) go(std::true_type{});
  else go(std::false_type{});
}

// ------------------------------------------------------------------ diagnostics
// E/E_lam = 6 sum' w |u|^2, D/D_lam = sum' w |w|^2, I/I_lam = 4 (1 + beta) int u_z00 r dr
__global__ void __launch_bounds__(256) k_energy(Dims d, const double* __restrict__ wq,
                                                const double2* __restrict__ W6, double* partial) {
  __shared__ double su[256], sw[256];
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  double eu = 0.0, ew = 0.0;
  if (idx < d.F) {
    const int n = (idx / d.nk) % d.N;
    const int m = idx / ((long)d.nk * d.N);
    const double w = (m == 0 ? 1.0 : 2.0) * wq[n];
    for (int f = 0; f < 3; ++f) {
      const double2 u = W6[f * d.F + idx], o = W6[(3 + f) * d.F + idx];
      eu += u.x * u.x + u.y * u.y;
      ew += o.x * o.x + o.y * o.y;
    }
    eu *= w;
    ew *= w;
  }
  su[threadIdx.x] = eu;
  sw[threadIdx.x] = ew;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      su[threadIdx.x] += su[threadIdx.x + h];
      sw[threadIdx.x] += sw[threadIdx.x + h];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = su[0];
    partial[2 * blockIdx.x + 1] = sw[0];
  }
}

__global__ void k_energy_final(Dims d, const double* __restrict__ partial, int nblk,
                               const double* __restrict__ wq, const double2* __restrict__ U,
                               const double* beta_p, const double* prm, double* out3) {
  __shared__ double su[256], sw[256], sq[256];
  double a = 0.0, b = 0.0, q = 0.0;
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
    a += partial[2 * i];
    b += partial[2 * i + 1];
  }
  const double2* uz = U + 2 * d.F + (d.K - 1);  // (k,m) = (0,0), u_z: the flux int u_z r dr
  for (int n = threadIdx.x; n < d.N; n += blockDim.x) q += wq[n] * uz[(long)n * d.nk].x;
  su[threadIdx.x] = a;
  sw[threadIdx.x] = b;
  sq[threadIdx.x] = q;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
      su[threadIdx.x] += su[threadIdx.x + h];
      sw[threadIdx.x] += sw[threadIdx.x + h];
      sq[threadIdx.x] += sq[threadIdx.x + h];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double beta = *beta_p * prm[kPrmRe] / 4.0;
    out3[0] = 6.0 * su[0];
    out3[1] = 4.0 * (1.0 + beta) * sq[0];
    out3[2] = sw[0];
  }
}

int energy_blocks(const Dims& d) { return (int)((d.F + 255) / 256); }

void launch_energy(const Dims& d, const DevSetup& s, const double2* U, const double2* W6,
                   const double* beta_p, double* partial, int nblk, double* out3, cudaStream_t st) {
  k_energy<<<nblk, 256, 0, st>>>(d, s.wq, W6, partial);
  k_energy_final<<<1, 256, 0, st>>>(d, partial, nblk, s.wq, U, beta_p, s.prm, out3);
}

// Boundary vector g of section 2 over all modes: max |u(1)| and max |div u(1)|.
__global__ void k_wall(Dims d, const double* __restrict__ d1, const double2* __restrict__ U,
                       unsigned long long* out2) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= d.M * d.nk) return;
  const int m = idx / d.nk, kk = idx % d.nk, N = d.N;
  const long fs = d.F;
  const double2* up = U + ((long)m * N) * d.nk + kk;
  const double2* um = up + fs;
  const double2* uz = up + 2 * fs;
  const long w = (long)(N - 1) * d.nk;
  const double2 a = up[w], b = um[w], c = uz[w];
  const double ur = hypot(0.5 * (a.x + b.x), 0.5 * (a.y + b.y));
  const double ut = hypot(0.5 * (a.y - b.y), 0.5 * (a.x - b.x));
  const double umax = fmax(fmax(ur, ut), hypot(c.x, c.y));
  atomicMax(out2, __double_as_longlong(umax));
  if (m == 0 && kk == d.K - 1) return;
  const int mt = d.m_p * m;
  const double ak = d.alpha * (kk - (d.K - 1));
  const double* wr = d1 + ((long)((mt & 1) ^ 1) * N + N - 1) * 9;
  double sx = 0.0, sy = 0.0;
  for (int q = 0; q < 9; ++q) {
    const long o = (long)(N - 9 + q) * d.nk;
    sx += wr[q] * (up[o].x + um[o].x);
    sy += wr[q] * (up[o].y + um[o].y);
  }
  const double dx = 0.5 * sx + 0.5 * ((1 + mt) * a.x + (1 - mt) * b.x) - ak * c.y;
  const double dy = 0.5 * sy + 0.5 * ((1 + mt) * a.y + (1 - mt) * b.y) + ak * c.x;
  atomicMax(out2 + 1, __double_as_longlong(hypot(dx, dy)));
}

void launch_wall(const Dims& d, const DevSetup& s, const double2* U, double* out2, cudaStream_t st) {
  cudaMemsetAsync(out2, 0, 2 * sizeof(double), st);
  const int nm = d.M * d.nk;
  k_wall<<<(nm + 127) / 128, 128, 0, st>>>(d, s.d1, U, (unsigned long long*)out2);
}

__global__ void k_nan(const double* __restrict__ x, long n, int* flag) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    if (!isfinite(x[i])) {
      atomicOr(flag, 1);
      return;
    }
}

void launch_nan_check(const double* x, long n, int* flag, cudaStream_t st) {
  cudaMemsetAsync(flag, 0, sizeof(int), st);
  k_nan<<<304, 256, 0, st>>>(x, n, flag);
}

}  // namespace opf
