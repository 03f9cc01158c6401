// Proposal network for Newton-Krylov initial guesses: a 1-D convolution net
// over the radial points acting on the lowest Fourier modes of a state.
//
//   h1 = gelu(conv3(x;  W1, b1))          x: [B][L][Cin]   (L radial points)
//   h2 = gelu(conv3(h1; W2, b2))          h: [B][L][H]
//   y  = conv3(h2; W3, b3)                y: [B][L][Cin]   (correction of x)
//   z  = Wh mean_l(h2) + bh               z: [B][2]        (period, shift)
//   loss = mean((y - ty)^2) + lambda mean((z - tz)^2)
//
// conv3 is a width-3 convolution along l with zero padding.  Every
// convolution and its two backward products is one GEMM on BF16 operands
// with FP32 accumulation on the tcgen05 tensor cores (opf_tcgemm.cu).  The
// products over channels take im2col rows (x[b][l + j - 1][c] at column
// j*C + c, zero padded), which the producer of the activations -- the first
// kernel, or the previous GEMM's epilogue -- writes directly; the weight
// gradients take the same rows by columns, so nothing is transposed.  Master
// weights and Adam moments are FP32.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>

#include "opf_internal.h"

namespace {

using bf16 = __nv_bfloat16;

// ------------------------------------------------------------------ operand layouts
// d/dx of gelu(x) = x Phi(x): Phi(x) + x phi(x) (the forward GELU is applied
// in the GEMM epilogue)
__device__ __forceinline__ float gelu_grad(float x) {
  const float cdf = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
  const float pdf = 0.39894228040143268f * expf(-0.5f * x * x);
  return cdf + x * pdf;
}

long pad128(long v) { return (v + 127) / 128 * 128; }
long pad64(long v) { return (v + 63) / 64 * 64; }

int gs(long n);

// V channels at c of one row's BF16 values into the im2col rows of a width-3
// convolution: row m's block j holds x[l + s (j - 1)], s = +1 (forward) or -1
// (its transpose), zeros past the ends.  col: row m, channel c of block 0.
template <typename T>
__device__ __forceinline__ void put_cols(T v, T zero, bf16* col, long ldc, int C, int l, int L, bool rev) {
  const int up = rev ? 2 : 0, down = 2 - up;  // the block in row l + 1 and in row l - 1
  *(T*)(col + C) = v;
  if (l + 1 < L) *(T*)(col + ldc + up * C) = v;
  else *(T*)(col + down * C) = zero;
  if (l > 0) *(T*)(col - ldc + down * C) = v;
  else *(T*)(col + up * C) = zero;
}

// x (FP32 [BL][C]) as BF16 im2col rows; VEC: eight channels per thread (C a
// multiple of 8, x 16-byte aligned).
template <bool VEC>
__global__ void k_x_cols(const float* __restrict__ x, int L, int C, bf16* __restrict__ col, long ldc) {
  const long m = blockIdx.x;
  const int l = (int)(m % L), c = (blockIdx.y * blockDim.x + threadIdx.x) * (VEC ? 8 : 1);
  if (c >= C) return;
  const float* s = x + m * C + c;
  bf16* d = col + m * ldc + c;
  if constexpr (VEC) {
    const float4 a = *(const float4*)s, b = *(const float4*)(s + 4);
    const __nv_bfloat162 p[4] = {__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(a.z, a.w),
                                 __floats2bfloat162_rn(b.x, b.y), __floats2bfloat162_rn(b.z, b.w)};
    put_cols(*(const uint4*)p, make_uint4(0u, 0u, 0u, 0u), d, ldc, C, l, L, false);
  } else {
    put_cols(__float2bfloat16(*s), __float2bfloat16(0.f), d, ldc, C, l, L, false);
  }
}

// padded copy: out[r][c] = src[r][c] for r < R, c < C, else 0; out is [Rp][Cp]
__global__ void k_pad(const bf16* __restrict__ src, int R, int C, bf16* __restrict__ out, int Rp, int Cp) {
  const long n = (long)Rp * Cp;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const int r = (int)(i / Cp), c = (int)(i - (long)r * Cp);
    out[i] = (r < R && c < C) ? src[(long)r * C + c] : __float2bfloat16(0.f);
  }
}

// weights of the input-gradient product: out[c][j*Cout + o] = W[o][j*Cin + c]; out is [Cinp][Kp]
__global__ void k_wshift(const bf16* __restrict__ W, int Cout, int Cin, bf16* __restrict__ out, int Cinp, int Kp) {
  const long n = (long)Cinp * Kp;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const int c = (int)(i / Kp), k = (int)(i - (long)c * Kp);
    bf16 v = __float2bfloat16(0.f);
    if (c < Cin && k < 3 * Cout) {
      const int j = k / Cout, o = k - j * Cout;
      v = W[(long)o * 3 * Cin + (long)j * Cin + c];
    }
    out[i] = v;
  }
}

// ------------------------------------------------------------------ small kernels
__global__ void k_to_bf16(const float* __restrict__ x, bf16* __restrict__ y, long n) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16(x[i]);
}

// mean over l of h2 (the middle block of its im2col rows) and the head:
// pooled[b][c], z[b][o] = sum_c Wh[o][c] pooled[b][c] + bh[o]; one block per
// b, two thirds of a channel's rows in flight at a time
constexpr int kPoolThreads = 512;
__global__ void __launch_bounds__(kPoolThreads) k_pool_head(const bf16* __restrict__ col, long ldc, int L, int C,
                                                            int O, const float* __restrict__ Wh,
                                                            const float* __restrict__ bh, float* pooled,
                                                            float* __restrict__ z) {
  const long b = blockIdx.x;
  float* sp = pooled + b * C;
  const bf16* h = col + b * L * ldc + C;
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float s = 0.f;
    for (int l0 = 0; l0 < L; l0 += 32) {
      bf16 v[32];
#pragma unroll
      for (int q = 0; q < 32; ++q) v[q] = l0 + q < L ? h[(l0 + q) * ldc + c] : __float2bfloat16(0.f);
#pragma unroll
      for (int q = 0; q < 32; ++q) s += __bfloat162float(v[q]);
    }
    sp[c] = s / L;
  }
  __syncthreads();
  for (int o = threadIdx.x >> 5; o < O; o += blockDim.x >> 5) {
    float s = 0.f;
#pragma unroll 8
    for (int c = threadIdx.x & 31; c < C; c += 32) s += Wh[(long)o * C + c] * sp[c];
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if ((threadIdx.x & 31) == 0) z[b * O + o] = bh[o] + s;
  }
}

// Gradient tiles: a block takes 32 rows x 64 columns, thread (tx, ty) columns
// 2 tx, 2 tx + 1 of rows ty, ty + 8, ..; column sums (bias gradients) of the
// block go to csum[block row][C], added up by k_bias_sum in a fixed order.
// Blocks along one grid axis, a row's tiles next to one another (the other
// axes end at 65,535).
constexpr int kGradRows = 32, kGradCols = 64;
int grad_tiles(int C) { return (C + kGradCols - 1) / kGradCols; }

__device__ __forceinline__ void grad_column_sums(float s0, float s1, long row, int c, int C, float* csum) {
  __shared__ float2 part[8][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  part[ty][tx] = make_float2(s0, s1);
  __syncthreads();
  if (ty == 0) {
    for (int q = 1; q < 8; ++q) {
      s0 += part[q][tx].x;
      s1 += part[q][tx].y;
    }
    if (c < C) csum[row * C + c] = s0;
    if (c + 1 < C) csum[row * C + c + 1] = s1;
  }
}

// one gradient pair as BF16: rows dz (ldz apart, an even number) and, if
// dzcol, the im2col rows of the transposed convolution
__device__ __forceinline__ void put_grad(float v0, float v1, long m, int c, int C, int L, bf16* dz, long ldz,
                                         bf16* dzcol, long ldc) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(v0, v1);
  const int l = (int)(m % L);
  if (c + 1 < C) {
    *(__nv_bfloat162*)(dz + m * ldz + c) = p;
  } else {
    dz[m * ldz + c] = p.x;
  }
  if (!dzcol) return;
  bf16* d = dzcol + m * ldc + c;
  if (!(C & 1)) {
    put_cols(*reinterpret_cast<const unsigned*>(&p), 0u, d, ldc, C, l, L, true);
  } else {
    put_cols(p.x, __float2bfloat16(0.f), d, ldc, C, l, L, true);
    if (c + 1 < C) put_cols(p.y, __float2bfloat16(0.f), d + 1, ldc, C, l, L, true);
  }
}

// dL/dy = 2 scale (y - t) of the output layer, and sum (y - t)^2
__global__ void __launch_bounds__(256) k_out_grad(const float* __restrict__ y, const float* __restrict__ t, int BL,
                                                  int L, int C, float scale, bf16* __restrict__ dz, long ldz,
                                                  bf16* __restrict__ dzcol, long ldc, float* __restrict__ csum,
                                                  double* __restrict__ sum) {
  const int tiles = (C + kGradCols - 1) / kGradCols, row = blockIdx.x / tiles;
  const int c = (blockIdx.x - row * tiles) * kGradCols + 2 * (threadIdx.x & 31);
  double acc = 0.0;
  float s0 = 0.f, s1 = 0.f;
#pragma unroll
  for (int q = 0; q < kGradRows / 8; ++q) {
    const long m = (long)row * kGradRows + q * 8 + (threadIdx.x >> 5);
    if (m >= BL || c >= C) continue;
    const long i = m * C + c;
    const float r0 = y[i] - t[i], r1 = c + 1 < C ? y[i + 1] - t[i + 1] : 0.f;
    acc += (double)r0 * r0;
    acc += (double)r1 * r1;
    const float g0 = 2.f * scale * r0, g1 = 2.f * scale * r1;
    s0 += g0;
    s1 += g1;
    put_grad(g0, g1, m, c, C, L, dz, ldz, dzcol, ldc);
  }
  grad_column_sums(s0, s1, row, c, C, csum);
  __shared__ double sh[8];
  for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) acc += sh[q];
    atomicAdd(sum, acc);
  }
}

// dZ = dH gelu'(pre) of a hidden layer; dH = sum over splits of dh [split][BL][C]
// plus, under the head, the pooled mean's gradient dpool[b][c]
__global__ void __launch_bounds__(256) k_hidden_grad(const float* __restrict__ dh, int nsplit,
                                                     const float* __restrict__ pre, int BL, int L, int C,
                                                     const float* __restrict__ dpool, bf16* __restrict__ dz, long ldz,
                                                     bf16* __restrict__ dzcol, long ldc, float* __restrict__ csum) {
  const int tiles = (C + kGradCols - 1) / kGradCols, row = blockIdx.x / tiles;
  const int c = (blockIdx.x - row * tiles) * kGradCols + 2 * (threadIdx.x & 31);
  const long total = (long)BL * C;
  float s0 = 0.f, s1 = 0.f;
#pragma unroll
  for (int q = 0; q < kGradRows / 8; ++q) {
    const long m = (long)row * kGradRows + q * 8 + (threadIdx.x >> 5);
    if (m >= BL || c >= C) continue;
    const long i = m * C + c;
    float v[2] = {0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (c + u >= C) continue;
      float h = 0.f;
      for (int k = 0; k < nsplit; ++k) h += dh[k * total + i + u];
      if (dpool) h += dpool[m / L * C + c + u];
      v[u] = h * gelu_grad(pre[i + u]);
    }
    s0 += v[0];
    s1 += v[1];
    put_grad(v[0], v[1], m, c, C, L, dz, ldz, dzcol, ldc);
  }
  grad_column_sums(s0, s1, row, c, C, csum);
}

// head, dz = 2 zscale (z - tz).  A row of 128-channel blocks for each output o:
// dWh[o][c] = sum_b dz[b][o] pooled[b][c], dbh[o] and sum (z - tz)^2; then one
// for each sample: dpool[b][c] = sum_o dz[b][o] Wh[o][c] / L.
__global__ void __launch_bounds__(128) k_head_grad(const float* __restrict__ z, const float* __restrict__ tz,
                                                   float zscale, const float* __restrict__ pooled,
                                                   const float* __restrict__ Wh, int B, int L, int C, int O,
                                                   float* __restrict__ dWh, float* __restrict__ dbh,
                                                   float* __restrict__ dpool, double* __restrict__ sum) {
  const int per = (C + 127) / 128, o = blockIdx.x / per, cb = blockIdx.x - o * per;
  const int c = cb * 128 + threadIdx.x;
  if (o >= O) {
    const long b = o - O;
    if (c >= C) return;
    float p = 0.f;
#pragma unroll 4
    for (int q = 0; q < O; ++q) p += 2.f * zscale * (z[b * O + q] - tz[b * O + q]) * Wh[(long)q * C + c];
    dpool[b * C + c] = p / L;
    return;
  }
  __shared__ float dz[128];
  float s = 0.f;
  for (int b0 = 0; b0 < B; b0 += 128) {
    const int nb = min(128, B - b0), b = b0 + threadIdx.x;
    __syncthreads();
    if ((int)threadIdx.x < nb) dz[threadIdx.x] = 2.f * zscale * (z[(long)b * O + o] - tz[(long)b * O + o]);
    __syncthreads();
    if (c < C) {
#pragma unroll 16
      for (int q = 0; q < nb; ++q) s += dz[q] * pooled[(long)(b0 + q) * C + c];
    }
  }
  if (c < C) dWh[(long)o * C + c] = s;
  if (cb == 0 && threadIdx.x < 32) {  // one warp per output
    double acc = 0.0;
    float t = 0.f;
    for (int b = threadIdx.x; b < B; b += 32) {
      const float r = z[(long)b * O + o] - tz[(long)b * O + o];
      acc += (double)r * r;
      t += 2.f * zscale * r;
    }
    for (int d = 16; d > 0; d >>= 1) {
      acc += __shfl_xor_sync(0xffffffffu, acc, d);
      t += __shfl_xor_sync(0xffffffffu, t, d);
    }
    if (threadIdx.x == 0) {
      dbh[o] = t;
      atomicAdd(sum, acc);
    }
  }
}

// bias gradients of the three layers (grid y): db[c] = sum of the tiles' sums;
// block of 32 channels x 8 groups of tiles
struct BiasSums {
  const float* csum[3];
  float* db[3];
  int C[3];
};
__global__ void __launch_bounds__(256) k_bias_sum(BiasSums a, int rows) {
  __shared__ float part[8][32];
  const int q = blockIdx.y, tx = threadIdx.x & 31, ty = threadIdx.x >> 5, c = blockIdx.x * 32 + tx, C = a.C[q];
  float s = 0.f;
  if (c < C) {
#pragma unroll 4
    for (int r = ty; r < rows; r += 8) s += a.csum[q][(long)r * C + c];
  }
  part[ty][tx] = s;
  __syncthreads();
  if (ty == 0 && c < C) {
    for (int u = 1; u < 8; ++u) s += part[u][tx];
    a.db[q][c] = s;
  }
}

__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, long n, float lr, float b1, float b2, float c1, float c2,
                       float eps, bf16* __restrict__ wb) {
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    m1[i] = b1 * m1[i] + (1.f - b1) * g[i];
    m2[i] = b2 * m2[i] + (1.f - b2) * g[i] * g[i];
    w[i] -= lr * (m1[i] / c1) / (sqrtf(m2[i] / c2) + eps);
    if (wb) wb[i] = __float2bfloat16(w[i]);
  }
}

int gs(long n) { return (int)std::min<long>((n + 255) / 256, 4096); }

}  // namespace

// ====================================================================== net object
struct opf_net {
  int Cin, H, L, O;
  // parameters (f32 master) in one block: W1 b1 W2 b2 W3 b3 Wh bh
  long off[8], count[8], total;
  float *P = nullptr, *G = nullptr, *M1 = nullptr, *M2 = nullptr;
  bf16* Pb = nullptr;  // bf16 copies of the weight matrices (same offsets)
  long step = 0;
  int Bcap = 0;
  // activations / workspace for batch capacity Bcap: im2col rows of the three
  // layer inputs, an output gradient by rows (ldz apart), im2col rows of the
  // transposed convolution for layers 2 and 3, padded and shifted weights
  bf16 *col[3] = {nullptr, nullptr, nullptr}, *dz = nullptr, *dzcol[2] = {nullptr, nullptr};
  bf16 *wp[3] = {nullptr, nullptr, nullptr}, *ws[2] = {nullptr, nullptr};
  float* gwork = nullptr;  // split-K partial sums of the weight-gradient GEMMs
  long gwork_floats = 0;
  float *pre1 = nullptr, *pre2 = nullptr, *y = nullptr, *dh = nullptr;
  float *pooled = nullptr, *dpool = nullptr, *z = nullptr, *csum = nullptr;
  double* sums = nullptr;  // the two loss sums, then the GEMMs' error flag
  double* read = nullptr;  // pinned host copy of sums and flag
  int* aug_idx = nullptr;    // minibatch rows of opf_net_gather_augment (device)
  float* aug_ang = nullptr;  // their shift / rotation phases
  int aug_cap = 0;
  cudaStream_t st = nullptr;
};

namespace {
int nfail(const std::string& m) {
  opf::set_last_error(m);
  return OPF_ECUDA;
}
#define NCU(call)                                                                    \
  do {                                                                               \
    cudaError_t e_ = (call);                                                         \
    if (e_ != cudaSuccess) return nfail(std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

long net_ldz(const opf_net* n) { return pad64(std::max(n->H, n->Cin)); }

int net_reserve(opf_net* n, int B) {
  if (B <= n->Bcap) return OPF_OK;
  n->Bcap = 0;
  for (void** p : {(void**)&n->col[0], (void**)&n->col[1], (void**)&n->col[2], (void**)&n->dz, (void**)&n->dzcol[0],
                   (void**)&n->dzcol[1],
                   (void**)&n->pre1, (void**)&n->pre2, (void**)&n->y, (void**)&n->dh, (void**)&n->pooled,
                   (void**)&n->dpool, (void**)&n->z, (void**)&n->csum}) {
    if (*p) cudaFree(*p);
    *p = nullptr;
  }
  const long BL = (long)B * n->L, W = std::max(n->H, n->Cin);
  const long BLp = pad128(BL), K1 = pad64(3L * n->Cin), K2 = pad64(3L * n->H), ldz = net_ldz(n);
  // the BF16 rows' padding is zero and stays so
  auto zeroed = [&](bf16** p, long count) {
    NCU(cudaMalloc(p, count * sizeof(bf16)));
    NCU(cudaMemsetAsync(*p, 0, count * sizeof(bf16), n->st));
    return (int)OPF_OK;
  };
  int rc;
  if ((rc = zeroed(&n->col[0], BLp * K1)) || (rc = zeroed(&n->col[1], BLp * K2)) ||
      (rc = zeroed(&n->col[2], BLp * K2)) || (rc = zeroed(&n->dz, BLp * ldz)) ||
      (rc = zeroed(&n->dzcol[0], BLp * K2)) || (rc = zeroed(&n->dzcol[1], BLp * K1)))
    return rc;
  NCU(cudaMalloc(&n->pre1, BL * n->H * sizeof(float)));
  NCU(cudaMalloc(&n->pre2, BL * n->H * sizeof(float)));
  NCU(cudaMalloc(&n->y, BL * n->Cin * sizeof(float)));
  NCU(cudaMalloc(&n->dh, BL * W * sizeof(float)));
  NCU(cudaMalloc(&n->pooled, (long)B * n->H * sizeof(float)));
  NCU(cudaMalloc(&n->dpool, (long)B * n->H * sizeof(float)));
  NCU(cudaMalloc(&n->z, (long)B * n->O * sizeof(float)));
  NCU(cudaMalloc(&n->csum, (BL + kGradRows - 1) / kGradRows * (n->Cin + 2L * n->H) * sizeof(float)));
  n->Bcap = B;
  return OPF_OK;
}

float* Pf(opf_net* n, int i) { return n->P + n->off[i]; }
float* Gf(opf_net* n, int i) { return n->G + n->off[i]; }
bf16* Pbf(opf_net* n, int i) { return n->Pb + n->off[i]; }

int* net_err(opf_net* n) { return (int*)(n->sums + 2); }

// C = A B^T on padded operands with the given epilogue
int gemm(opf_net* n, const bf16* A, const bf16* Bm, int M, int N, int Kp, const opf::TcEpilogue& e,
         int* splits = nullptr) {
  return opf::tc_gemm(A, Bm, M, N, (int)pad128(M), (int)pad128(N), Kp, e, net_err(n), n->st, n->gwork,
                      n->gwork_floats, splits);
}

// the epilogue of a hidden layer: bias, GELU, the next layer's im2col rows
opf::TcEpilogue hidden_epilogue(opf_net* n, const float* bias, float* pre, bf16* col) {
  opf::TcEpilogue e{};
  e.ldo = n->H;
  e.bias = bias;
  e.gelu = 1;
  e.pre_f32 = pre;
  e.col = col;
  e.C = n->H;
  e.L = n->L;
  e.ldc = pad64(3L * n->H);
  return e;
}

// padded copies of the weight matrices (after every parameter change)
void prepare_weights(opf_net* n) {
  const int Ci = n->Cin, H = n->H;
  const int rows[3] = {H, H, Ci}, cols[3] = {3 * Ci, 3 * H, 3 * H};
  for (int i = 0; i < 3; ++i) {
    const long Rp = pad128(rows[i]), Cp = pad64(cols[i]);
    k_pad<<<gs(Rp * Cp), 256, 0, n->st>>>(Pbf(n, 2 * i), rows[i], cols[i], n->wp[i], (int)Rp, (int)Cp);
  }
  // input-gradient weights of layers 3 (Cout = Cin, input H) and 2 (Cout = H, input H)
  k_wshift<<<gs(pad128(H) * pad64(3L * Ci)), 256, 0, n->st>>>(Pbf(n, 4), Ci, H, n->ws[1], (int)pad128(H),
                                                               (int)pad64(3L * Ci));
  k_wshift<<<gs(pad128(H) * pad64(3L * H)), 256, 0, n->st>>>(Pbf(n, 2), H, H, n->ws[0], (int)pad128(H),
                                                              (int)pad64(3L * H));
}

// forward for B samples whose features are at x (f32 [B][L][Cin]) into y and
// z; grad: the hidden layers' inputs to the GELU are kept for the gradients
int net_forward(opf_net* n, const float* x, int B, float* y, float* z, bool grad) {
  const int L = n->L, Ci = n->Cin, H = n->H, O = n->O;
  const long BL = (long)B * L, K1 = pad64(3L * Ci), K2 = pad64(3L * H);
  int rc;
  if (Ci % 8 == 0 && !((uintptr_t)x & 15))
    k_x_cols<true><<<dim3((unsigned)BL, (unsigned)((Ci / 8 + 127) / 128)), 128, 0, n->st>>>(x, L, Ci, n->col[0], K1);
  else
    k_x_cols<false><<<dim3((unsigned)BL, (unsigned)((Ci + 127) / 128)), 128, 0, n->st>>>(x, L, Ci, n->col[0], K1);
  // h1 = gelu(col(x) W1^T + b1), h2 likewise, y linear
  if ((rc = gemm(n, n->col[0], n->wp[0], (int)BL, H, (int)K1,
                 hidden_epilogue(n, Pf(n, 1), grad ? n->pre1 : nullptr, n->col[1]))))
    return rc;
  if ((rc = gemm(n, n->col[1], n->wp[1], (int)BL, H, (int)K2,
                 hidden_epilogue(n, Pf(n, 3), grad ? n->pre2 : nullptr, n->col[2]))))
    return rc;
  opf::TcEpilogue e{};
  e.ldo = Ci;
  e.bias = Pf(n, 5);
  e.out_f32 = y;
  if ((rc = gemm(n, n->col[2], n->wp[2], (int)BL, Ci, (int)K2, e))) return rc;
  k_pool_head<<<B, kPoolThreads, 0, n->st>>>(n->col[2], K2, L, H, O, Pf(n, 6), Pf(n, 7), n->pooled, z);
  return OPF_OK;
}

// loss and all parameter gradients into n->G for targets ty [B][L][Cin], tz [B][O]:
//   dW[o][k] = sum_m dZ[m][o] col[m][k],  db[o] = sum_m dZ[m][o],
//   dx[m][c] = sum_{j,o} dZ[(b, l + 1 - j)][o] W[o][j*Cin + c]
int net_gradients(opf_net* n, const float* x, const float* ty, const float* tz, int B, float lambda) {
  const int L = n->L, Ci = n->Cin, H = n->H, O = n->O;
  const long BL = (long)B * L, K1 = pad64(3L * Ci), K2 = pad64(3L * H), ldz = net_ldz(n);
  const int rows = (int)((BL + kGradRows - 1) / kGradRows);
  const float zscale = lambda / (float)(B * O);
  float *cs3 = n->csum, *cs2 = cs3 + (long)rows * Ci, *cs1 = cs2 + (long)rows * H;
  NCU(cudaMemsetAsync(n->sums, 0, 2 * sizeof(double), n->st));
  int rc = net_forward(n, x, B, n->y, n->z, true);
  if (rc) return rc;
  auto weights = [&](const bf16* col, long ldc, int Cin, int Cout, float* dW) {
    return opf::tc_gemm_columns(n->dz, ldz, col, ldc, Cout, 3 * Cin, (int)BL, dW, 3L * Cin, net_err(n), n->st,
                                n->gwork, n->gwork_floats);
  };
  // the gradient of the layer's input: dh, or split sums in the work space
  const float* dh = nullptr;
  int nsplit = 1;
  auto inputs = [&](const bf16* dzcol, const bf16* ws, int Cin, int Kd) {
    opf::TcEpilogue e{};
    e.ldo = Cin;
    e.out_f32 = n->dh;
    const int r = gemm(n, dzcol, ws, (int)BL, Cin, Kd, e, &nsplit);
    dh = nsplit > 1 ? n->gwork : n->dh;
    return r;
  };
  auto hidden = [&](const float* pre, bool head, bf16* dzcol, float* csum) {
    k_hidden_grad<<<(unsigned)grad_tiles(H) * rows, 256, 0, n->st>>>(
        dh, nsplit, pre, (int)BL, L, H, head ? n->dpool : nullptr, n->dz, ldz, dzcol, K2, csum);
  };
  // layer 3 (linear): dZ = dL/dy = 2 (y - ty) / (BL Ci); head: dL/dz = 2 lambda (z - tz) / (B O)
  k_out_grad<<<(unsigned)grad_tiles(Ci) * rows, 256, 0, n->st>>>(
      n->y, ty, (int)BL, L, Ci, 1.f / (float)(BL * Ci), n->dz, ldz, n->dzcol[1], K1, cs3, n->sums);
  k_head_grad<<<(unsigned)((H + 127) / 128) * (unsigned)(O + B), 128, 0, n->st>>>(
      n->z, tz, zscale, n->pooled, Pf(n, 6), B, L, H, O, Gf(n, 6), Gf(n, 7), n->dpool, n->sums + 1);
  if ((rc = weights(n->col[2], K2, H, Ci, Gf(n, 4)))) return rc;
  if ((rc = inputs(n->dzcol[1], n->ws[1], H, (int)K1))) return rc;
  // layer 2
  hidden(n->pre2, true, n->dzcol[0], cs2);
  if ((rc = weights(n->col[1], K2, H, H, Gf(n, 2)))) return rc;
  if ((rc = inputs(n->dzcol[0], n->ws[0], H, (int)K2))) return rc;
  // layer 1 (input gradient not needed)
  hidden(n->pre1, false, nullptr, cs1);
  if ((rc = weights(n->col[0], K1, Ci, H, Gf(n, 0)))) return rc;
  const BiasSums bs{{cs3, cs2, cs1}, {Gf(n, 5), Gf(n, 3), Gf(n, 1)}, {Ci, H, H}};
  k_bias_sum<<<dim3((unsigned)((std::max(Ci, H) + 31) / 32), 3), 256, 0, n->st>>>(bs, rows);
  NCU(cudaGetLastError());
  return OPF_OK;
}

// Minibatch gather with the pipe-flow symmetries applied (training-data
// augmentation): sample b is row idx[b] of the device-resident set, its
// complex channel (component, axial index kidx, azimuthal m) turned by
// e^{i (ang[2b] k + ang[2b+1] m)}, k = kidx - (nkf - 1)/2 -- an axial shift
// (ang[2b] = alpha a) and an azimuthal rotation (ang[2b+1] = m_p phi).  The
// head targets are gathered unchanged (period and shift are invariant).
__global__ void k_gather_augment(const float2* __restrict__ x, const float2* __restrict__ y,
                                 const float* __restrict__ z, const int* __restrict__ idx,
                                 const float* __restrict__ ang, int B, int L, int ncomp, int nkf, int mf, int nz,
                                 float2* __restrict__ bx, float2* __restrict__ by, float* __restrict__ bz) {
  const long C = (long)ncomp * nkf * mf;
  const long total = (long)B * L * C;
  const long stride = (long)gridDim.x * blockDim.x;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < total; t += stride) {
    const long ch = t % C, bl = t / C;
    const int l = (int)(bl % L), b = (int)(bl / L);
    const int m = (int)(ch % mf), kidx = (int)((ch / mf) % nkf);
    const float ph = ang[2 * b] * (float)(kidx - (nkf - 1) / 2) + ang[2 * b + 1] * (float)m;
    float sn, cs;
    sincosf(ph, &sn, &cs);
    const long src = ((long)idx[b] * L + l) * C + ch, dst = ((long)b * L + l) * C + ch;
    const float2 xv = x[src], yv = y[src];
    bx[dst] = make_float2(xv.x * cs - xv.y * sn, xv.x * sn + xv.y * cs);
    by[dst] = make_float2(yv.x * cs - yv.y * sn, yv.x * sn + yv.y * cs);
  }
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < (long)B * nz; t += stride)
    bz[t] = z[(long)idx[t / nz] * nz + t % nz];
}

void refresh_bf16(opf_net* n) {
  k_to_bf16<<<gs(n->total), 256, 0, n->st>>>(n->P, n->Pb, n->total);
  prepare_weights(n);
}

}  // namespace

extern "C" {

opf_net_t* opf_net_create(int cin, int hidden, int L, int nout, unsigned long long seed) {
  if (cin < 1 || hidden < 1 || L < 1 || nout < 1) {
    opf::set_last_error("opf_net_create: sizes must be positive");
    return nullptr;
  }
  opf_net* n = new opf_net();
  n->Cin = cin;
  n->H = hidden;
  n->L = L;
  n->O = nout;
  const long cnt[8] = {(long)hidden * 3 * cin, hidden, (long)hidden * 3 * hidden, hidden,
                       (long)cin * 3 * hidden, cin, (long)nout * hidden, nout};
  long t = 0;
  for (int i = 0; i < 8; ++i) {
    n->off[i] = t;
    n->count[i] = cnt[i];
    t += (cnt[i] + 63) / 64 * 64;
  }
  n->total = t;
  // deterministic init: uniform(-a, a), a = 1/sqrt(fan_in), biases 0
  std::vector<float> h(t, 0.f);
  unsigned long long z = seed;
  auto next = [&]() {
    z += 0x9E3779B97F4A7C15ull;
    unsigned long long q = z;
    q = (q ^ (q >> 30)) * 0xBF58476D1CE4E5B9ull;
    q = (q ^ (q >> 27)) * 0x94D049BB133111EBull;
    q ^= q >> 31;
    return (double)(q >> 11) * (1.0 / 9007199254740992.0);
  };
  const long fan[8] = {3L * cin, 0, 3L * hidden, 0, 3L * hidden, 0, hidden, 0};
  for (int i = 0; i < 8; i += 2) {
    const double a = 1.0 / std::sqrt((double)fan[i]);
    for (long j = 0; j < cnt[i]; ++j) h[n->off[i] + j] = (float)((2.0 * next() - 1.0) * a);
  }
  if (cudaStreamCreateWithFlags(&n->st, cudaStreamNonBlocking) != cudaSuccess ||
      cudaMalloc(&n->P, t * sizeof(float)) != cudaSuccess || cudaMalloc(&n->G, t * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->M1, t * sizeof(float)) != cudaSuccess || cudaMalloc(&n->M2, t * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->Pb, t * sizeof(bf16)) != cudaSuccess ||
      cudaMalloc(&n->wp[0], pad128(hidden) * pad64(3L * cin) * sizeof(bf16)) != cudaSuccess ||
      cudaMalloc(&n->wp[1], pad128(hidden) * pad64(3L * hidden) * sizeof(bf16)) != cudaSuccess ||
      cudaMalloc(&n->wp[2], pad128(cin) * pad64(3L * hidden) * sizeof(bf16)) != cudaSuccess ||
      cudaMalloc(&n->ws[0], pad128(hidden) * pad64(3L * hidden) * sizeof(bf16)) != cudaSuccess ||
      cudaMalloc(&n->ws[1], pad128(hidden) * pad64(3L * cin) * sizeof(bf16)) != cudaSuccess ||
      cudaMalloc(&n->sums, 3 * sizeof(double)) != cudaSuccess ||
      cudaMallocHost(&n->read, 3 * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&n->gwork, (n->gwork_floats = 8L * std::max(3L * hidden * std::max(cin, hidden), 1L)) *
                                sizeof(float)) != cudaSuccess) {
    opf::set_last_error("opf_net_create: device allocation failed");
    opf_net_destroy(n);
    return nullptr;
  }
  cudaMemcpy(n->P, h.data(), t * sizeof(float), cudaMemcpyHostToDevice);
  cudaMemset(n->G, 0, t * sizeof(float));
  cudaMemset(n->M1, 0, t * sizeof(float));
  cudaMemset(n->M2, 0, t * sizeof(float));
  cudaMemset(n->sums, 0, 3 * sizeof(double));
  refresh_bf16(n);
  if (cudaStreamSynchronize(n->st) != cudaSuccess) {
    opf::set_last_error("opf_net_create: initialisation failed");
    opf_net_destroy(n);
    return nullptr;
  }
  return n;
}

void opf_net_destroy(opf_net_t* n) {
  if (!n) return;
  if (n->st) cudaStreamSynchronize(n->st);
  for (void* p : {(void*)n->P, (void*)n->G, (void*)n->M1, (void*)n->M2, (void*)n->Pb, (void*)n->pre1,
                  (void*)n->pre2, (void*)n->y, (void*)n->dh, (void*)n->pooled, (void*)n->dpool, (void*)n->z, (void*)n->csum,
                  (void*)n->sums, (void*)n->col[0], (void*)n->col[1], (void*)n->col[2], (void*)n->dz,
                  (void*)n->dzcol[0], (void*)n->dzcol[1], (void*)n->wp[0], (void*)n->wp[1], (void*)n->wp[2], (void*)n->ws[0],
                  (void*)n->ws[1], (void*)n->gwork, (void*)n->aug_idx, (void*)n->aug_ang})
    if (p) cudaFree(p);
  if (n->read) cudaFreeHost(n->read);
  if (n->st) cudaStreamDestroy(n->st);
  delete n;
}

int opf_net_param_count(opf_net_t* n, long* total, long* sizes8) {
  if (!n || !total) return OPF_EINVAL;
  long s = 0;
  for (int i = 0; i < 8; ++i) {
    s += n->count[i];
    if (sizes8) sizes8[i] = n->count[i];
  }
  *total = s;
  return OPF_OK;
}

int opf_net_get_params(opf_net_t* n, float* host, int grads) {
  if (!n || !host) return OPF_EINVAL;
  // straight into the caller's buffer, one copy per run of arrays that follow
  // one another without padding (a staging copy and a loop over its elements
  // took 0.7 ms of the 2.1 M parameters, this 0.06 ms into touched pages)
  const float* src = grads ? n->G : n->P;
  for (int i = 0; i < 8;) {
    const long first = n->off[i];
    long count = n->count[i++];
    while (i < 8 && n->off[i] == first + count) count += n->count[i++];
    NCU(cudaMemcpy(host, src + first, count * sizeof(float), cudaMemcpyDeviceToHost));
    host += count;
  }
  return OPF_OK;
}

int opf_net_set_params(opf_net_t* n, const float* host) {
  if (!n || !host) return OPF_EINVAL;
  std::vector<float> h(n->total, 0.f);
  long o = 0;
  for (int i = 0; i < 8; ++i)
    for (long j = 0; j < n->count[i]; ++j) h[n->off[i] + j] = host[o++];
  NCU(cudaMemcpy(n->P, h.data(), n->total * sizeof(float), cudaMemcpyHostToDevice));
  refresh_bf16(n);
  NCU(cudaStreamSynchronize(n->st));
  return OPF_OK;
}

// Waits for the stream with the loss sums and the error flag in n->read; a
// tensor-core GEMM whose bounded wait ran out leaves the flag set.
static int net_finish(opf_net_t* n) {
  NCU(cudaMemcpyAsync(n->read, n->sums, 3 * sizeof(double), cudaMemcpyDeviceToHost, n->st));
  NCU(cudaStreamSynchronize(n->st));
  NCU(cudaGetLastError());
  int h;
  std::memcpy(&h, n->read + 2, sizeof h);
  if (h) {
    cudaMemset(net_err(n), 0, sizeof(int));
    opf::set_last_error("proposal network: a tensor-core GEMM timed out waiting for its operands");
    return OPF_ETIMEOUT;
  }
  return OPF_OK;
}

int opf_net_forward(opf_net_t* n, const float* d_x, int B, float* d_y, float* d_z) {
  if (!n || !d_x || B < 1) return OPF_EINVAL;
  int rc = net_reserve(n, B);
  if (rc) return rc;
  rc = net_forward(n, d_x, B, d_y ? d_y : n->y, d_z ? d_z : n->z, false);
  if (rc) return rc;
  return net_finish(n);
}

int opf_net_gradients(opf_net_t* n, const float* d_x, const float* d_ty, const float* d_tz, int B,
                      float lambda, double* loss) {
  if (!n || !d_x || !d_ty || !d_tz || B < 1) return OPF_EINVAL;
  int rc = net_reserve(n, B);
  if (rc) return rc;
  rc = net_gradients(n, d_x, d_ty, d_tz, B, lambda);
  if (rc) return rc;
  rc = net_finish(n);
  if (rc) return rc;
  if (loss) *loss = n->read[0] / (double)((long)B * n->L * n->Cin) + lambda * n->read[1] / (double)(B * n->O);
  return OPF_OK;
}

int opf_net_train_step(opf_net_t* n, const float* d_x, const float* d_ty, const float* d_tz, int B,
                       float lambda, float lr, double* loss) {
  int rc = opf_net_gradients(n, d_x, d_ty, d_tz, B, lambda, loss);
  if (rc) return rc;
  n->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)n->step), c2 = 1.f - std::pow(b2, (float)n->step);
  k_adam<<<gs(n->total), 256, 0, n->st>>>(n->P, n->G, n->M1, n->M2, n->total, lr, b1, b2, c1, c2, 1e-8f, n->Pb);
  prepare_weights(n);
  NCU(cudaStreamSynchronize(n->st));
  NCU(cudaGetLastError());
  return OPF_OK;
}

int opf_net_gather_augment(opf_net_t* n, int B, int L, int ncomp, int nkf, int mf, int nz, const float* d_x,
                           const float* d_y, const float* d_z, long rows, const int* idx, const float* ang,
                           float* d_bx, float* d_by, float* d_bz) {
  if (!n || B < 1 || L < 1 || ncomp < 1 || nkf < 1 || mf < 1 || nz < 1 || rows < 1 || !d_x || !d_y || !d_z ||
      !idx || !ang || !d_bx || !d_by || !d_bz) {
    opf::set_last_error("opf_net_gather_augment: bad arguments");
    return OPF_EINVAL;
  }
  for (int b = 0; b < B; ++b)
    if (idx[b] < 0 || idx[b] >= rows) {
      opf::set_last_error("opf_net_gather_augment: sample index out of range");
      return OPF_EINVAL;
    }
  if (n->aug_cap < B) {
    if (n->aug_idx) cudaFree(n->aug_idx);
    if (n->aug_ang) cudaFree(n->aug_ang);
    n->aug_idx = nullptr;
    n->aug_ang = nullptr;
    n->aug_cap = 0;
    NCU(cudaMalloc((void**)&n->aug_idx, (size_t)B * sizeof(int)));
    NCU(cudaMalloc((void**)&n->aug_ang, (size_t)2 * B * sizeof(float)));
    n->aug_cap = B;
  }
  NCU(cudaMemcpyAsync(n->aug_idx, idx, (size_t)B * sizeof(int), cudaMemcpyHostToDevice, n->st));
  NCU(cudaMemcpyAsync(n->aug_ang, ang, (size_t)2 * B * sizeof(float), cudaMemcpyHostToDevice, n->st));
  const long total = (long)B * L * ncomp * nkf * mf;
  k_gather_augment<<<gs(total), 256, 0, n->st>>>((const float2*)d_x, (const float2*)d_y, d_z, n->aug_idx,
                                                 n->aug_ang, B, L, ncomp, nkf, mf, nz, (float2*)d_bx,
                                                 (float2*)d_by, d_bz);
  NCU(cudaGetLastError());
  return OPF_OK;
}

}  // extern "C"
