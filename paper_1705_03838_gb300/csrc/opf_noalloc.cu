// opf_nonlinear_noalloc: the nonlinear-term evaluation of opf_nonlinear with
// every intermediate placed in one file-scope device array instead of
// memory from cudaMalloc.
//
// Who needs it: callers that must not allocate device memory at the point of
// the call -- a serving process whose device memory is entirely handed out
// by its own pool, code that may not trigger the device-wide synchronisation
// cudaMalloc/cudaFree can cause, or a loop that forbids allocation after
// start-up.  They pass device input and output buffers; everything else
// lives in g_noalloc_scratch below.
//
// Limits and sharing:
//  * g_noalloc_scratch holds kNoallocScratchBytes (16 MiB) on every GPU that
//    loads the library, for the life of the process.  Sizes whose working set
//    does not fit are rejected with OPF_EINVAL before any launch.
//  * All calls share the array and it keeps the last call's contents.  Every
//    region is fully written before it is read within a call, so nothing has
//    to start at zero.  Calls whose GPU work overlaps (different streams or
//    threads without ordering) race on the array.
//  * The first call on a device looks up the array's device address there
//    (cudaGetSymbolAddress) and sets the kernels' shared-memory limits; make
//    that first call before any stream capture.  CUDA loads modules lazily,
//    so it is also that first call (not loading the library) that places the
//    16 MiB array and the kernels' code on the device: make it at start-up,
//    before the caller's own pool takes the device memory.
//  * The call waits for its result (it synchronises the stream) before it
//    returns, so it refuses, with OPF_EINVAL and before launching anything,
//    a stream that is being captured.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include "opf_dft.cuh"
#include "opf_internal.h"

namespace {

constexpr size_t kNoallocScratchBytes = 16u << 20;
constexpr int kMaxDevices = 64;

// Scratch for the no-allocation entry point.  In host code this name is only
// a stand-in for the symbol; kernels get the device address looked up below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

void* g_scratch_addr[kMaxDevices] = {nullptr};

// Transform lengths (3K, 3M) whose kernels already have their shared-memory
// limit raised, per device, in a fixed table (no host allocation either); the
// attributes are set once per device and shape (every call, once the table
// is full).
constexpr int kAttrSlots = 32;
std::mutex g_attr_mutex;
long g_attr_done[kMaxDevices][kAttrSlots] = {};
int g_attr_count[kMaxDevices] = {};

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

bool smooth235(int n) {
  for (int p : {2, 3, 5})
    while (n % p == 0) n /= p;
  return n == 1;
}

// Radial points, 9-point first-derivative stencils for both axis parities
// (same points and folding as the handle's setup) and the z / theta twiddle
// tables, computed on the device into the scratch.  One thread per weight:
// with a_i = prod_(j != i) (x_i - x_j), the weight of node i at node c is
// a_c / (a_i (x_c - x_i)), that of c itself sum_(j != c) 1 / (x_c - x_j).  A
// block's rows are two tiles of the curl's digit table, which it fills in.  (A
// thread per row running a recursion over the nodes took 101 us at N = 32 on
// chains of divisions, more than the rest of the call.)
constexpr int kConstRows = 16;                   // radial rows per block
constexpr int kConstThreads = kConstRows * 9;    // a thread per (row, node)
__global__ void __launch_bounds__(kConstThreads)
    k_noalloc_consts(int N, int nz, int nth, double Re, double* prm, double* d1, double* rinv, double2* twz,
                     double2* twth, uint2* tab, int* ew) {
  __shared__ double xs[kConstRows + 16], as[kConstRows][9], ws[kConstRows][9], inv[kConstRows][9];
  const int tiles = opf::stencil_tiles(N), n0 = blockIdx.x * kConstRows - (8 * tiles - N);
  if (n0 >= N) {  // blocks behind the rows': the twiddles
    int t = (blockIdx.x - (tiles + 1) / 2) * blockDim.x + threadIdx.x;
    if (t < opf::kPrmCount) prm[t] = t == opf::kPrmRe ? Re : 0.0;
    const int n = t < nz ? nz : nth;
    double2* tw = t < nz ? twz : twth;
    t = t < nz ? t : t - nz;
    if (t < n) {
      double s, c;
      sincospi(2.0 * t / n, &s, &c);
      tw[t] = double2{c, s};
    }
    return;
  }
  // extended nodes e0, e0 + 1, .. of the block's rows: e < N is -r_(N-1-e)
  const int e0 = min(N + max(n0, 0) - 4, 2 * N - 9);
  auto rad = [&](int j) { return j == N - 1 ? 1.0 : cospi((double)(N - 1 - j) / (2.0 * N - 1.0)); };
  if (threadIdx.x < kConstRows + 8 && e0 + (int)threadIdx.x < 2 * N) {
    const int e = e0 + threadIdx.x;
    xs[threadIdx.x] = e < N ? -rad(N - 1 - e) : rad(e - N);
  }
  __syncthreads();
  const int row = threadIdx.x / 9, u = threadIdx.x - row * 9, n = n0 + row;
  const bool in = n >= 0 && n < N;
  const int first = min(N + n - 4, 2 * N - 9);  // this row's first node
  const double* x = xs + (in ? first - e0 : 0);
  const int c = in ? N + n - first : 0;
  if (in) {
    double a = 1.0;
    for (int j = 0; j < 9; ++j)
      if (j != u) a *= x[u] - x[j];
    as[row][u] = a;
    if (u == 0) rinv[n] = 1.0 / rad(n);
  }
  __syncthreads();
  if (in && u != c) {
    const double dist = x[c] - x[u];
    ws[row][u] = as[row][c] / (as[row][u] * dist);
    inv[row][u] = 1.0 / dist;
  }
  __syncthreads();
  if (in && u == c) {
    double s = 0.0;
    for (int j = 0; j < 9; ++j)
      if (j != c) s += inv[row][j];
    ws[row][c] = s;
  }
  __syncthreads();
  // slot u of the row's columns lo .. lo + 8: the real node there, plus the
  // ghost that folds onto it
  if (in) {
    const int lo = min(max(n - 4, 0), N - 9), col = lo + u;
    double even = 0.0, odd = 0.0;
    const int real = N + col - first, ghost = N - 1 - col - first;
    if (real >= 0 && real < 9) even = odd = ws[row][real];
    if (ghost >= 0 && ghost < 9) {
      even += ws[row][ghost];
      odd -= ws[row][ghost];
    }
    d1[(0 * N + n) * 9 + u] = even;
    d1[(1 * N + n) * 9 + u] = odd;
  }
  __syncthreads();  // (the tiles' weights are this block's own)
  const int tile = blockIdx.x * 2 + (threadIdx.x >> 6), par = (threadIdx.x >> 5) & 1;
  if (threadIdx.x < 128 && tile < tiles)
    opf::stencil_entry((par * tiles + tile) * 32 + (threadIdx.x & 31), d1, N, tab, ew);
}

int fail(int code, const std::string& m) {
  opf::set_last_error(m);  // reported by opf_last_error()
  return code;
}

}  // namespace

extern "C" int opf_nonlinear_noalloc(int N, int K, int M, int m_p, double alpha, double Re,
                                     const double* d_state, double* d_out, void* stream) {
  if (N < 9 || K < 1 || M < 1 || m_p < 1 || !(alpha > 0) || !(Re > 0))
    return fail(OPF_EINVAL, "opf_nonlinear_noalloc: need N>=9, K>=1, M>=1, m_p>=1, alpha>0, Re>0");
  if (!d_state || !d_out) return fail(OPF_EINVAL, "opf_nonlinear_noalloc: NULL buffer");
  if (!smooth235(3 * K) || !smooth235(3 * M))
    return fail(OPF_EINVAL, "opf_nonlinear_noalloc: 3K and 3M must have no prime factor other than 2, 3, 5");
  opf::Dims d{};
  d.N = N;
  d.K = K;
  d.M = M;
  d.m_p = m_p;
  d.nk = 2 * K - 1;
  d.nz = 3 * K;
  d.nth = 3 * M;
  d.inv_grid = 1.0 / ((double)d.nz * d.nth);
  d.alpha = alpha;
  d.Re = Re;
  d.dt = 1.0;
  d.F = (long)M * N * d.nk;
  opf::choose_chunks(&d);
  opf::FftPlan pz{}, pth{};
  if (!opf::make_plan(d.nz, &pz) || !opf::make_plan(d.nth, &pth))
    return fail(OPF_EINVAL, "opf_nonlinear_noalloc: no FFT plan for 3K or 3M");

  // scratch layout: constants | U (3F) | W6 (6F) | Z6 (6P) | ZN (3P) | N (3F)
  const size_t F16 = (size_t)d.F * sizeof(double2);
  const size_t P16 = (size_t)N * d.nz * M * sizeof(double2);
  const size_t o_prm = 0;
  const size_t o_d1 = align256(o_prm + opf::kPrmCount * sizeof(double));
  const size_t o_rinv = align256(o_d1 + 2 * (size_t)N * 9 * sizeof(double));
  const size_t o_twz = align256(o_rinv + N * sizeof(double));
  const size_t o_twth = align256(o_twz + d.nz * sizeof(double2));
  const size_t o_U = align256(o_twth + d.nth * sizeof(double2));
  const size_t o_W6 = align256(o_U + 3 * F16);
  const size_t o_Z6 = align256(o_W6 + 6 * F16);
  const size_t o_ZN = align256(o_Z6 + 6 * P16);
  const size_t o_N = align256(o_ZN + 3 * P16);
  const size_t need = align256(o_N + 3 * F16);
  if (need > kNoallocScratchBytes)
    return fail(OPF_EINVAL, "opf_nonlinear_noalloc: resolution needs " + std::to_string(need) +
                                " bytes of scratch, more than the fixed " +
                                std::to_string(kNoallocScratchBytes));

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return fail(OPF_ECUDA, "opf_nonlinear_noalloc: no usable CUDA device");
  cudaStream_t st = (cudaStream_t)stream;
  {  // the call ends with a stream synchronisation, which a capture forbids
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
      if (e != cudaSuccess) cudaGetLastError();  // leave no sticky status behind
      return fail(OPF_EINVAL, "opf_nonlinear_noalloc: the stream is being captured (or its capture state "
                              "cannot be read); this call synchronises its stream and cannot run inside a capture");
    }
  }
  // (on every call: what the transforms need is checked once per pair of lengths)
  if (!opf::nonlinear_radial_fits(d))
    return fail(OPF_EINVAL, "opf_nonlinear_noalloc: resolution needs more shared memory than a block has");
  if (!g_scratch_addr[dev]) {  // once per device, with that device current
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return fail(OPF_ECUDA, std::string("opf_nonlinear_noalloc: cudaGetSymbolAddress: ") +
                                 cudaGetErrorString(e));
    g_scratch_addr[dev] = p;
  }
  {
    const long key = (long)d.nz << 20 | d.nth;
    std::lock_guard<std::mutex> lock(g_attr_mutex);
    long* done = g_attr_done[dev];
    int& count = g_attr_count[dev];
    if (std::find(done, done + count, key) == done + count) {
      if (!opf::prepare_nonlinear_attrs(d))
        return fail(OPF_EINVAL, "opf_nonlinear_noalloc: resolution needs more shared memory than a block has");
      if (count < kAttrSlots) done[count++] = key;
    }
  }
  unsigned char* base = (unsigned char*)g_scratch_addr[dev];
  opf::DevSetup s{};
  s.prm = (double*)(base + o_prm);
  d.prm = s.prm;
  s.d1 = (double*)(base + o_d1);
  s.rinv = (double*)(base + o_rinv);
  s.tw_z = (double2*)(base + o_twz);
  s.tw_th = (double2*)(base + o_twth);
  double2* U = (double2*)(base + o_U);
  double2* W6 = (double2*)(base + o_W6);
  double2* Z6 = (double2*)(base + o_Z6);
  double2* ZN = (double2*)(base + o_ZN);
  double2* Nn = (double2*)(base + o_N);

  // the curl's digit table: behind the other regions, or in the half-physical
  // fields', which are not in use yet, where the scratch ends before
  s.stab = need + opf::stencil_bytes(N) <= kNoallocScratchBytes ? base + need : base + o_Z6;
  const opf::StencilTable stab = opf::stencil_at(s.stab, s.d1, N);
  const int nb = (stab.tiles + 1) / 2 + (d.nz + d.nth + kConstThreads - 1) / kConstThreads;
  k_noalloc_consts<<<nb, kConstThreads, 0, st>>>(N, d.nz, d.nth, Re, s.prm, s.d1, s.rinv, s.tw_z, s.tw_th,
                                                 (uint2*)stab.tab, (int*)stab.ew);
  opf::launch_abi_to_internal(d, (const double2*)d_state, U, st);
  opf::launch_curl(d, s, U, W6, st);
  // the transforms' tables: behind the other regions (over the curl's), or over U, which the
  // curl has read, where the scratch ends before (a working set that fills it
  // has a U of a megabyte and more)
  unsigned char* tab = need + opf::dft_table_bytes(K, M) <= kNoallocScratchBytes ? base + need : base + o_U;
  opf::dft_device_tables(K, M, d.inv_grid, s.tw_z, s.tw_th, tab, &s.dft, st);
  opf::launch_zsynth(d, s, pz, W6, Z6, st);
  opf::launch_product(d, s, pth, Z6, ZN, st);
  opf::launch_zanalysis(d, s, pz, ZN, Nn, st);
  opf::launch_internal_to_abi(d, Nn, (double2*)d_out, 1, st);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess)
    return fail(OPF_ECUDA, std::string("opf_nonlinear_noalloc: ") + cudaGetErrorString(e));
  return OPF_OK;
}
