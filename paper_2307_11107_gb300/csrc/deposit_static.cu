// apic_deposit_static: the cloud-in-cell charge deposit with its 64-bit
// fixed-point accumulator in library-owned static device memory, for callers
// that cannot allocate device memory themselves.
//
// Some callers cannot call cudaMalloc where they need a density: a component
// that runs under a device-memory budget owned by another part of the
// program, a host framework that only hands out the buffers it manages, or a
// latency-critical loop that must not enter the allocator.  This entry point
// takes the caller's particle positions, node volumes and output array and
// needs no other device memory: its scratch is the file-scope array below,
// which every GPU that loads the library keeps until the process exits
// (8 MiB per device).  The first call on a device looks up the array's device
// address; make that first call before any stream capture.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "../../include/apic.h"

namespace {

#include "cell_fixed.cuh"

constexpr long long kStaticNodes = 1ll << 20;  // node capacity of the static accumulator
constexpr int kMaxDevices = 64;
constexpr int kWindowBytes = 48 * 1024;  // shared-memory window of the outermost rows (no opt-in needed)
constexpr int kMaxCopies = 64;  // copies of a small grid's accumulator in the static array at most

// Shared by every call on a device: calls that overlap on the GPU race on it.
__device__ __align__(256) unsigned long long g_static_acc[kStaticNodes];

std::mutex g_mu;
void* g_acc_ptr[kMaxDevices] = {};

// Device address of the static accumulator on the current device, looked up
// once per device (host code cannot use the symbol's name as an address).
cudaError_t static_acc(unsigned long long** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_acc_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_acc);
    if (e != cudaSuccess) return e;
    g_acc_ptr[dev] = p;
  }
  *out = (unsigned long long*)g_acc_ptr[dev];
  return cudaSuccess;
}

// SMs of the current device, looked up once per device.
int sm_count() {
  static int n[kMaxDevices] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  std::lock_guard<std::mutex> lk(g_mu);
  if (n[dev] == 0 && cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n[dev] = 0;
  return n[dev];
}

__global__ void k_clear(unsigned long long* acc, long long nodes) {
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < nodes;
       k += (long long)gridDim.x * blockDim.x)
    acc[k] = 0ull;
}

// Bits of a coordinate inside [lo, hi] (both negative, lo <= hi): the range
// test of a negative double on its bit pattern, whose order is that of the
// magnitudes (a NaN's exceeds every number's; positive ones lie below).
__device__ __forceinline__ bool in_negative(double v, unsigned long long hi_bits, unsigned long long lo_bits) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return b >= hi_bits && b <= lo_bits;
}

// Bilinear (cloud-in-cell) weights of each particle in the logical (x1, x2)
// grid, rounded to F fractional bits and added with 64-bit integer atomics
// (order-independent sums) to the CTA's copy of the accumulator.  A particle
// outside [-1, x1_outer] x [-1, 1], or with a non-finite coordinate, carries no
// charge onto the grid (as a freed or escaped slot of a simulation does) and
// is skipped.
//
// Bound: the atomics.  The particles per unit of x1 grow as r^4 (Eq. 5), so a
// plasma puts most of them into the outermost rows (uniform in volume between
// the grain and 20 R0, 512 rows: a tenth in the last one, 84 % in the last
// 23), and additions to one address follow one another at L2.  So the CTAs
// write to several copies of the accumulator, and, with enough particles
// (kWin), to a shared-memory window over the last `rows` node rows, flushed at
// the end, by 32-bit atomics (the low word passes its carry; 64-bit ones cost
// three times as much).  1e7 such particles on 512 x 256 cells: 0.88 ms with
// one copy, 0.81 with the weights in integer arithmetic (cell_fixed.cuh),
// 0.31 with seven copies too, 0.13 with the window; on 1000 x 500 cells
// (where the static array holds two copies) 0.32 and 0.24; spread evenly over
// 512 x 256 cells, where the window catches a twentieth, 0.20 and 0.22.
__device__ __forceinline__ void add_lo_hi(unsigned long long* s, unsigned long long v) {
  unsigned* p = (unsigned*)s;
  const unsigned lo = (unsigned)v, old = atomicAdd(p, lo);
  const unsigned hi = (unsigned)(v >> 32) + (old + lo < old ? 1u : 0u);
  if (hi) atomicAdd(p + 1, hi);
}

template <bool kWin>
__global__ void __launch_bounds__(kWin ? 1024 : 256) k_weigh(unsigned long long* acc, const double* x1,
                                                              const double* x2, long long n, int n1, int n2,
                                                              unsigned long long out_bits, double s1, double s2, int b,
                                                              int F, int copies, int nodes, int rows) {
  extern __shared__ unsigned long long s_acc[];  // kWin: [rows * N2], node rows n1 + 1 - rows .. n1
  const int N2 = n2 + 1;
  const unsigned long long one_bits = 0x3ff0000000000000ull, neg_one = one_bits | 1ull << 63;
  acc += (long long)(blockIdx.x % copies) * nodes;
  const int w0 = nodes - rows * N2;  // first node of the window
  if (kWin) {
    for (int e = threadIdx.x; e < rows * N2; e += blockDim.x) s_acc[e] = 0ull;
    __syncthreads();
  }
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x) {
    const double a = x1[k], c = x2[k];
    if (!in_negative(a, out_bits, neg_one)) continue;
    if (((unsigned long long)__double_as_longlong(c) & ~(1ull << 63)) > one_bits) continue;  // |x2| > 1, NaN
    unsigned long long f1, f2;
    const int i = cell_fixed(a, s1, n1, b, f1), j = cell_fixed(c, s2, n2, b, f2);
    const W4 w = weights_fixed(f1, f2, b, F);
    const int m = i * N2 + j;
    if (kWin && m >= w0) {
      unsigned long long* p = s_acc + (m - w0);
      add_lo_hi(p, w.w00);
      add_lo_hi(p + N2, w.w10);
      add_lo_hi(p + 1, w.w01);
      add_lo_hi(p + N2 + 1, w.w11);
    } else {
      unsigned long long* p = acc + m;
      atomicAdd(p, w.w00);
      atomicAdd(p + N2, w.w10);
      atomicAdd(p + 1, w.w01);
      atomicAdd(p + N2 + 1, w.w11);
    }
  }
  if (kWin) {
    __syncthreads();
    for (int e = threadIdx.x; e < rows * N2; e += blockDim.x) {
      const unsigned long long v = s_acc[e];
      if (v) atomicAdd(acc + w0 + e, v);
    }
  }
}

__global__ void __launch_bounds__(256) k_density(const unsigned long long* acc, const double* V, double* rho,
                                                 long long nodes, int copies, double scale) {
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < nodes;
       k += (long long)gridDim.x * blockDim.x) {
    unsigned long long q = 0;
#pragma unroll 4
    for (int c = 0; c < copies; ++c) q += acc[c * nodes + k];
    rho[k] = scale * (double)q / V[k];
  }
}

}  // namespace

extern "C" int apic_deposit_static(const apic_grid_t* grid, const double* x1, const double* x2, int64_t n,
                                   double qw, const double* volume, double* rho, void* stream) {
  if (!grid || !volume || !rho || n < 0 || (n > 0 && (!x1 || !x2))) return APIC_ERR_INVALID_ARG;
  if (grid->n1 < 1 || grid->n2 < 1 || !(grid->x1_outer > -1.0 && grid->x1_outer < 0.0)) return APIC_ERR_INVALID_ARG;
  long long nodes = (long long)(grid->n1 + 1) * (grid->n2 + 1);
  if (nodes > kStaticNodes) return APIC_ERR_INVALID_ARG;  // larger than the static scratch
  if (n >= (1ll << 40)) return APIC_ERR_INVALID_ARG;
  unsigned long long* acc = nullptr;
  if (static_acc(&acc) != cudaSuccess) return APIC_ERR_CUDA;
  cudaStream_t s = (cudaStream_t)stream;
  int bits = 0;
  for (long long v = n; v > 0; v >>= 1) ++bits;
  int F = 62 - bits;  // n weights of at most 2^F each cannot overflow 2^62
  // fraction bits: the largest cell index and the fraction share 62 bits
  int cb = kCellBits;
  while (cb > 1 && ((long long)std::max(grid->n1, grid->n2) >> (62 - cb)) > 0) --cb;
  // copies of the accumulator, as many as the static array holds, but no more
  // than the particles per node (clearing and adding a copy costs what as
  // many particles as nodes do)
  int copies = (int)std::min<long long>(kMaxCopies, std::min(kStaticNodes / nodes, n / nodes));
  copies = std::max(1, copies);
  auto blocks = [](long long k) { return (unsigned)std::min<long long>(4096, (k + 255) / 256); };
  k_clear<<<blocks(nodes * copies), 256, 0, s>>>(acc, nodes * copies);
  if (cudaGetLastError() != cudaSuccess) return APIC_ERR_CUDA;
  if (n > 0) {
    const double h1 = (grid->x1_outer + 1.0) / grid->n1, h2 = 2.0 / grid->n2;
    long long wb = (n + 255) / 256;
    wb = wb > 16384 ? 16384 : wb;  // grid-stride loop beyond 2^22 particles
    unsigned long long out_bits;
    std::memcpy(&out_bits, &grid->x1_outer, sizeof(out_bits));
    const double s1 = ldexp(1.0 / h1, cb), s2 = ldexp(1.0 / h2, cb);
    // the window: two CTAs of 1024 threads per SM share it out; worth its
    // clearing and flushing from a few dozen particles per entry and CTA pair on
    const int rows = (int)std::min<long long>(grid->n1 + 1, kWindowBytes / (8ll * (grid->n2 + 1)));
    int sms = 0;
    if (rows >= 2 && n >= 64ll * rows * (grid->n2 + 1) && (sms = sm_count()) > 0) {
      k_weigh<true><<<2 * sms, 1024, rows * (grid->n2 + 1) * sizeof(unsigned long long), s>>>(
          acc, x1, x2, n, grid->n1, grid->n2, out_bits, s1, s2, cb, F, copies, (int)nodes, rows);
    } else {
      k_weigh<false><<<(unsigned)wb, 256, 0, s>>>(acc, x1, x2, n, grid->n1, grid->n2, out_bits, s1, s2, cb, F, copies,
                                                  (int)nodes, 0);
    }
    if (cudaGetLastError() != cudaSuccess) return APIC_ERR_CUDA;  // rho is not written
  }
  k_density<<<blocks(nodes), 256, 0, s>>>(acc, volume, rho, nodes, copies, qw * ldexp(1.0, -F));
  return cudaGetLastError() == cudaSuccess ? APIC_OK : APIC_ERR_CUDA;
}
