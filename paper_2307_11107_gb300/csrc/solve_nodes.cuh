// Node phases of the cooperative direct solves (bcr.cu, nd_solve.cu): node
// tasks with fixed-order partial sums, and the sums of the partials.
// Included inside namespace apic::{anonymous} after solver_common.cuh.
#pragma once

// Instance of task t of a phase: pre[k] <= t < pre[k + 1] (prefix in shared memory).
__device__ __forceinline__ int task_inst_s(const int* pre, int ni, int t) {
  int lo = 0, hi = ni - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= t) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Sums of part[r chunks + npre[k] .. r chunks + npre[k + 1]) for every system
// v = r ni + k (right-hand side r < nrhs, instance k) with sel[v] (all when
// sel is null); out[v] in shared memory, the same in every CTA.  A system's
// partials are summed in segments of kSumSeg, one warp each, and the segments
// in order: the result depends on the system alone.  With many partials (an
// FP64 addition of a warp takes 16 cycles of its SM) the segments are shared
// out over the CTAs, whose sums meet in part2 after one more grid barrier
// (48 instances, 3e4 partials: 8 us if every CTA adds them all).  seg:
// kSumSlots doubles of shared memory.  False: the barrier timed out.
constexpr int kSumSeg = 128, kSumLocal = 4096, kSumSlots = kSumLocal / kSumSeg + kCoopMaxInst;

// Prefix of the instances' segments (one right-hand side), sp[ni + 1]; ends
// without a barrier.
__device__ __forceinline__ void sum_prefix(const int* npre, int ni, int* sp) {
  for (int k = threadIdx.x; k <= ni; k += blockDim.x) {
    int a = 0;
    for (int z = 0; z < k; ++z) a += (npre[z + 1] - npre[z] + kSumSeg - 1) / kSumSeg;
    sp[k] = a;
  }
}

__device__ __noinline__ bool inst_sums(const DevPtrs& d, const double* part, double* part2, const int* npre,
                                       const int* sp, int nrhs, long long chunks, const int* sel, double* out,
                                       double* seg) {
  const int ni = d.n_inst, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  const int per_rhs = sp[ni], jobs = nrhs * per_rhs;
  const bool grid = (long long)nrhs * npre[ni] > kSumLocal;  // else every CTA adds all of them
  double* to = grid ? part2 : seg;
  for (int j = grid ? warp * (int)gridDim.x + (int)blockIdx.x : warp; j < jobs; j += grid ? nw * (int)gridDim.x : nw) {
    const int r = nrhs == 1 ? 0 : j / per_rhs, k = task_inst_s(sp, ni, j - r * per_rhs);
    if (sel && !sel[r * ni + k]) continue;
    const int q = j - r * per_rhs - sp[k], n = npre[k + 1] - npre[k];
    const double* pr = part + (long long)r * chunks + npre[k];
    double x = 0.0;
#pragma unroll
    for (int i = 0; i < kSumSeg / 32; ++i) {
      const int c = q * kSumSeg + lane + 32 * i;
      if (c < n) x += pr[c];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(kFull, x, o);
    if (lane == 0) to[j] = x;
  }
  if (grid) {
    if (!grid_sync(d, gridDim.x)) return false;
  } else {
    __syncthreads();
  }
  for (int v = threadIdx.x; v < nrhs * ni; v += blockDim.x) {
    if (sel && !sel[v]) continue;
    const int r = v / ni, k = v - r * ni;
    double x = 0.0;
    for (int q = sp[k]; q < sp[k + 1]; ++q) x += to[r * per_rhs + q];
    out[v] = x;
  }
  __syncthreads();
  return true;
}

// Node tasks over the ranges of range_nodes() nodes of every instance, the
// ranges of all instances (and right-hand sides r < nrhs) spread over the
// warps of all CTAs, consecutive ranges to a warp.  body(r, k, I, nd) returns
// the node's contributions (one or two) to its range's sums, which go to
// part[r chunks + npre[k] + c] and part2 (when not null) as the lanes' sums
// and a warp-shuffle tree: the sums do not depend on the CTA or the other
// instances of a batch.  sel: systems whose body runs (all when null).
template <class F>
__device__ __forceinline__ void node_tasks(const DevPtrs& d, const int* npre, int nrhs, long long chunks, const int* sel, double* part,
                           double* part2, F body) {
  const int ni = d.n_inst, nb = gridDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  const int per_rhs = npre[ni], total = nrhs * per_rhs;
  const int per = (total + nw * nb - 1) / (nw * nb);
  const int t0 = (warp * nb + (int)blockIdx.x) * per, t1 = min(total, t0 + per);
  int rh = 0, k = -1;
  const Inst* I = nullptr;
  for (int t = t0; t < t1; ++t) {
    const int c = t - rh * per_rhs;
    if (k < 0 || c >= npre[k + 1]) {  // another system
      rh = nrhs == 1 ? 0 : t / per_rhs;
      k = task_inst_s(npre, ni, t - rh * per_rhs);
      I = d.inst + k;
    }
    if (sel && !sel[rh * ni + k]) continue;
    const int cc = t - rh * per_rhs;
    const int sub = range_nodes(I->nodes), n0 = (cc - npre[k]) * sub + lane, n1 = (int)I->nodes;
    double2 x = make_double2(0.0, 0.0);
    if (n0 < n1) x = body(rh, k, *I, n0);
    if (sub == 64 && n0 + 32 < n1) {
      const double2 y = body(rh, k, *I, n0 + 32);
      x.x += y.x;
      if (part2) x.y += y.y;
    }
    if (part) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x.x += __shfl_down_sync(kFull, x.x, o);
      if (lane == 0) part[(long long)rh * chunks + cc] = x.x;
    }
    if (part2) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x.y += __shfl_down_sync(kFull, x.y, o);
      if (lane == 0) part2[(long long)rh * chunks + cc] = x.y;
    }
  }
}
