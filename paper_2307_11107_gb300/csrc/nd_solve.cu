// Nested-dissection solve of the Poisson problem of Eqs. 6-7 (Sec. 2) for
// every instance of a batch in one cooperative launch: iterative refinement
//   r = b - A x (FP64),  e = A^-1 r by two sweeps over the front tree,  x += e
// until |r| <= tol |b| per instance, with the step's density before and its
// node gradients and surface quantities after it.  The sweeps run in T: FP32
// fronts (about 1e-7 of the residual left per pass) for FP32 particles, FP64
// fronts (one pass reaches FP64 rounding) for FP64 particles.
//
// Dataflow: each CTA is several workers of four warps.  Worker u takes the
// records u, u + workers, ... of the sweep's list (nd_records.h): forward the
// fronts' leaves first, backward the roots first, so that every record comes
// after those it reads from; all CTAs are resident, so the earliest unfinished
// record always runs.  The values carry their own readiness: the update
// vectors and the backward result are filled with a mark (a NaN no arithmetic
// gives) before the sweeps, writers store values with relaxed stores, readers
// load with relaxed loads and load again what still holds the mark (bounded).
// No counter, no fence and no release stands between a front and its parent,
// and no acquire invalidates L1 around the others' loads: a level of a 256 x
// 128 tree takes 1.8 us (with per-front counters 4 us).
//
// Bound: latency on single grids, FP64 additions of the node phases and the
// gathers' round trips on batches.  The 48-instance scan streams 1 GB of
// fronts per pass, 0.15 ms at HBM speed, so everything static is taken out of
// a task's chain: a record (gather tables and matrix rows of a task) is copied
// whole by one bulk copy issued while the task before runs, right-hand side and
// correction are kept front by front (contiguous), and results go from the dot
// products straight to global memory.  The warps of a worker are independent
// but for the stage they share.  Per step, ms, against sweeps that signal
// through counters and gather through global index tables: 1024 x 512 0.79 ->
// 0.39, 48 instances 2.37 -> 1.05, 256 x 128 0.32 -> 0.15 (block cyclic
// reduction 0.18); FP64 256 x 128 1.25 (multigrid) -> 0.11.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdlib>

#include "apic_internal.h"
#include "nd_records.h"

namespace apic {
namespace {

#include "solver_common.cuh"
#include "fields_common.cuh"
#include "bulk_copy.cuh"
#include "solve_nodes.cuh"

constexpr int kWkThreads = 32 * kNdFlowWarps;
constexpr int kStageBytes = 4 * kNdFlowStage;
constexpr int kVecBytes = 14 * 1024;  // a worker's vectors
constexpr int kWkBytes = kStageBytes + kVecBytes;
static_assert(kStageBytes % 128 == 0, "aligned stages");
// a warp's and an 8-lane group's share of the vectors, in FP64
static_assert(kVecBytes / 4 >= (192 + 64) * 8 + 64 * 8 && kVecBytes / 16 >= (kNdTinyU + kNdTinyS) * 8 + kNdTinyS * 8 &&
                  kVecBytes % 256 == 0,
              "vector areas");

// Elements of a kind-0 front's vector: what the rows' values (backward: z and
// x, forward: the update rows' right-hand sides) leave of a worker's area.
template <class T>
constexpr int vec_cap() {
  return (kVecBytes - kNdFlowRows * ((int)sizeof(T) + 8)) / (int)sizeof(T) & ~3;
}

// The mark of a value not written yet, relaxed stores and loads at GPU scope.
template <class T>
struct Dyn;
template <>
struct Dyn<float> {
  __device__ static float mark() { return __uint_as_float(0xffc0deadu); }
  __device__ static bool missing(float x) { return __float_as_uint(x) == 0xffc0deadu; }
  // p[i], or 0 for i < 0 (predicated: no branch)
  __device__ static float load(const float* p, int i) {
    float x;
    asm volatile(
        "{\n .reg .pred q;\n setp.ge.s32 q, %2, 0;\n mov.f32 %0, 0f00000000;\n"
        " @q ld.relaxed.gpu.global.f32 %0, [%1];\n}\n"
        : "=f"(x)
        : "l"(p + i), "r"(i)
        : "memory");
    return x;
  }
  __device__ static void store(float* p, float x) {
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(p), "f"(x) : "memory");
  }
};
template <>
struct Dyn<double> {
  __device__ static double mark() { return __longlong_as_double((long long)0xfff8deadfff8deadull); }
  __device__ static bool missing(double x) { return (unsigned)__double2hiint(x) == 0xfff8deadu; }
  __device__ static double load(const double* p, int i) {
    double x;
    asm volatile(
        "{\n .reg .pred q;\n setp.ge.s32 q, %2, 0;\n mov.f64 %0, 0d0000000000000000;\n"
        " @q ld.relaxed.gpu.global.f64 %0, [%1];\n}\n"
        : "=d"(x)
        : "l"(p + i), "r"(i)
        : "memory");
    return x;
  }
  __device__ static void store(double* p, double x) {
    asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(x) : "memory");
  }
};

// 16-byte vectors of T.
template <class T>
struct V16;
template <>
struct V16<float> {
  using V = float4;
  static constexpr int kN = 4;
  __device__ static float dot(const float4& a, const float4& b, float acc) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, acc))));
  }
};
template <>
struct V16<double> {
  using V = double2;
  static constexpr int kN = 2;
  __device__ static double dot(const double2& a, const double2& b, double acc) {
    return fma(a.x, b.x, fma(a.y, b.y, acc));
  }
};

// Dot products of rows [0, nr) (nv vectors of 16 bytes each, stride vectors
// apart) at `mat` with `v`, both in shared memory, G lanes per row with A
// partial sums each: vector t goes to partial sum t mod (G A), which lane
// t mod G keeps, and the partial sums are added in a butterfly from the
// farthest pairs down, a lane's own first: the result depends on G A alone, not
// on G, the CTA or the batch.  Lane q of the rows' `lanes` lanes takes the rows
// q / G, q / G + lanes / G, ....  Every lane runs as many passes (nr is the
// same for all lanes that shuffle).  fn(row, value) on the first lane of a row.
template <class T, int G, int A, class Fn>
__device__ __forceinline__ void rows_dot(const T* mat, int stride, int nv, int nr, const T* v, int q, int lanes,
                                         Fn fn) {
  using V = typename V16<T>::V;
  const int sl = q & (G - 1), step = lanes / G;
  const V* v4 = (const V*)v;
  for (int a0 = 0; a0 < nr; a0 += step) {
    const int a = a0 + q / G;
    const V* m4 = (const V*)mat + a * stride;
    T acc[A];
#pragma unroll
    for (int i = 0; i < A; ++i) acc[i] = T(0);
    if (a < nr) {
      for (int t = sl; t < nv; t += G * A) {
#pragma unroll
        for (int i = 0; i < A; ++i)
          if (t + i * G < nv) acc[i] = V16<T>::dot(m4[t + i * G], v4[t + i * G], acc[i]);
      }
    }
#pragma unroll
    for (int o = A / 2; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < o; ++i) acc[i] += acc[i + o];
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(kFull, acc[0], o);
    if (a < nr && sl == 0) fn(a, acc[0]);
  }
}

// The forms of nd_records.cpp's shape_of: lanes 2^lg for 2^sum partial sums.
// (Few forms: every tree level of a chain of dependent tasks pays for the
// instructions it is first to run.)
template <class T, class Fn>
__device__ __forceinline__ void rows_any(int lg, int sum, const T* mat, int stride, int nv, int nr, const T* v, int q,
                                         int lanes, Fn fn) {
  if (sum == 2) rows_dot<T, 1, 4>(mat, stride, nv, nr, v, q, lanes, fn);
  else if (lg == 0) rows_dot<T, 1, 8>(mat, stride, nv, nr, v, q, lanes, fn);
  else if (lg == 1) rows_dot<T, 2, 8>(mat, stride, nv, nr, v, q, lanes, fn);
  else if (lg == 2) rows_dot<T, 4, 8>(mat, stride, nv, nr, v, q, lanes, fn);
  else rows_dot<T, 32, 1>(mat, stride, nv, nr, v, q, lanes, fn);
}

// Loads src[ix[0 .. kUnroll)] (0 for a negative index) until none holds the
// mark.  Lanes that miss one first wait for the two entries rep (negative:
// none), which are written last, one load at a time, then load again.  False
// after d.wait_ns (kErrTimeout) or when another wait gave up.
constexpr int kUnroll = 8;

template <class T>
__device__ __noinline__ bool wait_ready(const DevPtrs& d, const T* src, const int2 rep) {
  unsigned long long t0 = 0;
  for (int spins = 1; Dyn<T>::missing(Dyn<T>::load(src, rep.x)) || Dyn<T>::missing(Dyn<T>::load(src, rep.y)); ++spins) {
    __nanosleep(20);
    if ((spins & 63) == 0) {
      if ((*(volatile int*)d.err) & kErrTimeout) return false;
      const unsigned long long now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > d.wait_ns) {
        atomicOr(d.err, kErrTimeout);
        return false;
      }
    }
  }
  return true;
}

template <class T>
__device__ __forceinline__ bool load_ready(const DevPtrs& d, const T* src, const int (&ix)[kUnroll], T (&v)[kUnroll],
                                           const int2 rep) {
  for (unsigned long long t0 = 0;;) {
    bool miss = false;
#pragma unroll
    for (int i = 0; i < kUnroll; ++i) v[i] = Dyn<T>::load(src, ix[i]);
#pragma unroll
    for (int i = 0; i < kUnroll; ++i) miss |= Dyn<T>::missing(v[i]);
    if (!miss) return true;
    if (!wait_ready<T>(d, src, rep)) return false;
    // the last entries are there: the others follow within a store's time
    const unsigned long long now = global_ns();
    if (t0 == 0) t0 = now;
    else if (now - t0 > d.wait_ns) {
      atomicOr(d.err, kErrTimeout);
      return false;
    }
  }
}

// A front's vectors of a record from global memory, by `lanes` lanes (this
// one is q).  Forward: v[p], p < s, the front's right-hand side f[p] plus what
// the children's update vectors hold for it (pairs; null: a leaf), child 0
// then child 1, zeros up to s_pad, and, unless a leaf, z[k], k < nu, the same
// for the task's update rows (no right-hand side).
template <class T>
__device__ __forceinline__ bool gather_fwd(const DevPtrs& d, T* v, int s, int s_pad, T* z, int nu, const int2* pairs,
                                           const T* f, const T* w, const int2 rep, int q, int lanes) {
  if (!pairs) {
    for (int p = q; p < s_pad; p += lanes) v[p] = p < s ? f[p] : T(0);
    return true;
  }
  // positions: the separator's, its padding, the update rows'; the tables
  // skip the padding
  const int n = s_pad + nu, gap = s_pad - s;
  constexpr int H = kUnroll / 2;  // entries of two children each
  for (int b = q; b < n; b += H * lanes) {
    T x[H], y[kUnroll];
    int a[kUnroll];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const int p = b + i * lanes, k = p < s_pad ? p : p - gap;
      const bool in = p < n && (p < s || p >= s_pad);
      int2 g = make_int2(-1, -1);
      if (in) g = pairs[k];
      x[i] = p < s ? f[p] : T(0);
      a[2 * i] = g.x;
      a[2 * i + 1] = g.y;
    }
    if (!load_ready<T>(d, w, a, y, rep)) return false;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const int p = b + i * lanes;
      T* o = p < s_pad ? v + p : z + (p - s_pad);
      if (p < n) *o = x[i] + y[2 * i] + y[2 * i + 1];
    }
  }
  return true;
}

// Backward: v[p] = e at the update set's places tab[p], p < u, zeros up to
// u_pad, and for the task's rows a < nr z[a] = z0[a] (the forward sweep's) and
// xs[a] = x at the unknowns tab[u + a].
template <class T>
__device__ __forceinline__ bool gather_back(const DevPtrs& d, T* v, int u, int u_pad, T* z, double* xs, int nr,
                                            const int* tab, const T* e, const T* z0, const double* x, const int2 rep,
                                            int q, int lanes) {
  T zr = T(0);
  double xr = 0.0;
  if (q < nr) {  // (the first row's loads run beside the update set's)
    zr = z0[q];
    xr = x[tab[u + q]];
  }
  for (int b = q; b < u_pad; b += kUnroll * lanes) {
    T y[kUnroll];
    int a[kUnroll];
#pragma unroll
    for (int i = 0; i < kUnroll; ++i) a[i] = b + i * lanes < u ? tab[b + i * lanes] : -1;
    if (!load_ready<T>(d, e, a, y, rep)) return false;
#pragma unroll
    for (int i = 0; i < kUnroll; ++i)
      if (b + i * lanes < u_pad) v[b + i * lanes] = y[i];
  }
  if (q < nr) {
    z[q] = zr;
    xs[q] = xr;
  }
  for (int a = q + lanes; a < nr; a += lanes) {
    z[a] = z0[a];
    xs[a] = x[tab[u + a]];
  }
  return true;
}

// Bounded wait of a warp for a stage's copy (all lanes).
__device__ __forceinline__ bool wait_stage(uint64_t* bar, unsigned parity, int32_t* err) {
  bool ok = false;
  for (long long k = 0; k < (1ll << 22); ++k) {
    if (mbar_try_wait(bar, parity)) {
      ok = true;
      break;
    }
    if ((k & 1023) == 1023 && ((*(volatile int32_t*)err) & kErrTimeout)) break;
    __nanosleep(32);
  }
  if (!ok) {
    atomicOr(err, kErrTimeout);
    for (long long k = 0; k < (1ll << 22); ++k) {  // the copy in flight lands before the stage or the CTA goes
      if (mbar_try_wait(bar, parity)) break;
      __nanosleep(64);
    }
  }
  return __all_sync(kFull, ok) != 0;
}

// One record of a sweep by one warp of a worker.  f: the right-hand side's
// residual, z, e: what the sweeps give (forward, backward), x: its solution,
// all of the record's instance; w: its update vectors; vec: the worker's
// vectors.  False: a wait gave up.
template <class T, bool kFwd>
__device__ __forceinline__ bool run_record(const DevPtrs& d, const int* rec, char* vec, const T* f, T* zb, T* e,
                                           double* x, T* w, int kind, int warp, int lane, int bar_id) {
  const int nf = rec[1];
  // the lanes that share a front, this lane's place among them and its front:
  // kind 0 the worker, 1 the warp, 2 an 8-lane group
  const int lanes = kind == 0 ? kWkThreads : (kind == 1 ? 32 : 8);
  const int q = kind == 0 ? 32 * warp + lane : (kind == 1 ? lane : lane & 7);
  const int k = kind == 0 ? 0 : (kind == 1 ? warp : warp + kNdFlowWarps * (lane >> 3));
  if (kind != 0 && warp >= nf) return true;
  const bool has = k < nf;
  const int* E = rec + kNdHead + kNdEntry * (has ? k : 0);
  const int s = E[kNdS], u = E[kNdU], nv = E[kNdVecs], stride = E[kNdStride], r0 = E[kNdR0], lg = E[kNdLg] & 255;
  const bool leaf = (E[kNdLg] & kNdHas) == 0;
  const int nr = has ? E[kNdNr] : 0, pad = nv * V16<T>::kN;
  const int* tab = rec + E[kNdTab];
  const T* mat = (const T*)(rec + E[kNdMat]);
  T* out = (kFwd ? zb : e) + E[kNdP0] + r0;  // the task's first row
  constexpr int kWarpVec = kVecBytes / kNdFlowWarps;
  T* v = (T*)(vec + (kind == 0 ? 0 : warp * kWarpVec + (kind == 2 ? (lane >> 3) * (kWarpVec / 4) : 0)));
  T* z = v + (kind == 0 ? vec_cap<T>() : (kind == 1 ? (kFwd ? 64 : 192) : (kFwd ? kNdTinyS : kNdTinyU)));
  double* xs = (double*)(z + (kind == 0 ? kNdFlowRows : (kind == 1 ? 64 : kNdTinyS)));
  const int skip = kFwd ? max(r0, s) - s : 0;  // update rows before the task's
  bool ok = true;
  if (has) {
    const int2 rep = make_int2(E[kNdRep0], E[kNdRep1]);
    if (kFwd)
      ok = gather_fwd<T>(d, v, s, pad, z, max(0, r0 + nr - max(r0, s)), leaf ? nullptr : (const int2*)tab, f + E[kNdP0],
                         w, rep, q, lanes);
    else ok = gather_back<T>(d, v, u, pad, z, xs, nr, tab, e, zb + E[kNdP0] + r0, x, rep, q, lanes);
  }
  ok = __all_sync(kFull, ok) != 0;  // (and orders the vectors' stores)
  if (kind == 0) {
    asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(kWkThreads) : "memory");
  }
  if (!ok) return false;
  __syncwarp();
  T* wo = w + E[kNdW];
  auto put = [=](int a, T acc) {
    if (kFwd) {
      const int r = r0 + a;
      if (r < s) out[a] = acc;
      else Dyn<T>::store(wo + (r - s), leaf ? -acc : z[r - s - skip] - acc);
    } else {
      const T val = z[a] - acc;
      Dyn<T>::store(out + a, val);
      x[tab[u + a]] = xs[a] + (double)val;
    }
  };
  rows_any<T>(lg, E[kNdLgSum], mat, stride, nv, nr, v, q, lanes, put);
  return true;
}

// One sweep: the records of `list` (n entries: record offset in 16-byte
// units, bytes, instance, kind) for every right-hand side, worker by worker.
// i0: copies the worker has issued so far (its stage's parity).  A worker
// whose wait gave up takes the rest of its records' copies without running
// them, so its barriers stay in step; the grid barrier that follows ends the
// kernel.
template <class T, bool kFwd>
__device__ __forceinline__ void sweep(const DevPtrs& d, const BcrPlan& pl, const int4* list, int n, int R,
                                      const int* s_act, char* wk, uint64_t* bar, unsigned& i0, const BcrRhs& rhs) {
  constexpr int kWk = nd_workers(sizeof(T) / 4);
  const int ni = d.n_inst;
  const int h = (int)threadIdx.x / kWkThreads, t = (int)threadIdx.x % kWkThreads, warp = t >> 5, lane = t & 31;
  const int total = R * n, nu = kWk * (int)gridDim.x;
  auto x_of = [&](int r) { return r == 0 ? rhs.x[0] : (r == 1 ? rhs.x[1] : rhs.x[2]); };
  // the next record from q on whose system still iterates
  auto next = [&](int q, int4& en) {
    for (; q < total; q += nu) {
      const int r = R == 1 ? 0 : q / n;
      en = list[q - r * n];
      if (s_act[r * ni + en.z]) break;
    }
    return q;
  };
  auto issue = [&](const int4& en) {
    if (t == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_expect_tx(bar, (unsigned)en.y);
      const char* src = (const char*)d.nd_rec + 16ll * en.x;
      if (pl.nd_stream) bulk_g2s_stream(wk, src, (unsigned)en.y, bar);
      else bulk_g2s(wk, src, (unsigned)en.y, bar);
    }
  };
  bool good = true;
  int4 en0 = make_int4(0, 0, 0, 0);
  int q0 = next(h * (int)gridDim.x + (int)blockIdx.x, en0);
  if (q0 < total) issue(en0);
  for (; q0 < total; ++i0) {
    int4 en1 = en0;
    const int q1 = next(q0 + nu, en1);  // its loads run beside this record
    if (!wait_stage(bar, i0 & 1u, d.err)) good = false;
    const int rh = R == 1 ? 0 : q0 / n;
    const int* rec = (const int*)wk;
    const long long at = rh * pl.rows + rec[3];
    if (good)
      good = run_record<T, kFwd>(d, rec, wk + kStageBytes, (const T*)d.bcr_f + at, (T*)d.bcr_e + at, (T*)d.nd_e2 + at,
                                 x_of(rh) + rec[4] + rec[2], (T*)d.nd_w + rh * pl.nd_wrows, en0.w, warp, lane, 1 + h);
    else if (en0.w == 0)  // the barrier inside a shared record
      asm volatile("bar.sync %0, %1;" ::"r"(1 + h), "r"(kWkThreads) : "memory");
    // every warp is done with the stage (and with its vectors)
    asm volatile("bar.sync %0, %1;" ::"r"(1 + h), "r"(kWkThreads) : "memory");
    if (q1 < total) issue(en1);
    q0 = q1;
    en0 = en1;
  }
}

// mode, only, rhs as k_solve_bcr (bcr.cu).
constexpr double kFloor64 = 1e-11;  // relative residual below which an FP64 solve may stop at its rounding floor

template <class T, class Real>  // of the fronts, of the particles
__global__ void __launch_bounds__(nd_threads(sizeof(T) / 4), 1)
k_solve_nd(const __grid_constant__ DevPtrs d, const __grid_constant__ BcrPlan pl, int mode, int only,
           const __grid_constant__ BcrRhs rhs) {
  constexpr int kWk = nd_workers(sizeof(T) / 4);
  extern __shared__ __align__(128) char s_dyn[];
  __shared__ double sh[40];
  __shared__ double s_bn[kCoopMaxInst];
  __shared__ double s_rn[kCoopMaxInst];
  __shared__ double s_rp[kCoopMaxInst];  // |r|^2 of the pass before
  __shared__ int s_act[kCoopMaxInst];
  __shared__ int s_npre[kCoopMaxInst + 1];
  __shared__ double s_seg[kSumSlots];
  __shared__ int s_sp[kCoopMaxInst + 1];
  __shared__ int s_foff[kCoopMaxInst];
  __shared__ __align__(8) uint64_t s_bar[kWk];
  const int nb = gridDim.x, ni = d.n_inst, R = rhs.n, nv = R * ni;
  static_assert(kBcrMaxRhs == 3, "selections below");
  auto x_of = [&](int r) { return r == 0 ? rhs.x[0] : (r == 1 ? rhs.x[1] : rhs.x[2]); };
  auto b_of = [&](int r) { return r == 0 ? rhs.b[0] : (r == 1 ? rhs.b[1] : rhs.b[2]); };
  double* part_b = d.bcr_part;              // |b|^2 per range
  double* part_r = d.bcr_part + pl.chunks;  // |r|^2 per range and right-hand side
  double* seg_b = d.bcr_part + (1 + kBcrMaxRhs) * pl.chunks;  // the sums' second stage
  double* seg_r = seg_b + kBcrMaxRhs * (pl.chunks + ni);
  for (int k = threadIdx.x; k <= ni; k += blockDim.x) {
    s_npre[k] = d.bcr_npre[k];
    if (k < ni) s_foff[k] = (int)d.bcr_inst[k].foff;
  }
  for (int v = threadIdx.x; v < nv; v += blockDim.x) s_act[v] = only < 0 || v % ni == only;
  if (threadIdx.x < kWk) mbar_init(&s_bar[threadIdx.x], 1);
  __syncthreads();
  sum_prefix(s_npre, ni, s_sp);
  __syncthreads();
  // FP64 residual at a node, stored as the sweeps' right-hand side; returns
  // its square
  auto residual = [&](int rh, int k, const Inst& I, int nd, double bv) {
    const int N = I.N2, i = nd / N, j = nd - i * N;
    if (i <= 0 || i >= I.n1) return 0.0;
    const double r = bv - apply_st<double, double>(d.st64 + (long long)kSt * I.node_off, I.nodes, x_of(rh) + I.node_off,
                                                   nd, i, j, I.n2, N, 1);
    ((T*)d.bcr_f)[rh * pl.rows + s_foff[k] + d.nd_perm[s_foff[k] + nd - N]] = (T)r;
    return r * r;
  };
  auto gradient = [&](const Inst& I, int nd) {
    if constexpr (sizeof(Real) == 4) grad_node<float, float2>(d, I, nd);
    else grad_node<double, double2>(d, I, nd);
  };
  // the density and the first residual in one phase where every instance
  // starts from its last potential (an extrapolated start is written by this
  // phase, and its neighbours' residuals read it)
  bool fused = (mode & kBcrRho) != 0;
  for (int k = 0; k < ni && fused; ++k) fused = !(d.inst[k].guess && d.stp[k].step >= 2);
  if (mode & kBcrRho) {
    if (!fused) {
      node_tasks(d, s_npre, 1, pl.chunks, nullptr, part_b, nullptr, [&](int, int k, const Inst& I, int nd) {
        const double bv = rho_node(d, I, k, nd);
        return make_double2(bv * bv, 0.0);
      });
      if (!grid_sync(d, nb)) return;
      if (!inst_sums(d, part_b, seg_b, s_npre, s_sp, 1, pl.chunks, nullptr, s_bn, s_seg)) return;
    }
  } else {
    for (int v = threadIdx.x; v < nv; v += blockDim.x) {
      const int r = v / ni, k = v - r * ni;
      const int slot = r == 0 ? rhs.slot[0] : (r == 1 ? rhs.slot[1] : rhs.slot[2]);
      const double* pr = d.red + ((long long)k * kNRed + slot) * kRedBlocks;
      double s0 = 0.0;
      for (int q = 0; q < kRedBlocks; ++q) s0 += pr[q];
      s_bn[v] = s0;
    }
    __syncthreads();
  }
  bool graded = false;  // the last residual phase took the node gradients along
  const int h = (int)threadIdx.x / kWkThreads;
  char* wk = s_dyn + h * kWkBytes;
  unsigned copies = 0;  // this worker's copies so far
  for (int it = 0;; ++it) {
    // residual of every system still iterating; where this should be the last
    // one (two passes of FP32 fronts, one of FP64 ones), the node gradients too
    graded = (mode & kBcrFields) && it == (sizeof(T) == 4 ? 2 : 1);
    if (it == 0 && fused) {
      node_tasks(d, s_npre, 1, pl.chunks, nullptr, part_r, part_b, [&](int, int k, const Inst& I, int nd) {
        const double bv = rho_node(d, I, k, nd);
        return make_double2(residual(0, k, I, nd, bv), bv * bv);
      });
    } else if (graded) {
      node_tasks(d, s_npre, 1, pl.chunks, nullptr, part_r, nullptr, [&](int, int k, const Inst& I, int nd) {
        gradient(I, nd);
        return make_double2(s_act[k] ? residual(0, k, I, nd, b_of(0)[I.node_off + nd]) : 0.0, 0.0);
      });
    } else {
      node_tasks(d, s_npre, R, pl.chunks, s_act, part_r, nullptr, [&](int rh, int k, const Inst& I, int nd) {
        return make_double2(residual(rh, k, I, nd, b_of(rh)[I.node_off + nd]), 0.0);
      });
    }
    // the mark in what this pass's sweeps write
    for (int rh = 0; rh < R; ++rh) {
      const int n = (int)pl.rows + (int)pl.nd_wrows, rows = (int)pl.rows;
      T* e2 = (T*)d.nd_e2 + rh * pl.rows;
      T* w = (T*)d.nd_w + rh * pl.nd_wrows;
      for (int z = blockIdx.x * (int)blockDim.x + threadIdx.x; z < n; z += nb * (int)blockDim.x)
        (z < rows ? e2[z] : w[z - rows]) = Dyn<T>::mark();
    }
    if (!grid_sync(d, nb)) return;
    if (!inst_sums(d, part_r, seg_r, s_npre, s_sp, R, pl.chunks, s_act, s_rn, s_seg)) return;
    if (it == 0 && fused && !inst_sums(d, part_b, seg_b, s_npre, s_sp, 1, pl.chunks, nullptr, s_bn, s_seg)) return;
    int more = 0;
    for (int v = threadIdx.x; v < nv; v += blockDim.x) {
      if (!s_act[v]) continue;
      const int k = v % ni;
      const Inst& I = d.inst[k];
      const double rn = s_rn[v], bn = s_bn[v];
      // FP64 fronts: a residual near FP64 rounding that a further pass did not
      // halve is as small as it gets, whatever the tolerance
      const bool floor64 = sizeof(T) == 8 && it >= 2 && rn <= kFloor64 * kFloor64 * bn && rn > 0.25 * s_rp[v];
      const bool conv = rn <= I.tol * I.tol * bn || floor64, bad = !(rn == rn);
      s_rp[v] = rn;
      if (conv || bad || it >= I.max_iter) {
        if (blockIdx.x == 0) {
          if (v < ni) {  // the first right-hand side reports the solver state
            SolverState& S = d.sol[k];
            S.res = bn > 0.0 ? sqrt(rn / bn) : 0.0;
            S.iters = it;
            S.done = 1;
          }
          if (!conv) atomicOr(d.err, bad ? kErrNonFinite : kErrNotConverged);
        }
        s_act[v] = 0;
      } else {
        more = 1;
      }
    }
    if (!__syncthreads_or(more)) break;
    sweep<T, true>(d, pl, d.nd_list, pl.nd_nf, R, s_act, wk, s_bar + h, copies, rhs);
    if (!grid_sync(d, nb)) return;
    sweep<T, false>(d, pl, d.nd_list + pl.nd_nf, pl.nd_nb, R, s_act, wk, s_bar + h, copies, rhs);
    if (!grid_sync(d, nb)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) d.cnt[0] += 1;
  }
  if (mode & kBcrFields) {
    // phi is final everywhere (the last pass ended at a grid barrier)
    if (!graded)
      node_tasks(d, s_npre, 1, pl.chunks, nullptr, nullptr, nullptr, [&](int, int, const Inst& I, int nd) {
        gradient(I, nd);
        return make_double2(0.0, 0.0);
      });
    for (int k = nb - 1 - (int)blockIdx.x; k < ni; k += nb) surface_block(d, k, sh);
  }
}

// lambda_b = A^-T lambda_phi for the reverse sweep (adjoint.cu): the records
// hold the transposed fronts.  lphi: by node; out: by unknown (from each
// instance's foff).  256 x 128: 88 us, with one launch per tree level (28 of
// them, a CTA per front) 840.
__global__ void __launch_bounds__(nd_threads(2), 1)
k_nd_transposed(const __grid_constant__ DevPtrs d, const __grid_constant__ BcrPlan pl, const double* lphi,
                const __grid_constant__ BcrRhs rhs) {
  constexpr int kWk = nd_workers(2);
  extern __shared__ __align__(128) char s_dyn[];
  __shared__ int s_act[kCoopMaxInst];
  __shared__ __align__(8) uint64_t s_bar[kWk];
  const int nb = gridDim.x, ni = d.n_inst;
  for (int k = threadIdx.x; k < ni; k += blockDim.x) s_act[k] = 1;
  if (threadIdx.x < kWk) mbar_init(&s_bar[threadIdx.x], 1);
  const int t = blockIdx.x * (int)blockDim.x + threadIdx.x, nt = nb * (int)blockDim.x;
  for (int k = 0; k < ni; ++k) {
    const BcrInst& B = d.bcr_inst[k];
    if (!B.nd) continue;
    const double* src = lphi + d.inst[k].node_off + B.N;
    for (int z = t; z < B.M * B.N; z += nt) {
      ((double*)d.bcr_f)[B.foff + d.nd_perm[B.foff + z]] = src[z];
      rhs.x[0][B.foff + z] = 0.0;
    }
  }
  for (int z = t; z < (int)pl.rows; z += nt) ((double*)d.nd_e2)[z] = Dyn<double>::mark();
  for (int z = t; z < (int)pl.nd_wrows; z += nt) ((double*)d.nd_w)[z] = Dyn<double>::mark();
  if (!grid_sync(d, nb)) return;
  const int h = (int)threadIdx.x / kWkThreads;
  char* wk = s_dyn + h * kWkBytes;
  unsigned copies = 0;
  sweep<double, true>(d, pl, d.nd_list, pl.nd_nf, 1, s_act, wk, s_bar + h, copies, rhs);
  if (!grid_sync(d, nb)) return;
  sweep<double, false>(d, pl, d.nd_list + pl.nd_nf, pl.nd_nb, 1, s_act, wk, s_bar + h, copies, rhs);
}

const void* kernel_of(const BcrPlan& b) {
  if (b.nd_elem == 1) return (const void*)k_solve_nd<float, float>;
  return b.nd_f64 ? (const void*)k_solve_nd<double, double> : (const void*)k_solve_nd<double, float>;
}

}  // namespace

const void* nd_kernel(const SolvePlan& pl) { return kernel_of(pl.bcr); }

int nd_vec_cap(int elem) { return elem == 2 ? vec_cap<double>() : vec_cap<float>(); }

static int configure(const void* kern, BcrPlan& b, int sms) {
  b.dyn = nd_workers(b.nd_elem) * kWkBytes;
  int per_sm = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, b.dyn) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nd_threads(b.nd_elem), (size_t)b.dyn) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return 0;
  }
  return sms < kCoopMaxBlocks ? sms : kCoopMaxBlocks;
}

int nd_configure(SolvePlan& pl, int sms) { return configure(kernel_of(pl.bcr), pl.bcr, sms); }

int nd_transposed_configure(BcrPlan& b, int sms) { return configure((const void*)k_nd_transposed, b, sms); }

cudaError_t launch_nd_transposed(const DevPtrs& d, const BcrPlan& b, int blocks, const double* lphi, double* out,
                                 cudaStream_t s) {
  BcrRhs rhs{};
  rhs.n = 1;
  rhs.x[0] = out;
  void* args[] = {(void*)&d, (void*)&b, (void*)&lphi, (void*)&rhs};
  return cudaLaunchCooperativeKernel((const void*)k_nd_transposed, dim3(blocks), dim3(nd_threads(2)), args,
                                     (size_t)b.dyn, s);
}

}  // namespace apic
