// Reverse sweep (adjoint) of a K-step window of the APIC step
// (arXiv:2307.11107, Secs. 1-2): the gradient of L = sum_o dL/dout_o out_o
// (window means of drag F_Z, electric F_Z, current, torque T_z and grain
// charge Q) with respect to the grain shape alpha (Eqs. 2-5, 7), the grain
// potential phi_g (boundary value of Eq. 6) and the axial field B (Eq. 9), at
// fixed decisions (absorbed, escaped or kept, injection counts, cells): the
// transpose of the forward-mode window's Jacobian, computed backwards.
//
// Forward pass (the ordinary step, with per-step checkpoints): the particle
// state at the start of each step, rho and phi, each slot's fate in the push
// and each injection draw's slot.  Reverse pass, step K-1 down to 0, in the
// reverse order of the step:
//   injection   the adjoint of an injected particle's state times its
//               alpha-derivative (Eq. 4 sampling at the same random numbers);
//   push        per particle, the transpose of its local Jacobian (the step's
//               gather of Eq. 10, Boris push of Eq. 9, chord, rotation and
//               Eq. 2, or the tallies of an absorbed particle) applied to its
//               adjoint, stage by stage;
//   surface     the seeds of the electric force and grain charge on phi;
//   gradients   the transpose of the node differences;
//   Poisson     lambda_b = A^-T lambda_phi with the nested-dissection fronts
//               of A applied transposed (FP64; as dataflow sweeps, nd_solve.cu,
//               or, where a front exceeds their records, level by level), and the terms of phi_g (the
//               Dirichlet row) and alpha (the operator's derivative);
//   deposit     the transpose of the bilinear weighing onto the particles and
//               the alpha-derivative of w = V_domain / N and of the volumes.
//
// Compiled once per particle precision (-DAPIC_REAL=double | float); the
// node-side kernels only in the double build (APIC_ADJOINT_COMMON).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "apic_internal.h"
#include "dual.cuh"
#include "geom.cuh"

#ifndef APIC_REAL
#error "compile with -DAPIC_REAL=float or -DAPIC_REAL=double"
#endif

namespace apic {
namespace {

#include "particle_common.cuh"

using Real2 = typename Pair<Real>::T;
using D1 = ad::Dual<Real, 1>;

__device__ __forceinline__ const Real* ckc(const AdjPtrs& a, int k, int c) {
  return (const Real*)a.ck + ((long long)k * 5 + c) * a.stride;
}

// Prefix of the populations' slot counts at the start of step k (one thread).
__device__ __forceinline__ void pop_prefix_at(const DevPtrs& d, const PopState* ps, long long* pre) {
  if (threadIdx.x == 0) {
    long long s = 0;
    for (int p = 0; p < d.n_pop; ++p) {
      pre[p] = s;
      s += ps[p].n;
    }
    pre[d.n_pop] = s;
  }
  __syncthreads();
}

// What a population's particles share in the forward push, in their precision
// (a conversion or a division of the FP64 parameters per particle bounds the
// kernel: the FP64 pipe takes two lanes a clock per SM; 2e6 particles 70 us
// with them, 49 without).
struct FwdPop {
  Real h, al, dt, B, h1, h2, x1_out;
  long long base, node_off;
  int n1, n2, N2, pad;
};

// One particle's push, the same sequence as the step's push (gather of Eq. 10
// with the bilinear weights of its cell, Boris push with the field vector
// -B z-hat, straight chord, rotation back to the meridional plane, Eq. 2).
struct PushIO {
  Real x1n, x2n, vRn, vz, vTn;  // the new state of a kept particle
  Real R, Z, vx, vy;            // chord start and the velocity at n + 1/2 (tallies)
  bool hit, out;
};

__device__ __forceinline__ void push_eval(const FwdPop& C, const Real2* G, Real x1, Real x2, Real vR, Real vZ, Real vT,
                                          PushIO& o) {
  const Real dt = C.dt, al = C.al, h = C.h;
  Real r = radius(al, x1, x2);
  Real sn = sqrt((Real(1) - x2) * (Real(1) + x2));
  Real R = r * sn, Z = r * x2;
  Real u1 = (x1 + Real(1)) / C.h1;
  Real u2 = (x2 + Real(1)) / C.h2;
  int ci = (int)floor(u1), cj = (int)floor(u2);
  ci = ci < 0 ? 0 : (ci > C.n1 - 1 ? C.n1 - 1 : ci);
  cj = cj < 0 ? 0 : (cj > C.n2 - 1 ? C.n2 - 1 : cj);
  Real f1 = u1 - (Real)ci, f2 = u2 - (Real)cj;
  if (f1 < Real(0)) f1 = Real(0);
  if (f1 > Real(1)) f1 = Real(1);
  if (f2 < Real(0)) f2 = Real(0);
  if (f2 > Real(1)) f2 = Real(1);
  const long long n00 = C.node_off + (long long)ci * C.N2 + cj;
  const Real2 a00 = G[n00], a10 = G[n00 + C.N2], a01 = G[n00 + 1], a11 = G[n00 + C.N2 + 1];
  Real w00 = (Real(1) - f1) * (Real(1) - f2), w10 = f1 * (Real(1) - f2);
  Real w01 = (Real(1) - f1) * f2, w11 = f1 * f2;
  Real g1 = w00 * a00.x + w10 * a10.x + w01 * a01.x + w11 * a11.x;
  Real g2 = w00 * a00.y + w10 * a10.y + w01 * a01.y + w11 * a11.y;
  Metric<Real> m = metric(al, r, x2);
  Real ER = -(m.x1R * g1 + m.x2R * g2);
  Real EZ = -(m.x1Z * g1 + m.x2Z * g2);
  Real vx = vR + h * ER, vy = vT, vz = vZ + h * EZ;
  Real tz = h * (-C.B);
  Real sz = Real(2) * tz / (Real(1) + tz * tz);
  Real px_ = vx + vy * tz, py_ = vy - vx * tz;
  vx = vx + py_ * sz;
  vy = vy - px_ * sz;
  vx = vx + h * ER;
  vz = vz + h * EZ;
  Real Xc = R + vx * dt, Yc = vy * dt, Zn = Z + vz * dt;
  Real Rn = sqrt(Xc * Xc + Yc * Yc);
  Real cr(Real(1)), sr(Real(0));
  if (Rn > Real(0)) {
    cr = Xc / Rn;
    sr = Yc / Rn;
  }
  o.vRn = cr * vx + sr * vy;
  o.vTn = -sr * vx + cr * vy;
  Real rn = sqrt(Rn * Rn + Zn * Zn);
  o.x2n = Zn / rn;
  o.hit = rn < r_grain(al, o.x2n);
  o.x1n = x1_at(al, rn, o.x2n);
  o.out = !o.hit && o.x1n > C.x1_out;
  o.vz = vz;
  o.R = R;
  o.Z = Z;
  o.vx = vx;
  o.vy = vy;
}

// ---- forward pass ----
// The step's push (values), each live slot's state before it (the step's
// checkpoint) and every slot's fate recorded: 0 kept, 1 absorbed, 2 escaped, 3
// no live particle.
__global__ void __launch_bounds__(256) k_adj_fwd_push(DevPtrs d, AdjPtrs a, int k) {
  extern __shared__ __align__(16) char s_raw[];
  FwdPop* s_pop = (FwdPop*)s_raw;
  __shared__ long long s_pre[kMaxPop + 1];
  for (int p = threadIdx.x; p < d.n_pop; p += blockDim.x) {
    const Pop& P = d.pop[p];
    const Inst& I = d.inst[P.inst];
    s_pop[p] = FwdPop{Real(0.5) * (Real)(P.q / P.m) * (Real)I.dt, (Real)I.alpha, (Real)I.dt, (Real)I.B, (Real)I.h1,
                      (Real)I.h2, (Real)I.x1_out, P.base, I.node_off, I.n1, I.n2, I.N2, 0};
  }
  pop_prefix_at(d, d.ps, s_pre);
  const long long total = s_pre[d.n_pop];
  const Real2* G = (const Real2*)d.G;
  uint8_t* fate = a.fate + (long long)k * a.stride;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const int pop = find_pop(s_pre, d.n_pop, q);
    const FwdPop& C = s_pop[pop];
    const long long kk = q - s_pre[pop], slot = C.base + kk;
    const Real x1 = ((const Real*)d.x1)[slot];
    if (!(x1 < Real(0))) {
      fate[slot] = 3;
      continue;
    }
    const Real x2 = ((const Real*)d.x2)[slot], vR = ((const Real*)d.vR)[slot], vZ = ((const Real*)d.vZ)[slot],
               vT = ((const Real*)d.vT)[slot];
    Real* ck = (Real*)a.ck + (long long)k * 5 * a.stride + slot;
    ck[0] = x1;
    ck[a.stride] = x2;
    ck[2 * a.stride] = vR;
    ck[3 * a.stride] = vZ;
    ck[4 * a.stride] = vT;
    PushIO o;
    push_eval(C, G, x1, x2, vR, vZ, vT, o);
    if (o.hit) {
      const Pop& P = d.pop[pop];
      const Inst& I = d.inst[P.inst];
      absorb_tally(d, I, P, o.R, o.Z, o.vx, o.vz, o.vy, C.dt);
      atomicAdd((unsigned long long*)&d.ps[pop].absorbed, 1ull);
      ((Real*)d.x1)[slot] = Real(2);
      push_hole(d, P, pop, kk);
      fate[slot] = 1;
      continue;
    }
    if (o.out) {
      atomicAdd((unsigned long long*)&d.ps[pop].escaped, 1ull);
      ((Real*)d.x1)[slot] = Real(2);
      push_hole(d, d.pop[pop], pop, kk);
      fate[slot] = 2;
      continue;
    }
    ((Real*)d.x1)[slot] = o.x1n;
    ((Real*)d.x2)[slot] = o.x2n;
    ((Real*)d.vR)[slot] = o.vRn;
    ((Real*)d.vZ)[slot] = o.vz;
    ((Real*)d.vT)[slot] = o.vTn;
    fate[slot] = 0;
  }
}

// Threads per CTA of the injection kernels: a long chain of FP64 and special
// functions for a few thousand particles, spread over the SMs.
constexpr int kInjThreads = 64;

// An injected particle's state (values and alpha-derivative) from its draws:
// x2 from the inverse CDF of Eq. 4 on x1_out (its alpha-derivative from the
// table's), a flux-weighted half-Maxwellian along -grad x1 and Maxwellian
// tangential and Theta components, a free flight of a uniform fraction of dt.
struct Inj {
  D1 x1n, x2n, vRn, vz, vTn;  // stored state
  D1 R, Z, vx, vy;            // flight start and velocity (tallies)
  Real tau;
  bool hit, out;
};

__device__ __forceinline__ void inject_eval(const DevPtrs& d, const TanPtrs& t, const Inst& I, const Pop& P,
                                            long long g, Inj& o) {
  uint32_t u[8];
  draws8(I, P, g, 2u, u);
  const D1 al = D1::seed((Real)I.alpha, 0);
  const Real dt = (Real)I.dt;
  const double* cdf = d.tab + I.tab_off + (kTable + 1);
  const double* dcdf = t.dtab + I.tab_off + (kTable + 1);
  const Real u0 = unit(u[0]);
  const double tq = (double)u0 * cdf[kTable];
  const int lo = table_interval(cdf, d.guide + I.tab_off + (kTable + 1), (double)u0, tq);
  const double dlt = cdf[lo + 1] - cdf[lo];
  const double f = dlt > 0.0 ? (tq - cdf[lo]) / dlt : 0.5;
  const double ht = 2.0 / kTable;
  const double dtq = (double)u0 * dcdf[kTable];
  const double df = dlt > 0.0 ? (dtq - dcdf[lo] - f * (dcdf[lo + 1] - dcdf[lo])) / dlt : 0.0;
  D1 x2((Real)(-1.0 + lo * ht + f * ht));
  x2.d[0] = (Real)(df * ht);
  const Real vth = (Real)P.vth;
  const Real vn = vth * sqrt(Real(-2) * log(unit(u[1])));
  const Real ra = sqrt(Real(-2) * log(unit(u[2])));
  const Real pa = Real(2 * kPi) * unit(u[3]);
  const Real vt = vth * (ra * cos(pa)), vth_ = vth * (ra * sin(pa));
  o.tau = unit(u[4]) * dt;
  D1 r = radius(al, D1((Real)I.x1_out), x2);
  D1 sn = sqrt((Real(1) - x2) * (Real(1) + x2));
  o.R = r * sn;
  o.Z = r * x2;
  Metric<D1> m = metric(al, r, x2);
  D1 gn = sqrt(m.x1R * m.x1R + m.x1Z * m.x1Z);
  D1 nR = -m.x1R / gn, nZ = -m.x1Z / gn;
  D1 tR = nZ, tZ = -nR;
  o.vx = vn * nR + vt * tR;
  o.vz = vn * nZ + vt * tZ;
  o.vy = D1(vth_);
  D1 Xc = o.R + o.vx * o.tau, Yc = o.vy * o.tau, Zn = o.Z + o.vz * o.tau;
  D1 Rn = sqrt(Xc * Xc + Yc * Yc);
  D1 cr(Real(1)), sr(Real(0));
  if (Rn.v > Real(0)) {
    cr = Xc / Rn;
    sr = Yc / Rn;
  }
  D1 rn = sqrt(Rn * Rn + Zn * Zn);
  o.x2n = Zn / rn;
  o.hit = rn.v < r_grain(al.v, o.x2n.v);
  o.x1n = x1_at(al, rn, o.x2n);
  o.out = !o.hit && o.x1n.v > (Real)I.x1_out;
  o.vRn = cr * o.vx + sr * o.vy;
  o.vTn = -sr * o.vx + cr * o.vy;
}

// The step's surface injection (values), each draw's slot recorded (from the
// population's base; -1 absorbed in its first flight, -2 escaped).
__global__ void __launch_bounds__(kInjThreads) k_adj_fwd_inject(DevPtrs d, AdjPtrs a, TanPtrs t, int k) {
  const int pop = blockIdx.y;
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  PopState& S = d.ps[pop];
  const Pop& P = d.pop[pop];
  const Inst& I = d.inst[P.inst];
  if (q >= S.n_inj) return;
  int64_t* rec = a.inj + ((long long)k * d.n_pop + pop) * a.inj_cap;
  Inj o;
  inject_eval(d, t, I, P, S.draws + q, o);
  if (o.hit) {
    absorb_tally(d, I, P, o.R.v, o.Z.v, o.vx.v, o.vz.v, o.vy.v, o.tau);
    atomicAdd((unsigned long long*)&S.absorbed, 1ull);
    if (q < a.inj_cap) rec[q] = -1;
    return;
  }
  if (o.out) {
    atomicAdd((unsigned long long*)&S.escaped, 1ull);
    if (q < a.inj_cap) rec[q] = -2;
    return;
  }
  const long long sidx = (long long)atomicAdd((unsigned long long*)&S.inj_stored, 1ull);
  const long long nh = S.n_holes, n = S.n;
  const long long kk = sidx < nh ? d.holes[P.base + nh - 1 - sidx] : n + (sidx - nh);
  if (kk >= P.cap) {
    atomicAdd((unsigned long long*)&S.dropped, 1ull);
    atomicOr(d.err, kErrCapacity);
    if (q < a.inj_cap) rec[q] = -2;
    return;
  }
  const long long slot = P.base + kk;
  ((Real*)d.x1)[slot] = o.x1n.v;
  ((Real*)d.x2)[slot] = o.x2n.v;
  ((Real*)d.vR)[slot] = o.vRn.v;
  ((Real*)d.vZ)[slot] = o.vz.v;
  ((Real*)d.vT)[slot] = o.vTn.v;
  if (q < a.inj_cap) rec[q] = kk;
}

// ---- reverse pass ----
// Parameter adjoints of one thread (instance inst) added to the instance's
// totals: a warp whose lanes share the instance adds its sum once.
__device__ __forceinline__ void add_grad(const AdjPtrs& a, int inst, double ga, double gp, double gb) {
  const unsigned full = 0xffffffffu;
  const int i0 = __shfl_sync(full, inst, 0);
  if (__all_sync(full, inst == i0)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ga += __shfl_down_sync(full, ga, o);
      gp += __shfl_down_sync(full, gp, o);
      gb += __shfl_down_sync(full, gb, o);
    }
    if ((threadIdx.x & 31) == 0 && i0 >= 0) {
      if (ga != 0.0) atomicAdd(a.grad + i0 * kNPar + 0, ga);
      if (gp != 0.0) atomicAdd(a.grad + i0 * kNPar + 1, gp);
      if (gb != 0.0) atomicAdd(a.grad + i0 * kNPar + 2, gb);
    }
  } else if (inst >= 0) {
    if (ga != 0.0) atomicAdd(a.grad + inst * kNPar + 0, ga);
    if (gp != 0.0) atomicAdd(a.grad + inst * kNPar + 1, gp);
    if (gb != 0.0) atomicAdd(a.grad + inst * kNPar + 2, gb);
  }
}

// Injection of step k backwards: a stored particle's adjoint (from the later
// steps) times its state's alpha-derivative, and the slot's adjoint cleared
// (before the step's injection it held no particle, or one that left in
// this step's push); a particle absorbed in its first flight adds its
// tallies' alpha-derivatives (w = V_domain / N moves with alpha too).
__global__ void __launch_bounds__(kInjThreads) k_adj_rev_inject(DevPtrs d, AdjPtrs a, TanPtrs t, int k) {
  const int pop = blockIdx.y;
  const Pop& P = d.pop[pop];
  const Inst& I = d.inst[P.inst];
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long g0 = a.ck_ps[(long long)k * d.n_pop + pop].draws;
  const long long n_inj = a.ck_ps[(long long)(k + 1) * d.n_pop + pop].draws - g0;
  double ga = 0.0;
  int inst = -1;
  if (q < n_inj && q < a.inj_cap) {
    const int64_t rec = a.inj[((long long)k * d.n_pop + pop) * a.inj_cap + q];
    if (rec != -2) {
      inst = P.inst;
      Inj o;
      inject_eval(d, t, I, P, g0 + q, o);
      if (rec >= 0) {
        const long long slot = P.base + rec;
        double* L = a.lam;
        const D1* st[5] = {&o.x1n, &o.x2n, &o.vRn, &o.vz, &o.vTn};
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          ga += L[(long long)c * a.stride + slot] * (double)st[c]->d[0];
          L[(long long)c * a.stride + slot] = 0.0;
        }
      } else {
        const double* sd = a.seed + (long long)P.inst * kNOut;
        const double dt = I.dt, w = P.w, dl = t.dlnw[P.inst];
        const double vz = o.vz.v, Rvy = (double)o.R.v * o.vy.v;
        const double dvz = o.vz.d[0], dRvy = (double)o.R.d[0] * o.vy.v + (double)o.R.v * o.vy.d[0];
        ga += sd[0] / dt * P.m * w * (dvz + vz * dl) + sd[3] / dt * P.m * w * (dRvy + Rvy * dl) +
              sd[2] / dt * P.q * w * dl;
      }
    }
  }
  add_grad(a, inst, ga, 0.0, 0.0);
}

// A float as a double by integer arithmetic (exact; subnormals as zero): the
// FP64 pipe, which a conversion instruction takes as long as a product, does
// two lanes a clock per SM and bounds the reverse particle kernels.
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  unsigned hi = (m >> 3) + 0x38000000u;
  if (m >= 0x7f800000u) hi += 0x38000000u;  // infinities and NaN keep the largest exponent
  if (m < 0x00800000u) hi = 0u;
  return __hiloint2double((int)(hi | (b & 0x80000000u)), m < 0x00800000u ? 0 : (int)(b << 29));
}

// What a population's particles share in the reverse push.
struct RevPop {
  double c, s, dt;       // the magnetic rotation
  double k0, k3, k2;     // the absorbed particle's seeds: dL/d(vz), dL/d(R vy) and its constant part
  double dl;             // d ln w / d alpha
  Real h, al, fdt, tz, sz, cB, sB;
  Real h1, h2, ih1, ih2;
  long long base, node_off;
  int n1, n2, N2, inst;
};

// Cell and fractions of (x1, x2) as push_eval's, and the fractions' derivatives
// (zero where the fraction is clamped).
struct RevCell {
  long long n00;
  Real f1, f2, d1, d2;
};
__device__ __forceinline__ RevCell rev_cell(const RevPop& C, Real x1, Real x2) {
  const Real u1 = (x1 + Real(1)) / C.h1, u2 = (x2 + Real(1)) / C.h2;
  int ci = (int)floor(u1), cj = (int)floor(u2);
  ci = ci < 0 ? 0 : (ci > C.n1 - 1 ? C.n1 - 1 : ci);
  cj = cj < 0 ? 0 : (cj > C.n2 - 1 ? C.n2 - 1 : cj);
  RevCell r{C.node_off + (long long)ci * C.N2 + cj, u1 - (Real)ci, u2 - (Real)cj, C.ih1, C.ih2};
  if (r.f1 < Real(0) || r.f1 > Real(1)) {
    r.f1 = r.f1 < Real(0) ? Real(0) : Real(1);
    r.d1 = Real(0);
  }
  if (r.f2 < Real(0) || r.f2 > Real(1)) {
    r.f2 = r.f2 < Real(0) ? Real(0) : Real(1);
    r.d2 = Real(0);
  }
  return r;
}

// Push of step k backwards.  For each slot live at the start of the step
// (the checkpoint), the transpose of the particle's local Jacobian applied to
// the adjoint of its push's result: the new state's adjoint for a kept
// particle, the output seeds of its tallies for an absorbed one, nothing for
// an escaped one.  The slot's adjoint becomes that of its state at the start
// of the step; the gathered field's adjoint goes to the four corner nodes with
// the bilinear weights.
//
// The push is taken backwards stage by stage (end point in Eq. 2, rotation to
// the meridional plane, chord, Boris rotation, field and metric, Eq. 3), with
// the stages' derivatives in closed form in the particles' precision and the
// adjoints in FP64.  Bound: with float particles the FP64 pipe (about 45
// products a particle and the corner sums), with double ones its operations
// altogether.  Dual numbers three directions at a time, the form before,
// evaluated the push's values three times and spent as much of the FP64 pipe
// on converting the Jacobian's 45 entries as on their products.
// The corner sums of a plasma that fills its volume meet on the outermost rows'
// nodes, where the additions follow one another at L2 (its busiest slice at 87 %
// while the mean is at 13 %): the CTAs add to several copies of lambda_G
// (a.copies), folded before the gradients' transpose.  2e6 float particles on
// 256 x 128 cells: 1.00 ms by duals, 0.48 in this form, 0.23 with eight copies.
template <class F>
__device__ __forceinline__ void load_pops(const DevPtrs& d, const AdjPtrs& a, const TanPtrs& t, F* pop) {
  for (int p = threadIdx.x; p < d.n_pop; p += blockDim.x) {
    const Pop& P = d.pop[p];
    const Inst& I = d.inst[P.inst];
    F& C = pop[p];
    const double* sd = a.seed + (long long)P.inst * kNOut;
    const double dt = I.dt, w = P.w;
    C.h = Real(0.5) * (Real)(P.q / P.m) * (Real)I.dt;
    C.al = (Real)I.alpha;
    C.fdt = (Real)I.dt;
    C.tz = C.h * -(Real)I.B;
    const Real den = Real(1) + C.tz * C.tz;
    C.sz = Real(2) * C.tz / den;
    const Real cr = (Real(1) - C.tz * C.tz) / den;  // 1 - t s
    C.c = cr;
    C.s = C.sz;
    // along B: dt = -h dB, ds = 2 c / (1 + t^2) dt, dc = -2 s / (1 + t^2) dt
    C.sB = -C.h * (Real(2) * cr / den);
    C.cB = C.h * (Real(2) * C.sz / den);
    C.dt = (Real)I.dt;
    C.dl = t.dlnw[P.inst];
    C.k0 = sd[0] / dt * P.m * w;
    C.k3 = sd[3] / dt * P.m * w;
    C.k2 = sd[2] / dt * P.q * w;
    C.h1 = (Real)I.h1;
    C.h2 = (Real)I.h2;
    C.ih1 = Real(1) / C.h1;
    C.ih2 = Real(1) / C.h2;
    C.base = P.base;
    C.node_off = I.node_off;
    C.n1 = I.n1;
    C.n2 = I.n2;
    C.N2 = I.N2;
    C.inst = P.inst;
  }
  __syncthreads();
}

constexpr int kRevThreads = 256;
__global__ void __launch_bounds__(kRevThreads) k_adj_rev_push(DevPtrs d, AdjPtrs a, TanPtrs t, int k) {
  extern __shared__ __align__(16) char s_raw[];
  RevPop* s_pop = (RevPop*)s_raw;
  __shared__ long long s_pre[kMaxPop + 1];
  const PopState* ps = a.ck_ps + (long long)k * d.n_pop;
  load_pops(d, a, t, s_pop);
  pop_prefix_at(d, ps, s_pre);
  const long long total = s_pre[d.n_pop];
  const Real2* G = (const Real2*)a.Gk;
  const uint8_t* fate = a.fate + (long long)k * a.stride;
  const long long tn = d.total_nodes;
  double* L = a.lam;
  double* lG = a.lG + 2 * tn * (blockIdx.x % (unsigned)a.copies);
  double ga = 0.0, gb = 0.0;
  int inst = -1;  // the instance that ga, gb belong to
  for (long long q0 = (long long)blockIdx.x * blockDim.x; q0 < total; q0 += (long long)gridDim.x * blockDim.x) {
    const long long q = q0 + threadIdx.x;
    const int pop = q < total ? find_pop(s_pre, d.n_pop, q) : -1;
    const int in_q = pop < 0 ? inst : s_pop[pop].inst;
    if (__any_sync(0xffffffffu, in_q != inst)) {
      add_grad(a, inst, ga, 0.0, gb);
      ga = gb = 0.0;
      inst = in_q;
    }
    if (pop < 0) continue;
    const RevPop& C = s_pop[pop];
    const long long slot = C.base + (q - s_pre[pop]);
    const int f = fate[slot];
    if (f > 1) {
#pragma unroll
      for (int c = 0; c < 5; ++c) L[(long long)c * a.stride + slot] = 0.0;
      continue;
    }
    const Real x1 = ckc(a, k, 0)[slot], x2 = ckc(a, k, 1)[slot], vR = ckc(a, k, 2)[slot], vZ = ckc(a, k, 3)[slot],
               vT = ckc(a, k, 4)[slot];
    const Real al = C.al, h = C.h, dt = C.fdt;
    // Eq. 3 and the position: derivatives along x1, x2, alpha
    const Real qs = sqrt(Real(1) - Real(4) * al * x1 * x2), iq = Real(1) / qs, ix = Real(1) / x1;
    const Real r = -(Real(1) + qs) * (Real(0.5) * ix), ir = Real(1) / r;
    const Real s2 = (Real(1) - x2) * (Real(1) + x2), sn = sqrt(s2);
    const Real sn2 = sn > Real(0) ? -x2 / sn : Real(0);
    const Real r1 = (al * x2 * iq - r) * ix, r2 = al * iq, ra = x2 * iq;
    const Real R = r * sn, Z = r * x2;
    const Real R1 = r1 * sn, R2 = r2 * sn + r * sn2, Ra = ra * sn;
    const Real Z1 = r1 * x2, Z2 = r2 * x2 + r, Za = ra * x2;
    // the field of Eq. 10 and its derivatives
    const RevCell e = rev_cell(C, x1, x2);
    const Real2 a00 = G[e.n00], a10 = G[e.n00 + C.N2], a01 = G[e.n00 + 1], a11 = G[e.n00 + C.N2 + 1];
    const Real o1 = Real(1) - e.f1, o2 = Real(1) - e.f2;
    const Real w00 = o1 * o2, w10 = e.f1 * o2, w01 = o1 * e.f2, w11 = e.f1 * e.f2;
    const Real g1 = w00 * a00.x + w10 * a10.x + w01 * a01.x + w11 * a11.x;
    const Real g2 = w00 * a00.y + w10 * a10.y + w01 * a01.y + w11 * a11.y;
    const Real g11 = e.d1 * (o2 * (a10.x - a00.x) + e.f2 * (a11.x - a01.x));
    const Real g12 = e.d2 * (o1 * (a01.x - a00.x) + e.f1 * (a11.x - a10.x));
    const Real g21 = e.d1 * (o2 * (a10.y - a00.y) + e.f2 * (a11.y - a01.y));
    const Real g22 = e.d2 * (o1 * (a01.y - a00.y) + e.f1 * (a11.y - a10.y));
    // the metric (geom.cuh) and its derivatives along r, x2, alpha
    const Real ir3 = ir * ir * ir;
    const Real p1 = r + Real(3) * al * x2, p2 = Real(3) * x2 * x2 - Real(1);
    const Real mR1 = sn * p1 * ir3, mZ1 = (r * x2 + al * p2) * ir3, mR2 = -x2 * sn * ir, mZ2 = s2 * ir;
    const Real mR1r = sn * ir3 - Real(3) * mR1 * ir, mZ1r = x2 * ir3 - Real(3) * mZ1 * ir;
    const Real mR1x = (sn2 * p1 + Real(3) * al * sn) * ir3, mZ1x = (r + Real(6) * al * x2) * ir3;
    const Real mR2x = -(sn + x2 * sn2) * ir, mZ2x = Real(-2) * x2 * ir;
    const Real ER = -(mR1 * g1 + mR2 * g2), EZ = -(mZ1 * g1 + mZ2 * g2);
    const Real ERr = -(mR1r * g1 - mR2 * ir * g2), EZr = -(mZ1r * g1 - mZ2 * ir * g2);
    const Real ER1 = ERr * r1 - (mR1 * g11 + mR2 * g21), EZ1 = EZr * r1 - (mZ1 * g11 + mZ2 * g21);
    const Real ER2 = ERr * r2 - (mR1x * g1 + mR2x * g2 + mR1 * g12 + mR2 * g22);
    const Real EZ2 = EZr * r2 - (mZ1x * g1 + mZ2x * g2 + mZ1 * g12 + mZ2 * g22);
    const Real ERa = ERr * ra - Real(3) * sn * x2 * ir3 * g1, EZa = EZr * ra - p2 * ir3 * g1;
    // Boris push
    const Real bx = vR + h * ER, bz = vZ + h * EZ;
    const Real px = bx + vT * C.tz, py = vT - bx * C.tz;
    const Real vx = bx + py * C.sz + h * ER, vy = vT - px * C.sz, vz = bz + h * EZ;
    double aX = 0.0, aY = 0.0, aZ = 0.0;     // of the chord's end
    double avx = 0.0, avy = 0.0, avz, aR = 0.0, aa = 0.0;
    if (f == 0) {
      const double l1 = L[slot], l2 = L[a.stride + slot], lR = L[2 * a.stride + slot], lZ = L[3 * a.stride + slot],
                   lT = L[4 * a.stride + slot];
      const Real Xc = R + vx * dt, Yc = vy * dt, Zn = Z + vz * dt;
      const Real Rn = sqrt(Xc * Xc + Yc * Yc), rn = sqrt(Rn * Rn + Zn * Zn), irn = Real(1) / rn;
      Real cr = Real(1), sr = Real(0), iRn = Real(0);
      if (Rn > Real(0)) {
        iRn = Real(1) / Rn;
        cr = Xc * iRn;
        sr = Yc * iRn;
      }
      const Real xn = Zn * irn, st = Rn * irn, i2 = irn * irn;
      // Eq. 2, then x2 = Z / r and r of the end point
      aa = l1 * wide(-xn * i2);
      const double ax2 = fma(l1, wide(-al * i2), l2);
      const double arn = l1 * wide(i2 + Real(2) * al * xn * i2 * irn);
      aZ = fma(arn, wide(xn), ax2 * wide(st * st * irn));
      const double aRn = iRn > Real(0) ? wide(st) * fma(ax2, wide(-xn * irn), arn) : 0.0;
      // rotation to the meridional plane
      const Real vRn = cr * vx + sr * vy, vTn = cr * vy - sr * vx;
      const double tt = fma(lR, wide(vTn), -(lT * wide(vRn)));
      aX = fma(aRn, wide(cr), tt * wide(-sr * iRn));
      aY = fma(aRn, wide(sr), tt * wide(cr * iRn));
      const double c = wide(cr), s = wide(sr);
      avx = fma(C.dt, aX, fma(lR, c, -(lT * s)));
      avy = fma(C.dt, aY, fma(lR, s, lT * c));
      avz = fma(C.dt, aZ, lZ);
      aR = aX;
    } else {
      const double Rw = wide(R), vyw = wide(vy);
      avz = C.k0;
      aR = C.k3 * vyw;
      avy = C.k3 * Rw;
      aa = C.dl * (C.k0 * wide(vz) + C.k3 * Rw * vyw + C.k2);  // w moves with alpha
    }
    // Boris rotation: vx = c bx + s vT + h ER, vy = c vT - s bx
    gb += avx * wide(bx * C.cB + vT * C.sB) + avy * wide(vT * C.cB - bx * C.sB);
    const double abx = fma(C.c, avx, -(C.s * avy)), aT = fma(C.s, avx, C.c * avy);
    const double aE = avx + abx;  // over h; that of h EZ is 2 avz
    const Real hz = Real(2) * h;
    const double l1 = fma(aR, wide(R1), fma(aZ, wide(Z1), fma(aE, wide(h * ER1), avz * wide(hz * EZ1))));
    const double l2 = fma(aR, wide(R2), fma(aZ, wide(Z2), fma(aE, wide(h * ER2), avz * wide(hz * EZ2))));
    ga += aa + fma(aR, wide(Ra), fma(aZ, wide(Za), fma(aE, wide(h * ERa), avz * wide(hz * EZa))));
    const double lg1 = -fma(aE, wide(h * mR1), avz * wide(hz * mZ1));
    const double lg2 = -fma(aE, wide(h * mR2), avz * wide(hz * mZ2));
    L[slot] = l1;
    L[a.stride + slot] = l2;
    L[2 * a.stride + slot] = abx;
    L[3 * a.stride + slot] = avz;
    L[4 * a.stride + slot] = aT;
    const Real w[4] = {w00, w10, w01, w11};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (w[c] == Real(0)) continue;
      const long long n = e.n00 + (c & 1 ? C.N2 : 0) + (c >> 1);
      const double wd = wide(w[c]);
      atomicAdd(lG + n, wd * lg1);
      atomicAdd(lG + tn + n, wd * lg2);
    }
  }
  add_grad(a, inst, ga, 0.0, gb);
}

// Deposit of step k backwards: rho = sum_p q w S(x_p) / V, so the adjoint of
// a live particle's (x1, x2) gains q w sum_c (dS_c / dx) lambda_rho_c / V_c
// (bilinear weights of its cell; a clamped fraction carries none; a.lrho holds
// lambda_rho / V).  Bound by the FP64 pipe: a coordinate's cell and fraction
// come from one fused product and a conversion (as in cell_fixed.cuh), the
// corner sum from the cell's differences.
// 2e6 float particles on 256 x 128 cells: 475 us with divisions, 63 so.
struct DepPop {
  double s1, s2;            // 2^b / h1, 2^b / h2
  double k1, k2;            // q w / h1, q w / h2
  long long base, node_off;
  int n1, n2, N2, b;        // b: a fraction's bits (the largest cell index and a fraction share 62)
};

// Cell of a logical coordinate and the fraction in it (to 2^-b); the
// fraction's derivative is zero (d = 0) where it is clamped to [0, 1].
__device__ __forceinline__ int dep_cell(double x, double s, int n, int b, double& f, double& d) {
  const long long t = __double2ll_rn(fma(x, s, s));
  const int i = (int)(t >> b);
  unsigned long long m = (unsigned long long)t & ((1ull << b) - 1ull);
  if ((unsigned)i >= (unsigned)n) {  // outside the grid, or on its last node
    m = i < 0 ? 0ull : 1ull << b;
    if (t != (long long)n << b) d = 0.0;
  }
  f = __longlong_as_double((long long)(0x3ff0000000000000ull + (m << (52 - b)))) - 1.0;
  return min(max(i, 0), n - 1);
}

__global__ void __launch_bounds__(kRevThreads) k_adj_rev_deposit(DevPtrs d, AdjPtrs a, int k) {
  extern __shared__ __align__(16) char s_raw[];
  DepPop* s_pop = (DepPop*)s_raw;
  __shared__ long long s_pre[kMaxPop + 1];
  for (int p = threadIdx.x; p < d.n_pop; p += blockDim.x) {
    const Pop& P = d.pop[p];
    const Inst& I = d.inst[P.inst];
    const double qw = P.q * P.w;
    int b = 50;
    while (b > 1 && (long long)max(I.n1, I.n2) >> (62 - b)) --b;
    s_pop[p] = DepPop{ldexp(1.0 / I.h1, b), ldexp(1.0 / I.h2, b), qw / I.h1, qw / I.h2, P.base, I.node_off, I.n1, I.n2,
                      I.N2, b};
  }
  pop_prefix_at(d, a.ck_ps + (long long)k * d.n_pop, s_pre);
  const long long total = s_pre[d.n_pop];
  const uint8_t* fate = a.fate + (long long)k * a.stride;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (long long)gridDim.x * blockDim.x) {
    const int pop = find_pop(s_pre, d.n_pop, q);
    const DepPop& C = s_pop[pop];
    const long long slot = C.base + (q - s_pre[pop]);
    if (fate[slot] == 3) continue;
    double f1, f2, k1 = C.k1, k2 = C.k2;
    const int ci = dep_cell(wide(ckc(a, k, 0)[slot]), C.s1, C.n1, C.b, f1, k1);
    const int cj = dep_cell(wide(ckc(a, k, 1)[slot]), C.s2, C.n2, C.b, f2, k2);
    const double* l = a.lrho + C.node_off + (long long)ci * C.N2 + cj;
    // l00 .. l11 = l[0], l[N2], l[1], l[N2 + 1]:  d/dx1 = (l10 - l00) + f2 m, d/dx2 = (l01 - l00) + f1 m,
    // m = (l11 - l01) - (l10 - l00)
    const double l00 = l[0], l10 = l[C.N2], l01 = l[1], l11 = l[C.N2 + 1];
    const double e1 = l10 - l00, e2 = l01 - l00, m = (l11 - l01) - e1;
    a.lam[slot] = fma(k1, fma(f2, m, e1), a.lam[slot]);
    a.lam[a.stride + slot] = fma(k2, fma(f1, m, e2), a.lam[a.stride + slot]);
  }
}

#ifdef APIC_ADJOINT_COMMON
__device__ __forceinline__ double x2_node(const Inst& I, int j) { return j == I.n2 ? 1.0 : -1.0 + j * I.h2; }

// Deterministic block sum (fixed tree) of one double per thread; blockDim 256.
__device__ double block_sum(double v, double* sh) {
  int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int o = blockDim.x >> 1; o > 0; o >>= 1) {
    if (t < o) sh[t] += sh[t + o];
    __syncthreads();
  }
  double r = sh[0];
  __syncthreads();
  return r;
}

// Constants of the grain surface per node j of instance blockIdx.x, and their
// alpha-derivatives: |grad x1|, dA of Eq. 4 and n_Z dA (once, at set-up).
__global__ void __launch_bounds__(256) k_adj_surface_geom(DevPtrs d, AdjPtrs a, int n2_max) {
  const Inst& I = d.inst[blockIdx.x];
  double* o = a.sgeo + 6ll * blockIdx.x * (n2_max + 1);
  for (int j = threadIdx.x; j <= I.n2; j += blockDim.x) {
    using DD = ad::Dual<double, 1>;
    DD al = DD::seed(I.alpha, 0), X2(x2_node(I, j));
    DD r = r_grain(al, X2);
    Metric<DD> m = metric(al, r, X2);
    DD g = sqrt(m.x1R * m.x1R + m.x1Z * m.x1Z);
    DD dA = area_density(al, DD(-1.0), X2);
    DD nzda = (m.x1Z / g) * dA;
    const double v[6] = {g.v, g.d[0], dA.v, dA.d[0], nzda.v, nzda.d[0]};
    for (int c = 0; c < 6; ++c) o[6 * j + c] = v[c];
  }
}

// Seeds of the electric force and grain charge of step k on phi (rows 0..2
// through the one-sided dphi/dx1 on the grain), and their alpha-derivative at
// fixed phi (|grad x1|, n_Z and dA of Eq. 4 on the grain).
__global__ void __launch_bounds__(256) k_adj_surface(DevPtrs d, AdjPtrs a, int k, int n2_max) {
  __shared__ double sh[256];
  const int inst = blockIdx.x;
  const Inst& I = d.inst[inst];
  const bool nofield = (I.flags & APIC_NO_FIELD) != 0;
  const int N2 = I.N2;
  const double* p0 = a.ck_phi + (long long)k * d.total_nodes + I.node_off;
  const double* geo = a.sgeo + 6ll * inst * (n2_max + 1);
  const double sF = a.seed[(long long)inst * kNOut + 1], sQ = a.seed[(long long)inst * kNOut + 4];
  double ga = 0.0;
  for (int j = threadIdx.x; j <= I.n2 && !nofield; j += blockDim.x) {
    const double g = geo[6 * j], gd = geo[6 * j + 1], dA = geo[6 * j + 2], dAd = geo[6 * j + 3], nz = geo[6 * j + 4],
                 nzd = geo[6 * j + 5];
    const double G1 = (-3.0 * p0[j] + 4.0 * p0[N2 + j] - p0[2 * N2 + j]) / (2.0 * I.h1);
    const double En = -G1 * g;
    const double tw = (j == 0 || j == I.n2) ? 0.5 * I.h2 : I.h2;
    // dL/dE_n and the E_n derivative along alpha at fixed phi
    const double dLdE = sQ * tw * dA + sF * tw * En * nz;
    const double dEa = -G1 * gd;
    ga += dLdE * dEa + sQ * tw * En * dAd + sF * tw * 0.5 * En * En * nzd;
    const double c = -g / (2.0 * I.h1);  // dE_n / dphi = c (-3, 4, -1) on rows 0, 1, 2
    double* lp = a.lphi + I.node_off;
    lp[j] += dLdE * c * -3.0;
    lp[N2 + j] += dLdE * c * 4.0;
    lp[2 * N2 + j] += dLdE * c * -1.0;
  }
  const double tot = block_sum(ga, sh);
  if (threadIdx.x == 0 && tot != 0.0) atomicAdd(a.grad + (long long)inst * kNPar + 0, tot);
}

// The copies of lambda_G added into the first.
__global__ void __launch_bounds__(256) k_adj_fold(double* lG, long long n, int copies) {
  for (long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x; z < n; z += (long long)gridDim.x * blockDim.x) {
    double s = lG[z];
#pragma unroll 4
    for (int c = 1; c < copies; ++c) s += lG[c * n + z];
    lG[z] = s;
  }
}

// lambda_phi += D^T lambda_G: the transpose of the node gradients (central
// differences inside, one-sided second order on the four edges).
__global__ void __launch_bounds__(256) k_adj_gradT(DevPtrs d, AdjPtrs a) {
  const Inst& I = d.inst[blockIdx.y];
  const int n1 = I.n1, n2 = I.n2, N2 = I.N2;
  const double* l1 = a.lG + I.node_off;
  const double* l2 = a.lG + d.total_nodes + I.node_off;
  const double c1 = 1.0 / (2.0 * I.h1), c2 = 1.0 / (2.0 * I.h2);
  for (long long nd = (long long)blockIdx.x * blockDim.x + threadIdx.x; nd < I.nodes;
       nd += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(nd / N2), j = (int)(nd % N2);
    double s = 0.0;
    // G1 at row i' = i - 1 (central: + phi(i' + 1)) and i' = i + 1 (central: - phi(i' - 1))
    if (i - 1 > 0 && i - 1 < n1) s += c1 * l1[(long long)(i - 1) * N2 + j];
    if (i + 1 > 0 && i + 1 < n1) s -= c1 * l1[(long long)(i + 1) * N2 + j];
    if (i <= 2) s += c1 * (i == 0 ? -3.0 : (i == 1 ? 4.0 : -1.0)) * l1[j];
    if (i >= n1 - 2) s += c1 * (i == n1 ? 3.0 : (i == n1 - 1 ? -4.0 : 1.0)) * l1[(long long)n1 * N2 + j];
    const long long b = (long long)i * N2;
    if (j - 1 > 0 && j - 1 < n2) s += c2 * l2[b + j - 1];
    if (j + 1 > 0 && j + 1 < n2) s -= c2 * l2[b + j + 1];
    if (j <= 2) s += c2 * (j == 0 ? -3.0 : (j == 1 ? 4.0 : -1.0)) * l2[b];
    if (j >= n2 - 2) s += c2 * (j == n2 ? 3.0 : (j == n2 - 1 ? -4.0 : 1.0)) * l2[b + n2];
    a.lphi[I.node_off + nd] += s;
  }
}

// The interior of lambda_phi as the right-hand side of the transposed solve
// (unknown (i, j) of instance k at unk_off[k] + (i - 1) N2 + j).
__global__ void __launch_bounds__(256) k_adj_to_unknowns(DevPtrs d, AdjPtrs a) {
  const int inst = blockIdx.y;
  const Inst& I = d.inst[inst];
  for (long long nd = (long long)blockIdx.x * blockDim.x + threadIdx.x; nd < I.nodes;
       nd += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(nd / I.N2);
    if (i < 1 || i >= I.n1) continue;
    a.rhs[a.unk_off[inst] + nd - I.N2] = a.lphi[I.node_off + nd];
  }
}

// The transposed sweeps of the nested dissection (the fronts of A^T are the
// transposes of A's): forward z_S = F_SS^-T v_S, W = v_U - (F_SS^-1 F_SU)^T v_S;
// backward x_S = z_S - (F_US F_SS^-1)^T x_U.  One CTA per front, threads over
// the outputs (reading matrix rows, coalesced).
__global__ void __launch_bounds__(256) k_adj_ndT(AdjPtrs a, int f0, long long unk0, int forward) {
  extern __shared__ double s_v[];
  const NdFront F = a.nd_front[f0 + blockIdx.x];
  double* x = a.rhs + unk0;
  if (forward) {
    for (int p = threadIdx.x; p < F.s + F.u; p += blockDim.x) {
      const int2 g = *(const int2*)(a.nd_gather + F.G + 2 * p);
      double v = p < F.s ? x[a.nd_idx[F.S + p]] : 0.0;
      if (g.x >= 0) v += a.ndw[g.x];
      if (g.y >= 0) v += a.ndw[g.y];
      s_v[p] = v;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < F.s + F.u; c += blockDim.x) {
      double acc = 0.0;
      if (c < F.s) {
        for (int r = 0; r < F.s; ++r) acc += a.nd_mat[F.FM + (long long)r * F.sp + c] * s_v[r];
        x[a.nd_idx[F.S + c]] = acc;
      } else {
        const int qq = c - F.s;
        for (int r = 0; r < F.s; ++r) acc += a.nd_mat[F.NB + (long long)r * F.up + qq] * s_v[r];
        a.ndw[F.W + qq] = s_v[c] - acc;
      }
    }
  } else {
    for (int p = threadIdx.x; p < F.u; p += blockDim.x) s_v[p] = x[a.nd_idx[F.U + p]];
    __syncthreads();
    for (int c = threadIdx.x; c < F.s; c += blockDim.x) {
      double acc = 0.0;
      for (int r = 0; r < F.u; ++r) acc += a.nd_mat[F.FM + (long long)(F.s + r) * F.sp + c] * s_v[r];
      x[a.nd_idx[F.S + c]] -= acc;
    }
  }
}

// After the transposed solve (lambda_b in rhs): lambda_rho = -rscale lambda_b;
// the phi_g adjoint from the Dirichlet term of the scaled right-hand side and
// from lambda_phi on the grain row; the alpha adjoint from the operator's
// derivative, -lambda_b rscale (dL/dalpha phi), and from rho's explicit
// alpha-dependence, lambda_rho rho (d ln w - dV / V).
__global__ void __launch_bounds__(256) k_adj_after_solve(DevPtrs d, AdjPtrs a, TanPtrs t, int k) {
  __shared__ double sh[256];
  const int inst = blockIdx.y;
  const Inst& I = d.inst[inst];
  const bool nofield = (I.flags & APIC_NO_FIELD) != 0;
  const double* phi = a.ck_phi + (long long)k * d.total_nodes + I.node_off;
  const double* rho = a.ck_rho + (long long)k * d.total_nodes + I.node_off;
  const double* st = t.dst + (long long)kSt * I.node_off;
  const double dl = t.dlnw[inst];
  double ga = 0.0, gp = 0.0;
  for (long long nd = (long long)blockIdx.x * blockDim.x + threadIdx.x; nd < I.nodes;
       nd += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(nd / I.N2), j = (int)(nd % I.N2);
    const long long g = I.node_off + nd;
    double lr = 0.0;
    if (i == 0) gp += a.lphi[g];
    if (i > 0 && i < I.n1 && !nofield) {
      const double lb = a.rhs[a.unk_off[inst] + nd - I.N2];
      gp += lb * t.bbc_g[g];
      double dL = 0.0;
      for (int di = -1; di <= 1; ++di)
        for (int dj = -1; dj <= 1; ++dj) {
          const int jj = j + dj;
          if (jj < 0 || jj > I.n2) continue;
          dL += st[(long long)st_slot(di, dj) * I.nodes + nd] * phi[(long long)(i + di) * I.N2 + jj];
        }
      const double sp = st[(long long)kStPole * I.nodes + nd];
      if (j == 0) dL += sp * phi[(long long)i * I.N2 + 2];
      if (j == I.n2) dL += sp * phi[(long long)i * I.N2 + I.n2 - 2];
      ga -= lb * d.rscale[g] * dL;
      lr = -d.rscale[g] * lb;
    }
    a.lrho[g] = lr / d.V[g];  // as the deposit's weighing takes it
    ga += lr * rho[nd] * (dl - t.dV[g] / d.V[g]);
  }
  const double ta = block_sum(ga, sh), tp = block_sum(gp, sh);
  if (threadIdx.x == 0) {
    if (ta != 0.0) atomicAdd(a.grad + (long long)inst * kNPar + 0, ta);
    if (tp != 0.0) atomicAdd(a.grad + (long long)inst * kNPar + 1, tp);
  }
}
#endif  // APIC_ADJOINT_COMMON

}  // namespace

// CTAs of 256 threads over `n` nodes.
[[maybe_unused]] static unsigned node_blocks(long long n) {
  return (unsigned)std::max<long long>(1, std::min<long long>(608, (n + 255) / 256));
}

// CTAs of 256 threads over every slot.
static unsigned adj_blocks(const AdjPtrs& a) {
  return (unsigned)std::max<long long>(1, std::min<long long>(kAdjBlocks, (a.stride + 255) / 256));
}

template <>
void launch_adj_fwd_push<Real>(const DevPtrs& d, const AdjPtrs& a, int k, cudaStream_t s) {
  k_adj_fwd_push<<<adj_blocks(a), 256, sizeof(FwdPop) * (size_t)d.n_pop, s>>>(d, a, k);
}
template <>
void launch_adj_fwd_inject<Real>(const DevPtrs& d, const AdjPtrs& a, const TanPtrs& t, int k, long long max_inj,
                                 cudaStream_t s) {
  if (max_inj <= 0) return;
  const unsigned gx = (unsigned)((max_inj + kInjThreads - 1) / kInjThreads);
  k_adj_fwd_inject<<<dim3(gx, d.n_pop), kInjThreads, 0, s>>>(d, a, t, k);
}
template <>
void launch_adj_rev_inject<Real>(const DevPtrs& d, const AdjPtrs& a, const TanPtrs& t, int k, long long max_inj,
                                 cudaStream_t s) {
  if (max_inj <= 0) return;
  const unsigned gx = (unsigned)((max_inj + kInjThreads - 1) / kInjThreads);
  k_adj_rev_inject<<<dim3(gx, d.n_pop), kInjThreads, 0, s>>>(d, a, t, k);
}
template <>
void launch_adj_rev_push<Real>(const DevPtrs& d, const AdjPtrs& a, const TanPtrs& t, int k, cudaStream_t s) {
  k_adj_rev_push<<<adj_blocks(a), kRevThreads, sizeof(RevPop) * (size_t)d.n_pop, s>>>(d, a, t, k);
}
template <>
void launch_adj_rev_deposit<Real>(const DevPtrs& d, const AdjPtrs& a, int k, cudaStream_t s) {
  k_adj_rev_deposit<<<adj_blocks(a), kRevThreads, sizeof(DepPop) * (size_t)d.n_pop, s>>>(d, a, k);
}

#ifdef APIC_ADJOINT_COMMON
void launch_adj_surface_geom(const DevPtrs& d, const AdjPtrs& a, int n2_max, cudaStream_t s) {
  k_adj_surface_geom<<<d.n_inst, 256, 0, s>>>(d, a, n2_max);
}
void launch_adj_surface(const DevPtrs& d, const AdjPtrs& a, int k, int n2_max, cudaStream_t s) {
  k_adj_surface<<<d.n_inst, 256, 0, s>>>(d, a, k, n2_max);
}
void launch_adj_gradT(const DevPtrs& d, const AdjPtrs& a, cudaStream_t s) {
  if (a.copies > 1) k_adj_fold<<<node_blocks(2 * d.total_nodes), 256, 0, s>>>(a.lG, 2 * d.total_nodes, a.copies);
  k_adj_gradT<<<dim3(node_blocks(d.total_nodes / d.n_inst), d.n_inst), 256, 0, s>>>(d, a);
}
void launch_adj_to_unknowns(const DevPtrs& d, const AdjPtrs& a, cudaStream_t s) {
  k_adj_to_unknowns<<<dim3(kRedBlocks, d.n_inst), 256, 0, s>>>(d, a);
}
void launch_adj_ndT(const AdjPtrs& a, int f0, int f1, long long unk0, int smem_doubles, bool forward, cudaStream_t s) {
  if (f1 <= f0) return;
  k_adj_ndT<<<f1 - f0, 256, sizeof(double) * (size_t)smem_doubles, s>>>(a, f0, unk0, forward ? 1 : 0);
}
void launch_adj_after_solve(const DevPtrs& d, const AdjPtrs& a, const TanPtrs& t, int k, cudaStream_t s) {
  k_adj_after_solve<<<dim3(node_blocks(d.total_nodes / d.n_inst), d.n_inst), 256, 0, s>>>(d, a, t, k);
}
const void* adj_ndT_kernel() { return (const void*)k_adj_ndT; }
#endif

}  // namespace apic
