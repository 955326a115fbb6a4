// Walks the records of transposed fronts (nd_transpose64) on the host for a
// batch with an instance without fronts in the middle and prints the largest
// relative difference of y . A^-1 r and (A^-T y) . r, per instance.
// argv: M N of the two instances, workers.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>
#include <vector>

#include "../../paper_2307_11107_gb300/csrc/nd_records.h"

using namespace apic;

struct Op {
  int N;
  std::vector<double> c;
};
static double coef(const void* ctx, int i, int j, int slot) {
  const Op& o = *(const Op*)ctx;
  return o.c[((size_t)(i - 1) * o.N + j) * 11 + slot];
}

int main(int argc, char** argv) {
  if (argc < 6) return 2;
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  const int units = std::atoi(argv[5]);
  NdFlowPlan P;
  std::vector<NdFactor> fs(3);
  std::vector<int64_t> at;
  for (int k = 0; k < 3; ++k) {
    at.push_back(P.rows);
    if (k == 1) {
      if (!nd_flow_add(P, nullptr, 77, 2, units, 1280, 1 << 30)) return 3;
      continue;
    }
    const int M = std::atoi(argv[1 + k]), N = std::atoi(argv[2 + k]);
    Op op{N, std::vector<double>((size_t)M * N * 11, 0.0)};
    for (size_t q = 0; q < (size_t)M * N; ++q) {  // unsymmetric, diagonally dominant
      double* r = op.c.data() + q * 11;
      double off = 0.0;
      for (int s = 0; s < 10; ++s) off += std::fabs(r[s] = 0.3 + 0.25 * U(rng));
      r[4] = -1.1 * off;
    }
    std::string why;
    if (!nd_build(M, N, coef, &op, 16, 4, true, fs[k], why)) return 4;
    if (!nd_flow_add(P, &fs[k], (int64_t)M * N, 2, units, 1280, 1 << 30)) return 5;
  }
  nd_flow_lists(P);
  std::vector<double> r((size_t)P.rows), y(r.size()), f(r.size(), 0.0), z(r.size(), 0.0);
  for (double& v : r) v = U(rng);
  for (double& v : y) v = U(rng);
  double lhs[3] = {0, 0, 0}, scale[3] = {0, 0, 0};
  std::vector<int32_t> rec((size_t)P.words.back());
  for (int k = 0; k < 3; k += 2) {
    const int n = fs[k].M * fs[k].N;
    std::vector<double> x(n);
    nd_solve_host(fs[k], r.data() + at[k], x.data(), true);
    for (int q = 0; q < n; ++q) {
      lhs[k] += y[at[k] + q] * x[q];
      scale[k] += std::fabs(y[at[k] + q] * x[q]);
      f[at[k] + P.perm[at[k] + q]] = y[at[k] + q];
    }
    nd_transpose64(fs[k]);
    const NdFlowInst I{fs[k].N, (int)at[k], (int)at[k] - fs[k].N};
    for (size_t t = 0; t < P.tasks.size(); ++t)
      if (P.tasks[t].inst == k)
        nd_flow_write<double>(P.up, P.tasks[t], P.place, P.perm.data() + at[k], I, fs[k].fm64.data(), 0,
                              fs[k].nb64.data(), fs[k].fm_total, rec.data() + P.off[t]);
  }
  std::vector<int64_t> fw, bw;
  for (int q = 0; q < P.nf + P.nb; ++q) (q < P.nf ? fw : bw).push_back(4ll * P.list[q].at);
  if (nd_flow_solve_host<double>(rec, fw, bw, f, z.data(), std::max<int64_t>(1, P.w)) != 0) return 6;
  double worst = 0.0;
  for (int k = 0; k < 3; k += 2) {
    double rhs = 0.0;
    for (int q = 0; q < fs[k].M * fs[k].N; ++q) rhs += z[at[k] + q] * r[at[k] + q];
    worst = std::max(worst, std::fabs(rhs - lhs[k]) / scale[k]);
  }
  for (int q = 0; q < 77; ++q)
    if (z[at[1] + q] != 0.0) return 7;
  std::printf("OK %.3e\n", worst);
  return 0;
}
