// Host check of the dataflow sweeps' task records (nd_records.cpp): two
// instances of a batch (random operators with the library's stencil pattern),
// their records walked on the host in list order as the device walks them, in
// FP32 and FP64.  Prints the largest deviation from the host sweeps of the
// factorisation, relative to the largest value; FAIL if a record breaks a
// device limit, overlaps the next or comes before one it waits for.
//   nd_records_check M N M2 N2 leaf units
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>
#include <vector>

#include "../../paper_2307_11107_gb300/csrc/nd_records.h"

using namespace apic;

struct Op {
  int M, N;
  std::vector<double> c;
};

static double coef(const void* ctx, int i, int j, int slot) {
  const Op& o = *(const Op*)ctx;
  return o.c[((size_t)(i - 1) * o.N + j) * 10 + slot];
}

static Op random_op(int M, int N, unsigned seed) {
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  Op op{M, N, std::vector<double>((size_t)M * N * 10, 0.0)};
  for (size_t q = 0; q < (size_t)M * N; ++q) {
    double* r = &op.c[q * 10];
    const int j = (int)(q % N);
    double off = 0.0;
    for (int s = 0; s < 10; ++s) {
      if (s == 4 || (s == 9 && j != 0 && j != N - 1)) continue;
      r[s] = 0.3 + U(rng) * 0.2;
      off += std::fabs(r[s]);
    }
    r[4] = -1.1 * off;
  }
  return op;
}

template <class M>
static double run(const std::vector<NdFactor>& fs, const std::vector<int>& Ns, int units) {
  const int elem = (int)sizeof(M) / 4, ni = (int)fs.size();
  NdUpload up;
  std::vector<NdFlowTask> tasks;
  std::vector<int64_t> off;
  std::vector<NdFlowInst> inst;
  std::vector<int> firsts;
  int64_t w = 0, foff = 0, node = 0, words = 0;
  for (int k = 0; k < ni; ++k) {
    NdLevels lv;
    const int f0 = (int)up.fronts.size();
    nd_layout(fs[k], 0, w, 64, 192, 2048, 8192, 512, 4, 8192, 1, up, lv);
    const size_t t0 = tasks.size();
    for (int sw = 0; sw < 2; ++sw)
      if (!nd_flow_tasks(up, f0, (int)up.fronts.size() - f0, fs[k].depth, k, sw == 0, elem, units, elem == 2 ? 1280 : 2816, k == 0 ? 16 : 1 << 30, tasks))
        return -1.0;
    for (size_t t = t0; t < tasks.size(); ++t) {
      off.push_back(words);
      words += tasks[t].words;
      if (tasks[t].words > kNdFlowStage || tasks[t].words % 4) return -2.0;
    }
    inst.push_back(NdFlowInst{Ns[k], (int)foff, (int)node});
    firsts.push_back(f0);
    foff += (int64_t)fs[k].M * fs[k].N;
    node += (int64_t)(fs[k].M + 2) * fs[k].N;
    w += (fs[k].w_total + 63) & ~63ll;
  }
  std::vector<int32_t> rec((size_t)words), place, perm;
  firsts.push_back((int)up.fronts.size());
  for (int k = 0; k < ni; ++k)
    nd_flow_places(up, firsts[k], firsts[k + 1] - firsts[k], (int64_t)fs[k].M * fs[k].N, place, perm);
  std::vector<int> order[2];
  for (size_t t = 0; t < tasks.size(); ++t) {
    const NdFactor& F = fs[tasks[t].inst];
    // (a record must not write past its words: the next one's are written after and checked by the walk)
    if (elem == 2)
      nd_flow_write<double>(up, tasks[t], place, perm.data() + inst[tasks[t].inst].foff, inst[tasks[t].inst], F.fm64.data(), 0, F.nb64.data(), F.fm_total,
                            rec.data() + off[t]);
    else
      nd_flow_write<float>(up, tasks[t], place, perm.data() + inst[tasks[t].inst].foff, inst[tasks[t].inst], F.fm.data(), 0, F.nb.data(), F.fm_total,
                           rec.data() + off[t]);
    order[tasks[t].fwd ? 0 : 1].push_back((int)t);
  }
  std::vector<int64_t> list[2];
  for (int sw = 0; sw < 2; ++sw) {
    std::stable_sort(order[sw].begin(), order[sw].end(), [&](int a, int b) {
      auto key = [&](int t) { return sw == 0 ? fs[tasks[t].inst].depth - tasks[t].level : tasks[t].level; };
      return key(a) < key(b);
    });
    for (int t : order[sw]) list[sw].push_back(off[t]);
  }
  std::mt19937_64 rng(5);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  std::vector<M> f((size_t)foff);
  std::vector<double> xs((size_t)foff, 0.0);
  for (M& x : f) x = (M)U(rng);
  std::vector<char> seen((size_t)foff, 0);
  for (int k = 0; k < ni; ++k)
    for (int q = 0; q < fs[k].M * fs[k].N; ++q) {
      const int p = perm[inst[k].foff + q];
      if (p < 0 || p >= fs[k].M * fs[k].N || seen[inst[k].foff + p]++) return -4.0;  // a permutation
    }
  if (nd_flow_solve_host<M>(rec, list[0], list[1], f, xs.data(), std::max<int64_t>(1, w)) != 0) return -3.0;
  double worst = 0.0;
  for (int k = 0; k < ni; ++k) {
    std::vector<double> r((size_t)fs[k].M * fs[k].N), x(r.size());
    for (size_t q = 0; q < r.size(); ++q) r[q] = f[inst[k].foff + perm[inst[k].foff + q]];
    nd_solve_host(fs[k], r.data(), x.data(), elem == 2);
    double d = 0.0, m = 0.0;
    for (size_t q = 0; q < r.size(); ++q) {
      d = std::max(d, std::fabs(xs[inst[k].foff + q] - x[q]));
      m = std::max(m, std::fabs(x[q]));
    }
    worst = std::max(worst, d / m);
  }
  return worst;
}

int main(int argc, char** argv) {
  if (argc < 7) return 2;
  const int leaf = std::atoi(argv[5]), units = std::atoi(argv[6]);
  std::vector<NdFactor> fs(2);
  std::vector<int> Ns;
  for (int k = 0; k < 2; ++k) {
    const int M = std::atoi(argv[1 + 2 * k]), N = std::atoi(argv[2 + 2 * k]);
    Op op = random_op(M, N, 11 + k);
    std::string why;
    if (!nd_build(M, N, coef, &op, leaf, 4, true, fs[k], why)) {
      std::printf("FAIL %s\n", why.c_str());
      return 1;
    }
    Ns.push_back(N);
  }
  const double a = run<float>(fs, Ns, units), b = run<double>(fs, Ns, units);
  std::printf("%s %.3e %.3e\n", a < 0.0 || b < 0.0 ? "FAIL" : "OK", a, b);
  return 0;
}
