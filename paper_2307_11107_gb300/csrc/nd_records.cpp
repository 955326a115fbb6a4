// Task records of the nested-dissection dataflow sweeps (see nd_records.h).
#include "nd_records.h"

#include <algorithm>
#include <cstring>

namespace apic {
namespace {

constexpr int kWarpS = 64, kWarpU = 192;  // a warp's vector areas

bool has_gather(const NdFront& F) { return F.child[0] >= 0 || F.child[1] >= 0; }

// Shape of a task's dot products: vectors of a row, lanes per row (as a power
// of two) and the padded row stride in vectors.
struct Shape {
  int vecs, lg, sum, stride;
};

Shape shape_of(const NdFront& F, bool fwd, int elem, bool sum8) {
  const int cols = fwd ? F.s : F.u, per = 4 / elem;
  Shape h{(cols + per - 1) / per, 0, 0, 0};
  // partial sums: 4 up to 4 vectors, 8 up to 8, 16 up to 16, else 32
  h.sum = h.vecs > 16 ? 5 : (h.vecs > 8 ? 4 : (h.vecs > 4 ? 3 : 2));
  if (!fwd && sum8 && F.s <= kNdTinyS && F.u <= kNdTinyU) h.sum = 3;
  // lanes: one per row with up to eight partial sums each, two, four, or (rows
  // of more than 64 vectors, of which a record holds few) a warp
  h.lg = h.sum <= 3 ? 0 : (h.sum == 4 ? 1 : (h.vecs > 64 ? 5 : 2));
  const int G = 1 << h.lg;
  h.stride = h.vecs;
  if (G < 8)
    while (h.stride % (2 * G) != G) ++h.stride;
  return h;
}

// Words of one front's entry, tables and matrix in a record that holds rows
// [r0, r0 + nr) of it (all rows for kinds 1 and 2).
int front_words(const NdFront& F, bool fwd, int r0, int nr, int elem, bool sum8) {
  const int mat = 4 * nr * shape_of(F, fwd, elem, sum8).stride;
  int w = kNdEntry;
  if (fwd) {
    const int nu = std::max(0, r0 + nr - std::max(r0, F.s));
    w += (has_gather(F) ? 2 * (F.s + nu) : 0) + mat;
  } else {
    w += nr + F.u + ((nr + F.u) & 1) + (F.u > 0 ? mat : 0);
  }
  return w + 3;  // the matrix starts on four words
}

int rows_of(const NdFront& F, bool fwd) { return fwd ? F.s + F.u : F.s; }

}  // namespace

bool nd_flow_tasks(const NdUpload& up, int front0, int nf, int depth, int inst, bool fwd, int elem, int units,
                   int vec_cap, int sum8, std::vector<NdFlowTask>& tasks) {
  auto large = [&](const NdFront& F) {
    return F.s > kWarpS || F.u > kWarpU ||
           4 * rows_of(F, fwd) * shape_of(F, fwd, elem, false).stride > kNdFlowWarpWords;
  };
  auto tiny0 = [&](const NdFront& F) { return F.s <= kNdTinyS && F.u <= kNdTinyU && !large(F); };
  const int c = std::max(1, units);
  for (int l = 0; l <= depth; ++l) {
    int q = 0;
    while (q < nf && up.fronts[front0 + q].level != l) ++q;
    int small = 0, nt = 0, ns = 0;
    for (int z = q; z < nf && up.fronts[front0 + z].level == l; ++z) {
      small += !large(up.fronts[front0 + z]);
      nt += tiny0(up.fronts[front0 + z]);
      ns += up.fronts[front0 + z].s <= kNdTinyS && up.fronts[front0 + z].u <= kNdTinyU;
    }
    // tiny fronts four to a warp when that still leaves every worker some,
    // else one to a warp like the small ones
    const bool use_tiny = nt >= 4 * c;
    // (the eight lanes of a tiny front run rows of their own number: one lane a row)
    const bool s8 = ns >= sum8 || use_tiny;
    const int per = std::max(1, std::min(kNdFlowWarps, (small + c - 1) / c));
    const int per_tiny = std::max(1, std::min(4 * kNdFlowWarps, (nt + c - 1) / c));
    while (q < nf && up.fronts[front0 + q].level == l) {
      const NdFront& F = up.fronts[front0 + q];
      if (large(F)) {
        if (std::max(F.sp, F.up) > vec_cap) return false;
        const int rows = rows_of(F, fwd);
        for (int r = 0; r < rows;) {
          int n = std::min(kNdFlowRows, rows - r);
          while (n > 0 && kNdHead + front_words(F, fwd, r, n, elem, s8) > kNdFlowStage) --n;
          if (n < 1) return false;
          tasks.push_back(NdFlowTask{front0 + q, r, n, 0, l, inst, fwd, s8, 0});
          r += n;
        }
        ++q;
        continue;
      }
      const bool t = use_tiny && tiny0(F);
      const int cap = t ? per_tiny : per;
      int n = 0, w = kNdHead;
      while (q + n < nf && n < cap) {
        const NdFront& G = up.fronts[front0 + q + n];
        if (G.level != l || large(G) || (use_tiny && tiny0(G)) != t) break;
        const int g = front_words(G, fwd, 0, rows_of(G, fwd), elem, s8);
        if (w + g > kNdFlowStage) break;
        w += g;
        ++n;
      }
      if (n < 1) return false;
      tasks.push_back(NdFlowTask{front0 + q, 0, n, t ? 2 : 1, l, inst, fwd, s8, 0});
      q += n;
    }
  }
  for (NdFlowTask& T : tasks) {
    if (T.inst != inst || T.fwd != fwd) continue;
    int w = kNdHead;
    if (T.kind == 0) w += front_words(up.fronts[T.front], fwd, T.r0, T.n, elem, T.sum8);
    else
      for (int k = 0; k < T.n; ++k) {
        const NdFront& G = up.fronts[T.front + k];
        w += front_words(G, fwd, 0, rows_of(G, fwd), elem, T.sum8);
      }
    T.words = (w + 3) & ~3;
  }
  return true;
}

void nd_flow_places(const NdUpload& up, int front0, int nf, int64_t unknowns, std::vector<int32_t>& place,
                    std::vector<int32_t>& perm) {
  const size_t base = perm.size();
  perm.resize(base + (size_t)unknowns, 0);
  int p = 0;
  for (int q = front0; q < front0 + nf; ++q) {
    const NdFront& F = up.fronts[q];
    place.push_back(p);
    for (int a = 0; a < F.s; ++a) perm[base + up.idx[F.S + a]] = p + a;
    p += F.s;
  }
}

bool nd_flow_add(NdFlowPlan& P, const NdFactor* f, int64_t unknowns, int elem, int units, int vec_cap, int sum8) {
  const int inst = (int)P.depth.size(), f0 = (int)P.up.fronts.size();
  P.words.push_back(P.words.back());
  P.depth.push_back(f ? f->depth : 0);
  bool ok = true;
  if (f) {
    NdLevels lv;
    nd_layout(*f, 0, P.w, kWarpS, kWarpU, 2048, 8192, 512, 4, 8192, 1, P.up, lv);  // (its level-by-level tasks are not used)
    const size_t t0 = P.tasks.size();
    for (int sw = 0; sw < 2 && ok; ++sw)
      ok = nd_flow_tasks(P.up, f0, (int)P.up.fronts.size() - f0, f->depth, inst, sw == 0, elem, units, vec_cap, sum8,
                         P.tasks);
    for (size_t t = t0; t < P.tasks.size(); ++t) {
      P.off.push_back(P.words.back());
      P.words.back() += P.tasks[t].words;
    }
    P.w += (f->w_total + 63) & ~63ll;
  }
  nd_flow_places(P.up, f0, (int)P.up.fronts.size() - f0, unknowns, P.place, P.perm);
  P.rows += unknowns;
  return ok && P.words.back() / 4 < (1ll << 31) && P.rows + P.w < (1ll << 31);
}

void nd_flow_lists(NdFlowPlan& P) {
  std::vector<int> v[2];
  for (size_t t = 0; t < P.tasks.size(); ++t) v[P.tasks[t].fwd ? 0 : 1].push_back((int)t);
  auto key = [&](int t) {
    const NdFlowTask& T = P.tasks[t];
    return std::make_pair(T.fwd ? P.depth[T.inst] - T.level : T.level, T.inst);
  };
  P.list.clear();
  for (std::vector<int>& q : v) {
    std::stable_sort(q.begin(), q.end(), [&](int a, int b) { return key(a) < key(b); });
    for (int t : q)
      P.list.push_back(NdFlowEntry{(int)(P.off[t] / 4), 4 * P.tasks[t].words, P.tasks[t].inst, P.tasks[t].kind});
  }
  P.nf = (int)v[0].size();
  P.nb = (int)v[1].size();
}

void nd_transpose64(NdFactor& f) {
  for (const NdFront& F : f.fronts) {
    double *a = f.fm64.data() + F.FM, *b = f.nb64.data() + F.NB;
    for (int r = 0; r < F.s; ++r)
      for (int c = 0; c < r; ++c) std::swap(a[(int64_t)r * F.sp + c], a[(int64_t)c * F.sp + r]);
    for (int r = 0; r < F.s; ++r)
      for (int q = 0; q < F.u; ++q) std::swap(b[(int64_t)r * F.up + q], a[(int64_t)(F.s + q) * F.sp + r]);
  }
}

template <class M>
void nd_flow_write(const NdUpload& up, const NdFlowTask& T, const std::vector<int32_t>& place, const int32_t* perm,
                   const NdFlowInst& I, const M* fm,
                   int64_t fm0, const M* nb, int64_t nb0, int32_t* out) {
  const int elem = (int)(sizeof(M) / sizeof(int32_t));
  std::memset(out, 0, sizeof(int32_t) * (size_t)T.words);
  const int nfr = T.kind == 0 ? 1 : T.n;
  out[0] = T.kind;
  out[1] = nfr;
  out[2] = I.N;
  out[3] = I.foff;
  out[4] = I.node_off;
  int pos = kNdHead + kNdEntry * nfr;
  for (int k = 0; k < nfr; ++k) {
    const NdFront& F = up.fronts[T.front + k];
    int32_t* E = out + kNdHead + kNdEntry * k;
    const int r0 = T.kind == 0 ? T.r0 : 0, nr = T.kind == 0 ? T.n : rows_of(F, T.fwd);
    E[kNdS] = F.s;
    E[kNdU] = F.u;
    const Shape h = shape_of(F, T.fwd, elem, T.sum8);
    E[kNdStride] = h.stride;
    E[kNdVecs] = h.vecs;
    E[kNdLgSum] = h.sum;
    E[kNdLg] = h.lg | (has_gather(F) ? kNdHas : 0);
    E[kNdW] = (int32_t)F.W;
    // a front's last update entry, or separator row
    auto rep = [&](int q) {
      if (q < 0) return -1;
      const NdFront& G = up.fronts[q];
      return T.fwd ? (G.u > 0 ? (int32_t)(G.W + G.u - 1) : -1) : place[q] + G.s - 1;
    };
    E[kNdRep0] = rep(T.fwd ? F.child[0] : F.parent);
    E[kNdRep1] = T.fwd ? rep(F.child[1]) : -1;
    E[kNdR0] = r0;
    E[kNdNr] = nr;
    E[kNdP0] = place[T.front + k];
    E[kNdTab] = pos;
    if (T.fwd) {
      if (has_gather(F)) {
        for (int p = 0; p < 2 * F.s; ++p) out[pos++] = up.gather[F.G + p];
        for (int a = std::max(r0, F.s); a < r0 + nr; ++a) {
          out[pos++] = up.gather[F.G + 2 * a];
          out[pos++] = up.gather[F.G + 2 * a + 1];
        }
      }
    } else {
      for (int p = 0; p < F.u; ++p) out[pos++] = perm[up.idx[F.U + p]];
      for (int a = r0; a < r0 + nr; ++a) out[pos++] = up.idx[F.S + a];
      pos += pos & 1;
    }
  }
  for (int k = 0; k < nfr; ++k) {
    const NdFront& F = up.fronts[T.front + k];
    int32_t* E = out + kNdHead + kNdEntry * k;
    pos = (pos + 3) & ~3;
    E[kNdMat] = pos;
    const int cols = T.fwd ? F.s : F.u, width = T.fwd ? F.sp : F.up, stride = 4 * E[kNdStride];
    const M* src = T.fwd ? fm + (F.FM - fm0) + (int64_t)E[kNdR0] * F.sp : nb + (F.NB - nb0) + (int64_t)E[kNdR0] * F.up;
    for (int a = 0; a < E[kNdNr] && cols > 0; ++a, pos += stride)
      std::memcpy(out + pos, src + (int64_t)a * width, sizeof(M) * (size_t)cols);
  }
}

template <class M>
int64_t nd_flow_solve_host(const std::vector<int32_t>& rec, const std::vector<int64_t>& fwd_list,
                           const std::vector<int64_t>& back_list, const std::vector<M>& f, double* x, int64_t wn) {
  std::vector<M> z(f.size(), M(0)), e(f.size(), M(0)), w((size_t)wn, M(0));
  std::vector<char> has_z(f.size(), 0), has_e(f.size(), 0), has_w((size_t)wn, 0);
  int64_t late = 0;
  for (int sw = 0; sw < 2; ++sw) {
    const bool fwd = sw == 0;
    for (int64_t off : fwd ? fwd_list : back_list) {
      if (off % 4 || off + kNdHead > (int64_t)rec.size()) return -1;
      const int32_t* R = rec.data() + off;
      const int64_t fo = R[3];
      if (R[1] < 1 || R[1] > (R[0] == 0 ? 1 : (R[0] == 1 ? kNdFlowWarps : 4 * kNdFlowWarps))) return -1;
      for (int k = 0; k < R[1]; ++k) {
        const int32_t* E = R + kNdHead + kNdEntry * k;
        const int s = E[kNdS], u = E[kNdU], r0 = E[kNdR0], nr = E[kNdNr], per = 16 / (int)sizeof(M);
        const int st = per * E[kNdStride], nc = per * E[kNdVecs], lg = E[kNdLg] & 255;
        const bool has = (E[kNdLg] & kNdHas) != 0;
        const M* m = (const M*)(R + E[kNdMat]);
        if (E[kNdMat] % 4 || E[kNdMat] + (fwd || u > 0 ? 4 * nr * E[kNdStride] : 0) > kNdFlowStage) return -1;
        if (nc < (fwd ? s : u) || st < nc || (R[0] == 2 && lg)) return -1;
        const int sum = E[kNdLgSum];  // the forms rows_any (nd_solve.cu) knows
        if (!((lg == 0 && (sum == 2 || sum == 3)) || (lg == 1 && sum == 4) || (sum == 5 && (lg == 2 || lg == 5)))) return -1;
        if (sum == 2 && E[kNdVecs] > 4) return -1;
        if (R[0] == 2 && (s > kNdTinyS || u > kNdTinyU)) return -1;
        if (R[0] == 1 && (s > kWarpS || u > kWarpU)) return -1;
        if (R[0] == 0 && nr > kNdFlowRows) return -1;
        for (int q = 0; q < 2; ++q) {
          const int rp = E[kNdRep0 + q];
          if (rp >= 0 && !(fwd ? has_w[rp] : has_e[fo + rp])) ++late;
        }
        const int32_t* tab = R + E[kNdTab];
        std::vector<M> v(std::max(nc, 1), M(0));
        if (fwd) {
          if (has && (tab - R) % 2) return -1;  // pairs are read as 8-byte words
          auto pair = [&](const int32_t* p) {
            M sum = M(0);
            for (int c = 0; c < 2; ++c)
              if (p[c] >= 0) {
                late += !has_w[p[c]];
                sum += w[p[c]];
              }
            return sum;
          };
          for (int p = 0; p < s; ++p) v[p] = f[fo + E[kNdP0] + p] + (has ? pair(tab + 2 * p) : M(0));
          for (int a = r0; a < r0 + nr; ++a) {
            M acc = M(0);
            for (int t = 0; t < nc; ++t) acc += m[(int64_t)(a - r0) * st + t] * v[t];
            if (a < s) {
              late += has_z[fo + E[kNdP0] + a]++;
              z[fo + E[kNdP0] + a] = acc;
            } else {
              late += has_w[E[kNdW] + a - s]++;
              w[E[kNdW] + a - s] = (has ? pair(tab + 2 * (s + a - std::max(r0, s))) : M(0)) - acc;
            }
          }
        } else {
          for (int p = 0; p < u; ++p) {
            late += !has_e[fo + tab[p]];
            v[p] = e[fo + tab[p]];
          }
          for (int a = 0; a < nr; ++a) {
            M acc = M(0);
            for (int t = 0; t < nc && u > 0; ++t) acc += m[(int64_t)a * st + t] * v[t];
            const int64_t at = fo + E[kNdP0] + r0 + a;
            late += !has_z[at];
            late += has_e[at]++;
            e[at] = z[at] - acc;
            x[fo + tab[u + a]] += (double)e[at];
          }
        }
      }
    }
  }
  return late;
}

template void nd_flow_write<float>(const NdUpload&, const NdFlowTask&, const std::vector<int32_t>&, const int32_t*,
                                   const NdFlowInst&, const float*, int64_t, const float*, int64_t, int32_t*);
template void nd_flow_write<double>(const NdUpload&, const NdFlowTask&, const std::vector<int32_t>&, const int32_t*,
                                    const NdFlowInst&, const double*, int64_t, const double*, int64_t, int32_t*);
template int64_t nd_flow_solve_host<float>(const std::vector<int32_t>&, const std::vector<int64_t>&,
                                           const std::vector<int64_t>&, const std::vector<float>&, double*, int64_t);
template int64_t nd_flow_solve_host<double>(const std::vector<int32_t>&, const std::vector<int64_t>&,
                                            const std::vector<int64_t>&, const std::vector<double>&, double*, int64_t);

}  // namespace apic
