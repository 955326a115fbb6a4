// Task records of the nested-dissection dataflow sweeps (nd_solve.cu): every
// task's static data (its fronts' sizes, node indices and gather tables, then
// its matrix rows) in one contiguous run of words, so that
// one bulk copy brings a task whole into shared memory before it runs.
// Host-only C++.
#pragma once
#include <cstdint>
#include <vector>

#include "nd_factor.h"

namespace apic {

// A record, in 32-bit words:
//   [0] kind, [1] fronts, [2] N, [3] first unknown of the instance, [4] its
//   first node, [5..7] unused; then one entry of kNdEntry words per front;
//   then the tables; then, from a multiple of four words, the matrix rows.
// Kinds: 0 rows [r0, r0 + nr) of one front by all warps of a worker, 1 up to
// kNdFlowWarps fronts, one per warp (front k by warp k), 2 up to
// 4 kNdFlowWarps tiny fronts, one per 8-lane group (front k by warp
// k % kNdFlowWarps, group k / kNdFlowWarps).
// The right-hand side and the correction are kept front by front: a front's
// separator has consecutive places from kNdP0 on (nd_flow_places).
// Tables, forward: unless the front is a leaf the gather pairs (offsets into
// the update vectors, -1: none) of its separator [2 s] and of the task's
// update rows [2 each].  Backward: the places of the update set [u], then the
// unknowns of the task's separator rows [nr].
// kNdRep0, kNdRep1: an entry of what each child (forward: its update vector)
// or the parent (backward: its separator) writes last, to wait for (-1: none).
// Matrix, forward: rows of [F_SS^-1; F_US F_SS^-1]; backward: rows of
// F_SS^-1 F_SU (none when u = 0).  A row of kNdVecs 16-byte vectors is summed
// in a form that does not depend on how the rows are shared out: vector t goes
// to partial sum t mod 2^kNdLgSum, and the partial sums are added in a tree.
// 2^kNdLg lanes share a row; the row stride is padded so that eight
// neighbouring lanes' 16-byte loads fall into different shared-memory banks.
constexpr int kNdHead = 8, kNdEntry = 16;
enum NdEntryWord {
  kNdS, kNdU, kNdStride /* 16-byte vectors */, kNdW, kNdRep0, kNdRep1, kNdTab, kNdMat, kNdR0, kNdNr, kNdP0,
  kNdVecs, kNdLg, /* + kNdHas unless the front is a leaf */
  kNdLgSum
};
constexpr int kNdHas = 0x100;
constexpr int kNdFlowWarps = 4;       // warps of a worker
constexpr int kNdFlowStage = 4480;    // words of a record at most
constexpr int kNdFlowRows = 256;      // rows of a kind-0 task at most
constexpr int kNdFlowWarpWords = 1536;  // matrix words of a front that one warp takes at most

struct NdFlowTask {
  int front, r0, n, kind;  // as NdTask (n: rows of kind 0, fronts otherwise)
  int level, inst;
  bool fwd, sum8;  // sum8: eight partial sums for backward rows of tiny fronts
  int words;
};

// Tasks of instance `inst` (its fronts are up.fronts [front0, front0 + nf),
// level by level) for one sweep, `elem` words per matrix element, spread over
// `units` workers; appended to `tasks`.  vec_cap: elements of a kind-0 front's
// vector the device holds.  sum8: the tiny fronts of a level from which on
// their backward rows take eight partial sums whatever their length (the FP32
// sums of the level-by-level sweeps, kept bit for bit).  False: a front does
// not fit.
bool nd_flow_tasks(const NdUpload& up, int front0, int nf, int depth, int inst, bool fwd, int elem, int units,
                   int vec_cap, int sum8, std::vector<NdFlowTask>& tasks);

// Appends the first places of the fronts [front0, front0 + nf) of one instance
// to `place` and the places of its `unknowns` unknowns to `perm`.
void nd_flow_places(const NdUpload& up, int front0, int nf, int64_t unknowns, std::vector<int32_t>& place,
                    std::vector<int32_t>& perm);

struct NdFlowInst {
  int N, foff, node_off;
};

// Writes task T's record (T.words words) at out.  fm, nb: the instance's
// matrices, of element type M (float or double), with fm0, nb0 the values of
// NdFront::FM, NB that they start at; perm: the instance's places.
template <class M>
void nd_flow_write(const NdUpload& up, const NdFlowTask& T, const std::vector<int32_t>& place, const int32_t* perm,
                   const NdFlowInst& I, const M* fm,
                   int64_t fm0, const M* nb, int64_t nb0, int32_t* out);

// A list entry, same layout as CUDA's int4: a record's first word / 4, its
// bytes, instance and kind.
struct NdFlowEntry {
  int at, bytes, inst, kind;
};

// The records of a batch: instances are added in order, then the lists made.
struct NdFlowPlan {
  NdUpload up;
  std::vector<NdFlowTask> tasks;        // instance by instance
  std::vector<int64_t> off;             // their first words
  std::vector<int64_t> words{0};        // first word of each instance's records (and the end)
  std::vector<int32_t> place, perm;     // nd_flow_places
  std::vector<int> depth;               // of each instance's tree
  std::vector<NdFlowEntry> list;        // the forward sweep's entries, then the backward one's
  int nf = 0, nb = 0;
  int64_t rows = 0, w = 0;              // unknowns and update-vector entries so far
};

// Adds f as the next instance (its right-hand side at P.rows, its update
// vectors at P.w); unknowns: M N, also where the instance has no fronts (f
// null).  False: a front does not fit, or an offset exceeds 31 bits.
bool nd_flow_add(NdFlowPlan& P, const NdFactor* f, int64_t unknowns, int elem, int units, int vec_cap, int sum8);

// The lists, forward from the deepest tree level, backward from the root:
// every record after those it reads from.
void nd_flow_lists(NdFlowPlan& P);

// The fronts of the transposed system in place (FP64): those of A^T are the
// transposes of A's, F_SS^-T and, as the lower block, (F_SS^-1 F_SU)^T; the
// lower block's transpose in place of F_SS^-1 F_SU.
void nd_transpose64(NdFactor& f);

// The sweeps as the device runs them, record by record in list order (offsets
// in words into rec): f in places, x += A^-1 f for the unknowns of every
// instance, w: the update vectors' total.  Returns the entries that were read
// before they were written (0 in a valid order) or written twice, or -1 for a
// record that breaks a limit.
template <class M>
int64_t nd_flow_solve_host(const std::vector<int32_t>& rec, const std::vector<int64_t>& fwd_list,
                           const std::vector<int64_t>& back_list, const std::vector<M>& f, double* x, int64_t w);

}  // namespace apic
