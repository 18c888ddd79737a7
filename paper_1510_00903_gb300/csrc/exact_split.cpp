// exact_split.cpp -- which block-pair products of the FP64-accurate paths run
// as digit-sliced tensor-core products (tc_exact.cu).
//
// Two task forms of the planner (Sec. 3 Eq. LN.pLLp.FFT) are matrix products
// whose operands are shared by many tasks:
//   trace form (4 x 4 spins, 12 x 12 open indices): tr(M_A(q) M_B(-q)) of whole
//     12 x 12 blocks, over all such blocks one nb x nb product of 144 terms;
//     G(-q) = G(q)^T, so one product serves a pair {q, -q};
//   slice form (8 x 2 or 2 x 8 spins, 12 x 3 open indices): 36 consecutive rows
//     of one block against 36 of another, one nA x nB product per q.
// Every product the tasks need gets its place in the product buffer P through
// the item tables; tasks with few open indices are made one product per thread.
// A plan with any other task (or more operands than the kernel holds) keeps the
// CUDA-core products of field-major blocks.
#include <algorithm>
#include <map>
#include <set>

#include "kernels.cuh"
#include "planner.hpp"

namespace bbc {

namespace {

constexpr int kTraceForm[6] = {12, 12, 12, 1, 1, 12};  // n1, n2, sA1, sA2, sB1, sB2
constexpr int kSliceForm[6] = {12, 3, 1, 12, 1, 12};

bool has_form(const PairTask& t, const int (&f)[6]) {
  return t.n1 == f[0] && t.n2 == f[1] && t.sA1 == f[2] && t.sA2 == f[3] && t.sB1 == f[4] && t.sB2 == f[5];
}

int index_of(const std::vector<int>& v, int x) { return (int)(std::lower_bound(v.begin(), v.end(), x) - v.begin()); }

}  // namespace

void make_exact_split(const Plan& plan, ExactSplit* out) {
  ExactSplit S;
  const int n = (int)plan.tasks.size();
  S.done.assign(n, 0);
  *out = ExactSplit();
  if (n * 16 > 32767) return;  // the item tables hold 16-bit indices
  // trace form
  std::set<int> blocks;
  for (const PairTask& t : plan.tasks)
    if (t.nA == 4 && t.nB == 4 && has_form(t, kTraceForm))
      for (int r = 0; r < 4; r++) {
        blocks.insert(t.offA[r]);
        blocks.insert(t.offB[r]);
      }
  ExactSet& T = S.trace;
  if (!blocks.empty() && (int)blocks.size() <= kExactMaxBlocks) {
    T.rowA.assign(blocks.begin(), blocks.end());
    T.rowB = T.rowA;
    T.nAp = T.nBp = ((int)blocks.size() + 15) / 16 * 16;
    T.itemQ.assign((size_t)T.nAp * T.nBp, -1);
    for (int ti = 0; ti < n; ti++) {
      const PairTask& t = plan.tasks[ti];
      if (!(t.nA == 4 && t.nB == 4 && has_form(t, kTraceForm))) continue;
      std::vector<size_t> at;
      for (int ra = 0; ra < 4; ra++)
        for (int rb = 0; rb < 4; rb++) at.push_back((size_t)index_of(T.rowA, t.offA[ra]) * T.nBp + index_of(T.rowB, t.offB[rb]));
      bool free_all = std::set<size_t>(at.begin(), at.end()).size() == 16;
      for (size_t a : at) free_all &= T.itemQ[a] < 0;
      if (!free_all) continue;  // a second task on the same products stays on the CUDA cores
      for (int i = 0; i < 16; i++) T.itemQ[at[i]] = (short)(16 * ti + i);
      S.done[ti] = 1;
    }
    T.itemNQ.assign(T.itemQ.size(), -1);
    for (int i = 0; i < T.nAp; i++)
      for (int j = 0; j < T.nBp; j++) T.itemNQ[(size_t)i * T.nBp + j] = T.itemQ[(size_t)j * T.nBp + i];
  }
  // slice form: the 8-side's rows are A, the 2-side's B; a 2 x 8 task reads B at
  // q and A at -q, so its product belongs to the place of -q
  auto slice = [&](const PairTask& t, const int** a8, const int** b2, bool* swapped) {
    if (!has_form(t, kSliceForm) || !((t.nA == 8 && t.nB == 2) || (t.nA == 2 && t.nB == 8))) return false;
    *swapped = t.nA == 2;
    *a8 = *swapped ? t.offB : t.offA;
    *b2 = *swapped ? t.offA : t.offB;
    return true;
  };
  std::set<int> rowsA, rowsB;
  for (const PairTask& t : plan.tasks) {
    const int *a8, *b2;
    bool sw;
    if (!slice(t, &a8, &b2, &sw)) continue;
    rowsA.insert(a8, a8 + 8);
    rowsB.insert(b2, b2 + 2);
  }
  ExactSet& C = S.slice;
  if (!rowsA.empty() && (int)rowsA.size() <= kExactMaxSliceA && (int)rowsB.size() <= kExactMaxSliceB) {
    C.rowA.assign(rowsA.begin(), rowsA.end());
    C.rowB.assign(rowsB.begin(), rowsB.end());
    C.nAp = ((int)rowsA.size() + 15) / 16 * 16;
    C.nBp = ((int)rowsB.size() + 15) / 16 * 16;
    C.itemQ.assign((size_t)C.nAp * C.nBp, -1);
    C.itemNQ.assign((size_t)C.nAp * C.nBp, -1);
    for (int ti = 0; ti < n; ti++) {
      const PairTask& t = plan.tasks[ti];
      const int *a8, *b2;
      bool sw;
      if (!slice(t, &a8, &b2, &sw)) continue;
      std::vector<short>& items = sw ? C.itemNQ : C.itemQ;
      bool free_all = true;
      std::set<size_t> seen;
      for (int a = 0; a < 8; a++)
        for (int b = 0; b < 2; b++) {
          const size_t at = (size_t)index_of(C.rowA, a8[a]) * C.nBp + index_of(C.rowB, b2[b]);
          free_all &= items[at] < 0 && seen.insert(at).second;
        }
      if (!free_all) continue;
      for (int a = 0; a < 8; a++)
        for (int b = 0; b < 2; b++)
          items[(size_t)index_of(C.rowA, a8[a]) * C.nBp + index_of(C.rowB, b2[b])] =
              (short)(16 * ti + (sw ? b * 8 + a : a * 2 + b));
      S.done[ti] = 1;
    }
  }
  // exponent jobs (first row, rows): one per trace block, and one per slice that
  // lies in no trace block (a slice inside one shares its exponent)
  std::map<std::pair<int, int>, int> job_of;
  auto job = [&](int first, int rows) {
    auto it = job_of.find({first, rows});
    if (it != job_of.end()) return it->second;
    const int id = (int)(S.jobs.size() / 2);
    S.jobs.push_back(first);
    S.jobs.push_back(rows);
    job_of[{first, rows}] = id;
    return id;
  };
  for (int r : T.rowA) T.expA.push_back(job(r, 144));
  T.expB = T.expA;
  auto slice_job = [&](int r) {
    auto it = std::upper_bound(T.rowA.begin(), T.rowA.end(), r);
    if (it != T.rowA.begin() && r + 36 <= *(it - 1) + 144) return job(*(it - 1), 144);
    return job(r, 36);
  };
  for (int r : C.rowA) C.expA.push_back(slice_job(r));
  for (int r : C.rowB) C.expB.push_back(slice_job(r));
  if (S.jobs.empty()) return;
  // every operand row lies inside the block rows, at an even row (32-byte loads)
  bool ok = plan.n_out % 2 == 0;
  auto inside = [&](const std::vector<int>& rows, int len) {
    for (int r : rows) ok &= r >= 0 && r % 2 == 0 && r + len <= plan.n_out;
  };
  inside(T.rowA, 144);
  inside(C.rowA, 36);
  inside(C.rowB, 36);
  for (int ti = 0; ti < n; ti++) {
    const PairTask& t = plan.tasks[ti];
    if (S.done[ti]) continue;
    if (t.n1 * t.n2 > kExactSmallSteps) return;
    S.small.push_back(ti);
  }
  S.all = ok;
  *out = std::move(S);
}

}  // namespace bbc
