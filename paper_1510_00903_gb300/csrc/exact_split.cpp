// exact_split.cpp -- which block-pair products run as digit-sliced tensor-core
// products (tc_exact.cu).
//
// Most tasks of the planner (Sec. 3 Eq. LN.pLLp.FFT) have forms that are matrix
// products whose operands are shared by many tasks:
//   trace forms (4 x 4 spins, 12 x 12 open indices): sums over whole 12 x 12
//     blocks, tr(M_A(q) M_B(-q)) or the same without the transpose, over all such
//     blocks one nb x nb product of 144 terms; G(-q) = G(q)^T, so one product
//     serves a pair {q, -q};
//   slice forms (8 x 2 or 2 x 8 spins, 12 x 3 open indices): 36 consecutive rows
//     of one block (or three columns of it) against 36 consecutive rows of
//     another, one nA x nB product per q.
// Every product the tasks need gets its place in the product buffer P through
// the item tables; tasks with few open indices are made one product per thread.
// A plan with any other task (or more operands than the kernel holds) keeps the
// CUDA-core products, and so does one that they serve faster (exact_pays).
#include <algorithm>
#include <cmath>
#include <iterator>
#include <map>
#include <set>

#include "kernels.cuh"
#include "planner.hpp"

namespace bbc {

namespace {

// n1, n2, sA1, sA2, sB1, sB2
constexpr int kTraceForms[2][6] = {{12, 12, 12, 1, 1, 12}, {12, 12, 12, 1, 12, 1}};
// slices, seen from the 8-spin side: both of consecutive rows, or the 8-side of columns
constexpr int kSliceForms[2][6] = {{12, 3, 1, 12, 1, 12}, {12, 3, 12, 1, 1, 12}};

bool has_form(const PairTask& t, const int (&f)[6], bool swapped) {
  return t.n1 == f[0] && t.n2 == f[1] && (swapped ? t.sB1 : t.sA1) == f[2] && (swapped ? t.sB2 : t.sA2) == f[3] &&
         (swapped ? t.sA1 : t.sB1) == f[4] && (swapped ? t.sA2 : t.sB2) == f[5];
}

int index_of(const std::vector<int>& v, int x) { return (int)(std::lower_bound(v.begin(), v.end(), x) - v.begin()); }

// trace form f: operands, item tables, done tasks
void trace_set(const Plan& plan, int f, ExactSet* T, std::vector<char>* done) {
  const int n = (int)plan.tasks.size();
  auto is = [&](const PairTask& t) { return t.nA == 4 && t.nB == 4 && has_form(t, kTraceForms[f], false); };
  std::set<int> blocks;
  for (const PairTask& t : plan.tasks)
    if (is(t))
      for (int r = 0; r < 4; r++) {
        blocks.insert(t.offA[r]);
        blocks.insert(t.offB[r]);
      }
  if (blocks.empty() || (int)blocks.size() > kExactMaxBlocks) return;
  T->rowA.assign(blocks.begin(), blocks.end());
  T->rowB = T->rowA;
  T->nAp = T->nBp = ((int)blocks.size() + 15) / 16 * 16;
  T->itemQ.assign((size_t)T->nAp * T->nBp, -1);
  for (int ti = 0; ti < n; ti++) {
    const PairTask& t = plan.tasks[ti];
    if (!is(t)) continue;
    std::set<size_t> seen;
    std::vector<size_t> at;
    bool free_all = true;
    for (int ra = 0; ra < 4; ra++)
      for (int rb = 0; rb < 4; rb++) {
        at.push_back((size_t)index_of(T->rowA, t.offA[ra]) * T->nBp + index_of(T->rowB, t.offB[rb]));
        free_all &= T->itemQ[at.back()] < 0 && seen.insert(at.back()).second;
      }
    if (!free_all) continue;  // a second task on the same products: not for this kernel
    for (int i = 0; i < 16; i++) T->itemQ[at[i]] = (short)(16 * ti + i);
    (*done)[ti] = 1;
  }
  T->itemNQ.assign(T->itemQ.size(), -1);
  for (int i = 0; i < T->nAp; i++)
    for (int j = 0; j < T->nBp; j++) T->itemNQ[(size_t)i * T->nBp + j] = T->itemQ[(size_t)j * T->nBp + i];
}

// slice form f: the 8-side's rows are A, the 2-side's B; a 2 x 8 task reads B at
// q and A at -q, so its product belongs to the place of -q
void slice_set(const Plan& plan, int f, ExactSet* C, std::vector<char>* done) {
  const int n = (int)plan.tasks.size();
  auto is = [&](const PairTask& t, const int** a8, const int** b2, bool* swapped) {
    *swapped = t.nA == 2 && t.nB == 8;
    if (!(*swapped || (t.nA == 8 && t.nB == 2)) || !has_form(t, kSliceForms[f], *swapped)) return false;
    *a8 = *swapped ? t.offB : t.offA;
    *b2 = *swapped ? t.offA : t.offB;
    return true;
  };
  std::set<int> rowsA, rowsB;
  const int *a8, *b2;
  bool sw;
  for (const PairTask& t : plan.tasks)
    if (is(t, &a8, &b2, &sw)) {
      rowsA.insert(a8, a8 + 8);
      rowsB.insert(b2, b2 + 2);
    }
  if (rowsA.empty() || (int)rowsA.size() > kExactMaxSliceA || (int)rowsB.size() > kExactMaxSliceB) return;
  C->rowA.assign(rowsA.begin(), rowsA.end());
  C->rowB.assign(rowsB.begin(), rowsB.end());
  C->nAp = ((int)rowsA.size() + 15) / 16 * 16;
  C->nBp = ((int)rowsB.size() + 15) / 16 * 16;
  C->itemQ.assign((size_t)C->nAp * C->nBp, -1);
  C->itemNQ.assign((size_t)C->nAp * C->nBp, -1);
  for (int ti = 0; ti < n; ti++) {
    if (!is(plan.tasks[ti], &a8, &b2, &sw)) continue;
    std::vector<short>& items = sw ? C->itemNQ : C->itemQ;
    std::set<size_t> seen;
    bool free_all = true;
    auto at = [&](int a, int b) { return (size_t)index_of(C->rowA, a8[a]) * C->nBp + index_of(C->rowB, b2[b]); };
    for (int a = 0; a < 8; a++)
      for (int b = 0; b < 2; b++) free_all &= items[at(a, b)] < 0 && seen.insert(at(a, b)).second;
    if (!free_all) continue;
    for (int a = 0; a < 8; a++)
      for (int b = 0; b < 2; b++) items[at(a, b)] = (short)(16 * ti + (sw ? b * 8 + a : a * 2 + b));
    (*done)[ti] = 1;
  }
}

}  // namespace

void make_exact_split(const Plan& plan, ExactSplit* out) {
  constexpr int align = 2;  // field rows per 32 bytes: operands are read in such pieces
  ExactSplit S;
  const int n = (int)plan.tasks.size();
  std::vector<char> done(n, 0);
  *out = ExactSplit();
  if (n * 16 > 32767) return;  // the item tables hold 16-bit indices
  for (int f = 0; f < 2; f++) {
    trace_set(plan, f, &S.set[kExactTrace + f], &done);
    slice_set(plan, f, &S.set[kExactSlice + f], &done);
  }
  // One exponent per operand row (first field row, rows or kExactColumns).  A slice
  // inside a trace block has its own: it is one Dirac component of an open index and
  // may be orders of magnitude smaller than the rest of the block.  Its rows are read
  // once, with the block's.
  using Job = std::pair<int, int>;
  std::map<Job, int> job_of;
  auto span = [](const Job& j) { return j.second == kExactColumns ? 11 * 12 + 3 : j.second; };
  for (int f = 0; f < 2; f++) {
    for (int r : S.set[f].rowA) job_of[{r, 144}] = 0;
    for (int r : S.set[kExactSlice + f].rowA) job_of[{r, f == 0 ? 36 : kExactColumns}] = 0;
    for (int r : S.set[kExactSlice + f].rowB) job_of[{r, 36}] = 0;
  }
  if (job_of.empty()) return;
  std::map<Job, std::vector<Job>> loads;
  for (const auto& j : job_of)
    if (j.first.second == 144) loads[j.first].push_back(j.first);
  for (const auto& j : job_of) {
    if (j.first.second == 144) continue;
    auto it = loads.upper_bound({j.first.first, 144});
    const bool inside = it != loads.begin() && j.first.first + span(j.first) <= span(std::prev(it)->first) + std::prev(it)->first.first;
    loads[inside ? std::prev(it)->first : Job(j.first.first, span(j.first))].push_back(j.first);
  }
  bool ok = plan.n_out % align == 0;
  for (const auto& l : loads) {
    const int id = (int)S.jobs.size() / 2, first = l.first.first;
    S.loads.insert(S.loads.end(), {first, l.first.second, id, id + (int)l.second.size()});
    // every operand row lies inside the block rows
    ok &= first >= 0 && first + l.first.second <= plan.n_out;
    for (const Job& j : l.second) {
      job_of[j] = (int)S.jobs.size() / 2;
      S.jobs.insert(S.jobs.end(), {j.first - first, j.second});
    }
  }
  for (int f = 0; f < 2; f++) {
    ExactSet& T = S.set[f];
    for (int r : T.rowA) {
      T.expA.push_back(job_of[{r, 144}]);
      ok &= r % align == 0;
    }
    T.expB = T.expA;
    ExactSet& C = S.set[kExactSlice + f];
    for (int r : C.rowA) {
      C.expA.push_back(job_of[{r, f == 0 ? 36 : kExactColumns}]);
      ok &= f == 1 || r % align == 0;
    }
    for (int r : C.rowB) {
      C.expB.push_back(job_of[{r, 36}]);
      ok &= r % align == 0;
    }
  }
  for (int ti = 0; ti < n; ti++) {
    const PairTask& t = plan.tasks[ti];
    if (done[ti]) continue;
    if (t.n1 * t.n2 > kExactSmallSteps) return;
    S.small.push_back(ti);
  }
  // signed sums
  const int n_o = (int)plan.tcontrib_ptr.size() - 1;
  std::vector<int> order(n_o);
  for (int o = 0; o < n_o; o++) order[o] = o;
  auto terms = [&](int o) { return plan.tcontrib_ptr[o + 1] - plan.tcontrib_ptr[o]; };
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return terms(a) > terms(b); });
  std::map<double, int> coef_of;
  for (int c0 = 0; c0 < n_o; c0 += 32) {
    const int len = terms(order[c0]), base = (int)S.wick_ell.size();
    S.wick_chunks.push_back({base, len});
    S.wick_ell.resize(base + 32 * (size_t)len, 0u);
    for (int l = 0; l < 32; l++) {
      const int o = c0 + l < n_o ? order[c0 + l] : -1, nt = o < 0 ? 0 : terms(o);
      S.wick_outputs.push_back({o, nt});
      for (int k = 0; k < nt; k++) {
        const double x = plan.tcontrib_coef[plan.tcontrib_ptr[o] + k];
        auto it = coef_of.emplace(x, (int)S.wick_coefs.size());
        if (it.second) S.wick_coefs.push_back(x);
        S.wick_ell[base + 32 * (size_t)k + l] =
            (uint32_t)plan.tcontrib_item[plan.tcontrib_ptr[o] + k] | ((uint32_t)it.first->second << 16);
      }
    }
  }
  ok &= S.wick_coefs.size() <= 65536;
  S.all = ok;
  *out = std::move(S);
}

// The estimates behind the choice, in us per slice on 152 SMs (one persistent CTA
// each), fitted to the contraction stages of twelve lists (one channel to all 52 or
// 90) on L = 8 .. 48 and met within 25%:
//   digits: a launch, and per operand set as many rounds as it has products per SM,
//     whose time has a constant part (the chunks of one product follow one another)
//     and grows with the rows cut;
//   CUDA cores: the chain of the longest task list, then the complex multiply-adds
//     on the FP64 pipe or on the FP32 pipes (and a pass over the rows).
// The digits read q-major blocks, whose forward transform takes 3 ps more per value
// than the field-major one, but 5 ps less in double-float at L = 24 and 32 (two
// passes, k_fft_xy_split).  Both sides measured, contraction in us:
// double-float 48^3, channel 0: digits 5569, CUDA cores 3185 (the whole call 13958
// and 11639); 52 channels: 13103 and 35969; 16^3, channel 0: 240 and 277; FP64 24^3,
// channel 51: 710 and 608; channel 0: 712 and 1003; 8^3: 54 and 331.
bool exact_pays(const Plan& plan, const ExactSplit& s, int L, bool df) {
  const double V = (double)L * L * L, sms = 152;
  double digits = 23 + V * plan.n_out * (df && (L == 24 || L == 32) ? -5e-6 : 3e-6);
  for (int f = 0; f < kExactSets; f++) {
    const ExactSet& x = s.set[f];
    if (!x.nAp) continue;
    if (f < kExactSlice) digits += std::ceil((V + 8) / 2 / sms) * (4 + 0.34 * x.nAp);
    else digits += std::ceil(V / sms) * (2.5 + 0.027 * x.nAp + 0.0095 * x.nAp * (x.nBp - 16));
  }
  const double macs = (double)plan.pair_macs;
  const double cores = df ? 130 + V * (0.018 + 1.83e-6 * macs) : 305 + V * 5.2e-6 * macs;
  return digits < cores;
}

}  // namespace bbc
