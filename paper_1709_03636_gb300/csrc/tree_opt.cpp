// Contraction trees for execution in double precision (host).
//
// A plan's tree follows its elimination ordering (Section 3.1): a large tensor
// meets one small gate tensor per eliminated wire.  The scalar does not depend
// on the tree (Eq. 1 is associative), so the graph executor contracts a
// complex128 network along a tree of its own: below every node that touches a
// large tensor the tree is cut off at a few subtrees (largest tensors opened
// first) and the best way to contract those is found exactly, by dynamic
// programming over their subsets, under a model of the step's time on the
// device.  What bounds these programs is the FP64 pipe, so fewer multiply-adds
// pay: 7-regular n=20 full networks 0.227 -> 0.168 G forward (and half the
// elements moved), value + gradient 5.66 -> 4.30 ms.  The plan itself
// (qtc_plan_*, qtc_batch_stats) stays as the ordering gave it.
#include <algorithm>
#include <cmath>

#include "qtc_internal.h"

namespace qtc {

namespace {

constexpr int kMaxFrontier = 8;   // subtrees rearranged at once: up to 3^8 splits per node
// Passes over the nodes, by width of the frontier: two schedules end in
// different local optima, the better one is taken.
constexpr int kSchedule[2][6] = {{8, 8, 8, 8, 8, 8}, {4, 5, 6, 7, 8, 8}};
constexpr double kWorthIt = 0.03; // share of the tree's time below which steps are left alone

struct Tree {
  int n_leaves = 0, root = 0, words = 0;
  std::vector<int> left, right;
  std::vector<uint64_t> bits;      // label set of every tensor
  std::vector<uint64_t> seen;      // per node: what it was last found best for

  uint64_t* labels(int t) { return &bits[(size_t)t * words]; }
  int rank(int t) {
    int c = 0;
    for (int w = 0; w < words; ++w) c += __builtin_popcountll(labels(t)[w]);
    return c;
  }
};

// Labels of one step, at most: trees with wider steps stay as they are (they are
// far beyond the device's memory).
constexpr int kMaxStepLabels = 64;

// Expected time (ns over the whole device) of one step, from tables over the
// ranks of its tensors and the number of its labels.
struct StepTimes {
  double move[kMaxStepLabels + 1], work[kMaxStepLabels + 1], fixed;
  explicit StepTimes(const TreeModel& m) : fixed(m.step_ns) {
    for (int i = 0; i <= kMaxStepLabels; ++i) {
      move[i] = m.elem * std::ldexp(1.0, i) / m.bytes_per_ns;
      work[i] = std::ldexp(1.0, i) / m.macs_per_ns;
    }
  }
  double operator()(int ra, int rb, int rc, int all) const {
    // the larger of moving and computing, and part of the other (they overlap
    // within a step, but not perfectly)
    const double mv = move[ra] + move[rb] + move[rc], wk = work[all];
    return std::max(mv, wk) + 0.25 * std::min(mv, wk) + fixed;
  }
};

int labels_of_step(Tree& t, int x) {
  int all = 0;
  for (int w = 0; w < t.words; ++w)
    all += __builtin_popcountll(t.labels(t.left[x])[w] | t.labels(t.right[x])[w]);
  return all;
}

// (no step of a tree under search has more than kMaxStepLabels labels: the given
// ones were looked at, the new ones hold labels of one 64-bit word)
double step_of(Tree& t, int x, const StepTimes& time) {
  return time(t.rank(t.left[x]), t.rank(t.right[x]), t.rank(x), labels_of_step(t, x));
}

// Rearranges the tree below `node`; true when that made it faster.
bool rearrange(Tree& t, int node, int width, const StepTimes& time, double least) {
  int frontier[kMaxFrontier], k = 1;
  int inner[kMaxFrontier], n_inner = 0;
  frontier[0] = node;
  while (k < width) {
    int at = -1, best = -1;
    for (int i = 0; i < k; ++i)
      if (frontier[i] >= t.n_leaves) {
        const int r = t.rank(frontier[i]);
        if (r > best) best = r, at = i;
      }
    if (at < 0) break;
    const int x = frontier[at];
    inner[n_inner++] = x;
    frontier[at] = t.left[x];
    frontier[k++] = t.right[x];
  }
  if (k < 3) return false;
  double old = 0;
  for (int i = 0; i < n_inner; ++i) old += step_of(t, inner[i], time);
  if (old < least) return false;
  // the labels in play as bits of one word
  std::vector<int> local;
  for (int w = 0; w < t.words; ++w) {
    uint64_t any = 0;
    for (int i = 0; i < k; ++i) any |= t.labels(frontier[i])[w];
    for (; any; any &= any - 1) local.push_back(64 * w + __builtin_ctzll(any));
  }
  if (local.size() > kMaxStepLabels) return false;
  auto pack = [&](int x) {
    uint64_t v = 0;
    const uint64_t* l = t.labels(x);
    for (size_t i = 0; i < local.size(); ++i)
      v |= ((l[local[i] >> 6] >> (local[i] & 63)) & 1ull) << i;
    return v;
  };
  const uint64_t out = pack(node);
  const int all = (1 << k) - 1;
  // held: labels of a subset's subtrees; open: those still needed outside it
  uint64_t held[1 << kMaxFrontier], open[1 << kMaxFrontier];
  double cost[1 << kMaxFrontier];
  int split[1 << kMaxFrontier];
  uint8_t rank[1 << kMaxFrontier];
  held[0] = 0;
  for (int s = 1; s <= all; ++s)
    held[s] = held[s & (s - 1)] | ((s & (s - 1)) ? held[s & -s] : pack(frontier[__builtin_ctz(s)]));
  for (int s = 1; s <= all; ++s) {
    open[s] = held[s] & (out | held[all ^ s]);
    rank[s] = (uint8_t)__builtin_popcountll(open[s]);
    cost[s] = (s & (s - 1)) ? HUGE_VAL : 0.0;
    split[s] = 0;
  }
  // the same subtrees under the same tree as at the last look: nothing to find
  uint64_t sign = 1469598103934665603ull;
  auto mix = [&](uint64_t v) { sign = (sign ^ v) * 1099511628211ull + (sign >> 29); };
  for (int i = 0; i < k; ++i) {
    mix((uint64_t)frontier[i]);
    mix(held[1 << i]);
  }
  for (size_t i = 0; i < local.size(); ++i) mix((uint64_t)local[i]);
  for (int i = 0; i < n_inner; ++i) {
    const int x = inner[i];
    mix((uint64_t)t.left[x] << 32 | (uint64_t)t.right[x]);
  }
  if (t.seen[node] == sign) return false;
  t.seen[node] = sign;
  for (int s = 3; s <= all; ++s) {
    // (a subset whose result alone takes longer is no use either)
    if (!(s & (s - 1)) || time.move[rank[s]] >= old) continue;
    for (int a = (s - 1) & s; a; a = (a - 1) & s) {
      const int b = s ^ a;
      if (a < b) break;            // the other half of the splits
      const double parts = cost[a] + cost[b];
      if (parts >= cost[s] || parts >= old) continue;   // `old`: no use to the whole
      const double c =
          parts + time(rank[a], rank[b], rank[s], __builtin_popcountll(open[a] | open[b]));
      if (c < cost[s]) cost[s] = c, split[s] = a;
    }
  }
  if (!(cost[all] < 0.999 * old)) return false;
  // rebuild with the same inner nodes, `node` staying the top
  int next = 1;
  auto build = [&](auto&& self, int s, int id) -> int {
    if (!(s & (s - 1))) return frontier[__builtin_ctz(s)];
    if (id < 0) id = inner[next++];
    const int a = self(self, split[s], -1), b = self(self, s ^ split[s], -1);
    t.left[id] = a;
    t.right[id] = b;
    if (id != node) {
      uint64_t* l = t.labels(id);
      std::fill(l, l + t.words, 0ull);
      for (size_t i = 0; i < local.size(); ++i)
        if ((open[s] >> i) & 1ull) l[local[i] >> 6] |= 1ull << (local[i] & 63);
    }
    return id;
  };
  build(build, all, node);
  return true;
}

}  // namespace

TreeModel tree_model(int dtype) {
  TreeModel m;
  m.elem = (double)elem_bytes(dtype);
  if (dtype == QTC_C128) {
    // multiply-adds run on the narrow FP64 pipe (0.16 per ps at its peak): fewer
    // of them is what pays
    m.macs_per_ns = 150;
  } else {
    // Single precision keeps the plan's own order of every sum: expectation
    // values are often far below one (p=1 on a 7-regular graph: under 5e-3 for a
    // third of all angles), and another tree moves them by their whole rounding
    // error (1.5e-3 relative seen on 7-regular n=26), for all that it was 2.0x
    // faster there and 1.7x on p=3 n=60.
    m.small_rank = 1 << 20;
  }
  return m;
}

Plan execution_plan(const Plan& plan, const TreeModel& m) {
  const int L = (int)plan.net.leaves.size(), S = (int)plan.steps.size();
  if (plan.max_rank <= m.small_rank) return plan;
  Tree t;
  t.n_leaves = L;
  t.root = L + S - 1;
  t.words = (plan.net.n_labels + 63) / 64;
  t.left.assign(L + S, -1);
  t.right.assign(L + S, -1);
  t.bits.assign((size_t)(L + S) * t.words, 0);
  t.seen.assign(L + S, 0);
  for (int i = 0; i < L + S; ++i)
    for (int x : plan.labels[i]) t.labels(i)[x >> 6] |= 1ull << (x & 63);
  for (int s = 0; s < S; ++s) {
    t.left[L + s] = plan.steps[s].a;
    t.right[L + s] = plan.steps[s].b;
  }
  for (int x = L; x < L + S; ++x)
    if (labels_of_step(t, x) > kMaxStepLabels) return plan;
  const StepTimes time(m);
  std::vector<int> order;          // inner nodes, children before parents
  auto walk = [&](Tree& t) {
    order.clear();
    std::vector<int> todo{t.root};
    while (!todo.empty()) {        // parents first, then reversed
      const int x = todo.back();
      todo.pop_back();
      if (x < L) continue;
      order.push_back(x);
      todo.push_back(t.left[x]);
      todo.push_back(t.right[x]);
    }
    std::reverse(order.begin(), order.end());
    double total = 0;
    for (int x : order) total += step_of(t, x, time);
    return total;
  };
  const Tree given = t;
  double best = walk(t);
  bool changed = false;
  for (const auto& schedule : kSchedule) {
    Tree u = given;
    for (int width : schedule) {
      const double least = kWorthIt * walk(u);
      bool moved = false;
      for (auto it = order.rbegin(); it != order.rend(); ++it) {
        const int x = *it;
        if (std::max({u.rank(x), u.rank(u.left[x]), u.rank(u.right[x])}) < m.small_rank) continue;
        if (rearrange(u, x, width, time, least)) moved = true;
      }
      if (!moved && width == kMaxFrontier) break;
    }
    const double total = walk(u);
    if (total < best) {
      best = total;
      t = std::move(u);
      changed = true;
    }
  }
  if (!changed) return plan;
  walk(t);
  Plan out;
  out.net = plan.net;
  out.lg_width = plan.lg_width;
  std::vector<int> id(L + S, -1);
  for (int i = 0; i < L; ++i) id[i] = i;
  for (int x : order) {
    id[x] = L + (int)out.steps.size();
    out.steps.push_back({id[t.left[x]], id[t.right[x]]});
  }
  layout_labels(out);
  return out;
}

}  // namespace qtc
