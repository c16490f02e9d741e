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
constexpr int kSmallRank = 10;    // trees of tensors up to this rank stay as they are
// What a step costs on the device (complex128): bytes moved by all SMs per ns,
// multiply-adds per ns on the narrow FP64 pipe (160 at its peak; fewer of them is what
// pays), and ns per step over the networks that run beside it.
constexpr double kElemBytes = 16, kBytesPerNs = 6000, kMacsPerNs = 150, kStepNs = 1;

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
  double move[kMaxStepLabels + 1], work[kMaxStepLabels + 1];
  StepTimes() {
    for (int i = 0; i <= kMaxStepLabels; ++i) {
      move[i] = kElemBytes * std::ldexp(1.0, i) / kBytesPerNs;
      work[i] = std::ldexp(1.0, i) / kMacsPerNs;
    }
  }
  double operator()(int ra, int rb, int rc, int all) const {
    // the larger of moving and computing, and part of the other (they overlap
    // within a step, but not perfectly)
    const double mv = move[ra] + move[rb] + move[rc], wk = work[all];
    return std::max(mv, wk) + 0.25 * std::min(mv, wk) + kStepNs;
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
  // made: a subset's cost and the move of its result, what any split above it pays
  double made[1 << kMaxFrontier];
  for (int i = 0; i < k; ++i) made[1 << i] = time.move[rank[1 << i]];
  for (int s = 3; s <= all; ++s) {
    if (!(s & (s - 1))) continue;
    made[s] = HUGE_VAL;
    // (what the subset may cost to be of use to the whole)
    const double out_move = time.move[rank[s]];
    const double useful = s == all ? old : old - out_move - time.move[rank[all]];
    if (out_move >= useful) continue;
    double least_made = useful - out_move;
    for (int a = (s - 1) & s; a; a = (a - 1) & s) {
      const int b = s ^ a;
      if (a < b) break;            // the other half of the splits
      if (made[a] + made[b] >= least_made) continue;
      const double c = cost[a] + cost[b] +
                       time(rank[a], rank[b], rank[s], __builtin_popcountll(open[a] | open[b]));
      if (c < cost[s]) {
        cost[s] = c;
        split[s] = a;
        least_made = std::min(c, useful) - out_move;
      }
    }
    made[s] = cost[s] + out_move;
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

namespace {

// The best tree found for `plan`; no steps when that is its own.
void search_tree(const Plan& plan, bool alone, ExecutionTree& out) {
  const int L = (int)plan.net.leaves.size(), S = (int)plan.steps.size();
  Tree given;
  given.n_leaves = L;
  given.root = L + S - 1;
  given.words = (plan.net.n_labels + 63) / 64;
  given.left.assign(L + S, -1);
  given.right.assign(L + S, -1);
  given.bits.assign((size_t)(L + S) * given.words, 0);
  given.seen.assign(L + S, 0);
  for (int i = 0; i < L + S; ++i)
    for (int x : plan.labels[i]) given.labels(i)[x >> 6] |= 1ull << (x & 63);
  for (int s = 0; s < S; ++s) {
    given.left[L + s] = plan.steps[s].a;
    given.right[L + s] = plan.steps[s].b;
  }
  for (int x = L; x < L + S; ++x)
    if (labels_of_step(given, x) > kMaxStepLabels) return;
  const StepTimes time;
  // inner nodes, children before parents; the time of all steps
  auto walk = [&](Tree& t, std::vector<int>& order) {
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
  Tree found[2];
  std::vector<int> orders[2];
  double totals[2];
  auto search = [&](int k) {
    Tree& u = found[k] = given;
    std::vector<int>& order = orders[k];
    for (int width : kSchedule[k]) {
      const double least = kWorthIt * walk(u, order);
      bool moved = false;
      for (auto it = order.rbegin(); it != order.rend(); ++it) {
        const int x = *it;
        if (std::max({u.rank(x), u.rank(u.left[x]), u.rank(u.right[x])}) < kSmallRank) continue;
        if (rearrange(u, x, width, time, least)) moved = true;
      }
      if (!moved && width == kMaxFrontier) break;
    }
    totals[k] = walk(u, order);
  };
  if (alone) {
    parallel_for(2, search, true);
  } else {
    search(0);
    search(1);
  }
  const int best = totals[1] < totals[0] ? 1 : 0;
  {
    std::vector<int> order;
    if (!(totals[best] < walk(given, order))) return;
  }
  // its steps, and the labels in storage order as layout_labels gives them (a label
  // that survives longer comes first), from the label sets at hand
  Tree& t = found[best];
  const std::vector<int>& nodes = orders[best];
  std::vector<int> id(L + S, -1), death(plan.net.n_labels, S);
  out.labels.assign(plan.labels.begin(), plan.labels.begin() + L);
  out.labels.resize(L + S);
  for (int i = 0; i < L; ++i) id[i] = i;
  auto each = [&](uint64_t bits, int w, auto&& f) {
    for (; bits; bits &= bits - 1) f(64 * w + __builtin_ctzll(bits));
  };
  double elems = 0;
  for (int s = 0; s < S; ++s) {
    const int x = nodes[s], a = t.left[x], b = t.right[x];
    id[x] = L + s;
    out.steps.push_back({id[a], id[b]});
    for (int w = 0; w < t.words; ++w)
      each((t.labels(a)[w] | t.labels(b)[w]) & ~t.labels(x)[w], w, [&](int l) { death[l] = s; });
    out.cmacs += std::ldexp(1.0, labels_of_step(t, x));
    elems += std::ldexp(1.0, t.rank(a)) + std::ldexp(1.0, t.rank(b)) + std::ldexp(1.0, t.rank(x));
    out.max_rank = std::max(out.max_rank, t.rank(x));
  }
  out.bytes_c64 = 8.0 * elems;
  for (int s = 0; s < S; ++s) {
    std::vector<int>& r = out.labels[L + s];
    for (int w = 0; w < t.words; ++w)
      each(t.labels(nodes[s])[w], w, [&](int l) { r.push_back(l); });
    std::sort(r.begin(), r.end(), [&](int x, int y) {
      if (death[x] != death[y]) return death[x] > death[y];
      return x < y;
    });
  }
}

}  // namespace

Plan execution_plan(const Plan& plan, int dtype, bool alone) {
  // Single precision keeps the plan's own order of every sum: expectation values are
  // often far below one (p=1 on a 7-regular graph: under 5e-3 for a third of all
  // angles), and another tree moves them by their whole rounding error (1.5e-3 relative
  // seen on 7-regular n=26), for all that it was 2.0x faster there and 1.7x on p=3 n=60.
  if (dtype != QTC_C128 || plan.max_rank <= kSmallRank) return plan;
  ExecutionTree& tree = *plan.tree;
  std::lock_guard<std::mutex> lock(tree.mutex);
  if (!tree.known) {
    search_tree(plan, alone, tree);
    tree.known = true;
  }
  if (tree.steps.empty()) return plan;
  Plan out;
  out.net = plan.net;
  out.lg_width = plan.lg_width;
  out.steps = tree.steps;
  out.labels = tree.labels;
  out.max_rank = tree.max_rank;
  out.cmacs = tree.cmacs;
  out.bytes_c64 = tree.bytes_c64;
  return out;
}

}  // namespace qtc
