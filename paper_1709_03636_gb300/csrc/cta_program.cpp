// Order of a task's shared-memory ops for a team of warps (CTA teams of the
// shared-memory executor, subtree tasks of the graph executor).
//
// The lowered ops of a network or subtree (Eq. 1 step by step, then the
// adjoint sweep) form a graph through the arena elements they read and write.
// They are put in levels: an op goes one level after the last op it conflicts
// with (read after write, write after read, write after write; the arena
// reuses buffers), and the team meets at one barrier per level instead of one
// per op.  Within a level the ops of few outputs are dealt to the team's warps
// by cost, the others use the whole team.  A leaf's adjoint is fused with its
// dot against the leaf's derivative, and adjoint sums that are long for their
// few outputs are shared by a warp's lanes.  Forward sums keep their order.
// The ops of up to 16 outputs and four terms, nine of ten, are then written as
// lanes (one output each, its offsets formed here), so that a level of them is
// one step of the team.
#include <algorithm>
#include <cstring>

#include "qtc_internal.h"

namespace qtc {

namespace {

int max_pos(const uint8_t* a, int n, const uint8_t* y, int m) {
  int v = 0;
  for (int i = 0; i < n; ++i)
    if (a[i] != kAbsent) v |= 1 << a[i];
  for (int i = 0; i < m; ++i)
    if (y[i] != kAbsent) v |= 1 << y[i];
  return v;
}

// An element range an op touches.
struct Range {
  uint32_t at, size;
  bool global, write;
};

int op_code(const SOp& op) { return op.code & 15; }

// Ranges of one op (gate-table operands are read-only and left out).
int op_ranges(const SOp& op, uint32_t table_elems, Range (&r)[3]) {
  int n = 0;
  auto add = [&](uint32_t at, uint32_t size, bool global, bool write) {
    if (global || at >= table_elems) r[n++] = {at, size, global, write};
  };
  const uint32_t nout = 1u << op.rc;
  switch (op_code(op)) {
    case SOP_CONTRACT:
      add(op.in1, (uint32_t)max_pos(op.p1, op.rc, op.y1, op.ry) + 1, op.flags & SOPF_IN1_GLOBAL,
          false);
      add(op.in2, (uint32_t)max_pos(op.p2, op.rc, op.y2, op.ry) + 1, op.flags & SOPF_IN2_GLOBAL,
          false);
      if (!(op.flags & SOPF_LEAFDOT)) add(op.out, nout, op.flags & SOPF_OUT_GLOBAL, true);
      break;
    case SOP_LEAFGRAD:
      add(op.in1, nout, false, false);
      break;
    case SOP_RESULT:
      add(op.in1, 1, op.flags & SOPF_IN1_GLOBAL, false);
      break;
    case SOP_SEED:
      add(op.out, 1, op.flags & SOPF_OUT_GLOBAL, true);
      break;
    default:
      break;
  }
  return n;
}

// Rough cycles of an op on one warp (narrow) or on the team.
double op_cycles(const SOp& op) {
  const double nout = 1u << op.rc, ny = 1u << op.ry;
  if (op_code(op) != SOP_CONTRACT) return 60;
  if (op.flags & SOPF_LANES) return 150 + nout * (100 + ny / 128 * 90);
  return 200 + std::max(1.0, nout / 128) * ny * 12;
}

}  // namespace

double schedule_cta_ops(std::vector<SOp>& ops, uint32_t table_elems, int n_warps) {
  // leaf dots into the adjoints that produce their operand (nothing else
  // reads a leaf's adjoint)
  std::vector<SOp> in;
  for (size_t i = 0; i < ops.size(); ++i) {
    const SOp& op = ops[i];
    if (op.code == SOP_LEAFGRAD && !in.empty()) {
      SOp& prev = in.back();
      if (prev.code == SOP_CONTRACT && !(prev.flags & (SOPF_LEAFDOT | SOPF_OUT_GLOBAL)) &&
          prev.out == op.in1 && prev.rc == op.rc && op.rc <= 4) {
        prev.flags |= SOPF_LEAFDOT;
        prev.p1[kLeafSlotByte] = (uint8_t)op.out;
        prev.out = op.in2;   // d(leaf)/dparam
        continue;
      }
    }
    in.push_back(op);
  }
  const int n = (int)in.size();
  for (int i = 0; i < n; ++i) {
    SOp& op = in[i];
    const uint32_t nout = 1u << op.rc, ny = 1u << op.ry;
    if (op_code(op) != SOP_CONTRACT || (op.flags & SOPF_LEAFDOT) || nout <= 32 ||
        (nout <= kNarrowMax && ny <= 2))
      op.flags |= SOPF_NARROW;
    // the lowering marks the ops whose sums may be taken in another order
    if (nout > 32 || ny < 64 || nout * (100.0 + ny / 128.0 * 90) >= ny * 12.0)
      op.flags &= (uint8_t)~SOPF_LANES;
  }
  // levels
  std::vector<int> level(n, 0);
  int n_levels = 0;
  uint32_t top = table_elems;
  Range r[3];
  for (const SOp& op : in) {
    const int k = op_ranges(op, table_elems, r);
    for (int j = 0; j < k; ++j)
      if (!r[j].global) top = std::max(top, r[j].at + r[j].size);
  }
  std::vector<int> wrote(top - table_elems, -1), read(top - table_elems, -1);
  std::vector<std::pair<Range, int>> global_uses;   // few per task
  for (int i = 0; i < n; ++i) {
    const int k = op_ranges(in[i], table_elems, r);
    int lv = 0;
    for (int j = 0; j < k; ++j) {
      if (r[j].global) {
        for (const auto& g : global_uses)
          if ((g.first.write || r[j].write) && g.first.at < r[j].at + r[j].size &&
              r[j].at < g.first.at + g.first.size)
            lv = std::max(lv, g.second + 1);
        continue;
      }
      for (uint32_t e = r[j].at - table_elems, end = e + r[j].size; e < end; ++e) {
        lv = std::max(lv, wrote[e] + 1);
        if (r[j].write) lv = std::max(lv, read[e] + 1);
      }
    }
    level[i] = lv;
    n_levels = std::max(n_levels, lv + 1);
    for (int j = 0; j < k; ++j) {
      if (r[j].global) {
        global_uses.push_back({r[j], lv});
        continue;
      }
      std::vector<int>& v = r[j].write ? wrote : read;
      for (uint32_t e = r[j].at - table_elems, end = e + r[j].size; e < end; ++e)
        v[e] = std::max(v[e], lv);
    }
  }
  std::vector<std::vector<int>> by_level(n_levels);
  for (int i = 0; i < n; ++i) by_level[level[i]].push_back(i);
  ops.clear();
  std::vector<double> load(n_warps);
  double cycles = 0;
  for (auto& members : by_level) {
    // narrow ops first, longest first, each to the warp with the least to do
    // (leaf dots to the first warp, so that the order of their terms is fixed);
    // then the team's ops
    std::stable_sort(members.begin(), members.end(), [&](int x, int y) {
      const bool nx = in[x].flags & SOPF_NARROW, ny = in[y].flags & SOPF_NARROW;
      if (nx != ny) return nx;
      return nx && op_cycles(in[x]) > op_cycles(in[y]);
    });
    std::fill(load.begin(), load.end(), 0.0);
    cycles += 200;
    for (int i : members) {
      SOp op = in[i];
      if (!(op.flags & SOPF_NARROW)) cycles += op_cycles(op);
      if (op.flags & SOPF_NARROW) {
        int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
        if (op.code == SOP_LEAFGRAD || (op.flags & SOPF_LEAFDOT)) w = 0;
        load[w] += op_cycles(op);
        op.code = (uint8_t)(op.code | w << 4);
      }
      ops.push_back(op);
    }
    if (!members.empty()) ops.back().flags |= SOPF_SYNC;
    cycles += *std::max_element(load.begin(), load.end());
  }
  return cycles;
}

void validate_cta_ops(const SOp* ops, size_t n, uint32_t table_elems, uint32_t arena_elems,
                      uint64_t global_elems, int n_params, int n_warps) {
  auto need = [&](bool ok, size_t k, const char* what) {
    if (!ok) fail(QTC_ERR_INVALID, "internal: shared-memory op %zu: %s", k, what);
  };
  auto inside = [&](uint32_t off, bool global, uint64_t elems, size_t k, const char* what) {
    const uint64_t end = (uint64_t)off + elems;
    if (global) need(end <= global_elems, k, what);
    else if (off < table_elems) need(end <= table_elems, k, what);
    else need(end <= (uint64_t)table_elems + arena_elems, k, what);
  };
  need(n == 0 || (ops[n - 1].flags & SOPF_SYNC), n, "no barrier at the end");
  size_t first = 0;   // of the current level
  for (size_t k = 0; k < n; ++k) {
    const SOp& op = ops[k];
    const int code = op_code(op);
    const bool narrow = op.flags & SOPF_NARROW, dot = op.flags & SOPF_LEAFDOT;
    need(narrow || code == SOP_CONTRACT, k, "a team op that is no contraction");
    need(!narrow || (op.code >> 4) < n_warps, k, "warp");
    int slot = -1;
    if (code == SOP_CONTRACT) {
      need(op.rc <= kMaxSmemRank && op.ry <= kMaxSmemRank, k, "shape");
      need(!narrow || (1u << op.rc) <= kNarrowMax, k, "narrow op with many outputs");
      need(!(op.flags & (SOPF_LANES | SOPF_LEAFDOT)) || (narrow && op.rc <= 5), k, "adjoint op");
      need(!(op.flags & SOPF_LANES) || op.ry >= 5, k, "lanes over a short sum");
      need(!dot || op.rc <= 4, k, "leaf rank");
      inside(op.in1, op.flags & SOPF_IN1_GLOBAL,
             (uint64_t)max_pos(op.p1, op.rc, op.y1, op.ry) + 1, k, "first operand");
      inside(op.in2, op.flags & SOPF_IN2_GLOBAL,
             (uint64_t)max_pos(op.p2, op.rc, op.y2, op.ry) + 1, k, "second operand");
      if (dot) {
        need((uint64_t)op.out + (1u << op.rc) <= table_elems, k, "leaf derivative");
        slot = op.p1[kLeafSlotByte];
      } else {
        need((op.flags & SOPF_OUT_GLOBAL) || op.out >= table_elems, k, "output in the table");
        inside(op.out, op.flags & SOPF_OUT_GLOBAL, 1ull << op.rc, k, "output");
      }
    } else if (code == SOP_LEAFGRAD) {
      inside(op.in1, false, 1ull << op.rc, k, "leaf adjoint");
      inside(op.in2, false, 1ull << op.rc, k, "leaf derivative");
      slot = (int)op.out;
    } else if (code == SOP_RESULT) {
      inside(op.in1, op.flags & SOPF_IN1_GLOBAL, 1, k, "result");
    } else if (code == SOP_SEED) {
      inside(op.out, op.flags & SOPF_OUT_GLOBAL, 1, k, "seed");
    } else {
      need(false, k, "code");
    }
    if (code == SOP_LEAFGRAD || dot) {
      need(slot >= 0 && slot < n_params, k, "gradient slot");
      need((op.code >> 4) == 0, k, "leaf dot away from the first warp");
    }
    // no conflict with the level's earlier ops
    Range a[3], b[3];
    const int na = op_ranges(op, table_elems, a);
    for (size_t q = first; q < k; ++q) {
      const int nb = op_ranges(ops[q], table_elems, b);
      for (int i = 0; i < na; ++i)
        for (int j = 0; j < nb; ++j)
          need(!(a[i].write || b[j].write) || a[i].global != b[j].global ||
                   a[i].at >= b[j].at + b[j].size || b[j].at >= a[i].at + a[i].size,
               k, "conflicts with an op of its level");
    }
    if (op.flags & SOPF_SYNC) first = k + 1;
  }
}

namespace {

// The small contractions of a level, one output per lane.
bool fits_lanes(const SOp& op, uint32_t lane_limit, bool dots) {
  if (op_code(op) != SOP_CONTRACT || !(op.flags & SOPF_NARROW) || (op.flags & SOPF_LANES) ||
      (op.flags & (SOPF_OUT_GLOBAL | SOPF_IN1_GLOBAL | SOPF_IN2_GLOBAL)))
    return false;
  if (op.ry > 2 || (1u << op.rc) > lane_limit) return false;
  if ((op.flags & SOPF_LEAFDOT) && (!dots || op.p1[kLeafSlotByte] >= kLaneDotSlots)) return false;
  return op.out + (1u << op.rc) <= 0x10000u &&
         op.in1 + (uint32_t)max_pos(op.p1, op.rc, op.y1, op.ry) < 0x10000u &&
         op.in2 + (uint32_t)max_pos(op.p2, op.rc, op.y2, op.ry) < 0x10000u;
}

uint32_t spread(const uint8_t* pos, int n, uint32_t v) {
  uint32_t off = 0;
  for (int i = 0; i < n; ++i)
    if (((v >> i) & 1u) && pos[i] != kAbsent) off |= 1u << pos[i];
  return off;
}

CLane make_lane(const SOp& op, uint32_t c) {
  CLane l{};
  const bool dot = op.flags & SOPF_LEAFDOT;
  l.out = (uint16_t)(op.out + c);
  l.a = (uint16_t)(op.in1 + spread(op.p1, op.rc, c));
  l.b = (uint16_t)(op.in2 + spread(op.p2, op.rc, c));
  l.flags = (uint8_t)(op.ry | (dot ? CLF_DOT : CLF_STORE));
  l.slot = dot ? op.p1[kLeafSlotByte] : (uint8_t)0;
  if (op.ry >= 1) {
    l.ya1 = (uint16_t)spread(op.y1, op.ry, 1);
    l.yb1 = (uint16_t)spread(op.y2, op.ry, 1);
  }
  if (op.ry >= 2) {
    l.ya2 = (uint16_t)spread(op.y1, op.ry, 2);
    l.yb2 = (uint16_t)spread(op.y2, op.ry, 2);
  }
  return l;
}

}  // namespace

uint32_t build_cta_stream(const std::vector<SOp>& ops, uint32_t half_units, uint32_t lane_limit,
                          bool dots, std::vector<uint4>& out) {
  if (ops.empty()) return 0;
  if (half_units < 1 + kSOpUnits)
    fail(QTC_ERR_INVALID, "internal: a stage of %u units", 2 * half_units);
  struct Record {
    std::vector<uint4> units;
    bool level_end = false;
  };
  std::vector<Record> records;
  const uint32_t max_lanes = std::min(half_units - 2, 1024u);
  auto unit_of = [](const void* p) {
    uint4 u;
    std::memcpy(&u, p, sizeof u);
    return u;
  };
  for (size_t first = 0; first < ops.size();) {
    size_t last = first;
    while (!(ops[last].flags & SOPF_SYNC)) ++last;
    // lanes: leaf dots (first 32 lanes of a record), then the others
    std::vector<CLane> leaf, rest;
    std::vector<const SOp*> whole;
    for (size_t k = first; k <= last; ++k) {
      if (!fits_lanes(ops[k], lane_limit, dots)) {
        whole.push_back(&ops[k]);
        continue;
      }
      for (uint32_t c = 0; c < (1u << ops[k].rc); ++c)
        ((ops[k].flags & SOPF_LEAFDOT) ? leaf : rest).push_back(make_lane(ops[k], c));
    }
    size_t nl = 0, nr = 0;
    while (nl < leaf.size() || nr < rest.size()) {
      Record r;
      uint4 head{SOP_LANES, 0, 0, 0};
      r.units.push_back(head);
      for (uint32_t i = 0; i < max_lanes; ++i) {
        CLane l{};
        if (i < 32 && nl < leaf.size()) l = leaf[nl++];
        else if (nr < rest.size()) l = rest[nr++];
        else break;
        r.units.push_back(unit_of(&l));
      }
      r.units[0].y = (uint32_t)r.units.size() - 1;
      records.push_back(std::move(r));
    }
    for (const SOp* op : whole) {
      Record r;
      SOp plain = *op;
      plain.flags &= (uint8_t)~SOPF_SYNC;
      const unsigned char* p = reinterpret_cast<const unsigned char*>(&plain);
      for (uint32_t u = 0; u < kSOpUnits; ++u) r.units.push_back(unit_of(p + 16 * u));
      records.push_back(std::move(r));
    }
    records.back().level_end = true;
    first = last + 1;
  }
  // batches; a level that ends with its batch needs no barrier of its own
  std::vector<std::pair<size_t, size_t>> batches;
  for (size_t i = 0; i < records.size();) {
    size_t j = i;
    uint32_t units = i ? 1 : 0;
    while (j < records.size() && units + records[j].units.size() <= half_units)
      units += (uint32_t)records[j++].units.size();
    batches.push_back({i, j});
    i = j;
  }
  std::vector<uint32_t> sizes;
  for (const auto& b : batches) {
    uint32_t units = b.first ? 1 : 0;
    for (size_t k = b.first; k < b.second; ++k) units += (uint32_t)records[k].units.size();
    sizes.push_back(units);
  }
  for (size_t n = 0; n < batches.size(); ++n) {
    const auto& b = batches[n];
    if (n) out.push_back(uint4{0, n + 1 < sizes.size() ? sizes[n + 1] : 0u, 0, 0});
    for (size_t k = b.first; k < b.second; ++k) {
      if (records[k].level_end && k + 1 < b.second) records[k].units[0].x |= SOPF_SYNC << 24;
      out.insert(out.end(), records[k].units.begin(), records[k].units.end());
    }
  }
  return sizes[0] | (sizes.size() > 1 ? sizes[1] << 16 : 0u);
}

uint32_t build_smallest_stream(const std::vector<SOp>& ops, uint32_t half_units, bool dots,
                               std::vector<uint4>& out) {
  std::vector<uint4> best;
  uint32_t units = 0;
  for (uint32_t limit : {4u, 2u, 0u}) {
    std::vector<uint4> s;
    const uint32_t first = build_cta_stream(ops, half_units, limit, dots, s);
    if (limit < 4u && s.size() >= best.size()) continue;
    best.swap(s);
    units = first;
  }
  out.insert(out.end(), best.begin(), best.end());
  return units;
}

void validate_cta_stream(const uint4* stream, size_t n, uint32_t batches, uint32_t half_units,
                         uint32_t table_elems, uint32_t arena_elems, int n_params) {
  auto need = [&](bool ok, const char* what) {
    if (!ok) fail(QTC_ERR_INVALID, "internal: task stream: %s", what);
  };
  const uint32_t team_elems = table_elems + arena_elems;
  size_t at = 0;
  uint32_t units = batches & 0xffffu;
  while (units) {
    need(units <= half_units && at + units <= n, "batch beyond the stage or the stream");
    const uint32_t next = at ? stream[at].y : batches >> 16;
    size_t u = at ? at + 1 : at;
    while (u < at + units) {
      if ((stream[u].x & 15u) != SOP_LANES) {
        u += kSOpUnits;   // (checked op by op before)
        continue;
      }
      const uint32_t lanes = stream[u].y;
      need(lanes >= 1 && u + 1 + lanes <= at + units, "lanes beyond their batch");
      for (uint32_t i = 0; i < lanes; ++i) {
        CLane l;
        std::memcpy(&l, &stream[u + 1 + i], sizeof l);
        const uint32_t ma = (uint32_t)(l.ya1 | l.ya2), mb = (uint32_t)(l.yb1 | l.yb2);
        need((l.flags & 3) <= 2 && l.a + ma < team_elems && l.b + mb < team_elems, "lane operand");
        // the two regions are addressed apart: an operand stays in its own
        need((l.a < table_elems) == (l.a + ma < table_elems) &&
                 (l.b < table_elems) == (l.b + mb < table_elems),
             "lane operand across the table's end");
        if (l.flags & CLF_STORE) need(l.out >= table_elems && l.out < team_elems, "lane output");
        if (l.flags & CLF_DOT)
          need(i < 32 && l.out < table_elems && l.slot < n_params && l.slot < kLaneDotSlots,
               "lane leaf dot");
      }
      u += 1 + lanes;
    }
    need(u == at + units, "batch size");
    at += units;
    units = next;
  }
  need(at == n, "stream size");
}

}  // namespace qtc
