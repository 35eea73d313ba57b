// Sweeps: a registered program as independent element-wise expressions
// (host side; hiccl_sweep.cu executes them).
//
// The factorized schedule of a primitive moves the same byte range through
// every step of its tree, so the value that reaches a destination is a
// function of the sources at the same offset: a copy of the root's value, or
// the nested fold that the hierarchy (and the ring) fixes -- independent of
// stripe, pipeline depth and representatives.  Evaluating that expression
// directly gives the schedule's result bit for bit and needs no relay, no
// second read of a partial result and no signalling between steps.
//
// A fence is handled by substitution: a copy whose source is exactly what an
// earlier expression stores becomes more destinations of that expression
// (All-reduce's All-gather half).  Any other conflict across a fence leaves
// the program to the step executor.

#include <algorithm>
#include <map>
#include <string>
#include <tuple>

#include "hiccl_internal.h"

namespace hiccl {

namespace {

// ---- expressions -------------------------------------------------------------

// Emits the evaluation order and tokens of one reduction: the leaves of
// [lo, hi) of the sorted leaf list, grouped by the hierarchy.
struct Expr {
  const std::vector<int> &h;
  const std::vector<int> &leaves;
  bool rounds;                       // the payload is rounded after every fold
  std::vector<long long> G;
  std::vector<int> order;            // ranks in evaluation order
  std::vector<uint32_t> toks;
  std::vector<uint32_t> nops;
  bool ok = true;

  Expr(const std::vector<int> &hier, const std::vector<int> &lv, bool rnd) : h(hier), leaves(lv), rounds(rnd) {
    G.assign(h.size() + 1, 1);
    for (size_t l = h.size(); l-- > 0;) G[l] = G[l + 1] * h[l];
    order.reserve(lv.size());
    toks.reserve(lv.size());
    nops.reserve(lv.size());
  }
  void leaf(int rank, bool start, bool push) {
    order.push_back(rank);
    toks.push_back((start ? TOK_START : 0u) | (push ? TOK_PUSH : 0u));
    nops.push_back(0);
  }
  void op(uint32_t o) {
    if (nops.back() >= 12) {
      ok = false;
      return;
    }
    toks.back() |= o << (TOK_OPS + 2 * nops.back()++);
  }
  // ends of the level-l subgroups inside leaves[lo, hi)
  size_t next(size_t lo, size_t hi, int l) const { return next_in(leaves, lo, hi, l); }
  size_t next_in(const std::vector<int> &v, size_t lo, size_t hi, int l) const {
    const long long end = (v[lo] / G[l + 1] + 1) * G[l + 1];
    if (v[hi - 1] < end) return hi;
    size_t k = lo + 1;
    while (v[k] < end) ++k;
    return k;
  }
  // the value of a group: the left fold of its non-empty subgroups'
  // values in ascending order; a group with one passes its value through.
  // The accumulator is started (push: after saving it).
  void group(size_t lo, size_t hi, int l, bool push) {
    if (hi - lo == 1) {
      leaf(leaves[lo], true, push);
      return;
    }
    if (next(lo, hi, l) == hi) {
      group(lo, hi, l + 1, push);
      return;
    }
    parts(lo, hi, l, push);
    if (rounds) op(TOK_ROUND);
  }
  // the same fold without the rounding that ends it
  void parts(size_t lo, size_t hi, int l, bool push) {
    for (size_t a = lo; a < hi;) {
      const size_t z = next(a, hi, l);
      if (a == lo) {
        group(a, z, l + 1, push);
      } else if (z - a == 1) {
        leaf(leaves[a], false, false);
      } else {
        group(a, z, l + 1, true);
        op(TOK_POP);
      }
      a = z;
    }
  }
  // ring across the nodes of level lr, node a0 first: every node folds its
  // subgroups' values and then the value coming from the next node, so the
  // chain is evaluated from its last node back
  void chain(int ring, int lr, long long a0) {
    const long long N = G[lr];
    std::vector<std::pair<size_t, size_t>> nodes;
    for (int i = 0; i < ring; ++i) {
      const long long a = (a0 + i) % ring;
      const size_t lo = std::lower_bound(leaves.begin(), leaves.end(), (int)(a * N)) - leaves.begin();
      const size_t hi = std::lower_bound(leaves.begin(), leaves.end(), (int)((a + 1) * N)) - leaves.begin();
      if (lo < hi) nodes.emplace_back(lo, hi);
    }
    for (size_t k = nodes.size(); k-- > 0;) {
      if (k + 1 == nodes.size()) {
        group(nodes[k].first, nodes[k].second, lr, false);
        continue;
      }
      if (lr == (int)h.size()) leaf(leaves[nodes[k].first], true, true);
      else parts(nodes[k].first, nodes[k].second, lr, true);
      op(TOK_JOIN);
      if (rounds) op(TOK_ROUND);
    }
  }
  // Drop the rounding that the store does anyway and count the saved values;
  // false when the expression does not fit the kernels.
  bool finish(uint32_t &depth) {
    if (!ok) return false;
    uint32_t &last = toks.back();
    const uint32_t n = nops.back();
    if (n && ((last >> (TOK_OPS + 2 * (n - 1))) & 3u) == TOK_ROUND) last &= ~(3u << (TOK_OPS + 2 * (n - 1)));
    uint32_t sp = 0, most = 0;
    for (uint32_t t : toks) {
      if (t & TOK_PUSH) most = std::max(most, ++sp);
      for (uint32_t o = t >> TOK_OPS; o; o >>= 2)
        if ((o & 3u) >= TOK_POP) --sp;
    }
    depth = most;
    return most <= SWEEP_MAX_DEPTH;
  }
};

struct Program {   // an expression shared by members: evaluation order and tokens
  std::vector<int> leaves;
  long long node;  // the chain's first node (-1: tree)
  bool rounds, exact;
  std::vector<int> order;
  uint32_t tok, team, ttok;
};

// The two-step form of a program's expression (see SweepClass::team): the
// groups of one level, or equal parts where the operator is exact (the order of exact
// operations does not change the result).  Returns the number of sections (0: none) and
// appends their tokens, bounds and the tokens of their values.
uint32_t two_steps(const std::vector<int> &h, const std::vector<int> &leaves, bool rounds, bool exact, bool chained, bool few,
                   std::vector<uint32_t> &toks, uint32_t &depth) {
  const uint32_t n = (uint32_t)leaves.size();
  if (n < 8 || (chained && !exact)) return 0;
  std::vector<uint32_t> lower, bounds, upper;
  if (exact) {
    uint32_t T = 2;
    while (T < SWEEP_TEAM_MAX && (T + 1) * (T + 1) <= n) ++T;
    for (uint32_t s = 0; s <= T; ++s) bounds.push_back((uint32_t)((unsigned long long)n * s / T));
    lower.assign(n, 0);
    for (uint32_t s = 0; s < T; ++s) lower[bounds[s]] = TOK_START;
    upper.assign(T, 0);
    upper[0] = TOK_START;
  } else {
    std::vector<int> reps;
    Expr top(h, reps, rounds);
    int level = -1;
    // the level that makes a section and the list of sections shortest together;
    // with more than 32 sections where there is no other, or in a pass of few
    // units where that leaves fewer sources in series: those of the sections
    // that a warp takes in turn, and the values, which come from shared memory
    // and take two thirds of the time
    auto series = [&](uint32_t T) { return 3 * ((T + 15) / 16 * ((n + T - 1) / T)) + 2 * T; };
    for (int l = 0; l < (int)h.size(); ++l) {
      std::vector<uint32_t> b;
      for (size_t a = 0; a < n; a = top.next_in(leaves, a, n, l)) b.push_back((uint32_t)a);
      const uint32_t T = (uint32_t)b.size(), T0 = (uint32_t)bounds.size();
      if (T > SWEEP_TEAM_MAX || T == n) break;
      if (T < 2) continue;
      if (level >= 0 && (T <= 32 ? n / T + T >= n / T0 + T0 : !few || series(T) >= series(T0))) continue;
      level = l;
      bounds = b;
    }
    if (level < 0) return 0;
    for (uint32_t a : bounds) reps.push_back(leaves[a]);
    bounds.push_back(n);
    // (sections of one shape have the same tokens: for 64 groups of one size
    // planning takes 6 us less)
    const long long below = top.G[level + 1];
    for (size_t s = 0; s + 1 < bounds.size(); ++s) {
      const uint32_t lo = bounds[s], hi = bounds[s + 1];
      bool same = s > 0 && hi - lo == lo - bounds[s - 1];
      for (uint32_t k = 0; same && k < hi - lo; ++k)
        same = leaves[lo + k] % below == leaves[bounds[s - 1] + k] % below;
      if (same) {
        for (uint32_t k = 0; k < hi - lo; ++k) lower.push_back(lower[bounds[s - 1] + k]);
        continue;
      }
      Expr e(h, leaves, rounds);
      e.group(lo, hi, level + 1, false);
      uint32_t d = 0;
      if (!e.finish(d)) return 0;
      depth = std::max(depth, d);
      lower.insert(lower.end(), e.toks.begin(), e.toks.end());
    }
    top.group(0, reps.size(), 0, false);
    uint32_t d = 0;
    if (!top.finish(d)) return 0;
    depth = std::max(depth, d);
    upper = top.toks;
  }
  toks.insert(toks.end(), lower.begin(), lower.end());
  toks.insert(toks.end(), bounds.begin(), bounds.end());
  toks.insert(toks.end(), upper.begin(), upper.end());
  return (uint32_t)upper.size();
}

constexpr uint32_t NONE = 0xffffffffu;

// The operands of a member are ops[src .. src + nsrc) and ops[dst .. dst + ndst),
// where up to `room` fit.
struct Member {
  unsigned long long nbytes;
  uint32_t src, nsrc, dst, ndst, room;
  uint32_t rop, tok, team, ttok;
};

// Width of the accesses that every operand of a member allows: 16 bytes when
// all lie equally far off a 16-byte boundary (whole vectors between a few
// elements at both ends), told as 32 when they lie equally far off a 32-byte
// sector (the vectors then start with one), else the widest of 4 and 2 that
// the addresses (and the length) share.
uint32_t width_log2(const Member &m, const std::vector<unsigned long long> &ops) {
  const unsigned long long *src = &ops[m.src], *dst = &ops[m.dst], base = src[0];
  unsigned long long a = 0, off = 0;
  for (uint32_t k = 0; k < m.nsrc; ++k) a |= src[k], off |= src[k] ^ base;
  for (uint32_t k = 0; k < m.ndst; ++k) a |= dst[k], off |= dst[k] ^ base;
  if (off % 16 == 0) return off % 32 == 0 ? 5 : 4;
  return a % 4 == 0 && m.nbytes % 4 == 0 ? 2 : 1;
}

// bytes of a member that a warp moves with one vector per lane
unsigned long long row_bytes(uint32_t kern, const SweepClass &k) {
  if (kern == SWEEP_FP8 || kern == SWEEP_FP8_TEAM) return 4 * FP8_BLOCK_BYTES;
  return kern == SWEEP_SHIFT ? 31 * 16 : 32ull << std::min(sweep_lw(k.meta), 4u);
}

// units that store one range of a member to all its destinations
unsigned long long groups(const SweepClass &k) {
  return k.nsrc > 1 ? 1 : (k.ndst + SWEEP_GROUP - 1) / SWEEP_GROUP;
}

// Launches, vectors per lane and units of a sweep's classes.
void plan_launches(Sweep &sw) {
  bool folds = false;   // a launch of SWEEP_FOLD, which copies can join
  unsigned long long fold_units = 0;
  auto fold_kernel = [](const SweepClass &k) -> uint32_t {
    return sweep_dtype(k.meta) == HICCL_FP8E4M3 ? SWEEP_FP8 : SWEEP_FOLD;
  };
  auto folded = [](const SweepClass &k) { return k.nsrc > 1 && sweep_lw(k.meta) >= 4; };
  for (const SweepClass &k : sw.classes)
    if (folded(k)) fold_units += (k.nbytes + row_bytes(fold_kernel(k), k) - 1) / row_bytes(fold_kernel(k), k) * k.nmem;
  auto teamed = [&](const SweepClass &k) {
    return k.team > 1 && fold_units < (k.team > 32 ? SWEEP_TEAM_MANY : SWEEP_TEAM_UNITS);
  };
  for (const SweepClass &k : sw.classes) folds |= folded(k) && !teamed(k) && fold_kernel(k) == SWEEP_FOLD;
  auto kernel_of = [&](const SweepClass &k) -> uint32_t {
    if (sweep_lw(k.meta) < 4) return k.nsrc > 1 ? SWEEP_NARROW : SWEEP_SHIFT;
    if (!folded(k)) return folds ? SWEEP_FOLD : SWEEP_COPY;
    if (teamed(k)) return fold_kernel(k) == SWEEP_FP8 ? SWEEP_FP8_TEAM : SWEEP_TEAM;
    return fold_kernel(k);
  };
  std::stable_sort(sw.classes.begin(), sw.classes.end(),
                   [&](const SweepClass &a, const SweepClass &b) { return kernel_of(a) < kernel_of(b); });
  sw.launches.clear();
  sw.hints.clear();
  for (size_t a = 0; a < sw.classes.size();) {
    const uint32_t kern = kernel_of(sw.classes[a]);
    size_t z = a;
    unsigned long long rows = 0;   // units of one vector per lane
    for (; z < sw.classes.size() && kernel_of(sw.classes[z]) == kern; ++z) {
      const SweepClass &k = sw.classes[z];
      const unsigned long long row = row_bytes(kern, k);
      rows += (k.nbytes + row - 1) / row * k.nmem * groups(k);
    }
    unsigned long long units = 0;
    uint32_t words = 0;
    for (size_t i = a; i < z; ++i) {
      SweepClass &k = sw.classes[i];
      const uint32_t dt = sweep_dtype(k.meta), lw = sweep_lw(k.meta);
      uint32_t v = 1;
      constexpr uint32_t WARPS = SWEEP_SMS * 16;   // that keep every SM busy
      if (kern == SWEEP_SHIFT) v = rows >= 4 * WARPS ? 4 : 1;
      else if (kern == SWEEP_NARROW) v = rows >= 8 * WARPS ? 8 : rows >= 2 * WARPS ? 2 : 1;
      else if (k.nsrc == 1) v = rows >= 4096 ? 4 : rows >= 2048 ? 2 : 1;
      const unsigned long long unit = row_bytes(kern, k) * v;
      const unsigned long long upm = (k.nbytes + unit - 1) / unit;
      k.meta = sweep_meta(dt, sweep_rop(k.meta), lw, v, kern);
      k.unit0 = (uint32_t)units;
      k.upm = (uint32_t)upm;
      k.group = k.nsrc > 1 ? k.ndst : SWEEP_GROUP;
      units += upm * k.nmem * groups(k);
      if (units > 0xF0000000ull) {   // far beyond device memory
        sw.valid = false;
        return;
      }
      // accumulator words of a lane: 32-bit values, or BF16 / FP8 values widened to 32 bits
      const uint32_t acc = kern == SWEEP_FP8 || kern == SWEEP_FP8_TEAM ? 16 : lw >= 4 ? (dt == HICCL_BF16 ? 8 : 4) : lw == 2 && dt == HICCL_BF16 ? 2 : 1;
      if (k.nsrc > 1) words = std::max(words, sw.depth * acc * v);
    }
    SweepLaunch L{kern, (uint32_t)a, (uint32_t)z, (uint32_t)units, 0, words, (uint32_t)sw.hints.size(), 0};
    if (z - a > SWEEP_PREFIX)
      for (size_t i = a, u = 0; u <= units + (1u << SWEEP_HINT_SHIFT); u += 1u << SWEEP_HINT_SHIFT) {
        while (i + 1 < z && sw.classes[i + 1].unit0 <= u) ++i;
        sw.hints.push_back((uint32_t)(i - a));
      }
    const uint32_t most = SWEEP_THREADS[kern];
    // a short pass uses small CTAs, so that its units reach every SM
    uint32_t warps = most / 32;
    const bool team = kern == SWEEP_TEAM || kern == SWEEP_FP8_TEAM;
    while (!team && warps > 1 && units < (unsigned long long)warps * (2 * SWEEP_SMS)) warps /= 2;
    // a team's warps: no more than sections, and enough for SWEEP_TEAM_WARPS in all
    uint32_t sections = 1;
    for (size_t i = a; team && i < z; ++i) sections = std::max(sections, sw.classes[i].team);
    L.sections = team ? sections : 0;
    while (team && warps > sections) warps /= 2;
    while (team && warps > 1 && units * (warps / 2) >= SWEEP_TEAM_WARPS) warps /= 2;
    L.threads = warps * 32;
    sw.launches.push_back(L);
    a = z;
  }
}

// Classes of equal shape, in order of first appearance.  (Neighbours are mostly
// alike: the maps are searched where a member differs from the one before.)
void make_classes(const hiccl_comm &c, const std::vector<Member> &ms, const std::vector<unsigned long long> &ops,
                  Sweep &sw) {
  // copies of one shape go together, as misaligned as the worst of them: in an
  // All-to-all of odd chunks one pair of ranks in eight happens to agree, and a
  // launch of its own costs its ramp (64 ranks x 1 MiB of BF16: 27.5 us with
  // it, 25.1 us without)
  std::map<std::pair<unsigned long long, uint32_t>, uint32_t> shapes;
  std::vector<uint32_t> widths(ms.size());
  auto alike = [](const Member &a, const Member &b) { return a.nbytes == b.nbytes && a.nsrc == b.nsrc && a.ndst == b.ndst; };
  uint32_t *worst = nullptr;
  auto shape_of = [&](size_t i) -> uint32_t & {
    if (!i || !worst || !alike(ms[i], ms[i - 1])) worst = &shapes.emplace(std::make_pair(ms[i].nbytes, ms[i].ndst), 5u).first->second;
    return *worst;
  };
  for (size_t i = 0; i < ms.size(); ++i) {
    widths[i] = width_log2(ms[i], ops);
    if (ms[i].nsrc > 1) continue;
    uint32_t &w = shape_of(i);
    w = std::min(w, widths[i]);
  }
  using Key = std::tuple<unsigned long long, uint32_t, uint32_t, uint32_t, uint32_t, uint32_t>;
  std::map<Key, uint32_t> at;
  std::vector<uint32_t> first, class_of(ms.size());   // first member of a class, class of a member
  size_t nptrs = 0;
  for (size_t i = 0; i < ms.size(); ++i) {
    const Member &m = ms[i];
    if (m.nsrc == 1) widths[i] = shape_of(i);
    if (i && alike(m, ms[i - 1]) && m.rop == ms[i - 1].rop && m.tok == ms[i - 1].tok && widths[i] == widths[i - 1]) {
      class_of[i] = class_of[i - 1];
    } else {
      const Key k(m.nbytes, m.nsrc, m.ndst, m.rop, m.tok, widths[i]);
      class_of[i] = at.emplace(k, (uint32_t)first.size()).first->second;
      if (class_of[i] == first.size()) first.push_back((uint32_t)i);
    }
    nptrs += m.nsrc + m.ndst;
  }
  for (uint32_t i : first) {
    const Member &m = ms[i];
    SweepClass k{};
    k.nbytes = m.nbytes;
    k.nsrc = m.nsrc;
    k.ndst = m.ndst;
    k.tok = m.tok;
    k.team = m.team;
    k.ttok = m.ttok;
    k.meta = sweep_meta((uint32_t)c.dtype, m.rop, widths[i], 1, 0);
    sw.classes.push_back(k);
  }
  for (uint32_t k : class_of) ++sw.classes[k].nmem;
  size_t ptr = 0;
  std::vector<size_t> to;
  for (SweepClass &k : sw.classes) {
    k.ptr = ptr;
    to.push_back(ptr);
    ptr += (size_t)k.nmem * (k.nsrc + k.ndst);
  }
  sw.ptrs.resize(nptrs);
  for (size_t i = 0; i < ms.size(); ++i) {
    const Member &m = ms[i];
    size_t &q = to[class_of[i]];
    for (uint32_t k = 0; k < m.nsrc; ++k) sw.ptrs[q++] = ops[m.src + k];
    for (uint32_t k = 0; k < m.ndst; ++k) sw.ptrs[q++] = ops[m.dst + k];
  }
  sw.valid = true;
  plan_launches(sw);
}

// ---- the check of a sweep ------------------------------------------------------

// Byte ranges joined to disjoint spans.
struct Bytes {
  struct Span {
    unsigned long long lo, hi;
  };
  std::vector<Span> v;
  void join() {
    auto before = [](const Span &a, const Span &b) { return a.lo < b.lo; };
    if (!std::is_sorted(v.begin(), v.end(), before)) std::sort(v.begin(), v.end(), before);
    size_t w = 0;
    for (size_t k = 1; k < v.size(); ++k) {
      if (v[k].lo <= v[w].hi) v[w].hi = std::max(v[w].hi, v[k].hi);
      else v[++w] = v[k];
    }
    if (!v.empty()) v.resize(w + 1);
  }
  // the span that holds [lo, hi), if any
  const Span *find(unsigned long long lo, unsigned long long hi) const {
    auto it = std::upper_bound(v.begin(), v.end(), lo, [](unsigned long long a, const Span &s) { return a < s.lo; });
    return it == v.begin() || hi > (--it)->hi ? nullptr : &*it;
  }
};
// Ranges of nbytes, each mostly in the span of the one before or in the next one
// (members take the ranks' rows in turn).
struct Inside {
  const Bytes &in;
  const unsigned long long nbytes;
  size_t at = 0;
  Inside(const Bytes &b, unsigned long long n) : in(b), nbytes(n) {}
  bool holds(size_t k, unsigned long long a) const {
    return k < in.v.size() && a >= in.v[k].lo && a + nbytes <= in.v[k].hi;
  }
  bool operator()(unsigned long long a) {
    if (holds(at, a)) return true;
    if (holds(at + 1, a)) {
      ++at;
      return true;
    }
    const Bytes::Span *s = in.find(a, a + nbytes);
    if (s) at = s - in.v.data();
    return s != nullptr;
  }
};
// what a program reads or writes, and what it writes
void join_ranges(const Ranges &ranges, int P, Bytes &all, Bytes &written) {
  struct Open {
    unsigned long long lo = 0, hi = 0;
  };
  std::vector<Open> open(2 * (size_t)P);   // by direction and rank: its ranges mostly continue one another
  all.v.reserve(open.size());
  written.v.reserve(P);
  auto close = [&](const Open &o, bool write) {
    if (o.lo == o.hi) return;
    all.v.push_back(Bytes::Span{o.lo, o.hi});
    if (write) written.v.push_back(Bytes::Span{o.lo, o.hi});
  };
  for (const Range &r : ranges.all) {
    Open &o = open[(r.write ? P : 0) + r.rank];
    if (r.lo <= o.hi && r.hi >= o.lo && o.lo != o.hi) {
      o.lo = std::min(o.lo, r.lo);
      o.hi = std::max(o.hi, r.hi);
    } else {
      close(o, r.write);
      o.lo = r.lo;
      o.hi = r.hi;
    }
  }
  for (size_t k = 0; k < open.size(); ++k) close(open[k], k >= (size_t)P);
  all.join();
  written.join();
}

// Do n tokens start with a value, save and take back in balance and never hold
// more than `most` values?
bool balanced(const uint32_t *tok, uint32_t n, uint32_t most) {
  if (n == 0 || (tok[0] & 3u) != TOK_START) return false;
  uint32_t sp = 0;
  for (uint32_t k = 0; k < n; ++k) {
    if (k && (tok[k] & 3u) == TOK_START) return false;   // would lose the accumulator
    if ((tok[k] & 3u) == TOK_PUSH) return false;
    if ((tok[k] & TOK_PUSH) && ++sp > most) return false;
    for (uint32_t o = tok[k] >> TOK_OPS; o; o >>= 2) {
      if ((o & 3u) == 0) return false;
      if ((o & 3u) >= TOK_POP && sp-- == 0) return false;
    }
  }
  return sp == 0;
}

}  // namespace

// (Every plan pays for its sweep, so this shares the ranges and conflicts that
// the step table needs anyway and keeps all operands in one list.  Planning's
// share for 64 ranks: All-reduce 33 us, with ranges sorted anew and two vectors
// a member 330 us; All-to-all 150 against 490 us.)
void build_sweep(const hiccl_comm &c, const std::vector<int> &hierarchy, int ring_lvl,
                 const Ranges &ranges, const std::vector<Conflict> &conflicts, Sweep &sw) {
  sw = Sweep();
  if (c.epochs > 32) return;   // (nothing measured beyond)
  std::vector<Member> ms;
  std::vector<unsigned long long> ops, mine;
  std::vector<uint32_t> member_of(c.prims.size(), NONE);
  std::vector<Program> progs;
  ms.reserve(c.prims.size());
  ops.reserve(ranges.all.size());
  const long long node_ranks = c.P / c.ring;
  const unsigned long long row = c.dtype == HICCL_FP8E4M3 ? 4 * FP8_BLOCK_BYTES : 512;
  unsigned long long units = 0;   // of the folds
  for (const Prim &p : c.prims)
    if (p.kind == 1 && p.leaves.size() > 1) units += ((unsigned long long)p.count * c.esize + row - 1) / row;
  const bool few = c.dtype != HICCL_FP8E4M3 && units < SWEEP_TEAM_FEW;
  size_t next = 0;   // conflict
  for (size_t i = 0; i < c.prims.size(); ++i) {
    const Prim &p = c.prims[i];
    while (next < conflicts.size() && conflicts[next].later < i) ++next;
    const size_t r0 = ranges.of[i], r1 = ranges.of[i + 1], ops0 = ops.size();
    if (r0 == r1) continue;
    Member m{};
    m.nbytes = ranges.all[r0].hi - ranges.all[r0].lo;
    m.src = (uint32_t)ops0;
    if (p.kind == 0 || p.leaves.size() == 1) {   // copies (one input: the operator is omitted)
      if (ranges.all[r0].write || r1 - r0 < 2) continue;   // in place: nothing to do
      m.nsrc = 1;
      ops.resize(ops0 + (r1 - r0));
      for (size_t r = r0; r < r1; ++r) ops[ops0 + (r - r0)] = ranges.all[r].lo;
    } else {
      const bool rounds = p.op == HICCL_SUM && (c.dtype == HICCL_BF16 || c.dtype == HICCL_FP8E4M3);
      const bool exact = p.op != HICCL_SUM || c.dtype == HICCL_I32;
      const long long node = c.ring > 1 ? p.root / node_ranks : -1;
      const Program *pg = nullptr;
      for (size_t k = progs.size(); k-- > 0 && !pg && k + 64 > progs.size();)
        if (progs[k].node == node && progs[k].rounds == rounds && progs[k].exact == exact && progs[k].leaves == p.leaves) pg = &progs[k];
      if (!pg) {
        Expr e(hierarchy, p.leaves, rounds);
        if (c.ring > 1) e.chain(c.ring, ring_lvl, node);
        else e.group(0, p.leaves.size(), 0, false);
        uint32_t depth = 0;
        if (!e.finish(depth)) return;
        const uint32_t tok = (uint32_t)sw.toks.size();
        sw.toks.insert(sw.toks.end(), e.toks.begin(), e.toks.end());
        const uint32_t ttok = (uint32_t)sw.toks.size();
        const uint32_t team = two_steps(hierarchy, p.leaves, rounds, exact, c.ring > 1, few, sw.toks, depth);
        sw.depth = std::max(sw.depth, depth);
        progs.push_back(Program{p.leaves, node, rounds, exact, e.order, tok, team, ttok});
        pg = &progs.back();
      }
      m.nsrc = (uint32_t)pg->order.size();
      for (int r : pg->order) ops.push_back(p.send[r]);
      ops.push_back(p.recv[p.root]);
      m.rop = (uint32_t)p.op;
      m.tok = pg->tok;
      m.team = pg->team;
      m.ttok = pg->ttok;
    }
    m.dst = m.src + m.nsrc;
    m.ndst = m.room = (uint32_t)(ops.size() - m.dst);
    // earlier epochs: no conflict, or a copy of exactly what one expression
    // stores (whose sources it may overwrite in place)
    uint32_t with = NONE;
    bool again = false;   // a destination that was written before
    for (; next < conflicts.size() && conflicts[next].later == i; ++next) {
      const Conflict &x = conflicts[next];
      const uint32_t k = member_of[x.earlier];
      if (k == NONE) continue;                                  // it does nothing
      if (!x.same || (with != NONE && with != k)) return;       // part of a value, or two of them
      with = k;
      again |= x.rewrites;
    }
    if (with == NONE) {
      member_of[i] = (uint32_t)ms.size();
      ms.push_back(m);
      continue;
    }
    // the copy's source has to hold the expression's value
    Member &x = ms[with];
    auto stored = [&](unsigned long long a) {
      return std::find(ops.begin() + x.dst, ops.begin() + x.dst + x.ndst, a) != ops.begin() + x.dst + x.ndst;
    };
    const unsigned long long from = ops[m.src];
    if (m.nsrc != 1 || !(stored(from) || (x.nsrc == 1 && ops[x.src] == from))) return;
    member_of[i] = with;
    // its destinations follow those that the expression has; a list without
    // room moves to the end, with room for as many again
    mine.clear();
    for (uint32_t k = m.dst; k < m.dst + m.ndst; ++k)
      if (!again || !stored(ops[k])) mine.push_back(ops[k]);
    ops.resize(ops0);
    const uint32_t all = x.ndst + (uint32_t)mine.size();
    if (all > x.room) {
      x.room = std::max(all, 2 * x.ndst);
      ops.resize(ops0 + x.room);
      std::copy_n(ops.begin() + x.dst, x.ndst, ops.begin() + ops0);
      x.dst = (uint32_t)ops0;
    }
    std::copy(mine.begin(), mine.end(), ops.begin() + x.dst + x.ndst);
    x.ndst = all;
  }
  make_classes(c, ms, ops, sw);
}

bool check_sweep(const hiccl_comm &c, const Ranges &ranges, const Sweep &sw, std::string &why) {
  auto bad = [&](const std::string &m) {
    why = "sweep: " + m;
    return false;
  };
  Bytes all, written;   // (a group has no primitives; its members were checked)
  if (!c.group) join_ranges(ranges, c.P, all, written);
  size_t next = 0;       // class
  for (const SweepLaunch &L : sw.launches) {
    if (L.class_lo != next || L.class_hi <= L.class_lo || L.class_hi > sw.classes.size() || L.kernel >= SWEEP_KERNELS)
      return bad("launches do not divide the classes");
    next = L.class_hi;
    if (L.threads < 32 || L.threads % 32 || L.threads > SWEEP_THREADS[L.kernel] || L.stack_words > SWEEP_MAX_DEPTH * 16)
      return bad("a launch has a bad shape");
    const bool team = L.kernel == SWEEP_TEAM || L.kernel == SWEEP_FP8_TEAM;
    unsigned long long units = 0;
    for (size_t i = L.class_lo; i < L.class_hi; ++i) {
      const SweepClass &k = sw.classes[i];
      const std::string at = "class " + std::to_string(i);
      const uint32_t dt = sweep_dtype(k.meta), lw = sweep_lw(k.meta), v = sweep_v(k.meta);
      const bool fold = k.nsrc > 1, fp8 = dt == HICCL_FP8E4M3;
      const uint32_t elem = fp8 ? 16 : dt == HICCL_BF16 ? 2 : 4;
      // a kernel that handles the class
      bool runs = sweep_kernel(k.meta) == L.kernel && k.nsrc && k.ndst && k.nmem && k.nbytes;
      switch (L.kernel) {
        case SWEEP_COPY: runs = runs && !fold && lw >= 4; break;
        case SWEEP_FOLD: runs = runs && lw >= 4 && !(fold && fp8); break;
        case SWEEP_FP8: case SWEEP_FP8_TEAM: runs = runs && fold && fp8 && lw >= 4; break;
        case SWEEP_NARROW: runs = runs && fold && !fp8 && (lw == 2 || (lw == 1 && dt == HICCL_BF16)); break;
        case SWEEP_SHIFT: runs = runs && !fold; break;
        default: runs = runs && fold && !fp8 && lw >= 4; break;
      }
      if (!runs) return bad(at + " does not fit its kernel");
      // units that tile the members
      const unsigned long long unit = row_bytes(L.kernel, k) * v;
      if (!v || k.unit0 != units || (k.upm - 1ull) * unit >= k.nbytes || k.upm * unit < k.nbytes || !k.group ||
          (fold && k.group != k.ndst))
        return bad("units of " + at + " do not tile it");
      units += (unsigned long long)k.upm * k.nmem * ((k.ndst + k.group - 1) / k.group);
      // operands inside the buffers, as far off a boundary as the kernel's accesses allow
      const unsigned long long n = (unsigned long long)k.nsrc + k.ndst;
      if (k.ptr > sw.ptrs.size() || k.nmem > (sw.ptrs.size() - k.ptr) / n) return bad("operands of " + at + " are missing");
      Inside readable(all, k.nbytes), writable(written, k.nbytes);
      const unsigned long long mask = (1ull << lw) - 1;
      for (uint32_t m = 0; m < k.nmem; ++m) {
        const unsigned long long *p = &sw.ptrs[k.ptr + m * n];
        bool in = true;
        unsigned long long off = 0, low = 0;
        for (uint32_t q = 0; q < k.nsrc; ++q) in = in && (c.group || readable(p[q]));
        for (uint32_t q = k.nsrc; q < n; ++q) in = in && (c.group || writable(p[q]));
        if (!in) return bad("an operand of " + at + " lies outside the primitives' buffers");
        for (uint32_t q = 0; q < n; ++q) off |= p[q] ^ p[0], low |= p[q];
        if (((low | k.nbytes) & (elem - 1)) || ((lw >= 4 ? off : fold ? low | k.nbytes : 0) & mask))
          return bad("operands of " + at + " are not aligned");
      }
      if (!fold) continue;
      // expressions that fit the saved values
      const uint32_t acc = fp8 ? 16 : lw >= 4 ? (dt == HICCL_BF16 ? 8 : 4) : lw == 2 && dt == HICCL_BF16 ? 2 : 1;
      const uint32_t most = L.stack_words / (acc * v);
      if (k.tok > sw.toks.size() || k.nsrc > sw.toks.size() - k.tok || !balanced(&sw.toks[k.tok], k.nsrc, most))
        return bad("tokens of " + at + " are not an expression");
      if (!team) continue;
      const size_t need = (size_t)k.nsrc + 2 * k.team + 1;
      if (k.team < 2 || k.team > L.sections || L.sections > SWEEP_TEAM_MAX || k.ttok > sw.toks.size() || need > sw.toks.size() - k.ttok)
        return bad("the two steps of " + at + " are missing");
      const uint32_t *t = &sw.toks[k.ttok], *b = t + k.nsrc;
      bool good = b[0] == 0 && b[k.team] == k.nsrc && balanced(b + k.team + 1, k.team, most);
      for (uint32_t s = 0; s < k.team && good; ++s)
        good = b[s] < b[s + 1] && b[s + 1] <= k.nsrc && balanced(t + b[s], b[s + 1] - b[s], most);
      if (!good) return bad("the two steps of " + at + " are not an expression");
    }
    if (units != L.units) return bad("a launch has another number of units than its classes");
    if (L.class_hi - L.class_lo > SWEEP_PREFIX) {   // every unit's class lies between two hints
      const size_t nh = (size_t)((units - 1) >> SWEEP_HINT_SHIFT) + 2, nc = L.class_hi - L.class_lo;
      if (L.hint > sw.hints.size() || nh > sw.hints.size() - L.hint) return bad("hints are missing");
      const SweepClass *k = &sw.classes[L.class_lo];
      for (size_t i = 0; i < nh; ++i) {
        const size_t h = sw.hints[L.hint + i];
        const unsigned long long u = (unsigned long long)i << SWEEP_HINT_SHIFT;
        if (h >= nc || k[h].unit0 > u || (h + 1 < nc && k[h + 1].unit0 <= u)) return bad("a hint names a wrong class");
      }
    }
  }
  return next == sw.classes.size() || bad("launches do not divide the classes");
}

void group_sweep(const std::vector<const Sweep *> &members, Sweep &sw) {
  sw = Sweep();
  for (const Sweep *m : members)
    if (!m->valid) return;
  for (const Sweep *m : members) {
    for (SweepClass k : m->classes) {
      k.ptr += sw.ptrs.size();
      k.tok += (uint32_t)sw.toks.size();
      k.ttok += (uint32_t)sw.toks.size();
      sw.classes.push_back(k);
    }
    sw.ptrs.insert(sw.ptrs.end(), m->ptrs.begin(), m->ptrs.end());
    sw.toks.insert(sw.toks.end(), m->toks.begin(), m->toks.end());
    sw.depth = std::max(sw.depth, m->depth);
  }
  sw.valid = true;
  plan_launches(sw);
}

}  // namespace hiccl
