// Step programs: which steps of a pass share a launch, how their work is cut
// into CTA-sized units, and in which order the units are taken (host only;
// the kernel is k_program in exec.cu).
#include <algorithm>
#include <cmath>

#include "host.h"

namespace qgm {

namespace {

// A step is launched on its own when it loads at least kAlone values (its
// 2^(w + k) products times its inputs, counted in 16-byte pairs of batch
// entries) for at least kAloneItems items (rows times pairs): there the
// kernels specialised by input count and tile, with every CTA on one step,
// beat the program's units.  A long sum over few items stays in the program,
// which splits it over the machine.
constexpr double kAlone = 4194304.0;
constexpr double kAloneItems = 65536.0;

// Lanes wanted for one step: about two CTAs of 256 on each SM
constexpr int64_t kLanes = 65536;
// Units of a step: as many as two CTAs an SM can take (a pass over 256 lanes
// each: the passes of a unit run one after another, about 0.6 us each), then
// larger units up to kLoads loads per thread, which amortises a unit's setup
constexpr int kUnits = 304, kLoads = 32;

double step_items(const StepDesc &d, int Bp) { return std::ldexp(d.batched_out ? Bp / 2 : 1.0, d.w_out); }

bool fits(const StepDesc &d, int Bp) {
  for (int i = 0; i < d.m; ++i) {
    int rank = 0;
    for (int q = 0; q < d.in[i].nruns; ++q) rank += d.in[i].len[q];
    if (rank + 3 > 30 || std::ldexp(d.in[i].batched ? 8.0 * Bp : 8.0, rank) >= 2147483648.0) return false;
  }
  return d.k < 24 && step_items(d, Bp) < 1073741824.0;
}

// Input i of a step summing union bits [w, w + k): row runs and term runs
// (term bits counted from w).
PIn make_in(const InDesc &in, int w, int64_t off_meta) {
  PIn p{};
  p.off = in.off;
  p.meta = in.meta >= 0 ? off_meta + 8 * (int64_t)in.meta : -1;
  p.batched = in.batched;
  std::vector<uint32_t> row, term;
  for (int q = 0; q < in.nruns; ++q) {
    const int s = in.src[q], l = in.len[q], d = in.dst[q];
    const int nr = std::max(0, std::min(l, w - s));
    if (nr > 0) row.push_back((uint32_t)(s | nr << 8 | d << 16));
    if (nr < l) term.push_back((uint32_t)((s + nr - w) | (l - nr) << 8 | (d + nr) << 16));
  }
  p.nrow = (int16_t)row.size();
  p.nterm = (int16_t)term.size();
  std::copy(row.begin(), row.end(), p.run);
  std::copy(term.begin(), term.end(), p.run + row.size());
  return p;
}

void set_units(PStep &s) {
  s.lg = 0;
  while (s.lg < 5 && s.k - s.lg > 2 && ((int64_t)s.items << (s.lg + 1)) <= kLanes / 2) ++s.lg;
  const int per_pass = 256 >> s.lg;
  const int64_t loads = ((int64_t)1 << (s.k - s.lg)) * s.m;  // per item and lane
  const int64_t one_pass = (s.items + per_pass - 1) / per_pass;
  const int64_t passes = std::max<int64_t>(1, std::min<int64_t>(kLoads / loads, (one_pass + kUnits - 1) / kUnits));
  s.unit_items = (int)std::min<int64_t>(per_pass * passes, s.items);
  s.n_units = (s.items + s.unit_items - 1) / s.unit_items;
}

}  // namespace

bool program_alone(const StepDesc &d, int Bp) {
  const double items = step_items(d, Bp);
  // (the kernels for single steps tabulate at most 16 summed variables)
  return d.gemm >= 0 || (items >= kAloneItems && d.k <= 16 && std::ldexp(items * d.m, d.k) >= kAlone) || !fits(d, Bp);
}

void build_program(Program &P, int Bp, int64_t off_meta, const std::vector<char> &alone) {
  const int n = (int)P.all.size();
  P.steps.clear();
  P.tasks.clear();
  P.ops.clear();
  P.n_segments = 0;
  P.n_tmp = 0;
  P.tmp_bytes = 0;
  // phase of a step: a large step b of the launch order belongs to phase b
  // (after segment b), a small one to the first segment after its producers
  std::vector<int> phase(n, 0), big_of;
  std::vector<char> big(n, 0);
  for (int s = 0; s < n; ++s) {
    const StepDesc &d = P.all[s];
    big[s] = alone[s] || program_alone(d, Bp);
    if (big[s]) {
      phase[s] = (int)big_of.size();
      big_of.push_back(s);
    } else {
      for (int q : P.prod[s])
        if (q >= 0) phase[s] = std::max(phase[s], big[q] ? phase[q] + 1 : phase[q]);
    }
  }
  // small steps as PSteps; a long sum over few outputs is split in two: the
  // sum over its low summed variables for every value of the high ones, into
  // a temporary, then the sum over those
  struct Node {
    PStep s;
    int phase;
    std::vector<int> deps;  // nodes
    double height = 0;
    int chain = -1;
  };
  std::vector<Node> nodes;
  std::vector<int> node_of(n, -1);
  std::vector<std::vector<int>> readers;
  auto add = [&](Node &&nd) {
    nodes.push_back(std::move(nd));
    readers.emplace_back();
    const int id = (int)nodes.size() - 1;
    for (int q : nodes[id].deps) readers[q].push_back(id);
    return id;
  };
  for (int s = 0; s < n; ++s) {
    if (big[s]) continue;
    const StepDesc &d = P.all[s];
    Node nd;
    PStep &t = nd.s;
    t = PStep{};
    nd.phase = phase[s];
    t.m = d.m;
    t.k = d.k;
    t.w_out = d.w_out;
    t.batched = d.batched_out;
    t.out_off = d.out_off;
    t.out_meta = off_meta + 8 * (int64_t)d.out_meta;
    t.pairs = d.batched_out ? Bp / 2 : 1;
    t.items = t.pairs << d.w_out;
    for (int q : P.prod[s])
      if (q >= 0 && !big[q] && phase[q] == phase[s] && std::find(nd.deps.begin(), nd.deps.end(), node_of[q]) == nd.deps.end())
        nd.deps.push_back(node_of[q]);
    set_units(t);
    int hi = 0;  // summed variables left to the second step
    while (t.k - hi - t.lg > 5 && ((int64_t)t.items << (t.lg + hi)) < kLanes) ++hi;
    if (hi < 2) {
      for (int i = 0; i < d.m; ++i) t.in[i] = make_in(d.in[i], d.w_out, off_meta);
      node_of[s] = add(std::move(nd));
      continue;
    }
    const int64_t rows = (int64_t)1 << d.w_out;
    Node second = nd;
    second.deps.clear();
    // first: summed bits [w, w + k - hi); the high summed bits become its top
    // row bits.  In the union the kept bits are [0, w) and the summed ones
    // above, so the first step's union has its rows' high part above its
    // terms: the runs' sources are moved accordingly.
    const int w = d.w_out, lo = d.k - hi;
    t.w_out = w + hi;
    t.k = lo;
    t.items = (int)((int64_t)t.pairs << t.w_out);
    for (int i = 0; i < d.m; ++i) {
      PIn p{};
      const PIn f = make_in(d.in[i], w, off_meta);
      p.off = f.off;
      p.meta = f.meta;
      p.batched = f.batched;
      std::vector<uint32_t> row(f.run, f.run + f.nrow), term;
      for (int q = 0; q < f.nterm; ++q) {
        const uint32_t r = f.run[f.nrow + q];
        const int src = r & 255, len = r >> 8 & 255, dst = r >> 16;
        const int a = std::max(0, std::min(len, lo - src));
        if (a > 0) term.push_back((uint32_t)(src | a << 8 | dst << 16));
        if (a < len) row.push_back((uint32_t)((src + a - lo + w) | (len - a) << 8 | (dst + a) << 16));
      }
      p.nrow = (int16_t)row.size();
      p.nterm = (int16_t)term.size();
      std::copy(row.begin(), row.end(), p.run);
      std::copy(term.begin(), term.end(), p.run + row.size());
      t.in[i] = p;
    }
    t.out_off = -1 - P.tmp_bytes;  // placed by place_program
    t.out_meta = -1 - P.n_tmp;
    set_units(t);
    PStep &u = second.s;
    u.m = 1;
    u.k = hi;
    u.in[0] = PIn{};
    u.in[0].off = t.out_off;
    u.in[0].meta = t.out_meta;
    u.in[0].batched = d.batched_out;
    if (w > 0) u.in[0].run[u.in[0].nrow++] = (uint32_t)(0 | w << 8 | 0 << 16);
    u.in[0].run[u.in[0].nrow] = (uint32_t)(0 | hi << 8 | w << 16);
    u.in[0].nterm = 1;
    set_units(u);
    P.tmp_bytes += ((rows << hi) * (d.batched_out ? Bp : 1) * 8 + 255) & ~int64_t(255);
    P.n_tmp += 1;
    second.deps.push_back(add(std::move(nd)));
    node_of[s] = add(std::move(second));
  }
  const int nn = (int)nodes.size();
  // order within a phase: longest remaining path first.  A step's cost is
  // its fixed latency and its share of the machine; every cost is positive,
  // so producers come before consumers.
  for (int i = nn - 1; i >= 0; --i) {
    const PStep &t = nodes[i].s;
    double h = 0;
    for (int r : readers[i]) h = std::max(h, nodes[r].height);
    const double work = std::ldexp((double)t.items * t.m, t.k);
    nodes[i].height = h + 2.0 + work / (256.0 * 304.0) * 0.2;
  }
  // chains: a one-unit step joins the one-unit step it alone waits for
  std::vector<int> next(nn, -1), first(nn, 1);
  for (int i = 0; i < nn; ++i) {
    if (nodes[i].s.n_units != 1 || nodes[i].deps.size() != 1) continue;
    const int q = nodes[i].deps[0];
    if (nodes[q].s.n_units == 1 && next[q] < 0) {
      next[q] = i;
      first[i] = 0;
    }
  }
  std::vector<int> order;
  for (int i = 0; i < nn; ++i)
    if (first[i]) order.push_back(i);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    if (nodes[a].phase != nodes[b].phase) return nodes[a].phase < nodes[b].phase;
    return nodes[a].height > nodes[b].height;
  });
  std::vector<int> at(nn, -1);  // node -> index in P.steps
  size_t o = 0;
  for (int ph = 0; ph <= (int)big_of.size(); ++ph) {
    const int task0 = (int)P.tasks.size();
    for (; o < order.size() && nodes[order[o]].phase == ph; ++o) {
      const int i0 = order[o];
      PTask t{(int)P.steps.size(), 0, 0, 0};
      for (int i = i0; i >= 0; i = next[i]) {
        at[i] = (int)P.steps.size();
        PStep s = nodes[i].s;
        // within a chain the previous step is this CTA's own
        if (i == i0)
          for (int q : nodes[i].deps) {
            s.dep[s.n_deps] = at[q];
            s.dep_units[s.n_deps++] = nodes[q].s.n_units;
          }
        for (int r : readers[i]) s.signal |= r != next[i];
        P.steps.push_back(s);
        ++t.count;
      }
      const int units = P.steps[t.step].n_units;
      for (int u = 0; u < units; ++u) {
        t.unit = u;
        P.tasks.push_back(t);
      }
    }
    if ((int)P.tasks.size() > task0) {
      P.ops.push_back({-1, task0, (int)P.tasks.size() - task0});
      P.n_segments += 1;
    }
    if (ph < (int)big_of.size()) P.ops.push_back({big_of[ph], 0, 0});
  }
}

int64_t place_program(Program &P, int64_t off) {
  auto take = [&](int64_t bytes) {
    const int64_t o = off;
    off += (bytes + 255) & ~int64_t(255);
    return o;
  };
  P.off_sync = take(P.sync_words() * 4);
  P.off_steps = take((int64_t)P.steps.size() * (int64_t)sizeof(PStep));
  P.off_tasks = take((int64_t)P.tasks.size() * (int64_t)sizeof(PTask));
  P.off_tmp = take(P.tmp_bytes);
  const int64_t tmp_meta = P.off_sync + P.meta_word() * 4;
  for (PStep &s : P.steps) {
    if (s.out_off < 0) {
      s.out_off = P.off_tmp + (-1 - s.out_off);
      s.out_meta = tmp_meta + 8 * (-1 - s.out_meta);
    }
    for (int i = 0; i < s.m; ++i)
      if (s.in[i].off < 0) {
        s.in[i].off = P.off_tmp + (-1 - s.in[i].off);
        s.in[i].meta = tmp_meta + 8 * (-1 - s.in[i].meta);
      }
  }
  return off;
}

}  // namespace qgm
