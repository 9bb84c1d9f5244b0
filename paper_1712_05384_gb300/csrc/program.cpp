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
  uint32_t term[MAXRUN];
  for (int q = 0; q < in.nruns; ++q) {
    const int s = in.src[q], l = in.len[q], d = in.dst[q];
    const int nr = std::max(0, std::min(l, w - s));
    if (nr > 0) p.run[p.nrow++] = (uint32_t)(s | nr << 8 | d << 16);
    if (nr < l) term[p.nterm++] = (uint32_t)((s + nr - w) | (l - nr) << 8 | (d + nr) << 16);
  }
  std::copy(term, term + p.nterm, p.run + p.nrow);
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

void program_phases(Program &P, int Bp, int run) {
  const int n = (int)P.all.size();
  P.big.assign(n, 0);
  P.phase.assign(n, 0);
  P.big_at.clear();
  int in_run = 0;  // small steps in the present segment (run > 0)
  for (int s = 0; s < n; ++s) {
    P.big[s] = program_alone(P.all[s], Bp);
    if (P.big[s] || (run > 0 && in_run == run)) {
      // the present phase ends, with this step or without a large one
      P.big_at.push_back(P.big[s] ? s : -1);
      in_run = 0;
      if (P.big[s]) {
        P.phase[s] = (int)P.big_at.size() - 1;
        continue;
      }
    }
    ++in_run;
    if (run > 0) P.phase[s] = (int)P.big_at.size();
    else
      for (int q : P.prod[s])
        if (q >= 0) P.phase[s] = std::max(P.phase[s], P.big[q] ? P.phase[q] + 1 : P.phase[q]);
  }
  P.big_at.push_back(-1);
}

void build_program(Program &P, int Bp, int64_t off_meta, bool split) {
  const int n = (int)P.all.size();
  P.steps.clear();
  P.steps.reserve(n + n / 4 + 8);
  P.tasks.clear();
  P.ops.clear();
  P.n_segments = 0;
  P.n_tmp = 0;
  P.tmp_bytes = 0;
  const std::vector<char> &big = P.big;
  const std::vector<int> &phase = P.phase;
  std::vector<int64_t> tmp(P.big_at.size(), 0);  // bytes of temporaries, which a later segment reuses
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
  nodes.reserve(n + n / 4 + 8);
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
    while (split && t.k - hi - t.lg > 5 && ((int64_t)t.items << (t.lg + hi)) < kLanes) ++hi;
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
    t.out_off = -1 - tmp[nd.phase];  // placed by place_program
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
    tmp[nd.phase] += ((rows << hi) * (d.batched_out ? Bp : 1) * 8 + 255) & ~int64_t(255);
    P.tmp_bytes = std::max(P.tmp_bytes, tmp[nd.phase]);
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
  for (int ph = 0; ph < (int)P.big_at.size(); ++ph) {
    const int task0 = (int)P.tasks.size();
    double loads = 0;
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
        loads += std::ldexp((double)s.items * s.m, s.k);
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
      // a wait lasts at most as long as the segment: a second, and a
      // nanosecond for each of its loads (some hundred times their time), up
      // to a minute
      P.ops.push_back({-1, task0, (int)P.tasks.size() - task0, 1000000000 + (int64_t)std::min(loads, 6e10)});
      P.n_segments += 1;
    }
    if (P.big_at[ph] >= 0) P.ops.push_back({P.big_at[ph], 0, 0, 0});
  }
}

namespace {

// Runs of an index that is linear in the bits of x: bit b of x has value
// 2^pos[b] (pos < 0: absent).
int runs_of(const std::vector<int> &pos, uint32_t *run) {
  int n = 0;
  for (size_t b = 0; b < pos.size();) {
    if (pos[b] < 0) {
      ++b;
      continue;
    }
    size_t l = 1;
    while (b + l < pos.size() && pos[b + l] == pos[b] + (int)l) ++l;
    if (n == PMAXRUN) return -1;
    run[n++] = (uint32_t)(b | l << 8 | (size_t)pos[b] << 16);
    b += l;
  }
  return n;
}

}  // namespace

bool reg_step(const StepDesc &d, int Bp, RegStep &r) {
  const int w = d.w_out, k = d.k;
  if (!d.batched_out || d.m != 2 || k > 8 || w < 3) return false;
  // position of each union bit in each input
  std::vector<std::vector<int>> pos(2, std::vector<int>(w + k, -1));
  for (int i = 0; i < 2; ++i)
    for (int q = 0; q < d.in[i].nruns; ++q)
      for (int l = 0; l < d.in[i].len[q]; ++l) pos[i][d.in[i].src[q] + l] = d.in[i].dst[q] + l;
  int pa = 0, pb = 0;
  for (int u = 0; u < w; ++u) {
    pa += pos[0][u] >= 0 && pos[1][u] < 0;
    pb += pos[1][u] >= 0 && pos[0][u] < 0;
  }
  const int A = pa >= pb ? 0 : 1, B = 1 - A;
  int tm = std::min(std::max(pa, pb), REG_TM), tn = std::min(std::min(pa, pb), REG_TN);
  // enough threads: smaller tiles while the step would leave SMs idle
  while (tm + tn > 2 && (w - tm - tn < 1 || std::ldexp((double)Bp, w - tm - tn) < 65536.0)) {
    if (tm > tn && tm > 2) --tm;
    else if (tn > 0) --tn;
    else break;
  }
  if (tm == 2 && tn == 1) tn = 0;  // forms compiled: 3+2, 3+1, 3+0, 2+2, 2+0
  if (tm < 2 || w - tm - tn < 1) return false;
  // an output with no bit A lacks, and a gate table for B: nothing to reuse;
  // only short sums gain (several rows' loads in flight; 2^25 outputs, one
  // term 0.51 -> 0.44 ms; 2^9 outputs x 1000 entries, 64 terms 0.068 -> 0.096)
  if (tn == 0 && !d.in[B].batched && k > 2) return false;
  r = RegStep{};
  r.k = k;
  r.tm = tm;
  r.tn = tn;
  r.out_off = d.out_off;
  r.out_meta = d.out_meta;
  // batch entries per block: lanes of a warp along the batch, as many as
  // waste few on the last block
  r.lb = 5;
  while (r.lb > 2 && (((Bp + (1 << r.lb) - 1) >> r.lb) << r.lb) * 8 > Bp * 9) --r.lb;
  r.nblk = (Bp + (1 << r.lb) - 1) >> r.lb;
  // tile bits: the highest private bits (the low ones stay neighbours in a row)
  std::vector<int> tile, row;
  std::vector<char> is_tile(w, 0);
  auto pick = [&](int x, int y, int n) {
    for (int u = w - 1; u >= 0 && n > 0; --u)
      if (!is_tile[u] && pos[x][u] >= 0 && pos[y][u] < 0) {
        is_tile[u] = 1;
        tile.push_back(u);
        --n;
      }
  };
  pick(A, B, tm);
  pick(B, A, tn);
  // row bits: with whole warps along the batch, one bit of either kind below
  // the batch block, so that the warps of a CTA share their operands in L1
  if (r.lb == 5)
    for (int side = 0; side < 2; ++side)
      for (int u = 0; u < w; ++u)
        if (!is_tile[u] && std::find(row.begin(), row.end(), u) == row.end() && pos[side ? B : A][u] >= 0 &&
            pos[side ? A : B][u] < 0) {
          row.push_back(u);
          break;
        }
  r.rl = r.lb == 5 ? (int)row.size() : std::min(w - tm - tn, 7 - r.lb);
  for (int u = 0; u < w; ++u)
    if (!is_tile[u] && std::find(row.begin(), row.end(), u) == row.end()) row.push_back(u);
  r.wr = (int)row.size();
  std::vector<int> term;
  for (int u = w; u < w + k; ++u) term.push_back(u);
  auto at = [&](const std::vector<int> &p, const std::vector<int> &bits) {
    std::vector<int> v;
    for (int u : bits) v.push_back(p[u]);
    return v;
  };
  for (int q = 0; q < 2; ++q) {
    const int i = q ? B : A;
    RegIn &x = r.in[q];
    x.off = d.in[i].off;
    x.meta = d.in[i].meta;
    x.batched = d.in[i].batched;
    x.nrow = runs_of(at(pos[i], row), x.run);
    if (x.nrow < 0) return false;
    uint32_t tr[PMAXRUN];
    x.nterm = runs_of(at(pos[i], term), tr);
    if (x.nterm < 0 || x.nrow + x.nterm > PMAXRUN) return false;
    std::copy(tr, tr + x.nterm, x.run + x.nrow);
    for (size_t b = 0; b < tile.size(); ++b) {
      const int ps = pos[i][tile[b]];
      x.tile[(int)b < tm ? b : REG_TM + b - tm] = ps < 0 ? 0 : (int64_t)1 << ps;
    }
  }
  r.norun = runs_of(row, r.orun);
  if (r.norun < 0) return false;
  for (size_t b = 0; b < tile.size(); ++b) r.otile[(int)b < tm ? b : REG_TM + b - tm] = (int64_t)1 << tile[b];
  return true;
}

bool mm_step(const StepDesc &d, int Bp, MmStep &r) {
  const int w = d.w_out, k = d.k, m = d.m;
  if (!d.batched_out || m < 2 || m > 2 + MM_MAXX || k < 2 || k > 16) return false;
  std::vector<std::vector<int>> pos(m, std::vector<int>(w + k, -1));
  for (int i = 0; i < m; ++i)
    for (int q = 0; q < d.in[i].nruns; ++q)
      for (int l = 0; l < d.in[i].len[q]; ++l) pos[i][d.in[i].src[q] + l] = d.in[i].dst[q] + l;
  // batch entries per CTA: 8 unless that wastes lanes (64-byte copies, and
  // the fewer the entries the larger the tile, so the fewer re-reads)
  const int lb = Bp % 8 == 0 || Bp > 32 ? 3 : 2;
  // the pair: least work per output; its tile: as many tile rows and columns
  // as the pair's private bits and 256 threads allow
  double best = 1e300;
  int A = -1, B = -1, mgb = 0, ngb = 0, k2 = 0;
  for (int a = 0; a < m; ++a)
    for (int b = 0; b < m; ++b) {
      if (a == b) continue;
      int pa = 0, pb = 0, in2 = 0;
      for (int u = 0; u < w; ++u) {
        pa += pos[a][u] >= 0 && pos[b][u] < 0;
        pb += pos[b][u] >= 0 && pos[a][u] < 0;
      }
      for (int u = w; u < w + k; ++u) {
        bool out = false;
        for (int i = 0; i < m; ++i) out = out || (i != a && i != b && pos[i][u] >= 0);
        in2 += !out;
      }
      if (pa < MM_TM || pb < MM_TN || in2 < 2 || in2 > 8 || k - in2 > 8) continue;
      // forms compiled: thread groups 3+3, 2+3, 2+2, 1+2, 1+1
      static const int form[5][2] = {{3, 3}, {2, 3}, {2, 2}, {1, 2}, {1, 1}};
      int f = 0;
      while (f < 5 && (form[f][0] + MM_TM > pa || form[f][1] + MM_TN > pb || form[f][0] + form[f][1] + lb > 8)) ++f;
      if (f == 5) continue;
      const double cost = std::ldexp(1.0, k - in2) * (std::ldexp(1.0, in2) + 3.0 * (m - 2)) * (1.0 + 0.05 * f);
      if (cost < best) {
        best = cost;
        A = a;
        B = b;
        mgb = form[f][0];
        ngb = form[f][1];
        k2 = in2;
      }
    }
  if (A < 0) return false;
  r = MmStep{};
  r.nx = m - 2;
  r.k1 = k - k2;
  r.k2 = k2;
  r.mgb = mgb;
  r.ngb = ngb;
  r.lb = lb;
  r.nblk = (Bp + (1 << lb) - 1) >> lb;
  r.out_off = d.out_off;
  r.out_meta = d.out_meta;
  std::vector<int> tile, row;
  std::vector<char> used(w, 0);
  auto priv = [&](int x, int y, int u) { return !used[u] && pos[x][u] >= 0 && pos[y][u] < 0; };
  auto pick = [&](int x, int y, int n) {
    for (int u = 0; u < w && n > 0; ++u)
      if (priv(x, y, u)) {
        used[u] = 1;
        tile.push_back(u);
        --n;
      }
  };
  pick(A, B, MM_TM + mgb);
  pick(B, A, MM_TN + ngb);
  // rows: the rb lowest share a CTA; then the pair's other private bits (CTAs
  // that run together re-read the pair's operands from L2), then the rest
  const int wr = w - (int)tile.size();
  r.wr = wr;
  r.rb = std::min(wr, 8 - lb - mgb - ngb);
  if (r.rb != 8 - lb - mgb - ngb) return false;  // a CTA's threads are all in use
  for (int u = 0; u < w && (int)row.size() < r.rb; ++u)
    if (!used[u]) {
      used[u] = 1;
      row.push_back(u);
    }
  for (int pass = 0; pass < 2; ++pass)
    for (int u = 0; u < w; ++u)
      if (!used[u] && (pass || priv(A, B, u) || priv(B, A, u))) {
        used[u] = 1;
        row.push_back(u);
        r.wp += pass == 0;
      }
  std::vector<int> term;
  for (int pass = 0; pass < 2; ++pass)
    for (int u = w; u < w + k; ++u) {
      bool out = false;
      for (int i = 0; i < m; ++i) out = out || (i != A && i != B && pos[i][u] >= 0);
      if (out == (pass == 1)) term.push_back(u);
    }
  auto at = [&](const std::vector<int> &p, const std::vector<int> &bits) {
    std::vector<int> v;
    for (int u : bits) v.push_back(p[u]);
    return v;
  };
  std::vector<int> order = {A, B};
  for (int i = 0; i < m; ++i)
    if (i != A && i != B) order.push_back(i);
  const int mb = MM_TM + mgb;
  for (int q = 0; q < m; ++q) {
    const InDesc &in = d.in[order[q]];
    MmIn &x = r.in[q];
    x.off = in.off;
    x.meta = in.meta;
    x.batched = in.batched;
    x.nrow = runs_of(at(pos[order[q]], row), x.run);
    if (x.nrow < 0) return false;
    uint32_t tr[PMAXRUN];
    x.nterm = runs_of(at(pos[order[q]], term), tr);
    if (x.nterm < 0 || x.nrow + x.nterm > PMAXRUN) return false;
    std::copy(tr, tr + x.nterm, x.run + x.nrow);
    for (int b = 0; b < (int)tile.size(); ++b) {
      const int ps = pos[order[q]][tile[b]];
      x.tile[b < mb ? b : MM_MBITS + b - mb] = ps < 0 ? 0 : (int64_t)1 << ps;
    }
  }
  r.norun = runs_of(row, r.orun);
  if (r.norun < 0) return false;
  for (int b = 0; b < (int)tile.size(); ++b) r.otile[b < mb ? b : MM_MBITS + b - mb] = (int64_t)1 << tile[b];
  return true;
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
