// Plan-specialised resident kernel (compiled at bind time with NVRTC).
//
// The resident executor runs the whole elimination of one chunk of
// bitstrings inside one CTA (Sec. IV, App. A: every bucket's product-sum
// with all tensors in shared memory).  Its generic form reads a descriptor
// per step (index-map tables, warp schedule) and walks it at run time; for
// the small steps that dominate low-depth circuits that bookkeeping costs
// more than the arithmetic.  This file writes the same computation as CUDA
// source with every plan constant in place (shared-memory offsets, index
// maps, loop bounds, the warp schedule of each dependency level), so that
// each step is only its loads, complex products and stores, and compiles it
// for the device with NVRTC (loaded with dlopen; when it is missing, or the
// compile fails, the generic resident kernel runs instead).
//
// Arithmetic follows the generic kernel: per-tensor power-of-two exponents
// (the producer records max |re|,|im|; the consumer scales by 2^-e), one
// combined scale per output entry while raw products stay clear of both ends
// of FP32's range, the inputs rescaled in place otherwise.  Three additions.
// Most steps take a static bound as their recorded maximum (static_bounds): their consumers' scales are constants and nothing is
// measured.  In wide steps a thread forms two or four entries that share
// loads and addresses (emit_tile).  Shared memory starts from the chunks of a
// plan image that hold something, built at bind.
//
// What bounds it: one CTA alone, the chain of dependency levels (5x5 depth 20:
// 17 levels, 27.9 us before these additions, 20.5 now, caches cold; 4x4 depth
// 12: 7.1 and 5.7 us); a full SM (7 CTAs, shared memory), instruction issue:
// 1024 bitstrings of 5x5 depth 20 26.9 -> 21.5 M warp instructions, 36.5 ->
// 28.7 us (20 -> 26 TFLOP/s).
#include <cuda_runtime.h>
#include <dlfcn.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include "host.h"

namespace qgm {

namespace {

// Value of union bit b in input i of step d, in float2 elements (0 when the
// input does not hold that variable).
std::vector<int64_t> union_values(const InDesc &in, int U, int64_t unit) {
  std::vector<int64_t> v(U, 0);
  for (int q = 0; q < in.nruns; ++q)
    for (int l = 0; l < in.len[q]; ++l) v[in.src[q] + l] = ((int64_t)1 << (in.dst[q] + l)) * unit;
  return v;
}

// C expression for sum_b bit_b(x) * val[lo + b], b < n, with val[] powers of
// two or 0: runs of consecutive bits whose values double become one
// shift-and-mask term.
std::string bit_map_expr(const std::string &x, const std::vector<int64_t> &val, int lo, int n) {
  std::string e;
  int b = 0;
  while (b < n) {
    if (val[lo + b] == 0) {
      ++b;
      continue;
    }
    int l = 1;
    while (b + l < n && val[lo + b + l] == val[lo + b] * ((int64_t)1 << l)) ++l;
    const int s = __builtin_ctzll((unsigned long long)val[lo + b]);
    std::ostringstream t;
    t << "(((" << x << " >> " << b << ") & " << ((1 << l) - 1) << ") << " << s << ")";
    e += (e.empty() ? "" : " + ") + t.str();
    b += l;
  }
  return e.empty() ? "0" : e;
}

int64_t bit_map_value(int64_t x, const std::vector<int64_t> &val, int lo, int n) {
  int64_t r = 0;
  for (int b = 0; b < n; ++b)
    if ((x >> b) & 1) r += val[lo + b];
  return r;
}

const char *kPrelude = R"(
typedef unsigned long long u64;
struct Header { int status; int slice_id; int pad[62]; };
struct Meta { unsigned maxbits; int exp; };
struct RJob { int src; int dst; unsigned char n_out, q0, q1, batched; };
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a += x * y (complex), as four fused multiply-adds
__device__ __forceinline__ void cmac(float2 &a, float2 x, float2 y) {
  a.x = fmaf(x.x, y.x, a.x);
  a.x = fmaf(-x.y, y.y, a.x);
  a.y = fmaf(x.x, y.y, a.y);
  a.y = fmaf(x.y, y.x, a.y);
}
__device__ __forceinline__ void opscale(const Meta *meta, int slot, float &s, int &lo, int &hi, int &esum) {
  const unsigned bits = meta[slot].maxbits;
  const int E = (int)((bits >> 23) & 0xff);
  s = 1.f;
  int e = 0;
  // Inf or NaN (E = 0xff) stays unscaled: it reaches the final tensor,
  // whose check sets the status
  if (E != 0 && E != 0xff) {
    e = E - 126;
    if (e > 126) e = 126;
    s = __int_as_float((127 - e) << 23);
  }
  lo += min(e, 0);
  hi += max(e, 0);
  esum += e + meta[slot].exp;
}
)";

constexpr int kUnroll = 16;  // terms per unrolled block

// "acc += f0 * f1 * ... " for the given operand expressions: products in a
// chain, the last factor fused into the accumulation
void emit_term(std::ostringstream &o, const std::vector<std::string> &f, const std::string &acc,
               const std::string &ind) {
  if (f.size() == 1) {
    o << ind << "{ const float2 p = " << f[0] << "; " << acc << ".x += p.x; " << acc << ".y += p.y; }\n";
    return;
  }
  o << ind << "{ float2 p = " << f[0] << ";\n";
  for (size_t i = 1; i + 1 < f.size(); ++i) o << ind << "  p = cmul(p, " << f[i] << ");\n";
  o << ind << "  cmac(" << acc << ", p, " << f.back() << "); }\n";
}

// Wide steps (every thread forms T = 2 or 4 entries): the T entries of a
// thread differ in item bits J chosen so that the fewest values are loaded
// (an input is loaded once for all entries that agree in the bits it holds),
// with constant offsets between them: one address per input, and loads, not
// index arithmetic, for the other entries.
void emit_tile(std::ostringstream &o, const ResidentLayout &L, const RStep &r, const StepRec &st,
               const std::vector<std::vector<int64_t>> &v, int w, int k, int lb, int nw, int64_t n_iter, int64_t shift,
               bool track_max) {
  const int m = (int)v.size(), W = w + lb;
  const int jt = n_iter >= 4 ? 2 : 1, T = 1 << jt;
  auto log2i = [](int64_t x) { return 63 - __builtin_clzll((unsigned long long)x); };
  const int lt = log2i(32 * nw), lo = log2i(n_iter) - jt;  // thread bits, loop bits
  // value of item bit p in input i (bits below lb: the batch entry)
  auto val = [&](int i, int p) -> int64_t { return p < lb ? (r.in[i].batched ? (int64_t)1 << p : 0) : v[i][p - lb]; };
  // nested evaluation, as in emit_body
  const int k2 = st.k_inner, k1 = k - k2;
  const bool nested = k2 > 0 && k2 <= 4 && (int)st.inner.size() == m;
  // the bits J: item bits of whole warps (from 5 on, the batch entry below)
  std::vector<int> J;
  double best = 1e300;
  for (int a = std::max(5, lb); a < W; ++a)
    for (int b = jt == 2 ? a + 1 : a; b < (jt == 2 ? W : a + 1); ++b) {
      double c = 0;
      for (int i = 0; i < m; ++i) {
        int h = val(i, a) != 0;
        if (jt == 2) h += val(i, b) != 0;
        c += std::ldexp(nested && !st.inner[i] ? std::ldexp(1.0, -k2) : 1.0, h);
      }
      if (c < best) {
        best = c;
        J = jt == 2 ? std::vector<int>{a, b} : std::vector<int>{a};
      }
    }
  std::vector<int> tb, ob;
  for (int p = 0; p < W; ++p)
    if (std::find(J.begin(), J.end(), p) == J.end()) ((int)tb.size() < lt ? tb : ob).push_back(p);
  auto expr = [&](const char *x, const std::vector<int> &bits, int i) {  // i < 0: the output
    std::vector<int64_t> a;
    for (int p : bits) a.push_back(i < 0 ? (int64_t)1 << p : val(i, p));
    return bit_map_expr(x, a, 0, (int)a.size());
  };
  auto jval = [&](int i, int c) {
    int64_t x = 0;
    for (int q = 0; q < jt; ++q)
      if ((c >> q) & 1) x += i < 0 ? (int64_t)1 << J[q] : val(i, J[q]);
    return x;
  };
  if (track_max) o << "    unsigned lmax = 0u;\n";
  if (lo) o << "#pragma unroll 1\n    for (int j = 0; j < " << (1 << lo) << "; ++j) {\n";
  else o << "    {\n";
  for (int i = 0; i < m; ++i) {
    o << "      const int b" << i << " = " << ((r.in[i].soff - shift) / 8) << " + " << expr("gt", tb, i);
    if (lo) o << " + " << expr("j", ob, i);
    o << ";\n";
  }
  o << "      const int bo = " << ((r.out_soff - shift) / 8) << " + " << expr("gt", tb, -1);
  if (lo) o << " + " << expr("j", ob, -1);
  o << ";\n";
  for (int c = 0; c < T; ++c) o << "      float2 a" << c << " = make_float2(0.f, 0.f);\n";
  // inputs that hold fewer of J first: their products are shared
  std::vector<int> in_order(m);
  for (int i = 0; i < m; ++i) in_order[i] = i;
  std::stable_sort(in_order.begin(), in_order.end(), [&](int a, int b) {
    int ha = 0, hb = 0;
    for (int p : J) {
      ha += val(a, p) != 0;
      hb += val(b, p) != 0;
    }
    return ha < hb;
  });
  // one term: the values each entry needs (an entry's value named after the
  // first entry with the same one), then the T products
  auto term = [&](int64_t e, bool inner_only, bool outer_only, const std::string &acc, const std::string &lead,
                  const std::string &base, const std::string &ind) {
    o << ind << "{\n";
    std::vector<std::vector<std::string>> f(T);
    if (!lead.empty())
      for (int c = 0; c < T; ++c) f[c].push_back(lead + std::to_string(c));
    for (int i : in_order) {
      if ((inner_only && !st.inner[i]) || (outer_only && st.inner[i])) continue;
      std::map<int64_t, int> seen;
      for (int c = 0; c < T; ++c) {
        const int64_t x = jval(i, c);
        auto it = seen.find(x);
        if (it == seen.end()) {
          it = seen.emplace(x, c).first;
          o << ind << "  const float2 x" << i << "_" << c << " = F[" << base << i << " + "
            << (bit_map_value(e, v[i], w, k) + x) << "];\n";
        }
        f[c].push_back("x" + std::to_string(i) + "_" + std::to_string(it->second));
      }
    }
    for (int c = 0; c < T; ++c) emit_term(o, f[c], acc + std::to_string(c), ind + "  ");
    o << ind << "}\n";
  };
  if (nested) {
    const int u2n = 1 << k2;
    const int u1_log = std::min(k1, std::max(0, 4 - k2 - jt)), blk_log = k1 - u1_log;
    if (blk_log) o << "#pragma unroll 1\n      for (int blk = 0; blk < " << (1 << blk_log) << "; ++blk) {\n";
    else o << "      {\n";
    for (int i = 0; i < m; ++i)
      o << "        const int c" << i << " = b" << i << " + "
        << (blk_log ? bit_map_expr("blk", v[i], w + k2 + u1_log, blk_log) : std::string("0")) << ";\n";
    for (int u1 = 0; u1 < (1 << u1_log); ++u1) {
      o << "        {\n";
      for (int c = 0; c < T; ++c) o << "          float2 i" << c << " = make_float2(0.f, 0.f);\n";
      for (int u2 = 0; u2 < u2n; ++u2) term(((int64_t)u1 << k2) | u2, true, false, "i", "", "c", "          ");
      term((int64_t)u1 << k2, false, true, "a", "i", "c", "          ");
      o << "        }\n";
    }
    o << "      }\n";
  } else {
    const int unr_log = std::min(k, std::max(0, 4 - jt)), blk_log = k - unr_log;
    if (blk_log) o << "#pragma unroll 1\n      for (int blk = 0; blk < " << (1 << blk_log) << "; ++blk) {\n";
    else o << "      {\n";
    for (int i = 0; i < m; ++i)
      o << "        const int c" << i << " = b" << i << " + "
        << (blk_log ? bit_map_expr("blk", v[i], w + unr_log, blk_log) : std::string("0")) << ";\n";
    for (int u = 0; u < (1 << unr_log); ++u) term(u, false, false, "a", "", "c", "        ");
    o << "      }\n";
  }
  for (int c = 0; c < T; ++c) {
    o << "      a" << c << " = make_float2(a" << c << ".x * comb, a" << c << ".y * comb); F[bo + " << jval(-1, c) << "] = a" << c
      << ";\n";
    if (track_max)
      o << "      lmax = max(lmax, max(__float_as_uint(a" << c << ".x) & 0x7fffffffu, __float_as_uint(a" << c
        << ".y) & 0x7fffffffu));\n";
  }
  o << "    }\n";
}

// One step's body for the threads of its warps (gt = thread index in the
// group): every item's product-sum with raw operand values, times `comb`
// (2^-es, the inputs' combined scale) per entry.  Shared-memory offsets are
// the layout's minus `shift` (the generic kernel's work lists are not kept).
void emit_body(std::ostringstream &o, const qgm_plan *p, const ResidentLayout &L, size_t q, int64_t shift,
               bool track_max) {
  const RStep &r = L.steps[q];
  const StepDesc &d = p->steps[L.src_step[q]];
  const int logBc = __builtin_ctz(L.chunk);
  const int m = d.m, k = d.k, w = d.w_out, U = w + k;
  const int nw = (r.sched >> 4) & 15, lg = (r.sched >> 8) & 15;
  const int lb = r.batched_out ? logBc : 0;
  const int64_t items = ((int64_t)1 << w) << lb;
  const int G = 32 * nw, tpi = 1 << lg, sit = G >> lg;
  const int64_t n_iter = (items * tpi + G - 1) / G;
  const bool always_live = (items * tpi) % G == 0 && items * tpi >= G;
  const int tpt_log = k - lg;  // terms per thread per item: 2^tpt_log
  const int unr_log = std::min(tpt_log, __builtin_ctz(kUnroll));
  const int blk_log = tpt_log - unr_log;
  std::vector<std::vector<int64_t>> v(m);
  for (int i = 0; i < m; ++i) v[i] = union_values(d.in[i], U, r.in[i].batched ? L.chunk : 1);
  const std::string live = always_live ? "true" : "it < " + std::to_string(items);
  // nested evaluation: the lanes of an entry split the outer terms, each
  // lane runs all 2^k2 inner terms per outer term
  const StepRec &st = p->sim.steps[L.src_step[q]];
  const int k2 = st.k_inner, k1 = k - k2;
  const bool nested = k2 > 0 && k2 <= 4 && lg <= k1 && (int)st.inner.size() == m;
  const int glo = nested ? w + k2 : w;  // union bit of the lane index's bit 0
  if (lg == 0 && n_iter >= 2 && always_live && (n_iter & (n_iter - 1)) == 0 && w + lb >= 7) {
    emit_tile(o, L, r, st, v, w, k, lb, nw, n_iter, shift, track_max);
    return;
  }
  if (track_max) o << "    unsigned lmax = 0u;\n";
  if (lg) {
    o << "    const int g = gt & " << (tpi - 1) << ";\n";
    for (int i = 0; i < m; ++i) o << "    const int go" << i << " = " << bit_map_expr("g", v[i], glo, lg) << ";\n";
  }
  o << "#pragma unroll 1\n    for (int j = 0; j < " << n_iter << "; ++j) {\n";
  o << "      const int it = (gt >> " << lg << ") + j * " << sit << ";\n";
  o << "      float2 acc = make_float2(0.f, 0.f);\n";
  o << "      if (" << live << ") {\n";
  if (w) o << "        const int row = it >> " << lb << ";\n";
  if (lb) o << "        const int beta = it & " << ((1 << lb) - 1) << ";\n";
  for (int i = 0; i < m; ++i) {
    o << "        const int b" << i << " = " << ((r.in[i].soff - shift) / 8);
    if (r.in[i].batched && lb) o << " + beta";
    o << " + " << bit_map_expr("row", v[i], 0, w);
    if (lg) o << " + go" << i;
    o << ";\n";
  }
  if (nested) {
    // term index e = (e1 << k2) | e2 with e1 = (blk << (u1_log + lg)) | (u1 << lg) | g
    const int u2n = 1 << k2;
    const int u1_log = std::min(k1 - lg, std::max(0, 4 - k2));
    const int blk_log1 = k1 - lg - u1_log;
    o << "        float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);\n";
    o << "#pragma unroll 1\n        for (int blk = 0; blk < " << (1 << blk_log1) << "; ++blk) {\n";
    for (int i = 0; i < m; ++i) {
      const std::string e = blk_log1 ? bit_map_expr("blk", v[i], w + k2 + lg + u1_log, blk_log1) : std::string("0");
      o << "          const int c" << i << " = b" << i << " + " << e << ";\n";
    }
    for (int u1 = 0; u1 < (1 << u1_log); ++u1) {
      o << "          { float2 i0 = make_float2(0.f, 0.f), i1 = make_float2(0.f, 0.f);\n";
      for (int u2 = 0; u2 < u2n; ++u2) {
        const int64_t e = ((int64_t)u1 << (lg + k2)) | u2;
        std::vector<std::string> f;
        for (int i = 0; i < m; ++i)
          if (st.inner[i]) f.push_back("F[c" + std::to_string(i) + " + " + std::to_string(bit_map_value(e, v[i], w, k)) + "]");
        emit_term(o, f, "i" + std::to_string(u2 & 1), "            ");
      }
      const int64_t e = (int64_t)u1 << (lg + k2);
      std::vector<std::string> f = {"make_float2(i0.x + i1.x, i0.y + i1.y)"};
      for (int i = 0; i < m; ++i)
        if (!st.inner[i]) f.push_back("F[c" + std::to_string(i) + " + " + std::to_string(bit_map_value(e, v[i], w, k)) + "]");
      emit_term(o, f, "a" + std::to_string(u1 & 1), "            ");
      o << "          }\n";
    }
    o << "        }\n";
  } else {
  // unrolled blocks of 2^unr_log terms: the block's offsets at run time,
  // the term offsets inside a block as constants; term index
  // e = (blk << (unr_log + lg)) | (u << lg) | g
  o << "        float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);\n";
  o << "#pragma unroll 1\n        for (int blk = 0; blk < " << (1 << blk_log) << "; ++blk) {\n";
  for (int i = 0; i < m; ++i) {
    const std::string e = blk_log ? bit_map_expr("blk", v[i], w + lg + unr_log, blk_log) : std::string("0");
    o << "          const int c" << i << " = b" << i << " + " << e << ";\n";
  }
  for (int u = 0; u < (1 << unr_log); ++u) {
    std::vector<std::string> f;
    for (int i = 0; i < m; ++i)
      f.push_back("F[c" + std::to_string(i) + " + " + std::to_string(bit_map_value((int64_t)u << lg, v[i], w, k)) + "]");
    emit_term(o, f, "a" + std::to_string(u & 1), "          ");
  }
  o << "        }\n";
  }
  o << "        acc = make_float2((a0.x + a1.x) * comb, (a0.y + a1.y) * comb);\n";
  o << "      }\n";
  for (int s2 = 1; s2 < tpi; s2 <<= 1)
    o << "      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, " << s2
      << "); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, " << s2 << ");\n";
  o << "      if (" << live << (lg ? " && g == 0" : "") << ") {\n";
  o << "        F[" << ((r.out_soff - shift) / 8) << " + it] = acc;\n";
  if (track_max)
    o << "        lmax = max(lmax, max(__float_as_uint(acc.x) & 0x7fffffffu, __float_as_uint(acc.y) & 0x7fffffffu));\n";
  o << "      }\n";
  o << "    }\n";
}

}  // namespace

std::vector<int> rotations(const qgm_plan *p) {
  std::vector<int> n(p->sim.tensors.size(), 0);
  for (size_t li = 0; li < p->leaves.size(); ++li)
    for (int fi : p->leaves[li].members) n[li] += p->model.gates[p->model.factors[fi].gate].kind == QGM_GATE_RXY;
  for (const StepRec &st : p->sim.steps)
    for (int id : st.inputs) n[st.out] += n[id];
  return n;
}

std::map<int, StaticBound> static_bounds(const qgm_plan *p, const ResidentLayout &L) {
  std::map<int, StaticBound> bound;
  struct Slack {
    int bits;
    int64_t entries;
  };
  std::map<int, Slack> loose;  // by metadata slot
  const std::vector<int> rot = rotations(p);
  for (size_t q = 0; q < L.steps.size(); ++q) {
    const RStep &r = L.steps[q];
    const StepRec &st = p->sim.steps[L.src_step[q]];
    const int64_t entries = ((int64_t)1 << r.w_out) * (r.batched_out ? L.chunk : 1);
    // slack of the leaves and of the inputs with a static bound; inputs scaled
    int leaf = 0, slack = 0, scaled = 0;
    for (int i = 0; i < r.m; ++i) {
      if (r.in[i].meta < 0) leaf += ROTATION_BITS * rot[st.inputs[i]];
      else ++scaled;
      if (bound.count(r.in[i].meta)) slack += loose[r.in[i].meta].bits;
    }
    auto loosest = [&]() {
      int best = -1;
      for (int i = 0; i < r.m; ++i)
        if (bound.count(r.in[i].meta) && (best < 0 || loose[r.in[i].meta].bits > loose[r.in[best].meta].bits)) best = i;
      return best;
    };
    auto measure = [&](int i) {
      slack -= loose[r.in[i].meta].bits;
      bound.erase(r.in[i].meta);
    };
    while (slack > 0 && leaf + slack > SLACK_BITS) measure(loosest());
    if (r.out_meta == L.final_meta) continue;
    const int own = r.k + scaled + leaf;
    if (own + slack > SLACK_BITS) {
      // measure an input in place of the output where that is less work
      const int i = loosest();
      if (i < 0 || slack - loose[r.in[i].meta].bits > SLACK_BITS - own || loose[r.in[i].meta].entries >= entries) continue;
      measure(i);
    }
    StaticBound s;
    s.k = r.k;
    s.exp_known = true;
    bool ok = true;
    for (int i = 0; i < r.m; ++i) {
      if (r.in[i].meta < 0) continue;
      auto it = bound.find(r.in[i].meta);
      if (it == bound.end()) {
        s.exp_known = false;  // measured at run time
        ok = ok && rot[st.inputs[i]] == 0;
        continue;
      }
      s.exp_known = s.exp_known && it->second.exp_known;
      s.exp += it->second.k + 1 + it->second.exp;  // scale exponent k+1, recorded exponent
    }
    if (!ok) continue;
    bound[r.out_meta] = s;
    loose[r.out_meta] = {own + slack, entries};
  }
  return bound;
}

std::vector<uint32_t> image_chunks(const qgm_plan *p, const ResidentLayout &L) {
  std::vector<char> used((size_t)(compiled_smem(L) / 16), 0);
  const int64_t shift = worklist_bytes(L);
  for (int64_t b = 0; b < (int64_t)p->n_meta_fwd * 8; b += 16) used[b / 16] = 1;
  for (const RJob &j : L.jobs)
    if (!j.batched) used[(j.dst - shift) / 16] = 1;
  std::vector<uint32_t> at;
  for (size_t c = 0; c < used.size(); ++c)
    if (used[c]) at.push_back((uint32_t)c);
  return at;
}

// CUDA source of the resident kernel specialised to layout L of plan p.
// mode RES_WHOLE: the whole pass per CTA.  RES_MAIN: the steps with a batch
// axis; the bitstring-independent tensors they read come from the pre
// region, written by the RES_PRE kernel (one CTA running the steps without a
// batch axis), which the main kernel may overlap up to the point where it
// waits for them (programmatic dependent launch).
std::string resident_source(const qgm_plan *p, const ResidentLayout &L, const std::string &name, int minb,
                            int mode) {
  std::ostringstream o;
  o << kPrelude;
  const int logBc = __builtin_ctz(L.chunk);
  const int64_t shift = worklist_bytes(L);
  const bool pre = mode == RES_PRE, main_part = mode == RES_MAIN;
  o << "extern \"C\" __global__ void __launch_bounds__(256, " << minb << ") " << name
    << "(const char *ws, const RJob *jobs, int n_jobs, const u64 *bits, long long B, double c_re, double c_im, "
       "double2 *out, Header *hdr) {\n";
  o << "  extern __shared__ __align__(16) char sm[];\n";
  o << "  float2 *F = reinterpret_cast<float2 *>(sm);\n";
  o << "  Meta *meta = reinterpret_cast<Meta *>(sm);\n";
  o << "  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;\n";
  o << "  const long long b0 = (long long)blockIdx.x * " << L.chunk << ";\n";
  if (pre) o << "  asm volatile(\"griddepcontrol.launch_dependents;\");\n";
  // shared memory starts with the plan's image (image_chunks)
  const size_t n_img = image_chunks(p, L).size();
  o << "  {\n    const uint4 *img = reinterpret_cast<const uint4 *>(ws + " << p->off_image << ");\n";
  o << "    const unsigned *at = reinterpret_cast<const unsigned *>(img + " << n_img << ");\n";
  o << "    uint4 *S = reinterpret_cast<uint4 *>(sm);\n";
  o << "#pragma unroll 2\n    for (int i = tid; i < " << n_img << "; i += 256) S[__ldg(at + i)] = __ldg(img + i);\n  }\n";
  int n_batched = 0;
  for (const RJob &j : L.jobs) n_batched += j.batched != 0;
  if (!pre && n_batched) {
    // leaf rows that depend on the output bits of x_beta (listed first); no
    // tensor shares a 16-byte chunk with another, so they need not wait for
    // the image
    o << "  const float2 *wsf = reinterpret_cast<const float2 *>(ws);\n";
    if (L.chunk == 1) o << "  const u64 x1 = b0 < B ? __ldg(bits + b0) : 0ull;\n";
    o << "  for (int t = tid; t < " << (n_batched << logBc) << "; t += 256) {\n";
    o << "    const int b = t & " << (L.chunk - 1) << ";\n";
    o << "    const RJob jb = jobs[t >> " << logBc << "];\n";
    o << "    int ob = 0;\n";
    o << "    if (jb.n_out) {\n";
    if (L.chunk == 1) o << "      const u64 x = x1;\n";
    else o << "      const u64 x = (b0 + b < B) ? bits[b0 + b] : 0ull;\n";
    o << "      ob = jb.n_out == 1 ? (int)((x >> jb.q0) & 1ull) : (int)((((x >> jb.q0) & 1ull) << 1) | ((x >> jb.q1) & 1ull));\n";
    o << "    }\n";
    o << "    reinterpret_cast<float2 *>(sm + jb.dst - " << shift << ")[b] = __ldg(wsf + jb.src + ob);\n";
    o << "  }\n";
  }
  if (main_part) {
    // the pre kernel's outputs and their scales, once it has finished
    o << "  __syncthreads();\n";
    o << "  asm volatile(\"griddepcontrol.wait;\" ::: \"memory\");\n";
    o << "  {\n    const float2 *pd = reinterpret_cast<const float2 *>(ws + " << p->off_pre << ") + " << p->pre_data
      << ";\n";
    o << "    const int2 *pm = reinterpret_cast<const int2 *>(ws + " << p->off_pre << ");\n";
    for (size_t j = 0; j < L.pre.size(); ++j) {
      const auto &t = L.pre[j];
      o << "    for (int x = tid; x < " << t.entries << "; x += 256) F[" << ((t.soff - shift) / 8) << " + x] = pd["
        << t.goff << " + x];\n";
      o << "    if (tid == " << (j % 256) << ") { const int2 v = pm[" << j << "]; meta[" << t.meta
        << "].maxbits = (unsigned)v.x; meta[" << t.meta << "].exp = v.y; }\n";
    }
    o << "  }\n";
  }
  o << "  __syncthreads();\n";
  // recorded maxima known before the run: steps with a static bound
  const std::map<int, StaticBound> static_k = static_bounds(p, L);
  const std::vector<int> rot = rotations(p);
  // steps in level order; inside a level grouped by first warp, so that
  // each warp's code for the level is contiguous
  std::vector<size_t> emit_order(L.steps.size());
  for (size_t q = 0; q < emit_order.size(); ++q) emit_order[q] = q;
  std::stable_sort(emit_order.begin(), emit_order.end(), [&](size_t a, size_t b) {
    if (L.level[a] != L.level[b]) return L.level[a] < L.level[b];
    return (L.steps[a].sched & 15) < (L.steps[b].sched & 15);
  });
  int cur_level = -1;
  for (size_t q : emit_order) {
    const RStep &r = L.steps[q];
    if ((pre && r.batched_out) || (main_part && !r.batched_out)) continue;
    if (L.level[q] != cur_level) {
      if (cur_level >= 0) o << "  __syncthreads();\n";
      cur_level = L.level[q];
    }
    const StepDesc &d = p->steps[L.src_step[q]];
    const int w0 = r.sched & 15, nw = (r.sched >> 4) & 15;
    o << "  // step " << L.src_step[q] << ": " << d.m << " inputs, " << d.k << " summed, " << d.w_out
      << " kept (level " << L.level[q] << ")\n";
    o << "  if (wid >= " << w0 << " && wid < " << (w0 + nw) << ") {\n";
    o << "    const int gt = tid - " << (32 * w0) << ";\n";
    // inputs whose producer has a static bound 2^k' get the constant scale
    // 2^-(k'+1) (exponent k'+1); the others read theirs
    int es_static = 0, esum_static = 0;
    bool any_dynamic = false;
    std::string esum_late;  // recorded exponents read by the thread that records the output's
    for (int i = 0; i < d.m; ++i)
      if (r.in[i].meta >= 0) {
        auto it = static_k.find(r.in[i].meta);
        if (it == static_k.end()) {
          any_dynamic = true;
          continue;
        }
        es_static += it->second.k + 1;
        esum_static += it->second.k + 1;
        if (it->second.exp_known) esum_static += it->second.exp;
        else esum_late += " + meta[" + std::to_string(r.in[i].meta) + "].exp";
      }
    // exponents of the inputs: the negative ones (how small raw products may
    // be) and the others apart
    o << "    int lo = 0, hi = " << es_static << ", esum = " << esum_static << ";\n";
    for (int i = 0; i < d.m; ++i) {
      if (r.in[i].meta < 0) continue;
      auto it = static_k.find(r.in[i].meta);
      if (it != static_k.end())
        o << "    const float s" << i << " = __int_as_float(" << (126 - it->second.k) << " << 23);\n";
      else
        o << "    float s" << i << "; opscale(meta, " << r.in[i].meta << ", s" << i << ", lo, hi, esum);\n";
    }
    // scales: one combined factor per entry while products of raw values stay
    // clear of both ends of FP32's range (by more where small entries matter,
    // behind rotations); otherwise the intermediate inputs are rescaled in
    // place first (each feeds this step only) and the factor is 1
    bool any_meta = false;
    const int least = rot[p->sim.steps[L.src_step[q]].out] ? -16 : -40;
    for (int i = 0; i < d.m; ++i) any_meta |= r.in[i].meta >= 0;
    o << "    float comb = 1.f;\n";
    if (any_meta && !any_dynamic && es_static <= 60) {
      o << "    comb = __int_as_float(" << (127 - es_static) << " << 23);\n";
    } else if (any_meta) {
      o << "    if (lo >= " << least << " && hi <= 60) comb = __int_as_float((127 - lo - hi) << 23);\n";
      o << "    else {\n";
      for (int i = 0; i < d.m; ++i) {
        if (r.in[i].meta < 0) continue;
        const SymTensor &t = p->sim.tensors[p->sim.steps[L.src_step[q]].inputs[i]];
        const int64_t n = ((int64_t)1 << t.vars.size()) * (t.batched ? L.chunk : 1);
        o << "      for (int x = gt; x < " << n << "; x += " << 32 * nw << ") { float2 &y = F["
          << ((r.in[i].soff - shift) / 8) << " + x]; y.x *= s" << i << "; y.y *= s" << i << "; }\n";
      }
      if (nw > 1) o << "      asm volatile(\"bar.sync %0, %1;\" :: \"r\"(" << (1 + w0) << "), \"r\"(" << 32 * nw << "));\n";
      else o << "      __syncwarp();\n";
      o << "    }\n";
    }
    auto bound = static_k.find(r.out_meta);
    const bool track = bound == static_k.end();
    {
      std::ostringstream b;
      emit_body(b, p, L, q, shift, track);
      if (track) o << "    unsigned lm;\n    {\n" << b.str() << "    lm = lmax; }\n";
      else o << "    {\n" << b.str() << "    }\n";
    }
    if (track) {
      // max |re|,|im| over the step's entries: non-negative floats (and NaN,
      // which must reach the maximum) order like their bit patterns
      o << "    lm = __reduce_max_sync(0xffffffffu, lm);\n";
      o << "    if (lane == 0) {\n";
      o << "      if (lm) atomicMax(&meta[" << r.out_meta << "].maxbits, lm);\n";
      o << "      if (wid == " << w0 << ") meta[" << r.out_meta << "].exp = esum" << esum_late << ";\n";
      o << "    }\n";
    } else if (!bound->second.exp_known) {
      o << "    if (gt == 0) meta[" << r.out_meta << "].exp = esum" << esum_late << ";\n";
    }
    o << "  }\n";
  }
  o << "  __syncthreads();\n";
  if (pre) {
    // publish the outputs read by batched steps, with their scales
    o << "  {\n    float2 *pd = reinterpret_cast<float2 *>(const_cast<char *>(ws) + " << p->off_pre << ") + "
      << p->pre_data << ";\n";
    o << "    int2 *pm = reinterpret_cast<int2 *>(const_cast<char *>(ws) + " << p->off_pre << ");\n";
    for (size_t j = 0; j < L.pre.size(); ++j) {
      const auto &t = L.pre[j];
      o << "    for (int x = tid; x < " << t.entries << "; x += 256) pd[" << t.goff << " + x] = F["
        << ((t.soff - shift) / 8) << " + x];\n";
      o << "    if (tid == " << (j % 256) << ") pm[" << j << "] = make_int2((int)meta[" << t.meta << "].maxbits, meta["
        << t.meta << "].exp);\n";
    }
    o << "  }\n}\n";
    return o.str();
  }
  o << "  if (tid == 0 && ((meta[" << L.final_meta << "].maxbits >> 23) & 0xff) == 0xff) atomicCAS(&hdr->status, 0, -5);\n";
  o << "  if (tid < " << L.chunk << " && b0 + tid < B) {\n";
  o << "    const float2 v = F[" << ((L.final_soff - shift) / 8) << (p->final_batched ? " + tid" : "") << "];\n";
  o << "    const double scl = ldexp(1.0, meta[" << L.final_meta << "].exp);\n";
  o << "    const double re = (double)v.x * scl, im = (double)v.y * scl;\n";
  o << "    out[b0 + tid] = make_double2(re * c_re - im * c_im, re * c_im + im * c_re);\n";
  o << "  }\n}\n";
  return o.str();
}

}  // namespace qgm

// ---------------------------------------------------------------- NVRTC
namespace qgm {

namespace {

struct Nvrtc {
  bool ok = false;
  int (*create)(void **, const char *, const char *, int, const char *const *, const char *const *) = nullptr;
  int (*compile)(void *, int, const char *const *) = nullptr;
  int (*log_size)(void *, size_t *) = nullptr;
  int (*log)(void *, char *) = nullptr;
  int (*cubin_size)(void *, size_t *) = nullptr;
  int (*cubin)(void *, char *) = nullptr;
  int (*destroy)(void **) = nullptr;
};

Nvrtc &nvrtc() {
  static Nvrtc n;
  static std::once_flag once;
  std::call_once(once, [] {
    void *h = nullptr;
    for (const char *name : {"libnvrtc.so.13", "libnvrtc.so", "/usr/local/cuda/lib64/libnvrtc.so.13"})
      if ((h = dlopen(name, RTLD_NOW | RTLD_LOCAL))) break;
    if (!h) return;
    n.create = reinterpret_cast<decltype(n.create)>(dlsym(h, "nvrtcCreateProgram"));
    n.compile = reinterpret_cast<decltype(n.compile)>(dlsym(h, "nvrtcCompileProgram"));
    n.log_size = reinterpret_cast<decltype(n.log_size)>(dlsym(h, "nvrtcGetProgramLogSize"));
    n.log = reinterpret_cast<decltype(n.log)>(dlsym(h, "nvrtcGetProgramLog"));
    n.cubin_size = reinterpret_cast<decltype(n.cubin_size)>(dlsym(h, "nvrtcGetCUBINSize"));
    n.cubin = reinterpret_cast<decltype(n.cubin)>(dlsym(h, "nvrtcGetCUBIN"));
    n.destroy = reinterpret_cast<decltype(n.destroy)>(dlsym(h, "nvrtcDestroyProgram"));
    n.ok = n.create && n.compile && n.log_size && n.log && n.cubin_size && n.cubin && n.destroy;
  });
  return n;
}

struct CacheKey {
  int device;
  size_t hash, len;
  bool operator<(const CacheKey &o) const {
    return device != o.device ? device < o.device : hash != o.hash ? hash < o.hash : len < o.len;
  }
};

std::mutex g_cache_mu;
std::map<CacheKey, cudaKernel_t> g_cache;

}  // namespace

// Compile `src` for the current device (sm_103a) and return kernel `name`.
// Kernels are cached per device and source for the life of the process.
// Returns false (with a message in *err) when NVRTC is unavailable or the
// compile or load fails.
bool jit_kernel(const std::string &src, const std::string &name, int device, cudaKernel_t *out,
                std::string *err) {
  const CacheKey key{device, std::hash<std::string>()(src), src.size()};
  {
    std::lock_guard<std::mutex> lk(g_cache_mu);
    auto it = g_cache.find(key);
    if (it != g_cache.end()) {
      *out = it->second;
      return true;
    }
  }
  Nvrtc &n = nvrtc();
  if (!n.ok) {
    *err = "NVRTC library not found";
    return false;
  }
  void *prog = nullptr;
  if (n.create(&prog, src.c_str(), "qgm_resident.cu", 0, nullptr, nullptr) != 0) {
    *err = "nvrtcCreateProgram failed";
    return false;
  }
  const char *opts[] = {"--gpu-architecture=sm_103a", "-std=c++17", "-default-device"};
  const int rc = n.compile(prog, 3, opts);
  if (rc != 0) {
    size_t ls = 0;
    n.log_size(prog, &ls);
    std::string log(ls, '\0');
    if (ls) n.log(prog, &log[0]);
    *err = "NVRTC compile failed: " + log.substr(0, 2000);
    n.destroy(&prog);
    return false;
  }
  size_t cs = 0;
  n.cubin_size(prog, &cs);
  std::vector<char> cubin(cs);
  n.cubin(prog, cubin.data());
  n.destroy(&prog);
  cudaLibrary_t lib;
  cudaError_t e = cudaLibraryLoadData(&lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0);
  if (e != cudaSuccess) {
    *err = std::string("cudaLibraryLoadData: ") + cudaGetErrorString(e);
    return false;
  }
  cudaKernel_t k;
  e = cudaLibraryGetKernel(&k, lib, name.c_str());
  if (e != cudaSuccess) {
    *err = std::string("cudaLibraryGetKernel: ") + cudaGetErrorString(e);
    return false;
  }
  std::lock_guard<std::mutex> lk(g_cache_mu);
  g_cache[key] = k;
  *out = k;
  return true;
}

}  // namespace qgm
