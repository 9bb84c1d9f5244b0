// Internal host-side structures shared by host.cpp (circuit, model, plan)
// and exec.cu (device execution).  Not part of the C ABI.
#pragma once

#include <algorithm>
#include <complex>
#include <cstdint>
#include <map>
#include <string>
#include <vector>

#include "qgm.h"

struct qgm_plan;

namespace qgm {

using cd = std::complex<double>;

void set_error(const char *fmt, ...);

// ---------------------------------------------------------------- circuit
struct Circuit {
  int n = 0, rows = 0, cols = 0, depth = 0;
  uint64_t seed = 0;
  int param = 0;
  std::vector<qgm_gate> gates;
  std::vector<int> param_gates;
};

// ------------------------------------------------------------------ model
// One factor per gate (Sec. III.B).  Table index = (bit(v[0]) << (nv-1)) | bit(v[1]).
struct MFactor {
  int nv = 0;
  int v[2] = {-1, -1};
  cd t[4];
  int gate = -1;
  int half_pow = 0;  // number of 2^{-1/2} factors pulled out of the table
};

struct Model {
  int n = 0, rows = 0, cols = 0;
  int n_vars = 0;
  std::vector<int> var_qubit, var_k, inputs, outputs;
  std::vector<MFactor> factors;
  int L = 0;                       // non-diagonal gates
  std::vector<int> param_factor;   // factor index of each RXY gate
  std::vector<qgm_gate> gates;     // copy of the circuit's gates
};

// ------------------------------------------------------------------- plan
constexpr int MAXIN = 8;    // tensors multiplied in one step
constexpr int MAXRUN = 16;  // contiguous bit runs of an index map
constexpr int ADJOINT_K = 30;  // most variables an adjoint step sums
constexpr int MAXLEAFV = 4; // variables of a leaf factor (internal+slice+output)
constexpr int RES_WARPS = 8; // warps of a resident CTA

// Index map of one step input: the input's index is the union index with
// the bits of absent variables squeezed out (a "pext" by contiguous runs).
struct InDesc {
  int64_t off;       // byte offset of the tensor in the workspace
  int32_t meta;      // tensor metadata slot (intermediates), -1 for leaves
  int32_t batched;   // 1: rows of batch_padded complex values
  int32_t nruns;
  uint8_t src[MAXRUN], len[MAXRUN], dst[MAXRUN];
};

struct StepDesc {
  int32_t m;            // inputs
  int32_t k;            // variables summed (top k bits of the union index)
  int32_t w_out;        // output rank (binary variables)
  int32_t batched_out;
  int64_t out_off;
  int32_t out_meta;
  int32_t gemm;         // index of the step's GemmDesc, or -1
  // register tile: output bits (union positions < w_out) that the largest
  // input does not hold; a thread loads that input once per term and forms
  // the 2^tile_t outputs that share it
  int32_t tile_t;
  uint8_t tile_pos[4];
  InDesc in[MAXIN];
};

// A GEMM-shaped step: out[s, m, n] = sum_k A[s, m, k] B[s, n, k] with s the
// kept variables both operands hold, m (n) the kept variables only A (B)
// holds and k the summed variables (both hold all of them).  Each operand
// and the output are addressed through the bit positions of those
// variables in their own index (no transposition); the batch axis, when
// present, stays innermost.
constexpr int GMAXB = 24;
struct GemmDesc {
  int64_t a_off, b_off, o_off;
  int32_t a_meta, b_meta, o_meta;
  int32_t a_bat, b_bat, o_bat;
  int32_t nm, nn, nk, ns;
  // batch entry outermost (a tensor written by one tensor-core product per
  // entry and read only by another tensor-core step): entry beta's values
  // are a whole tensor of 2^rank complex64 at beta * 2^rank * 8 bytes
  int32_t a_bout, b_bout, o_bout;
  uint8_t mA[GMAXB], mO[GMAXB], nB[GMAXB], nO[GMAXB];
  uint8_t kA[GMAXB], kB[GMAXB], sA[GMAXB], sB[GMAXB], sO[GMAXB];
};

// Exchange the roles of the two operands: out[s, n, m] = sum_k B A is the
// same product.
inline void gemm_swap_roles(GemmDesc &g) {
  std::swap(g.a_off, g.b_off);
  std::swap(g.a_meta, g.b_meta);
  std::swap(g.a_bat, g.b_bat);
  std::swap(g.a_bout, g.b_bout);
  std::swap(g.nm, g.nn);
  for (int b = 0; b < GMAXB; ++b) {
    std::swap(g.mA[b], g.nB[b]);
    std::swap(g.mO[b], g.nO[b]);
    std::swap(g.kA[b], g.kB[b]);
    std::swap(g.sA[b], g.sB[b]);
  }
}

// Tensor-core form of a GEMM-shaped step.  One operand takes the MMA's M
// side (tiles of 128 rows), the other the N side (tiles of nt = min(256,
// 2^nN) rows); both are first split into planes of 16-bit terms stored as
// the MMA reads them.  When only one operand carries the batch axis it takes
// the M side and its batch entries become rows there (row = m * Bp + beta),
// so the other operand's tile serves every entry; when both carry it, each
// (shared index, batch entry) is a product of its own ("per entry").  A
// plane block holds, for one instance (shared index, and batch entry when
// per entry), one row tile and one chunk of 16 summed entries, P planes of
// TR x 16 terms in 8-row x 16-byte core matrices (row group stride 256 B,
// the two 8-entry halves of a row 128 B apart).
constexpr int TC_M = 128;
struct TcCfg {
  bool ok = false;
  bool swap = false;     // B takes the M side
  bool fold = false;     // batch entries are rows of the M side
  bool perbeta = false;  // one product per (shared index, batch entry)
  int nM = 0, nN = 0;    // private kept variables of the M and N sides
  int nt = 0;            // N tile
  int64_t mrows = 0, mtiles = 0, ntiles = 0, kc = 0, inst = 0;
  int64_t bytesM = 0, bytesN = 0;  // plane bytes of the M and N sides
};

// planes: 16-bit terms per complex value (4: FP16 high and low parts of the
// real and imaginary parts; 6: three BF16 terms of each)
inline TcCfg tc_config(const GemmDesc &g, int Bp, int planes, int nt_cap = 256) {
  TcCfg c;
  const bool one = g.o_bat && (g.a_bat != g.b_bat);
  c.swap = one ? (g.b_bat != 0) : (g.nn > g.nm);
  c.fold = one && Bp > 1;
  c.perbeta = g.o_bat && g.a_bat && g.b_bat && Bp > 1;
  c.nM = c.swap ? g.nn : g.nm;
  c.nN = c.swap ? g.nm : g.nn;
  if (g.nk < 1 || c.nN < 5 || g.ns > 15 || c.nM > 30) return c;
  c.mrows = ((int64_t)1 << c.nM) * (c.fold ? Bp : 1);
  if (c.mrows < TC_M) return c;
  c.mtiles = (c.mrows + TC_M - 1) / TC_M;
  c.nt = c.nN >= 8 ? 256 : (1 << c.nN);
  if (c.nt > nt_cap && nt_cap >= 32) c.nt = nt_cap;  // narrower N tiles: two accumulators in tensor memory
  c.ntiles = ((int64_t)1 << c.nN) / c.nt;
  c.kc = (((int64_t)1 << g.nk) + 15) / 16;  // fewer than 16 summed entries: one chunk, zero-padded
  c.inst = ((int64_t)1 << g.ns) * (c.perbeta ? Bp : 1);
  if (c.inst * c.mtiles * c.ntiles >= ((int64_t)1 << 31)) return c;
  c.bytesM = c.inst * c.mtiles * c.kc * planes * TC_M * 32;
  c.bytesN = c.inst * c.ntiles * c.kc * planes * c.nt * 32;
  c.ok = true;
  return c;
}

// Launch parameters of one step chosen by the autotuner (qgm_plan_opts.autotune)
// by timing its candidates on the bound device; zeros are the fixed rules.
struct StepTune {
  int32_t nt_cap = 0;     // tensor-core GEMM: N tile at most 256, 128 or 64 (0: the rule)
  int32_t T = 0;          // batched product-sum: term groups per row (0: rule)
  int32_t conv = 0;       // folded tensor-core step: 1 converts the M side in the product kernel
  int32_t U = 0;          // batched product-sum: terms in flight per thread (4 or 8, else 2)
  int32_t ps = 0;         // GEMM-shaped step: 1 runs it with the product-sum kernels
  float ms_rule = 0.f;    // measured time with the fixed rules (ms)
  float ms_best = 0.f;    // measured time of the chosen candidate (ms)
};

// A GEMM step runs on the tensor cores when its tensor-core form exists: the
// M side has at least 128 rows (batch entries counted when they become
// rows), the N side at least 32 (summed entries are zero-padded to whole
// chunks of 16, one MMA's K).
inline bool gemm_tc_eligible(const GemmDesc &g, int Bp) { return tc_config(g, Bp, 4).ok; }

// The FP32-core GEMM kernel's shapes: 64-row A tiles, 32- or 64-column B
// tiles, chunks of 16 summed entries.  Other GEMM steps (accepted for the
// tensor cores) run with the product-sum kernels where the tensor cores are
// not used.
inline bool gemm_fp32_ok(const GemmDesc &g) { return g.nk >= 4 && g.nm >= 6 && g.nn >= 5; }

// ------------------------------------------------------------- step program
// Most steps of a plan are small: alone in a launch they cost its latency and
// the setup of its index tables (5 to 8 us a step).  They run instead as
// segments of a program: one launch takes all small steps between two large
// ones, cut into units of one CTA's work, which CTAs take in the order of a
// ticket counter; a unit waits for the units of the steps it reads (counters
// in the workspace).  Units are numbered so that a step's producers come
// first, so a unit only ever waits for units taken before it.
// (a descriptor's runs: a map's, one split between rows and terms, one more
// where a long sum is cut in two)
constexpr int PMAXRUN = MAXRUN + 2;

// One input: index = the row's and the term's bits by contiguous runs, each
// packed as source bit | length << 8 | destination bit << 16 (row runs first).
struct PIn {
  int64_t off;       // byte offset of the tensor in the workspace (below 2 GiB in size)
  int64_t meta;      // byte offset of its Meta, -1 for leaves
  int32_t batched;
  int16_t nrow, nterm;
  uint32_t run[PMAXRUN];
};

struct PStep {
  int32_t m, k, w_out, batched;
  int64_t out_off, out_meta;  // byte offsets
  int32_t lg;                 // 2^lg lanes share an item's terms
  int32_t items, pairs;       // items = rows x batch pairs (1 without a batch axis)
  int32_t unit_items, n_units;
  int32_t n_deps, signal;     // steps waited for; 1: another task waits for this one
  int32_t dep[MAXIN], dep_units[MAXIN];
  PIn in[MAXIN];
};

// One ticket: unit `unit` of step `step`, or (count > 1) the one-unit steps
// step .. step + count - 1, each reading the one before it, run in turn by
// the same CTA.
struct PTask {
  int32_t step, unit, count, pad_;
};

struct ProgramOp {
  int32_t big;          // >= 0: index of a step launched on its own; -1: a segment
  int32_t task0, tasks; // the segment's tasks
  int64_t wait_ns;      // longest wait of a unit for another step
};

struct Program {
  std::vector<StepDesc> all;     // every step, offsets as the program uses them
  std::vector<GemmDesc> gemms;
  std::vector<std::vector<int>> prod;  // producer step of each input (-1: a leaf or another pass's tensor)
  // phase by phase: a segment of small steps, then (if any) one large step
  std::vector<char> big;           // per step: launched on its own
  std::vector<int> phase, big_at;  // phase of each step; the large step of each phase (-1: none)
  int time(int s) const { return 2 * phase[s] + big[s]; }
  std::vector<PStep> steps;
  std::vector<PTask> tasks;
  std::vector<ProgramOp> ops;
  int32_t n_segments = 0, n_tmp = 0;  // segments; temporary tensors of split sums
  int64_t tmp_bytes = 0;
  // workspace layout: sync words (abort, a ticket per segment, a counter per
  // step), the temporaries' Meta (both cleared with the leaves), descriptors
  int64_t off_sync = 0, off_steps = 0, off_tasks = 0, off_tmp = 0;
  int64_t done_word() const { return 1 + n_segments; }
  int64_t meta_word() const { return (done_word() + (int64_t)steps.size() + 1) & ~int64_t(1); }
  int64_t sync_words() const { return meta_word() + 2 * n_tmp; }
};

// --------------------------------------------------- register-tiled step
// A large batched product-sum step of two inputs,
//   out[c] = sum_e A[e, cm] B[e, cn]
// for the tile c = (cm, cn) of outputs one thread forms for one batch entry:
// cm runs over output bits only A holds, cn over bits only B holds, so each
// loaded value serves a row or a column of the tile.
constexpr int REG_TM = 3, REG_TN = 2;  // most tile bits of either kind
struct RegIn {
  int64_t off;
  int32_t meta, batched;
  int32_t nrow, nterm;
  uint32_t run[PMAXRUN];               // row runs, then term runs (as PIn)
  int64_t tile[REG_TM + REG_TN];       // index steps of the tile bits (0: not held), cm first
};
struct RegStep {
  int32_t k, tm, tn;                   // summed variables; tile bits
  int32_t wr, rl;                      // row bits outside the tile; of them below the batch block
  int32_t lb, nblk;                    // batch entries per block (log2), blocks per row
  int32_t out_meta, norun;
  int64_t out_off;
  uint32_t orun[PMAXRUN];
  int64_t otile[REG_TM + REG_TN];
  RegIn in[2];
};

// A step of two to five inputs as
//   out[c] = sum_{e1} prod_{i >= 2} F_i[e1, c] * sum_{e2} A[e1, e2, cm] B[e1, e2, cn]
// with the pair's operands staged in shared memory: e2 are the summed
// variables the pair (A, B) alone holds; a CTA of 256 threads forms tiles of
// 2^(3 + mgb) x 2^(2 + ngb) outputs (cm and cn as in RegStep) for 2^lb batch
// entries and 2^rb rows, a thread 8 x 4 of them.
constexpr int MM_MAXX = 3;                                  // most further inputs
constexpr int MM_TM = 3, MM_TN = 2, MM_KC = 4;  // thread tile (log2); summed entries per stage
constexpr int MM_MBITS = MM_TM + 3, MM_NBITS = MM_TN + 3;
struct MmIn {
  int64_t off;
  int32_t meta, batched;
  int32_t nrow, nterm;
  uint32_t run[PMAXRUN];
  int64_t tile[MM_MBITS + MM_NBITS];  // index steps of the tile bits (0: not held), rows (m) first
};
struct MmStep {
  int32_t nx, k1, k2;      // further inputs; summed variables outside and inside
  int32_t mgb, ngb, rb;    // thread groups along m and n, rows of a CTA (log2)
  int32_t lb, nblk;        // batch entries of a CTA (log2), blocks
  int32_t wr, wp;          // row bits outside the tile; of them, above the rb lowest, held by A or B alone
  int32_t out_meta, norun;
  int64_t out_off;
  uint32_t orun[PMAXRUN];
  int64_t otile[MM_MBITS + MM_NBITS];
  MmIn in[2 + MM_MAXX];
};

// Leaf factor built on the device per slice: base table over
// (internal vars | slice vars | output vars), MSB first.
struct LeafDesc {
  int64_t base_off;  // complex64 base table (bytes into the workspace)
  int64_t out_off;   // built table
  int32_t n_int, n_slice, n_out, batched;
  int32_t slice_bit[MAXLEAFV];  // bit of the slice id for each slice var
  int32_t out_qubit[MAXLEAFV];  // qubit of each output var
};

// Resident executor: one CTA per chunk of Bc batch entries runs every step
// with its tensors in shared memory.  Offsets are bytes into dynamic smem.
// Input index = pext(row, runs) | (pext(e, emask) << rowbits): the summed
// variables are the top bits of the union index and, the input's variables
// being sorted the same way, the top bits of the input index too.
// One input of a resident step with its address tables precomputed by the
// planner (every input index is linear in the bits of the union index; all
// entries are byte offsets in shared memory):
//   lrow[b]  value of row bit b (b < r0), for a thread's first row;
//   lterm[b] value of summed bit b (b < lg), for a thread's first term;
//   rinc[t]  change when the thread's row counter carries into bit t;
//   tinc[t]  change when its term counter carries into bit t.
struct RIn {
  int32_t soff;      // smem byte offset of the tensor
  int32_t meta;      // smem metadata slot (intermediates), -1 for leaves
  int32_t batched;
  int32_t nlow;      // entries of lrow in use (min(r0, w_out))
  int32_t rinc[16];
  int32_t tinc[8];
  int32_t lrow[8];
  int32_t lterm[8];
};

struct RStep {
  int32_t m, k, w_out, batched_out;
  int32_t out_soff, out_meta;
  // warps [w0, w0 + nw) run the step with 2^lg lanes per output entry;
  // bit 16: the last step of its dependency level (a block barrier follows)
  int32_t sched;
  int32_t bytes;     // bytes of this descriptor in use (header + m inputs)
  RIn in[MAXIN];
};
constexpr int SCHED_LAST = 1 << 16;

struct RLeaf {        // leaf materialised in smem per chunk
  int32_t leaf;       // index into the LeafDesc table
  int32_t soff;
  int32_t batched;    // 1: rows x Bc entries from the bitstrings; 0: the table
  int32_t pad_;
};

// One row of a leaf staged into shared memory: entry (row, beta) is base
// entry src + (output bits of x_beta) stored at smem byte dst + 8 * beta
// (batched) or dst (unbatched).
struct RJob {
  int32_t src;      // float2 index into the workspace base tables
  int32_t dst;      // smem byte offset of (row, beta = 0)
  uint8_t n_out;    // output qubits of the leaf (0..2)
  uint8_t q0, q1;   // their qubits, most significant first
  uint8_t batched;
};

// Work list of the warps: entry = step | level << 12 | descriptor words << 22;
// warp w owns entries [wstart[w], wstart[w + 1]), ordered by level.
struct ResidentLayout {
  int chunk = 0;            // Bc
  int64_t smem_bytes = 0;   // dynamic shared memory per CTA
  std::vector<RStep> steps;
  std::vector<RLeaf> leaves;
  std::vector<RJob> jobs;
  std::vector<uint32_t> wlist;
  int32_t wstart[RES_WARPS + 1] = {0};
  int n_levels = 0;
  int wlist_soff = 0;       // smem byte offset of the work lists
  int final_soff = -1, final_meta = -1;
  std::vector<int> src_step, level;  // per entry of `steps`: plan step, dependency level
  // The bitstring-independent part: steps without a batch axis, run once per
  // call by a one-CTA kernel (compiled executor); `pre` lists their outputs
  // read by batched steps, staged through the workspace's pre region.
  struct PreT {
    int32_t soff;     // smem byte offset in this layout
    int32_t meta;     // metadata slot
    int32_t entries;  // complex64 entries
    int32_t goff;     // float2 index in the pre region's data
  };
  std::vector<PreT> pre;
  bool split_pre = false;  // the compiled executor runs the pre kernel
};

// Shared-memory bytes of the work lists, which sit between the metadata and
// the tensors (the compiled kernel has no work lists and drops them).
inline int64_t worklist_bytes(const ResidentLayout &L) { return ((int64_t)L.wlist.size() * 4 + 15) & ~int64_t(15); }
// Parametrised gates each tensor of the elimination is formed from.
std::vector<int> rotations(const qgm_plan *p);
// Steps of the compiled resident kernel with a static bound on their output:
// inputs are scaled to maxima at most 1 (gate tables have entries of modulus
// at most 1), so |out| <= 2^k for k summed variables.  That bound serves as
// the recorded maximum (no run-time reduction, and a constant scale in the
// consumer).  Powers of two cost no precision; what a loose bound gives away
// is headroom towards FP32's smallest values, as the consumer multiplies raw
// values.
//
// The slack is counted along the tree: k bits and one per scaled input (fixed
// gates have entries of modulus 1: a step's values are sums of phases), and
// ROTATION_BITS for every parametrised gate, whose table (the plan is kept over
// new angles) may have entries as small as one likes.  It is an estimate (sums
// may cancel further, angles be smaller), so it stays far from the range:
// tensors are measured instead, the loosest first, such that no step's output,
// and no step's inputs together, have more than SLACK_BITS.  Behind a rotation, a product of measured tensors may
// be small everywhere (large entries of one meeting small ones of the other):
// a step that reads one measured is itself measured, as is the final tensor
// (non-finite values reach it and set the status there).
//
// Over grids of up to 28 qubits and depths of 8 to 60 the largest product of
// raw values of any step is above 2^-70 (2^-133, out of range, when only a
// step's own output was held to 48 bits).
constexpr int SLACK_BITS = 48, ROTATION_BITS = 9;
struct StaticBound {
  int k = 0;               // |out| <= 2^k
  bool exp_known = false;  // every input's exponent is known too:
  int exp = 0;             //   the output's, else it is formed at run time
};
std::map<int, StaticBound> static_bounds(const qgm_plan *p, const ResidentLayout &L);  // by metadata slot
// 16-byte chunks of the compiled resident kernel's initial shared memory that
// hold something (tensor metadata, bitstring-independent leaf rows); the
// others are written before they are read
std::vector<uint32_t> image_chunks(const qgm_plan *p, const ResidentLayout &L);
// Dynamic shared memory of the compiled resident kernel (16-byte multiple).
inline int64_t compiled_smem(const ResidentLayout &L) { return (L.smem_bytes - worklist_bytes(L) + 15) & ~int64_t(15); }

// Gradient of one parametrised gate (adjoint elimination): the adjoint of
// the leaf holding the gate, and the leaf's derivative tables with respect to
// theta and phi in the leaf's base-table layout.
struct GradParam {
  int64_t dbase_off[2];  // complex64 derivative base tables (bytes into the workspace)
  int64_t adj_off;       // adjoint of the leaf: rows x batch_padded complex64
  int32_t adj_meta;
  int32_t n_int, n_out, n_slice;  // derivative table over (internal | slice | output) variables
  int32_t out_qubit[MAXLEAFV];
  int32_t slice_bit[MAXLEAFV];    // bit of the slice id for each slice variable
};

struct SymTensor {
  std::vector<int> vars;  // sorted by elimination position
  bool batched = false;
  int leaf = -1;          // leaf index or -1
  int meta = -1;          // metadata slot for intermediates
  int64_t off = -1;       // byte offset in the workspace
  int64_t entries = 0;
};

struct StepRec {
  std::vector<int> inputs;  // SymTensor ids
  std::vector<int> uni;     // union vars (sorted)
  int k = 0;
  int out = -1;
  bool batched = false;
  double bytes = 0, flops = 0;
  bool gemm = false;        // two operands, run by the GEMM kernel
  // nested evaluation (compiled resident kernel): the last k_inner summed
  // variables occur only in the inputs flagged inner, so
  // out = sum_outer prod(outer inputs) * sum_inner prod(inner inputs)
  int k_inner = 0;
  std::vector<char> inner;
};

struct LeafFactor {          // merged factor after fixing the inputs
  std::vector<int> scope;    // var ids (table is C-order over scope)
  std::vector<cd> table;
  int half_pow = 0;
  std::vector<int> members; // model factor ids merged into it
};

struct SimResult {
  double bytes = 0, flops = 0, max_step_bytes = 0;
  int64_t max_entries = 0;
  int64_t arena_peak = 0;
  int max_clique = 0;
  std::vector<SymTensor> tensors;
  std::vector<StepRec> steps;
  std::vector<int> final_tensors;
  int final_tensor = -1;
  int tree_error = -1;  // a tensor consumed other than once (plan invariant broken)
};

}  // namespace qgm

struct qgm_circuit {
  qgm::Circuit c;
};
struct qgm_model {
  qgm::Model m;
};

struct qgm_exec_state;  // device-side state (exec.cu)

struct qgm_plan {
  const qgm::Model *model_copy_owner = nullptr;
  qgm::Model model;
  qgm_plan_opts opts{};
  int order_kind = 0;
  int output_mode = 0;
  int64_t batch = 1;
  int32_t Bp = 1;
  std::vector<int> order;        // eliminated vars
  std::vector<int> open_vars;    // never eliminated (open outputs)
  std::vector<int> slice_vars;
  std::vector<int> pos;          // elimination position per var (-1: not in graph)
  std::vector<int> var_role;     // 0 free, 1 input, 2 output(batched), 3 open, 4 slice
  std::vector<qgm::LeafFactor> leaves;
  qgm::cd constant = 1.0;        // product of scope-free factors and 2^{-L/2}
  int half_pow_total = 0;
  qgm::SimResult sim;
  // device layout
  std::vector<qgm::StepDesc> steps;
  std::vector<qgm::GemmDesc> gemms;
  std::vector<qgm::LeafDesc> leafdesc;
  std::vector<float> base_tables;  // interleaved complex64
  int n_meta = 0;
  int64_t off_header = 0, off_meta = 0, off_leafdesc = 0, off_base = 0, off_leaf = 0, off_bits = 0,
          off_outstage = 0, off_acc = 0, off_arena = 0, ws_bytes = 0;
  int64_t final_entries = 0;     // rows of the final tensor (2^n_open or 1)
  int open_in_batch = 0;         // open output qubits of a batch plan (k)
  int final_batched = 0;
  int64_t final_off = 0;
  int final_meta = -1;
  // adjoint elimination (qgm_plan_opts.gradients): forward steps that keep
  // every intermediate, the seed, backward steps, one record per parameter
  bool grad = false;
  std::vector<qgm::StepDesc> gfwd, gbwd;
  std::vector<qgm::GradParam> gparams;
  int64_t g_final_off = 0, g_seed_off = 0, off_gparams = 0;
  int g_final_meta = -1, g_seed_meta = -1, g_final_batched = 0;
  int n_meta_fwd = 0;
  // resident executor layouts for Bc = 1, 2, 4, 8 (empty when infeasible)
  std::vector<qgm::ResidentLayout> resident;
  int64_t off_rsteps = 0;   // workspace region for the chosen layout's steps
  int64_t off_pre = 0;      // pre region: per pre tensor (maxbits, exp), then the data (16-byte aligned)
  int64_t pre_data = 0;     // float2 index of the data inside the pre region
  int64_t off_image = 0;    // compiled resident kernel: initial shared-memory image (bitstring-independent leaves)
  int executor_pref = 0;    // qgm_plan_opts.executor
  bool gemm_ok = true;      // GEMM-shaped steps run by the GEMM kernel
  bool gemm_tc = false;     // eligible GEMM steps run on the tensor cores (split terms)
  int tc_planes = 4;        // 16-bit terms per complex value: 4 (FP16 x 2) or 6 (BF16 x 3)
  int64_t off_planes = 0;   // workspace region of the split operand planes
  int64_t planes_bytes = 0; // its size (the largest tensor-core step's two operands)
  int64_t ws_fwd_bytes = 0; // workspace the forward pass needs without that region
  std::vector<qgm::StepTune> tune;  // per step of `steps` (autotuner choices)
  qgm::Program fprog, gprog;  // the forward and the gradient pass as step programs
  int64_t f_final_off = 0;    // the forward program's final tensor
  int64_t prog_end = 0;       // end of the tensors' region (both layouts)
  int64_t live_bytes = 0;     // live intermediates of the larger layout, split sums' temporaries included
  // per leaf: table layout (internal | slice | output variables), offset of
  // its base table and of its derivative tables (floats), its RXY member
  std::vector<std::vector<int>> leaf_layout;
  std::vector<int64_t> base_at, dbase_at;
  std::vector<int> rxy_member;
  // leaves holding an RXY gate (qgm_plan_set_params): per member its factor
  // and, per entry of the leaf's base table, the entry of the factor's table
  struct ParamLeaf {
    int leaf;
    std::vector<int> factor;
    std::vector<std::vector<uint8_t>> entry;
  };
  std::vector<ParamLeaf> param_leaf;
  bool trees_ok = false;    // buckets of three or more inputs may run as contraction trees
  bool nest_ok = true;      // buckets may be marked for nested evaluation
  qgm_exec_state *exec = nullptr;
};

namespace qgm {
int build_plan(const Model &m, const qgm_plan_opts &o, qgm_plan *p);
int plan_set_params(qgm_plan *p, const double *params);
// The phases of P.all (program.cpp): run = 0 gives every small step the first
// segment after its producers; else the steps keep their order, at most `run`
// small ones to a segment (less memory is live then).
void program_phases(Program &P, int Bp, int run);
// Cut P.all into segments of small steps and large steps launched on their
// own, by its phases.  split: long sums over few outputs in two, through a
// temporary.
void build_program(Program &P, int Bp, int64_t off_meta, bool split);
// Whether a step is launched on its own by its size and form.
bool program_alone(const StepDesc &d, int Bp);
// The register-tiled form of a step, where it has one that pays.
bool reg_step(const StepDesc &d, int Bp, RegStep &r);
// Its form with operands staged in shared memory, likewise.
bool mm_step(const StepDesc &d, int Bp, MmStep &r);
// Sizes of the program's workspace region, laid out from `off` on; returns its end.
int64_t place_program(Program &P, int64_t off);
// CUDA source of the resident kernel specialised to one layout (jit.cpp):
// the whole pass, its batched part, or its bitstring-independent part
enum { RES_WHOLE = 0, RES_MAIN = 1, RES_PRE = 2 };
std::string resident_source(const qgm_plan *p, const ResidentLayout &L, const std::string &name, int minb,
                            int mode);
}
