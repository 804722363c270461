// Schedules an SSA program for the interpreter kernel and places its values.
//
// This is the sequential traversal of CusADi §III-A ("traversing across the
// instructions sequentially") kept for programs too large to compile, with W
// warps sharing the instructions of each group of 32 instances (lane =
// instance): walking one stream with one thread per instance left the kernel
// waiting for one instruction's operands at a time, and a work vector of
// ~1,000 slots per instance lived in HBM (LDL^T with 47 unknowns, N = 16,384:
// 16.7 ms).  Ops get a warp and a phase (pack_phases): an op may read its own
// warp's values at once and another warp's from earlier phases; a CTA barrier
// separates phases.  A multiply whose only reader is an add or subtract is
// evaluated by it (rounded on its own, so the results keep their bits).
//
// Work slots come in two tiers: slots in shared memory (32 instances each) and,
// beyond them, rows of a global workspace.  A value holds one slot from its
// phase to the phase of its last read; a value read only by its own warp in its
// own phase gives its slot back at that read.  Which values get shared slots is
// decided by linear scan over the phases (M. Poletto and V. Sarkar, "Linear
// scan register allocation", TOPLAS 21(5), 1999): when the shared slots are
// full, whichever of the new value and the live ones is read last moves to the
// workspace for its whole life.  Inputs and constants are read where they are.
#include <algorithm>
#include <cmath>
#include <set>

#include "internal.h"

namespace cusadi {

namespace {

// shared memory of one CTA that slots can take (the rest stages the streams)
constexpr int64_t kSlotBytesMax = 200 * 1024;

// One program's ops, fused multiplies and dependences; build() lays it out for a
// number of warps and a phase length.
struct Packer {
  const Graph& g;
  const int dtype, shared_kb;
  const int64_t n, elt;
  std::vector<std::vector<int64_t>> out_rows;
  std::vector<int32_t> fused;      // per add or subtract: the multiply it evaluates, -1
  PhaseDag d;

  Packer(const Graph& g_, int dtype_, int shared_kb_);
  bool leaf(int64_t i) const { return g.nodes[i].op == INPUT || g.nodes[i].op == CONST; }
  // operands of the (possibly fused) op: multiply's factors first, then the other
  std::array<int32_t, 3> operands(int64_t i) const {
    const Node& x = g.nodes[i];
    const int32_t m = fused[i];
    if (m < 0) return {x.a, x.b, -1};
    return {g.nodes[m].a, g.nodes[m].b, x.a == m ? x.b : x.a};
  }
  // target < 0: one warp, the program's own order
  bool build(int ways, double target, InterpProgram& p, std::string& err) const;
};

Packer::Packer(const Graph& g_, int dtype_, int shared_kb_)
    : g(g_), dtype(dtype_), shared_kb(shared_kb_), n((int64_t)g_.nodes.size()), elt(dtype_ == CUSADI_F32 ? 4 : 8) {
  out_rows.assign(n, {});
  for (size_t r = 0; r < g.out.size(); ++r) out_rows[g.out[r]].push_back((int64_t)r);
  std::vector<int32_t> reads(n, 0);
  for (const Node& x : g.nodes) {
    if (x.a >= 0) ++reads[x.a];
    if (x.b >= 0) ++reads[x.b];
  }
  fused.assign(n, -1);
  d.deps.assign(n, {-1, -1, -1});
  d.skip.assign(n, 0);
  d.cost.assign(n, 0.0);
  for (int64_t i = 0; i < n; ++i) {
    if (leaf(i)) { d.skip[i] = 1; continue; }
    const Node& x = g.nodes[i];
    if (x.op != ADD && x.op != SUB) continue;
    for (int32_t m : {x.a, x.b})
      if (fused[i] < 0 && g.nodes[m].op == MUL && reads[m] == 1 && out_rows[m].empty() && g.nodes[m].f64 == x.f64) {
        fused[i] = m;
        d.skip[m] = 1;
      }
  }
  const double dispatch = 8.0;   // decoding and operand reads, in op_cost's units
  for (int64_t i = 0; i < n; ++i) {
    if (d.skip[i]) continue;
    const std::array<int32_t, 3> o = operands(i);
    for (int k = 0; k < 3; ++k) d.deps[i][k] = o[k] >= 0 && !leaf(o[k]) ? o[k] : -1;
    d.cost[i] = dispatch + op_cost(g.nodes[i], dtype) + (fused[i] >= 0 ? op_cost(g.nodes[fused[i]], dtype) : 0.0);
  }
  d.finish();
}

bool Packer::build(int ways, double target, InterpProgram& p, std::string& err) const {
  p = InterpProgram();
  p.ways = ways;
  const int64_t AUX_MAX = (1 << 24) - 1, IDX_MAX = (int64_t)kOperandMask;
  const bool own_order = target < 0;
  CoopPlan plan;
  if (own_order) {
    plan.owner.assign(n, 0);
    plan.phase.assign(n, 0);
  } else {
    plan = pack_phases(d, ways, target);
  }
  p.estimate = estimate_phases(d, plan, 30.0);
  // per phase and warp, the order: bundles of up to kBundle multiply-adds on work
  // slots that do not read one another's results, each as early as the results it
  // reads allow, and every other instruction (an op or an output store) alone
  struct Item { int64_t node, row; };                       // row >= 0: store of that output row
  typedef std::vector<std::vector<Item>> Bundles;
  std::vector<std::vector<Bundles>> work(plan.n_phases, std::vector<Bundles>(p.ways));
  std::vector<int> bundle_of(n, -1);
  {
    auto multiply_add = [&](const Item& it) {
      if (own_order || it.row >= 0 || fused[it.node] < 0) return false;
      for (int32_t o : operands(it.node))
        if (leaf(o)) return false;
      return dtype != CUSADI_MIXED;
    };
    std::vector<std::vector<size_t>> room(plan.n_phases, std::vector<size_t>(p.ways, 0));
    auto place = [&](Bundles& B, size_t& first, size_t from, Item it) -> int {
      if (!multiply_add(it)) {
        B.push_back({it});
        return (int)B.size() - 1;
      }
      auto fits = [&](size_t k) { return B[k].size() < (size_t)kBundle && multiply_add(B[k][0]); };
      size_t b = std::max(first, from);                      // no bundle before `first` has room
      while (b < B.size() && !fits(b)) ++b;
      if (b == B.size()) B.push_back({it});
      else B[b].push_back(it);
      while (first < B.size() && !fits(first)) ++first;
      return (int)b;
    };
    for (int64_t i = 0; i < n; ++i) {
      if (leaf(i)) {                                        // outputs fed directly by inputs or constants
        for (int64_t r : out_rows[i]) place(work[0][0], room[0][0], 0, {i, r});
        continue;
      }
      if (d.skip[i]) continue;
      const int q = plan.phase[i], w = plan.owner[i];
      size_t from = 0;
      for (int32_t o : operands(i))
        if (o >= 0 && !leaf(o) && plan.phase[o] == q) from = std::max(from, (size_t)bundle_of[o] + 1);
      bundle_of[i] = place(work[q][w], room[q][w], from, {i, -1});
      for (int64_t r : out_rows[i]) place(work[q][w], room[q][w], (size_t)bundle_of[i] + 1, {i, r});
    }
    // what did not fill a bundle runs one by one
    for (std::vector<Bundles>& phase : work)
      for (Bundles& B : phase) {
        Bundles out;
        for (const std::vector<Item>& b : B)
          if (b.size() == (size_t)kBundle) out.push_back(b);
          else
            for (const Item& it : b) out.push_back({it});
        B.swap(out);
      }
  }

  // 3. slots.  last[i]: phase of the last read; own_last[i]: the bundle that reads
  // a private value (all reads by its own warp in its own phase) last
  std::vector<int> last(n, -1), own_last(n, -1);
  std::vector<uint8_t> priv(n, 1);
  for (int q = 0; q < plan.n_phases; ++q)
    for (int w = 0; w < p.ways; ++w)
      for (size_t b = 0; b < work[q][w].size(); ++b)
        for (const Item& it : work[q][w][b]) {
          const std::array<int32_t, 3> o3 = it.row >= 0 ? std::array<int32_t, 3>{(int32_t)it.node, -1, -1} : operands(it.node);
          for (int32_t o : o3) {
            if (o < 0 || leaf(o)) continue;
            last[o] = std::max(last[o], q);
            if (plan.phase[o] != q || plan.owner[o] != w) priv[o] = 0;
            else own_last[o] = std::max(own_last[o], (int)b);
          }
        }
  const int64_t budget = std::min<int64_t>((int64_t)shared_kb * 1024 * p.ways / 4, kSlotBytesMax) / (32 * elt);
  std::vector<int64_t> slot(n, -1);
  std::vector<uint8_t> global(n, 0);
  // one tier's allocation: values in order of definition; with a limit, the value
  // read last leaves (it is marked global and gets its row in the second pass)
  auto assign = [&](bool second, int64_t limit) -> int64_t {
    std::set<std::pair<int, int64_t>> active;              // (last phase, value)
    std::vector<int64_t> free_slots;
    int64_t next = 0;
    std::vector<int64_t> ret;                              // private slots back at the phase's end
    for (int q = 0; q < plan.n_phases; ++q) {
      while (!active.empty() && active.begin()->first < q) {
        free_slots.push_back(slot[active.begin()->second]);
        active.erase(active.begin());
      }
      for (int64_t s : ret) free_slots.push_back(s);
      ret.clear();
      for (int w = 0; w < p.ways; ++w) {
        std::vector<int64_t> mine;                         // this warp's own free slots in this phase
        const uint8_t tier = second ? 1 : 0;
        for (size_t b = 0; b < work[q][w].size(); ++b) {
          // private values read here for the last time give their slots back (the
          // bundle's results are written after its reads)
          for (const Item& it : work[q][w][b]) {
            const std::array<int32_t, 3> o3 = it.row >= 0 ? std::array<int32_t, 3>{(int32_t)it.node, -1, -1} : operands(it.node);
            for (int32_t o : o3)
              if (o >= 0 && !leaf(o) && priv[o] && own_last[o] == (int)b && global[o] == tier && slot[o] >= 0 &&
                  std::find(mine.begin(), mine.end(), slot[o]) == mine.end())
                mine.push_back(slot[o]);
          }
          for (const Item& it : work[q][w][b]) {
            const int64_t i = it.node;
            if (it.row >= 0 || global[i] != tier) continue;
            const bool pv = priv[i] && own_last[i] >= 0;
            const int end = std::max(last[i], q);
            if (!mine.empty() && pv) { slot[i] = mine.back(); mine.pop_back(); continue; }
            if (!free_slots.empty() || next < limit) {
              if (!free_slots.empty()) { slot[i] = free_slots.back(); free_slots.pop_back(); }
              else slot[i] = next++;
            } else if (!pv && !active.empty() && std::prev(active.end())->first > end) {
              auto far = std::prev(active.end());
              const int64_t u = far->second;
              slot[i] = slot[u];
              slot[u] = -1;
              global[u] = 1;
              active.erase(far);
            } else {
              global[i] = 1;
              continue;
            }
            if (!pv) active.insert({end, i});
          }
        }
        for (int64_t s : mine) ret.push_back(s);
      }
    }
    return next;
  };
  p.n_shared = assign(false, budget);
  p.n_global = assign(true, (int64_t)1 << 40);
  for (int64_t v = 0; v < n; ++v)
    if (global[v]) slot[v] += p.n_shared;                  // global rows follow the shared slots
  p.n_slots = std::max<int64_t>(p.n_shared + p.n_global, 1);
  if (p.n_slots > AUX_MAX) { err = "too many live values for the interpreter"; return false; }

  // 4. the streams.  A reduced (broadcast) row carries its index among the reduced
  // rows + 1, the same in every layout.
  std::vector<uint32_t> reduced(g.out.size(), 0);
  for (size_t r = 0; r < g.out.size(); ++r)
    if (!g.out_reduce.empty() && g.out_reduce[r]) {
      p.reduce_rows.push_back((int64_t)r);
      reduced[r] = (uint32_t)p.reduce_rows.size();
    }
  std::vector<int64_t> const_at(n, -1);
  auto constant = [&](double v) -> int64_t {
    p.k.push_back(v);
    return (int64_t)p.k.size() - 1;
  };
  auto operand = [&](int32_t i) -> uint32_t {
    if (i < 0) return 0;
    const Node& x = g.nodes[i];
    if (x.op == CONST) {
      if (const_at[i] < 0) const_at[i] = constant(x.k);
      return 3u << kOperandShift | (uint32_t)const_at[i];
    }
    if (x.op == INPUT) return (x.bcast ? 2u : 1u) << kOperandShift | (uint32_t)x.io;
    return (uint32_t)slot[i];
  };
  auto code = [&](uint32_t op, int f64, int64_t aux) { return op | (uint32_t)(f64 ? 1 : 0) << 7 | (uint32_t)aux << 8; };
  if ((int64_t)g.out.size() > AUX_MAX) { err = "too many output rows for the interpreter"; return false; }
  if (g.nnz_in > IDX_MAX) { err = "too many input rows for the interpreter"; return false; }
  for (int w = 0; w < p.ways; ++w) {
    p.begin.push_back((int32_t)p.ops.size());
    for (int q = 0; q < plan.n_phases; ++q) {
      for (const std::vector<Item>& bundle : work[q][w]) {
        // a full bundle starts at a multiple of its size
        while (bundle.size() == (size_t)kBundle && (p.ops.size() - p.begin.back()) % kBundle != 0)
          p.ops.push_back({I_NOP, 0, 0, 0});
        for (const Item& it : bundle) {
          const int64_t i = it.node;
          if (it.row >= 0) {
            p.ops.push_back({code(I_OUTPUT, 0, it.row), operand((int32_t)i), reduced[it.row], 0});
            continue;
          }
          const Node& x = g.nodes[i];
          const std::array<int32_t, 3> o = operands(i);
          IOp I{code(x.op, x.f64, slot[i]), operand(o[0]), operand(o[1]), operand(o[2])};
          if (fused[i] >= 0)
            I.code = code(x.op == ADD ? I_MUL_ADD : (x.a == fused[i] ? I_MUL_SUB : I_SUB_MUL), x.f64, slot[i]);
          else if (x.op == FMA_CONST)
            I.c = 3u << kOperandShift | (uint32_t)constant(x.k);
          p.ops.push_back(I);
        }
        if (bundle.size() < (size_t)kBundle) continue;
        IOp* const B = &p.ops[p.ops.size() - kBundle];
        bool far = false;
        for (int k = 0; k < kBundle; ++k)
          for (uint32_t o : {B[k].a, B[k].b, B[k].c, B[k].code >> 8}) far |= o >= (uint32_t)p.n_shared;
        for (int k = 0; k < kBundle; ++k)
          B[k].code += (far ? I_FAST_FAR : I_FAST) - I_MUL_ADD;
      }
      if (q + 1 < plan.n_phases) p.ops.push_back({I_SYNC, 0, 0, 0});
    }
  }
  p.begin.push_back((int32_t)p.ops.size());
  if ((int64_t)p.k.size() > IDX_MAX) { err = "too many constants for the interpreter"; return false; }
  p.has_reduce = !p.reduce_rows.empty();
  return true;
}

}  // namespace

// Two layouts: `few` for at most kInterpFew instances (one group of 32 per SM: as
// many warps as help each), `many` beyond (more groups per SM: their phases fill
// each other's barriers, so fewer warps and fewer slots each).  Measured, FP64
// LDL^T with 47 unknowns, 4 / 8 / 16 warps: N = 16,384 2.80 / 3.09 / 4.16 ms, N =
// 300 - / 1.75 / 1.00 ms; FP32 programs have no FP64 unit to wait for and keep 8.
// The phase length that takes least estimated time is kept, per resident group for
// `many`.  A layout may not need more workspace rows than the values live at once
// in the program's own order, past 48 KB's worth; one warp in that order never does.
bool pack_interp(const Graph& g, InterpProgram& many, InterpProgram& few, std::string& err, int dtype,
                 int shared_kb) {
  const Packer P(g, dtype, shared_kb);
  const int64_t n_ops = count_ops(g), elt = P.elt;
  const int64_t max_rows = std::max<int64_t>(0, max_live(g) - (int64_t)shared_kb * 1024 / (128 * elt));
  auto choose = [&](InterpProgram& best, int ways, bool resident) -> bool {
    double best_t = -1;
    for (double target : {150.0, 600.0, 2400.0}) {
      if (n_ops > 100000 && target != 600.0) continue;     // packing time
      InterpProgram p;
      if (!P.build(ways, ways > 1 ? target : 1e30, p, err)) return false;
      const int64_t smem = p.n_shared * 32 * elt + ways * 1024;
      const double groups = std::min(std::min(64.0 / ways, 32.0), (double)(220 * 1024) / (double)std::max<int64_t>(smem, 1));
      const double t = resident ? p.estimate / std::max(1.0, std::floor(groups)) : p.estimate;
      if (p.n_global <= max_rows && (best_t < 0 || t < best_t)) { best_t = t; best = std::move(p); }
      if (ways == 1) break;
    }
    return best_t >= 0 || P.build(1, -1, best, err);
  };
  const int narrow = n_ops < 200 ? 1 : (dtype == CUSADI_F32 && n_ops > 1000 ? 8 : 4);
  if (!choose(many, narrow, true) || !choose(few, n_ops < 200 ? 1 : (n_ops > 1000 ? 16 : 8), false)) return false;
  // Ops that need one another in a chain leave warps idle, which hold the places of
  // further groups: half the warps where the program takes as long with them (35 FP32
  // quotients in a row, N = 65,536, 4 warps 144 us, one 78; FP64 162 and 91; four such
  // rows side by side FP32, 8 warps 421 us, 4 warps 254).
  double work = 0;
  for (int64_t i = 0; i < P.n; ++i)
    if (!P.d.skip[i]) work += P.d.cost[i];
  while (many.ways > 1 && work < 0.6 * many.ways * many.estimate) {
    InterpProgram p;
    if (!choose(p, many.ways / 2, true)) return false;
    if (p.ways != many.ways / 2 || p.estimate > 1.05 * many.estimate) break;
    many = std::move(p);
  }
  // workspace rows of the groups in flight: past 256 MB they come from HBM at every
  // use, and one wide group per SM is faster (LDL^T with 100 unknowns, N = 8,192:
  // 124 ms with four narrow groups per SM)
  const int64_t smem = many.n_shared * 32 * elt + many.ways * 1024;
  const int64_t groups = std::max<int64_t>(1, std::min<int64_t>(64 / many.ways, 220 * 1024 / smem));
  if (groups * kInterpFew * many.n_global * elt > (int64_t)256 << 20) many = few;
  return true;
}

}  // namespace cusadi
