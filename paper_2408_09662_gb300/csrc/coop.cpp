// Within-instance parallelism: W warps cooperate on each group of 32
// instances (lane = instance), splitting one program's ops between them.
//
// CusADi parallelises across instances only and names parallelism inside one
// expression graph as future work (§VI).  Ops are assigned a warp and a phase;
// phases are separated by a CTA barrier, an op may read a value of its own
// warp from its own or an earlier phase and a value of another warp from an
// earlier phase (through shared memory).  Two schedulers are tried and the
// one with the lower estimated time (sum over phases of the busiest warp's
// op cost plus a barrier cost) is kept:
//  * earliest finish time: each op goes to the warp where it finishes first,
//    counting a fixed cost for a value that crosses warps; phases follow;
//  * phase packing: phases are filled one at a time, up to a target cost per
//    warp, always with the ready op of longest remaining critical path (bottom
//    level), so every warp carries about the same work between barriers.
//    Several targets are tried.
#include <algorithm>
#include <cstdlib>
#include <map>
#include <queue>

#include "internal.h"

namespace cusadi {

// Cost of one node in units of about 5 clocks (an FP32 add's latency).  FP64:
// 64 clocks of the FP64 unit per add or multiply, the measured latency of the
// integer-pipe functions (math64.cuh: division 344, square root 298, exp 408,
// sin/cos 551 clocks), the library's for the rest.
double op_cost(const Node& x, int dtype) {
  const bool f64 = dtype == CUSADI_F64 || (dtype == CUSADI_MIXED && x.f64);
  switch (x.op) {
    case SIN: case COS:
      return f64 ? 110.0 : 24.0;
    case TAN: case ATAN: case ATAN2: case TANH: case ASIN: case ACOS:
    case SINH: case COSH: case ERF: case POW: case LOG: case HYPOT: case LOG1P: case EXPM1:
    case FMOD:
      return f64 ? 300.0 : 24.0;
    case EXP: return f64 ? 80.0 : 12.0;
    case DIV: case SQRT: case INV: return f64 ? 65.0 : 8.0;
    default: return f64 ? 13.0 : 1.0;
  }
}

namespace {

// a CTA barrier plus the shared-memory hand-off, in op costs (CUSADI_COOP_BARRIER_COST
// overrides it, for sweeps of the phase count against compile time and run time);
// FP64: six adds, as for FP32 (random 20k program, N = 4,096, 8 warps: 272 us from
// 20 to 150 units here, 317 us at 6)
double barrier_cost(int dtype) {
  static const double c = [] {
    const char* e = std::getenv("CUSADI_COOP_BARRIER_COST");
    return e ? std::max(0.0, std::atof(e)) : -1.0;
  }();
  return c >= 0 ? c : (dtype == CUSADI_F64 ? 78.0 : 6.0);
}

bool is_leaf(const Graph& g, int64_t i) {   // no value of its own to compute (Gen::leaf)
  return g.nodes[i].op == INPUT || g.nodes[i].op == CONST || (!g.gone.empty() && g.gone[i]);
}

struct Ready {
  double pri;
  int64_t i;
  bool operator<(const Ready& o) const { return pri < o.pri || (pri == o.pri && i > o.i); }
};

CoopPlan plan_eft(const PhaseDag& d, int ways, double comm_cost);

}  // namespace

void PhaseDag::finish() {
  const int64_t n = (int64_t)deps.size();
  bottom.assign(n, 0.0);
  users.assign(n, {});
  for (int64_t i = 0; i < n; ++i) {
    if (skip[i]) continue;
    bottom[i] = cost[i];
    for (int32_t o : deps[i])
      if (o >= 0) users[o].push_back(i);
  }
  for (int64_t i = n - 1; i >= 0; --i)
    if (!skip[i])
      for (int32_t o : deps[i])
        if (o >= 0) bottom[o] = std::max(bottom[o], cost[o] + bottom[i]);
}

double estimate_phases(const PhaseDag& d, const CoopPlan& P, double barrier) {
  std::vector<double> load((size_t)P.n_phases * P.ways, 0.0);
  for (int64_t i = 0; i < (int64_t)d.deps.size(); ++i)
    if (!d.skip[i]) load[(size_t)P.phase[i] * P.ways + P.owner[i]] += d.cost[i];
  double t = 0;
  for (int q = 0; q < P.n_phases; ++q)
    t += *std::max_element(load.begin() + (size_t)q * P.ways, load.begin() + (size_t)(q + 1) * P.ways) + barrier;
  return t;
}

CoopPlan pack_phases(const PhaseDag& d, int ways, double target) {
  const int64_t n = (int64_t)d.deps.size();
  CoopPlan P;
  P.ways = ways;
  P.owner.assign(n, -1);
  P.phase.assign(n, 0);
  std::vector<int> pending(n, 0);
  int64_t todo = 0;
  std::priority_queue<Ready> open;                        // any warp may take these
  std::vector<std::priority_queue<Ready>> mine(ways);     // need a value of this warp's phase
  std::vector<int64_t> later;                             // need values of two warps' phase
  for (int64_t i = 0; i < n; ++i) {
    if (d.skip[i]) continue;
    ++todo;
    for (int32_t o : d.deps[i])
      if (o >= 0) ++pending[i];
    if (pending[i] == 0) open.push({d.bottom[i], i});
  }
  int q = 0;
  std::vector<double> load(ways);
  std::vector<char> full(ways);
  while (todo > 0) {
    std::fill(load.begin(), load.end(), 0.0);
    std::fill(full.begin(), full.end(), 0);
    int active = ways;
    while (active > 0) {
      int w = -1;
      for (int k = 0; k < ways; ++k)
        if (!full[k] && (w < 0 || load[k] < load[w])) w = k;
      const bool has_mine = !mine[w].empty(), has_open = !open.empty();
      if (!has_mine && !has_open) { full[w] = 1; --active; continue; }
      const bool take_mine = has_mine && (!has_open || !(mine[w].top() < open.top()));
      const Ready r = take_mine ? mine[w].top() : open.top();
      const double c = d.cost[r.i];
      if (load[w] > 0 && load[w] + c > target) { full[w] = 1; --active; continue; }
      (take_mine ? mine[w] : open).pop();
      P.owner[r.i] = w;
      P.phase[r.i] = q;
      load[w] += c;
      --todo;
      for (int64_t u : d.users[r.i]) {
        if (--pending[u] != 0) continue;
        int same = -1;   // warp of the operands computed in this phase, -2 if two warps
        for (int32_t o : d.deps[u])
          if (o >= 0 && P.phase[o] == q)
            same = (same == -1 || same == P.owner[o]) ? P.owner[o] : -2;
        if (same == -1) open.push({d.bottom[u], u});
        else if (same >= 0) mine[same].push({d.bottom[u], u});
        else later.push_back(u);
      }
    }
    // what waited on this phase's values of one warp, or of two, is open next phase
    for (auto& m : mine)
      while (!m.empty()) { open.push(m.top()); m.pop(); }
    for (int64_t u : later) open.push({d.bottom[u], u});
    later.clear();
    ++q;
  }
  P.n_phases = std::max(q, 1);
  return P;
}

CoopPlan plan_coop(const Graph& g, int ways, double comm_cost, int dtype) {
  const int64_t n = (int64_t)g.nodes.size();
  PhaseDag d;
  d.deps.assign(n, {-1, -1, -1});
  d.skip.assign(n, 0);
  d.cost.assign(n, 0.0);
  // An FP64 multiply whose only reader is an add or subtract goes with it, so that the
  // compiler contracts the two as it does in the one-thread kernel: one instruction of
  // the FP64 unit less.  Not in FP32, where the schedule matters more than the
  // instruction (50,000 random ops, N = 8,192, 4 warps: 0.60 ms together, 0.45 apart).
  std::vector<int32_t> reads(n, 0), fused(n, -1);
  for (const Node& x : g.nodes) {
    if (x.a >= 0) ++reads[x.a];
    if (x.b >= 0) ++reads[x.b];
  }
  for (int32_t o : g.out) ++reads[o];
  for (int64_t i = 0; i < n; ++i) {
    const Node& x = g.nodes[i];
    if (is_leaf(g, i)) { d.skip[i] = 1; continue; }
    if ((x.op != ADD && x.op != SUB) || !g.fused.empty()) continue;   // else contract() has decided
    for (int32_t m : {x.a, x.b})
      if (fused[i] < 0 && (g.nodes[m].op == MUL || g.nodes[m].op == SQ) && reads[m] == 1 &&
          g.nodes[m].f64 == x.f64 && (dtype == CUSADI_F64 || (dtype == CUSADI_MIXED && x.f64))) {
        fused[i] = m;
        d.skip[m] = 1;
      }
  }
  for (int64_t i = 0; i < n; ++i) {
    if (d.skip[i]) continue;
    const Node& x = g.nodes[i];
    const int32_t m = fused[i];
    d.cost[i] = op_cost(x, dtype);
    std::array<int32_t, 3> o = operands(g, i);
    if (m >= 0) o = {g.nodes[m].a, g.nodes[m].b, x.a == m ? x.b : x.a};
    for (int k = 0; k < 3; ++k) d.deps[i][k] = o[k] >= 0 && !is_leaf(g, o[k]) ? o[k] : -1;
  }
  d.finish();
  CoopPlan best = plan_eft(d, ways, comm_cost);
  double best_t = estimate_phases(d, best, barrier_cost(dtype));
  // FP64 phases hold as many ops at 13 times the cost
  const double unit = dtype == CUSADI_F64 ? 13.0 : 1.0;
  for (double target : {8.0, 16.0, 32.0, 64.0, 128.0, 256.0, 512.0}) {
    CoopPlan P = pack_phases(d, ways, target * unit);
    const double t = estimate_phases(d, P, barrier_cost(dtype));
    if (t < best_t) { best_t = t; best = std::move(P); }
  }
  for (int64_t i = 0; i < n; ++i)
    if (fused[i] >= 0) {
      best.owner[fused[i]] = best.owner[i];
      best.phase[fused[i]] = best.phase[i];
    }
  return best;
}

namespace {

CoopPlan plan_eft(const PhaseDag& d, int ways, double comm_cost) {
  const int64_t n = (int64_t)d.deps.size();
  CoopPlan P;
  P.ways = ways;
  P.owner.assign(n, -1);
  P.phase.assign(n, 0);
  std::vector<double> finish(n, 0.0), avail(ways, 0.0);
  P.n_phases = 1;
  for (int64_t i = 0; i < n; ++i) {
    if (d.skip[i]) continue;
    int best = 0;
    double best_f = 1e300;
    for (int w = 0; w < ways; ++w) {
      double start = avail[w];
      for (int32_t o : d.deps[i])
        if (o >= 0) start = std::max(start, finish[o] + (P.owner[o] == w ? 0.0 : comm_cost));
      const double f = start + d.cost[i];
      if (f < best_f - 1e-12 || (f < best_f + 1e-12 && avail[w] < avail[best])) {
        best = w;
        best_f = f;
      }
    }
    P.owner[i] = best;
    finish[i] = best_f;
    avail[best] = best_f;
    int ph = 0;
    for (int32_t o : d.deps[i])
      if (o >= 0) ph = std::max(ph, P.phase[o] + (P.owner[o] == best ? 0 : 1));
    P.phase[i] = ph;
    P.n_phases = std::max(P.n_phases, ph + 1);
  }
  return P;
}

}  // namespace

int assign_coop_slots(const Graph& g, const CoopPlan& P, const std::vector<int>& seg_of_node,
                      int max_slots, std::vector<int>& slot, std::vector<int>& gslot,
                      int& n_gslots) {
  // Values read by another warp of the same kernel get a shared-memory slot for
  // the phases [producer phase, last such reader's phase]; a slot is free again
  // from the phase after its last reader.  When all max_slots are taken, the
  // value goes to a workspace row instead (the CTA barrier orders global
  // memory as well).  Reads from a later kernel go through the workspace.
  const int64_t n = (int64_t)g.nodes.size();
  auto leaf = [&](int64_t i) { return is_leaf(g, i); };
  slot.assign(n, -1);
  gslot.assign(n, -1);
  std::vector<int> last_read(n, -1);
  for (int64_t i = 0; i < n; ++i) {
    if (leaf(i)) continue;
    for (int32_t o : operands(g, i))
      if (o >= 0 && !leaf(o) && P.owner[o] != P.owner[i] && seg_of_node[o] == seg_of_node[i])
        last_read[o] = std::max(last_read[o], P.phase[i]);
  }
  std::vector<std::vector<int64_t>> by_phase(P.n_phases);
  for (int64_t i = 0; i < n; ++i)
    if (last_read[i] >= 0) by_phase[P.phase[i]].push_back(i);
  std::vector<std::vector<int>> release(P.n_phases + 1), grelease(P.n_phases + 1);
  std::vector<int> free_slots, free_g;
  int slots = 0;
  n_gslots = 0;
  for (int q = 0; q < P.n_phases; ++q) {
    for (int s : release[q]) free_slots.push_back(s);
    for (int s : grelease[q]) free_g.push_back(s);
    for (int64_t i : by_phase[q]) {
      const int end = std::min(last_read[i] + 1, P.n_phases);
      if (!free_slots.empty() || slots < max_slots) {
        int s;
        if (!free_slots.empty()) { s = free_slots.back(); free_slots.pop_back(); }
        else s = slots++;
        slot[i] = s;
        release[end].push_back(s);
      } else {
        int s;
        if (!free_g.empty()) { s = free_g.back(); free_g.pop_back(); }
        else s = n_gslots++;
        gslot[i] = s;
        grelease[end].push_back(s);
      }
    }
  }
  return slots;
}

}  // namespace cusadi
