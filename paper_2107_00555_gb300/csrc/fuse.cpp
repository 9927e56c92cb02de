// Planning passes over the SSA graph (Sec. 3.1 auto-optimisation):
//  * map fusion -- greedy merging of elementwise maps that share an iteration
//    space into one expression DAG evaluated in registers (Sec. 3.1, "greedy
//    subgraph fusion": fuse the largest contiguous subgraphs over the same
//    iteration space, checking that what a map consumes is a subset of what
//    the fused scope produces);
//  * subgraph fusion -- reductions become epilogues of the kernel that
//    produces their operand (tiled write-conflict resolution, Sec. 3.1);
//    an axis reduction takes the elementwise maps producing its operand as
//    the prologue of its own kernel, and reductions along the same axis of
//    that prologue share the kernel;
//    elementwise maps feeding a stencil become its prologue, evaluated at
//    every cell the stencil tile reads; unary maps after a stencil step
//    become that step's epilogue; maps after the last step become a post
//    stage; consecutive stencils with the same neighbourhood chain into one
//    group that can be time tiled;
//  * transient mitigation -- a value gets a device buffer only if it is a
//    program output or is read by another kernel (Sec. 3.1: temporaries are
//    persistent and fused-away temporaries are never allocated);
//  * batching -- independent stencil groups running the same step program
//    on different shapes are packed into one launch (the side-by-side
//    connected components of Sec. 2.4 state fusion).
#include <algorithm>
#include <cmath>
#include <map>
#include <set>
#include <sstream>

#include "dcp_internal.h"

namespace dcp {

namespace {

struct Planner {
  GraphImpl& g;
  uint32_t flags;
  std::vector<std::vector<int>> users;
  std::vector<char> live, is_out;
  std::map<int, int> axis_map;  // map planned into an axis-reduce group before its turn

  std::vector<Group>& batch_store;
  Planner(GraphImpl& gi, uint32_t f) : g(gi), flags(f), batch_store(gi.batch_store) {}

  bool fmaps() const { return flags & DCP_FUSE_MAPS; }
  bool fsub() const { return flags & DCP_FUSE_SUBGRAPH; }

  int live_users(int v) const {
    int c = 0;
    for (int u : users[v])
      if (live[u]) ++c;
    return c;
  }

  bool in_vec(const std::vector<int>& a, int v) const {
    return std::find(a.begin(), a.end(), v) != a.end();
  }

  // Is `v` computed in registers by group `gi` (member, stencil output, post)?
  bool computed_in(int gi, int v) const {
    const Group& G = g.groups[gi];
    if (G.kind == GroupKind::Map || G.kind == GroupKind::AxisReduce) return in_vec(G.members, v);
    if (G.kind == GroupKind::Stencil) return v == G.st_out || in_vec(G.post, v);
    if (G.kind == GroupKind::AdjTile) return v == G.st_out;
    return false;
  }

  // Value available in memory before group gi runs (an input, or produced by
  // an earlier group).
  bool available_before(int v, int gi) const {
    int pg = g.value_group[v];
    return pg < 0 || pg < gi;
  }

  void add_operand(Group& G, int gi, int a) {
    if (computed_in(gi, a)) return;
    const Node& n = g.nodes[a];
    bool scalar = n.shape.empty() && !G.shape.empty();
    std::vector<int>& dst = scalar ? G.scalars : (G.kind == GroupKind::Stencil ? G.post_loads : G.loads);
    if (!in_vec(dst, a)) dst.push_back(a);
  }

  void plan() {
    const int N = (int)g.nodes.size();
    users.assign(N, {});
    for (int v = 0; v < N; ++v)
      for (int a : g.nodes[v].in) users[a].push_back(v);
    is_out.assign(N, 0);
    for (int o : g.outputs) is_out[o] = 1;
    // liveness: everything an output depends on
    live.assign(N, 0);
    std::vector<int> stack(g.outputs.begin(), g.outputs.end());
    while (!stack.empty()) {
      int v = stack.back();
      stack.pop_back();
      if (live[v]) continue;
      live[v] = 1;
      for (int a : g.nodes[v].in) stack.push_back(a);
    }
    g.groups.clear();
    g.value_group.assign(N, -1);

    for (int v = 0; v < N; ++v) {
      if (!live[v]) continue;
      const Node& n = g.nodes[v];
      switch (n.kind) {
        case Kind::Input: break;
        case Kind::Map: plan_map(v); break;
        case Kind::Reduce: plan_reduce(v); break;
        case Kind::Stencil: plan_stencil(v); break;
        case Kind::AdjChain: plan_adj(v); break;
      }
    }
    if (flags & DCP_BATCH) plan_batch();
    finalize();
  }

  // What an axis-reduce group will hold once the rest of its prologue has
  // been planned: room other reductions over the same space must leave.
  struct AxisDue {
    std::set<int> maps, reds, loads, scalars;
  };
  std::map<int, AxisDue> axis_due;

  // The maps reached from those of map group M (group gi) that may join the
  // prologue of reductions along `axis` of the group that will replace it:
  // same space, read only by such maps or by reductions along that axis,
  // every operand computed there or before.
  bool axis_closure(const Group& M, int gi, int axis, AxisDue& due) const {
    const std::set<int> own(M.members.begin(), M.members.end());
    std::vector<int> todo = M.members;
    while (!todo.empty()) {
      const int m = todo.back();
      todo.pop_back();
      if (is_out[m] || g.nodes[m].kind != Kind::Map) return false;
      for (int u : users[m]) {
        if (!live[u] || own.count(u) || due.maps.count(u)) continue;
        const Node& un = g.nodes[u];
        if (un.kind == Kind::Reduce && un.axis == axis) {
          due.reds.insert(u);
          continue;
        }
        if (un.kind != Kind::Map || un.shape != M.shape) return false;
        due.maps.insert(u);
        todo.push_back(u);
      }
    }
    due.loads.insert(M.loads.begin(), M.loads.end());
    due.scalars.insert(M.scalars.begin(), M.scalars.end());
    for (int u : due.maps)
      for (int b : g.nodes[u].in) {
        if (own.count(b) || due.maps.count(b)) continue;
        if (g.nodes[b].kind != Kind::Input && !(g.value_group[b] >= 0 && g.value_group[b] < gi)) return false;
        (g.nodes[b].shape.empty() ? due.scalars : due.loads).insert(b);
      }
    return true;
  }

  void plan_map(int v) {
    const Node& n = g.nodes[v];
    auto planned = axis_map.find(v);
    if (planned != axis_map.end()) {  // fused into an axis reduction's prologue
      Group& G = g.groups[planned->second];
      G.members.push_back(v);
      g.value_group[v] = planned->second;
      for (int a : n.in) add_operand(G, planned->second, a);
      return;
    }
    // (1) stencil step epilogue: a unary / immediate map of a stencil group's
    //     current output, which nothing else reads.
    if (fsub() && (op_is_unary(n.op) || op_is_scalar_imm(n.op))) {
      int a = n.in[0];
      int gi = g.value_group[a];
      if (gi >= 0 && gi == (int)g.groups.size() - 1) {
        Group& G = g.groups[gi];
        if (G.kind == GroupKind::Stencil && G.st_out == a && G.post.empty() && G.reds.empty() &&
            !is_out[a] && live_users(a) == 1 && !G.steps.empty()) {
          G.steps.back().epi.push_back(v);
          G.st_out = v;
          g.value_group[v] = gi;
          return;
        }
      }
    }
    // (2) join a group that computes one of the operands.
    int best = -1;
    if (fmaps() || fsub()) {
      for (int a : n.in) {
        int gi = g.value_group[a];
        if (gi < 0 || !computed_in(gi, a)) continue;
        const Group& G = g.groups[gi];
        if (G.shape != n.shape) continue;
        if (G.kind == GroupKind::Map && !fmaps()) continue;
        if (G.kind == GroupKind::Stencil && !fsub()) continue;
        if (G.kind == GroupKind::Batch || G.kind == GroupKind::AxisReduce ||
            G.kind == GroupKind::AdjTile)
          continue;
        bool ok = true;
        for (int b : n.in)
          if (!computed_in(gi, b) && !available_before(b, gi)) ok = false;
        if (ok && gi > best) best = gi;
      }
    }
    // (3) no producer group qualifies (e.g. every operand is a program input):
    //     extend the contiguous subgraph, i.e. join the latest group if it is
    //     a map group over the same iteration space.
    if (best < 0 && fmaps() && !n.shape.empty() && !g.groups.empty()) {
      int gi = (int)g.groups.size() - 1;
      const Group& G = g.groups[gi];
      if (G.kind == GroupKind::Map && G.shape == n.shape) {
        bool ok = true;
        for (int b : n.in)
          if (!computed_in(gi, b) && !available_before(b, gi)) ok = false;
        if (ok) best = gi;
      }
    }
    if (best >= 0) {
      Group& G = g.groups[best];
      if (G.kind == GroupKind::Map) G.members.push_back(v);
      else G.post.push_back(v);
      g.value_group[v] = best;
      for (int a : n.in) add_operand(G, best, a);
      return;
    }
    Group G;
    G.kind = GroupKind::Map;
    G.dtype = n.dtype;
    G.shape = n.shape;
    G.members.push_back(v);
    g.groups.push_back(G);
    int gi = (int)g.groups.size() - 1;
    g.value_group[v] = gi;
    for (int a : n.in) add_operand(g.groups[gi], gi, a);
  }

  // Axis reduction (tiled write-conflict resolution with one partial per
  // remaining index): joins the axis-reduce group computing its operand, or
  // the latest one over the same space and axis; otherwise starts a group
  // that takes the producer map group as its prologue when every value of
  // that group is consumed inside it or by reductions along the same axis.
  void plan_axis_reduce(int v) {
    const Node& n = g.nodes[v];
    int a = n.in[0];
    const Node& an = g.nodes[a];
    auto same_space = [&](const Group& G) {
      return G.kind == GroupKind::AxisReduce && G.shape == an.shape && G.axis == n.axis &&
             G.dtype == an.dtype;
    };
    int gi = g.value_group[a];
    if (gi >= 0 && g.groups[gi].kind == GroupKind::AxisReduce && computed_in(gi, a)) {
      Group& G = g.groups[gi];
      if (!same_space(G) || (int)G.reds.size() >= kMaxIO)
        fail(DCP_E_UNSUPPORTED, "too many reductions of one fused prologue");
      G.reds.push_back(v);
      g.value_group[v] = gi;
      return;
    }
    if (fsub() && !g.groups.empty()) {
      int li = (int)g.groups.size() - 1;
      Group& G = g.groups[li];
      if (same_space(G) && available_before(a, li) && axis_room(G, li, a)) {
        G.reds.push_back(v);
        g.value_group[v] = li;
        add_operand(G, li, a);
        return;
      }
    }
    Group R;
    R.kind = GroupKind::AxisReduce;
    R.dtype = an.dtype;
    R.shape = an.shape;
    R.axis = n.axis;
    bool absorbed = false;
    AxisDue due;
    if (fsub() && gi >= 0 && gi == (int)g.groups.size() - 1 &&
        g.groups[gi].kind == GroupKind::Map && computed_in(gi, a)) {
      const Group& M = g.groups[gi];
      bool ok = M.reds.empty() && M.shape == an.shape && axis_closure(M, gi, n.axis, due);
      // binary64 maps with tanh, exp, sin and the like are bound by the FP64
      // pipe, which the map kernel keeps busier than a row tree: maps still to
      // come then stay in its one pass (sum of x^4 and maximum of tanh(x^4): the
      // columns of 8063 x 140 53 us against 70 in one kernel, of 500 x 500 33
      // against 66; of sin(x^4): 70 against 107 and 39 against 103)
      double cost = 0;
      for (int m : M.members) cost += op_cycles(g.nodes[m].op, an.dtype);
      for (int m : due.maps) cost += op_cycles(g.nodes[m].op, an.dtype);
      if (!due.maps.empty() && !fmaps()) ok = false;  // (maps are not to be fused with one another)
      if (an.dtype == DCP_F64 && !due.maps.empty() && cost >= 8 * op_cycles(DCP_ADD, DCP_F64)) ok = false;
      if (ok && (int)due.loads.size() <= kMaxIO && (int)due.scalars.size() <= kMaxIO &&
          (int)due.reds.size() <= kMaxIO) {
        R.members = M.members;
        R.loads = M.loads;
        R.scalars = M.scalars;
        g.groups.pop_back();
        absorbed = true;
      }
    }
    if (!absorbed) R.loads.push_back(a);
    R.reds.push_back(v);
    g.groups.push_back(R);
    int ri = (int)g.groups.size() - 1;
    g.value_group[v] = ri;
    for (int m : R.members) g.value_group[m] = ri;
    if (absorbed) {
      for (int u : due.maps) axis_map[u] = ri;
      axis_due[ri] = due;
    }
  }

  // Can axis-reduce group gi take another reduction, of value a, beside those
  // its own prologue still brings?
  bool axis_room(const Group& G, int gi, int a) const {
    std::set<int> reds(G.reds.begin(), G.reds.end()), loads(G.loads.begin(), G.loads.end());
    auto due = axis_due.find(gi);
    if (due != axis_due.end()) {
      reds.insert(due->second.reds.begin(), due->second.reds.end());
      loads.insert(due->second.loads.begin(), due->second.loads.end());
    }
    if (!computed_in(gi, a)) loads.insert(a);
    return (int)reds.size() < kMaxIO && (int)loads.size() <= kMaxIO;
  }

  void plan_reduce(int v) {
    const Node& n = g.nodes[v];
    if (n.axis >= 0) {
      plan_axis_reduce(v);
      return;
    }
    int a = n.in[0];
    int gi = g.value_group[a];
    if (fsub() && gi >= 0 && computed_in(gi, a) && g.groups[gi].kind != GroupKind::Batch &&
        g.groups[gi].kind != GroupKind::AxisReduce && g.groups[gi].kind != GroupKind::AdjTile &&
        (int)g.groups[gi].reds.size() < kMaxIO) {
      g.groups[gi].reds.push_back(v);
      g.value_group[v] = gi;
      return;
    }
    Group G;
    G.kind = GroupKind::Map;
    G.dtype = g.nodes[a].dtype;
    G.shape = g.nodes[a].shape;
    G.loads.push_back(a);
    G.reds.push_back(v);
    g.groups.push_back(G);
    g.value_group[v] = (int)g.groups.size() - 1;
  }

  static std::vector<int32_t> pad_offsets(const Node& n) {
    std::vector<int32_t> o;
    int nd = n.ndim();
    for (int k = 0; k < n.npts(); ++k)
      for (int d = 0; d < 3; ++d) {
        int src = d - (3 - nd);
        o.push_back(src >= 0 ? n.offsets[k * nd + src] : 0);
      }
    return o;
  }

  void plan_stencil(int v) {
    const Node& n = g.nodes[v];
    int a = n.in[0];
    if (n.steps == 0) {  // identity: a copy kernel
      Group G;
      G.kind = GroupKind::Map;
      G.dtype = n.dtype;
      G.shape = n.shape;
      G.members.push_back(v);
      G.loads.push_back(a);
      g.groups.push_back(G);
      g.value_group[v] = (int)g.groups.size() - 1;
      return;
    }
    std::vector<int32_t> offs = pad_offsets(n);
    int gi = g.value_group[a];
    // stencil -> stencil: extend the chain (time tiling candidate)
    if (fsub() && gi >= 0 && gi == (int)g.groups.size() - 1) {
      Group& G = g.groups[gi];
      if (G.kind == GroupKind::Stencil && G.st_out == a && G.post.empty() && G.reds.empty() &&
          !is_out[a] && live_users(a) == 1 && G.bc == n.bc && G.offsets == offs &&
          G.dtype == n.dtype) {
        for (int t = 0; t < n.steps; ++t) G.steps.push_back(StepDesc{v, {}});
        G.st_out = v;
        g.value_group[v] = gi;
        return;
      }
    }
    Group S;
    S.kind = GroupKind::Stencil;
    S.dtype = n.dtype;
    S.shape = n.shape;
    S.bc = n.bc;
    S.offsets = offs;
    for (int d = 0; d < 3; ++d) {
      int r = 0;
      for (int k = 0; k < n.npts(); ++k) r = std::max(r, std::abs(offs[k * 3 + d]));
      S.radius[d] = r;
    }
    // map -> stencil prologue: the producer map group is the latest group, has
    // no reductions, and none of its values is read outside this stencil.
    if (fsub() && gi >= 0 && gi == (int)g.groups.size() - 1 &&
        g.groups[gi].kind == GroupKind::Map && computed_in(gi, a)) {
      Group& M = g.groups[gi];
      bool ok = M.reds.empty() && M.shape == n.shape;
      for (int m : M.members) {
        if (is_out[m]) ok = false;
        for (int u : users[m])
          if (live[u] && u != v && !in_vec(M.members, u)) ok = false;
        if (g.nodes[m].kind != Kind::Map) ok = false;
      }
      if (ok) {
        S.members = M.members;
        S.loads = M.loads;
        S.scalars = M.scalars;
        g.groups.pop_back();
      }
    }
    S.st_in = a;
    for (int t = 0; t < n.steps; ++t) S.steps.push_back(StepDesc{v, {}});
    S.st_out = v;
    g.groups.push_back(S);
    int si = (int)g.groups.size() - 1;
    g.value_group[v] = si;
    for (int m : S.members) g.value_group[m] = si;
  }

  // Reverse of a chunk of a stencil chain (built by the adjoint): one group
  // reading u_t and the cotangent of u_{t+k} from memory, storing the
  // cotangent of u_t.
  void plan_adj(int v) {
    const Node& n = g.nodes[v];
    Group A;
    A.kind = GroupKind::AdjTile;
    A.dtype = n.dtype;
    A.shape = n.shape;
    A.bc = n.bc;
    A.offsets = pad_offsets(n);
    for (int d = 0; d < 3; ++d) {
      int r = 0;
      for (int k = 0; k < n.npts(); ++k) r = std::max(r, std::abs(A.offsets[k * 3 + d]));
      A.radius[d] = r;
    }
    A.loads = {n.in[0], n.in[1]};
    A.st_in = n.in[0];
    A.st_out = v;
    A.depth = (int)n.chain.size();
    A.members.push_back(v);
    g.groups.push_back(A);
    g.value_group[v] = (int)g.groups.size() - 1;
  }

  // Pack independent stencil groups that run one step program into batches.
  void plan_batch() {
    std::map<std::string, std::vector<int>> classes;
    for (int gi = 0; gi < (int)g.groups.size(); ++gi) {
      Group& G = g.groups[gi];
      if (G.kind != GroupKind::Stencil || !G.members.empty() || !G.post.empty() ||
          !G.reds.empty() || G.shape.size() != 2)
        continue;
      if (!is_out[G.st_out] || live_users(G.st_out) != 0) continue;
      if (g.value_group[G.st_in] >= 0) continue;  // batch members read program inputs
      std::ostringstream key;
      key.precision(17);
      key << G.dtype << "|" << G.bc << "|";
      for (auto o : G.offsets) key << o << ",";
      for (const StepDesc& s : G.steps) {
        key << "[";
        for (double w : g.nodes[s.node].weights) key << w << ",";
        for (int e : s.epi) key << g.nodes[e].op << ":" << g.nodes[e].imm << ",";
        key << "]";
      }
      classes[key.str()].push_back(gi);
    }
    for (auto& kv : classes) {
      if (kv.second.size() < 2) continue;
      Group B = g.groups[kv.second.front()];
      B.kind = GroupKind::Batch;
      B.shape.clear();
      B.batch_members = kv.second;
      for (int gi : kv.second) g.groups[gi].absorbed = true;
      g.groups.push_back(B);
    }
  }

  void finalize() {
    // Drop absorbed groups, keeping execution order; batch groups run where
    // they were appended (after every member's producers).
    std::vector<Group> out;
    std::vector<int> remap(g.groups.size(), -1);
    for (int gi = 0; gi < (int)g.groups.size(); ++gi) {
      if (g.groups[gi].absorbed) continue;
      remap[gi] = (int)out.size();
      out.push_back(g.groups[gi]);
    }
    // store the absorbed groups' descriptions inside the batch for codegen
    std::vector<Group> all = g.groups;
    for (Group& G : out)
      if (G.kind == GroupKind::Batch) {
        std::vector<int> members = G.batch_members;
        G.batch_members.clear();
        for (int m : members) {
          G.batch_members.push_back((int)batch_store.size());
          batch_store.push_back(all[m]);
        }
      }
    g.groups = out;
    const int N = (int)g.nodes.size();
    for (int v = 0; v < N; ++v)
      if (g.value_group[v] >= 0) g.value_group[v] = remap[g.value_group[v]];
    // batch: member values belong to the batch group
    for (int gi = 0; gi < (int)g.groups.size(); ++gi)
      if (g.groups[gi].kind == GroupKind::Batch)
        for (int m : g.groups[gi].batch_members) {
          const Group& M = batch_store[m];
          g.value_group[M.st_out] = gi;
          for (const StepDesc& s : M.steps) {
            g.value_group[s.node] = gi;
            for (int e : s.epi) g.value_group[e] = gi;
          }
        }

    // Materialisation: a value computed by group G is stored when it is an
    // output or read by a live node outside G.
    g.materialized.assign(N, 0);
    for (int v = 0; v < N; ++v)
      if (g.nodes[v].kind == Kind::Input) g.materialized[v] = 1;
    for (int gi = 0; gi < (int)g.groups.size(); ++gi) {
      Group& G = g.groups[gi];
      G.stores.clear();
      std::vector<int> cand;
      if (G.kind == GroupKind::Map) cand = G.members;
      if (G.kind == GroupKind::Stencil) {
        cand.push_back(G.st_out);
        cand.insert(cand.end(), G.post.begin(), G.post.end());
      }
      if (G.kind == GroupKind::AdjTile) cand.push_back(G.st_out);
      for (int v : cand) {
        bool need = is_out[v];
        for (int u : users[v])
          if (live[u] && g.value_group[u] != gi) need = true;
        // in a stencil group, the stencil output feeds post members in registers
        if (need) {
          G.stores.push_back(v);
          g.materialized[v] = 1;
        }
      }
      for (int r : G.reds) g.materialized[r] = 1;
      if (G.kind == GroupKind::Batch) {
        for (int m : G.batch_members) g.materialized[batch_store[m].st_out] = 1;
      }
      if ((int)G.loads.size() > kMaxIO || (int)G.post_loads.size() > kMaxIO ||
          (int)G.stores.size() > kMaxIO || (int)G.scalars.size() > kMaxIO)
        fail(DCP_E_UNSUPPORTED, "a fused group exceeds 16 loads/stores; split the program");
    }
    // Launch shapes
    int nl = 0;
    for (Group& G : g.groups) {
      if (G.kind == GroupKind::Map) {
        G.threads = 256;
        G.blocks_per_sm = (int)opt(DCP_OPT_MAP_BLOCKS_PER_SM, 8);
        G.unroll = (int)opt(DCP_OPT_MAP_UNROLL, 2);
        nl += 1;
      } else if (G.kind == GroupKind::AxisReduce) {
        G.threads = 256;
        nl += 1;
      } else if (G.kind == GroupKind::AdjTile) {
        // output tile; the halo is 2 k r (the forward k steps grow the
        // region the reverse k steps consume)
        const bool one_d = G.shape.size() == 1;
        G.tile[0] = 1;
        G.tile[1] = one_d ? 1 : (int)opt(DCP_OPT_TILE_Y, G.dtype == DCP_F32 ? 32 : 16);
        G.tile[2] = (int)opt(DCP_OPT_TILE_X, one_d ? 512 : 32);
        G.threads = 256;
        nl += 1;
      } else {
        choose_stencil_tiling(G);
        int S = (int)G.steps.size();
        nl += (S + G.depth - 1) / G.depth;
      }
    }
    g.n_launches = nl;
  }

  int64_t opt(int key, int64_t def) const {
    auto it = g.options.find(key);
    return it == g.options.end() ? def : it->second;
  }

  // The planner runs without a GPU: a GB300's SMs and their warp schedulers.
  static constexpr int64_t kSMs = 152, kSchedulers = 4 * kSMs;

  // Issue cycles of one operation on the C columns a lane holds (binary64
  // operations cost the FP64 pipe 64 cycles per warp and scheduler).
  double op_cycles(int op, int dtype) const {
    if (dtype == DCP_F64) {
      const double n = op == DCP_EXP || op == DCP_SQRT || op == DCP_DIV ? 10
                       : op == DCP_SIN || op == DCP_COS                ? 15
                       : op == DCP_TANH                                ? 7 : 1;
      return 2 * 64 * n;
    }
    const double n = op == DCP_EXP || op == DCP_SQRT || op == DCP_DIV ? 10
                     : op == DCP_SIN || op == DCP_COS || op == DCP_TANH ? 25 : 1;
    return 4 * n;
  }

  // FP64 operations per cell of a 2-D step: a run on its deferred weight
  // shares the pairs of a 5-point star (two operations fewer).
  double step_ops64(const Group& G) const {
    const int pts = (int)G.offsets.size() / 3;
    const Node& n = g.nodes[G.steps[0].node];
    auto opt_on = g.options.find(DCP_OPT_DEFERRED_WEIGHT);
    const bool run = G.steps.size() > 1 && G.steps[0].epi.empty() && defer_chunk_steps(n) > 0 &&
                     (opt_on == g.options.end() || opt_on->second != 0);
    return run ? std::max(1, pts == 5 ? pts - 2 : pts - 1) : pts;
  }

  // Input arrays of a stencil group, and issue cycles of its prologue per row
  // of a warp (binary64: a product and the add that takes it are one
  // instruction, 0.6 per map).
  int64_t arrays_in(const Group& G) const {
    return G.members.empty() ? 1 : std::max<int64_t>(1, (int64_t)G.loads.size());
  }
  double pro_cycles(const Group& G) const {
    double c = 0;
    for (int m : G.members) c += op_cycles(g.nodes[m].op, G.dtype);
    return G.dtype == DCP_F64 ? 0.6 * c : c;
  }
  // Issue cycles of a step's epilogue maps, averaged over the steps.
  double epi_cycles(const Group& G) const {
    double c = 0;
    for (const StepDesc& st : G.steps)
      for (int e : st.epi) c += op_cycles(g.nodes[e].op, G.dtype);
    return c / (double)G.steps.size();
  }

  // Cycles of one launch of K steps of the warp-stream kernel, and the rows
  // per work item that give them: nw warps per scheduler (4 per SM) stream
  // seg + 2 K ry rows each, a row taking the larger of its latency and the
  // nw warps' issue.  Fitted to 24 steps on 64^2 .. 4000 x 4100 binary32 and
  // 64^2 .. 2047 x 2051 binary64 grids (within 15 %): binary32 issues 27
  // cycles per level and 42 per row with a latency of 45 per level and 130
  // per row; binary64 is bound by the FP64 pipe (p operations on 2 columns),
  // with a latency of 500 per level and 300 per row.
  // With `pro` the launch evaluates the group's prologue; ctas: CTAs of it.
  double stream_cycles(const Group& G, int K, bool pro, int64_t& seg, int& nw, int64_t& ctas) const {
    const int64_t ny = G.shape.size() == 2 ? G.shape[0] : 1, nx = G.shape.back();
    const int ry = G.shape.size() == 2 ? G.radius[1] : 0;
    const int W = stream_width(G, K);
    const int64_t strips = (nx + W - 1) / W;
    const int pts = (int)G.offsets.size() / 3;
    double issue, latency;
    if (G.dtype == DCP_F64) {
      issue = K * 2.0 * 64 * step_ops64(G) + 60;
      latency = 300.0 + 500.0 * K;
    } else {
      issue = K * (7.0 + 4.0 * pts) + 42;
      latency = 130.0 + 45.0 * K;
    }
    issue += K * epi_cycles(G);
    const int64_t inputs = pro ? arrays_in(G) : 1;
    if (pro) issue += pro_cycles(G);
    const int64_t cells = ny * nx;
    const double bytes = 2.0 * cells * dtype_size(G.dtype);
    // 3237 bytes per clock from HBM (6.7 TB/s at 2.07 GHz), about twice that
    // where both arrays stay in L2
    const double mem = bytes / (bytes > 100e6 ? 3237.0 : 6500.0);
    double best = 1e300;
    const int64_t slots = kSchedulers;
    // the rows in flight of every input take shared memory (227 KB per SM)
    const int64_t resident = kSMs * std::max<int64_t>(1, 227 * 1024 / (inputs * 8 * 512));
    for (int n = 1; n <= 4 && (n == 1 || n * slots <= resident); ++n) {
      const int64_t segs = std::max<int64_t>(1, std::min<int64_t>(ny, std::min(n * slots, resident) / strips));
      const int64_t sg = (ny + segs - 1) / segs;
      const int64_t items = strips * ((ny + sg - 1) / sg);
      const int64_t per = (items + slots - 1) / slots;  // warps one scheduler runs
      const int64_t waves = (per + n - 1) / n;
      // the share of its time a scheduler's FP64 pipe is busy with nn warps
      const int nn = (int)std::min<int64_t>(per, n);
      const double busy = G.dtype == DCP_F64 ? (nn == 1 ? 0.7 : 0.85) : 1.0;
      const double c = std::max(mem, (double)waves * (sg + 2 * K * ry) * std::max(latency, issue * nn / busy));
      if (c < best * 0.999) best = c, seg = sg, nw = n, ctas = items;
    }
    return best;
  }

  // Cycles the tickets of a launch's CTAs take where it reduces: about 7 ns
  // each, those of the first few hundred beside the other CTAs' work.
  double ticket_cycles(const Group& G, int64_t ctas) const {
    return G.reds.empty() ? 0 : 14.0 * std::max<int64_t>(0, ctas - 512);
  }

  // Cycles of one batched launch of K steps with seg rows per work item: the
  // issue of every item's rows over the GPU's schedulers plus half an item's
  // time for the uneven end, at least one item's latency.  (4096 binary32
  // instances of 32^2 to 512^2, 20 steps at 5 per launch: 32, 64, 128 and 256
  // rows took 2.51, 2.23, 2.18 and 2.24 ms.)
  double batch_cycles(const Group& G, int K, int seg) const {
    const int W = stream_width(G, K), ry = G.radius[1];
    const int pts = (int)G.offsets.size() / 3;
    const bool f64 = G.dtype == DCP_F64;
    double epi = 0;
    for (const StepDesc& st : G.steps)
      for (int e : st.epi) epi += op_cycles(g.nodes[e].op, G.dtype);
    const double issue = (f64 ? (K * 2.0 * 64 * step_ops64(G) + 60) / 0.9 : K * (11.0 + 4.0 * pts) + 100) +
                         K * epi / (double)G.steps.size();
    const double latency = f64 ? 300.0 + 500.0 * K : 130.0 + 45.0 * K;
    double rows = 0, bytes = 0;
    int64_t items = 0, longest = 1;
    for (int m : G.batch_members) {
      const Group& M = batch_store[m];
      const int64_t ny = M.shape[0], nx = M.shape[1];
      if (ny * nx == 0) continue;
      const int64_t strips = (nx + W - 1) / W, segs = (ny + seg - 1) / seg;
      rows += (double)strips * (ny + segs * 2 * K * ry);
      items += strips * segs;
      longest = std::max(longest, std::min<int64_t>(ny, seg) + 2 * K * ry);
      bytes += 2.0 * ny * nx * dtype_size(G.dtype);
    }
    // (binary64: the other warps of the scheduler keep its FP64 pipe busy)
    const double n = f64 ? 1.0 : std::min(4.0, items / (double)kSchedulers);
    const double c = std::max(rows * issue / kSchedulers + 0.5 * longest * std::max(latency, n * issue),
                              longest * latency);
    return std::max(c, bytes / (bytes > 100e6 ? 3237.0 : 6500.0));
  }

  // Cycles of one launch of K steps of the shared-memory tile kernel (256
  // threads per CTA) on `tiles` tiles.  Binary32: about 290 cycles per step and
  // 256 cells of the region, two CTAs per SM in parallel (fitted to 24 steps
  // on 64^2 .. 512^2).  Binary64: per tile 350 cycles and the operations of
  // its regions at 2 per clock, 0.7 operations per cell more than the sum's and
  // 5 % over, and per step 1000 cycles of latency, 1200 where the SM has no
  // other tile (within 10 %: 5-, 9- and 13-point steps of radius 1 and 2, one
  // and two per launch, with prologues of 3, 8 and 14 arrays, on 500 x 513 ..
  // 3000 x 3100; 5 and 10 steps on 256^2 .. 512^2).
  double tile_cycles(const Group& G, int K, int ty, int tx, int64_t tiles, bool pro = false) const {
    const int64_t per = (tiles + kSMs - 1) / kSMs;  // tiles of one SM
    const int pts = (int)G.offsets.size() / 3;
    const int ry = G.radius[1], rx = G.radius[2];
    const bool f64 = G.dtype == DCP_F64;
    const double epi = epi_cycles(G), parallel = std::max(1.0, per / 2.0);
    const double ops = f64 ? std::min(pts, (int)step_ops64(G) + 1) + 0.7 + epi / 128 : 0;
    double t = 0;
    for (int s = 0; s < K; ++s) {
      const double cells = (double)(ty + 2 * (K - 1 - s) * ry) * (tx + 2 * (K - 1 - s) * rx);
      if (f64) t += (per == 1 ? 1200 : 1000) + per * cells * 1.05 * ops / 2;
      else t += parallel * (290.0 * pts / 5 + 0.6 * epi) * std::ceil(cells / 256);
    }
    if (f64) t += per * 350;
    if (pro && f64) t += per * (double)(ty + 2 * K * ry) * (tx + 2 * K * rx) * pro_cycles(G) / 128 / 2;
    return t;
  }
  int64_t tiles_of(const std::vector<int64_t>& shape, int ty, int tx) const {
    return ((shape[0] + ty - 1) / ty) * ((shape[1] + tx - 1) / tx);
  }

  // 3-D stars without a prologue run as warp-streamed columns where those are
  // faster, unless a tile option asks for the shared-memory planes: binary64
  // one step per launch, binary32 two.  A warp (nw per scheduler) streams seg + 2 K planes, one
  // plane costing the larger of its latency and the issue (binary32, fitted: 870
  // cycles for two steps of four rows) or FP64 pipe time (64 cycles per
  // operation of the warp) of the scheduler's warps.
  void choose_columns(Group& G) {
    G.variant = 0;
    const auto has = [&](int key) { return g.options.count(key) > 0; };
    if (!column_eligible(g, G) || has(DCP_OPT_TILE_X) || has(DCP_OPT_TILE_Y) || has(DCP_OPT_TILE_Z) ||
        has(DCP_OPT_CELLS_PER_THREAD) || G.shape[0] * G.shape[1] * G.shape[2] == 0)
      return;
    const bool f64 = G.dtype == DCP_F64;
    const int S = (int)G.steps.size();
    int kmax = f64 || !(flags & DCP_TIME_TILE) ? 1 : 2;
    kmax = std::min<int64_t>({kmax, S, std::max<int64_t>(1, opt(DCP_OPT_TIME_TILE_DEPTH, 2))});
    const int64_t nz = G.shape[0], ny = G.shape[1], nx = G.shape[2];
    double epi = 0;
    for (const StepDesc& st : G.steps)
      for (int e : st.epi) epi += op_cycles(g.nodes[e].op, G.dtype);
    epi /= S;
    const int pts = (int)G.offsets.size() / 3;
    const double bytes = 2.0 * nz * ny * nx * dtype_size(G.dtype);
    const double mem = bytes / (bytes > 100e6 ? 3237.0 : 6500.0);
    // measured over the counted cycles (512^3, 256^3, 300 x 333 x 381)
    const double busy = G.bc == DCP_BC_PERIODIC ? 1.15 : 1.09;
    int bcy = 4, blx = 32;
    int64_t bseg = 1;
    // the shared-memory planes: whole tiles of 8 x 32 cells, one operation more
    // (binary32: 63 instructions per cell, 3.84e-3 cycles of the whole GPU)
    const double padded = (double)nz * ((ny + 7) / 8 * 8) * ((nx + 31) / 32 * 32);
    double best =
        0.95 * S *
            ((f64 ? std::max(mem, 1.12 * padded * (pts - 1 + epi / 128) / (2 * kSMs) + 3000)
                 : std::max(mem, 3.84e-3 * padded * (0.6 + 0.4 * pts / 7 + epi / 252) + 5000)) + 6200) +
           (f64 ? 0 : ticket_cycles(G, (nz + 15) / 16 * ((ny + 7) / 8) * ((nx + 31) / 32)));
    const int lx0 = G.lx, cy0 = G.cy;
    const bool odd = nx % 4 != 0;
    bool column = false;
    const int K = kmax;  // (binary32: two steps beat one at every size measured)
    for (int lx : {32, 16})
      for (int cy : {8, 4, 2}) {
        if (!f64 && (cy == 8 || lx != 32)) continue;
        G.lx = lx;
        const int rows_w = 32 / lx * cy;  // rows per warp
        if (rows_w > 2 && rows_w / 2 >= ny) continue;
        const int64_t strips = (nx + column_width(G, K) - 1) / column_width(G, K);
        const int64_t blocks = (ny + rows_w - 1) / rows_w;
        const double rows = K == 1 ? cy : 2 * cy + 2;  // rows summed per plane, all levels
        const double issue = f64 ? cy * (2 * 64 * (pts - 3 + (cy + 1.0) / cy) + epi) + 100
                                 : rows * (52 + 4.0 * pts + epi) + 70 + (odd ? (cy + 2 * K) * 25 : 0);
        const double latency = f64 ? 1500 : 900 + 700.0 * K;
        const double ends = f64 ? 0.5 : 2.0 * K;  // planes an item pays for beside its own
        // warps per scheduler: what the registers of the form allow without
        // spills (512^3 binary64, 8 rows per lane: 1.22 ms per step at 2,
        // 1.41 at 3; 300 x 333 x 381 binary32: 59 us at 3, 72 at 4)
        const int nmax = f64 && cy == 8 ? 2 : 3;
        for (int n = 1; n <= nmax; ++n)
          for (int wv = 1; wv <= (n == nmax ? 16 : 1); ++wv) {  // whole waves of the resident warps
            const int64_t segs = (int64_t)wv * n * kSchedulers / (strips * blocks);
            if (segs < 1) continue;
            const int64_t sg = (nz + std::min(segs, nz) - 1) / std::min(segs, nz);
            const int64_t items = strips * blocks * ((nz + sg - 1) / sg);
            const int64_t per = (items + kSchedulers - 1) / kSchedulers;
            const int64_t waves = (per + n - 1) / n;
            // (one warp alone keeps its scheduler's FP64 pipe busy 70 % of the time)
            const int64_t nn = std::min<int64_t>(per, n);
            const double c = (std::max(mem, waves * (double)(sg + ends) *
                                                std::max(latency, issue * nn * busy * (f64 && nn == 1 ? 1.3 : 1.0))) +
                              6200) * ((S + K - 1) / K) +
                             (f64 ? 0 : ticket_cycles(G, items / (K * cy < 8 ? 4 : 1)));
            if (c < best * 0.999) best = c, G.depth = K, bcy = cy, blx = lx, bseg = sg, column = true;
            if (segs >= nz) break;
          }
        if (strips * blocks > 16 * nmax * kSchedulers) {  // wide grids: long columns
          const int64_t sg = std::min<int64_t>(nz, 64);
          const double c = ((double)strips * blocks * nz / sg / kSchedulers * (sg + ends) * issue + 6200) * ((S + K - 1) / K);
          if (c < best * 0.999) best = c, G.depth = K, bcy = cy, blx = lx, bseg = sg, column = true;
        }
      }
    G.lx = lx0;
    G.cy = cy0;
    if (!column) return;
    G.cy = bcy;
    G.lx = blx;
    G.seg = (int)bseg;
    G.variant = 3;
    G.threads = 32;
    G.min_ctas = column_min_ctas(G);
  }

  // Kernel form, depth, rows per work item or tile of a 1-D / 2-D stencil
  // group, each unless an option sets it.
  void choose_stencil_tiling(Group& G) {
    choose_stencil_tiling_impl(G);
    const int nd = G.kind == GroupKind::Batch ? 2 : (int)G.shape.size();
    if (nd == 3) {
      choose_columns(G);
      return;
    }
    const auto has = [&](int key) { return g.options.count(key) > 0; };
    const int S = (int)G.steps.size();
    const bool tt = (flags & DCP_TIME_TILE) != 0;
    const bool free_depth = tt && !has(DCP_OPT_TIME_TILE_DEPTH);
    // launches of equal depth: at most `most` steps each
    auto even = [S](int most) {
      const int n = (S + most - 1) / most;
      return (S + n - 1) / n;
    };
    // a launch costs about 3 us (6200 cycles) besides its rows
    const double launch = 6200;
    const int64_t cells = G.kind == GroupKind::Batch ? 0 : G.shape.size() == 2 ? G.shape[0] * G.shape[1] : G.shape[0];
    // the warp-stream kernel when it applies (1-D or 2-D, radius <= 2); the
    // shared-memory tile kernel otherwise
    int var = stream_eligible(G, G.depth) ? 1 : 0;
    auto it = g.options.find(DCP_OPT_STENCIL_KERNEL);
    if (it != g.options.end()) var = (it->second == 1 && stream_eligible(G, G.depth)) ? 1 : 0;
    int64_t seg = 0;
    int nw = 4;
    if (G.kind == GroupKind::Stencil && var == 1 && cells > 0) {
      // (the last launch of an uneven split runs fewer steps; the first alone
      // evaluates a prologue, which binary32 counts in every launch: it then
      // takes deeper ones, 9 steps on the sum of 8 arrays of 3000 x 3100 82 us in
      // one launch against 94 in two)
      auto total = [&](double cycles, double first, int K) {
        return first - cycles + std::max(1.0, (double)S / K) * cycles + launch * ((S + K - 1) / K);
      };
      const int wpc = G.reds.empty() ? 1 : G.dtype == DCP_F32 ? 4 : 2;  // warps per CTA of a launch that reduces
      auto stream_total = [&](int K, int64_t& sg, int& n) {
        int64_t ctas = 0, sg1;
        int n1;
        const bool pro = !G.members.empty();
        const double first = stream_cycles(G, K, pro, sg, n, ctas);
        if (K == S || !pro || G.dtype != DCP_F64) return total(first, first, K) + ticket_cycles(G, ctas / wpc);
        const double rest = stream_cycles(G, K, false, sg1, n1, ctas);
        sg = sg1, n = n1;
        return total(rest, first, K) + ticket_cycles(G, ctas / wpc);
      };
      double best = stream_total(G.depth, seg, nw);
      if (free_depth)
        for (int most = 1; most <= std::min(S, G.dtype == DCP_F32 ? 10 : 4); ++most) {
          const int K = even(most);
          int64_t sg;
          int n;
          if (!stream_eligible(G, K)) continue;
          const double c = stream_total(K, sg, n);
          // (strips of 1-D binary64 arrays: 24 steps of 10^7 elements, fixed ring,
          // 1.50 ms two at a time, 1.55 three, which the model holds equal)
          if (c < best * (stream_exact(G) && K > 2 ? 0.97 : 1.0)) best = c, G.depth = K, seg = sg, nw = n;
        }
      // Small grids run faster in shared-memory tiles, where every cell of a
      // step is in flight at once (256^2 binary64, 24 steps: 46 us against 91;
      // 64^2 binary32: 17 against 25).  From 512^2 on the stream wins, but for
      // prologues of many arrays, whose rings leave few warps (the step of a sum
      // of 8 arrays of 1000 x 1001, periodic: binary32 14 us streamed, 8 in
      // tiles, binary64 45 and 31), and for periodic binary64 grids: a step
      // whose sums share no pairs pays for the strip's halo columns (1000 x
      // 1001, 9 points of radius 2, 7 steps: 191 us streamed, 156 in tiles) and
      // a narrow one for idle lanes.
      const bool small = cells <= 512 * 512, f64 = G.dtype == DCP_F64;
      const bool periodic = G.bc == DCP_BC_PERIODIC;
      const int64_t n_in = arrays_in(G);
      const bool many = f64 ? n_in >= 3
                            : periodic && n_in >= 6 && cells >= 1 << 17 && S <= 4 &&
                                  (S == 1 || cells * S <= 5000000 || (S == 2 && n_in >= 8));
      if (nd == 2 && (small || many || (f64 && periodic)) && !has(DCP_OPT_STENCIL_KERNEL) &&
          !has(DCP_OPT_TILE_X) && !has(DCP_OPT_TILE_Y) && !has(DCP_OPT_STREAM_ROWS)) {
        const bool fixed = !small || (!f64 && many);  // the default tile
        for (int most = 1; most <= std::min(S, fixed ? 4 : 12); ++most) {
          const int K = free_depth ? even(most) : G.depth;
          for (int tx : fixed ? std::vector<int>{f64 ? 32 : 64} : std::vector<int>{16, 32}) {
            std::vector<int> heights = {16, 32};
            if (!fixed) {
              heights = {4, 8, 12, 16, 24, 32};
              // heights that give every SM the same number of tiles, one or two
              // (256 rows in 8 strips: 14, 152 tiles; 16 rows would leave 24 SMs idle)
              const int64_t strips = (G.shape[1] + tx - 1) / tx;
              for (int per : {1, 2})
                if (per * kSMs >= strips) {
                  const int64_t rows = per * kSMs / strips, ty = (G.shape[0] + rows - 1) / rows;
                  if (ty >= 4 && ty <= 32) heights.push_back((int)ty);
                }
            }
            for (int ty : heights) {
              const long smem = 2L * (ty + 2 * K * G.radius[1]) * (tx + 2 * K * G.radius[2]) * dtype_size(G.dtype);
              if (smem > 96 * 1024) continue;
              const int64_t tiles = tiles_of(G.shape, ty, tx);
              const double rest = tile_cycles(G, K, ty, tx, tiles);
              const double first = G.members.empty() ? rest : tile_cycles(G, K, ty, tx, tiles, true);
              const double c = total(rest, first, K) + 0.3 * launch * ((S + K - 1) / K) + ticket_cycles(G, tiles);
              // (on large grids more than two steps only for a gain the model
              // resolves; binary32 takes tiles for a few steps on many inputs
              // whatever the model says, which has no term for the inputs)
              if (c < best * (small || K <= 2 || var == 1 ? 1.0 : 0.97) || (!f64 && many && K == S && ty == 32)) {
                best = c;
                var = 0;
                G.depth = K;
                G.tile[1] = ty;
                G.tile[2] = tx;
              }
            }
          }
          if (!free_depth) break;
        }
      }
    }
    if (G.kind == GroupKind::Batch && var == 1) {
      double best = 1e300;
      const int most0 = free_depth ? 1 : G.depth;
      const int most1 = free_depth ? std::min(S, G.dtype == DCP_F32 ? 8 : 3) : G.depth;
      for (int most = most0; most <= most1; ++most) {
        const int K = free_depth ? even(most) : G.depth;
        if (!stream_eligible(G, K)) continue;
        for (int sg : {16, 32, 64, 128, 256}) {
          const double c = batch_cycles(G, K, sg) * S / K + launch * ((S + K - 1) / K);
          if (c < best) best = c, G.depth = K, seg = sg;
        }
      }
      // small periodic binary64 batches in tiles (64 instances of 32^2 to 64^2,
      // 20 steps: 153 us streamed, 124 in tiles)
      if (G.bc == DCP_BC_PERIODIC && G.dtype == DCP_F64 && !has(DCP_OPT_STENCIL_KERNEL) &&
          !has(DCP_OPT_TILE_X) && !has(DCP_OPT_TILE_Y) && !has(DCP_OPT_STREAM_ROWS))
        for (int most = most0; most <= std::min(most1, 2); ++most) {
          const int K = free_depth ? even(most) : G.depth;
          int64_t tiles = 0;
          for (int m : G.batch_members) tiles += tiles_of(batch_store[m].shape, G.tile[1], G.tile[2]);
          const double c = (tile_cycles(G, K, G.tile[1], G.tile[2], tiles) * S / K + 1.3 * launch * ((S + K - 1) / K));
          if (c < best) best = c, var = 0, G.depth = K;
        }
    }
    if (it != g.options.end() && it->second == 2 && G.kind == GroupKind::Stencil &&
        G.shape.size() <= 2) {
      // cooperative form: every step in one launch on the tile the options
      // (or the defaults) give
      G.depth = (int)G.steps.size();
      if (!coop_eligible(G, G.tile[1], G.tile[2]))
        fail(DCP_E_UNSUPPORTED, "the cooperative stencil form needs at most 63 steps and edge "
                                "tiles at least a radius wide");
      var = 2;
      // one thread per tile cell (64..1024): the tile's cells are independent
      // chains, which a latency-bound small grid needs in flight
      const int cells = (G.shape.size() == 1 ? 1 : G.tile[1]) * G.tile[2];
      G.threads = std::min(1024, std::max(64, (cells + 31) / 32 * 32));
    }
    G.variant = var;
    if (var == 1) {
      // One warp per CTA: work items end at different times, and a CTA's slots
      // free together (batch of 4096 instances 2.28 -> 2.13 ms, 4000 x 4100
      // binary32 16 steps 100 -> 91 us).  Binary64 arrays take two: the few
      // warps an FP64-bound scheduler needs are then spread over all four
      // schedulers (5195 x 5862 plain steps 5.15 -> 4.66 ms).
      G.threads = (int)opt(DCP_OPT_STREAM_THREADS, default_stream_threads(G));
      G.prefetch = (int)opt(DCP_OPT_STREAM_PREFETCH, 1);
      // registers for the four warps per scheduler the plan counts on
      G.min_ctas = (int)opt(DCP_OPT_STREAM_MIN_CTAS, nw >= 4 ? std::min(32, 512 / G.threads) : 0);
      G.seg = (int)std::max<int64_t>(seg, 1);
      auto so = g.options.find(DCP_OPT_STREAM_ROWS);
      if (so != g.options.end()) G.seg = (int)so->second;
    }
  }

  void choose_stencil_tiling_impl(Group& G) {
    int S = (int)G.steps.size();
    bool tt = flags & DCP_TIME_TILE;
    int nd = G.kind == GroupKind::Batch ? 2 : (int)G.shape.size();
    int depth = 1;
    if (tt && nd <= 2) depth = std::min(S, G.dtype == DCP_F32 ? 4 : 2);
    depth = (int)opt(DCP_OPT_TIME_TILE_DEPTH, depth);
    if (nd == 3) depth = 1;  // 3-D kernels stream planes one step at a time
    depth = std::max(1, std::min(depth, S));
    G.depth = depth;
    if (nd == 3) {
      G.tile[0] = (int)opt(DCP_OPT_TILE_Z, 16);  // z chunk
      G.tile[1] = (int)opt(DCP_OPT_TILE_Y, 8);
      G.tile[2] = (int)opt(DCP_OPT_TILE_X, 32);
      // two cells per thread along x (two independent FP64 chains per
      // thread, aligned pair loads) where the tile and radius allow it
      const bool pairs_ok = G.tile[2] % 2 == 0 && G.radius[2] <= 2;
      G.cx = pairs_ok ? (int)opt(DCP_OPT_CELLS_PER_THREAD, 2) : 1;
      G.threads = 256;
    } else {
      G.tile[0] = 1;
      G.tile[1] = (int)opt(DCP_OPT_TILE_Y, 32);
      G.tile[2] = (int)opt(DCP_OPT_TILE_X, G.dtype == DCP_F32 ? 64 : 32);
      G.threads = 256;
    }
  }

};

}  // namespace

bool coop_eligible(const Group& G, int ty, int tx) {
  const int nd = (int)G.shape.size();
  if (G.kind != GroupKind::Stencil || nd > 2 || G.steps.empty() || G.steps.size() > 63) return false;
  const int64_t ny = nd == 2 ? G.shape[0] : 1, nx = G.shape.back();
  if (nd == 1) ty = 1;
  const int ry = nd == 2 ? G.radius[1] : 0, rx = G.radius[2];
  if (ty < std::max(1, ry) || tx < std::max(1, rx) || ny < 1 || nx < 1) return false;
  // the halo must come from the adjacent tiles only
  const int64_t ey = ny % ty, ex = nx % tx;
  if ((ey != 0 && ey < ry) || (ex != 0 && ex < rx)) return false;
  if (ny < ry || nx < rx) return false;
  return true;
}

bool stream_eligible(const Group& G, int depth) {
  const int nd = G.kind == GroupKind::Batch ? 2 : (int)G.shape.size();
  if (nd > 2) return false;
  if (G.radius[1] > 2 || G.radius[2] > 2) return false;
  const int C = stream_cols_per_lane(G.dtype);
  if (G.radius[2] > C) return false;
  return 32 * C - 2 * depth * G.radius[2] >= 8;
}

void plan_graph(GraphImpl& g, uint32_t flags) {
  g.flags = flags;
  g.batch_store.clear();
  Planner p(g, flags);
  p.plan();
}

}  // namespace dcp
