// Code generation (Sec. 3.3: the GPU backend emits CUDA for every fused
// scope): each fused group becomes one hand-written skeleton from kernels/
// specialised with the group's expression DAG, stencil weights, tile shape
// and boundary rule.  The expression is emitted as straight-line code in
// registers; constants are emitted bit-exactly.
#include <algorithm>
#include <cfloat>
#include <cinttypes>
#include <cstdint>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <sstream>

#include "dcp_internal.h"

namespace dcp {

namespace {

// Variable names in generated code are numbered per kernel in order of first
// use, not by graph node id, so that structurally identical groups (e.g. the
// same program on many arrays) generate identical sources and share one
// compiled module.
thread_local std::map<int, int>* t_names = nullptr;

struct NameScope {
  std::map<int, int> names;
  std::map<int, int>* prev;
  NameScope() : prev(t_names) { t_names = &names; }
  ~NameScope() { t_names = prev; }
};

std::string var(int v) {
  if (!t_names) return "v" + std::to_string(v);
  auto it = t_names->find(v);
  int id;
  if (it == t_names->end()) {
    id = (int)t_names->size();
    (*t_names)[v] = id;
  } else {
    id = it->second;
  }
  return "v" + std::to_string(id);
}

std::string imm_literal(int dtype, double imm) {
  char buf[96];
  switch (dtype) {
    case DCP_F32: {
      float f = (float)imm;
      uint32_t b;
      std::memcpy(&b, &f, 4);
      std::snprintf(buf, sizeof buf, "__int_as_float(0x%08" PRIx32 ")", b);
      break;
    }
    case DCP_F64: {
      uint64_t b;
      std::memcpy(&b, &imm, 8);
      std::snprintf(buf, sizeof buf, "__longlong_as_double(0x%016" PRIx64 "ll)", b);
      break;
    }
    case DCP_I32: {
      int64_t i = (int64_t)imm;
      uint32_t b = (uint32_t)(uint64_t)i;
      std::snprintf(buf, sizeof buf, "((int)0x%08" PRIx32 "u)", b);
      break;
    }
    default: {
      int64_t i = (int64_t)imm;
      std::snprintf(buf, sizeof buf, "((long long)0x%016" PRIx64 "ull)", (uint64_t)i);
      break;
    }
  }
  return buf;
}

// Weight literal in the group's dtype (stencils are floating).
std::string weight_literal(int dtype, double w) { return imm_literal(dtype, w); }

// C expression of map op `op` (dtype, immediate) applied to operand
// expressions.
std::string op_expr(int op, int dtype, double imm_v, const std::string& a, const std::string& b) {
  std::string imm = imm_literal(dtype, imm_v);
  switch (op) {
    case kOpBcast: return a;
    case kOpConst: return imm;
    case kOpSign: return "dcp_sign(" + a + ")";
    case kOpGt: return "dcp_gt(" + a + ", " + b + ")";
    case kOpLt: return "dcp_lt(" + a + ", " + b + ")";
    case DCP_NEG: return "dcp_neg(" + a + ")";
    case DCP_ABS: return "dcp_abs(" + a + ")";
    case DCP_EXP: return (dtype == DCP_F64 ? "dcp_exp64(" : "dcp_exp(") + a + ")";
    case DCP_SIN: return (dtype == DCP_F64 ? "dcp_sin64(" : "dcp_sin(") + a + ")";
    case DCP_COS: return (dtype == DCP_F64 ? "dcp_cos64(" : "dcp_cos(") + a + ")";
    case DCP_TANH: return (dtype == DCP_F64 ? "dcp_tanh64(" : "dcp_tanh(") + a + ")";
    case DCP_SQRT: return "dcp_sqrt(" + a + ")";
    case DCP_SQUARE: return "dcp_square(" + a + ")";
    case DCP_ADD: return "dcp_add(" + a + ", " + b + ")";
    case DCP_SUB: return "dcp_sub(" + a + ", " + b + ")";
    case DCP_MUL: return "dcp_mul(" + a + ", " + b + ")";
    case DCP_DIV: return "dcp_div(" + a + ", " + b + ")";
    case DCP_MAX: return "dcp_max(" + a + ", " + b + ")";
    case DCP_MIN: return "dcp_min(" + a + ", " + b + ")";
    case DCP_ADD_S: return "dcp_add(" + a + ", " + imm + ")";
    case DCP_MUL_S: return "dcp_mul(" + a + ", " + imm + ")";
    case DCP_SUB_S: return "dcp_sub(" + a + ", " + imm + ")";
    case DCP_RSUB_S: return "dcp_sub(" + imm + ", " + a + ")";
  }
  fail(DCP_E_INVALID_ARG, "codegen: unknown op");
}

// C expression of map node v applied to operand expressions.
std::string map_expr(const GraphImpl& g, int v, const std::string& a, const std::string& b) {
  const Node& n = g.nodes[v];
  if (n.kind == Kind::Stencil) return a;  // zero-step stencil: identity
  return op_expr(n.op, n.dtype, n.imm, a, b);
}

// Maps inside stencil kernels (prologues, step epilogues, the tiled reverse's
// derivatives) are emitted with explicit rounding: a product that feeds an add
// or a subtraction becomes one fused multiply-add, everything else rounds on
// its own.  Left to the compiler, that choice depends on how a kernel's blocks
// are cut, and the kernel forms of one program would differ in last bits.
struct Ex {
  std::string s;      // the value
  std::string x, y;   // a product: s = (neg ? -1 : 1) x y
  bool neg = false;
  int uses = 1;
  bool mul() const { return !x.empty(); }
};

Ex ex_op(int op, int dtype, double imm_v, const Ex& a, const Ex& b) {
  const std::string imm = imm_literal(dtype, imm_v);
  Ex r;
  auto product = [&](const std::string& x, const std::string& y) {
    r.s = "dcp_mul_rn(" + x + ", " + y + ")";
    r.x = x;
    r.y = y;
  };
  // p + q or p - q.  A product is fused into the sum, except with itself or with
  // another node of the same factors: that difference is 0, not the rounding
  // error of the product.
  auto sum = [&](const Ex& p, const Ex& q, bool minus) {
    auto neg = [](const std::string& v, bool n) { return n ? "dcp_neg(" + v + ")" : v; };
    const bool same = p.s == q.s || (p.mul() && q.mul() && ((p.x == q.x && p.y == q.y) || (p.x == q.y && p.y == q.x)));
    if (!same && p.mul() && !(q.mul() && q.uses < p.uses))
      r.s = "dcp_fma_rn(" + neg(p.x, p.neg) + ", " + p.y + ", " + neg(q.s, minus) + ")";
    else if (!same && q.mul())
      r.s = "dcp_fma_rn(" + neg(q.x, q.neg != minus) + ", " + q.y + ", " + p.s + ")";
    else
      r.s = std::string(minus ? "dcp_sub_rn(" : "dcp_add_rn(") + p.s + ", " + q.s + ")";
  };
  Ex c;
  c.s = imm;
  switch (op) {
    case DCP_MUL: product(a.s, b.s); break;
    case DCP_MUL_S: product(a.s, imm); break;
    case DCP_SQUARE: product(a.s, a.s); break;
    case DCP_NEG:
      r.s = "dcp_neg(" + a.s + ")";
      r.x = a.x;
      r.y = a.y;
      r.neg = !a.neg;
      break;
    case DCP_ADD: sum(a, b, false); break;
    case DCP_SUB: sum(a, b, true); break;
    case DCP_ADD_S: sum(a, c, false); break;
    case DCP_SUB_S: sum(a, c, true); break;
    case DCP_RSUB_S: sum(c, a, true); break;
    default: r.s = op_expr(op, dtype, imm_v, a.s, b.s);
  }
  return r;
}

// The maps `members` as in emit_members, with explicit rounding.
void emit_members_rn(std::ostringstream& os, const GraphImpl& g, const std::vector<int>& members) {
  std::map<int, Ex> ex;
  auto val = [&](int v) {
    auto it = ex.find(v);
    Ex e;
    if (it != ex.end()) e = it->second;
    e.s = var(v);
    return e;
  };
  for (int v : members) {
    const Node& n = g.nodes[v];
    const Ex a = n.in.empty() ? Ex() : val(n.in[0]);
    const Ex b = n.in.size() > 1 ? val(n.in[1]) : Ex();
    Ex e;
    if (n.kind == Kind::Stencil) e.s = a.s;  // zero-step stencil: identity
    else e = ex_op(n.op, n.dtype, n.imm, a, b);
    e.uses = 0;
    for (int m : members)
      for (int o : g.nodes[m].in) e.uses += o == v;
    os << "  const DCP_T " << var(v) << " = " << e.s << ";\n";
    ex[v] = e;
  }
}

void emit_members(std::ostringstream& os, const GraphImpl& g, const std::vector<int>& members) {
  for (int v : members) {
    const Node& n = g.nodes[v];
    std::string a = n.in.empty() ? "" : var(n.in[0]);
    std::string b = n.in.size() > 1 ? var(n.in[1]) : "";
    os << "  const DCP_T " << var(v) << " = " << map_expr(g, v, a, b) << ";\n";
  }
}

std::string red_op_fn(const GraphImpl& g, const std::vector<int>& reds) {
  std::ostringstream os;
  os << "__device__ __forceinline__ constexpr int dcp_red_op(int r) { return ";
  for (size_t i = 0; i < reds.size(); ++i) os << "r == " << i << " ? " << g.nodes[reds[i]].op << " : ";
  os << "0; }\n";
  return os.str();
}

// A kernel's name hashes its generated prefix together with the
// hand-written skeletons it includes (and those they include), so the name
// (and the compiled-module caches keyed by the source) changes exactly when
// one of them changes.
uint64_t skeleton_hash(const std::string& body) {
  const std::pair<const char*, const char*> skel[] = {
      {"k_map.cuh", kernel_map_source()},
      {"k_stencil2d.cuh", kernel_stencil2d_source()},
      {"k_stencil3d.cuh", kernel_stencil3d_source()},
      {"k_stencil2d_stream.cuh", kernel_stream_source()},
      {"k_axis.cuh", kernel_axis_source()},
      {"k_math64.cuh", kernel_math64_source()},
      {"k_stencil_adj.cuh", kernel_adj_source()},
      {"k_stencil2d_coop.cuh", kernel_coop_source()},
      {"k_tanh64.cuh", kernel_tanh64_source()},
      {"k_tanh64_table.cuh", kernel_tanh64_table_source()},
      {"k_stencil3d_col.cuh", kernel_column_source()}};
  constexpr size_t N = sizeof skel / sizeof skel[0];
  auto included = [&](const std::string& by) {
    unsigned m = 0;
    for (size_t i = 0; i < N; ++i)
      if (by.find(std::string("#include \"") + skel[i].first + "\"") != std::string::npos) m |= 1u << i;
    return m;
  };
  const unsigned used = included(body);
  // (the skeletons never change within a process: one hash per set of them)
  static std::mutex mu;
  static std::map<unsigned, uint64_t> known;
  std::lock_guard<std::mutex> lk(mu);
  auto it = known.find(used);
  if (it != known.end()) return it->second;
  unsigned all = used;  // with the skeletons they include themselves
  for (size_t i = 0; i < N; ++i)
    if (used >> i & 1u) all |= included(skel[i].second);
  std::string text = device_header_source();
  for (size_t i = 0; i < N; ++i)
    if (all >> i & 1u) text += skel[i].second;
  return known[used] = fnv1a(text);
}

std::string finish(const std::string& prefix, const std::string& b) {
  // binary64 exp / sin / cos come from k_math64.cuh and tanh from
  // k_tanh64.cuh; they are included only by kernels that call them, so other kernels' sources (and names) do not
  // depend on it
  std::string body = b;
  const std::string dev = "#include \"dcp_device.cuh\"\n";
  const size_t at = body.find(dev);
  if (at != std::string::npos && (body.find("dcp_exp64(") != std::string::npos ||
                                  body.find("dcp_sin64(") != std::string::npos ||
                                  body.find("dcp_cos64(") != std::string::npos))
    body.insert(at + dev.size(), "#include \"k_math64.cuh\"\n");
  if (at != std::string::npos && body.find("dcp_tanh64(") != std::string::npos)
    body.insert(at + dev.size(), "#include \"k_tanh64.cuh\"\n");
  char name[64];
  std::snprintf(name, sizeof name, "%s_%016" PRIx64, prefix.c_str(),
                fnv1a(body) ^ skeleton_hash(body));
  return std::string("#define DCP_KNAME ") + name + "\n" + body;
}

std::string kname_of(const std::string& src) {
  const char* p = std::strstr(src.c_str(), "#define DCP_KNAME ");
  std::string s(p + std::strlen("#define DCP_KNAME "));
  return s.substr(0, s.find('\n'));
}

}  // namespace

CodegenOut gen_map_kernel(const GraphImpl& g, const Group& G, bool vec_ok) {
  NameScope names;
  std::ostringstream os;
  const int T = G.dtype;
  int vec = vec_ok ? 16 / dtype_size(T) : 1;
  os << "// dcp fused map kernel: " << G.members.size() << " ops, " << G.loads.size() << " loads, "
     << G.stores.size() << " stores, " << G.reds.size() << " reductions\n";
  os << "#define DCP_T " << dtype_cname(T) << "\n";
  os << "#define DCP_VEC " << vec << "\n#define DCP_UNROLL " << (vec > 1 ? G.unroll : 1) << "\n";
  os << "#define DCP_NLOAD " << G.loads.size() << "\n#define DCP_NSTORE " << G.stores.size()
     << "\n#define DCP_NSCALAR " << G.scalars.size() << "\n#define DCP_NRED " << G.reds.size()
     << "\n#define DCP_THREADS " << G.threads << "\n";
  os << red_op_fn(g, G.reds);
  os << "#include \"dcp_device.cuh\"\n";
  os << "__device__ __forceinline__ void dcp_body(const DCP_T* ld, const DCP_T* sc, DCP_T* st, "
        "DCP_T* rv) {\n";
  for (size_t i = 0; i < G.loads.size(); ++i)
    os << "  const DCP_T " << var(G.loads[i]) << " = ld[" << i << "];\n";
  for (size_t i = 0; i < G.scalars.size(); ++i)
    os << "  const DCP_T " << var(G.scalars[i]) << " = sc[" << i << "];\n";
  emit_members(os, g, G.members);
  for (size_t i = 0; i < G.stores.size(); ++i) os << "  st[" << i << "] = " << var(G.stores[i]) << ";\n";
  for (size_t i = 0; i < G.reds.size(); ++i)
    os << "  rv[" << i << "] = " << var(g.nodes[G.reds[i]].in[0]) << ";\n";
  os << "  (void)ld; (void)sc; (void)st; (void)rv;\n}\n";
  os << "#include \"k_map.cuh\"\n";
  CodegenOut out;
  out.source = finish(vec > 1 ? "dcp_map_v" : "dcp_map_s", os.str());
  out.name = kname_of(out.source);
  out.threads = G.threads;
  out.smem_bytes = 0;
  return out;
}

// Axis reduction (k_axis.cuh): the reduced operands, with the fused
// prologue maps, at a flat index of the iteration space.
CodegenOut gen_axis_kernel(const GraphImpl& g, const Group& G, bool vec_ok) {
  NameScope names;
  std::ostringstream os;
  const int T = G.dtype;
  int64_t inner = 1;
  for (int d = G.axis + 1; d < (int)G.shape.size(); ++d) inner *= G.shape[d];
  const int64_t R = G.shape[G.axis];
  // 16-byte vectors along the contiguous axis when the shape allows it and
  // the reduction tree's shared memory stays within 32 KB
  const int axmode = inner > 1 ? 0 : 1;
  int vec = vec_ok ? 16 / dtype_size(T) : 1;
  // (rows shorter than four vectors per thread of a warp gain nothing from
  // unaligned ends)
  if ((axmode == 0 ? inner : R) % vec != 0 && (axmode == 0 || R < 4 * 32 * vec)) vec = 1;
  if ((int)G.reds.size() * vec > 16) vec = 1;
  os << "// dcp axis reduction kernel: " << G.members.size() << " prologue ops, " << G.loads.size()
     << " loads, " << G.reds.size() << " reductions along axis " << G.axis << "\n";
  os << "#define DCP_T " << dtype_cname(T) << "\n#define DCP_THREADS " << G.threads
     << "\n#define DCP_NRED " << G.reds.size() << "\n#define DCP_NLOAD " << G.loads.size()
     << "\n#define DCP_NSCALAR " << G.scalars.size() << "\n#define DCP_VEC " << vec
     << "\n#define DCP_AXMODE " << axmode << "\n#define DCP_RAGGED " << (axmode == 1 && R % vec != 0 ? 1 : 0)
     << "\n#define DCP_LONG " << (R >= 64 ? 1 : 0) << "\n";
  os << red_op_fn(g, G.reds);
  os << "#include \"dcp_device.cuh\"\n";
  os << "__device__ __forceinline__ void dcp_body(const DCP_T* ld, const DCP_T* sc, DCP_T* rv) {\n";
  for (size_t i = 0; i < G.loads.size(); ++i)
    os << "  const DCP_T " << var(G.loads[i]) << " = ld[" << i << "];\n";
  for (size_t i = 0; i < G.scalars.size(); ++i)
    os << "  const DCP_T " << var(G.scalars[i]) << " = sc[" << i << "];\n";
  emit_members(os, g, G.members);
  for (size_t i = 0; i < G.reds.size(); ++i)
    os << "  rv[" << i << "] = " << var(g.nodes[G.reds[i]].in[0]) << ";\n";
  os << "  (void)ld; (void)sc;\n}\n";
  os << "#include \"k_axis.cuh\"\n";
  CodegenOut out;
  out.source = finish("dcp_axis", os.str());
  out.name = kname_of(out.source);
  out.threads = G.threads;
  out.smem_bytes = 0;
  out.vec = vec;
  out.axmode = axmode;
  return out;
}

namespace {

// Maps, stores and reductions after the last step.
void emit_stencil_post(std::ostringstream& os, const GraphImpl& g, const Group& G, bool last) {
  os << "__device__ __forceinline__ void dcp_post(const DcpStParamsT<DCP_T>& p, const DCP_T* sc, "
        "long long gi, DCP_T v, DCP_T* st, DCP_T* rv) {\n";
  if (last) {
    os << "  const DCP_T " << var(G.st_out) << " = v;\n";
    for (size_t i = 0; i < G.post_loads.size(); ++i)
      os << "  const DCP_T " << var(G.post_loads[i]) << " = p.pld[" << i << "][gi];\n";
    for (size_t i = 0; i < G.scalars.size(); ++i)
      os << "  const DCP_T " << var(G.scalars[i]) << " = sc[" << i << "];\n";
    emit_members(os, g, G.post);
    for (size_t i = 0; i < G.stores.size(); ++i)
      os << "  st[" << i << "] = " << var(G.stores[i]) << ";\n";
    for (size_t i = 0; i < G.reds.size(); ++i)
      os << "  rv[" << i << "] = " << var(g.nodes[G.reds[i]].in[0]) << ";\n";
  }
  os << "  (void)p; (void)sc; (void)gi; (void)v; (void)st; (void)rv;\n}\n";
}

// Functions shared by 2-D and 3-D stencil sources: input (prologue), post.
void emit_stencil_io(std::ostringstream& os, const GraphImpl& g, const Group& G, bool first,
                     bool last) {
  os << "__device__ __forceinline__ DCP_T dcp_input(const DcpStParamsT<DCP_T>& p, const DCP_T* sc, "
        "long long gi) {\n";
  if (first && !G.members.empty()) {
    for (size_t i = 0; i < G.loads.size(); ++i)
      os << "  const DCP_T " << var(G.loads[i]) << " = p.ld[" << i << "][gi];\n";
    for (size_t i = 0; i < G.scalars.size(); ++i)
      os << "  const DCP_T " << var(G.scalars[i]) << " = sc[" << i << "];\n";
    emit_members_rn(os, g, G.members);
    os << "  (void)sc;\n  return " << var(G.st_in) << ";\n}\n";
  } else {
    os << "  (void)sc;\n  return p.ld[0][gi];\n}\n";
  }
  emit_stencil_post(os, g, G, last);
}
// Deferred common weight of a linear run of binary64 stencil steps.  A step
// u' = sum_k w_k u[p + o_k] whose weights are all exact multiples
// w_k = f r_k of one weight f (r_k = 1 at f's own points) is computed as
// w' = sum_k r_k w[p + o_k] on the scaled state w = u / f^t, and f^m is
// applied once at the end of every chunk of m steps.  The sum then starts
// from a point of ratio 1 with no multiply, so a p-point step takes p - 1
// FP64 operations instead of p (6 instead of 7 for the 7-point heat
// stencil, where 0.4 = 4 * 0.1 exactly; 4 adds instead of 5 operations for
// the 5-point average).  Only binary64 steps, which the FP64 pipe bounds,
// take this form.  A run is the consecutive steps of a group with equal
// weights (one stencil node, or a fused chain of equal ones), no epilogue
// map before its last step, a zero or periodic boundary (a fixed ring would
// need its border rescaled every step) and at least two steps.  Chunks are
// at most D steps with (sum |r_k|)^D <= 2^32, so the scaled state stays
// within 2^32 of the unscaled state's bound; f^m is the product of m
// roundings of f, applied with one more rounding.  Each step's arithmetic
// depends only on its place in its run, so every kernel form, tile shape,
// time-tile depth and split into launches computes the same bits.
//
// binary32 steps keep the plain sum: the float32 stencils are bound by
// instruction issue and memory latency, not by their arithmetic, and the
// deferred form measured no faster on the batched workload (slower at some
// time-tile depths).
struct Defer {
  bool on = false;
  std::vector<int> order;     // point order: a ratio-1 point first
  std::vector<double> ratio;  // r_k = w_k / f, exact
  double scale = 1.0;         // multiply after this step (1.0: none)
  double max_input = 0.0;     // largest finite |input| the run keeps finite
};

// f: the most frequent nonzero weight; of equally frequent ones, on 2 axes, one
// with a point in the neighbourhood's first row, where the row-by-row sums
// start (a 9-point star of radius 2, sides 0.1 and 0.05, then takes 8
// operations instead of 9).
bool defer_ratios(const Node& n, std::vector<double>& ratio, double& f_out, double& gsum) {
  const std::vector<double>& w = n.weights;
  const int P = (int)w.size();
  double f = 0.0;
  int best = 0;
  auto first_row = [&](double v) {
    int top = n.offsets[0];
    bool in = false;
    for (int k = 0; k < P; ++k) top = std::min(top, n.offsets[2 * k]);
    for (int k = 0; k < P; ++k) in = in || (w[k] == v && n.offsets[2 * k] == top);
    return in;
  };
  for (int k = 0; k < P; ++k) {
    if (w[k] == 0.0) continue;
    int c = 0;
    for (int j = 0; j < P; ++j) c += w[j] == w[k];
    if (c > best || (c == best && n.ndim() == 2 && !first_row(f) && first_row(w[k]))) best = c, f = w[k];
  }
  if (f == 0.0 || !std::isfinite(f)) return false;
  ratio.assign(P, 0.0);
  gsum = 0.0;
  for (int k = 0; k < P; ++k) {
    const double r = w[k] / f;
    if (!std::isfinite(r) || std::fma(r, f, -w[k]) != 0.0) return false;  // exact
    ratio[k] = r;
    gsum += std::fabs(r);
  }
  f_out = f;
  return true;
}

}  // namespace

// Longest chunk (steps between two applications of f^m) of a deferred run of
// stencil node n's steps; 0 when its steps keep the plain weighted sum.
// Unbounded growth limits (sum |r_k| <= 1) give INT32_MAX.
int defer_chunk_steps(const Node& n) {
  if (n.dtype != DCP_F64 || (n.bc != DCP_BC_ZERO && n.bc != DCP_BC_PERIODIC)) return 0;
  std::vector<double> r;
  double f = 0.0, gsum = 0.0;
  if (!defer_ratios(n, r, f, gsum)) return 0;
  if (gsum <= 1.0) return INT32_MAX;
  const int D = (int)std::floor(32.0 / std::log2(gsum));
  return D >= 2 ? D : 0;
}

namespace {

Defer plan_defer(const GraphImpl& g, const Group& G, int s) {
  Defer d;
  const Node& n = g.nodes[G.steps[s].node];
  if (n.dtype != DCP_F64 || (n.bc != DCP_BC_ZERO && n.bc != DCP_BC_PERIODIC)) return d;
  auto opt = g.options.find(DCP_OPT_DEFERRED_WEIGHT);
  if (opt != g.options.end() && opt->second == 0) return d;
  const int S = (int)G.steps.size();
  // steps of the group share their offsets; a run also needs the same
  // weights and boundary
  auto same = [&](int t) {
    const Node& m = g.nodes[G.steps[t].node];
    return m.bc == n.bc && m.weights == n.weights;
  };
  int a = s;
  while (a > 0 && same(a - 1) && G.steps[a - 1].epi.empty()) --a;
  int b = s + 1;
  while (b < S && same(b) && G.steps[b - 1].epi.empty()) ++b;
  const int L = b - a;
  if (L < 2) return d;
  std::vector<double> r;
  double f = 0.0, gsum = 0.0;
  if (!defer_ratios(n, r, f, gsum)) return d;
  const int Dmax = defer_chunk_steps(n);
  if (Dmax == 0) return d;
  const int D = std::min(L, Dmax);
  if (D < 2) return d;
  auto power = [f](int m) {
    double F = 1.0;
    for (int t = 0; t < m; ++t) F *= f;
    return std::isnormal(F) ? F : 0.0;
  };
  if (power(D) == 0.0 || (L % D != 0 && power(L % D) == 0.0)) return d;
  const int i = s - a;
  const int m = (i + 1) % D == 0 ? D : (s == b - 1 ? (i + 1) % D : 0);
  d.on = true;
  d.ratio = r;
  for (int k = 0; k < (int)r.size(); ++k)
    if (r[k] == 1.0) {
      d.order.push_back(k);
      break;
    }
  for (int k = 0; k < (int)r.size(); ++k)
    if (k != d.order[0]) d.order.push_back(k);
  d.scale = m > 0 ? power(m) : 1.0;
  // the scaled state of a chunk of D steps is at most (sum |r_k|)^D times the
  // largest |input| (sum |r_k| <= 1: no growth)
  const double growth = gsum <= 1.0 ? 1.0 : std::pow(gsum, (double)D);
  d.max_input = DBL_MAX / growth;
  return d;
}

// Multipliers of the binary64 weighted sums, held in registers.  On GB300 a
// binary64 fused multiply-add whose multiplier is a register of its own
// issues at the FP64 pipe's full rate (2 per clock per SM), while an add, a
// multiply, or fused multiply-adds that all share one multiplier issue at
// 1.68 (the library's FP64 probe).  So the terms of a sum are fused
// multiply-adds by multipliers kept in distinct registers -- an add becomes
// x * 1 + acc, which rounds exactly like acc + x -- loaded at kernel start
// from a small table in device memory (values the compiler cannot fold
// back into immediates).  Up to kMax slots (registers); beyond that, terms
// reuse slots holding the same value.  binary32 sums keep immediates.
struct MulRegs {
  static constexpr int kMax = 8;
  bool on = false;
  std::vector<double> vals;
  int next = 0;
  std::string get(int T, double w) {
    if (!on) return weight_literal(T, w);
    auto same = [w](double v) { return std::memcmp(&v, &w, sizeof v) == 0; };
    if ((int)vals.size() < kMax) {
      vals.push_back(w);
      return "km[" + std::to_string(vals.size() - 1) + "]";
    }
    for (int t = 0; t < kMax; ++t) {
      const int i = (next + t) % kMax;
      if (same(vals[i])) {
        next = i + 1;
        return "km[" + std::to_string(i) + "]";
      }
    }
    return weight_literal(T, w);
  }
  // The table the kernel loads its multiplier registers from.
  std::string table() const {
    std::ostringstream os;
    const int n = vals.empty() ? 1 : (int)vals.size();
    os << "#define DCP_NK " << n << "\n__device__ double dcp_km[DCP_NK] = {";
    for (int i = 0; i < n; ++i) {
      char buf[48];
      std::snprintf(buf, sizeof buf, "%a", vals.empty() ? 1.0 : vals[i]);  // exact
      os << (i ? ", " : "") << buf;
    }
    os << "};\n";
    return os.str();
  }
};

// One term of a weighted sum into accumulator a (declared by the first).
// Deferred sums: the first point is copied, the others are fused
// multiply-adds (ratio 1: x * 1 + acc, the same rounding as acc + x).
void emit_term(std::ostringstream& os, int T, const std::string& a, const std::string& x, double w,
               bool first, bool deferred, MulRegs& km) {
  if (deferred) {
    if (first) os << "  DCP_T " << a << " = " << x << ";\n";
    else if (w == 1.0 && !km.on) os << "  " << a << " = dcp_add(" << a << ", " << x << ");\n";
    else if (w == 1.0)
      os << "  " << a << " = dcp_fma_rn(" << x << ", " << km.get(T, 1.0) << ", " << a << ");\n";
    else os << "  " << a << " = dcp_fma_rn(" << weight_literal(T, w) << ", " << x << ", " << a << ");\n";
    return;
  }
  if (first) os << "  DCP_T " << a << " = dcp_mul_rn(" << weight_literal(T, w) << ", " << x << ");\n";
  else os << "  " << a << " = dcp_fma_rn(" << km.get(T, w) << ", " << x << ", " << a << ");\n";
}

// How every 1-D / 2-D kernel form evaluates one step's weighted sum, so that
// all of them round alike.
//
// Row order (any stencil): the points sorted by row offset dy (ascending, the
// listed order within a row), one multiply (or, on a deferred common weight,
// a copy of a ratio-1 point) and fused multiply-adds.  A kernel that streams
// rows then adds each arriving row to the sums of the rows it touches and
// keeps 2 ry partial sums per column instead of 2 ry + 1 rows.
//
// Pair order (a 5-point star on a deferred weight whose four sides have ratio
// 1): D(p) = w(west) + w(north) is also w(south) + w(east) of the cell one row
// up and one column left, so
//     sum(p) = (D(p) + r w(centre)) + D(p + (1, 1))
// and a kernel that keeps D pays one add for two pairs of neighbours: 3
// operations per cell instead of 4.  Steps that apply their weights keep the
// row order: sums before the weights could leave the plain sum's range, and
// weights before the sums round once more per point (measured: 1.3 times the
// error of 50 binary32 steps).
struct Sum2 {
  Defer df;
  bool pair = false;
  double wc = 1.0;            // pair: the centre's ratio
  std::vector<int> order;     // row order
  std::vector<double> w;      // row order: weights (ratios) by point index
};

bool star_sides(const std::vector<int32_t>& offs, int npts, int& centre, int (&side)[4]) {
  if (npts != 5) return false;
  centre = -1;
  for (int& v : side) v = -1;
  for (int k = 0; k < npts; ++k) {
    const int dz = offs[k * 3], dy = offs[k * 3 + 1], dx = offs[k * 3 + 2];
    int* slot = dz ? nullptr
                : dy == 0 && dx == 0 ? &centre
                : dy == 0 && dx == -1 ? &side[0]   // west
                : dy == -1 && dx == 0 ? &side[1]   // north
                : dy == 0 && dx == 1 ? &side[2]    // east
                : dy == 1 && dx == 0 ? &side[3] : nullptr;  // south
    if (!slot || *slot >= 0) return false;
    *slot = k;
  }
  return true;
}

// `offs`: the step's offsets (padded to 3 axes); `df`: its deferred weight.
Sum2 plan_sum2(const std::vector<int32_t>& offs, const std::vector<double>& weights,
               const Defer& df) {
  Sum2 p;
  p.df = df;
  p.w = df.on ? df.ratio : weights;
  const int n = (int)p.w.size();
  int c, sd[4];
  if (df.on && star_sides(offs, n, c, sd) && p.w[sd[0]] == 1.0 && p.w[sd[1]] == 1.0 &&
      p.w[sd[2]] == 1.0 && p.w[sd[3]] == 1.0) {
    p.pair = true;
    p.wc = p.w[c];
    return p;
  }
  for (int k = 0; k < n; ++k) p.order.push_back(k);
  std::stable_sort(p.order.begin(), p.order.end(),
                   [&](int a, int b) { return offs[a * 3 + 1] < offs[b * 3 + 1]; });
  if (df.on)  // start from a ratio-1 point of the first row, which needs no multiply
    for (int i = 1; i < n && offs[p.order[i] * 3 + 1] == offs[p.order[0] * 3 + 1]; ++i)
      if (p.w[p.order[0]] != 1.0 && p.w[p.order[i]] == 1.0) {
        std::rotate(p.order.begin(), p.order.begin() + i, p.order.begin() + i + 1);
        break;
      }
  return p;
}

// x + y as the kernels of dtype T add: binary64 as a fused multiply-add by a
// register of 1.0 (the same rounding at the pipe's full rate).
std::string add_expr(int T, const std::string& x, const std::string& y, MulRegs& km) {
  if (T == DCP_F64) return "dcp_fma_rn(" + x + ", " + km.get(T, 1.0) + ", " + y + ")";
  return "dcp_add_rn(" + x + ", " + y + ")";
}

// One row-order term into accumulator a (`fresh`: the sum's first term).
void emit_row_term(std::ostringstream& os, int T, const std::string& a, const std::string& from,
                   const std::string& x, double w, bool fresh, bool deferred, MulRegs& km) {
  os << "  " << a << " = ";
  if (fresh && deferred && w == 1.0) os << x;
  else if (fresh) os << "dcp_mul_rn(" << weight_literal(T, w) << ", " << x << ")";
  else if (w == 1.0 && deferred) os << add_expr(T, x, from, km);
  else os << "dcp_fma_rn(" << km.get(T, w) << ", " << x << ", " << from << ")";
  os << ";\n";
}

// The whole sum of one cell as straight-line code declaring `acc`; x(dy, dx)
// names the neighbour (kernels that hold a whole tile).
template <class X>
void emit_sum_cell(std::ostringstream& os, int T, const Sum2& p, const std::vector<int32_t>& offs,
                   X x, MulRegs& km) {
  os << "  DCP_T acc;\n";
  if (p.pair) {
    os << "  acc = " << add_expr(T, x(0, -1), x(-1, 0), km) << ";\n";
    if (p.wc == 1.0) os << "  acc = " << add_expr(T, x(0, 0), "acc", km) << ";\n";
    else os << "  acc = dcp_fma_rn(" << km.get(T, p.wc) << ", " << x(0, 0) << ", acc);\n";
    os << "  const DCP_T d2 = " << add_expr(T, x(1, 0), x(0, 1), km) << ";\n";
    os << "  acc = " << add_expr(T, "d2", "acc", km) << ";\n";
  } else {
    for (size_t i = 0; i < p.order.size(); ++i) {
      const int k = p.order[i];
      emit_row_term(os, T, "acc", "acc", x(offs[k * 3 + 1], offs[k * 3 + 2]), p.w[k], i == 0,
                    p.df.on, km);
    }
  }
  if (p.df.scale != 1.0)
    os << "  acc = dcp_mul_rn(" << weight_literal(T, p.df.scale) << ", acc);\n";
}

// Unary / immediate maps applied in order to `v`.
std::string epi_chain(const std::vector<std::pair<int, double>>& ops, int dtype) {
  std::ostringstream os;
  Ex cur;
  cur.s = "v";
  int k = 0;
  for (const auto& o : ops) {
    Ex e = ex_op(o.first, dtype, o.second, cur, Ex());
    const std::string nv = "e" + std::to_string(k++);
    os << "  const DCP_T " << nv << " = " << e.s << ";\n";
    cur = e;
    cur.s = nv;
  }
  os << "  return " << cur.s << ";\n";
  return os.str();
}

// Epilogue chain of one step as a function of the weighted sum.
std::string epi_body(const GraphImpl& g, const StepDesc& s) {
  std::vector<std::pair<int, double>> ops;
  for (int e : s.epi) ops.emplace_back(g.nodes[e].op, g.nodes[e].imm);
  return epi_chain(ops, s.epi.empty() ? DCP_F64 : g.nodes[s.epi[0]].dtype);
}

}  // namespace

// The arrival of one row in a level of the warp-stream kernel: dcp_row<S>
// takes the row `a`, adds it to the level's partial sums `st` and gives the
// finished row `out` (ry rows above `a`).  rm[k]: columns whose cells in
// output row (row of a) - ry + k belong to a fixed ring (RINGM only).
static void emit_stream_row(std::ostringstream& os, int T, int s, const Sum2& p,
                            const std::vector<int32_t>& offs, int C, int ry, int rx, MulRegs& km) {
  const int NST = 2 * ry;
  os << "template <> struct DcpRow<" << s << "> {\n  template <bool RINGM>\n"
     << "  static __device__ __forceinline__ void run(const DCP_T (&a)[" << C << "], DCP_T (&st)["
     << (NST > 0 ? NST : 1) << "][" << C << "], DCP_T (&out)[" << C
     << "], const DCP_T (&km)[DCP_NK], const unsigned (&rm)[" << ry + 1 << "]) {\n"
     << "  (void)km; (void)st; (void)rm;\n";
  if (p.df.on) os << "  // deferred common weight: the ratios w_k / f\n";
  auto at = [](const char* n, int i) { return std::string(n) + "[" + std::to_string(i) + "]"; };
  auto st = [](int k, int c) { return "st[" + std::to_string(k) + "][" + std::to_string(c) + "]"; };
  if (p.pair) {
    // (a deferred run has no fixed ring)
    os << "  DCP_T d[" << C << "];\n  const DCP_T al = __shfl_up_sync(0xffffffffu, a[" << C - 1 << "], 1);\n";
    for (int c = 0; c < C; ++c)
      os << "  " << at("d", c) << " = " << add_expr(T, c ? at("a", c - 1) : "al", st(0, c), km) << ";\n";
    os << "  const DCP_T dr = __shfl_down_sync(0xffffffffu, d[0], 1);\n";
    for (int c = 0; c < C; ++c)
      os << "  " << at("out", c) << " = " << add_expr(T, c + 1 < C ? at("d", c + 1) : "dr", st(1, c), km)
         << ";\n";
    for (int c = 0; c < C; ++c) {
      if (p.wc == 1.0) os << "  " << st(1, c) << " = " << add_expr(T, at("a", c), at("d", c), km) << ";\n";
      else os << "  " << st(1, c) << " = dcp_fma_rn(" << km.get(T, p.wc) << ", " << at("a", c) << ", "
              << at("d", c) << ");\n";
      os << "  " << st(0, c) << " = " << at("a", c) << ";\n";
    }
  } else {
    bool left = false, right = false;
    for (size_t k = 0; k < p.w.size(); ++k) {
      left = left || offs[k * 3 + 2] < 0;
      right = right || offs[k * 3 + 2] > 0;
    }
    if (left) {
      os << "  DCP_T lf[" << rx << "];\n";
      for (int q = 0; q < rx; ++q)
        os << "  lf[" << rx - 1 - q << "] = __shfl_up_sync(0xffffffffu, a[" << C - 1 - q << "], 1);\n";
    }
    if (right) {
      os << "  DCP_T rt[" << rx << "];\n";
      for (int q = 0; q < rx; ++q)
        os << "  rt[" << q << "] = __shfl_down_sync(0xffffffffu, a[" << q << "], 1);\n";
    }
    // stage k: output row (row of a) - ry + k receives its dy = ry - k points
    for (int k = 0; k <= 2 * ry; ++k) {
      const int dy = ry - k;
      bool started = false;
      std::vector<int> pts;
      for (int i : p.order) {
        if (offs[i * 3 + 1] < dy) started = true;
        if (offs[i * 3 + 1] == dy) pts.push_back(i);
      }
      // (term by term over the columns: neighbouring operations independent)
      const bool ring_sel = dy >= 0;  // a ring cell's sum is its own value
      auto src = [&](int c) { return k < 2 * ry ? st(k, c) : std::string("(DCP_T)0"); };
      os << "  {\n  DCP_T t[" << C << "];\n";
      if (started || pts.empty())
        for (int c = 0; c < C; ++c) os << "  t[" << c << "] = " << (started ? src(c) : "(DCP_T)0") << ";\n";
      bool fresh = !started;
      for (int i : pts) {
        for (int c = 0; c < C; ++c) {
          const int cc = c + offs[i * 3 + 2];
          const std::string x = cc < 0 ? at("lf", rx + cc) : (cc >= C ? at("rt", cc - C) : at("a", cc));
          emit_row_term(os, T, at("t", c), at("t", c), x, p.w[i], fresh, p.df.on, km);
        }
        fresh = false;
      }
      for (int c = 0; c < C; ++c) {
        if (ring_sel)
          os << "  if (RINGM && ((rm[" << k << "] >> " << c << ") & 1u)) t[" << c << "] = "
             << (dy == 0 ? at("a", c) : src(c)) << ";\n";
        os << "  " << (k == 0 ? at("out", c) : st(k - 1, c)) << " = t[" << c << "];\n";
      }
      os << "  }\n";
    }
  }
  if (p.df.scale != 1.0)
    for (int c = 0; c < C; ++c)
      os << "  " << at("out", c) << " = dcp_mul_rn(" << weight_literal(T, p.df.scale) << ", "
         << at("out", c) << ");\n";
  os << "  }\n};\n";
}

// Binary64 3-D stars on a deferred weight are summed by shared pairs (see
// k_stencil3d_col.cuh) when the points at y +- 1 and z +- 1 have ratio 1 and
// the others lie in the row (|dx| <= 1); every 3-D kernel form evaluates
// D = north + below, then the row's points in listed order, then south +
// above, so all forms round alike.  (Steps that apply their weights keep the
// listed order: a pair would take two operations, and the planes form, which
// runs their epilogues, does not share it.)
struct Sum3 {
  bool pairs = false;
  int n = -1, s = -1, b = -1, t = -1;  // north, south, below (z - 1), above (z + 1)
  std::vector<int> row;                // the row's points, listed order
};

Sum3 plan_sum3(int T, const std::vector<int32_t>& offs, const std::vector<double>& w, const Defer& df) {
  Sum3 p;
  if (T != DCP_F64 || !df.on) return p;
  for (int k = 0; k < (int)w.size(); ++k) {
    const int dz = offs[k * 3], dy = offs[k * 3 + 1], dx = offs[k * 3 + 2];
    int* slot = dz == 0 && dy == -1 && dx == 0 ? &p.n
                : dz == 0 && dy == 1 && dx == 0 ? &p.s
                : dz == -1 && dy == 0 && dx == 0 ? &p.b
                : dz == 1 && dy == 0 && dx == 0 ? &p.t : nullptr;
    if (slot) {
      if (*slot >= 0) return p;
      *slot = k;
    } else if (dz == 0 && dy == 0 && dx >= -1 && dx <= 1) {
      for (int r : p.row)
        if (offs[r * 3 + 2] == dx) return p;
      p.row.push_back(k);
    } else {
      return p;
    }
  }
  if (p.n < 0 || p.s < 0 || p.b < 0 || p.t < 0) return p;
  p.pairs = df.ratio[p.n] == 1.0 && df.ratio[p.s] == 1.0 && df.ratio[p.b] == 1.0 && df.ratio[p.t] == 1.0;
  return p;
}

// A row point of ratio r added to `acc`.
std::string row_expr(int T, double r, const std::string& x, MulRegs& km) {
  if (r == 1.0) return add_expr(T, x, "acc", km);
  return "dcp_fma_rn(" + km.get(T, r) + ", " + x + ", acc)";
}

// Does a binary32 3-D star list its points as the column kernel adds them:
// in-plane star points, then below, then above?
bool listed_star3(const std::vector<int32_t>& offs, int n) {
  if (n < 3) return false;
  for (int k = 0; k < n; ++k) {
    const int dz = offs[k * 3], dy = offs[k * 3 + 1], dx = offs[k * 3 + 2];
    if (k == n - 1 ? !(dz == 1 && !dy && !dx)
        : k == n - 2 ? !(dz == -1 && !dy && !dx)
                     : (dz != 0 || std::abs(dy) + std::abs(dx) > 1))
      return false;
  }
  return true;
}

// Can step s of the group be summed by the column kernel?
bool column_step(const GraphImpl& g, const Group& G, int s) {
  const Node& n = g.nodes[G.steps[s].node];
  return G.dtype == DCP_F64 ? plan_sum3(G.dtype, G.offsets, n.weights, plan_defer(g, G, s)).pairs
                            : listed_star3(G.offsets, n.npts());
}

// Warp-streamed columns of a 3-D star (k_stencil3d_col.cuh).
static CodegenOut gen_column_kernel(const GraphImpl& g, const Group& G, int s0, int s1, int max_vec) {
  NameScope names;
  const int T = G.dtype, K = s1 - s0, C = stream_cols_per_lane(T);
  const bool first = s0 == 0, last = s1 == (int)G.steps.size();
  const bool f64 = T == DCP_F64;
  for (int s = s0; s < s1; ++s)
    if (!column_step(g, G, s)) fail(DCP_E_UNSUPPORTED, "3-D columns do not suit this stencil group");
  int vec = std::min(C, max_vec);
  while (G.shape.back() % vec != 0) vec /= 2;
  // four warps share the ticket of a launch that reduces (see gen_stream_kernel),
  // but where two steps of four rows need every register
  const int threads = last && !G.reds.empty() && !f64 && K * G.cy < 8 ? 4 * G.threads : G.threads;
  std::ostringstream os;
  os << "// dcp 3-D column stencil kernel: " << K << " steps per launch, bc " << G.bc << "\n";
  os << "#define DCP_T " << dtype_cname(T) << "\n#define DCP_C " << C << "\n#define DCP_CY " << G.cy
     << "\n#define DCP_LX " << G.lx << "\n#define DCP_NSTEPS " << K << "\n#define DCP_R " << kColumnRing << "\n#define DCP_W "
     << column_width(G, K) << "\n#define DCP_VEC " << vec << "\n#define DCP_PAIRS " << (f64 ? 1 : 0)
     << "\n#define DCP_BC " << G.bc << "\n#define DCP_THREADS " << threads << "\n#define DCP_LAST "
     << (last ? 1 : 0) << "\n#define DCP_POST "
     << (last && (!G.post.empty() || !G.reds.empty() || G.stores.size() != 1) ? 1 : 0)
     << "\n#define DCP_MINB " << std::max(1, G.min_ctas * G.threads / threads) << "\n#define DCP_NSTORE "
     << (last ? (int)G.stores.size() : 1) << "\n#define DCP_NRED " << (last ? (int)G.reds.size() : 0)
     << "\n#define DCP_NSCALAR " << G.scalars.size() << "\n";
  const Defer guard = first ? plan_defer(g, G, 0) : Defer();
  os << "#define DCP_GUARD " << (guard.on ? 1 : 0) << "\n";
  os << red_op_fn(g, last ? G.reds : std::vector<int>{});
  os << "#include \"dcp_device.cuh\"\n";
  emit_stencil_post(os, g, G, last);
  const char* fn = "__device__ __forceinline__ DCP_T ";
  const std::string kp = ", const DCP_T (&km)[DCP_NK])";
  os << "template <int S> " << fn << "dcp_epi(DCP_T v);\n";
  MulRegs km;
  km.on = f64;
  std::ostringstream sums, decl;
  CodegenOut out;
  for (int s = 0; s < K; ++s) {
    const StepDesc& sd = G.steps[s0 + s];
    const Node& sn = g.nodes[sd.node];
    const Defer df = plan_defer(g, G, s0 + s);
    const std::string sp = "template <> " + std::string(fn);
    const std::string id = "<" + std::to_string(s) + ">";
    auto side = [&](int dx) { return dx < 0 ? "l" : (dx > 0 ? "r" : "c"); };
    if (f64) {
      const Sum3 p = plan_sum3(T, G.offsets, sn.weights, df);
      sums << "// deferred common weight: the ratios w_k / f\n";
      for (int c = 0; c < C; ++c) {
        const std::string ic = "<" + std::to_string(s) + ", " + std::to_string(c) + ">";
        sums << sp << "dcp_d" << ic << "(DCP_T up, DCP_T before" << kp << " {\n  (void)km;\n  return "
             << add_expr(T, "up", "before", km) << ";\n}\n";
        sums << sp << "dcp_in" << ic << "(DCP_T d, DCP_T c, DCP_T l, DCP_T r" << kp
             << " {\n  (void)km; (void)c; (void)l; (void)r;\n  DCP_T acc = d;\n";
        for (int k : p.row)
          sums << "  acc = " << row_expr(T, df.ratio[k], side(G.offsets[k * 3 + 2]), km) << ";\n";
        sums << "  return acc;\n}\n";
        sums << sp << "dcp_fin" << ic << "(DCP_T acc, DCP_T d" << kp << " {\n  (void)km;\n  acc = "
             << add_expr(T, "d", "acc", km) << ";\n";
        if (df.scale != 1.0) sums << "  acc = dcp_mul_rn(" << weight_literal(T, df.scale) << ", acc);\n";
        sums << "  return acc;\n}\n";
      }
      if (s == 0)
        decl << "template <int S, int I> " << fn << "dcp_d(DCP_T up, DCP_T before" << kp
             << ";\ntemplate <int S, int I> " << fn << "dcp_in(DCP_T d, DCP_T c, DCP_T l, DCP_T r" << kp
             << ";\ntemplate <int S, int I> " << fn << "dcp_fin(DCP_T acc, DCP_T d" << kp << ";\n";
    } else {
      sums << sp << "dcp_in" << id << "(DCP_T c, DCP_T l, DCP_T r, DCP_T up, DCP_T dn, DCP_T before) {\n"
           << "  (void)c; (void)l; (void)r; (void)up; (void)dn;\n";
      const int n = sn.npts();
      for (int k = 0; k + 1 < n; ++k) {
        const int dz = G.offsets[k * 3], dy = G.offsets[k * 3 + 1], dx = G.offsets[k * 3 + 2];
        const std::string x = dz ? "before" : (dy < 0 ? "up" : (dy > 0 ? "dn" : side(dx)));
        emit_term(sums, T, "acc", x, sn.weights[k], k == 0, false, km);
      }
      sums << "  return acc;\n}\n";
      sums << sp << "dcp_fin" << id << "(DCP_T acc, DCP_T c) {\n";
      emit_term(sums, T, "acc", "c", sn.weights[n - 1], false, false, km);
      sums << "  return acc;\n}\n";
      if (s == 0)
        decl << "template <int S> " << fn
             << "dcp_in(DCP_T c, DCP_T l, DCP_T r, DCP_T up, DCP_T dn, DCP_T before);\ntemplate <int S> " << fn
             << "dcp_fin(DCP_T acc, DCP_T c);\n";
    }
    if (df.on) out.defer_scales.push_back(df.scale);
    sums << sp << "dcp_epi" << id << "(DCP_T v) {\n" << epi_body(g, sd) << "}\n";
  }
  os << km.table() << decl.str() << sums.str();
  os << "#include \"k_stencil3d_col.cuh\"\n";
  out.threads = threads;
  out.vec = vec;
  out.guard_max_input = guard.on ? guard.max_input : 0.0;
  out.smem_bytes = threads / 32 * kColumnRing * (32 / G.lx * G.cy + 2 * K) * ((G.lx + 2) * C) * dtype_size(T);
  out.source = finish("dcp_col3d", os.str());
  out.name = kname_of(out.source);
  return out;
}

// Warp-stream form (k_stencil2d_stream.cuh) of a 1-D / 2-D stencil launch.
static CodegenOut gen_stream_kernel(const GraphImpl& g, const Group& G, int s0, int s1, int max_vec) {
  NameScope names;
  const bool batch = G.kind == GroupKind::Batch;
  const int nd = batch ? 2 : (int)G.shape.size();
  const int T = G.dtype;
  const int nsteps = s1 - s0;
  const bool first = s0 == 0, last = s1 == (int)G.steps.size();
  const int C = stream_cols_per_lane(T);
  const int ry = nd == 1 ? 0 : G.radius[1], rx = G.radius[2];
  const bool pro = !batch && first && !G.members.empty();
  // elements per access: the widest that divides a row (batched: per instance)
  int vec = 0;
  if (!batch)
    for (vec = std::min(C, max_vec); G.shape.back() % vec != 0;) vec /= 2;
  const bool exact = stream_exact(G);
  if (exact) vec = 1;
  std::ostringstream os;
  os << "// dcp warp-stream stencil kernel: " << nsteps << " steps per launch, bc " << G.bc << ", "
     << nd << "-D" << (batch ? ", batched" : "") << "\n";
  os << "#define DCP_T " << dtype_cname(T) << "\n#define DCP_C " << C << "\n";
  // shared-memory ring: 8 rows (a window of 7 rows ahead hides device-memory
  // latency from 4 warps per scheduler) per prefetch window and input array,
  // 512 bytes each; fewer rows, then fewer warps per CTA where 192 KB is short
  const int nload = pro ? (int)G.loads.size() : 1;
  const int nin = std::max(1, nload);  // a prologue of broadcast scalars loads no array
  // A 1-D array's items are one row each.
  int threads = G.threads, ring = nd == 1 ? 4 : 8;  // a power of two
  for (const int rows = ring * G.prefetch; ring < rows;) ring *= 2;
  // Every CTA of a launch that reduces takes a ticket, about 7 ns each, one
  // after the other: four binary32 warps share one (a step of 1000 x 1001 with
  // its maximum 18.5 -> 11 us).  The FP64 pipes would be shared out too
  // unevenly (3000 x 3100: 160 us in CTAs of two warps, 209 in CTAs of eight).
  if (last && !G.reds.empty() && T == DCP_F32 && !g.options.count(DCP_OPT_STREAM_THREADS))
    threads = std::max(threads, 128);
  auto smem = [&] { return threads / 32 * nin * ring * 512; };
  while (smem() > 192 * 1024 && ring > 4) ring /= 2;
  while (smem() > 192 * 1024 && threads > 32) threads = threads / 64 * 32;
  os << "#define DCP_THREADS " << threads << "\n#define DCP_BC " << G.bc << "\n";
  os << "#define DCP_LAST " << (last ? 1 : 0) << "\n#define DCP_BATCH " << (batch ? 1 : 0) << "\n";
  os << "#define DCP_NSTORE " << (last ? (int)G.stores.size() : 1) << "\n#define DCP_NRED "
     << (last ? (int)G.reds.size() : 0) << "\n#define DCP_NSCALAR " << G.scalars.size() << "\n";
  os << "#define DCP_NLOAD " << nload << "\n#define DCP_NIN " << nin << "\n#define DCP_PRO " << (pro ? 1 : 0)
     << "\n#define DCP_POST "
     << (last && (!G.post.empty() || !G.reds.empty() || G.stores.size() != 1) ? 1 : 0) << "\n";
  os << "#define DCP_RX " << rx << "\n#define DCP_RY " << ry << "\n#define DCP_NSTEPS " << nsteps
     << "\n#define DCP_R " << ring << "\n#define DCP_W " << stream_width(G, nsteps)
     << "\n#define DCP_HX " << (exact ? nsteps * rx : (nsteps * rx + C - 1) / C * C)
     << "\n#define DCP_VEC " << vec
     << "\n#define DCP_HUGE " << (!batch && G.shape.back() > 0x7fffffff - 4096 ? 1 : 0) << "\n";
  const Defer guard = first ? plan_defer(g, G, 0) : Defer();
  os << "#define DCP_GUARD " << (guard.on ? 1 : 0) << "\n";
  if (G.min_ctas > 0) os << "#define DCP_MINB " << std::max(1, G.min_ctas * G.threads / threads) << "\n";
  os << red_op_fn(g, last ? G.reds : std::vector<int>{});
  os << "#include \"dcp_device.cuh\"\n";
  if (!batch) {
    // the prologue as a function of the loaded values (the kernel keeps raw
    // loads in flight and evaluates the maps when the row arrives)
    os << "__device__ __forceinline__ DCP_T dcp_pro(const DCP_T (&ld)[DCP_NIN], const DCP_T* sc) {\n"
          "  (void)sc;\n";
    if (pro) {
      for (size_t i = 0; i < G.loads.size(); ++i)
        os << "  const DCP_T " << var(G.loads[i]) << " = ld[" << i << "];\n";
      for (size_t i = 0; i < G.scalars.size(); ++i)
        os << "  const DCP_T " << var(G.scalars[i]) << " = sc[" << i << "];\n";
      emit_members_rn(os, g, G.members);
      os << "  return " << var(G.st_in) << ";\n}\n";
    } else {
      os << "  return ld[0];\n}\n";
    }
    emit_stencil_post(os, g, G, last);
  }
  os << "template <int S> __device__ __forceinline__ DCP_T dcp_epi(DCP_T v);\n"
     << "template <int S> struct DcpRow;\n";
  std::vector<double> scales;
  MulRegs km;
  km.on = T == DCP_F64;
  std::ostringstream sums;  // emitted after the multiplier table they use
  for (int s = 0; s < nsteps; ++s) {
    const StepDesc& sd = G.steps[s0 + s];
    const Sum2 p = plan_sum2(G.offsets, g.nodes[sd.node].weights, plan_defer(g, G, s0 + s));
    scales.push_back(p.df.on ? p.df.scale : 0.0);
    emit_stream_row(sums, T, s, p, G.offsets, C, ry, rx, km);
    sums << "template <> __device__ __forceinline__ DCP_T dcp_epi<" << s << ">(DCP_T v) {\n"
         << epi_body(g, sd) << "}\n";
  }
  os << km.table() << sums.str();
  os << "#include \"k_stencil2d_stream.cuh\"\n";
  CodegenOut out;
  out.threads = threads;
  out.smem_bytes = smem();
  for (double x : scales)
    if (x != 0.0) out.defer_scales = scales;
  out.guard_max_input = guard.on ? guard.max_input : 0.0;
  out.vec = std::max(1, vec);
  out.source = finish(batch ? "dcp_bstream" : "dcp_stream", os.str());
  out.name = kname_of(out.source);
  return out;
}

CodegenOut gen_stencil_kernel(const GraphImpl& g, const Group& G, int s0, int s1, int max_vec) {
  if (G.variant == 1) return gen_stream_kernel(g, G, s0, s1, max_vec);
  if (G.variant == 3) return gen_column_kernel(g, G, s0, s1, max_vec);
  NameScope names;
  const bool batch = G.kind == GroupKind::Batch;
  const int nd = batch ? 2 : (int)G.shape.size();
  const int T = G.dtype;
  const int nsteps = s1 - s0;
  const bool first = s0 == 0, last = s1 == (int)G.steps.size();
  std::ostringstream os;
  os << "// dcp stencil kernel: " << nsteps << " steps per launch, bc " << G.bc << ", " << nd
     << "-D" << (batch ? ", batched" : "") << "\n";
  // 3-D: paired cells along x when requested and the tile allows it; rows of
  // the plane are then stored from an even offset so every pair is aligned
  const int rz = G.radius[0], ry = G.radius[1], rx = G.radius[2];
  const int CX3 = nd == 3 && G.cx == 2 && G.tile[2] % 2 == 0 && rx <= 2 ? 2 : 1;
  const int threads = nd == 3 ? G.tile[2] * G.tile[1] / CX3 : G.threads;
  os << "#define DCP_T " << dtype_cname(T) << "\n";
  os << "#define DCP_THREADS " << threads << "\n#define DCP_BC " << G.bc << "\n";
  os << "#define DCP_LAST " << (last ? 1 : 0) << "\n#define DCP_BATCH " << (batch ? 1 : 0) << "\n";
  int nstore = last ? (int)G.stores.size() : 1;
  int nred = last ? (int)G.reds.size() : 0;
  os << "#define DCP_NSTORE " << nstore << "\n#define DCP_NRED " << nred << "\n#define DCP_NSCALAR "
     << G.scalars.size() << "\n";
  const Defer guard = first ? plan_defer(g, G, 0) : Defer();
  os << "#define DCP_GUARD " << (guard.on ? 1 : 0) << "\n";
  os << red_op_fn(g, last ? G.reds : std::vector<int>{});
  os << "#include \"dcp_device.cuh\"\n";
  CodegenOut out;
  out.threads = threads;
  out.guard_max_input = guard.on ? guard.max_input : 0.0;
  // cooperative form: every step in one launch, a halo of one radius
  const bool coop = G.variant == 2 && nd <= 2 && !batch;
  if (coop && (!first || !last))
    fail(DCP_E_UNSUPPORTED, "the cooperative stencil form runs every step in one launch");
  if (nd <= 2) {
    const int TX = G.tile[2], TY = nd == 1 ? 1 : G.tile[1];
    const int RY = nd == 1 ? 0 : ry;
    const int hs = coop ? 1 : nsteps;  // halo width in radii
    const int PW = TX + 2 * hs * rx, PH = TY + 2 * hs * RY;
    os << "#define DCP_TX " << TX << "\n#define DCP_TY " << TY << "\n#define DCP_RX " << rx
       << "\n#define DCP_RY " << RY << "\n#define DCP_NSTEPS " << nsteps << "\n";
    if (!batch) emit_stencil_io(os, g, G, first, last);
    os << "template <int S> __device__ __forceinline__ DCP_T dcp_epi(DCP_T v);\n";
    std::vector<double> scales;
    MulRegs km;
    km.on = T == DCP_F64;
    std::ostringstream sums;  // emitted after the multiplier table they use
    for (int s = 0; s < nsteps; ++s) {
      std::ostringstream& os = sums;
      const StepDesc& sd = G.steps[s0 + s];
      const Node& sn = g.nodes[sd.node];
      os << "template <> __device__ __forceinline__ DCP_T dcp_sum<" << s
         << ">(const DCP_T* A, int c, const DCP_T (&km)[DCP_NK]) {\n  (void)km;\n";
      const Sum2 p = plan_sum2(G.offsets, sn.weights, plan_defer(g, G, s0 + s));
      if (p.df.on) os << "  // deferred common weight: the ratios w_k / f\n";
      scales.push_back(p.df.on ? p.df.scale : 0.0);
      emit_sum_cell(os, T, p, G.offsets, [&](int dy, int dx) {
        return "A[c + (" + std::to_string(dy * PW + dx) + ")]";
      }, km);
      os << "  return acc;\n}\n";
      os << "template <> __device__ __forceinline__ DCP_T dcp_epi<" << s << ">(DCP_T v) {\n"
         << epi_body(g, sd) << "}\n";
    }
    os << km.table();
    os << "template <int S> __device__ __forceinline__ DCP_T dcp_sum(const DCP_T* A, int c, "
          "const DCP_T (&km)[DCP_NK]);\n";
    os << sums.str();
    if (coop) {
      // host-side fault injection (DCP_FAULT=coop_wait): every neighbour wait
      // gives up after 1000 polls, so the bounded-wait error path runs
      // without a fault or a hang
      const char* f = std::getenv("DCP_FAULT");
      if (f && std::strcmp(f, "coop_wait") == 0)
        os << "#define DCP_SPIN_LIMIT 1000\n#define DCP_WAIT_SKEW 4096u\n";
    }
    os << (coop ? "#include \"k_stencil2d_coop.cuh\"\n" : "#include \"k_stencil2d.cuh\"\n");
    out.smem_bytes = 2 * PW * PH * dtype_size(T);
    for (double x : scales)
      if (x != 0.0) out.defer_scales = scales;
  } else {
    if (nsteps != 1) fail(DCP_E_UNSUPPORTED, "3-D stencil launches run one step each");
    const int TX = G.tile[2], TY = G.tile[1], TZ = G.tile[0];
    const int CX = CX3;
    const int AX = CX == 2 ? (rx + 1) / 2 * 2 : rx;
    const int PW = TX + 2 * AX, PH = TY + 2 * ry;
    os << "#define DCP_TX " << TX << "\n#define DCP_TY " << TY << "\n#define DCP_TZ " << TZ
       << "\n#define DCP_RX " << rx << "\n#define DCP_RY " << ry << "\n#define DCP_RZ " << rz
       << "\n#define DCP_CX " << CX << "\n#define DCP_AX " << AX << "\n";
    emit_stencil_io(os, g, G, first, last);
    const StepDesc& sd = G.steps[s0];
    const Node& sn = g.nodes[sd.node];
    MulRegs km;
    km.on = T == DCP_F64;
    std::ostringstream sums;  // emitted after the multiplier table it uses
    sums << "__device__ __forceinline__ void dcp_sum3(const DCP_T* const* pl, int c, DCP_T (&v)["
         << CX << "], const DCP_T (&km)[DCP_NK]) {\n  (void)km;\n";
    const Defer df = plan_defer(g, G, s0);
    std::vector<int> order(sn.npts());
    for (int k = 0; k < sn.npts(); ++k) order[k] = df.on ? df.order[k] : k;
    auto wt = [&](int k) { return df.on ? df.ratio[k] : sn.weights[k]; };
    if (df.on) sums << "  // deferred common weight: the ratios w_k / f\n";
    if (df.on) out.defer_scales = {df.scale};
    const Sum3 p3 = plan_sum3(T, G.offsets, sn.weights, df);
    // the weighted sum of one cell; x(k) names point k's value
    auto emit_cell = [&](const std::string& a, const std::function<std::string(int)>& x) {
      if (p3.pairs) {
        sums << "  DCP_T " << a << ";\n  {\n  DCP_T acc = " << add_expr(T, x(p3.n), x(p3.b), km)
             << ";\n";
        for (int k : p3.row) sums << "  acc = " << row_expr(T, df.ratio[k], x(k), km) << ";\n";
        sums << "  const DCP_T d2 = " << add_expr(T, x(p3.t), x(p3.s), km) << ";\n  " << a
             << " = " << add_expr(T, "d2", "acc", km) << ";\n  }\n";
      } else {
        for (int i = 0; i < sn.npts(); ++i)
          emit_term(sums, T, a, x(order[i]), wt(order[i]), i == 0, df.on, km);
      }
      if (df.scale != 1.0)
        sums << "  " << a << " = dcp_mul_rn(" << weight_literal(T, df.scale) << ", " << a << ");\n";
    };
    if (CX == 1) {
      emit_cell("a0", [&](int k) {
        int dz = G.offsets[k * 3], dy = G.offsets[k * 3 + 1], dx = G.offsets[k * 3 + 2];
        return "pl[" + std::to_string(dz + rz) + "][c + (" + std::to_string(dy * PW + dx) + ")]";
      });
      sums << "  v[0] = a0;\n";
    } else {
      // one aligned pair load per distinct (plane, pair index) the two cells read
      auto floor_div2 = [](int o) { return o >= 0 ? o / 2 : -((-o + 1) / 2); };
      std::map<std::pair<int, int>, std::string> pairs;
      sums << "  typedef typename DcpVec2<DCP_T>::type T2;\n";
      for (int k = 0; k < sn.npts(); ++k)
        for (int j = 0; j < 2; ++j) {
          int dz = G.offsets[k * 3], dy = G.offsets[k * 3 + 1], dx = G.offsets[k * 3 + 2];
          int q = floor_div2(dy * PW + dx + j);
          auto key = std::make_pair(dz + rz, q);
          if (pairs.count(key)) continue;
          std::string nm = "p" + std::to_string(pairs.size());
          pairs[key] = nm;
          sums << "  const T2 " << nm << " = *reinterpret_cast<const T2*>(pl[" << key.first
               << "] + c + (" << 2 * q << "));\n";
        }
      for (int j = 0; j < 2; ++j) {
        std::string a = "a" + std::to_string(j);
        emit_cell(a, [&](int k) {
          int dz = G.offsets[k * 3], dy = G.offsets[k * 3 + 1], dx = G.offsets[k * 3 + 2];
          int o = dy * PW + dx + j, q = floor_div2(o);
          return pairs[std::make_pair(dz + rz, q)] + (o - 2 * q == 0 ? ".x" : ".y");
        });
        sums << "  v[" << j << "] = " << a << ";\n";
      }
    }
    sums << "}\n";
    os << km.table() << sums.str();
    os << "__device__ __forceinline__ DCP_T dcp_epi3(DCP_T v) {\n" << epi_body(g, sd) << "}\n";
    os << "#include \"k_stencil3d.cuh\"\n";
    out.smem_bytes = (2 * rz + 2) * PW * PH * dtype_size(T);
  }
  out.source = finish(batch ? "dcp_batch" : (nd == 3 ? "dcp_st3d" : (coop ? "dcp_coop" : "dcp_st2d")),
                      os.str());
  out.name = kname_of(out.source);
  return out;
}

bool column_eligible(const GraphImpl& g, const Group& G) {
  if (G.kind != GroupKind::Stencil || G.shape.size() != 3 || !G.members.empty()) return false;
  if (G.radius[0] != 1 || G.radius[1] > 1 || G.radius[2] > 1) return false;
  if (G.shape[1] * G.shape[2] > 0x7fffffff) return false;  // offsets within a plane are 32-bit
  for (int64_t n : G.shape)
    if (n > 0x7fffffff - 4096) return false;  // a block may reach past the last cell
  for (int s = 0; s < (int)G.steps.size(); ++s)
    if (!column_step(g, G, s)) return false;
  return true;
}

CodegenOut gen_batch_kernel(const GraphImpl& g, const Group& G, int s0, int s1) {
  return gen_stencil_kernel(g, G, s0, s1);
}


// ---------------------------------------------------------------------------
// Time-tiled reverse pass of a 1-D / 2-D stencil chain (k_stencil_adj.cuh).
// ---------------------------------------------------------------------------
namespace {

// Which forward value the reverse rule of a unary / immediate op reads:
// 1 its operand X, 2 its result Y, 0 neither.  The rules are those of the
// adjoint's per-op reverse maps, so the fused reverse rounds alike.
int vjp_reads(int op) {
  switch (op) {
    case DCP_ABS: case DCP_SIN: case DCP_COS: case DCP_SQUARE: return 1;
    case DCP_EXP: case DCP_TANH: case DCP_SQRT: return 2;
    case DCP_NEG: case DCP_ADD_S: case DCP_SUB_S: case DCP_MUL_S: case DCP_RSUB_S: return 0;
  }
  fail(DCP_E_UNSUPPORTED, std::string("adjoint: no reverse rule for epilogue op ") + op_name(op));
}

// Cotangent of the operand of op from the cotangent a of its result (the
// same expressions as the per-op reverse maps of the adjoint builder).
std::string vjp_expr(int op, double imm, int T, const std::string& as, const std::string& Xs,
                     const std::string& Ys) {
  Ex a, X, Y;
  a.s = as;
  X.s = Xs;
  Y.s = Ys;
  auto e = [&](int o, double i, const Ex& p, const Ex& q = Ex()) { return ex_op(o, T, i, p, q); };
  switch (op) {
    case DCP_NEG: return e(DCP_NEG, 0, a).s;
    case DCP_ABS: return e(DCP_MUL, 0, e(kOpSign, 0, X), a).s;
    case DCP_EXP: return e(DCP_MUL, 0, Y, a).s;
    case DCP_SIN: return e(DCP_MUL, 0, e(DCP_COS, 0, X), a).s;
    case DCP_COS: return e(DCP_MUL, 0, e(DCP_NEG, 0, e(DCP_SIN, 0, X)), a).s;
    case DCP_TANH: return e(DCP_MUL, 0, e(DCP_RSUB_S, 1.0, e(DCP_SQUARE, 0, Y)), a).s;
    case DCP_SQRT: return e(DCP_DIV, 0, e(DCP_MUL_S, 0.5, a), Y).s;
    case DCP_SQUARE: return e(DCP_MUL, 0, e(DCP_MUL_S, 2.0, X), a).s;
    case DCP_ADD_S: case DCP_SUB_S: return as;
    case DCP_MUL_S: return e(DCP_MUL_S, imm, a).s;
    case DCP_RSUB_S: return e(DCP_NEG, 0, a).s;
  }
  fail(DCP_E_UNSUPPORTED, std::string("adjoint: no reverse rule for epilogue op ") + op_name(op));
}

}  // namespace

bool adj_needs_z(const std::vector<std::pair<int, double>>& epi) {
  const int m = (int)epi.size();
  for (int j = 0; j < m; ++j) {
    const int r = vjp_reads(epi[j].first);
    if (r == 1) return true;               // the operand: z or an intermediate
    if (r == 2 && j + 1 < m) return true;  // an intermediate result
  }
  return false;
}

CodegenOut gen_adj_kernel(const GraphImpl& g, const Group& G) {
  NameScope names;
  const Node& n = g.nodes[G.st_out];
  const int T = G.dtype;
  const int K = (int)n.chain.size();
  const int nd = (int)G.shape.size();
  const int ry = nd == 1 ? 0 : G.radius[1], rx = G.radius[2];
  const int TX = G.tile[2], TY = nd == 1 ? 1 : G.tile[1];
  const int PW = TX + 4 * K * rx, PH = TY + 4 * K * ry;
  bool needz = false;
  for (const AdjStep& st : n.chain) needz = needz || adj_needs_z(st.epi);
  std::ostringstream os;
  os << "// dcp time-tiled reverse stencil kernel: " << K << " steps per launch, bc " << G.bc << ", "
     << nd << "-D\n";
  os << "#define DCP_T " << dtype_cname(T) << "\n#define DCP_THREADS " << G.threads
     << "\n#define DCP_BC " << G.bc << "\n#define DCP_TX " << TX << "\n#define DCP_TY " << TY
     << "\n#define DCP_RX " << rx << "\n#define DCP_RY " << ry << "\n#define DCP_K " << K
     << "\n#define DCP_NEEDZ " << (needz ? 1 : 0) << "\n";
  os << "#include \"dcp_device.cuh\"\n";
  MulRegs km;
  km.on = T == DCP_F64;
  std::ostringstream fn;  // emitted after the multiplier table they use
  for (int s = 0; s < K; ++s) {
    const AdjStep& st = n.chain[s];
    for (int dir = 0; dir < 2; ++dir) {  // 0: forward sum, 1: transposed sum
      fn << "template <> __device__ __forceinline__ DCP_T " << (dir ? "dcp_bsum<" : "dcp_fsum<") << s
         << ">(const DCP_T* A, int c, const DCP_T (&km)[DCP_NK]) {\n  (void)km;\n";
      std::vector<int32_t> offs = G.offsets;  // transposed: negated offsets
      if (dir)
        for (auto& o : offs) o = -o;
      emit_sum_cell(fn, T, plan_sum2(offs, st.weights, Defer()), offs, [&](int dy, int dx) {
        return "A[c + (" + std::to_string(dy * PW + dx) + ")]";
      }, km);
      fn << "  return acc;\n}\n";
    }
    // forward epilogue
    fn << "template <> __device__ __forceinline__ DCP_T dcp_fepi<" << s << ">(DCP_T v) {\n";
    fn << epi_chain(st.epi, T) << "}\n";
    // reverse of the epilogue: intermediates recomputed from z when read
    fn << "template <> __device__ __forceinline__ DCP_T dcp_vjp<" << s
       << ">(DCP_T g, DCP_T z, DCP_T u) {\n  (void)z; (void)u;\n";
    const int m = (int)st.epi.size();
    std::vector<Ex> val(m + 1);  // val[0] = z, val[j] = result of op j-1
    val[0].s = "z";
    const bool need = adj_needs_z(st.epi);
    for (int j = 0; j < m; ++j) {
      if (need && j + 1 < m) {
        val[j + 1] = ex_op(st.epi[j].first, T, st.epi[j].second, val[j], Ex());
        fn << "  const DCP_T f" << j << " = " << val[j + 1].s << ";\n";
        val[j + 1].s = "f" + std::to_string(j);
      }
    }
    if (m > 0) val[m] = Ex(), val[m].s = "u";
    std::string a = "g";
    for (int j = m - 1; j >= 0; --j) {
      std::string nv = "a" + std::to_string(j);
      fn << "  const DCP_T " << nv << " = "
         << vjp_expr(st.epi[j].first, st.epi[j].second, T, a, val[j].s, val[j + 1].s) << ";\n";
      a = nv;
    }
    fn << "  return " << a << ";\n}\n";
  }
  os << km.table();
  os << "template <int S> __device__ __forceinline__ DCP_T dcp_fsum(const DCP_T* A, int c, const "
        "DCP_T (&km)[DCP_NK]);\n"
     << "template <int S> __device__ __forceinline__ DCP_T dcp_bsum(const DCP_T* A, int c, const "
        "DCP_T (&km)[DCP_NK]);\n"
     << "template <int S> __device__ __forceinline__ DCP_T dcp_fepi(DCP_T v);\n"
     << "template <int S> __device__ __forceinline__ DCP_T dcp_vjp(DCP_T g, DCP_T z, DCP_T u);\n";
  os << fn.str();
  os << "#include \"k_stencil_adj.cuh\"\n";
  CodegenOut out;
  out.threads = G.threads;
  out.smem_bytes = (K + 1 + (needz ? K : 0)) * PW * PH * dtype_size(T);
  out.source = finish("dcp_adj", os.str());
  out.name = kname_of(out.source);
  return out;
}

}  // namespace dcp
