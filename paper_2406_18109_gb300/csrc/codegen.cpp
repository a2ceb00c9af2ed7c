// codegen.cpp -- CUDA source for one launch group.
//
// The fused task body is the composition of the task bodies in program order
// (Section 4.2.2); loops of consecutive tasks with the same iteration space
// are fused and their temporaries become registers (Section 6.3, Fig. 8:
// compose, eliminate temporaries, fuse and parallelise loops, remove local
// allocations).  On the GPU:
//   * the launch domain is the set of work units (points); CTAs take points
//     in grid-stride order, so a fused group needs no communication between
//     CTAs (the fusion constraints guarantee point-wise dependencies);
//   * a launch holding several fused groups (persistent mode) separates them
//     by grid barriers wherever the previous group was not a replicated
//     scalar group; scalar groups (all stores 0-d) run redundantly in every
//     CTA on register copies of the 0-d values (after a barrier, on warp 0
//     with a shared-memory broadcast to the rest of the CTA);
//   * reductions keep one partial per point, finished in a fixed order after
//     the next barrier (or by the last CTA to exit), so every result is
//     reproducible and identical between fused and unfused execution.
// Every shape, tile and offset is a compile-time constant of the generated
// source; pointers and immediate values are kernel parameters, so isomorphic
// windows share one compiled kernel (Section 5.2).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <functional>
#include <sstream>
#include <stdexcept>
#include <tuple>

#include "runtime.hpp"

namespace dfs {

size_t dtype_size(int dt) {
  switch (dt) {
    case DFS_F32: return 4;
    case DFS_F64: return 8;
    case DFS_I32: return 4;
    case DFS_I64: return 8;
  }
  return 0;
}
const char* dtype_cname(int dt) {
  switch (dt) {
    case DFS_F32: return "float";
    case DFS_F64: return "double";
    case DFS_I32: return "int";
    case DFS_I64: return "long long";
  }
  return "void";
}
bool dtype_is_float(int dt) { return dt == DFS_F32 || dt == DFS_F64; }

namespace {

const char* op_fn(int op) {
  switch (op) {
    case DFS_OP_COPY: return "op_copy";
    case DFS_OP_NEG: return "op_neg";
    case DFS_OP_ABS: return "op_abs";
    case DFS_OP_EXP: return "op_exp";
    case DFS_OP_LOG: return "op_log";
    case DFS_OP_SQRT: return "op_sqrt";
    case DFS_OP_ERF: return "op_erf";
    case DFS_OP_NCDF: return "op_ncdf";
    case DFS_OP_ADD: return "op_add";
    case DFS_OP_SUB: return "op_sub";
    case DFS_OP_MUL: return "op_mul";
    case DFS_OP_DIV: return "op_div";
    case DFS_OP_POW: return "op_pow";
    case DFS_OP_MAX: return "op_max";
    case DFS_OP_MIN: return "op_min";
  }
  return nullptr;
}

bool is_elementwise(int op) { return op_fn(op) != nullptr; }
bool is_reduction(int op) { return op == DFS_OP_DOT || op == DFS_OP_SUM; }

// The argument whose sub-store drives the task's loop.
const Arg& space_arg(const Task& t) {
  if (is_reduction(t.op)) return t.args[0];
  if (t.op == DFS_OP_SPMV) return t.args[4];
  return t.args.back();
}

std::string akey(const Arg& a) { return std::to_string(a.root) + "@" + a.part.key(); }

struct Nest {
  int first, last;  // task indices [first, last)
  int dims;         // 1 (flat) or 2 (row loop)
  int vec;          // elements per vector access
  int rank = 1;     // rank of the iteration space (rows of a 3-D space are (plane, row) pairs)
  bool coop = false;  // an SpMV of the nest uses several lanes per row (spmv_warp)
  bool rows = false;  // the nest's SpMVs are computed a warp's rows at a time (spmv_rows)
  // realigned rows: vectors in the frame of the written views (`head` scalar
  // columns first); a read view whose column origin is `shift` elements past
  // that frame is loaded as two aligned vectors
  bool realign = false;
  int head = 0;
  std::map<std::string, int> shift;
};

// Whether an FP32 SpMV's rows are computed a warp's rows at a time (spmv_rows)
// or one per lane (spmv_row); the bits are the same.  spmv_rows wins as a rule
// (1M rows of 7 entries 58 -> 38 us, of 31 253 -> 160) and by far where rows
// differ in length, but not
//  * for rows of one entry over several million rows, nothing to coalesce (4M
//    rows: 18.0 us a lane each, 21.1 a warp's at a time);
//  * for a few points of long rows: a warp's chunks come one after another (40000
//    rows of 31 entries in 157 points 18.8, 21.8);
//  * in CTAs of more than 256 threads, whose registers (48 against 32) leave half
//    as many CTAs per SM, when the points then take another round and keep few
//    warps busy (100000 rows of 31 in 391 points, 512 threads 26, 41), at 1024
//    threads also for short rows (1M rows of 5 18.6, 22.0; of 16 133, 93).
bool rows_pay(const Task& t, int block, int sms) {
  const Arg& y = t.args[4];
  if (y.dtype != DFS_F32) return false;
  const int64_t nnz = t.args[1].part.vhi[0] - t.args[1].part.vlo[0], points = t.npoints();
  const int64_t rows = t.args[0].part.vhi[0] - t.args[0].part.vlo[0] - 1, tile = y.part.kind == 1 ? y.part.tile[0] : rows;
  if (rows >= (1 << 21) && nnz < 2 * rows) return false;
  if (points * 4 <= sms * 5 && nnz >= 24 * rows && rows > 0) return false;
  if (block <= 256 || points * block <= (int64_t)sms * 1024) return true;
  return tile >= block && (block < 1024 || nnz >= 8 * rows);
}

// Lanes per row of an SpMV task's matrix (col and rowptr extents).
int spmv_k(const Task& t) {
  const NPart& c = t.args[1].part;
  const NPart& r = t.args[0].part;
  return spmv_lanes(c.vhi[0] - c.vlo[0], r.vhi[0] - r.vlo[0] - 1);
}

class Gen {
 public:
  explicit Gen(const LaunchSpec& s) : S(s) {}

  KernelCode run();

  // How the loop nests of group g sweep their space (empty: several nests).
  std::string form(int g) {
    const std::vector<Nest> v = nests_of(g);
    if (v.size() != 1) return std::string();
    return std::to_string(v[0].dims) + "," + std::to_string(v[0].vec) + "," + std::to_string(v[0].realign) + "," +
           std::to_string(v[0].head);
  }

 private:
  const LaunchSpec& S;
  std::ostringstream o;
  KernelCode kc;
  std::map<int64_t, int> ptr_of;          // root -> pointer param index
  std::map<int64_t, std::string> sreg;    // 0-d root -> register name
  std::map<int64_t, bool> have;           // 0-d root holds a value in registers
  struct Red { int slot; int64_t root; int dtype; int64_t points; };
  std::vector<Red> pending_red;           // reductions awaiting finalisation
  int nbar = 0;
  int nbc = 0;  // shared broadcast slots of finished reductions
  bool stage = false;  // some per-point SpMV nest stages x windows in shared memory
  int wave_blocks = 0;  // CTAs per SM an in-place sweep needs resident

  const LaunchRoot& R(int64_t root) const { return S.roots[S.root_index.at(root)]; }
  bool temp_in(int g, int64_t root) const;
  std::string ptr(int64_t root) const { return "r" + std::to_string(ptr_of.at(root)); }
  std::string T(int dt) const { return dtype_cname(dt); }

  void emit_params();
  void emit_prologue();
  void emit_group(int g);
  void emit_scalar_group(int g);
  void emit_vector_group(int g);
  // memory reads of a loop nest: distinct (root, partition) read before any
  // in-nest write of it; reduction accumulators
  struct Rd { std::string key; const Arg* a; std::string var; bool ro; };
  struct Acc { int task; int slot; std::string var; int dt; };
  // What the body of a nest needs besides its loads: names of the base
  // offsets and immediates, SpMV values computed before the body, the SpMV
  // task that reads staged x windows.
  struct BodyEnv {
    std::vector<Rd> reads;
    std::vector<Acc> accs;
    std::map<std::string, std::string> base;
    std::map<std::pair<int, int>, std::string> immv;
    std::map<int, std::string> spre;
    int staged = -1;
  };
  void emit_nest(int g, const Nest& n, const std::string& red_pt, bool flat);
  std::map<std::string, std::vector<std::string>> emit_compute(const Nest& n, const BodyEnv& E, int w,
                                                               const std::vector<std::string>& slots,
                                                               const std::vector<std::string>& eflat,
                                                               const std::string& pad);
  void emit_wave(int g);
  // test hook: CTA 0 withholds the context's flag number -debug_skip
  std::string raises(const std::string& flag) const {
    return S.debug_skip < 0 ? ", blockIdx.x != 0 || " + flag + " != " + std::to_string(-(int64_t)S.debug_skip) + "ull" : std::string();
  }
  void emit_march(int g, int sweeps);
  std::string sweep_signature(int g) const;
  // Which tasks of nest n run two lanes per instruction in a body of w lanes
  // (index: task - n.first).
  std::vector<char> packed_tasks(const Nest& n, int w) const;
  // which phases use a store; sweeps that come back to one (emit_nest)
  bool uses(int h, int64_t root) const;
  int users(int64_t root) const;
  bool revisits(int g, const Nest& n) const;
  bool swept_after(int g, int h);
  void emit_finalise(const char* indent);
  int emit_warp0_scalars(int g);
  void realign(Nest& n, int vec);
  std::vector<Nest> nests_of(int g);
  std::string imm_expr(int task, int arg, int dt);
};

bool Gen::temp_in(int g, int64_t root) const {
  (void)g;
  const LaunchRoot& r = R(root);
  return r.temp;
}

std::string Gen::imm_expr(int task, int arg, int dt) {
  const int k = kc.nimm++;
  kc.imms.push_back(S.tasks[task].args[arg].immv);
  kc.imm_src.push_back({task, arg});
  return "((" + T(dt) + ")P.imm[" + std::to_string(k) + "])";
}

void Gen::emit_params() {
  // pointer params: every root with memory
  for (const LaunchRoot& r : S.roots) {
    if (r.param < 0) continue;
    ptr_of[r.root] = r.param;
  }
  kc.nptr = 0;
  for (const LaunchRoot& r : S.roots)
    if (r.param >= 0) kc.nptr = std::max(kc.nptr, r.param + 1);
  kc.ptr_roots.assign(kc.nptr, 0);
  for (const LaunchRoot& r : S.roots)
    if (r.param >= 0) kc.ptr_roots[r.param] = r.root;
}

void Gen::emit_prologue() {
  // typed root pointers
  for (const LaunchRoot& r : S.roots) {
    if (r.param < 0) continue;
    o << "  " << T(r.dtype) << "* __restrict__ " << ptr(r.root) << " = (" << T(r.dtype) << "*)P.p["
      << r.param << "];\n";
  }
  // 0-d registers
  int k = 0;
  for (const LaunchRoot& r : S.roots) {
    if (!r.zero_d) continue;
    const std::string nm = "s" + std::to_string(k++);
    sreg[r.root] = nm;
    const bool load = r.valid_before && r.param >= 0;
    o << "  " << T(r.dtype) << " " << nm << " = " << (load ? "ld(" + ptr(r.root) + ")" : T(r.dtype) + "(0)")
      << ";\n";
    have[r.root] = load;
  }
}

// Row nests whose views start at different column offsets (the shifted
// views of a stencil) still use vector accesses when every root row is a
// whole number of aligned vectors and no reduction's summation order would
// change: the nest iterates in the vector frame of its written views.
void Gen::realign(Nest& n, int vec) {
  int mw = -1, mr = -1;
  size_t esz = 0;
  std::map<std::string, int> phase;
  for (int t = n.first; t < n.last; ++t) {
    const Task& tk = S.tasks[t];
    if (tk.scalar()) continue;
    if (is_reduction(tk.op) || tk.op == DFS_OP_SPMV) return;
    for (size_t ai = 0; ai < tk.args.size(); ++ai) {
      const Arg& a = tk.args[ai];
      if (a.imm || a.nd == 0) continue;
      const LaunchRoot& r = R(a.root);
      if (r.temp) continue;  // lives in registers
      if (esz && esz != dtype_size(a.dtype)) return;
      esz = dtype_size(a.dtype);
      const int cd = a.nd - 1;
      if (!r.aligned16 || a.part.kind != 1 || tk.dom[a.part.proj[cd]] != 1) return;
      for (int d = 0; d < cd; ++d)
        if (r.stride[d] % vec) return;
      const int64_t c0 = std::max(a.part.off[cd], a.part.vlo[cd]);
      const int ph = (int)(((c0 % vec) + vec) % vec);
      phase[akey(a)] = ph;
      const bool out = is_elementwise(tk.op) && ai + 1 == tk.args.size();
      if (out) {
        if (mw >= 0 && mw != ph) return;
        mw = ph;
      } else if (mr < 0) {
        mr = ph;
      }
    }
  }
  if (!esz || (int)(16 / esz) != vec) return;
  n.realign = true;
  n.vec = vec;
  n.head = (vec - (mw >= 0 ? mw : std::max(mr, 0))) % vec;
  for (const auto& kv : phase) n.shift[kv.first] = (kv.second + n.head) % vec;
}

std::vector<Nest> Gen::nests_of(int g) {
  const Group& G = S.groups[g];
  std::vector<Nest> v;
  int i = G.begin;
  while (i < G.end && S.tasks[i].scalar()) ++i;  // scalar tasks are hoisted
  while (i < G.end) {
    const std::string key = iteration_space_key(S.tasks[i]);
    int j = i + 1;
    while (j < G.end && (S.tasks[j].scalar() || iteration_space_key(S.tasks[j]) == key)) ++j;
    Nest n;
    n.first = i;
    n.last = j;
    // dimensionality and vector width
    const Arg& sa = space_arg(S.tasks[i]);
    const int nd = sa.nd;
    // collapse a 2-D or 3-D space into a flat one when every access spans
    // whole root rows (and planes): its elements are then contiguous
    bool flat = nd <= 1;
    if (nd >= 2) {
      flat = true;
      for (int t = i; t < j && flat; ++t)
        for (const Arg& a : S.tasks[t].args) {
          if (a.imm || a.nd == 0) continue;
          if (S.tasks[t].op == DFS_OP_SPMV && &a != &S.tasks[t].args[4]) continue;
          const LaunchRoot& r = R(a.root);
          if (a.part.kind != 1) flat = false;
          for (int d = 1; d < nd && flat; ++d)
            if (a.part.vlo[d] != 0 || a.part.vhi[d] != r.shape[d] || a.part.off[d] > 0 ||
                a.part.tile[d] < r.shape[d] || r.stride[d - 1] != r.shape[d] * r.stride[d])  // no row padding
              flat = false;
        }
    }
    if (nd > 3) throw std::runtime_error("iteration spaces of rank > 3 are not supported");
    // rows mode: ext0 rows (2-D) or ext0 x ext1 rows (3-D) of the last dimension
    n.dims = flat ? 1 : 2;
    n.rank = nd;
    // widest element over the memory accesses of the nest
    size_t esz = 0;
    bool aligned = true;
    for (int t = i; t < j; ++t) {
      const Task& tk = S.tasks[t];
      for (size_t ai = 0; ai < tk.args.size(); ++ai) {
        const Arg& a = tk.args[ai];
        if (a.imm || a.nd == 0) continue;
        if (tk.op == DFS_OP_SPMV && ai != 4) continue;  // gathered, not streamed
        esz = std::max(esz, dtype_size(a.dtype));
      }
    }
    int vec = esz ? (int)(16 / esz) : 1;
    for (int t = i; t < j && vec > 1; ++t) {
      const Task& tk = S.tasks[t];
      for (size_t ai = 0; ai < tk.args.size(); ++ai) {
        const Arg& a = tk.args[ai];
        if (a.imm || a.nd == 0) continue;
        if (tk.op == DFS_OP_SPMV && ai != 4) continue;
        const LaunchRoot& r = R(a.root);
        if ((int)(16 / dtype_size(a.dtype)) != vec) aligned = false;
        if (!r.temp && !r.aligned16) aligned = false;
        if (n.dims == 1) {
          for (int d = 0; d < a.nd; ++d) {
            const int64_t st = r.stride[d];
            if ((a.part.tile[d] * st) % vec || (a.part.off[d] * st) % vec || (a.part.vlo[d] * st) % vec)
              aligned = false;
          }
        } else {
          const int cd = a.nd - 1;  // the column dimension
          for (int d = 0; d < cd; ++d)
            if (r.stride[d] % vec) aligned = false;
          if (a.part.tile[cd] % vec || a.part.off[cd] % vec || a.part.vlo[cd] % vec ||
              (a.part.vhi[cd] - a.part.vlo[cd]) % vec)
            aligned = false;
        }
      }
    }
    n.vec = aligned ? vec : 1;
    if (!aligned && vec > 1 && n.dims == 2) realign(n, vec);
    for (int t = i; t < j; ++t)
      if (S.tasks[t].op == DFS_OP_SPMV && spmv_k(S.tasks[t]) > 1) n.coop = true;
    for (int t = i; t < j; ++t)
      if (S.tasks[t].op == DFS_OP_SPMV && !n.coop && n.dims == 1 && rows_pay(S.tasks[t], S.block, S.sms)) n.rows = true;
    v.push_back(n);
    i = j;
    while (i < G.end && S.tasks[i].scalar()) ++i;
  }
  return v;
}

void Gen::emit_group(int g) {
  if (S.groups[g].scalar)
    emit_scalar_group(g);
  else
    emit_vector_group(g);
}

// A group of scalar tasks, evaluated on the register copies of the 0-d
// stores: by every thread at the start of a launch, by warp 0 after a grid
// barrier (emit_warp0_scalars).
void Gen::emit_scalar_group(int g) {
  const Group& G = S.groups[g];
  o << "    { // group " << g << " (scalar)\n";
  for (int i = G.begin; i < G.end; ++i) {
    const Task& t = S.tasks[i];
    const Arg& out = t.args.back();
    const int dt = out.dtype;
    std::vector<std::string> ins;
    for (size_t k = 0; k + 1 < t.args.size(); ++k) {
      const Arg& a = t.args[k];
      if (a.imm) ins.push_back(imm_expr(i, (int)k, dt));
      else ins.push_back("(" + T(dt) + ")" + sreg.at(a.root));
    }
    o << "      " << sreg.at(out.root) << " = " << op_fn(t.op) << "(";
    for (size_t k = 0; k < ins.size(); ++k) o << (k ? ", " : "") << ins[k];
    o << ");\n";
    have[out.root] = true;
  }
  o << "    }\n";
}

void Gen::emit_vector_group(int g) {
  const Group& G = S.groups[g];
  const Task& t0 = S.tasks[G.begin];
  const int64_t npts = t0.npoints();
  // Scalar tasks can share a group with vector tasks when the launch domain
  // has a single point.  They read and write 0-d values only, so every CTA
  // evaluates them first, in program order (the one point may run anywhere);
  // this is exact unless a vector task earlier in the group reads a value a
  // later scalar task overwrites.
  for (int i = G.begin; i < G.end; ++i) {
    if (!S.tasks[i].scalar()) continue;
    const int64_t out = S.tasks[i].args.back().root;
    for (int j = G.begin; j < i; ++j)
      if (!S.tasks[j].scalar())
        for (const Arg& a : S.tasks[j].args)
          if (!a.imm && a.root == out)
            throw std::runtime_error("a scalar task overwrites a value read earlier in its group");
    const Task& t = S.tasks[i];
    const int dt = t.args.back().dtype;
    std::vector<std::string> ins;
    for (size_t k = 0; k + 1 < t.args.size(); ++k) {
      const Arg& a = t.args[k];
      ins.push_back(a.imm ? imm_expr(i, (int)k, dt) : "(" + T(dt) + ")" + sreg.at(a.root));
    }
    o << "    " << sreg.at(t.args.back().root) << " = " << op_fn(t.op) << "(";
    for (size_t k = 0; k < ins.size(); ++k) o << (k ? ", " : "") << ins[k];
    o << ");\n";
    have[t.args.back().root] = true;
  }
  std::vector<Nest> nests = nests_of(g);
  // A group with one loop nest and no reduction needs no per-point
  // structure: the union of the points' sub-stores is one rectangle of
  // contiguous tiles (every operand has the same tile shape and offsets
  // relative to its view), so it is swept as one range with a grid stride,
  // which balances the work across CTAs at element granularity.
  bool flat = nests.size() == 1;
  for (int i = G.begin; i < G.end && flat; ++i)
    if (is_reduction(S.tasks[i].op)) flat = false;
  if (flat && space_arg(t0).nd > 3) flat = false;
  if (flat) {
    kc.has_flat = true;
    o << "    { // group " << g << ": tasks " << G.begin << ".." << G.end - 1 << ", one flat nest over "
      << npts << " points\n";
    emit_nest(g, nests[0], "", true);
    o << "    }\n";
    return;
  }
  kc.has_points = true;
  kc.max_points = std::max(kc.max_points, npts);
  o << "    { // group " << g << ": tasks " << G.begin << ".." << G.end - 1 << ", " << nests.size()
    << " loop nest(s), " << npts << " points\n";
  o << "      for (i64 pt = blockIdx.x; pt < " << npts << "LL; pt += gridDim.x) {\n";
  // point coordinates
  {
    int64_t rem = 1;
    for (int d = t0.dnd - 1; d >= 0; --d) {
      o << "        const i64 q" << d << " = (pt / " << rem << "LL) % " << t0.dom[d] << "LL;\n";
      rem *= t0.dom[d];
    }
  }
  for (size_t k = 0; k < nests.size(); ++k) {
    if (k) o << "        __syncthreads();\n";
    emit_nest(g, nests[k], "pt", false);
  }
  o << "      }\n";
  o << "    }\n";
}

// FP32 element-wise ADD, NCDF, ERF and LOG tasks run two lanes per
// instruction (pk_add, pk_ncdf_*, erf_mag2, log_f32x2) when that cannot change
// a bit.  The compiler contracts a packed product whose value reaches a sum
// into a fused multiply-add, so an NCDF (whose last step multiplies) whose
// value, possibly negated or copied on the way, reaches a sum of the body
// (ADD, SUB, a SUM reduction) keeps both operations scalar, and so does a sum
// of a MUL.  ERF and LOG are neither products nor sums (inside, their products
// reach sums only through explicit fused multiply-adds), so they always pair
// up.  MUL itself stays on single lanes: a packed multiply saves an issue slot
// but waits on the packed pipe, and measured on the fused Black-Scholes
// window, multiplies on lane pairs made the kernel 0.9 % slower.  Values
// loaded from memory or computed outside the body are not products of the
// body.
std::vector<char> Gen::packed_tasks(const Nest& n, int w) const {
  std::vector<char> pk(n.last - n.first, 0);
  if (w < 2 || w % 2) return pk;
  std::map<std::string, int> product_of;  // akey -> task whose product the value is
  std::vector<char> blocked(n.last - n.first, 0);
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    if (t.scalar()) continue;
    const bool sum = t.op == DFS_OP_ADD || t.op == DFS_OP_SUB || t.op == DFS_OP_SUM;
    const size_t nin = t.op == DFS_OP_SPMV ? 0 : t.args.size() - 1;
    int carried = -1;  // a product passed on by NEG or COPY
    for (size_t ai = 0; ai < nin; ++ai) {
      const Arg& a = t.args[ai];
      if (a.imm || a.nd == 0) continue;
      auto it = product_of.find(akey(a));
      if (it == product_of.end()) continue;
      if (sum) {
        blocked[it->second - n.first] = 1;
        blocked[i - n.first] = 1;
      }
      if (t.op == DFS_OP_NEG || t.op == DFS_OP_COPY) carried = it->second;
    }
    if (!is_elementwise(t.op)) continue;
    const std::string out = akey(t.args.back());
    product_of.erase(out);
    if (t.op == DFS_OP_MUL || t.op == DFS_OP_NCDF) product_of[out] = i;
    else if (carried >= 0) product_of[out] = carried;
  }
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    if (t.scalar() || blocked[i - n.first] || space_arg(t).dtype != DFS_F32) continue;
    pk[i - n.first] = t.op == DFS_OP_ADD || t.op == DFS_OP_NCDF || t.op == DFS_OP_ERF || t.op == DFS_OP_LOG;
  }
  return pk;
}

// The tasks of a nest over `slots` groups of w lanes, in program order, on
// values the caller has loaded as <read var>_<slot>.  Returns, per (root,
// partition) to store, the value names by slot * w + lane.
std::map<std::string, std::vector<std::string>> Gen::emit_compute(const Nest& n, const BodyEnv& E, int w,
                                                                  const std::vector<std::string>& slots,
                                                                  const std::vector<std::string>& eflat,
                                                                  const std::string& pad) {
  const int ns = (int)slots.size();
  // compute: per slot, tasks in program order, each over the lanes
  const std::vector<char> pk = packed_tasks(n, w);
  std::map<std::string, std::vector<std::string>> outvars;  // akey -> per (slot*w+lane) value
  for (int s = 0; s < ns; ++s) {
    std::vector<std::map<std::string, std::string>> curs(w);  // per lane: akey -> value expr
    std::vector<LaneOps> lanes(w);
    for (int l = 0; l < w; ++l)
      for (const Rd& rd : E.reads) {
        const std::string v = rd.var + "_" + slots[s];
        curs[l][rd.key] = (w > 1) ? v + ".v[" + std::to_string(l) + "]" : v;
      }
    for (int i = n.first; i < n.last; ++i) {
      const Task& t = S.tasks[i];
      if (t.scalar()) continue;
      const int dt = space_arg(t).dtype;   // the output's (y for an SpMV, whose last arg may be its windows)
      auto res_of = [&](int l) { return "v" + std::to_string(i) + "_" + slots[s] + "_" + std::to_string(l); };
      auto val_of = [&](int l, size_t ai) -> std::string {
        const Arg& a = t.args[ai];
        if (a.imm) return E.immv.at({i, (int)ai});
        if (a.nd == 0) return "(" + T(dt) + ")" + sreg.at(a.root);
        return curs[l].at(akey(a));
      };
      if (pk[i - n.first]) {
        // two lanes per instruction
        for (int l = 0; l < w; l += 2) {
          const std::string r0 = res_of(l), r1 = res_of(l + 1), pr = r0 + "_p";
          if (t.op == DFS_OP_NCDF || t.op == DFS_OP_ERF) {
            lanes[l].define(r0);
            lanes[l + 1].define(r1);
            const std::string a0 = val_of(l, 0), a1 = val_of(l + 1, 0);
            // the argument of erf: x / sqrt 2 for NCDF, x itself for ERF
            std::string y0 = a0, y1 = a1;
            if (t.op == DFS_OP_NCDF) {
              const std::string y = r0 + "_y2";
              o << pad << "const float2 " << y << " = pk_ncdf_arg(" << a0 << ", " << a1 << ");\n";
              y0 = y + ".x";
              y1 = y + ".y";
            }
            // erf(|y|) of both lanes in one packed evaluation, unless the
            // lanes reuse the magnitude of a negation (both do, or neither)
            std::string m0 = lanes[l].mag_of(t.op, a0), m1 = lanes[l + 1].mag_of(t.op, a1);
            if (m0.empty() && m1.empty()) {
              o << pad << "const float2 " << r0 << "_m2 = erf_mag2(" << y0 << ", " << y1 << ");\n";
              m0 = r0 + "_m2.x";
              m1 = r0 + "_m2.y";
            } else {
              if (m0.empty()) {
                m0 = r0 + "_m";
                o << pad << "const float " << m0 << " = erf_mag(" << y0 << ");\n";
              }
              if (m1.empty()) {
                m1 = r1 + "_m";
                o << pad << "const float " << m1 << " = erf_mag(" << y1 << ");\n";
              }
            }
            lanes[l].set_mag(t.op, a0, m0);
            lanes[l + 1].set_mag(t.op, a1, m1);
            if (t.op == DFS_OP_NCDF)
              o << pad << "const float2 " << pr << " = pk_ncdf_of_erf(erf_sign(" << m0 << ", " << y0 << "), erf_sign("
                << m1 << ", " << y1 << "));\n";
            else
              o << pad << "const float2 " << pr << " = make_float2(erf_sign(" << m0 << ", " << y0 << "), erf_sign("
                << m1 << ", " << y1 << "));\n";
          } else if (t.op == DFS_OP_LOG) {
            lanes[l].define(r0);
            lanes[l + 1].define(r1);
            o << pad << "const float2 " << pr << " = log_f32x2(" << val_of(l, 0) << ", " << val_of(l + 1, 0) << ");\n";
          } else {
            lanes[l].define(r0);
            lanes[l + 1].define(r1);
            o << pad << "const float2 " << pr << " = pk_add(" << val_of(l, 0) << ", " << val_of(l + 1, 0) << ", "
              << val_of(l, 1) << ", " << val_of(l + 1, 1) << ");\n";
          }
          o << pad << "const float " << r0 << " = " << pr << ".x;\n";
          o << pad << "const float " << r1 << " = " << pr << ".y;\n";
          curs[l][akey(t.args.back())] = r0;
          curs[l + 1][akey(t.args.back())] = r1;
        }
        continue;
      }
      for (int l = 0; l < w; ++l) {
        auto& cur = curs[l];
        LaneOps& lane = lanes[l];
        auto val = [&](size_t ai) { return val_of(l, ai); };
        const std::string res = res_of(l);
        if (is_elementwise(t.op)) {
          std::vector<std::string> in{val(0)};
          if (t.args.size() == 3) in.push_back(val(1));
          lane.emit(o, pad, T(dt), t.op, res, in);
          cur[akey(t.args.back())] = res;
        } else if (t.op == DFS_OP_SPMV && E.spre.count(i)) {
          o << pad << "const " << T(dt) << " " << res << " = " << E.spre.at(i) << "_" << l << ";\n";
          cur[akey(t.args[4])] = res;
        } else if (t.op == DFS_OP_SPMV) {
          const Arg& y = t.args[4];
          const std::string row = "(" + E.base.at(akey(y)) + " - " + std::to_string(y.part.vlo[0]) + "LL + " +
                                  eflat[s] + " + " + std::to_string(l) + ")";
          o << pad << "const " << T(dt) << " " << res << " = " << (i == E.staged ? "spmv_row_xs<" : "spmv_row<")
            << T(dt) << ">(" << ptr(t.args[0].root) << " + " << E.base.at(akey(t.args[0])) << ", "
            << ptr(t.args[1].root) << " + " << E.base.at(akey(t.args[1])) << ", " << ptr(t.args[2].root) << " + "
            << E.base.at(akey(t.args[2])) << ", " << ptr(t.args[3].root) << " + " << E.base.at(akey(t.args[3])) << ", "
            << row << (i == E.staged ? ", (const " + T(dt) + "*)dfs_xs_raw, xw_" : std::string()) << ");\n";
          cur[akey(y)] = res;
        } else if (is_reduction(t.op)) {
          const Acc* ac = nullptr;
          for (const Acc& x : E.accs)
            if (x.task == i) ac = &x;
          if (t.op == DFS_OP_DOT)
            o << pad << ac->var << " = red_fma(" << val(0) << ", " << val(1) << ", " << ac->var << ");\n";
          else
            o << pad << ac->var << " = " << ac->var << " + " << val(0) << ";\n";
        }
      }
    }
    // collect outputs to store
    for (int l = 0; l < w; ++l)
      for (int i = n.first; i < n.last; ++i) {
        const Task& t = S.tasks[i];
        if (t.scalar()) continue;
        const Arg* out = nullptr;
        if (is_elementwise(t.op)) out = &t.args.back();
        if (t.op == DFS_OP_SPMV) out = &t.args[4];
        if (!out || R(out->root).temp) continue;
        const std::string k = akey(*out);
        auto& vv = outvars[k];
        if (vv.size() < (size_t)(ns * w)) vv.resize(ns * w);
        vv[s * w + l] = curs[l].at(k);
      }
  }
  return outvars;
}

bool Gen::uses(int h, int64_t root) const {
  for (int i = S.groups[h].begin; i < S.groups[h].end; ++i)
    for (const Arg& a : S.tasks[i].args)
      if (!a.imm && a.nd > 0 && a.root == root) return true;
  return false;
}
int Gen::users(int64_t root) const {
  int k = 0;
  for (int h = 0; h < (int)S.groups.size(); ++h) k += uses(h, root) ? 1 : 0;
  return k;
}
// Nest n of group g reads an array that the last sweep before it used, and runs
// backwards over it: x + s with 3 y after a sum of x, 2^24 FP32 elements, 59.5 ->
// 54.7 us.  FP64 sweeps are bound by their pipe and lose by the addresses once
// their own arrays do not stay in L2 (2^24 elements 131.7 -> 140.4, 4M 39.4 ->
// 40.7; 2M 26.4 -> 25.1, CG at 1337^2 743 -> 736 us per ten iterations).
bool Gen::revisits(int g, const Nest& n) const {
  std::set<int64_t> arrays;
  int64_t bytes = 0;
  for (int i = n.first; i < n.last; ++i)
    for (const Arg& a : S.tasks[i].args) {
      if (a.imm || a.nd == 0 || R(a.root).temp || !arrays.insert(a.root).second) continue;
      int64_t e = (int64_t)dtype_size(a.dtype);
      for (int d = 0; d < a.nd; ++d) e *= R(a.root).shape[d];
      bytes += e;
    }
  if (space_arg(S.tasks[n.first]).dtype != DFS_F32 && bytes > 96000000) return false;
  int h = g - 1;
  while (h >= 0 && S.groups[h].scalar) --h;
  if (h < 0) return false;
  for (int i = n.first; i < n.last; ++i)
    for (const Arg& a : S.tasks[i].args)
      if (!a.imm && a.nd > 0 && a.is_r() && !R(a.root).temp && uses(h, a.root)) return true;
  return false;
}
// Group h is the next sweep after g, runs backwards, and reads what g uses.
bool Gen::swept_after(int g, int h) {
  for (int k = g + 1; k < h; ++k)
    if (!S.groups[k].scalar) return false;
  for (int i = S.groups[h].begin; i < S.groups[h].end; ++i)
    if (!is_elementwise(S.tasks[i].op)) return false;
  const std::vector<Nest> v = nests_of(h);
  return v.size() == 1 && v[0].dims == 1 && revisits(h, v[0]);
}

void Gen::emit_nest(int g, const Nest& n, const std::string& ptvar, bool flat) {
  const int BD = S.block;
  const int U = std::max(1, S.unroll);
  const int V = n.vec;
  const Task& first = S.tasks[n.first];
  const Arg& sa = space_arg(first);
  const int nd = sa.nd;
  const std::string ind = "        ";
  o << ind << "{ // nest: tasks " << n.first << ".." << n.last - 1 << ", vec " << V << ", "
    << (n.dims == 1 ? "flat" : "rows") << "\n";
  // ---- per-access base offsets (root coordinates flattened)
  BodyEnv E;
  std::map<std::string, std::string>& base = E.base;  // akey -> base variable
  int nb = 0;
  auto box_lo = [&](const Arg& a, int d) {
    std::ostringstream s;
    if (a.part.kind == 0) {
      s << a.part.vlo[d] << "LL";
    } else if (flat) {
      s << std::max(a.part.off[d], a.part.vlo[d]) << "LL";
    } else {
      s << "max(q" << a.part.proj[d] << " * " << a.part.tile[d] << "LL + (" << a.part.off[d] << "LL), "
        << a.part.vlo[d] << "LL)";
    }
    return s.str();
  };
  auto need_base = [&](const Arg& a) {
    const std::string k = akey(a);
    if (base.count(k)) return base[k];
    const std::string nm = "b" + std::to_string(nb++);
    const LaunchRoot& r = R(a.root);
    o << ind << "  const i64 " << nm << " = ";
    for (int d = 0; d < a.nd; ++d) o << (d ? " + " : "") << "(" << box_lo(a, d) << ") * " << r.stride[d] << "LL";
    if (a.nd == 0) o << "0";
    o << ";\n";
    base[k] = nm;
    return nm;
  };
  // ---- extents of the iteration space
  int64_t flat_cells = 1;  // elements of a flat range (constant)
  for (int d = 0; d < nd; ++d) {
    if (sa.part.kind == 0) {
      flat_cells *= std::max<int64_t>(0, sa.part.vhi[d] - sa.part.vlo[d]);
      o << ind << "  const i64 ext" << d << " = " << (sa.part.vhi[d] - sa.part.vlo[d]) << "LL;\n";
    } else if (flat) {
      const int64_t cnt = first.dom[sa.part.proj[d]];
      const int64_t lo = std::max(sa.part.off[d], sa.part.vlo[d]);
      const int64_t hi = std::min(cnt * sa.part.tile[d] + sa.part.off[d], sa.part.vhi[d]);
      flat_cells *= std::max<int64_t>(0, hi - lo);
      o << ind << "  const i64 ext" << d << " = " << std::max<int64_t>(0, hi - lo) << "LL;\n";
    } else {
      o << ind << "  const i64 ext" << d << " = min(q" << sa.part.proj[d] << " * " << sa.part.tile[d]
        << "LL + (" << sa.part.off[d] << "LL) + " << sa.part.tile[d] << "LL, " << sa.part.vhi[d]
        << "LL) - max(q" << sa.part.proj[d] << " * " << sa.part.tile[d] << "LL + (" << sa.part.off[d]
        << "LL), " << sa.part.vlo[d] << "LL);\n";
    }
  }
  // ---- classify accesses
  // reads from memory: distinct (root, partition) read before any in-nest write of it
  std::vector<Rd>& reads = E.reads;
  std::map<std::string, int> read_idx;
  std::set<std::string> written_keys;
  std::vector<Acc>& accs = E.accs;  // reduction accumulators
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    if (t.scalar()) continue;
    for (size_t ai = 0; ai < t.args.size(); ++ai) {
      const Arg& a = t.args[ai];
      if (a.imm || a.nd == 0) continue;
      if (t.op == DFS_OP_SPMV && ai != 4) continue;
      const std::string k = akey(a);
      if (a.is_r() && !(t.op != DFS_OP_SPMV && is_elementwise(t.op) && ai + 1 == t.args.size())) {
        if (!written_keys.count(k) && !read_idx.count(k)) {
          read_idx[k] = (int)reads.size();
          const LaunchRoot& r = R(a.root);
          reads.push_back({k, &a, "m" + std::to_string(reads.size()), !r.written});
          need_base(a);
        }
      }
      const bool is_out = (is_elementwise(t.op) && ai + 1 == t.args.size()) || (t.op == DFS_OP_SPMV && ai == 4);
      if (is_out) {
        written_keys.insert(k);
        // an SpMV output's offset also gives its row index, temporary or not
        if (!R(a.root).temp || t.op == DFS_OP_SPMV) need_base(a);
      }
    }
    if (is_reduction(t.op)) {
      const Arg& out = t.args.back();
      Acc ac;
      ac.task = i;
      ac.slot = kc.nred++;
      ac.var = "acc" + std::to_string(ac.slot);
      ac.dt = out.dtype;
      accs.push_back(ac);
      kc.red_points.push_back(t.npoints());
      pending_red.push_back({ac.slot, out.root, out.dtype, t.npoints()});
      o << ind << "  " << T(ac.dt) << " " << ac.var << " = " << T(ac.dt) << "(0);\n";
    }
  }
  // SpMV gathered operands: bases of rowptr/col/val/x (None partitions)
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    if (t.scalar()) continue;
    if (t.op != DFS_OP_SPMV) continue;
    for (int ai = 0; ai < 4; ++ai) need_base(t.args[ai]);
  }
  // the first SpMV of a per-point nest that carries x windows: stage them for
  // this point (every thread of the CTA is here, at the same point)
  int& staged = E.staged;
  if (stage && !flat && n.dims == 1 && !n.coop)
    for (int i = n.first; i < n.last && staged < 0; ++i)
      if (S.tasks[i].op == DFS_OP_SPMV && S.tasks[i].args.size() == 6) staged = i;
  if (staged >= 0) {
    const Task& t = S.tasks[staged];
    const Arg& x = t.args[3];
    const std::string tn = T(x.dtype);
    const std::string wb = need_base(t.args[5]);
    o << ind << "  const XWin xw_ = xstage<" << tn << ">((" << tn << "*)dfs_xs_raw, "
      << DFS_SPMV_STAGE_BYTES / (int)dtype_size(x.dtype) << ", " << ptr(x.root) << " + " << base.at(akey(x)) << ", "
      << (x.part.vhi[0] - x.part.vlo[0]) << "LL, (const int*)" << ptr(t.args[5].root) << " + " << wb
      << ", &xs_mbar_, xs_ph_, xs_live_, ctl, P.timeout_ns);\n";
  }
  // immediates hoisted once per nest
  std::map<std::pair<int, int>, std::string>& immv = E.immv;
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    if (t.scalar()) continue;
    const int dt = t.args.back().dtype;
    for (size_t ai = 0; ai < t.args.size(); ++ai) {
      const Arg& a = t.args[ai];
      if (!a.imm) continue;
      const std::string nm = "k" + std::to_string(i) + "_" + std::to_string(ai);
      o << ind << "  const " << T(dt) << " " << nm << " = " << imm_expr(i, (int)ai, dt) << ";\n";
      immv[{i, (int)ai}] = nm;
    }
  }

  const bool by_rows = n.rows && !stage;
  // A sweep over what an earlier phase has just been through runs from the
  // end: the L2 holds the tail of that phase, which a sweep from the start
  // would push out before it gets there.  And that phase reads what nothing
  // else of the launch uses with evict-first loads, so that the tail is longer.
  // (z = d / |d| after the phase that wrote d, 2^24 FP32: 65.3 -> 63.7 us a pass.)
  const bool backwards = flat && n.dims == 1 && !n.coop && !by_rows && revisits(g, n);
  bool revisited = false;
  for (int h = g + 1; h < (int)S.groups.size() && !revisited; ++h)
    if (!S.groups[h].scalar && !S.groups[h].wave) revisited = n.dims == 1 && swept_after(g, h);
  auto once = [&](const Rd& rd) { return revisited && rd.ro && users(rd.a->root) == 1; };
  std::map<int, std::string>& spre = E.spre;  // SpMV task -> value computed before the body (warp-cooperative rows)
  // ---- body generator for one element group: `u` unroll slot, lanes V,
  // element offset expression `eoff` (flat) or (row, col) expressions
  auto addr = [&](const Arg& a, const std::string& e_flat, const std::string& row, const std::string& col) {
    const LaunchRoot& r = R(a.root);
    if (n.dims == 1) return ptr(a.root) + " + " + base.at(akey(a)) + " + " + e_flat;
    if (n.rank == 3)
      return ptr(a.root) + " + " + base.at(akey(a)) + " + ((" + row + ") / ext1) * " + std::to_string(r.stride[0]) +
             "LL + ((" + row + ") % ext1) * " + std::to_string(r.stride[1]) + "LL + " + col;
    return ptr(a.root) + " + " + base.at(akey(a)) + " + (" + row + ") * " + std::to_string(r.stride[0]) + "LL + " + col;
  };
  // emits loads for slot u (vector width w), compute, stores; returns nothing
  auto body = [&](int w, const std::vector<std::string>& slots, const std::vector<std::string>& eflat,
                  const std::vector<std::string>& erow, const std::vector<std::string>& ecol,
                  const std::string& pad) {
    const int ns = (int)slots.size();
    // loads
    for (int s = 0; s < ns; ++s) {
      for (const Rd& rd : reads) {
        const Arg& a = *rd.a;
        const std::string ad = addr(a, eflat[s], erow[s], ecol[s]);
        const std::string v = rd.var + "_" + slots[s];
        const int sh = (w > 1 && n.realign) ? n.shift.at(rd.key) : 0;
        if (sh && w == 4 && a.dtype == DFS_F32) {
          o << pad << "const f32x4 " << v << " = " << (rd.ro ? "ld4sro<" : "ld4s<") << sh << ">(" << ad << " - " << sh
            << ");\n";
        } else if (sh && w == 2 && a.dtype == DFS_F64) {
          o << pad << "const f64x2 " << v << " = " << (rd.ro ? "ld2sro<" : "ld2s<") << sh << ">(" << ad << " - " << sh
            << ");\n";
        } else if (w == 4 && a.dtype == DFS_F32) {
          o << pad << "const f32x4 " << v << " = " << (once(rd) ? "ld4cs(" : rd.ro ? "ld4ro(" : "ld4(") << ad << ");\n";
        } else if (w == 2 && a.dtype == DFS_F64) {
          o << pad << "const f64x2 " << v << " = " << (once(rd) ? "ld2cs(" : rd.ro ? "ld2ro(" : "ld2(") << ad << ");\n";
        } else {
          o << pad << "const " << T(a.dtype) << " " << v << " = " << (rd.ro ? "ldro(" : "ld(") << ad << ");\n";
        }
      }
    }
    const auto outvars = emit_compute(n, E, w, slots, eflat, pad);
    // stores (the last value written to each (root, partition) in the nest)
    for (auto& kv : outvars) {
      const Arg* a = nullptr;
      for (int i = n.first; i < n.last && !a; ++i) {
        const Task& t = S.tasks[i];
        if (t.scalar()) continue;
        for (size_t ai = 0; ai < t.args.size(); ++ai)
          if (!t.args[ai].imm && akey(t.args[ai]) == kv.first) a = &t.args[ai];
      }
      for (int s = 0; s < ns; ++s) {
        const std::string ad = addr(*a, eflat[s], erow[s], ecol[s]);
        if (w == 4 && a->dtype == DFS_F32) {
          o << pad << "st4(" << ad << ", f32x4{{" << kv.second[s * w] << ", " << kv.second[s * w + 1] << ", "
            << kv.second[s * w + 2] << ", " << kv.second[s * w + 3] << "}});\n";
        } else if (w == 2 && a->dtype == DFS_F64) {
          o << pad << "st2(" << ad << ", f64x2{{" << kv.second[s * w] << ", " << kv.second[s * w + 1] << "}});\n";
        } else {
          o << pad << "*(" << ad << ") = " << kv.second[s * w] << ";\n";
        }
      }
    }
  };

  // block-stride loops inside a point, grid-stride loops over a flat range
  const std::string st0 = flat ? "((i64)blockIdx.x * " + std::to_string(BD) + " + threadIdx.x)" : "(i64)threadIdx.x";
  const std::string stp = flat ? "gs" : std::to_string(BD);
  if (flat) o << ind << "  const i64 gs = (i64)gridDim.x * " << BD << ";\n";
  auto slot_off = [&](int u) { return flat ? std::to_string(u) + " * gs" : std::to_string(u * BD); };
  if (n.dims == 1 && (n.coop || by_rows)) {
    // SpMV rows shared by lanes (spmv_warp), or a warp's rows summed from
    // shared memory (spmv_rows).  Elements are dealt to threads exactly as in
    // the plain loops (vectors of V in thread order, then the
    // scalar tail), so reductions fused here sum in the same order; each trip
    // a warp takes 32 consecutive vectors, so all its lanes run the same trips
    o << ind << "  const i64 n = ";
    for (int d = 0; d < nd; ++d) o << (d ? " * " : "") << "ext" << d;
    o << ";\n";
    o << ind << "  const int lane_ = threadIdx.x & 31;\n";
    auto coop_spmv = [&](int w, const std::string& first, const std::string& wfirst, const std::string& wrows,
                         const std::string& pad) {
      for (int i = n.first; i < n.last; ++i) {
        const Task& t = S.tasks[i];
        if (t.op != DFS_OP_SPMV) continue;
        const Arg& y = t.args[4];
        const int dt = y.dtype;
        const std::string ops = ptr(t.args[0].root) + " + " + base.at(akey(t.args[0])) + ", " + ptr(t.args[1].root) + " + " +
                                base.at(akey(t.args[1])) + ", " + ptr(t.args[2].root) + " + " + base.at(akey(t.args[2])) +
                                ", " + ptr(t.args[3].root) + " + " + base.at(akey(t.args[3])) + ", (" + base.at(akey(y)) +
                                " - " + std::to_string(y.part.vlo[0]) + "LL + ";
        const std::string sp = "sp" + std::to_string(i);
        if (by_rows) {
          o << pad << T(dt) << " " << sp << "[" << w << "];\n";
          o << pad << "spmv_rows<" << T(dt) << ", " << w << ">(" << ops << wfirst << "), " << wrows << ", (" << T(dt)
            << "*)(dfs_sp_raw + (threadIdx.x >> 5) * kSpmvWarpBytes), " << sp << ");\n";
          for (int l = 0; l < w; ++l) o << pad << "const " << T(dt) << " " << sp << "_" << l << " = " << sp << "[" << l << "];\n";
        } else {
          for (int l = 0; l < w; ++l)
            o << pad << "const " << T(dt) << " " << sp << "_" << l << " = spmv_warp<" << T(dt) << ">(" << ops << first
              << " + " << l << "), act_, " << spmv_k(t) << ");\n";
        }
        spre[i] = "sp" + std::to_string(i);
      }
    };
    if (V > 1) {
      o << ind << "  const i64 nv = n / " << V << ";\n";
      o << ind << "  for (i64 wb = " << st0 << " - lane_; wb < nv; wb += " << stp << ") {\n";
      o << ind << "    const i64 v = wb + lane_;\n";
      o << ind << "    const bool act_ = v < nv;\n";
      coop_spmv(V, "v * " + std::to_string(V), "wb * " + std::to_string(V),
                "(int)min(nv - wb, (i64)32) * " + std::to_string(V), ind + "    ");
      o << ind << "    if (act_) {\n";
      body(V, {"r"}, {"(v) * " + std::to_string(V)}, {""}, {""}, ind + "      ");
      o << ind << "    }\n";
      o << ind << "  }\n";
      o << ind << "  for (i64 wb = " << st0 << " - lane_; nv * " << V << " + wb < n; wb += " << stp << ") {\n";
      o << ind << "    const i64 e = nv * " << V << " + wb + lane_;\n";
    } else {
      o << ind << "  for (i64 wb = " << st0 << " - lane_; wb < n; wb += " << stp << ") {\n";
      o << ind << "    const i64 e = wb + lane_;\n";
    }
    o << ind << "    const bool act_ = e < n;\n";
    coop_spmv(1, "e", V > 1 ? "nv * " + std::to_string(V) + " + wb" : "wb", "(int)min(n - (e - lane_), (i64)32)",
              ind + "    ");
    o << ind << "    if (act_) {\n";
    body(1, {"t"}, {"e"}, {""}, {""}, ind + "      ");
    o << ind << "    }\n";
    o << ind << "  }\n";
  } else if (n.dims == 1) {
    // n elements in one contiguous range; vectors of V; main loop unrolled U
    o << ind << "  const i64 n = ";
    for (int d = 0; d < nd; ++d) o << (d ? " * " : "") << "ext" << d;
    o << ";\n";
    o << ind << "  if (n > 0) {\n";
    const std::string it = V > 1 ? "v" : "e";
    const std::string lim = V > 1 ? "nv" : "n";
    if (V > 1) o << ind << "    const i64 nv = n / " << V << ";\n";
    o << ind << "    i64 " << it << " = " << st0 << ";\n";
    auto flat_e = [&](const std::string& x) {
      const std::string at = backwards ? lim + " - 1 - (" + x + ")" : x;
      return V > 1 ? "(" + at + ") * " + std::to_string(V) : "(" + at + ")";
    };
    if (U > 1) {
      o << ind << "    for (; " << it << " + " << slot_off(U - 1) << " < " << lim << "; " << it << " += " << U
        << " * " << stp << ") {\n";
      std::vector<std::string> sl, ef, er, ec;
      for (int u = 0; u < U; ++u) {
        sl.push_back("u" + std::to_string(u));
        ef.push_back(flat_e(it + " + " + slot_off(u)));
        er.push_back("");
        ec.push_back("");
      }
      body(V, sl, ef, er, ec, ind + "      ");
      o << ind << "    }\n";
    }
    o << ind << "    for (; " << it << " < " << lim << "; " << it << " += " << stp << ") {\n";
    body(V, {"r"}, {flat_e(it)}, {""}, {""}, ind + "      ");
    o << ind << "    }\n";
    if (V > 1) {
      o << ind << "    for (i64 e = nv * " << V << " + " << st0 << "; e < n; e += " << stp << ") {\n";
      body(1, {"t"}, {"e"}, {""}, {""}, ind + "      ");
      o << ind << "    }\n";
    }
    o << ind << "  }\n";
  } else if (flat) {
    // a rectangle of nrows rows x ncols columns swept as one range of
    // (row, vector) cells with a grid stride; realigned rows start their
    // vectors after `hd` scalar columns and end with a scalar tail
    o << ind << "  const i64 nrows = " << (n.rank == 3 ? "ext0 * ext1" : "ext0") << ";\n";
    o << ind << "  const i64 ncols = " << (n.rank == 3 ? "ext2" : "ext1") << ";\n";
    o << ind << "  const i64 hd = " << (n.realign ? "min((i64)" + std::to_string(n.head) + ", ncols)" : "0") << ";\n";
    o << ind << "  const i64 nvr = (ncols - hd) / " << V << ";\n";
    o << ind << "  const i64 ncell = nrows * nvr;\n";
    o << ind << "  i64 c = " << st0 << ";\n";
    // 32-bit division by the constant row length when the range allows it
    const bool narrow = flat_cells < (int64_t(1) << 31);
    auto cell = [&](const std::string& cv, const std::string& sfx) {
      if (narrow)
        o << ind << "      const i64 i" << sfx << " = (i64)((u32)(" << cv << ") / (u32)nvr);\n";
      else
        o << ind << "      const i64 i" << sfx << " = (" << cv << ") / nvr;\n";
      o << ind << "      const i64 j" << sfx << " = hd + ((" << cv << ") - i" << sfx << " * nvr) * " << V << ";\n";
    };
    if (U > 1) {
      o << ind << "  for (; c + " << slot_off(U - 1) << " < ncell; c += " << U << " * gs) {\n";
      std::vector<std::string> sl, ef, er, ec;
      for (int u = 0; u < U; ++u) {
        cell("c + " + slot_off(u), std::to_string(u));
        sl.push_back("u" + std::to_string(u));
        ef.push_back("");
        er.push_back("i" + std::to_string(u));
        ec.push_back("j" + std::to_string(u));
      }
      body(V, sl, ef, er, ec, ind + "      ");
      o << ind << "  }\n";
    }
    o << ind << "  for (; c < ncell; c += gs) {\n";
    cell("c", "r");
    body(V, {"r"}, {""}, {"ir"}, {"jr"}, ind + "      ");
    o << ind << "  }\n";
    if (n.realign) {
      // the scalar head and tail columns of every row
      o << ind << "  const i64 nrem = ncols - nvr * " << V << ";\n";
      o << ind << "  if (nrem > 0) {\n";
      o << ind << "    for (i64 c2 = " << st0 << "; c2 < nrows * nrem; c2 += gs) {\n";
      o << ind << "      const i64 is = c2 / nrem;\n";
      o << ind << "      const i64 ks = c2 - is * nrem;\n";
      o << ind << "      const i64 js = ks < hd ? ks : hd + nvr * " << V << " + (ks - hd);\n";
      body(1, {"s"}, {""}, {"is"}, {"js"}, ind + "      ");
      o << ind << "    }\n";
      o << ind << "  }\n";
    }
  } else {
    // rows: each row of ncols elements is swept by the whole block
    o << ind << "  const i64 nrows = " << (n.rank == 3 ? "ext0 * ext1" : "ext0") << ";\n";
    o << ind << "  const i64 ncols = " << (n.rank == 3 ? "ext2" : "ext1") << ";\n";
    o << ind << "  for (i64 i = 0; i < nrows; ++i) {\n";
    if (V > 1 && n.realign) {
      o << ind << "    const i64 hd = min((i64)" << n.head << ", ncols);\n";
      o << ind << "    const i64 nv = (ncols - hd) / " << V << ";\n";
      o << ind << "    for (i64 v = threadIdx.x; v < nv; v += " << BD << ") {\n";
      body(V, {"r"}, {""}, {"i"}, {"hd + v * " + std::to_string(V)}, ind + "      ");
      o << ind << "    }\n";
      o << ind << "    for (i64 k = threadIdx.x; k < ncols - nv * " << V << "; k += " << BD << ") {\n";
      o << ind << "      const i64 js = k < hd ? k : hd + nv * " << V << " + (k - hd);\n";
      body(1, {"t"}, {""}, {"i"}, {"js"}, ind + "      ");
      o << ind << "    }\n";
    } else if (V > 1) {
      o << ind << "    const i64 nv = ncols / " << V << ";\n";
      o << ind << "    for (i64 v = threadIdx.x; v < nv; v += " << BD << ") {\n";
      body(V, {"r"}, {""}, {"i"}, {"v * " + std::to_string(V)}, ind + "      ");
      o << ind << "    }\n";
    } else {
      o << ind << "    i64 j = threadIdx.x;\n";
      if (U > 1) {
        o << ind << "    for (; j + " << (U - 1) * BD << " < ncols; j += " << U * BD << ") {\n";
        std::vector<std::string> sl, ef, er, ec;
        for (int u = 0; u < U; ++u) {
          sl.push_back("u" + std::to_string(u));
          ef.push_back("");
          er.push_back("i");
          ec.push_back("(j + " + std::to_string(u * BD) + ")");
        }
        body(1, sl, ef, er, ec, ind + "      ");
        o << ind << "    }\n";
      }
      o << ind << "    for (; j < ncols; j += " << BD << ") {\n";
      body(1, {"t"}, {""}, {"i"}, {"j"}, ind + "      ");
      o << ind << "    }\n";
    }
    o << ind << "  }\n";
  }
  // per-point partials of the reductions
  for (const Acc& ac : accs) {
    o << ind << "  { const " << T(ac.dt) << " tot = block_sum(" << ac.var << ", (" << T(ac.dt) << "*)red_buf);\n";
    o << ind << "    if (threadIdx.x == 0) ((" << T(ac.dt) << "*)P.partials)[" << ac.slot << "LL * P.red_stride + "
      << ptvar << "] = tot; }\n";
  }
  o << ind << "}\n";
  (void)g;
}

// Finishes every pending reduction: sum of the per-point partials in point
// order, folded into the register copy of the target.  Warp 0 sums (the
// order of sum_partials) and hands the totals to the CTA through shared
// memory: FP64 arithmetic is scarce on GB300 (about two lane operations per
// SM and clock), and every warp repeating the same sum cost about 0.5 us per
// reduction in an L2-resident CG iteration.  Called where every thread of the
// CTA arrives (after a grid barrier, or in the last CTA).
void Gen::emit_finalise(const char* ind) {
  if (pending_red.empty()) return;
  std::vector<std::string> bc;
  for (const Red& r : pending_red) {
    bc.push_back("bc" + std::to_string(nbc++));
    o << ind << "__shared__ " << T(r.dtype) << " " << bc.back() << ";\n";
  }
  o << ind << "if (threadIdx.x < 32) {\n";
  for (size_t j = 0; j < pending_red.size(); ++j) {
    const Red& r = pending_red[j];
    o << ind << "  const " << T(r.dtype) << " " << bc[j] << "_t = sum_partials8((const " << T(r.dtype)
      << "*)P.partials + " << r.slot << "LL * P.red_stride, " << r.points << "LL);\n";
    o << ind << "  if (threadIdx.x == 0) " << bc[j] << " = " << bc[j] << "_t;\n";
  }
  o << ind << "}\n" << ind << "__syncthreads();\n";
  for (size_t j = 0; j < pending_red.size(); ++j) {
    const Red& r = pending_red[j];
    const std::string nm = sreg.at(r.root);
    if (have[r.root])
      o << ind << nm << " = op_add(" << nm << ", " << bc[j] << ");\n";
    else
      o << ind << nm << " = " << bc[j] << ";\n";
    have[r.root] = true;
  }
  pending_red.clear();
}

// After a grid barrier: the pending reductions and the scalar groups that
// follow (g, g+1, ... while scalar) run on warp 0 alone, and every 0-d value
// they set reaches the CTA's other warps through shared memory.  The values
// are those every thread would compute (the same operations on the same
// register copies); only the repetition goes.  FP64 arithmetic is scarce on
// GB300 (about two lane operations per SM and clock), and eight warps
// repeating a 128-partial sum and an IEEE division cost about 1 us per CG
// phase at 256^2.  Returns the first group after the scalar run.
int Gen::emit_warp0_scalars(int g) {
  int h = g;
  while (h < (int)S.groups.size() && S.groups[h].scalar) ++h;
  std::vector<int64_t> set;
  auto add = [&](int64_t r) {
    if (std::find(set.begin(), set.end(), r) == set.end()) set.push_back(r);
  };
  for (const Red& r : pending_red) add(r.root);
  for (int k = g; k < h; ++k)
    for (int i = S.groups[k].begin; i < S.groups[k].end; ++i) add(S.tasks[i].args.back().root);
  if (set.empty()) return g;
  std::map<int64_t, std::string> bc;
  for (int64_t r : set) {
    bc[r] = "bc" + std::to_string(nbc++);
    o << "    __shared__ " << T(R(r).dtype) << " " << bc[r] << ";\n";
  }
  o << "    if (threadIdx.x < 32) {\n";
  for (const Red& r : pending_red) {
    const std::string nm = sreg.at(r.root);
    o << "      { const " << T(r.dtype) << " tot = sum_partials8((const " << T(r.dtype) << "*)P.partials + "
      << r.slot << "LL * P.red_stride, " << r.points << "LL);\n";
    if (have[r.root])
      o << "        " << nm << " = op_add(" << nm << ", tot); }\n";
    else
      o << "        " << nm << " = tot; }\n";
    have[r.root] = true;
  }
  pending_red.clear();
  for (int k = g; k < h; ++k) emit_scalar_group(k);
  o << "      if (threadIdx.x == 0) {\n";
  for (int64_t r : set) o << "        " << bc[r] << " = " << sreg.at(r) << ";\n";
  o << "      }\n    }\n    __syncthreads();\n";
  for (int64_t r : set) o << "    " << sreg.at(r) << " = " << bc[r] << ";\n";
  return h;
}

// ------------------------------------------------------- in-place sweeps
// See WaveGeom and MarchGeom.  The two-phase form of a Fig. 1 sweep (the
// stencil into a second array, a grid barrier, the copy back) moves 16 bytes
// per FP32 point and is bound by HBM; in place it is 8.  Measured on GB300, us
// per sweep, two phases -> in place:
//   8190^2 FP32 (512-thread CTAs)        175.6 -> 91.9 (5.84 TB/s, 86 % of the copy rate)
//   1021 x 1147 FP32, five per launch      7.9 -> 4.3
//   4000^2 FP64                          197.4 -> 174.4 (bound by the FP64 pipe: 5 operations per point)
//   251^3 FP32 (tiles)                    64.1 -> 42.1
//   251^3 FP64 (tiles)                   258.9 -> 242 (FP64 pipe: 7 operations per point, 176 us)
int64_t origin_of(const Arg& a, int d) { return std::max(a.part.off[d], a.part.vlo[d]); }
int64_t floor_div(int64_t a, int64_t b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// The sweeps' row and column numbers are 32-bit, sums of two of them included
// (the last bands start up to a band past the last row): stores with a longer
// side take the two phases, whose indices are 64-bit.
bool sides_fit(const LaunchSpec& S, int g) {
  for (int i = S.groups[g].begin; i < S.groups[g + 1].end; ++i)
    for (const Arg& a : S.tasks[i].args) {
      if (a.imm || a.nd == 0) continue;
      const LaunchRoot& r = S.roots[S.root_index.at(a.root)];
      for (int d = 0; d < r.ndim; ++d)
        if (r.shape[d] >= (int64_t(1) << 30)) return false;
    }
  return true;
}

}  // namespace

bool wave_legal(const LaunchSpec& S, int g) {
  if (g + 1 >= (int)S.groups.size()) return false;
  const Group &A = S.groups[g], &B = S.groups[g + 1];
  if (A.scalar || B.scalar) return false;
  const std::string space = iteration_space_key(S.tasks[A.begin]);
  for (int i = A.begin; i < B.end; ++i) {
    const Task& t = S.tasks[i];
    if (t.scalar() || !is_elementwise(t.op) || iteration_space_key(t) != space) return false;
    for (const Arg& a : t.args) {
      if (a.imm || a.nd == 0) continue;
      if (a.nd != 2 && a.nd != 3) return false;
      if (a.part.kind != 1) return false;
      for (int d = 0; d < a.nd; ++d)
        if (a.part.proj[d] != d) return false;
    }
  }
  // across the groups, accesses of one store through different partitions may
  // only be a read in A and a write in B (the anti-dependence the wave orders)
  bool cut = false;
  for (int i = A.begin; i < A.end; ++i)
    for (const Arg& a : S.tasks[i].args) {
      if (a.imm || a.nd == 0) continue;
      for (int j = B.begin; j < B.end; ++j)
        for (const Arg& b : S.tasks[j].args) {
          if (b.imm || b.root != a.root || b.part == a.part) continue;
          if (a.is_w()) return false;
          if (b.is_w()) cut = true;
        }
    }
  return cut;
}

namespace {

// Arithmetic operations per element of a pair of groups, in units of an
// addition (copies and signs cost no arithmetic).
double pair_ops(const LaunchSpec& S, int g) {
  double n = 0.0;
  for (int i = S.groups[g].begin; i < S.groups[g + 1].end; ++i) {
    const int op = S.tasks[i].op;
    if (op == DFS_OP_COPY || op == DFS_OP_NEG || op == DFS_OP_ABS) continue;
    n += op == DFS_OP_DIV || op == DFS_OP_SQRT ? 10.0 : op >= DFS_OP_ADD && op != DFS_OP_POW ? 1.0 : 25.0;
  }
  return n;
}

// What one sweep takes, in microseconds, as fitted to GB300 measurements (the
// 5-point stencil of 66^2 to 8190^2 points, tall and wide grids, one, five and
// nine operations a point, 128 to 1024 threads; within about 10 % of them).
// The forms are compared by these estimates only, so results do not depend on
// them: every form leaves the same bits.
//
// Two phases: a barrier and two flat sweeps; FP32 by L2 and HBM, FP64 by the
// FP64 pipe, which a flat sweep keeps busy on all SMs.
double phases_us(const LaunchSpec& S, double elems, int esz, double ops, int nd) {
  if (esz == 4) return 6.5 + elems / (8.0 * elems > 96e6 ? 0.385e6 : 0.48e6);
  const double pipe = elems / S.sms * (0.00045 + 0.00027 * ops);
  return nd == 3 ? std::max(std::min(10.0, 6.0 + elems / 8192.0), 7.5 + pipe) : std::max(S.block >= 1024 ? 11.0 : 9.0, 5.5 + pipe);
}
// Bands: the CTA's flags, then a row of the band (and the two next to it) at a
// time.  FP32: a row costs a round trip to L2, or what its vectors take; columns
// next to panels cost more.  FP64: the schedulers share the
// FP64 units in such a way that a row costs as if part of the warps were
// rounded up to eight (measured: 5, 6, 7, 8 warps 1.6, 1.7, 1.9, 2.0; 9, 10,
// 12, 14, 16 warps 3.1, 3.3, 3.5, 3.8, 4.0 times what a warp per scheduler
// should), whatever lanes are active: narrow rows waste it.
double bands_us(const LaunchSpec& S, const MarchGeom& M, int esz, double ops) {
  if (esz == 4) {
    const double row = 0.03 * ops * M.K * std::pow(S.block / 256.0, 0.6) * (1.0 + 0.05 * std::max(0, M.K - 6));
    const double trip = 0.23 * std::pow(S.block / 256.0, 0.3);
    return 3.5 + (M.BR + 2) * std::max(trip, row) * (1.0 + 0.2 * std::min<int64_t>(M.PN - 1, 3));
  }
  const int w = M.GT * M.G / 32 * std::max(1, S.min_blocks);
  const double busy = w <= 4 ? 1.1 : w / 8.0 + (w + 7) / 8;
  const double row = busy * M.K * (0.066 + 0.002 * ops) * ops * ((double)M.rows * M.cols * esz > 96e6 ? 1.12 : 1.0);
  return 4.5 + M.BR * std::max(0.8, row);
}

// Tiles: a CTA's first tile, then what the FP64 pipe takes for the tiles of the
// busiest SM (whole rounds of the resident CTAs once there are more tiles).
double tiles_us(const LaunchSpec& S, const WaveGeom& W, double elems, double ops) {
  const int64_t resident = (int64_t)W.min_blocks * S.sms;
  const double q = W.tiles <= resident ? (double)((W.tiles + S.sms - 1) / S.sms)
                                       : (double)((W.tiles + resident - 1) / resident) * W.min_blocks;
  const double us = 6.0 + q * (S.block - 32) * W.R * W.V * 0.000311 * ops;
  return W.nd == 2 && elems * 8 > 96e6 ? 1.15 * us : us;
}
// Whether tiles are below the two phases (us a sweep, tiles against phases).
// Their polling and their rounds cost more than the barrier saves but for small
// sweeps, where a tile is all that an SM has (5 x 10002 FP32 4.1 against 5.8;
// 34^3 FP32 5.7 against 6.7), and for 3-D grids of one result, whose planes a
// tile keeps in L1 (251^3 FP32 42 against 63, FP64 240 against 258).  With a
// second result in memory (200^3 FP32 31.5 against 22.5), lines much longer than
// a tile (48 x 48 x 2000 FP64 85 against 81) or readers most of a round away
// (20 x 500 x 500 FP64 125 against 81) they are slower.
bool tiles_pay(const LaunchSpec& S, const WaveGeom& W, double elems, int esz, double ops, int results) {
  const int64_t BD = S.block - 32, resident = (int64_t)W.min_blocks * S.sms;
  const bool small = W.tiles * 3 * std::max(1, S.block / 256) <= (int64_t)S.sms * 2;
  if (!small && ((W.nd == 3 && W.nvx > 2 * BD) || W.reach * 3 > resident * 2)) return false;
  if (esz == 8) return W.us + (small ? 0.0 : 0.3 * (results - 1)) < phases_us(S, elems, esz, ops, W.nd);
  return small || (W.nd == 3 && results == 1 && elems >= (1 << 21));
}

}  // namespace

WaveGeom wave_geometry(const LaunchSpec& S, int g) {
  WaveGeom W;
  const Group &A = S.groups[g], &B = S.groups[g + 1];
  const Task& last = S.tasks[B.end - 1];
  const Arg& sa = space_arg(last);
  W.nd = sa.nd;
  int64_t elems = 1;
  for (int d = 0; d < W.nd; ++d) {
    W.ext[d] = std::min(last.dom[d] * sa.part.tile[d] + sa.part.off[d], sa.part.vhi[d]) - origin_of(sa, d);
    if (W.ext[d] <= 0) return W;
    elems *= W.ext[d];
  }
  if (elems < kWaveMinElems || elems >= (int64_t(1) << 31) || !sides_fit(S, g)) return W;
  const int cd = W.nd - 1;
  // vector width: every row of every store in memory starts on a vector
  size_t esz = 0;
  bool aligned = true;
  for (int i = A.begin; i < B.end; ++i)
    for (const Arg& a : S.tasks[i].args) {
      if (a.imm || a.nd == 0) continue;
      const size_t es = dtype_size(a.dtype);
      if (esz && es != esz) return W;
      esz = es;
    }
  const int vec = (int)(16 / esz);
  for (int i = A.begin; i < B.end; ++i)
    for (const Arg& a : S.tasks[i].args) {
      if (a.imm || a.nd == 0) continue;
      const LaunchRoot& r = S.roots[S.root_index.at(a.root)];
      if (r.temp) continue;
      if (!r.aligned16) aligned = false;
      for (int d = 0; d < cd; ++d)
        if (r.stride[d] % vec) aligned = false;
    }
  W.V = aligned ? vec : 1;
  int phase = -1;
  for (int i = A.begin; i < B.end; ++i) {
    const Arg& a = S.tasks[i].args.back();
    if (S.roots[S.root_index.at(a.root)].temp) continue;
    const int ph = (int)(origin_of(a, cd) % W.V);
    if (phase >= 0 && ph != phase) return W;  // written views in different vector frames
    phase = ph;
  }
  W.lead = std::max(phase, 0);
  // slices per cell: a tile costs its CTA one round of flags whatever its
  // size, so more points per thread are better until registers spill or too
  // few warps stay (251^3 FP32, us per sweep at 256 threads: R = 2 67, 4 42,
  // 8 46; FP64 238, 242, 257).  1024-thread CTAs have 64 registers a thread.
  W.R = S.block >= 1024 ? 2 : 4;
  W.lines = W.nd == 3 ? W.ext[1] : 1;
  W.nvx = (W.lead + W.ext[cd] + W.V - 1) / W.V;
  const int64_t nrb = (W.ext[0] + W.R - 1) / W.R, BD = S.block - 32;  // cells per tile
  W.cells = nrb * W.lines * W.nvx;
  W.tiles = (W.cells + BD - 1) / BD;
  if (W.tiles > kWaveTilesMax || W.cells >= (int64_t(1) << 31) - BD) return W;
  // which tiles read tile t: a cell reads at every offset (read view's origin
  // less the written view's), as a range of cell numbers, hence of tiles
  std::set<int64_t> rel;
  for (int i = A.begin; i < A.end; ++i)
    for (const Arg& a : S.tasks[i].args) {
      if (a.imm || a.nd == 0 || !a.is_r()) continue;
      for (int j = B.begin; j < B.end; ++j) {
        const Arg& b = S.tasks[j].args.back();
        if (b.root != a.root || b.part == a.part) continue;
        const int64_t d0 = origin_of(a, 0) - origin_of(b, 0), dc = origin_of(a, cd) - origin_of(b, cd);
        const int64_t d1 = W.nd == 3 ? origin_of(a, 1) - origin_of(b, 1) : 0;
        const int64_t v0 = floor_div(dc, W.V), v1 = floor_div(W.V - 1 + dc, W.V);
        for (int64_t b0 = floor_div(d0, W.R); b0 <= floor_div(W.R - 1 + d0, W.R); ++b0) {
          const int64_t o = (b0 * W.lines + d1) * W.nvx;
          for (int64_t k = floor_div(-(o + v1), BD); k <= floor_div(BD - 1 - (o + v0), BD); ++k)
            if (k != 0) rel.insert(k);
          if (rel.size() > 4096) return W;
        }
      }
    }
  for (int64_t k : rel) {
    W.reach = std::max(W.reach, k < 0 ? -k : k);
    if (!W.readers.empty() && W.readers.back().second + 1 == k) W.readers.back().second = k;
    else W.readers.push_back({k, k});
  }
  // progress: a CTA waits for the readers of its previous tile before it
  // publishes its next one, `grid` tiles on, so a tile's readers must lie
  // less than a grid ahead (or every tile has a CTA of its own)
  W.min_blocks = S.min_blocks > 0 ? S.min_blocks : std::max(1, 1024 / S.block);
  const int64_t resident = (int64_t)W.min_blocks * S.sms;
  std::set<int64_t> results;
  for (int i = A.begin; i < B.end; ++i) {
    const Arg& a = S.tasks[i].args.back();
    if (!S.roots[S.root_index.at(a.root)].temp) results.insert(a.root);
  }
  const double ops = pair_ops(S, g);
  W.us = tiles_us(S, W, (double)elems, ops);
  W.ok = (W.tiles <= resident || W.reach < resident) &&
         tiles_pay(S, W, (double)elems, (int)esz, ops, (int)results.size());
  return W;
}

MarchGeom march_geometry(const LaunchSpec& S, int g) {
  MarchGeom M;
  const Group &A = S.groups[g], &B = S.groups[g + 1];
  const Arg& out = S.tasks[B.end - 1].args.back();
  if (out.nd != 2) return M;
  const LaunchRoot& X = S.roots[S.root_index.at(out.root)];
  if (X.temp) return M;
  M.w0 = origin_of(out, 0);
  M.wc = origin_of(out, 1);
  const Task& last = S.tasks[B.end - 1];
  M.rows = std::min(last.dom[0] * out.part.tile[0] + out.part.off[0], out.part.vhi[0]) - M.w0;
  M.cols = std::min(last.dom[1] * out.part.tile[1] + out.part.off[1], out.part.vhi[1]) - M.wc;
  if (M.rows <= 0 || M.cols <= 0 || M.rows * M.cols < kWaveMinElems || !sides_fit(S, g)) return M;
  const size_t esz = dtype_size(out.dtype);
  const int vec = (int)(16 / esz);
  M.V = X.aligned16 && X.stride[0] % vec == 0 ? vec : 1;
  const int64_t lead = M.wc % M.V, nv = M.V > 1 ? X.stride[0] / M.V : X.shape[1];
  std::set<std::pair<int64_t, int64_t>> edges;
  for (int i = A.begin; i < B.end; ++i)
    for (size_t ai = 0; ai < S.tasks[i].args.size(); ++ai) {
      const Arg& a = S.tasks[i].args[ai];
      if (a.imm || a.nd == 0) continue;
      if (S.roots[S.root_index.at(a.root)].temp) continue;
      if (a.root != out.root || a.dtype != out.dtype) return M;
      if (ai + 1 == S.tasks[i].args.size()) {
        if (!(a.part == out.part)) return M;
        continue;
      }
      const int64_t d0 = origin_of(a, 0) - M.w0, dc = origin_of(a, 1) - M.wc;
      if (d0 < -1 || d0 > 1 || dc < -M.V || dc > M.V) return M;
      if (dc < 0) M.edge_m = true;
      if (dc > 0) M.edge_p = true;
      for (int l = 0; l < M.V; ++l)
        if (floor_div(dc + l, M.V)) edges.insert({floor_div(dc + l, M.V), (dc + l + M.V) % M.V});
    }
  // vectors of a row: the written ones and the neighbours they read, as far
  // as the row has them
  const int64_t f0 = (M.wc - lead) / M.V, f1 = f0 + (lead + M.cols + M.V - 1) / M.V;
  M.pv0 = std::max<int64_t>(0, f0 - (M.edge_m ? 1 : 0));
  M.NC = std::min(nv, f1 + (M.edge_p ? 1 : 0)) - M.pv0;
  // threads, vectors per thread and rows ahead, from the registers of one CTA
  // per SM; narrow rows leave room for several bands in a CTA, and rows wider
  // than a CTA's registers are split into panels
  const int64_t words = M.V * (int64_t)esz / 4, 
                avail = std::min<int64_t>(255, 65536 / (S.block * std::max(1, S.min_blocks))) - 44;
  const int64_t kmax = avail / (words * 5);  // three rows around the computed one and two ahead
  const int64_t per_sm = S.min_blocks > 0 ? S.min_blocks : 1;
  // static shared memory: the row below the band, the warps' edge elements
  // and, between panels, the neighbours' edge columns; 48 KB less the kernel's
  // other arrays (the sums' buffer, broadcast slots)
  const int64_t limit = std::min<int64_t>(40 * 1024, 48 * 1024 - 8 * S.block - 1024);
  // vectors per thread: the fewest leave threads and warps of the last vector
  // idle, the most leave too few bands; taken by the estimate above, and only
  // where it is below that of the two phases.  Bands against two phases, us a
  // sweep: 1000002 x 5 FP64 659 -> 49, 200002 x 34 FP32 43 -> 20 (two phases
  // again); 20002 x 302 FP32 17.4 -> 11.3, 302 x 20002 FP32 16.6 -> 11.8 (other K).
  const double ops = pair_ops(S, g);
  double best = phases_us(S, (double)M.rows * M.cols, (int)esz, ops, 2);
  if (esz == 8) {
    const WaveGeom W = wave_geometry(S, g);
    if (W.ok) best = std::min(best, W.us);
  }
  MarchGeom pick;
  for (int64_t k = kmax; k >= 1; --k) {
    MarchGeom C = M;
    C.PN = (C.NC + S.block * k - 1) / (S.block * k);
    const int64_t per = (C.NC + C.PN - 1) / C.PN;
    C.K = (int)std::max(std::min(k, (per + 31) / 32), (per + S.block - 1) / S.block);
    C.GT = (int)(((per + C.K - 1) / C.K + 31) / 32 * 32);
    C.PC = (int64_t)C.K * C.GT;
    C.PN = (C.NC + C.PC - 1) / C.PC;
    C.G = C.PN > 1 ? 1 : S.block / C.GT;
    const int64_t ctas = std::max<int64_t>(1, per_sm * S.sms / C.PN);
    if (C.PN > per_sm * S.sms) continue;
    C.BR = (C.rows + ctas * C.G - 1) / (ctas * C.G);
    C.NB = ((C.rows + C.BR - 1) / C.BR + C.G - 1) / C.G;
    C.D = (int)std::min<int64_t>({6, avail / (words * C.K) - 3, C.BR});
    C.smem = (int64_t)C.K * C.GT * C.G * C.V * esz + (3 + C.D) * (int64_t)edges.size() * C.K * (C.GT * C.G / 32) * esz +
             (C.PN > 1 ? (C.BR + 2) * (int64_t)edges.size() * esz : 0);
    if (C.smem > limit || C.NB * C.PN > kWaveTilesMax) continue;
    const double us = bands_us(S, C, (int)esz, ops);
    // equal: fewer vectors per thread, unless that takes more panels
    if (pick.ok ? us > best + 1e-6 || (us > best - 1e-6 && C.PN > pick.PN) : us >= best) continue;
    pick = C;
    pick.ok = true;
    best = us;
  }
  return pick;
}

namespace {

// The band form of `sweeps` in-place sweeps in a row (MarchGeom): groups g,
// g+1 and the alike pairs after them, as one loop.  Between two of them the
// neighbours' "stored" flags take the place of a grid barrier.
void Gen::emit_march(int g, int sweeps) {
  const MarchGeom M = march_geometry(S, g);
  const Group &A = S.groups[g], &B = S.groups[g + 1];
  const int BD = S.block, V = M.V, K = M.K, RS = 3 + M.D, AT = M.GT * M.G, NW = AT / 32;  // AT: threads that own vectors
  const int steps = (int)std::min<int64_t>(RS, M.BR);  // rows per trip of the unrolled row loop
  Nest n;
  n.first = A.begin;
  n.last = B.end;
  n.dims = 2;
  n.vec = V;
  n.rank = 2;
  BodyEnv E;
  std::set<std::string> written, seen;
  std::string okey;
  const Arg* out = &S.tasks[B.end - 1].args.back();
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    for (size_t ai = 0; ai < t.args.size(); ++ai) {
      const Arg& a = t.args[ai];
      if (a.imm || a.nd == 0) continue;
      const std::string k = akey(a);
      if (ai + 1 == t.args.size()) {
        written.insert(k);
        if (!R(a.root).temp) okey = k;
      } else if (!written.count(k) && seen.insert(k).second) {
        E.reads.push_back({k, &a, "m" + std::to_string(E.reads.size()), false});
      }
    }
  }
  const LaunchRoot& X = R(out->root);
  const int dt = out->dtype;
  const std::string T1 = T(dt), TV = V == 4 ? "f32x4" : (V == 2 ? "f64x2" : T1);
  const std::string ldv = V == 4 ? "ld4" : (V == 2 ? "ld2" : "ld"), stv = V == 4 ? "st4" : "st2";
  const std::string ind = "      ", in2 = "        ", in3 = "            ";
  // elements of neighbouring vectors: (row offset, before/after, element)
  std::map<std::pair<int, int>, int> eidx;  // (dv, e) -> edge slot
  std::set<std::tuple<int, int, int>> need;
  auto src = [&](const Rd& rd, int l) {
    const int64_t d0 = origin_of(*rd.a, 0) - M.w0, q = origin_of(*rd.a, 1) - M.wc + l;
    const int dv = (int)floor_div(q, V);
    return std::make_tuple((int)d0, dv, (int)(q - (int64_t)dv * V));
  };
  for (const Rd& rd : E.reads)
    for (int l = 0; l < V; ++l) {
      const auto s = src(rd, l);
      if (std::get<1>(s) == 0) continue;
      eidx.emplace(std::make_pair(std::get<1>(s), std::get<2>(s)), (int)eidx.size());
      need.insert(s);
    }
  const int NE = (int)eidx.size();
  const int st0 = kc.nwaves + 1;  // "edges read"; the next value: "stored"
  kc.nwaves += 2 * sweeps;
  kc.wave_tiles = std::max(kc.wave_tiles, M.NB * M.PN);
  kc.march_ctas = std::max(kc.march_ctas, M.NB * M.PN);
  wave_blocks = std::max(wave_blocks, 1);
  const std::string sfx = std::to_string(g);
  o << "    { // groups " << g << ", " << g + 1 << ": tasks " << n.first << ".." << n.last - 1 << ", one in-place sweep of "
    << M.NB * M.G << " bands of " << M.BR << " rows, " << M.PN << " panel(s), " << K << " vector(s) per thread, " << M.D
    << " row(s) ahead\n";
  // immediates: those of every sweep in a row
  const int imm0 = kc.nimm, ntask = n.last - n.first;
  for (int w = 0; w < sweeps; ++w)
    for (int i = n.first; i < n.last; ++i)
      for (size_t ai = 0; ai < S.tasks[i].args.size(); ++ai)
        if (S.tasks[i].args[ai].imm) imm_expr(i + w * ntask, (int)ai, dt);
  const int nimm = (kc.nimm - imm0) / sweeps;
  const bool pan = M.PN > 1 && NE;
  o << ind << T1 << "* const mb" << sfx << " = (" << T1 << "*)march_raw;  // the row below the band\n";
  if (NE) o << ind << T1 << "* const me" << sfx << " = mb" << sfx << " + " << K * AT * V << ";  // edge elements of the warps' vectors\n";
  if (pan) o << ind << T1 << "* const mp" << sfx << " = me" << sfx << " + " << RS * NE * K * NW << ";  // edge columns of the next panels\n";
  o << ind << "bool mok = true;\n";
  const std::string sw = sweeps > 1 ? "sw" : "0";
  if (sweeps > 1) o << ind << "for (int sw = 0; sw < " << sweeps << " && mok; ++sw) {\n";
  o << ind << "const u64 fw = ep_ + " << st0 << "ull" << (sweeps > 1 ? " + 2 * sw" : "") << ";\n";
  for (int i = n.first, k = 0; i < n.last; ++i)
    for (size_t ai = 0; ai < S.tasks[i].args.size(); ++ai) {
      if (!S.tasks[i].args[ai].imm) continue;
      const std::string nm = "k" + std::to_string(i) + "_" + std::to_string(ai);
      o << ind << "const " << T1 << " " << nm << " = ((" << T1 << ")P.imm[" << imm0 + k++;
      if (sweeps > 1) o << " + sw * " << nimm;
      o << "]);\n";
      E.immv[{i, (int)ai}] = nm;
    }
  o << ind << "if (blockIdx.x < " << M.NB * M.PN << "u) {\n";
  if (sweeps > 1)
    o << in2 << "mok = sw == 0 || march_wait(P.flags, " << M.NB << "LL, " << M.PN << "LL, fw - 1, ctl, P.timeout_ns);\n"
      << in2 << "if (mok) {\n";
  else
    o << in2 << "{\n";
  if (M.G > 1) o << in2 << "const int grp = threadIdx.x / " << M.GT << ", q = threadIdx.x - grp * " << M.GT << ";\n";
  else o << in2 << "const int grp = 0, q = threadIdx.x;\n";
  // threads past the last group own nothing
  o << in2 << "const int ra = grp < " << M.G << " && q < " << M.GT << " ? min((int)((blockIdx.x / " << M.PN << "u) * " << M.G
    << "u + grp) * " << M.BR << ", " << M.rows << ") : " << M.rows << ", rz = min(ra + " << M.BR << ", " << M.rows << ");\n";
  o << in2 << "const bool act = ra < rz;\n";
  o << in2 << "const int pb = (int)(blockIdx.x % " << M.PN << "u) * " << M.PC << ";\n";
  // With several groups the warp's number comes through a shuffle: with it
  // written in place NVRTC 13.0 turned (threadIdx.x >> 5) * K + k, where only lane
  // 31 gets there and K is a power of two, into the address of K - 1 elements
  // further on.
  o << in2 << "const int lane = threadIdx.x & 31, lw = q >> 5;\n";
  o << in2 << "const int wid = " << (M.G > 1 ? "__shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0)" : "(int)(threadIdx.x >> 5)") << ";\n";
  // one warp's vectors k are consecutive; vectors past the row repeat its last
  for (int k = 0; k < K; ++k) {
    o << in2 << "const int c" << k << " = pb + " << k * M.GT << " + q;\n";
    o << in2 << T1 << "* const x" << k << " = " << ptr(out->root) << " + (i64)" << M.w0 << " * " << X.stride[0] << "LL + (i64)(min(c" << k
      << ", " << M.NC - 1 << ") + " << M.pv0 << ") * " << V << ";\n";
    o << in2 << "const bool s" << k << "_ = act && c" << k << " < " << (M.PN > 1 ? "min(pb + " + std::to_string(M.PC) + ", " + std::to_string(M.NC) + ")" : std::to_string(M.NC)) << ";\n";
    o << in2 << "const int j" << k << " = (c" << k << " + " << M.pv0 << ") * " << V << " - " << M.wc << ";\n";
  }
  auto sl = [&](int j, int k) { return "s" + std::to_string(((j % RS) + RS) % RS) + "_" + std::to_string(k); };
  for (int j = 0; j < RS; ++j)
    for (int k = 0; k < K; ++k) o << in2 << TV << " s" << j << "_" << k << (V > 1 ? " = {};\n" : " = 0;\n");
  auto row_at = [&](int k, const std::string& r) {
    return "x" + std::to_string(k) + " + (i64)(" + r + ") * " + std::to_string(X.stride[0]) + "LL";
  };
  // the rows next to the band, then the band's first rows
  o << in2 << "if (act) {\n";
  for (int k = 0; k < K; ++k) o << in3 << sl(0, k) << " = " << ldv << "(" << row_at(k, "max(ra - 1, " + std::to_string(-M.w0) + ")") << ");\n";
  for (int k = 0; k < K; ++k) o << in3 << "const " << TV << " b" << k << " = " << ldv << "(" << row_at(k, "min(rz, " + std::to_string(X.shape[0] - 1 - M.w0) + ")") << ");\n";
  for (int j = 1; j <= 1 + M.D; ++j) {
    o << in3 << "if (ra + " << j - 1 << " < rz) {\n";
    for (int k = 0; k < K; ++k) o << in3 << "  " << sl(j, k) << " = " << ldv << "(" << row_at(k, "ra + " + std::to_string(j - 1)) << ");\n";
    o << in3 << "}\n";
  }
  auto below = [&](int k) { return "mb" + sfx + " + (" + std::to_string(k * AT) + " + threadIdx.x) * " + std::to_string(V); };
  for (int k = 0; k < K; ++k) {
    if (V > 1) o << in3 << stv << "(" << below(k) << ", b" << k << ");\n";
    else o << in3 << "*(" << below(k) << ") = b" << k << ";\n";
  }
  for (int j = 2; j <= 1 + M.D; ++j) {
    o << in3 << "if (ra + " << j - 1 << " == rz) {\n";
    for (int k = 0; k < K; ++k) o << in3 << "  " << sl(j, k) << " = b" << k << ";\n";
    o << in3 << "}\n";
  }
  o << in2 << "}\n";
  if (pan) {
    // columns: element e of the vector before (after) the panel, rows -1 .. BR,
    // by the threads that own vectors (a panel is one group; the others have no rows)
    for (const auto& kv : eidx) {
      const int dv = kv.first.first, e = kv.first.second;
      const std::string v = dv < 0 ? "pb - 1" : "pb + " + std::to_string(M.PC);
      o << in2 << "if (" << v << " >= 0 && " << v << " < " << M.NC << ")\n";
      o << in2 << "  for (int i = threadIdx.x; i < rz - ra + 2; i += " << M.GT << ") mp" << sfx << "[" << kv.second * (M.BR + 2)
        << " + i] = ld(" << ptr(out->root) << " + (i64)min(max(ra - 1 + i + " << M.w0 << ", 0), " << X.shape[0] - 1 << ") * " << X.stride[0] << "LL + (i64)(" << v << " + "
        << M.pv0 << ") * " << V << " + " << e << ");\n";
    }
  }
  auto put_edges = [&](int j, const std::string& pad) {
    const int slot = ((j % RS) + RS) % RS;
    for (const auto& kv : eidx) {
      const int dv = kv.first.first, e = kv.first.second;
      o << pad << "if (lane == " << (dv < 0 ? 31 : 0) << " && act) {";
      for (int k = 0; k < K; ++k)
        o << " me" << sfx << "[" << (slot * NE + kv.second) * K * NW << " + wid * " << K << " + " << k << "] = " << sl(j, k)
          << (V > 1 ? ".v[" + std::to_string(e) + "]" : std::string()) << ";";
      o << " }\n";
    }
  };
  if (NE) {
    put_edges(0, in2);
    put_edges(1, in2);
  }
  // the rows and columns next to the band have been read (and used) here
  o << in2 << "{ u32 used_ = 0u";
  for (int k = 0; k < K; ++k)
    for (int l = 0; l < V; ++l) o << " ^ bits_of(" << sl(0, k) << (V > 1 ? ".v[" + std::to_string(l) + "]" : std::string()) << ")";
  o << ";\n" << in2 << "  if (used_ == 0x7fc5a3d1u) wave_pause(); }\n";
  o << in2 << "march_raise(P.flags, fw" << raises("fw") << ");\n";
  o << in2 << "for (int n0 = 0; n0 < " << M.BR << "; n0 += " << steps << ") {\n";
  for (int u = 0; u < steps; ++u) {
    o << in2 << "  { // row ra + n0 + " << u << "\n";
    o << in3 << "if (n0 + " << u << " >= " << M.BR << ") break;\n";
    o << in3 << "const int i = ra + n0 + " << u << ";\n";
    o << in3 << "const bool row = act && i < rz;\n";
    // the row D + 1 below, or the saved one under the band
    o << in3 << "if (act && i + " << M.D + 1 << " < rz) {\n";
    for (int k = 0; k < K; ++k)
      o << in3 << "  " << sl(u + RS - 1, k) << " = " << ldv << "(" << row_at(k, "i + " + std::to_string(M.D + 1)) << ");\n";
    o << in3 << "} else if (act && i + " << M.D + 1 << " == rz) {\n";
    for (int k = 0; k < K; ++k) o << in3 << "  " << sl(u + RS - 1, k) << " = " << ldv << "(" << below(k) << ");\n";
    o << in3 << "}\n";
    if (NE) {
      put_edges(u + 2, in3);
      o << in3 << "__syncthreads();\n";
    }
    std::map<std::tuple<int, int, int>, std::string> xv;
    for (const auto& s : need) {
      const int d0 = std::get<0>(s), dv = std::get<1>(s), e = std::get<2>(s), ei = eidx.at({dv, e});
      const int slot = (u + 1 + d0 + RS) % RS;
      const std::string nm = "x" + std::to_string(d0 + 1) + (dv < 0 ? "m" : "p") + std::to_string(e);
      xv[s] = nm;
      for (int k = 0; k < K; ++k) {
        o << in3 << T1 << " " << nm << "_" << k << " = " << (dv > 0 ? "__shfl_down_sync" : "__shfl_up_sync") << "(0xffffffffu, "
          << sl(u + 1 + d0, k) << (V > 1 ? ".v[" + std::to_string(e) + "]" : std::string()) << ", 1);\n";
        // across warps: the neighbouring vector is in the warp before
        // (after), or, past the group's last warp, in the next k
        const int base = (slot * NE + ei) * K * NW;
        const int wg = M.GT / 32;
        const std::string w = "wid";
        o << in3 << "if (lane == " << (dv > 0 ? 31 : 0) << " && act) {\n";
        const std::string at = "me" + sfx + "[" + std::to_string(base) + " + ";
        std::string panel = pan ? "mp" + sfx + "[" + std::to_string(ei * (M.BR + 2)) + " + i - ra + " + std::to_string(1 + d0) + "]" : "";
        if (dv > 0) {
          o << in3 << "  if (lw < " << wg - 1 << ") " << nm << "_" << k << " = " << at << "(" << w << " + 1) * " << K << " + " << k << "];\n";
          if (k + 1 < K)
            o << in3 << "  else " << nm << "_" << k << " = " << at << "(" << w << " - " << wg - 1 << ") * " << K << " + " << k + 1 << "];\n";
          else if (pan)
            o << in3 << "  else if (row) " << nm << "_" << k << " = " << panel << ";\n";
        } else {
          o << in3 << "  if (lw > 0) " << nm << "_" << k << " = " << at << "(" << w << " - 1) * " << K << " + " << k << "];\n";
          if (k > 0)
            o << in3 << "  else " << nm << "_" << k << " = " << at << "(" << w << " + " << wg - 1 << ") * " << K << " + " << k - 1 << "];\n";
          else if (pan)
            o << in3 << "  else if (row) " << nm << "_" << k << " = " << panel << ";\n";
        }
        o << in3 << "}\n";
      }
    }
    std::vector<std::string> slots, none;
    for (int k = 0; k < K; ++k) {
      slots.push_back("u" + std::to_string(k));
      none.push_back("");
      for (const Rd& rd : E.reads) {
        o << in3 << "const " << TV << " " << rd.var << "_u" << k << " = " << (V > 1 ? "{{" : "");
        for (int l = 0; l < V; ++l) {
          const auto s = src(rd, l);
          o << (l ? ", " : "");
          if (std::get<1>(s)) o << xv.at(s) << "_" << k;
          else o << sl(u + 1 + std::get<0>(s), k) << (V > 1 ? ".v[" + std::to_string(std::get<2>(s)) + "]" : std::string());
        }
        o << (V > 1 ? "}};\n" : ";\n");
      }
    }
    const auto outvars = emit_compute(n, E, V, slots, none, in3);
    const auto& vv = outvars.at(okey);
    if (u == 0)
      o << in3 << "if (n0 == 0 && !(mok = march_wait(P.flags, " << M.NB << "LL, " << M.PN << "LL, fw, ctl, P.timeout_ns))) break;\n";
    o << in3 << "if (row) {\n";
    for (int k = 0; k < K; ++k) {
      const std::string at = row_at(k, "i"), jn = "j" + std::to_string(k);
      if (V == 1) {
        o << in3 << "  if (s" << k << "_ && " << jn << " >= 0 && " << jn << " < " << M.cols << ") *(" << at << ") = " << vv[k] << ";\n";
        continue;
      }
      o << in3 << "  if (s" << k << "_ && " << jn << " >= 0 && " << jn << " + " << V << " <= " << M.cols << ") " << stv << "(" << at << ", " << TV << "{{";
      for (int l = 0; l < V; ++l) o << (l ? ", " : "") << vv[k * V + l];
      o << "}});\n" << in3 << "  else if (s" << k << "_) {\n";
      for (int l = 0; l < V; ++l)
        o << in3 << "    if (" << jn << " + " << l << " >= 0 && " << jn << " + " << l << " < " << M.cols << ") *(" << at << " + " << l << ") = "
          << vv[k * V + l] << ";\n";
      o << in3 << "  }\n";
    }
    o << in3 << "}\n";
    o << in2 << "  }\n";
  }
  o << in2 << "}\n";
  if (sweeps > 1) o << in2 << "if (mok && sw + 1 < " << sweeps << ") march_raise(P.flags, fw + 1" << raises("fw + 1") << ");\n";
  o << in2 << "}\n" << ind << "}\n";
  if (sweeps > 1) o << ind << "}\n";
  o << ind << "if (!mok) break;\n";
  o << "    }\n";
}

// The tasks of a sweep with its temporaries renamed: two sweeps with equal
// signatures differ in their temporaries and immediates only.
std::string Gen::sweep_signature(int g) const {
  std::map<int64_t, int> temps;
  std::string k;
  for (int i = S.groups[g].begin; i < S.groups[g + 1].end; ++i) {
    k += "|" + std::to_string(S.tasks[i].op);
    for (const Arg& a : S.tasks[i].args) {
      if (a.imm) k += ",i";
      else if (a.nd > 0 && R(a.root).temp)
        k += ",t" + std::to_string(temps.emplace(a.root, (int)temps.size()).first->second) + "@" + a.part.key();
      else k += "," + akey(a);
      k += ":" + std::to_string(a.priv);
    }
  }
  return k;
}

void Gen::emit_wave(int g) {
  const WaveGeom W = wave_geometry(S, g);
  const Group &A = S.groups[g], &B = S.groups[g + 1];
  const int BD = S.block - 32, V = W.V, Rr = W.R, cd = W.nd - 1;
  Nest n;
  n.first = A.begin;
  n.last = B.end;
  n.dims = 2;
  n.vec = V;
  n.rank = W.nd;
  BodyEnv E;
  std::set<std::string> written;
  struct Out { std::string key; const Arg* a; };
  std::vector<Out> outs;
  std::set<std::string> seen;
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    for (size_t ai = 0; ai < t.args.size(); ++ai) {
      const Arg& a = t.args[ai];
      if (a.imm || a.nd == 0) continue;
      const std::string k = akey(a);
      const bool out = ai + 1 == t.args.size();
      if (!out && a.is_r() && !written.count(k) && seen.insert(k).second)
        E.reads.push_back({k, &a, "m" + std::to_string(E.reads.size()), !R(a.root).written});
      if (out) {
        if (written.insert(k).second && !R(a.root).temp) outs.push_back({k, &a});
      }
    }
  }
  const std::string ind = "      ", in2 = ind + "    ";
  const int dt = outs[0].a->dtype;
  const std::string T1 = T(dt), TV = V == 4 ? "f32x4" : (V == 2 ? "f64x2" : T1);
  const std::string ldv = V == 4 ? "ld4" : "ld2", stv = V == 4 ? "st4" : "st2";
  ++kc.nwaves;
  kc.wave_tiles = std::max(kc.wave_tiles, W.tiles);
  if (W.reach > 0) kc.wave_reach = std::max(kc.wave_reach, W.reach);
  wave_blocks = std::max(wave_blocks, W.min_blocks);
  o << "    { // groups " << g << ", " << g + 1 << ": tasks " << n.first << ".." << n.last - 1
    << ", one in-place sweep of " << W.tiles << " tiles\n";
  for (int i = n.first; i < n.last; ++i) {
    const Task& t = S.tasks[i];
    for (size_t ai = 0; ai < t.args.size(); ++ai) {
      if (!t.args[ai].imm) continue;
      const std::string nm = "k" + std::to_string(i) + "_" + std::to_string(ai);
      o << ind << "const " << T1 << " " << nm << " = " << imm_expr(i, (int)ai, dt) << ";\n";
      E.immv[{i, (int)ai}] = nm;
    }
  }
  o << ind << "const u64 fw = ep_ + " << kc.nwaves << "ull;\n";
  // the ordering warp
  int64_t nflag = 0;
  for (const auto& rr : W.readers) nflag += rr.second - rr.first + 1;
  o << ind << "if (threadIdx.x >= " << BD << ") {\n";
  o << ind << "  for (i64 t = blockIdx.x; t < " << W.tiles << "LL; t += gridDim.x, ++wrd_) {\n";
  o << ind << "    bool ok_ = wave_raise(&wsync_, wrd_, P.flags + t, ctl, fw, P.timeout_ns" << raises("fw") << ");\n";
  if (nflag > 0) {
    o << ind << "    for (int i = threadIdx.x & 31; i < " << nflag << " && ok_; i += 32) {\n";
    o << ind << "      const i64 u = t + i + (";
    int64_t at = 0;
    for (size_t k = 0; k < W.readers.size(); ++k) {
      const std::string v = std::to_string(W.readers[k].first - at) + "LL";
      at += W.readers[k].second - W.readers[k].first + 1;
      o << (k + 1 < W.readers.size() ? "i < " + std::to_string(at) + " ? " + v + " : " : v);
    }
    o << ");\n";
    o << ind << "      if (u >= 0 && u < " << W.tiles << "LL && !wave_poll(P.flags + u, fw, ctl, P.timeout_ns)) ok_ = false;\n";
    o << ind << "    }\n";
  }
  o << ind << "    if (!wave_release(&wsync_, wrd_, ok_, ctl, fw)) break;\n";
  o << ind << "  }\n";
  o << ind << "} else {\n";
  o << ind << "bool live = false;\n" << ind << "u32 prb = 0, py = 0, pjv = 0;\n";
  o << ind << "bool pact = false;\n";
  for (size_t k = 0; k < outs.size(); ++k)
    for (int u = 0; u < Rr; ++u) o << ind << TV << " h" << k << "_" << u << (V > 1 ? " = {};\n" : " = 0;\n");
  o << ind << "for (i64 t = blockIdx.x;; t += gridDim.x) {\n";
  o << ind << "  const bool have = t < " << W.tiles << "LL;\n";
  // threads past the last cell repeat it (their results are not stored)
  o << ind << "  const u32 c = have ? min((u32)t * " << BD << "u + threadIdx.x, " << W.cells - 1 << "u) : 0u;\n";
  o << ind << "  const u32 rb = c / " << W.lines * W.nvx << "u;\n";
  if (W.nd == 3) {
    o << ind << "  const u32 rem = c - rb * " << W.lines * W.nvx << "u;\n";
    o << ind << "  const u32 y = rem / " << W.nvx << "u;\n" << ind << "  const u32 jv = rem - y * " << W.nvx << "u;\n";
  } else {
    o << ind << "  const u32 y = 0, jv = c - rb * " << W.nvx << "u;\n";
  }
  for (size_t k = 0; k < outs.size(); ++k)
    for (int u = 0; u < Rr; ++u) o << ind << "  " << TV << " n" << k << "_" << u << (V > 1 ? " = {};\n" : " = 0;\n");
  o << ind << "  if (have) {\n";
  // loads: distinct (root, slice, line, vector), one element where only one
  // of the vector is used
  struct Ld { std::string var; bool scalar = false; int elem = 0; bool ro = false; std::set<int> need; int64_t root; int64_t k0, o1, vb; };
  std::map<std::string, int> lidx;
  std::vector<Ld> loads;
  auto want = [&](const Rd& rd, int64_t k0, int64_t o1, int64_t vb, int e) -> int {
    const std::string k = std::to_string(rd.a->root) + "," + std::to_string(k0) + "," + std::to_string(o1) + "," + std::to_string(vb);
    auto it = lidx.find(k);
    if (it == lidx.end()) {
      Ld L;
      L.var = "w" + std::to_string(loads.size());
      L.ro = rd.ro;
      L.root = rd.a->root;
      L.k0 = k0;
      L.o1 = o1;
      L.vb = vb;
      it = lidx.emplace(k, (int)loads.size()).first;
      loads.push_back(L);
    }
    loads[it->second].need.insert(e);
    return it->second;
  };
  // element of lane l of read rd in slot u: (load, element)
  auto source = [&](const Rd& rd, int u, int l) {
    const int64_t q = origin_of(*rd.a, cd) - W.lead + l;
    const int64_t vb = floor_div(q, V);
    const int e = (int)(q - vb * V);
    return std::make_pair(want(rd, origin_of(*rd.a, 0) + u, W.nd == 3 ? origin_of(*rd.a, 1) : 0, vb, e), e);
  };
  for (int u = 0; u < Rr; ++u)
    for (const Rd& rd : E.reads)
      for (int l = 0; l < V; ++l) source(rd, u, l);
  std::map<std::string, std::string> rowp, colv;
  int nrow = 0;
  for (Ld& L : loads) {
    const LaunchRoot& r = R(L.root);
    const std::string rk = std::to_string(L.root) + "," + std::to_string(L.k0) + "," + std::to_string(L.o1);
    if (!rowp.count(rk)) {
      const std::string nm = "p" + std::to_string(nrow++);
      o << in2 << "const " << T1 << "* " << nm << " = " << ptr(L.root) << " + ";
      const std::string row = "rb * " + std::to_string(Rr) + "u + " + std::to_string(L.k0) + "u";
      // slices past the end (a ragged last block) repeat the store's last one
      if (W.ext[0] % Rr) o << "(i64)min(" << row << ", " << r.shape[0] - 1 << "u)";
      else o << "(i64)(" << row << ")";
      o << " * " << r.stride[0] << "LL";
      if (W.nd == 3) o << " + (i64)(y + " << L.o1 << "u) * " << r.stride[1] << "LL";
      o << ";\n";
      rowp[rk] = nm;
    }
    // vectors before the row's first or after its last serve no valid lane:
    // clamped into the row
    const int64_t nv = V > 1 ? r.stride[cd - 1] / V : r.shape[cd];
    const bool lo = L.vb < 0, hi = W.nvx - 1 + L.vb > nv - 1;
    const std::string ck = std::to_string(L.vb) + (lo ? "l" : "") + (hi ? "h" + std::to_string(nv) : "");
    if (!colv.count(ck)) {
      const std::string nm = "c" + std::to_string(colv.size());
      std::string e = "((int)jv + " + std::to_string(L.vb) + ")";
      if (lo) e = "max(" + e + ", 0)";
      if (hi) e = "min(" + e + ", " + std::to_string(nv - 1) + ")";
      o << in2 << "const int " << nm << " = " << e << " * " << V << ";\n";
      colv[ck] = nm;
    }
    const std::string ad = rowp[rk] + " + " + colv[ck];
    L.scalar = V > 1 && L.need.size() == 1;
    if (L.scalar) {
      L.elem = *L.need.begin();
      o << in2 << "const " << T1 << " " << L.var << " = " << (L.ro ? "ldro(" : "ld(") << ad << " + " << L.elem << ");\n";
    } else if (V > 1) {
      o << in2 << "const " << TV << " " << L.var << " = " << ldv << (L.ro ? "ro(" : "(") << ad << ");\n";
    } else {
      o << in2 << "const " << T1 << " " << L.var << " = " << (L.ro ? "ldro(" : "ld(") << ad << ");\n";
    }
  }
  // assemble the lanes, compute, keep the results
  std::vector<std::string> slots, none;
  for (int u = 0; u < Rr; ++u) {
    slots.push_back("u" + std::to_string(u));
    none.push_back("");
    for (const Rd& rd : E.reads) {
      o << in2 << "const " << TV << " " << rd.var << "_u" << u << " = ";
      if (V > 1) o << "{{";
      for (int l = 0; l < V; ++l) {
        const auto se = source(rd, u, l);
        const Ld& L = loads[se.first];
        o << (l ? ", " : "") << L.var;
        if (V > 1 && !L.scalar) o << ".v[" << se.second << "]";
      }
      o << (V > 1 ? "}};\n" : ";\n");
    }
  }
  const auto outvars = emit_compute(n, E, V, slots, none, in2);
  for (size_t k = 0; k < outs.size(); ++k) {
    const auto& vv = outvars.at(outs[k].key);
    for (int u = 0; u < Rr; ++u) {
      const std::string h = "n" + std::to_string(k) + "_" + std::to_string(u);
      if (V == 1) o << in2 << h << " = " << vv[u] << ";\n";
      else
        for (int l = 0; l < V; ++l) o << in2 << h << ".v[" << l << "] = " << vv[u * V + l] << ";\n";
    }
  }
  // Every value computed from the loads, as one word.  The elements of one
  // result are distinct cells, but two results may hold the same values (an
  // intermediate that the application keeps and the centre it is copied to) or
  // negated ones, so results are combined by a rotation and a sum, which do not
  // cancel as an exclusive or of equal words does.
  for (size_t k = 0; k < outs.size(); ++k) {
    std::string x;
    for (int u = 0; u < Rr; ++u)
      for (int l = 0; l < V; ++l)
        x += (x.empty() ? "" : " ^ ") + std::string("bits_of(n") + std::to_string(k) + "_" + std::to_string(u) +
             (V > 1 ? ".v[" + std::to_string(l) + "]" : std::string()) + ")";
    o << in2 << (k == 0 ? "u32 used_ = " + x : "used_ = __funnelshift_l(used_, used_, 1) + (" + x + ")") << ";\n";
  }
  o << ind << "  wave_read_done(&wsync_, wrd_ + (live ? 1u : 0u), used_);\n";
  o << ind << "  }\n";
  // the previous tile's results, once every tile that reads it has read
  o << ind << "  if (live) {\n";
  o << ind << "    if (!wave_ready(&wsync_, wrd_, ctl, fw, P.timeout_ns)) break;\n";
  o << ind << "    ++wrd_;\n";
  o << ind << "    if (pact) {\n";
  for (size_t k = 0; k < outs.size(); ++k) {
    const Arg& a = *outs[k].a;
    const LaunchRoot& r = R(a.root);
    o << ind << "      {\n";
    o << ind << "        " << T1 << "* q_ = " << ptr(a.root) << " + (i64)(prb * " << Rr << "u + " << origin_of(a, 0) << "u) * "
      << r.stride[0] << "LL";
    if (W.nd == 3) o << " + (i64)(py + " << origin_of(a, 1) << "u) * " << r.stride[1] << "LL";
    o << " + (i64)pjv * " << V << " + " << origin_of(a, cd) - W.lead << ";\n";
    o << ind << "        const int j_ = (int)pjv * " << V << " - " << W.lead << ";\n";
    for (int u = 0; u < Rr; ++u) {
      const std::string h = "h" + std::to_string(k) + "_" + std::to_string(u);
      const std::string at_ = "q_ + " + std::to_string(u * r.stride[0]) + "LL";
      o << ind << "        ";
      if (W.ext[0] % Rr) o << "if (prb * " << Rr << "u + " << u << "u < " << W.ext[0] << "u) ";
      if (V == 1) {
        o << "*(" << at_ << ") = " << h << ";\n";
        continue;
      }
      o << "{\n";
      o << ind << "          if (j_ >= 0 && j_ + " << V << " <= " << W.ext[cd] << ") " << stv << "(" << at_ << ", " << h << ");\n";
      o << ind << "          else {\n";
      for (int l = 0; l < V; ++l)
        o << ind << "            if (j_ + " << l << " >= 0 && j_ + " << l << " < " << W.ext[cd] << ") *(" << at_ << " + " << l
          << ") = " << h << ".v[" << l << "];\n";
      o << ind << "          }\n" << ind << "        }\n";
    }
    o << ind << "      }\n";
  }
  o << ind << "    }\n" << ind << "  }\n";
  o << ind << "  if (!have) break;\n";
  for (size_t k = 0; k < outs.size(); ++k)
    for (int u = 0; u < Rr; ++u) o << ind << "  h" << k << "_" << u << " = n" << k << "_" << u << ";\n";
  o << ind << "  live = true;\n";
  o << ind << "  pact = (u32)t * " << BD << "u + threadIdx.x < " << W.cells << "u;\n";
  o << ind << "  prb = rb;\n" << ind << "  py = y;\n" << ind << "  pjv = jv;\n";
  o << ind << "}\n";
  o << ind << "}\n" << ind << "__syncthreads();\n";
  o << ind << "if (wsync_.fail) break;\n";
  o << "    }\n";
}

KernelCode Gen::run() {
  emit_params();
  std::ostringstream body;
  // the kernel body is generated into `o`; header assembled afterwards
  // x windows are staged by per-point nests whose SpMV rows are not shared
  // between lanes (the same test emit_vector_group and emit_nest apply)
  for (int g = 0; g < (int)S.groups.size() && !stage; ++g) {
    if (S.groups[g].scalar) continue;
    const std::vector<Nest> ns = nests_of(g);
    bool flat = ns.size() == 1;
    for (int i = S.groups[g].begin; i < S.groups[g].end && flat; ++i)
      if (is_reduction(S.tasks[i].op)) flat = false;
    if (flat && space_arg(S.tasks[S.groups[g].begin]).nd > 3) flat = false;
    for (const Nest& n : ns)
      if (!flat && n.dims == 1 && !n.coop)
        for (int i = n.first; i < n.last; ++i)
          if (S.tasks[i].op == DFS_OP_SPMV && S.tasks[i].args.size() == 6) stage = true;
  }
  o << "  __shared__ double red_buf[" << S.block << "];\n";
  o << "  Ctl* ctl = P.ctl;\n";
  if (stage) {
    kc.dyn_smem = DFS_SPMV_STAGE_BYTES;
    o << "  extern __shared__ __align__(128) unsigned char dfs_xs_raw[];\n";
    o << "  __shared__ __align__(8) u64 xs_mbar_;\n  u32 xs_ph_ = 0;\n  bool xs_live_ = true;\n";
    o << "  xstage_init(&xs_mbar_);\n";
  }
  bool by_rows = false;
  for (int g = 0; g < (int)S.groups.size() && !stage && !by_rows; ++g)
    if (!S.groups[g].scalar)
      for (const Nest& n : nests_of(g)) by_rows = by_rows || n.rows;
  if (by_rows) {
    kc.dyn_smem = S.block / 32 * kSpmvWarpBytes;
    o << "  extern __shared__ __align__(128) unsigned char dfs_sp_raw[];\n";
  }
  emit_prologue();
  for (const Group& G : S.groups)
    if (G.wave) {
      o << "  const u64 ep_ = ctl->epoch;  // the last CTA to exit moves it on\n";
      o << "  __shared__ __align__(8) WaveSync wsync_;\n  u32 wrd_ = 0;\n  wave_init(&wsync_);\n";
      break;
    }
  int64_t march_smem = 0;
  for (int g = 0; g + 1 < (int)S.groups.size(); ++g)
    if (S.groups[g].wave) {
      const MarchGeom M = march_geometry(S, g);
      if (M.ok) march_smem = std::max(march_smem, M.smem);
    }
  if (march_smem) o << "  __shared__ __align__(16) unsigned char march_raw[" << march_smem << "];\n";
  o << "  do {\n";
  for (int g = 0; g < (int)S.groups.size(); ++g) {
    if (g > 0 && !S.groups[g - 1].scalar) {
      ++nbar;
      o << "    if (!grid_barrier(ctl, " << nbar << "u, P.timeout_ns"
        << (S.debug_skip == nbar ? ", blockIdx.x != 0" : "") << ")) break;\n";
      const int h = emit_warp0_scalars(g);
      if (h > g) {
        g = h - 1;
        continue;
      }
    }
    if (S.groups[g].wave) {
      if (march_geometry(S, g).ok) {
        int sweeps = 1;
        const std::string sig = sweep_signature(g);
        while (g + 2 * sweeps + 1 < (int)S.groups.size() && S.groups[g + 2 * sweeps].wave &&
               S.groups[g + 2 * sweeps + 1].end - S.groups[g + 2 * sweeps].begin == S.groups[g + 1].end - S.groups[g].begin &&
               sweep_signature(g + 2 * sweeps) == sig)
          ++sweeps;
        emit_march(g, sweeps);
        g += 2 * sweeps - 1;
        continue;
      }
      emit_wave(g);
      ++g;
      continue;
    }
    emit_group(g);
  }
  o << "  } while (0);\n";
  // The exit count costs every launch a round trip to L2 after its last store;
  // a kernel without barriers, sums, scalars to publish or sweeps leaves the
  // control block as it found it (Black-Scholes, 1,000,003 options, both in turn:
  // 10.27 -> 10.14 us).
  bool exits = nbar > 0 || !pending_red.empty() || kc.nwaves > 0;
  for (const LaunchRoot& r : S.roots) exits = exits || (r.zero_d && r.live_out && r.param >= 0);
  if (exits) {
    o << "  if (last_cta(ctl)) {\n";
    if (!pending_red.empty()) {
      o << "    if (ld_relaxed_int(&ctl->err) == 0) {\n";
      emit_finalise("      ");
      o << "    }\n";
    }
    o << "    if (threadIdx.x == 0) {\n";
    for (const LaunchRoot& r : S.roots) {
      if (!r.zero_d || !r.live_out || r.param < 0) continue;
      o << "      *" << ptr(r.root) << " = " << sreg.at(r.root) << ";\n";
    }
    if (kc.nwaves) o << "      ctl->epoch = ep_ + " << kc.nwaves << "ull;\n";
    o << "    }\n";
    o << "    ctl_reset(ctl);\n";
    o << "  }\n";
  }
  kc.nbarriers = nbar;

  std::ostringstream src;
  src << "#include \"dfs_device.cuh\"\nusing namespace dfs;\n";
  if (by_rows) src << "static_assert(kSpmvWarpBytes == " << kSpmvWarpBytes << ", \"shared memory of a warp\");\n";
  src << "struct Params {\n  void* p[" << std::max(1, kc.nptr) << "];\n  double imm[" << std::max(1, kc.nimm)
      << "];\n  void* partials;\n  Ctl* ctl;\n  u64 timeout_ns;\n  i64 red_stride;\n"
      << (kc.nwaves ? "  u64* flags;\n" : "") << "};\n";
  const std::string body_s = o.str();
  const size_t h = std::hash<std::string>{}(body_s);
  char nm[64];
  snprintf(nm, sizeof nm, "dfs_k%016zx", h);
  kc.name = nm;
  const int min_blocks = S.min_blocks > 0 ? S.min_blocks : wave_blocks;
  src << "extern \"C\" __global__ void __launch_bounds__(" << S.block << (min_blocks > 0 ? ", " + std::to_string(min_blocks) : std::string()) << ") " << kc.name
      << "(const __grid_constant__ Params P) {\n"
      << body_s << "}\n";
  kc.source = src.str();
  kc.key = kc.source;
  int64_t stride = 1;
  for (int64_t p : kc.red_points) stride = std::max(stride, p);
  kc.partial_bytes = (size_t)kc.nred * (size_t)stride * 8;
  return kc;
}

}  // namespace

const char* op_device_fn(int op) { return op_fn(op); }

std::string LaneOps::shared(const std::map<std::string, std::string>& m, const std::string& a) const {
  auto it = m.find(a);
  if (it != m.end()) return it->second;
  auto ng = neg_.find(a);
  if (ng != neg_.end()) {
    it = m.find(ng->second);
    if (it != m.end()) return it->second;
  }
  return std::string();
}

void LaneOps::emit(std::ostream& o, const std::string& pad, const std::string& T, int op, const std::string& res,
                   const std::vector<std::string>& in) {
  define(res);
  if (op == DFS_OP_ERF) {
    // |-a| = |a| bit for bit, so erf(|a|) serves a and its negation
    std::string m = shared(mag_, in[0]);
    if (m.empty()) {
      m = res + "_m";
      o << pad << "const " << T << " " << m << " = erf_mag(" << in[0] << ");\n";
    }
    mag_[in[0]] = m;
    o << pad << "const " << T << " " << res << " = erf_sign(" << m << ", " << in[0] << ");\n";
    return;
  }
  if (op == DFS_OP_NCDF) {
    // the scaled arguments of a and -a differ only in sign (round to
    // nearest is symmetric), so they share erf of their magnitude
    const std::string y = res + "_y";
    o << pad << "const " << T << " " << y << " = ncdf_arg(" << in[0] << ");\n";
    std::string m = shared(nmag_, in[0]);
    if (m.empty()) {
      m = res + "_m";
      o << pad << "const " << T << " " << m << " = erf_mag(" << y << ");\n";
    }
    nmag_[in[0]] = m;
    o << pad << "const " << T << " " << res << " = ncdf_of_erf(erf_sign(" << m << ", " << y << "));\n";
    return;
  }
  o << pad << "const " << T << " " << res << " = " << op_fn(op) << "(" << in[0];
  for (size_t k = 1; k < in.size(); ++k) o << ", " << in[k];
  o << ");\n";
  if (op == DFS_OP_NEG) {
    neg_.emplace(res, in[0]);
    neg_.emplace(in[0], res);
  }
}

std::string LaneOps::mag_of(int op, const std::string& in0) const {
  return shared(op == DFS_OP_NCDF ? nmag_ : mag_, in0);
}

void LaneOps::set_mag(int op, const std::string& in0, const std::string& m) {
  (op == DFS_OP_NCDF ? nmag_ : mag_)[in0] = m;
}

void LaneOps::define(const std::string& res) {
  if (!defined_.insert(res).second)
    throw std::runtime_error("code generator: value " + res + " defined twice in one loop body");
}

namespace {

// A task of one list writes or reduces a store that a task of the other uses.
bool conflict(const std::vector<Task>& T, const std::vector<int>& a, const std::vector<int>& b) {
  std::set<int64_t> used[2], set[2];
  for (int side = 0; side < 2; ++side)
    for (int i : side ? b : a)
      for (const Arg& x : T[i].args) {
        if (x.imm) continue;
        used[side].insert(x.root);
        if (x.is_w() || x.is_rd()) set[side].insert(x.root);
      }
  for (int side = 0; side < 2; ++side)
    for (int64_t r : set[side])
      if (used[1 - side].count(r)) return true;
  return false;
}

// Groups a (earlier) and b run as one loop nest: the fusion constraints hold
// for the tasks in a row, the nest sweeps as each of them alone does (so no
// sum changes its order), and b uses an array that a has in registers.
bool joins(const LaunchSpec& S, const std::vector<int>& a, const std::vector<int>& b) {
  LaunchSpec J;
  J.block = S.block;
  J.unroll = S.unroll;
  J.roots = S.roots;
  J.root_index = S.root_index;
  std::set<int64_t> arrays;
  bool shared = false;
  for (int side = 0; side < 2; ++side) {
    for (int i : side ? b : a) {
      const Task& t = S.tasks[i];
      if (t.scalar() || t.op == DFS_OP_SPMV) return false;
      for (const Arg& x : t.args) {
        if (x.imm || x.nd == 0) continue;
        if (side == 0) arrays.insert(x.root);
        else if (arrays.count(x.root)) shared = true;
      }
      J.tasks.push_back(t);
    }
  }
  if (!shared || longest_fusible_prefix(J.tasks, 0) != (int)J.tasks.size()) return false;
  const int na = (int)a.size(), n = (int)J.tasks.size();
  for (const auto& be : {std::make_pair(0, na), std::make_pair(na, n), std::make_pair(0, n)}) {
    Group G;
    G.begin = be.first;
    G.end = be.second;
    J.groups.push_back(G);
  }
  Gen gen(J);
  const std::string f = gen.form(2);
  return !f.empty() && f == gen.form(0) && f == gen.form(1);
}

}  // namespace

// The prefixes of a launch are cut wherever a scalar task stands between two
// sweeps of the same arrays (norm, then sum, then dot), and every sweep is a
// phase with its own grid barrier and its own pass over memory.  A group that
// uses nothing the phases between produce moves up into the earlier sweep.
// Bound by HBM: z = d / |d|, sum(y), x.y over 2^24 FP32 elements ran four
// sweeps (100.5 us a pass), the sums re-reading x and y; joined, two (65.5 us).
void pack_groups(LaunchSpec& S) {
  std::vector<std::vector<int>> out;
  std::vector<Group> gs;
  bool moved = false;
  for (const Group& G : S.groups) {
    std::vector<int> k;
    for (int i = G.begin; i < G.end; ++i) k.push_back(i);
    bool joined = false;
    if (!G.scalar)
      for (int j = (int)out.size() - 1; j >= 0 && !joined; --j) {
        if (!gs[j].scalar && joins(S, out[j], k)) {
          out[j].insert(out[j].end(), k.begin(), k.end());
          joined = moved = true;
        } else if (conflict(S.tasks, out[j], k)) {
          break;
        }
      }
    if (joined) continue;
    out.push_back(k);
    gs.push_back(G);
  }
  if (!moved) return;
  std::vector<Task> tasks;
  S.order.clear();
  for (size_t k = 0; k < out.size(); ++k) {
    gs[k].begin = (int)tasks.size();
    for (int i : out[k]) {
      tasks.push_back(S.tasks[i]);
      S.order.push_back(i);
    }
    gs[k].end = (int)tasks.size();
  }
  S.tasks = std::move(tasks);
  S.groups = std::move(gs);
}

KernelCode generate(const LaunchSpec& spec) {
  Gen g(spec);
  return g.run();
}

}  // namespace dfs
