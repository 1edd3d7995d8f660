// Host side of the library: the C ABI, the array-of-octrees build from
// refinement flags (Sec. II.B), the device block table and the per-step
// launch sequence (ghost refresh -> three PPM sweeps -> flux correction ->
// CFL/totals reduction), optionally replayed from a CUDA graph.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <unordered_set>
#include <vector>

#include "cello.h"
#include "cello_internal.h"
#include "morton.h"
#include "per_device.h"

using namespace cello;

namespace {

thread_local std::string g_last_error;

// Fields per cell: five conserved, plus rho e with the dual-energy formalism.
int nfields(const cello_mesh_desc& d) { return d.dual_energy ? 6 : 5; }

cello_status fail(cello_status st, const std::string& msg) {
  g_last_error = msg;
  return st;
}

// State pools and adjoints must start on a 256-byte boundary (the ABI's
// convention): the kernels move whole 32-byte sectors and 16-byte vectors,
// which a misaligned address would turn into a device fault.
bool misaligned(const void* p) { return p && (reinterpret_cast<uintptr_t>(p) & 255u) != 0; }
#define CELLO_REQUIRE_ALIGNED(p) \
  do { if (misaligned(p)) return fail(CELLO_EINVAL, #p " is not 256-byte aligned"); } while (0)

#define CELLO_CUDA(call)                                                                  \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess)                                                                \
      return fail(e_ == cudaErrorMemoryAllocation ? CELLO_ENOMEM : CELLO_ECUDA,           \
                  std::string(#call) + ": " + cudaGetErrorString(e_));                    \
  } while (0)

struct Node {
  int L, i, j, k;
};

inline unsigned long long pack(const Node& t) {
  return ((unsigned long long)t.L << 60) | ((unsigned long long)t.i << 40) | ((unsigned long long)t.j << 20) |
         (unsigned long long)t.k;
}

inline Node child(const Node& t, int o) {
  return Node{t.L + 1, 2 * t.i + (o & 1), 2 * t.j + ((o >> 1) & 1), 2 * t.k + (o >> 2)};
}

// Set of packed nodes: open addressing, linear probing.
class NodeSet {
 public:
  explicit NodeSet(size_t expected) {
    size_t cap = 64;
    while (cap < 2 * expected) cap *= 2;
    resize(cap);
  }
  bool insert(unsigned long long key) {   // false if it is there already
    if (2 * (count_ + 1) > slots_.size()) grow();
    const size_t i = find(key);
    if (slots_[i] == key + 1) return false;
    slots_[i] = key + 1;
    ++count_;
    return true;
  }
  bool contains(unsigned long long key) const { return slots_[find(key)] == key + 1; }

 private:
  std::vector<unsigned long long> slots_;   // key + 1, 0: empty (no packed node is all ones)
  size_t count_ = 0;
  int shift_ = 0;
  size_t find(unsigned long long key) const {
    size_t i = (size_t)((key * 0x9E3779B97F4A7C15ull) >> shift_);
    while (slots_[i] != 0 && slots_[i] != key + 1) i = (i + 1) & (slots_.size() - 1);
    return i;
  }
  void resize(size_t cap) {
    slots_.assign(cap, 0);
    shift_ = 64;
    for (size_t c = cap; c > 1; c /= 2) --shift_;
  }
  void grow() {
    std::vector<unsigned long long> old;
    old.swap(slots_);
    resize(old.size() * 2);
    for (unsigned long long v : old)
      if (v) slots_[find(v - 1)] = v;
  }
};

// The refined nodes of a mesh, by level; its leaves are their children that are
// not refined (and the roots that are not).
struct Tree {
  const cello_mesh_desc* d;
  NodeSet internal;
  std::vector<Node> level[12];
  Tree(const cello_mesh_desc& desc, size_t expected) : d(&desc), internal(expected) {}

  void refine(Node t) {   // the node and its ancestors
    while (internal.insert(pack(t))) {
      level[t.L].push_back(t);
      if (t.L == 0) break;
      t = Node{t.L - 1, t.i >> 1, t.j >> 1, t.k >> 1};
    }
  }

  bool wrap(int L, int a, int& v) const {
    const int nb = d->root[a] << L;
    if (v >= 0 && v < nb) return true;
    if (d->bc[a] != CELLO_PERIODIC) return false;
    v = ((v % nb) + nb) % nb;
    return true;
  }

  // True if a leaf two or more levels finer than node t touches it: some
  // same-level neighbour node is refined and one of its children that
  // touches t is refined too.
  bool touches_deeper(const Node& t) const {
    if (t.L + 2 > d->max_level) return false;
    for (int dz = -1; dz <= 1; ++dz)
      for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx) {
          if (!dx && !dy && !dz) continue;
          int v[3] = {t.i + dx, t.j + dy, t.k + dz};
          bool in = true;
          for (int a = 0; a < 3; ++a) in = in && wrap(t.L, a, v[a]);
          if (!in) continue;
          const Node nb{t.L, v[0], v[1], v[2]};
          if (!internal.contains(pack(nb))) continue;
          for (int o = 0; o < 8; ++o) {
            const int ox = o & 1, oy = (o >> 1) & 1, oz = o >> 2;
            if ((dx == 1 && ox) || (dx == -1 && !ox) || (dy == 1 && oy) || (dy == -1 && !oy) || (dz == 1 && oz) ||
                (dz == -1 && !oz))
              continue;
            if (internal.contains(pack(child(nb, o)))) return true;
          }
        }
    return false;
  }

  // 2:1 balance: a leaf that touches a leaf two levels finer is refined, until
  // there is none.  A refined node c asks for exactly the nodes one level
  // coarser that touch it, its parent's neighbours on the side of its octant (the
  // others are its parent), so one pass over the refined nodes from the finest
  // level up, 7 neighbours each, is the whole closure.
  void balance() {
    for (int L = d->max_level - 1; L >= 1; --L)
      for (size_t n = 0; n < level[L].size(); ++n) {
        const Node c = level[L][n];
        const int at[3] = {c.i, c.j, c.k};
        for (int mask = 1; mask < 8; ++mask) {
          int v[3];
          bool in = true;
          for (int a = 0; a < 3; ++a) {
            v[a] = at[a];
            if (mask >> a & 1) v[a] += (at[a] & 1) ? 1 : -1;
            in = in && wrap(L, a, v[a]);
          }
          if (in) refine(Node{L - 1, v[0] >> 1, v[1] >> 1, v[2] >> 1});
        }
      }
  }

  // The leaves under a node in Morton order.
  void emit(const Node& t, std::vector<Node>& out) const {
    if (!internal.contains(pack(t))) {
      out.push_back(t);
      return;
    }
    for (int o = 0; o < 8; ++o) emit(child(t, o), out);
  }
};

unsigned long long leaf_key(const cello_mesh_desc& d, const Node& t) {
  const int s = d.max_level - t.L;
  return morton3((unsigned)t.i << s, (unsigned)t.j << s, (unsigned)t.k << s);
}

}  // namespace

namespace cello {
void prepare_kernels() {
  static OncePerDevice once;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  once.run(dev, [] {
    prepare_kernels_f32();
    prepare_kernels_f64();
    // L2 fetch granularity of this process's context on the device: 64 bytes.
    // The ghost refresh reads 32-byte margin sectors of 160-byte rows; with the
    // limit left unset, misses fetched 128-byte lines (phase X: 3.2x its requested
    // sectors read from DRAM).  A hint of this context only, not a device setting.
    if (cudaDeviceSetLimit(cudaLimitMaxL2FetchGranularity, 64) != cudaSuccess)
      cudaGetLastError();   // a device that does not take the hint keeps its default
  });
}
}  // namespace cello

struct GraphEntry {
  const void* U;
  const double* dt;
  int parity;
  double cfl;
  double* dt_next;
  double* totals;
  cudaGraphExec_t exec;
  bool cfl_step = false;   // a cello_hydro_step_cfl graph (dt from the start state)
};

struct cello_mesh {
  cello_mesh_desc desc{};
  int B = 0, N = 0;
  std::vector<int4> leaves;
  std::vector<unsigned long long> keys;
  std::vector<int> face_slot;
  std::vector<CoarseFace> cfaces;   // fslot filled on the device only
  std::vector<int> group_start;
  int nslots = 0;
  // device tables: two allocations, d_table (sized by the leaves) and d_lists
  // (by the faces that are not same-level); the pointers below lie in them
  char* d_table = nullptr;
  char* d_lists = nullptr;
  int4* d_leaf = nullptr;
  unsigned long long* d_keys = nullptr;
  int8_t* d_kind = nullptr;
  int* d_idx = nullptr;
  int* d_fine8 = nullptr;
  int* d_face_slot = nullptr;
  CoarseFace* d_cfaces = nullptr;
  int* d_group_start = nullptr;
  double* d_reg = nullptr;
  double* d_partials = nullptr;
  int* d_slow = nullptr;           // faces the refresh computes (leaf * 6 + face): neighbour not same-level
  std::vector<int> slow_start;     // per-leaf offsets into d_slow, B + 1 entries
  int* d_slow_ax[3] = {nullptr, nullptr, nullptr};   // the same faces by axis, and their per-leaf offsets
  std::vector<int> slow_ax_start[3];
  int exec_mode = CELLO_EXEC_BATCHED;
  int sweep_variant[3] = {-1, -1, -1};   // per sweep axis; chosen by cello_autotune or set by the caller, -1: by rule
  unsigned* d_err = nullptr;       // error word: bit 0 set by the reduction, bit 1 by a sweep (ItemQueue)
  int* d_flag = nullptr;           // result word of the table and remap-map kernels
  RemapEntry* d_map = nullptr;     // remap entries of this mesh as the new one
  mutable std::mutex remap_lock;   // d_flag and d_map: one remap into this mesh at a time
  PoissonScratch* poisson = nullptr;   // multigrid levels, allocated by the first Poisson solve
  double* d_zero = nullptr;        // dt = 0, for timing sweeps without changing the state
  void* adj_scratch = nullptr;   // three states for the adjoint's forward recomputation
  size_t adj_bytes = 0;
  int* d_xlist = nullptr;        // index list of the last pack/unpack call (sharded step)
  size_t xlist_cap = 0;
  std::vector<GraphEntry> graphs;
  cudaStream_t capture_stream = nullptr;
  cudaStream_t side_stream = nullptr;          // the start-state reduction of cello_hydro_step_cfl
  cudaEvent_t fork_ev = nullptr, join_ev = nullptr;

  DevMesh dev() const {
    DevMesh m;
    m.n = desc.n;
    m.g = desc.ghosts;
    m.N = N;
    m.max_level = desc.max_level;
    for (int a = 0; a < 3; ++a) {
      m.root[a] = desc.root[a];
      m.bc[a] = desc.bc[a];
    }
    m.dx0 = (desc.hi[0] - desc.lo[0]) / (desc.root[0] * desc.n);
    m.gamma = desc.gamma;
    m.riemann = desc.riemann;
    m.steepen = desc.steepening;
    m.nf = desc.dual_energy ? 6 : 5;
    m.B = B;
    m.leaf = d_leaf;
    m.kind = d_kind;
    m.idx = d_idx;
    m.fine8 = d_fine8;
    m.face_slot = d_face_slot;
    m.err = d_err;
    return m;
  }

  void release() {
    poisson_free(poisson);
    poisson = nullptr;
    for (auto& g : graphs) cudaGraphExecDestroy(g.exec);
    graphs.clear();
    if (capture_stream) cudaStreamDestroy(capture_stream);
    capture_stream = nullptr;
    if (side_stream) cudaStreamDestroy(side_stream);
    side_stream = nullptr;
    if (fork_ev) cudaEventDestroy(fork_ev);
    if (join_ev) cudaEventDestroy(join_ev);
    fork_ev = join_ev = nullptr;
    if (adj_scratch) cudaFree(adj_scratch);
    adj_scratch = nullptr;
    if (d_xlist) cudaFree(d_xlist);
    d_xlist = nullptr;
    xlist_cap = 0;
    if (d_reg) cudaFree(d_reg);
    if (d_lists) cudaFree(d_lists);
    if (d_table) cudaFree(d_table);
    d_reg = nullptr;
    d_lists = d_table = nullptr;
  }
  ~cello_mesh() { release(); }
};

namespace {

cello_status check_desc(const cello_mesh_desc* d) {
  if (!d) return fail(CELLO_EINVAL, "desc is NULL");
  if (d->n != 8 && d->n != 16 && d->n != 32) return fail(CELLO_EINVAL, "n must be 8, 16 or 32");
  if (d->ghosts != kGhosts) return fail(CELLO_EINVAL, "ghosts must be 4");
  if (d->precision != 4 && d->precision != 8) return fail(CELLO_EINVAL, "precision must be 4 or 8");
  if (d->max_level < 0 || d->max_level > 10) return fail(CELLO_EINVAL, "max_level must be in [0, 10]");
  if (!(d->gamma > 1.0)) return fail(CELLO_EINVAL, "gamma must exceed 1");
  if (d->riemann != CELLO_RIEMANN_TWO_SHOCK && d->riemann != CELLO_RIEMANN_HLLC)
    return fail(CELLO_EINVAL, "riemann must be CELLO_RIEMANN_TWO_SHOCK or CELLO_RIEMANN_HLLC");
  if (d->steepening != 0 && d->steepening != 1) return fail(CELLO_EINVAL, "steepening must be 0 or 1");
  if (d->dual_energy != 0 && d->dual_energy != 1) return fail(CELLO_EINVAL, "dual_energy must be 0 or 1");
  double ext[3];
  for (int a = 0; a < 3; ++a) {
    if (d->root[a] < 1 || d->root[a] > 1024) return fail(CELLO_EINVAL, "root blocks per axis must be in [1, 1024]");
    if (d->bc[a] != CELLO_PERIODIC && d->bc[a] != CELLO_OUTFLOW) return fail(CELLO_EINVAL, "bc must be 0 or 1");
    ext[a] = (d->hi[a] - d->lo[a]) / d->root[a];
    if (!(ext[a] > 0)) return fail(CELLO_EINVAL, "hi must exceed lo");
  }
  for (int a = 1; a < 3; ++a)
    if (std::abs(ext[a] - ext[0]) > 1e-12 * ext[0]) return fail(CELLO_EINVAL, "cells must be cubes");
  return CELLO_OK;
}

// New leaf list, in Morton order, from the previous one and flags (see
// cello_octree_build).
std::vector<Node> build_leaves(const cello_mesh_desc& d, const cello_mesh* prev, const int8_t* flags) {
  std::vector<Node> out;
  if (!prev) {
    std::vector<std::pair<unsigned long long, Node>> roots;
    roots.reserve((size_t)d.root[0] * d.root[1] * d.root[2]);
    for (int k = 0; k < d.root[2]; ++k)
      for (int j = 0; j < d.root[1]; ++j)
        for (int i = 0; i < d.root[0]; ++i) roots.emplace_back(leaf_key(d, Node{0, i, j, k}), Node{0, i, j, k});
    std::sort(roots.begin(), roots.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
    out.reserve(roots.size());
    for (const auto& r : roots) out.push_back(r.second);
    return out;
  }
  const int B = prev->B;
  auto leaf = [&](int b) {
    const int4 l = prev->leaves[b];
    return Node{l.x, l.y, l.z, l.w};
  };
  // the previous mesh and the leaves to be refined
  auto mesh_tree = [&](const NodeSet* gone) {
    Tree t(d, (size_t)B / 4 + 64);
    for (int b = 0; b < B; ++b) {
      const Node n = leaf(b);
      if (flags && flags[b] > 0 && n.L < d.max_level) {
        t.refine(n);
      } else if (n.L > 0) {
        Node p{n.L - 1, n.i >> 1, n.j >> 1, n.k >> 1};
        if (gone && gone->contains(pack(p))) {   // the parent becomes a leaf
          if (p.L == 0) continue;
          p = Node{p.L - 1, p.i >> 1, p.j >> 1, p.k >> 1};
        }
        t.refine(p);
      }
    }
    return t;
  };
  Tree tree = mesh_tree(nullptr);
  // coarsening: octets of leaves (consecutive in Morton order) that are all -1
  // and whose parent would touch no leaf two levels finer
  std::vector<Node> coarsen;
  if (flags)
    for (int b = 0; b + 7 < B; ++b) {
      const Node t = leaf(b);
      if (flags[b] >= 0 || t.L == 0 || ((t.i | t.j | t.k) & 1)) continue;
      bool ok = true;
      for (int o = 1; o < 8 && ok; ++o) {
        const Node c = leaf(b + o);
        ok = flags[b + o] < 0 && c.L == t.L && (c.i >> 1) == (t.i >> 1) && (c.j >> 1) == (t.j >> 1) &&
             (c.k >> 1) == (t.k >> 1);
      }
      const Node p{t.L - 1, t.i >> 1, t.j >> 1, t.k >> 1};
      if (ok && !tree.touches_deeper(p)) coarsen.push_back(p);
    }
  if (!coarsen.empty()) {
    NodeSet gone(coarsen.size());
    for (const Node& p : coarsen) gone.insert(pack(p));
    tree = mesh_tree(&gone);
  }
  tree.balance();
  out.reserve((size_t)B);
  Node last{-1, 0, 0, 0};
  for (int b = 0; b < B; ++b) {   // the roots in the order of the leaves
    const Node t = leaf(b);
    const Node r{0, t.i >> t.L, t.j >> t.L, t.k >> t.L};
    if (last.L == 0 && r.i == last.i && r.j == last.j && r.k == last.k) continue;
    last = r;
    tree.emit(r, out);
  }
  return out;
}

#define CELLO_TRY(expr)               \
  do {                                \
    cello_status st_ = (expr);        \
    if (st_ != CELLO_OK) return st_;  \
  } while (0)

// Parts of one allocation, each on a 256-byte boundary.
struct Layout {
  size_t bytes = 0;
  template <typename V>
  size_t add(size_t count) {
    const size_t at = bytes;
    bytes += (count * sizeof(V) + 255) / 256 * 256;
    return at;
  }
};

template <typename V>
V* part(char* base, size_t at) { return reinterpret_cast<V*>(base + at); }

// The device tables of M->leaves.  The neighbour table stays on the device: what
// the host needs of it, whether the mesh is balanced and the kinds of each leaf's
// six faces, comes back in one copy, and the lists made from those go up in one
// (the whole table, 1 KB a leaf, walked on the host was a third of the build).
cello_status finish_build(cello_mesh* M) {
  const cello_mesh_desc& d = M->desc;
  const size_t B = (size_t)M->B;
  cudaStream_t s = cudaStreamPerThread;
  Layout t;
  const size_t o_leaf = t.add<int4>(B), o_keys = t.add<unsigned long long>(B), o_word = t.add<double>(32);
  const size_t head = t.bytes;   // uploaded: leaves, keys, the cleared words
  const size_t o_flag = t.add<int>(1), o_face = t.add<int8_t>(B * 6);
  const size_t tail = t.bytes - o_flag;   // downloaded
  const size_t o_kind = t.add<int8_t>(B * 27), o_idx = t.add<int>(B * 27), o_fine8 = t.add<int>(B * 27 * 8);
  const size_t o_part = t.add<double>(B * 6), o_map = t.add<RemapEntry>(B);
  CELLO_CUDA(cudaMalloc((void**)&M->d_table, t.bytes));
  M->d_leaf = part<int4>(M->d_table, o_leaf);
  M->d_keys = part<unsigned long long>(M->d_table, o_keys);
  M->d_err = part<unsigned>(M->d_table, o_word);
  M->d_zero = part<double>(M->d_table, o_word) + 16;
  M->d_flag = part<int>(M->d_table, o_flag);
  M->d_kind = part<int8_t>(M->d_table, o_kind);
  M->d_idx = part<int>(M->d_table, o_idx);
  M->d_fine8 = part<int>(M->d_table, o_fine8);
  M->d_partials = part<double>(M->d_table, o_part);
  M->d_map = part<RemapEntry>(M->d_table, o_map);
  std::vector<char> buf(std::max(head, tail), 0);
  std::memcpy(buf.data() + o_leaf, M->leaves.data(), B * sizeof(int4));
  std::memcpy(buf.data() + o_keys, M->keys.data(), B * sizeof(unsigned long long));
  CELLO_CUDA(cudaMemcpyAsync(M->d_table, buf.data(), head, cudaMemcpyHostToDevice, s));
  CELLO_CUDA(cudaMemsetAsync(M->d_flag, 0, sizeof(int), s));
  const DevMesh dm = M->dev();
  int8_t* d_face = part<int8_t>(M->d_table, o_face);
  launch_neighbour_table(dm, M->d_keys, M->d_kind, M->d_idx, M->d_fine8, d_face, M->d_flag, s);
  CELLO_CUDA(cudaGetLastError());
  CELLO_CUDA(cudaStreamSynchronize(s));   // buf is reused
  CELLO_CUDA(cudaMemcpyAsync(buf.data(), M->d_flag, tail, cudaMemcpyDeviceToHost, s));
  CELLO_CUDA(cudaStreamSynchronize(s));
  int flag;
  std::memcpy(&flag, buf.data(), sizeof(int));
  if (flag & 1) return fail(CELLO_EINTERNAL, "2:1 balance violated: a neighbour is two levels coarser");
  if (flag & 2) return fail(CELLO_EINTERNAL, "2:1 balance violated: a touching neighbour is two levels finer");
  const int8_t* face = reinterpret_cast<const int8_t*>(buf.data() + (o_face - o_flag));
  // flux-register slots: faces whose neighbour is finer (coarse side) or coarser
  // (fine side); the coarse sides, grouped by leaf; the faces whose phase region
  // the refresh computes instead of copying, those whose neighbour is not a
  // same-level leaf (coarser, finer, boundary), in leaf order and by axis
  M->face_slot.assign(B * 6, -1);
  std::vector<int> slow, by_axis[3];
  M->slow_start.assign(B + 1, 0);
  for (int a = 0; a < 3; ++a) M->slow_ax_start[a].assign(B + 1, 0);
  int ns = 0;
  for (size_t b = 0; b < B; ++b) {
    bool first = true;
    for (int f = 0; f < 6; ++f) {
      const int at = (int)b * 6 + f, k = face[at];
      if (k == kSame) continue;
      slow.push_back(at);
      by_axis[f >> 1].push_back(at);
      if (k == kBoundary) continue;
      M->face_slot[at] = ns++;
      if (k != kFine) continue;
      CoarseFace cf{};
      cf.leaf = (int)b;
      cf.axis = f >> 1;
      cf.side = (f & 1) ? 1 : -1;
      cf.cslot = M->face_slot[at];
      if (first) M->group_start.push_back((int)M->cfaces.size());
      first = false;
      M->cfaces.push_back(cf);
    }
    M->slow_start[b + 1] = (int)slow.size();
    for (int a = 0; a < 3; ++a) M->slow_ax_start[a][b + 1] = (int)by_axis[a].size();
  }
  M->nslots = ns;
  if (!M->cfaces.empty()) M->group_start.push_back((int)M->cfaces.size());
  Layout l;
  const size_t o_slot = l.add<int>(B * 6), o_cf = l.add<CoarseFace>(M->cfaces.size()),
               o_gs = l.add<int>(M->group_start.size()), o_slow = l.add<int>(slow.size());
  size_t o_ax[3];
  for (int a = 0; a < 3; ++a) o_ax[a] = l.add<int>(by_axis[a].size());
  CELLO_CUDA(cudaMalloc((void**)&M->d_lists, l.bytes));
  buf.resize(l.bytes);
  auto put = [&](size_t at, const auto& v) {
    if (!v.empty()) std::memcpy(buf.data() + at, v.data(), v.size() * sizeof(v[0]));
  };
  put(o_slot, M->face_slot);
  put(o_cf, M->cfaces);
  put(o_gs, M->group_start);
  put(o_slow, slow);
  for (int a = 0; a < 3; ++a) put(o_ax[a], by_axis[a]);
  CELLO_CUDA(cudaMemcpyAsync(M->d_lists, buf.data(), l.bytes, cudaMemcpyHostToDevice, s));
  M->d_face_slot = part<int>(M->d_lists, o_slot);
  if (!M->cfaces.empty()) {
    M->d_cfaces = part<CoarseFace>(M->d_lists, o_cf);
    M->d_group_start = part<int>(M->d_lists, o_gs);
    launch_fine_slots(M->dev(), M->d_cfaces, (int)M->cfaces.size(), s);
    CELLO_CUDA(cudaGetLastError());
  }
  if (!slow.empty()) M->d_slow = part<int>(M->d_lists, o_slow);
  for (int a = 0; a < 3; ++a)
    if (!by_axis[a].empty()) M->d_slow_ax[a] = part<int>(M->d_lists, o_ax[a]);
  if (ns > 0) CELLO_CUDA(cudaMalloc((void**)&M->d_reg, (size_t)ns * nfields(d) * d.n * d.n * sizeof(double)));
  CELLO_CUDA(cudaStreamSynchronize(s));   // the tables are read on any stream from here on
  return CELLO_OK;
}

void launch_refresh(const cello_mesh* M, const DevMesh& dm, void* U, int leaf0, int nleaf, cudaStream_t s,
                    int phases = kRefreshAll) {
  const int s0 = M->slow_start[leaf0], s1 = M->slow_start[leaf0 + nleaf];
  const int* slow = M->d_slow ? M->d_slow + s0 : nullptr;
  if (M->desc.precision == 4) launch_refresh_f32(dm, static_cast<float*>(U), leaf0, nleaf, slow, s1 - s0, phases, s);
  else launch_refresh_f64(dm, static_cast<double*>(U), leaf0, nleaf, slow, s1 - s0, phases, s);
}

// Transverse pencil ranges of a sweep along `axis`: a transverse axis already
// swept this step needs interior rows only, one not yet swept all N rows.
void sweep_ranges(const cello_mesh* M, int axis, const bool swept[3], int& a0, int& a1, int& b0, int& b1) {
  const int n = M->desc.n, g = M->desc.ghosts, N = M->N;
  const int ta = axis == 2 ? 1 : 2;   // transverse A: z, or y for the z sweep
  const int tb = axis == 0 ? 1 : 0;   // transverse B: y for the x sweep, else x
  a0 = swept[ta] ? g : 0;
  a1 = swept[ta] ? g + n : N;
  b0 = swept[tb] ? g : 0;
  b1 = swept[tb] ? g + n : N;
}

// The pencils of the step's oi-th sweep over leaves [leaf0, leaf0 + nleaf).
// whole: the sweep of a whole step, in which each leaf sweeps its interior rows
// and the ghost rows behind its faces that are not same-level, and stores the
// rows its same-level neighbours read behind the next sweep's faces into their
// ghost rows (push_offset in kernels.cuh); the ghost rows behind the last
// sweep's faces are needed by the second sweep only.  Otherwise (a leaf range, or
// a state whose ghost rows are read afterwards): every row a later sweep of the
// same leaf reads, nothing stored elsewhere.
void set_regions(const cello_mesh* M, SweepParams& p, const int order[3], int oi, int leaf0, int nleaf, bool whole) {
  const int n = M->desc.n, g = M->desc.ghosts, N = M->N;
  p.axis = order[oi];
  p.leaf0 = leaf0;
  p.nleaf = nleaf;
  p.push = -1;
  SweepRegion& r0 = p.reg3[0];
  if (!whole) {
    bool swept[3] = {false, false, false};
    for (int k = 0; k < oi; ++k) swept[order[k]] = true;
    int a1, b1;
    sweep_ranges(M, p.axis, swept, r0.a0, a1, r0.b0, b1);
    r0.cb = b1 - r0.b0;
    r0.count = (a1 - r0.a0) * r0.cb;
    return;
  }
  r0.a0 = r0.b0 = g;
  r0.cb = n;
  r0.count = n * n;
  if (oi < 2) p.push = order[oi + 1];
  const int ta = p.axis == 2 ? 1 : 2;
  for (int k = 1; oi + k < 3; ++k) {   // faces of the next sweep's axis, then (first sweep) of the last one's
    const int f = order[oi + k];
    const bool full = k == 2;          // behind those, the second sweep reads all rows of its own axis
    SweepRegion& r = p.reg3[k];
    const int along = full ? N : n, from = full ? 0 : g;
    if (f == ta) {
      r.a0 = 0; r.da = g + n;
      r.b0 = from; r.cb = along;
    } else {
      r.a0 = from;
      r.b0 = 0; r.db = g + n; r.cb = g;
    }
    r.count = g * along;
    const int s0 = M->slow_ax_start[f][leaf0];
    r.faces = M->d_slow_ax[f] ? M->d_slow_ax[f] + s0 : nullptr;
    r.nfaces = M->slow_ax_start[f][leaf0 + nleaf] - s0;
  }
}

void launch_sweep(const cello_mesh* M, const DevMesh& dm, const SweepParams& p, cudaStream_t s) {
  if (M->desc.precision == 4) launch_sweep_f32(dm, p, s);
  else launch_sweep_f64(dm, p, s);
}

// The three split sweeps of leaves [leaf0, leaf0 + nleaf) (x, y, z on even
// cycles, z, y, x on odd ones), face fluxes of coarse-fine faces into the
// registers; whole: see set_regions; plain: one launch per leaf and sweep; ev
// (nullable): events after each sweep at ev[2 ..].
void enqueue_sweeps(const cello_mesh* M, const DevMesh& dm, void* U, const double* dt, int cycle, int leaf0,
                    int nleaf, bool whole, bool plain, cudaStream_t s, cudaEvent_t* ev) {
  const int order[3] = {cycle % 2 == 0 ? 0 : 2, 1, cycle % 2 == 0 ? 2 : 0};
  for (int oi = 0; oi < 3; ++oi) {
    SweepParams p{};
    p.U = U;
    p.dt = dt;
    p.reg = M->d_reg;
    p.variant = M->sweep_variant[order[oi]];
    if (plain) {
      for (int b = leaf0; b < leaf0 + nleaf; ++b) {
        set_regions(M, p, order, oi, b, 1, whole);
        launch_sweep(M, dm, p, s);
      }
    } else if (nleaf > 0) {
      set_regions(M, p, order, oi, leaf0, nleaf, whole);
      launch_sweep(M, dm, p, s);
    }
    if (ev) cudaEventRecord(ev[2 + oi], s);
  }
}

// The ghost cells that the sweeps of a whole step read before writing them.
int step_refresh(int cycle) { return cycle % 2 == 0 ? kRefreshXFirst : kRefreshZFirst; }

// The launch sequence of one step on stream s.
void enqueue_step(const cello_mesh* M, void* U, const double* dt, int cycle, double cfl, double* dt_next,
                  double* totals, cudaStream_t s, cudaEvent_t* ev = nullptr) {
  const cello_mesh_desc& d = M->desc;
  const DevMesh dm = M->dev();
  const int B = M->B;
  const bool plain = M->exec_mode == CELLO_EXEC_PLAIN && !ev;
  if (ev) cudaEventRecord(ev[0], s);
  if (plain) {   // one launch per leaf and phase; each phase over every leaf before the next
    const int even[2] = {kRefreshSlow, kRefreshX}, odd[2] = {kRefreshZRows, kRefreshSlowZFirst};
    for (int ph : cycle % 2 == 0 ? even : odd)
      for (int b = 0; b < B; ++b) launch_refresh(M, dm, U, b, 1, s, ph);
  } else {
    launch_refresh(M, dm, U, 0, B, s, step_refresh(cycle));
  }
  if (ev) cudaEventRecord(ev[1], s);
  enqueue_sweeps(M, dm, U, dt, cycle, 0, B, true, plain, s, ev);
  if (!M->cfaces.empty())
    launch_fluxcorr(dm, U, d.precision, M->d_cfaces, M->d_group_start, (int)M->group_start.size() - 1, M->d_reg,
                    dt, s);
  if (ev) cudaEventRecord(ev[5], s);
  if (dt_next || totals || ev) launch_reduce(dm, U, d.precision, cfl, M->d_partials, dt_next, totals, s);
  if (ev) cudaEventRecord(ev[6], s);
}

// One step whose dt is the CFL step of its start state: the reduction of the
// start state (interiors only) on the side stream while the ghost refresh
// (ghosts only) runs on s; the sweeps wait for both.
constexpr int kSideReduceCtasPerSm = 2;

void enqueue_step_cfl(const cello_mesh* M, void* U, int cycle, double cfl, double* dt_used, double* totals,
                      cudaStream_t s) {
  const cello_mesh_desc& d = M->desc;
  const DevMesh dm = M->dev();
  cudaEventRecord(M->fork_ev, s);
  cudaStreamWaitEvent(M->side_stream, M->fork_ev, 0);
  // a few resident CTAs per SM walk the leaves, so that the reduction shares
  // the SMs with the refresh's kernels (latency-bound, DRAM not saturated)
  // instead of queueing behind them
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  launch_reduce(dm, U, d.precision, cfl, M->d_partials, dt_used, totals, M->side_stream, kSideReduceCtasPerSm * sms);
  cudaEventRecord(M->join_ev, M->side_stream);
  launch_refresh(M, dm, U, 0, M->B, s, step_refresh(cycle));
  cudaStreamWaitEvent(s, M->join_ev, 0);
  enqueue_sweeps(M, dm, U, dt_used, cycle, 0, M->B, true, false, s, nullptr);
  if (!M->cfaces.empty())
    launch_fluxcorr(dm, U, d.precision, M->d_cfaces, M->d_group_start, (int)M->group_start.size() - 1, M->d_reg,
                    dt_used, s);
}

cello_status adjoint_step(cello_mesh* M, const void* Un, void* lam, const double* dt, int cycle, cudaStream_t s) {
  const cello_mesh_desc& d = M->desc;
  bool uniform_periodic = true;   // then the ghost copy's transpose is a deterministic gather
  for (int a = 0; a < 3; ++a) uniform_periodic = uniform_periodic && d.bc[a] == CELLO_PERIODIC;
  for (int b = 1; b < M->B && uniform_periodic; ++b) uniform_periodic = M->leaves[b].x == M->leaves[0].x;
  const size_t state = (size_t)M->B * nfields(d) * M->N * M->N * M->N * d.precision;
  const size_t regs = (size_t)M->nslots * nfields(d) * d.n * d.n * sizeof(double);
  if (M->adj_bytes < 3 * state + regs) {
    if (M->adj_scratch) cudaFree(M->adj_scratch);
    M->adj_scratch = nullptr;
    M->adj_bytes = 0;
    CELLO_CUDA(cudaMalloc(&M->adj_scratch, 3 * state + regs));
    M->adj_bytes = 3 * state + regs;
  }
  char* S0 = static_cast<char*>(M->adj_scratch);
  char* S1 = S0 + state;
  char* S2 = S1 + state;
  const DevMesh dm = M->dev();
  const int B = M->B;
  // forward recomputation: refreshed start state, then the states entering
  // the second and third sweeps
  CELLO_CUDA(cudaMemcpyAsync(S0, Un, state, cudaMemcpyDeviceToDevice, s));
  launch_refresh(M, dm, S0, 0, B, s);
  const int order[3] = {cycle % 2 == 0 ? 0 : 2, 1, cycle % 2 == 0 ? 2 : 0};
  char* entry[3] = {S0, S1, S2};
  bool swept[3] = {false, false, false};
  int rng[3][4];
  for (int oi = 0; oi < 3; ++oi) {
    const int axis = order[oi];
    sweep_ranges(M, axis, swept, rng[oi][0], rng[oi][1], rng[oi][2], rng[oi][3]);
    if (oi < 2) {
      CELLO_CUDA(cudaMemcpyAsync(entry[oi + 1], entry[oi], state, cudaMemcpyDeviceToDevice, s));
      SweepParams p{};
      p.U = entry[oi + 1];
      p.dt = dt;
      p.reg = nullptr;
      p.variant = M->sweep_variant[axis];
      set_regions(M, p, order, oi, 0, B, false);   // the adjoint sweeps read every ghost row
      launch_sweep(M, dm, p, s);
    }
    swept[axis] = true;
  }
  // reverse: the adjoint of U_{n+1} lives on interior cells only; the
  // coarse-fine flux correction's adjoint gives the face-flux adjoints
  launch_zero_ghosts(dm, lam, d.precision, s);
  double* regb = nullptr;
  if (!M->cfaces.empty()) {
    regb = reinterpret_cast<double*>(S2 + state);
    launch_fluxcorr_adjoint(dm, lam, d.precision, M->d_cfaces, (int)M->cfaces.size(), regb, dt, s);
  }
  for (int oi = 2; oi >= 0; --oi) {
    AdjSweepParams p{};
    p.U = entry[oi];
    p.lam = lam;
    p.regb = regb;
    p.axis = order[oi];
    p.a0 = rng[oi][0]; p.a1 = rng[oi][1]; p.b0 = rng[oi][2]; p.b1 = rng[oi][3];
    const int pencils = (p.a1 - p.a0) * (p.b1 - p.b0);
    p.tiles_per_leaf = (pencils + adj_pencils(d.n, d.precision) - 1) / adj_pencils(d.n, d.precision);
    p.dt = dt;
    p.leaf0 = 0;
    p.nleaf = B;
    p.n_items = B * p.tiles_per_leaf;
    if (d.precision == 4) launch_adjoint_sweep_f32(dm, p, s);
    else launch_adjoint_sweep_f64(dm, p, s);
  }
  if (uniform_periodic) launch_adjoint_refresh(dm, lam, d.precision, s);
  else launch_adjoint_refresh_scatter(dm, S0, lam, d.precision, s);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

}  // namespace

namespace cello {
DevMesh mesh_dev(const cello_mesh* mesh) { return mesh->dev(); }
int mesh_precision(const cello_mesh* mesh) { return mesh->desc.precision; }
cello_status set_error(cello_status status, const char* message) { return fail(status, message); }
}  // namespace cello

// ====================================================================== ABI
extern "C" {

const char* cello_last_error(void) { return g_last_error.c_str(); }

cello_status cello_octree_build(const cello_mesh_desc* desc, const cello_mesh* prev, const int8_t* flags_host,
                                cello_mesh** out) {
  if (!out) return fail(CELLO_EINVAL, "out is NULL");
  *out = nullptr;
  CELLO_TRY(check_desc(desc));
  if (prev && std::memcmp(&prev->desc, desc, sizeof(cello_mesh_desc)) != 0)
    return fail(CELLO_EINVAL, "prev was built from a different description");
  prepare_kernels();
  auto* M = new (std::nothrow) cello_mesh();
  if (!M) return fail(CELLO_ENOMEM, "host allocation failed");
  M->desc = *desc;
  M->N = desc->n + 2 * desc->ghosts;
  const std::vector<Node> ls = build_leaves(*desc, prev, flags_host);
  M->B = (int)ls.size();
  M->keys.reserve(ls.size());
  M->leaves.reserve(ls.size());
  for (const Node& t : ls) {
    M->keys.push_back(leaf_key(*desc, t));
    M->leaves.push_back(make_int4(t.L, t.i, t.j, t.k));
  }
  cello_status st = finish_build(M);
  if (st != CELLO_OK) {
    delete M;
    return st;
  }
  *out = M;
  return CELLO_OK;
}

cello_status cello_mesh_from_leaves(const cello_mesh_desc* desc, const int32_t* leaves_host, int64_t count,
                                   cello_mesh** out) {
  if (!out || !leaves_host || count <= 0) return fail(CELLO_EINVAL, "NULL argument or empty leaf list");
  *out = nullptr;
  CELLO_TRY(check_desc(desc));
  std::vector<Node> ls((size_t)count);
  std::unordered_set<unsigned long long> seen;
  double volume = 0.0;
  for (int64_t b = 0; b < count; ++b) {
    const Node t{leaves_host[4 * b], leaves_host[4 * b + 1], leaves_host[4 * b + 2], leaves_host[4 * b + 3]};
    if (t.L < 0 || t.L > desc->max_level) return fail(CELLO_EINVAL, "leaf level out of range");
    const int p[3] = {t.i, t.j, t.k};
    for (int a = 0; a < 3; ++a)
      if (p[a] < 0 || p[a] >= (desc->root[a] << t.L)) return fail(CELLO_EINVAL, "leaf index out of range");
    if (!seen.insert(pack(t)).second) return fail(CELLO_EINVAL, "duplicate leaf");
    ls[(size_t)b] = t;
    volume += std::ldexp(1.0, -3 * t.L);
  }
  for (const Node& t : ls) {   // no leaf may contain another
    Node q = t;
    while (q.L > 0) {
      q = Node{q.L - 1, q.i >> 1, q.j >> 1, q.k >> 1};
      if (seen.count(pack(q))) return fail(CELLO_EINVAL, "leaves overlap");
    }
  }
  if (volume != (double)desc->root[0] * desc->root[1] * desc->root[2])
    return fail(CELLO_EINVAL, "leaves do not tile the domain");
  prepare_kernels();
  auto* M = new (std::nothrow) cello_mesh();
  if (!M) return fail(CELLO_ENOMEM, "host allocation failed");
  M->desc = *desc;
  M->N = desc->n + 2 * desc->ghosts;
  std::vector<std::pair<unsigned long long, Node>> keyed;
  for (const Node& t : ls) keyed.emplace_back(leaf_key(*desc, t), t);
  std::sort(keyed.begin(), keyed.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
  M->B = (int)keyed.size();
  for (const auto& kv : keyed) {
    M->keys.push_back(kv.first);
    M->leaves.push_back(make_int4(kv.second.L, kv.second.i, kv.second.j, kv.second.k));
  }
  cello_status st = finish_build(M);
  if (st != CELLO_OK) {
    delete M;
    return st;
  }
  *out = M;
  return CELLO_OK;
}

cello_status cello_check(cello_mesh* M, uint32_t* word) {
  if (!M) return fail(CELLO_EINVAL, "mesh is NULL");
  unsigned w = 0;
  CELLO_CUDA(cudaMemcpy(&w, M->d_err, sizeof(unsigned), cudaMemcpyDeviceToHost));
  CELLO_CUDA(cudaMemset(M->d_err, 0, sizeof(unsigned)));
  if (word) *word = w;
  if (w & 2u) return fail(CELLO_EINTERNAL, "a sweep gave up waiting for its next work item: the state is incomplete");
  if (w & 1u) return fail(CELLO_ENONFINITE, "a reduction saw a non-finite value or a non-positive density or pressure");
  return CELLO_OK;
}

void cello_mesh_free(cello_mesh* mesh) { delete mesh; }

cello_status cello_mesh_info(const cello_mesh* M, int64_t* n_leaves, int64_t* leaf_elems, int64_t* n_cf) {
  if (!M) return fail(CELLO_EINVAL, "mesh is NULL");
  if (n_leaves) *n_leaves = M->B;
  if (leaf_elems) *leaf_elems = (int64_t)nfields(M->desc) * M->N * M->N * M->N;
  if (n_cf) *n_cf = (int64_t)M->cfaces.size();
  return CELLO_OK;
}

cello_status cello_mesh_leaves(const cello_mesh* M, int32_t* out) {
  if (!M || !out) return fail(CELLO_EINVAL, "NULL argument");
  for (int b = 0; b < M->B; ++b) {
    out[4 * b] = M->leaves[b].x;
    out[4 * b + 1] = M->leaves[b].y;
    out[4 * b + 2] = M->leaves[b].z;
    out[4 * b + 3] = M->leaves[b].w;
  }
  return CELLO_OK;
}

cello_status cello_neighbour_table(const cello_mesh* M, int8_t* kind, int32_t* idx, int32_t* fine8) {
  if (!M) return fail(CELLO_EINVAL, "mesh is NULL");
  // the table stays on the device; a stream of its own in the relaxed capture
  // mode, so that a query during a graph capture neither joins nor breaks it
  const size_t entries = (size_t)M->B * 27;
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  CELLO_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
  cudaStream_t s = nullptr;
  cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  auto get = [&](void* to, const void* from, size_t bytes) {
    if (to && e == cudaSuccess) e = cudaMemcpyAsync(to, from, bytes, cudaMemcpyDeviceToHost, s);
  };
  get(kind, M->d_kind, entries);
  get(idx, M->d_idx, entries * sizeof(int));
  get(fine8, M->d_fine8, entries * 8 * sizeof(int));
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (s) cudaStreamDestroy(s);
  cudaThreadExchangeStreamCaptureMode(&mode);
  CELLO_CUDA(e);
  return CELLO_OK;
}

cello_status cello_refine_flags(cello_mesh* M, const void* U, int field, double tau, double tau_c, int8_t* flags,
                                void* stream) {
  if (!M || !U || !flags) return fail(CELLO_EINVAL, "NULL argument");
  if (field != 0 && field != 4) return fail(CELLO_EINVAL, "field must be 0 (density) or 4 (pressure)");
  CELLO_REQUIRE_ALIGNED(U);
  launch_flags(M->dev(), U, M->desc.precision, field, tau, tau_c, flags, (cudaStream_t)stream);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

cello_status cello_ghost_refresh(cello_mesh* M, void* U, void* stream) {
  if (!M || !U) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U);
  launch_refresh(M, M->dev(), U, 0, M->B, (cudaStream_t)stream);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

cello_status cello_reduce(cello_mesh* M, const void* U, double cfl, double* dt_next, double* totals, void* stream) {
  if (!M || !U) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U);
  launch_reduce(M->dev(), U, M->desc.precision, cfl, M->d_partials, dt_next, totals, (cudaStream_t)stream);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

// ------------------------------------------------------------- sharded step
namespace {

// The host index list copied to the mesh's device list (grown when needed),
// on the caller's stream.
cello_status upload_list(cello_mesh* M, const std::vector<int>& h, cudaStream_t s) {
  if (h.empty()) return CELLO_OK;
  if (M->xlist_cap < h.size()) {
    if (M->d_xlist) cudaFree(M->d_xlist);
    M->d_xlist = nullptr;
    M->xlist_cap = 0;
    CELLO_CUDA(cudaMalloc((void**)&M->d_xlist, h.size() * sizeof(int)));
    M->xlist_cap = h.size();
  }
  CELLO_CUDA(cudaMemcpyAsync(M->d_xlist, h.data(), h.size() * sizeof(int), cudaMemcpyHostToDevice, s));
  return CELLO_OK;
}

cello_status halo_copy(cello_mesh* M, void* U, const int32_t* leaf_ids, int64_t count, void* buf, int pack,
                       void* stream) {
  if (!M || count < 0 || (count > 0 && (!U || !leaf_ids || !buf))) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U);
  if (reinterpret_cast<uintptr_t>(buf) & 31u) return fail(CELLO_EINVAL, "buffer is not 32-byte aligned");
  std::vector<int> h((size_t)count);
  for (int64_t k = 0; k < count; ++k) {
    if (leaf_ids[k] < 0 || leaf_ids[k] >= M->B) return fail(CELLO_EINVAL, "leaf id out of range");
    h[k] = leaf_ids[k];
  }
  cudaStream_t s = (cudaStream_t)stream;
  CELLO_TRY(upload_list(M, h, s));
  launch_halo_copy(M->dev(), U, M->desc.precision, M->d_xlist, (long)count, buf, pack, s);
  CELLO_CUDA(cudaGetLastError());
  // the list is read by the kernel: a later call must not overwrite it before
  // the kernel has run, which the stream order guarantees for calls on one
  // stream
  return CELLO_OK;
}

cello_status flux_copy(cello_mesh* M, const int32_t* faces, int64_t count, double* buf, int pack, void* stream) {
  if (!M || count < 0 || (count > 0 && (!faces || !buf))) return fail(CELLO_EINVAL, "NULL argument");
  std::vector<int> h((size_t)count);
  for (int64_t k = 0; k < count; ++k) {
    if (faces[k] < 0 || faces[k] >= M->B * 6) return fail(CELLO_EINVAL, "face entry out of range");
    const int slot = M->face_slot[(size_t)faces[k]];
    if (slot < 0) return fail(CELLO_EINVAL, "a listed face is not on a coarse-fine face (no flux register)");
    h[k] = slot;
  }
  cudaStream_t s = (cudaStream_t)stream;
  CELLO_TRY(upload_list(M, h, s));
  launch_flux_copy(M->d_reg, M->d_xlist, (long)count, (long)nfields(M->desc) * M->desc.n * M->desc.n, buf, pack, s);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

cello_status check_range(const cello_mesh* M, int64_t leaf0, int64_t nleaf) {
  if (leaf0 < 0 || nleaf < 0 || leaf0 + nleaf > M->B) return fail(CELLO_EINVAL, "leaf range outside the mesh");
  return CELLO_OK;
}

}  // namespace

cello_status cello_halo_pack(cello_mesh* M, const void* U, const int32_t* leaf_ids, int64_t count, void* buf,
                             void* stream) {
  return halo_copy(M, const_cast<void*>(U), leaf_ids, count, buf, 1, stream);
}

cello_status cello_halo_unpack(cello_mesh* M, void* U, const int32_t* leaf_ids, int64_t count, const void* buf,
                               void* stream) {
  return halo_copy(M, U, leaf_ids, count, const_cast<void*>(buf), 0, stream);
}

cello_status cello_flux_pack(cello_mesh* M, const int32_t* faces, int64_t count, double* buf, void* stream) {
  return flux_copy(M, faces, count, buf, 1, stream);
}

cello_status cello_flux_unpack(cello_mesh* M, const int32_t* faces, int64_t count, const double* buf, void* stream) {
  return flux_copy(M, faces, count, const_cast<double*>(buf), 0, stream);
}

cello_status cello_hydro_step_part(cello_mesh* M, void* U, const double* dt, int cycle, int64_t leaf0, int64_t nleaf,
                                   int part, void* stream) {
  if (!M || !U || !dt) return fail(CELLO_EINVAL, "NULL argument");
  if (cycle < 0) return fail(CELLO_EINVAL, "cycle must be >= 0");
  if (part != 0 && part != 1) return fail(CELLO_EINVAL, "part must be 0 (refresh and sweeps) or 1 (flux correction)");
  CELLO_REQUIRE_ALIGNED(U);
  CELLO_TRY(check_range(M, leaf0, nleaf));
  cudaStream_t s = (cudaStream_t)stream;
  const DevMesh dm = M->dev();
  if (part == 0) {
    launch_refresh(M, dm, U, 0, M->B, s);
    enqueue_sweeps(M, dm, U, dt, cycle, (int)leaf0, (int)nleaf, false, false, s, nullptr);
  } else if (!M->cfaces.empty()) {
    // the groups (one per coarse leaf, in leaf order) whose leaf is in the range
    const int ng = (int)M->group_start.size() - 1;
    int g0 = 0, g1 = 0;
    while (g0 < ng && M->cfaces[M->group_start[g0]].leaf < leaf0) ++g0;
    g1 = g0;
    while (g1 < ng && M->cfaces[M->group_start[g1]].leaf < leaf0 + nleaf) ++g1;
    if (g1 > g0)
      launch_fluxcorr(dm, U, M->desc.precision, M->d_cfaces, M->d_group_start + g0, g1 - g0, M->d_reg, dt, s);
  }
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

cello_status cello_reduce_part(cello_mesh* M, const void* U, int64_t leaf0, int64_t nleaf, double* out_dev,
                               void* stream) {
  if (!M || !U || !out_dev) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U);
  CELLO_TRY(check_range(M, leaf0, nleaf));
  if (nleaf == 0) return fail(CELLO_EINVAL, "empty leaf range");
  launch_reduce_range(M->dev(), U, M->desc.precision, 1.0, M->d_partials, (int)leaf0, (int)nleaf, out_dev,
                      out_dev + 1, (cudaStream_t)stream);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

cello_status cello_set_exec(cello_mesh* M, int mode) {
  if (!M) return fail(CELLO_EINVAL, "mesh is NULL");
  if (mode < CELLO_EXEC_PLAIN || mode > CELLO_EXEC_GRAPH) return fail(CELLO_EINVAL, "unknown exec mode");
  M->exec_mode = mode;
  return CELLO_OK;
}

cello_status cello_hydro_step(cello_mesh* M, void* U, const double* dt, int cycle, double cfl, double* dt_next,
                              double* totals, void* stream) {
  if (!M || !U || !dt) return fail(CELLO_EINVAL, "NULL argument");
  if (cycle < 0) return fail(CELLO_EINVAL, "cycle must be >= 0");
  CELLO_REQUIRE_ALIGNED(U);
  cudaStream_t s = (cudaStream_t)stream;
  if (M->exec_mode != CELLO_EXEC_GRAPH) {
    enqueue_step(M, U, dt, cycle, cfl, dt_next, totals, s);
    CELLO_CUDA(cudaGetLastError());
    return CELLO_OK;
  }
  const int parity = cycle % 2;
  for (const GraphEntry& g : M->graphs)
    if (!g.cfl_step && g.U == U && g.dt == dt && g.parity == parity && g.cfl == cfl && g.dt_next == dt_next &&
        g.totals == totals) {
      CELLO_CUDA(cudaGraphLaunch(g.exec, s));
      return CELLO_OK;
    }
  if (!M->capture_stream) CELLO_CUDA(cudaStreamCreateWithFlags(&M->capture_stream, cudaStreamNonBlocking));
  cudaGraph_t graph;
  CELLO_CUDA(cudaStreamBeginCapture(M->capture_stream, cudaStreamCaptureModeThreadLocal));
  enqueue_step(M, U, dt, parity, cfl, dt_next, totals, M->capture_stream);
  CELLO_CUDA(cudaStreamEndCapture(M->capture_stream, &graph));
  cudaGraphExec_t exec;
  cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  CELLO_CUDA(e);
  if (M->graphs.size() >= 8) {
    cudaGraphExecDestroy(M->graphs.front().exec);
    M->graphs.erase(M->graphs.begin());
  }
  M->graphs.push_back(GraphEntry{U, dt, parity, cfl, dt_next, totals, exec});
  CELLO_CUDA(cudaGraphLaunch(exec, s));
  return CELLO_OK;
}

cello_status cello_hydro_step_cfl(cello_mesh* M, void* U, int cycle, double cfl, double* dt_used, double* totals,
                                  void* stream) {
  if (!M || !U || !dt_used) return fail(CELLO_EINVAL, "NULL argument");
  if (cycle < 0) return fail(CELLO_EINVAL, "cycle must be >= 0");
  CELLO_REQUIRE_ALIGNED(U);
  cudaStream_t s = (cudaStream_t)stream;
  if (!M->side_stream) CELLO_CUDA(cudaStreamCreateWithFlags(&M->side_stream, cudaStreamNonBlocking));
  if (!M->fork_ev) CELLO_CUDA(cudaEventCreateWithFlags(&M->fork_ev, cudaEventDisableTiming));
  if (!M->join_ev) CELLO_CUDA(cudaEventCreateWithFlags(&M->join_ev, cudaEventDisableTiming));
  if (M->exec_mode != CELLO_EXEC_GRAPH) {
    enqueue_step_cfl(M, U, cycle, cfl, dt_used, totals, s);
    CELLO_CUDA(cudaGetLastError());
    return CELLO_OK;
  }
  const int parity = cycle % 2;
  for (const GraphEntry& g : M->graphs)
    if (g.cfl_step && g.U == U && g.dt == dt_used && g.parity == parity && g.cfl == cfl && g.totals == totals) {
      CELLO_CUDA(cudaGraphLaunch(g.exec, s));
      return CELLO_OK;
    }
  if (!M->capture_stream) CELLO_CUDA(cudaStreamCreateWithFlags(&M->capture_stream, cudaStreamNonBlocking));
  cudaGraph_t graph;
  CELLO_CUDA(cudaStreamBeginCapture(M->capture_stream, cudaStreamCaptureModeThreadLocal));
  enqueue_step_cfl(M, U, parity, cfl, dt_used, totals, M->capture_stream);
  CELLO_CUDA(cudaStreamEndCapture(M->capture_stream, &graph));
  cudaGraphExec_t exec;
  cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  CELLO_CUDA(e);
  if (M->graphs.size() >= 8) {
    cudaGraphExecDestroy(M->graphs.front().exec);
    M->graphs.erase(M->graphs.begin());
  }
  GraphEntry ge{U, dt_used, parity, cfl, nullptr, totals, exec};
  ge.cfl_step = true;
  M->graphs.push_back(ge);
  CELLO_CUDA(cudaGraphLaunch(exec, s));
  return CELLO_OK;
}

cello_status cello_remap(const cello_mesh* old, const void* U_old, const cello_mesh* neu, void* U_new,
                         void* stream) {
  if (!old || !neu || !U_old || !U_new) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U_old);
  CELLO_REQUIRE_ALIGNED(U_new);
  if (std::memcmp(&old->desc, &neu->desc, sizeof(cello_mesh_desc)) != 0)
    return fail(CELLO_EINVAL, "meshes built from different descriptions");
  // the entries by binary search of the sorted keys on the device; if a new leaf
  // has no source there, nothing is written and the call says so.  The call ends
  // with its work, so calls from several threads take turns with the entries.
  const std::lock_guard<std::mutex> turn(neu->remap_lock);
  cudaStream_t s = (cudaStream_t)stream;
  CELLO_CUDA(cudaMemsetAsync(neu->d_flag, 0, sizeof(int), s));
  launch_remap(neu->dev(), neu->d_keys, old->dev(), old->d_keys, U_old, U_new, neu->d_map, neu->d_flag,
               neu->desc.precision, s);
  CELLO_CUDA(cudaGetLastError());
  int flag = 0;
  CELLO_CUDA(cudaMemcpyAsync(&flag, neu->d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
  CELLO_CUDA(cudaStreamSynchronize(s));
  if (flag) return fail(CELLO_EINVAL, "meshes are not one adaptation apart");
  return CELLO_OK;
}

cello_status cello_hydro_adjoint_step(cello_mesh* M, const void* Un, void* lam, const double* dt, int cycle,
                                      void* stream) {
  if (!M || !Un || !lam || !dt) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(Un);
  CELLO_REQUIRE_ALIGNED(lam);
  if (cycle < 0) return fail(CELLO_EINVAL, "cycle must be >= 0");
  if (M->desc.riemann != CELLO_RIEMANN_TWO_SHOCK || M->desc.steepening || M->desc.dual_energy)
    return fail(CELLO_EINVAL,
                "the adjoint step is written for the two-shock solver without contact steepening or dual energy");
  return adjoint_step(M, Un, lam, dt, cycle, (cudaStream_t)stream);
}

cello_status cello_set_sweep_variants(cello_mesh* M, const int* variants) {
  if (!M || !variants) return fail(CELLO_EINVAL, "NULL argument");
  const int nv = M->desc.precision == 4 ? sweep_variant_count_f32() : sweep_variant_count_f64();
  for (int a = 0; a < 3; ++a)
    if (variants[a] < -1 || variants[a] >= nv) return fail(CELLO_EINVAL, "sweep variant out of range");
  for (int a = 0; a < 3; ++a) M->sweep_variant[a] = variants[a];
  for (auto& g : M->graphs) cudaGraphExecDestroy(g.exec);
  M->graphs.clear();
  return CELLO_OK;
}

cello_status cello_set_sweep_variant(cello_mesh* M, int variant) {
  const int v[3] = {variant, variant, variant};
  return cello_set_sweep_variants(M, v);
}

cello_status cello_autotune(cello_mesh* M, void* U, int* variants_out, float* ms_out, int ms_len, void* stream) {
  if (!M || !U) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U);
  cudaStream_t s = (cudaStream_t)stream;
  const cello_mesh_desc& d = M->desc;
  const int nv = d.precision == 4 ? sweep_variant_count_f32() : sweep_variant_count_f64();
  const int nleaf = std::min(M->B, 4096);   // per-leaf cost is uniform: a sample of leaves suffices
  DevMesh dm = M->dev();
  dm.B = nleaf;
  // The sweeps of a whole step, stores into the neighbours' ghost rows included, on
  // a copy of the sample.  Where there is no room for one they run in place and
  // leave the neighbours' ghost rows alone (dt = 0: the interiors stay as they are,
  // but for a rho e that the dual-energy synchronisation resets).
  const size_t bytes = (size_t)nleaf * nfields(d) * M->N * M->N * M->N * d.precision;
  cudaEvent_t ev[4];
  for (int i = 0; i < 4; ++i) CELLO_CUDA(cudaEventCreate(&ev[i]));
  void* copy = nullptr;
  if (cudaMalloc(&copy, bytes) != cudaSuccess) {
    cudaGetLastError();
    copy = nullptr;
  }
  int best[3] = {0, 0, 0};
  float best_ms[3] = {1e30f, 1e30f, 1e30f};
  cudaError_t err = copy ? cudaMemcpyAsync(copy, U, bytes, cudaMemcpyDeviceToDevice, s) : cudaSuccess;
  float times[kMaxSweepVariants][3];
  for (int v = 0; v < nv && err == cudaSuccess; ++v) {
    float* vbest = times[v];
    std::fill(vbest, vbest + 3, 1e30f);
    const int twin = d.precision == 4 ? sweep_variant_twin_f32(v, d.dual_energy != 0) : v;
    if (twin != v)   // the same kernel and schedule: timed already
      std::copy(times[twin], times[twin] + 3, vbest);
    for (int rep = 0; rep < 4 && twin == v && err == cudaSuccess; ++rep) {
      float axis_ms[3] = {0, 0, 0};
      // the sweeps of an even (x, y, z) and an odd (z, y, x) cycle, dt = 0 (state unchanged):
      // each axis is timed in both of its positions
      for (int parity = 0; parity < 2 && err == cudaSuccess; ++parity) {
        const int order[3] = {parity == 0 ? 0 : 2, 1, parity == 0 ? 2 : 0};
        cudaEventRecord(ev[0], s);
        for (int oi = 0; oi < 3; ++oi) {
          SweepParams p{};
          p.U = copy ? copy : U;
          p.dt = M->d_zero;
          p.reg = nullptr;
          p.variant = v;
          set_regions(M, p, order, oi, 0, nleaf, true);
          if (!copy) p.push = -1;
          launch_sweep(M, dm, p, s);
          cudaEventRecord(ev[oi + 1], s);
        }
        err = cudaEventSynchronize(ev[3]);
        for (int oi = 0; oi < 3 && err == cudaSuccess; ++oi) {
          float ms = 0;
          err = cudaEventElapsedTime(&ms, ev[oi], ev[oi + 1]);
          axis_ms[order[oi]] += ms;
        }
      }
      if (rep > 0)   // the first repetition warms up
        for (int a = 0; a < 3; ++a) vbest[a] = std::min(vbest[a], axis_ms[a]);
    }
    for (int a = 0; a < 3; ++a) {
      if (ms_out && 3 * v + a < ms_len) ms_out[3 * v + a] = vbest[a];
      if (vbest[a] < best_ms[a]) {
        best_ms[a] = vbest[a];
        best[a] = v;
      }
    }
  }
  for (int i = 0; i < 4; ++i) cudaEventDestroy(ev[i]);
  if (copy) cudaFree(copy);
  CELLO_CUDA(err);
  CELLO_CUDA(cudaGetLastError());
  if (variants_out)
    for (int a = 0; a < 3; ++a) variants_out[a] = best[a];
  return cello_set_sweep_variants(M, best);
}

cello_status cello_hydro_step_host(cello_mesh* M, void* U_host, void* U_dev, double dt_host, double* dt_dev,
                                   int cycle, double cfl, double* scratch_dev, double* out_host, void* stream) {
  if (!M || !U_host || !U_dev || !dt_dev || !scratch_dev || !out_host) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U_dev);
  cudaStream_t s = (cudaStream_t)stream;
  const size_t bytes = (size_t)M->B * nfields(M->desc) * M->N * M->N * M->N * (size_t)M->desc.precision;
  // Host memory with a device address (page-locked, or any host memory where
  // the GPU reads the host's page tables), 16-byte aligned: the SMs read and
  // write its interior cells only (the step rewrites every ghost cell from
  // interiors before reading one).  Otherwise whole-buffer copies.
  void* h_dev = nullptr;
  bool mapped = false;
  if ((reinterpret_cast<uintptr_t>(U_host) & 15u) == 0) {
    if (cudaHostGetDevicePointer(&h_dev, U_host, 0) == cudaSuccess) mapped = h_dev != nullptr;
    else cudaGetLastError();   // no device address for this memory
  }
  const DevMesh dm = M->dev();
  if (mapped) launch_interior_copy(dm, h_dev, U_dev, M->desc.precision, s);
  else CELLO_CUDA(cudaMemcpyAsync(U_dev, U_host, bytes, cudaMemcpyHostToDevice, s));
  CELLO_CUDA(cudaMemcpyAsync(dt_dev, &dt_host, sizeof(double), cudaMemcpyHostToDevice, s));
  CELLO_TRY(cello_hydro_step(M, U_dev, dt_dev, cycle, cfl, scratch_dev, scratch_dev + 1, stream));
  if (mapped) launch_interior_copy(dm, U_dev, h_dev, M->desc.precision, s);
  else CELLO_CUDA(cudaMemcpyAsync(U_host, U_dev, bytes, cudaMemcpyDeviceToHost, s));
  CELLO_CUDA(cudaMemcpyAsync(out_host, scratch_dev, 6 * sizeof(double), cudaMemcpyDeviceToHost, s));
  CELLO_CUDA(cudaStreamSynchronize(s));
  return CELLO_OK;
}

cello_status cello_particles_locate(cello_mesh* M, const double* pos, int32_t* leaf, int64_t count, void* stream) {
  if (!M || (count > 0 && (!pos || !leaf)) || count < 0) return fail(CELLO_EINVAL, "NULL argument or negative count");
  launch_particles_locate(M->dev(), M->d_keys, M->desc.lo, M->desc.hi, pos, leaf, (long)count, (cudaStream_t)stream);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

cello_status cello_particles_push(cello_mesh* M, const void* U, double* pos, int32_t* leaf, int64_t count,
                                  const double* dt, void* stream) {
  if (!M || !U || !dt || (count > 0 && (!pos || !leaf)) || count < 0)
    return fail(CELLO_EINVAL, "NULL argument or negative count");
  CELLO_REQUIRE_ALIGNED(U);
  launch_particles_push(M->dev(), M->d_keys, M->desc.lo, M->desc.hi, U, M->desc.precision, pos, leaf, (long)count, dt,
                        (cudaStream_t)stream);
  CELLO_CUDA(cudaGetLastError());
  return CELLO_OK;
}

cello_status cello_poisson_solve(cello_mesh* M, const double* f, double* phi, int cycles, int inner,
                                 double* resid_host, void* stream) {
  if (!M || !f || !phi || cycles < 1) return fail(CELLO_EINVAL, "NULL argument or cycles < 1");
  if (inner != 4 && inner != 8) return fail(CELLO_EINVAL, "inner precision must be 4 or 8");
  const cello_mesh_desc& d = M->desc;
  for (int a = 0; a < 3; ++a)
    if (d.bc[a] != CELLO_PERIODIC || d.root[a] != d.root[0])
      return fail(CELLO_EINVAL, "the Poisson solver needs a cubic root array, periodic on every axis");
  const int L = M->leaves[0].x;
  for (const int4& lf : M->leaves)
    if (lf.x != L) return fail(CELLO_EINVAL, "the Poisson solver needs a uniform mesh (every leaf at one level)");
  const long Mg = (long)d.root[0] * (1L << L) * d.n;
  if (Mg / d.n > 512) return fail(CELLO_EINVAL, "grid too large for the Poisson solver (more than 512 blocks per axis)");
  const double h = std::ldexp((d.hi[0] - d.lo[0]) / (d.root[0] * d.n), -L);
  CELLO_CUDA(poisson_solve(&M->poisson, M->dev(), (int)Mg, h, f, phi, cycles, inner, resid_host,
                           (cudaStream_t)stream));
  return CELLO_OK;
}

cello_status cello_sweep_opcount(const cello_mesh* M, float* U_host, const int32_t* leaf_ids, int64_t count,
                                 double dt, int cycle, double* out) {
  if (!M || !U_host || !leaf_ids || !out || count <= 0) return fail(CELLO_EINVAL, "NULL argument or empty sample");
  if (M->desc.precision != 4) return fail(CELLO_EINVAL, "operation counts are taken on float32 meshes");
  for (int64_t i = 0; i < count; ++i)
    if (leaf_ids[i] < 0 || leaf_ids[i] >= M->B) return fail(CELLO_EINVAL, "leaf id out of range");
  const cello_mesh_desc& d = M->desc;
  const long slab = (long)nfields(d) * M->N * M->N * M->N;
  const double dx0 = (d.hi[0] - d.lo[0]) / (d.root[0] * d.n);
  for (int k = 0; k < 3 * 8; ++k) out[k] = 0.0;
  const int order[3] = {cycle % 2 == 0 ? 0 : 2, 1, cycle % 2 == 0 ? 2 : 0};
  bool swept[3] = {false, false, false};
  for (int oi = 0; oi < 3; ++oi) {
    const int axis = order[oi];
    int a0, a1, b0, b1;
    sweep_ranges(M, axis, swept, a0, a1, b0, b1);
    unsigned long long c[6] = {0, 0, 0, 0, 0, 0};
    for (int64_t i = 0; i < count; ++i) {
      const double dtdx = dt / std::ldexp(dx0, -M->leaves[leaf_ids[i]].x);
      opcount_leaf(U_host + i * slab, d.n, d.ghosts, axis, a0, a1, b0, b1, dtdx, d.gamma, d.riemann, d.steepening,
                   d.dual_energy, c);
    }
    for (int k = 0; k < 6; ++k) out[oi * 8 + k] = (double)c[k];
    out[oi * 8 + 6] = (double)count * (a1 - a0) * (b1 - b0);
    out[oi * 8 + 7] = out[oi * 8 + 6] * d.n;
    swept[axis] = true;
  }
  return CELLO_OK;
}

cello_status cello_profile_step(cello_mesh* M, void* U, const double* dt, int cycle, double cfl, float* phase_ms,
                                void* stream) {
  if (!M || !U || !dt || !phase_ms) return fail(CELLO_EINVAL, "NULL argument");
  CELLO_REQUIRE_ALIGNED(U);
  cudaStream_t s = (cudaStream_t)stream;
  cudaEvent_t ev[7];
  for (int i = 0; i < 7; ++i) CELLO_CUDA(cudaEventCreate(&ev[i]));
  enqueue_step(M, U, dt, cycle, cfl, nullptr, nullptr, s, ev);
  cudaError_t e = cudaEventSynchronize(ev[6]);
  for (int i = 0; i < 6 && e == cudaSuccess; ++i) e = cudaEventElapsedTime(&phase_ms[i], ev[i], ev[i + 1]);
  for (int i = 0; i < 7; ++i) cudaEventDestroy(ev[i]);
  CELLO_CUDA(e);
  return CELLO_OK;
}

}  // extern "C"
