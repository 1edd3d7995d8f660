// Internal types shared by the host orchestration and the kernel translation
// units.  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "cello.h"

namespace cello {

constexpr int kGhosts = 4;
constexpr int kFields = 5;
// Pencils per adjoint-sweep CTA for blocks of n cells per edge and values of elem
// bytes: 16 fill whole warps (float64, gradient on 64 leaves of 16^3: 26.4 ms against 28.3
// with 8) as far as one CTA's registers go; float32 waits for latency instead, and two
// smaller CTAs per SM hide it (2.16 -> 1.83 ms).
constexpr int adj_pencils(int n, int elem) { return n == 32 || (n == 16 && elem == 4) ? 8 : 16; }

// Launch variants of the PPM sweep: pencils per CTA, the minimum number of
// resident CTAs per SM the register allocation is bounded for, and the
// schedule (static: one CTA per item; persistent: resident CTAs take over the
// items that have not started, ItemQueue in kernels.cuh).  The autotuner times them.
struct SweepVariant {
  int pencils;       // pencils per CTA (the CTA size of the streaming form)
  int min_blocks;    // resident CTAs per SM the register bound is set for
  bool persistent;
  bool stream;       // register-streaming form (sweep_stream_kernel)
  int vec;           // streaming form moving x pencils four cells at a time, staged by cp.async (3), or not (0)
};
constexpr int kMaxSweepVariants = 24;   // of a precision
int sweep_variant_count_f32();
// The first variant with the kernel and schedule of variant v: v itself, but for
// dual-energy meshes, whose streaming kernels all have one register bound.
int sweep_variant_twin_f32(int v, bool dual);
int sweep_variant_count_f64();

// Neighbour kinds of the 27-entry table.
enum NbKind : int8_t { kSame = 0, kCoarse = 1, kFine = 2, kBoundary = 3 };

// Read-only view of the device-resident block table.
struct DevMesh {
  int n, g, N;            // cells per block edge, ghosts, padded edge
  int max_level;
  int root[3];
  int bc[3];              // 0 periodic, 1 outflow
  double dx0;             // cell width at level 0
  double gamma;
  int riemann;            // CELLO_RIEMANN_TWO_SHOCK or CELLO_RIEMANN_HLLC
  int steepen;            // contact steepening of the density edge values
  int nf;                 // fields per cell: 5, or 6 with the dual-energy formalism's rho e
  int B;                  // leaves
  const int4* leaf;       // (level, i, j, k)
  const int8_t* kind;     // [B][27]
  const int* idx;         // [B][27]
  const int* fine8;       // [B][27][8]
  const int* face_slot;   // [B][6] flux-register slot of each face or -1
  unsigned* err;          // error word: bit 0 set by the reduction on a non-finite or non-positive state
};

// Face order used by registers and corrections: -x, +x, -y, +y, -z, +z.
__host__ __device__ inline int face_dir(int axis, int side) {
  int d[3] = {0, 0, 0};
  d[axis] = side;
  return (d[2] + 1) * 9 + (d[1] + 1) * 3 + (d[0] + 1);
}

// One coarse face that touches four finer leaves.
struct CoarseFace {
  int leaf;       // coarse leaf
  int axis, side; // face
  int cslot;      // register slot of the coarse flux
  int fslot[4];   // register slots of the fine fluxes, index o2*2 + o1
};

// Unsigned division by a launch-time constant as a multiply-high and shift
// (Granlund & Montgomery): valid for dividends below 2^31.
struct FastDiv {
  unsigned d, m, s;
  __host__ __device__ static FastDiv make(unsigned d) {
    FastDiv f;
    f.d = d;
    f.s = 0;
    while ((1u << f.s) < d) ++f.s;
    f.m = (unsigned)((((unsigned long long)1 << 32) * ((1ull << f.s) - d)) / d + 1);
    return f;
  }
  __device__ __forceinline__ unsigned div(unsigned x) const { return (__umulhi(x, m) + x) >> s; }
};

// Padded index of the lower corner of a tracer, v cells from its leaf's first cell.
// A tracer inside its leaf has v in [-1, n); one that is not (a NaN, a step across
// the box, a leaf index that is not the position's) reads the block's outermost
// cells instead of memory outside it.
__host__ __device__ __forceinline__ int corner_index(int v, int g, int N) {
  const int lo = -g, hi = N - 2 - g;
  return (v < lo ? lo : (v > hi ? hi : v)) + g;
}

// Transverse pencils of one work item's leaf: cb pencils along transverse axis
// B times count / cb along A, from (a0, b0).  Region 0 of a sweep is a
// rectangle of every leaf; regions 1 and 2 belong to listed faces (leaf * 6 +
// face), the ghost rows behind one face, shifted by (da, db) on its + side.
struct SweepRegion {
  int a0, b0, da, db;
  int cb, count;
  int tiles;               // work items per leaf or face, set by the launcher from the pencils per CTA
  int items;               // set by the launcher
  FastDiv div_cb, div_tiles;
  const int* faces;        // null in region 0
  int nfaces;
};

// Where a pencil of a work item lies.
struct PencilAt {
  int leaf;
  int q;                   // first pencil of the item within its region
  int r;                   // region
  int a0, b0;
};

struct SweepParams {
  void* U;
  int leaf0, nleaf;        // leaves [leaf0, leaf0 + nleaf)
  int axis;
  SweepRegion reg3[3];
  int push;                // transverse axis across whose same-level faces the updated rows are also stored, or -1
  const double* dt;        // device scalar
  double* reg;             // flux registers (may be null)
  int n_items;             // set by the launcher: the grid, one CTA per item
  bool persistent;         // set by the launcher: CTAs take over items that have not started
  int variant;             // index into the sweep variants of the precision; -1: the launcher's rule

  // The items of the three regions for per_cta pencils per item.
  void plan(int per_cta) {
    n_items = 0;
    for (int r = 0; r < 3; ++r) {
      SweepRegion& g = reg3[r];
      const int owners = r == 0 ? nleaf : g.nfaces;
      g.tiles = owners > 0 ? (g.count + per_cta - 1) / per_cta : 0;
      g.items = owners * g.tiles;
      if (g.items > 0) {
        g.div_cb = FastDiv::make((unsigned)g.cb);
        g.div_tiles = FastDiv::make((unsigned)g.tiles);
      }
      n_items += g.items;
    }
  }

  __device__ __forceinline__ PencilAt locate(int item, int per_cta) const {
    PencilAt w;
    w.r = 0;
    if (item >= reg3[0].items) {
      item -= reg3[0].items;
      w.r = item < reg3[1].items ? 1 : 2;
      if (w.r == 2) item -= reg3[1].items;
    }
    const SweepRegion& g = reg3[w.r];
    const int owner = (int)g.div_tiles.div((unsigned)item);
    w.q = (item - owner * g.tiles) * per_cta;
    w.a0 = g.a0;
    w.b0 = g.b0;
    if (w.r == 0) {
      w.leaf = leaf0 + owner;
    } else {
      const int f = g.faces[owner];
      w.leaf = f / 6;
      if (f & 1) {
        w.a0 += g.da;
        w.b0 += g.db;
      }
    }
    return w;
  }
};

struct AdjSweepParams {
  const void* U;           // state entering the forward sweep (ghosts refreshed)
  void* lam;               // adjoint, updated in place
  const double* regb;      // adjoints of the face fluxes kept for flux correction (may be null)
  int leaf0, nleaf;
  int axis;
  int a0, a1, b0, b1;
  int tiles_per_leaf;
  const double* dt;
  int n_items;
};

// Remap of one new leaf from the old mesh: copy (src[0]), prolongation from
// the old leaf src[0] that is k levels coarser, or restriction from the 8 old
// children src[octant].
struct RemapEntry {
  int kind;   // 0 copy, 1 prolong, 2 restrict
  int k;
  int src[8];
};
// The entries of every new leaf into map, then the cells; where a new leaf has
// no source, *bad is set and no cell is written.
void launch_remap(const DevMesh& neu, const unsigned long long* nkeys, const DevMesh& old,
                  const unsigned long long* okeys, const void* Uold, void* Unew, RemapEntry* map, int* bad,
                  int precision, cudaStream_t s);
void launch_remap_map(const DevMesh& neu, const unsigned long long* nkeys, const DevMesh& old,
                      const unsigned long long* okeys, RemapEntry* map, int* bad, cudaStream_t s);

// Accessors for translation units that see cello_mesh only as an opaque type.
DevMesh mesh_dev(const cello_mesh* mesh);
int mesh_precision(const cello_mesh* mesh);
cello_status set_error(cello_status status, const char* message);

// Kernel attributes (dynamic shared memory limits) for the current device, set
// once per device, outside any stream capture.
void prepare_kernels();
void prepare_kernels_f32();
void prepare_kernels_f64();

// Launchers (defined in the kernel translation units).
void launch_neighbour_table(const DevMesh& m, const unsigned long long* keys, int8_t* kind, int* idx,
                            int* fine8, int8_t* face, int* bad, cudaStream_t s);
void launch_fine_slots(const DevMesh& m, CoarseFace* faces, int count, cudaStream_t s);
// Ghost refresh of leaves [leaf0, leaf0+nleaf) in phases, in this order: the
// listed slow faces (leaf * 6 + face of the faces of these leaves whose
// neighbour is not a same-level leaf: their phase regions computed from leaf
// interiors), then the same-level face copies along x, y and z (each phase
// reads the margins the earlier ones filled in the face neighbours).
// `phases` selects a subset; a phase must have run on every leaf before the
// next one starts.
//
// The two forms a step needs, whose sweeps fill the ghost rows behind
// same-level faces themselves (see push_offset in kernels.cuh): an x, y, z step
// reads the x margins of the interior rows and the slow regions (kRefreshXFirst);
// a z, y, x step the z ghosts of the interior columns (kRefreshZRows, whole rows
// of interior y) and then the slow regions nested the other way round
// (kRefreshSlowZFirst: the interior columns behind a z face, all z behind a y
// face, all y and z behind an x face).
enum RefreshPhase : int {
  kRefreshSlow = 1, kRefreshX = 2, kRefreshY = 4, kRefreshZ = 8, kRefreshAll = 15,
  kRefreshZRows = 16, kRefreshSlowZFirst = 32,
  kRefreshXFirst = kRefreshSlow | kRefreshX, kRefreshZFirst = kRefreshZRows | kRefreshSlowZFirst
};
void launch_refresh_f32(const DevMesh& m, float* U, int leaf0, int nleaf, const int* slow, int nslow,
                        int phases, cudaStream_t s);
void launch_refresh_f64(const DevMesh& m, double* U, int leaf0, int nleaf, const int* slow, int nslow,
                        int phases, cudaStream_t s);
void launch_sweep_f32(const DevMesh& m, const SweepParams& p, cudaStream_t s);
void launch_sweep_f64(const DevMesh& m, const SweepParams& p, cudaStream_t s);
template <int NB>
void prepare_sweep_f32();
template <int NB>
void launch_sweep_f32_nb(const DevMesh& m, const SweepParams& p, cudaStream_t s);
// Dual-energy sweeps (both float32 forms, sweep_de_f32.cuh; float64, k_de_f64.cu),
// launched by the planners above with the items they planned.
template <int NB, int P, int MINB>
void launch_sweep_de_f32(const DevMesh& m, const SweepParams& p, cudaStream_t s);
template <int NB, int CT, int VEC>
void launch_stream_de_f32(const DevMesh& m, const SweepParams& p, cudaStream_t s);
template <int NB>
void launch_sweep_de_f64(const DevMesh& m, const SweepParams& p, cudaStream_t s);
// Attributes of the dual-energy kernels.
template <int NB>
void prepare_sweep_de_f32();
void prepare_kernels_de_f64();
void launch_fluxcorr(const DevMesh& m, void* U, int precision, const CoarseFace* faces,
                     const int* group_start, int ngroups, const double* reg, const double* dt,
                     cudaStream_t s);
// grid > 0: that many CTAs walk the leaves (a reduction that is to run
// alongside other kernels); 0: one CTA per leaf.  The result is the same.
void launch_reduce(const DevMesh& m, const void* U, int precision, double cfl, double* partials,
                   double* dt_next, double* totals, cudaStream_t s, int grid = 0);
// The same over leaves [leaf0, leaf0 + nleaf): partials of those leaves at
// their own offsets, the min and the sums over the range only.
void launch_reduce_range(const DevMesh& m, const void* U, int precision, double cfl, double* partials, int leaf0,
                         int nleaf, double* dt_next, double* totals, cudaStream_t s, int grid = 0);
void launch_adjoint_sweep_f32(const DevMesh& m, const AdjSweepParams& p, cudaStream_t s);
void launch_adjoint_sweep_f64(const DevMesh& m, const AdjSweepParams& p, cudaStream_t s);
void launch_adjoint_refresh(const DevMesh& m, void* lam, int precision, cudaStream_t s);
// AMR form: scatter each ghost cell's adjoint onto its sources (copies,
// restrictions, limited prolongations evaluated at the refreshed state U),
// then clear the ghost adjoints.
void launch_adjoint_refresh_scatter(const DevMesh& m, const void* U, void* lam, int precision, cudaStream_t s);
void launch_fluxcorr_adjoint(const DevMesh& m, const void* lam, int precision, const CoarseFace* faces, int nfaces,
                             double* regb, const double* dt, cudaStream_t s);
void launch_zero_ghosts(const DevMesh& m, void* lam, int precision, cudaStream_t s);
void launch_reduce_partials_f32(const DevMesh& m, const float* U, double* partials, int leaf0, int nleaf, int grid,
                                cudaStream_t s);
void launch_flags(const DevMesh& m, const void* U, int precision, int field, double tau, double tau_c,
                  int8_t* flags, cudaStream_t s);
// Multigrid Poisson solver (poisson.cu) on the M^3 grid of a uniform periodic mesh.
struct PoissonScratch;
void poisson_free(PoissonScratch* p);
cudaError_t poisson_solve(PoissonScratch** scratch, const DevMesh& m, int M, double h, const double* f_leaves,
                          double* phi_leaves, int cycles, int inner, double* resid_host, cudaStream_t s);
// Tracer particles (particles.cu): lookup of the containing leaf, and one push.
void launch_particles_locate(const DevMesh& m, const unsigned long long* keys, const double lo[3], const double hi[3],
                             const double* pos, int* leaf, long count, cudaStream_t s);
void launch_particles_push(const DevMesh& m, const unsigned long long* keys, const double lo[3], const double hi[3],
                           const void* U, int precision, double* pos, int* leaf, long count, const double* dt,
                           cudaStream_t s);
// Sharded step (k_f64.cu): interiors of the listed leaves to (pack = 1) or
// from (pack = 0) buf[count][nf][n^3]; float64 flux-register slots (per
// doubles each) to or from buf[count][per].
void launch_halo_copy(const DevMesh& m, void* U, int precision, const int* ids, long count, void* buf, int pack,
                      cudaStream_t s);
void launch_flux_copy(double* reg, const int* slots, long count, long per, double* buf, int pack, cudaStream_t s);
// Interior cells of every leaf and field from src to dst (same layout, both
// device-addressable, 16-byte aligned).
void launch_interior_copy(const DevMesh& m, const void* src, void* dst, int precision, cudaStream_t s);
// Host: counted operations of one leaf's sweep (opcount.cu), update applied.
void opcount_leaf(float* slab, int n, int g, int axis, int a0, int a1, int b0, int b1, double dtdx, double gamma,
                  int riemann, int steepen, int dual, unsigned long long counts[6]);

}  // namespace cello
