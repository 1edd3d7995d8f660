// Tracer particles (Sec. II.B: Lagrangian particles that move between
// Blocks; Sec. III: the hydro scaling workload carries tracers).  Positions
// are float64 in structure-of-arrays form pos[3][count]; each tracer keeps
// the index of the leaf that contains it, -1 once lost through an outflow
// face.  Built without FMA contraction: every position is the same float64
// arithmetic as a term-by-term evaluation.
//
// Lookup: the block index at max_level of the point, b = floor((x - lo) /
// w) clamped into the root array, gives a Morton key; the containing leaf is
// the last leaf whose key does not exceed it (leaves tile the domain and
// are sorted by key).  Velocity: momentum over floored density, trilinear
// between the cell centres of the leaf's padded block (ghosts refreshed),
// along x, then y, then z.  Push: x += dt u, periodic wrap or outflow loss,
// lookup again (migration).
//
// Where the block width at max_level and the level-0 cell width are powers
// of two (a box whose extent over the root count is one), each division by a
// width is a multiplication by its reciprocal, also a power of two: both
// give the correctly rounded value of the same exact quotient, so the
// results are bit-identical, and six float64 divisions per tracer leave the
// slow float64 pipe.
#include "cello_internal.h"
#include "morton.h"
#include "ppm.cuh"
#include "widen.cuh"

namespace cello {
namespace {

struct PartMesh {
  DevMesh m;
  const unsigned long long* keys;
  double lo[3], hi[3];
  double w;   // block width at max_level
  double inv_w, inv_dx0;   // 1 / w and 1 / (level-0 cell width), exact when pow2
  bool pow2;               // both widths powers of two
};

// floor(v) of |v| < 2^31 from the low word of v + 1.5 2^52 rounded down: one
// float64 instruction, where floor and a conversion are two of the same pipe.
__device__ __forceinline__ int floor_int(double v) {
  const int big = __double2hiint(v) & 0x7fffffff;   // exponent and top of the fraction
  if (big < 0x41e00000) return __double2loint(__dadd_rd(v, 6755399441055744.0));
  return __double2int_rd(v);   // saturates
}

__device__ __forceinline__ double over_w(const PartMesh& P, double d) { return P.pow2 ? d * P.inv_w : d / P.w; }

__device__ __forceinline__ unsigned long long point_key(const PartMesh& P, const double x[3]) {
  unsigned b[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int nb = P.m.root[a] << P.m.max_level;   // at most 2^20
    const int v = floor_int(over_w(P, x[a] - P.lo[a]));
    b[a] = (unsigned)(v < 0 ? 0 : (v > nb - 1 ? nb - 1 : v));
  }
  return morton3(b[0], b[1], b[2]);
}

__device__ __forceinline__ int locate_key(const PartMesh& P, unsigned long long k) {
  int lo = 0, hi = P.m.B;   // first key > k
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (P.keys[mid] <= k) lo = mid + 1;
    else hi = mid;
  }
  return lo - 1;
}

// Velocity (3 components) of the cell at offset o of a padded block: momentum
// times 1/rho, the reciprocal a float32 seed refined in float64 by r (1 + e +
// e^2), e = 1 - rho r, |e| < 2^-22 (within 1 ulp; a float64 division costs ten
// instructions of the float64 pipe, which bounds the push).
__device__ __forceinline__ void cell_velocity(const double* blk, long SLAB, long o, double v[3]) {
  const double r = blk[o];
  const double rho = r > kRhoFloor ? r : kRhoFloor;
  const double s = (double)__frcp_rn((float)rho);
  const double e = fma(-rho, s, 1.0);
  const double ir = fma(s, fma(e, e, e), s);
#pragma unroll
  for (int c = 0; c < 3; ++c) v[c] = blk[(1 + c) * SLAB + o] * ir;
}

// Float32 state: e = 1 - rho r is exact in float32, e^2 needs no more, and the
// values reach float64 by integer instructions (widen): 5 float64 instructions a
// corner instead of 16 with the conversions.
__device__ __forceinline__ double density_reciprocal(float rho) {
  if (rho > 1e-9f && rho < 1e30f) {   // seed and remainder are normal numbers
    const float s = __frcp_rn(rho), e = __fmaf_rn(-rho, s, 1.0f);
    const double sd = widen(s);
    return fma(sd, widen(e) + widen(__fmul_rn(e, e)), sd);
  }
  return 1.0 / ((double)rho > kRhoFloor ? (double)rho : kRhoFloor);
}

// The eight corner velocities, x fastest: corner (dz, dy, dx) at 4 dz + 2 dy + dx.
__device__ __forceinline__ void corner_velocities(const double* blk, long SLAB, long o, long sy, long sz,
                                                  double cv[8][3]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) cell_velocity(blk, SLAB, o + (q >> 2) * sz + ((q >> 1) & 1) * sy + (q & 1), cv[q]);
}

// Float32: every value is asked for before the first is used (the branches between
// the corners kept the loads apart, and randomly placed tracers wait on them).
__device__ __forceinline__ void corner_velocities(const float* blk, long SLAB, long o, long sy, long sz,
                                                  double cv[8][3]) {
  float u[4][8];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int q = 0; q < 8; ++q) u[c][q] = __ldg(blk + c * SLAB + o + (q >> 2) * sz + ((q >> 1) & 1) * sy + (q & 1));
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const double ir = density_reciprocal(u[0][q]);
#pragma unroll
    for (int c = 0; c < 3; ++c) cv[q][c] = widen(u[1 + c][q]) * ir;
  }
}

// Three CTAs of 256 per SM (80 registers, a few spilled to L1): the corner
// gathers of randomly placed tracers are latency bound, and the extra warps
// hide more of it.
template <typename T>
__global__ void __launch_bounds__(256, 3) particles_push_kernel(PartMesh P, const T* U, double* pos, int* leaf, long count,
                                      const double* dt_dev) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int b = leaf[i];
  if (b < 0 || b >= P.m.B) return;
  const DevMesh& m = P.m;
  const int n = m.n, g = m.g, N = m.N;
  const long SLAB = (long)N * N * N;
  const int4 lf = m.leaf[b];
  const double dx = ldexp(m.dx0, -lf.x);
  const double inv_dx = ldexp(P.inv_dx0, lf.x);
  const int lidx[3] = {lf.y, lf.z, lf.w};
  double x[3], f[3];
  int i0[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    x[a] = pos[a * count + i];
    const double d = x[a] - (P.lo[a] + (double)(lidx[a] * n) * dx);
    const double s = (P.pow2 ? d * inv_dx : d / dx) - 0.5;
    const double c = floor(s);
    i0[a] = corner_index(floor_int(c), g, N);
    f[a] = s - c;
  }
  const T* blk = U + (long)b * m.nf * SLAB;
  const long o000 = ((long)i0[2] * N + i0[1]) * N + i0[0];
  const double dt = *dt_dev;
  const unsigned long long here = P.keys[b], beyond = b + 1 < m.B ? P.keys[b + 1] : ~0ull;
  double cv[8][3];
  corner_velocities(blk, SLAB, o000, N, (long)N * N, cv);
  bool lost = false;
#pragma unroll
  for (int comp = 0; comp < 3; ++comp) {
    const double fx = f[0], fy = f[1], fz = f[2];
    const double c00 = cv[0][comp] * (1.0 - fx) + cv[1][comp] * fx;
    const double c10 = cv[2][comp] * (1.0 - fx) + cv[3][comp] * fx;
    const double c01 = cv[4][comp] * (1.0 - fx) + cv[5][comp] * fx;
    const double c11 = cv[6][comp] * (1.0 - fx) + cv[7][comp] * fx;
    const double c0 = c00 * (1.0 - fy) + c10 * fy;
    const double c1 = c01 * (1.0 - fy) + c11 * fy;
    const double v = c0 * (1.0 - fz) + c1 * fz;
    double xn = x[comp] + dt * v;
    const double ext = P.hi[comp] - P.lo[comp];
    if (m.bc[comp] == CELLO_PERIODIC) {
      xn = xn < P.lo[comp] ? xn + ext : (xn >= P.hi[comp] ? xn - ext : xn);
    } else if (xn < P.lo[comp] || xn >= P.hi[comp]) {
      lost = true;
    }
    x[comp] = xn;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) pos[a * count + i] = x[a];
  // most tracers stay in their leaf, whose keys are at hand: the search is a chain
  // of loads
  if (lost) {
    leaf[i] = -1;
  } else {
    const unsigned long long k = point_key(P, x);
    if (k < here || k >= beyond) leaf[i] = locate_key(P, k);
  }
}

__global__ void particles_locate_kernel(PartMesh P, const double* pos, int* leaf, long count) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const double x[3] = {pos[i], pos[count + i], pos[2 * count + i]};
  leaf[i] = locate_key(P, point_key(P, x));
}

bool is_pow2(double v) {
  int e;
  return v > 0.0 && std::frexp(v, &e) == 0.5;
}

PartMesh part_mesh(const DevMesh& m, const unsigned long long* keys, const double lo[3], const double hi[3]) {
  PartMesh P{m, keys, {lo[0], lo[1], lo[2]}, {hi[0], hi[1], hi[2]}, ldexp((hi[0] - lo[0]) / m.root[0], -m.max_level)};
  P.pow2 = is_pow2(P.w) && is_pow2(m.dx0);
  P.inv_w = 1.0 / P.w;
  P.inv_dx0 = 1.0 / m.dx0;
  return P;
}

}  // namespace

void launch_particles_locate(const DevMesh& m, const unsigned long long* keys, const double lo[3], const double hi[3],
                             const double* pos, int* leaf, long count, cudaStream_t s) {
  if (count <= 0) return;
  const PartMesh P = part_mesh(m, keys, lo, hi);
  particles_locate_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(P, pos, leaf, count);
}

void launch_particles_push(const DevMesh& m, const unsigned long long* keys, const double lo[3], const double hi[3],
                           const void* U, int precision, double* pos, int* leaf, long count, const double* dt,
                           cudaStream_t s) {
  if (count <= 0) return;
  const PartMesh P = part_mesh(m, keys, lo, hi);
  const unsigned grid = (unsigned)((count + 255) / 256);
  if (precision == 4)
    particles_push_kernel<float><<<grid, 256, 0, s>>>(P, static_cast<const float*>(U), pos, leaf, count, dt);
  else
    particles_push_kernel<double><<<grid, 256, 0, s>>>(P, static_cast<const double*>(U), pos, leaf, count, dt);
}

}  // namespace cello
