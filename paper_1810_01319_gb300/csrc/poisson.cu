// Multigrid Poisson solver (Sec. II.C: Enzo-P's mg0, a geometric multigrid
// V-cycle, the self-gravity solver of the paper's uniform-grid runs) on the
// block table of a uniform periodic mesh.
//
// Each leaf block carries its own grid on every level where a block still
// has at least 4 cells per edge (n, n/2, ..., 4), stored without ghost layers
// ([B][n_l^3]; on the finest level the layout of the caller's f and phi): a
// kernel stages a tile of a block with its halo in shared memory and reads the
// halo from the same-level neighbour blocks through the 27-entry neighbour
// table of the hydro refresh (the periodic wrap is in the table).  Below the
// last block level the restricted residual of the blocks forms one grid of 2
// cells per block edge with periodic indexing: tiles while the edge is a
// multiple of 4, then every remaining level in one CTA.  float64, no
// contraction.
//
// What bounds it: float32 cycles on large grids, HBM and L2 traffic, hence one
// kernel per leg and level (two sweeps, residual and restriction read f once and
// write phi once; interpolation and two sweeps read phi and f once and write
// once); float64 cycles and the float64 residual of mixed ones, the float64 pipe;
// small grids, the number of dependent launches (8 per mixed cycle on 64^3).
//
// V-cycle (spacing h): two damped Jacobi sweeps (w = 6/7), the residual of
// the 8 children of each coarse cell restricted by their mean, a V-cycle for
// the coarse error from zero with spacing 2h, its trilinear prolongation
// added, two more sweeps; a 1-cell grid gives 0, an odd grid above 1 takes
// 50 sweeps.  Mean of f removed first, mean of phi removed last.  Every value
// is the plain expression in its order on the same grid values (the block
// layout only changes where they are stored), with 1/h^2 and 1/6 as
// multiplications by reciprocals computed once (float64: and multiply-adds fused).
#include <vector>

#include "cello_internal.h"
#include "per_device.h"
#include "widen.cuh"

namespace cello {
namespace {

constexpr double kOmega = 6.0 / 7.0;
constexpr int kNu = 2;
constexpr int kCoarseSweeps = 50;
constexpr int kRedThreads = 256;

// M <= 1024 (checked by cello_poisson_solve): M^3 <= 2^30 and every grid
// offset fits 32-bit unsigned arithmetic.
__device__ __forceinline__ unsigned gidx(int x, int y, int z, int M) {
  return ((unsigned)z * (unsigned)M + (unsigned)y) * (unsigned)M + (unsigned)x;
}
__device__ __forceinline__ int wrapm(int v, int M) { return v < 0 ? v + M : (v >= M ? v - M : v); }

// The cycle's formulas.  Float64, bound by the float64 pipe, fuses multiplies with
// adds.  Float32 rounds term by term: after a few cycles of a mixed-precision
// solve its rounding is what is left of the error, and fused values would differ
// there by 1e-9 of the potential and more.
//
// Damped Jacobi value of a cell from its value c, neighbour sum s and
// right-hand side f.
__device__ __forceinline__ double relax(double c, double s, double f, double h2) {   // 3 instructions
  return fma(kOmega / 6.0, fma(-h2, f, s), (1.0 - kOmega) * c);
}
__device__ __forceinline__ float relax(float c, float s, float f, float h2) {
  return float(1.0 - kOmega) * c + float(kOmega) * ((s - h2 * f) * float(1.0 / 6.0));
}
// The same from a zero field (neighbour sum and cell 0).
__device__ __forceinline__ double relax_zero(double f, double h2) { return (kOmega / 6.0) * (-h2 * f); }
__device__ __forceinline__ float relax_zero(float f, float h2) { return float(kOmega) * ((-h2 * f) * float(1.0 / 6.0)); }
// f - lap(phi).
__device__ __forceinline__ double residual_of(double c, double s, double f, double ih2) {
  return fma(-ih2, fma(-6.0, c, s), f);
}
__device__ __forceinline__ float residual_of(float c, float s, float f, float ih2) { return f - (s - 6.0f * c) * ih2; }
// Linear interpolation a quarter of the way from p to q (q / 4 is exact).
__device__ __forceinline__ double quarter(double p, double q) { return fma(0.25, q, 0.75 * p); }
__device__ __forceinline__ float quarter(float p, float q) { return fmaf(0.25f, q, 0.75f * p); }

template <typename T>
__device__ __forceinline__ T nbsum(const T* p, int x, int y, int z, int M) {
  const T xm = p[gidx(wrapm(x - 1, M), y, z, M)], xp = p[gidx(wrapm(x + 1, M), y, z, M)];
  const T ym = p[gidx(x, wrapm(y - 1, M), z, M)], yp = p[gidx(x, wrapm(y + 1, M), z, M)];
  const T zm = p[gidx(x, y, wrapm(z - 1, M), M)], zp = p[gidx(x, y, wrapm(z + 1, M), M)];
  return ((((xm + xp) + ym) + yp) + zm) + zp;
}

// The grid kernels run one thread per cell of an M^3 (or, for the
// restriction, (M/2)^3) grid on a 3-D launch: 32 x 8 threads per CTA in
// (x, y), one CTA row per z plane, so no division recovers the coordinates.
// The Jacobi sweep instead walks kZC planes per thread along z, keeping the
// z-1, z and z+1 values of its column in registers.
constexpr int kBX = 32, kBY = 8, kZC = 8;
dim3 grid3(int M) { return dim3((unsigned)((M + kBX - 1) / kBX), (unsigned)((M + kBY - 1) / kBY), (unsigned)M); }
dim3 grid_zc(int M) {
  return dim3((unsigned)((M + kBX - 1) / kBX), (unsigned)((M + kBY - 1) / kBY), (unsigned)((M + kZC - 1) / kZC));
}
const dim3 kBlock3(kBX, kBY, 1);

__device__ __forceinline__ bool cell3(int M, int& x, int& y, int& z) {
  x = blockIdx.x * kBX + threadIdx.x;
  y = blockIdx.y * kBY + threadIdx.y;
  z = blockIdx.z;
  return x < M && y < M;
}

template <typename T>
__global__ void jacobi_kernel(const T* __restrict__ in, T* __restrict__ out, const T* __restrict__ f, int M, T h2) {
  const int x = blockIdx.x * kBX + threadIdx.x;
  const int y = blockIdx.y * kBY + threadIdx.y;
  if (x >= M || y >= M) return;
  const int z0 = blockIdx.z * kZC;
  const int z1 = z0 + kZC < M ? z0 + kZC : M;
  const unsigned uM = (unsigned)M, P = uM * uM;
  const unsigned xm = (unsigned)wrapm(x - 1, M), xp = (unsigned)wrapm(x + 1, M);
  const unsigned row = (unsigned)y * uM, rym = (unsigned)wrapm(y - 1, M) * uM, ryp = (unsigned)wrapm(y + 1, M) * uM;
  unsigned zb = (unsigned)z0 * P;
  T cm = in[(unsigned)wrapm(z0 - 1, M) * P + row + x];   // column values at z-1 and z
  T cc = in[zb + row + x];
  for (int z = z0; z < z1; ++z) {
    const T cp = in[(unsigned)wrapm(z + 1, M) * P + row + x];
    // the neighbour sum in the order of nbsum: x-1, x+1, y-1, y+1, z-1, z+1
    const T s = ((((in[zb + row + xm] + in[zb + row + xp]) + in[zb + rym + x]) + in[zb + ryp + x]) + cm) + cp;
    const unsigned i = zb + row + x;
    out[i] = relax(cc, s, f[i], h2);
    cm = cc;
    cc = cp;
    zb += P;
  }
}

// Coarse right-hand side: mean of the residuals f - lap(phi) of the 8
// children, in (dz, dy, dx) order.
template <typename T>
__global__ void residual_restrict_kernel(const T* __restrict__ phi, const T* __restrict__ f, T* __restrict__ fc,
                                         int M, T ih2) {
  const int Mc = M / 2;
  int X, Y, Z;
  if (!cell3(Mc, X, Y, Z)) return;
  const unsigned i = gidx(X, Y, Z, Mc);
  T s = T(0);
  bool first = true;
  for (int dz = 0; dz < 2; ++dz)
    for (int dy = 0; dy < 2; ++dy)
      for (int dx = 0; dx < 2; ++dx) {
        const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
        const unsigned o = gidx(x, y, z, M);
        const T r = residual_of(phi[o], nbsum(phi, x, y, z, M), f[o], ih2);
        s = first ? r : s + r;
        first = false;
      }
  fc[i] = s * T(0.125);
}

// Trilinear prolongation of the coarse error ec (Mc cells per edge) at a fine cell.
template <typename T>
__device__ __forceinline__ T prolonged(const T* ec, int x, int y, int z, int Mc) {
  const int X = x >> 1, Y = y >> 1, Z = z >> 1;
  const int sx = (x & 1) ? 1 : -1, sy = (y & 1) ? 1 : -1, sz = (z & 1) ? 1 : -1;
  const int X1 = wrapm(X + sx, Mc), Y1 = wrapm(Y + sy, Mc), Z1 = wrapm(Z + sz, Mc);
  const T c00 = quarter(ec[gidx(X, Y, Z, Mc)], ec[gidx(X1, Y, Z, Mc)]);
  const T c10 = quarter(ec[gidx(X, Y1, Z, Mc)], ec[gidx(X1, Y1, Z, Mc)]);
  const T c01 = quarter(ec[gidx(X, Y, Z1, Mc)], ec[gidx(X1, Y, Z1, Mc)]);
  const T c11 = quarter(ec[gidx(X, Y1, Z1, Mc)], ec[gidx(X1, Y1, Z1, Mc)]);
  return quarter(quarter(c00, c10), quarter(c01, c11));
}

template <typename T>
__global__ void prolong_add_kernel(const T* __restrict__ ec, T* __restrict__ phi, int M) {
  int x, y, z;
  if (!cell3(M, x, y, z)) return;
  const unsigned i = gidx(x, y, z, M);
  phi[i] = phi[i] + prolonged(ec, x, y, z, M / 2);
}

template <typename T>
__global__ void fill_kernel(T* p, long count, T v) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) p[i] = v;
}

__global__ void add_kernel(double* p, long count, const double* shift, double scale) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) p[i] = p[i] - *shift * scale;
}

// Partial sums per CTA; one CTA folds them (or maxima: op 1).
__global__ void reduce_kernel(const double* __restrict__ a, long count, double* __restrict__ partial) {
  __shared__ double sh[kRedThreads];
  double acc = 0.0;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long)gridDim.x * blockDim.x) acc += a[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] = sh[threadIdx.x] + sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

__global__ void fold_kernel(const double* __restrict__ partial, long n, int op, double scale, double* out) {
  __shared__ double sh[kRedThreads];
  double acc = 0.0;
  for (long i = threadIdx.x; i < n; i += blockDim.x) acc = op == 0 ? acc + partial[i] : fmax(acc, partial[i]);
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = kRedThreads / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      sh[threadIdx.x] = op == 0 ? sh[threadIdx.x] + sh[threadIdx.x + s] : fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0] * scale;
}

// ---------------------------------------------------------------------------
// Tile levels: arrays [B][n^3] of blocks without ghost layers; a CTA stages one
// E^3 tile of a block and a halo of one or two cells in shared memory, the halo
// cells read from the neighbour blocks through the 27-entry table (a periodic
// single array is one block that is its own neighbour in all 27 directions).
// Two cells of halo let one kernel run two sweeps and a residual, or an
// interpolation and two sweeps, on values that never leave the SM.
struct TileLevel {
  int n;                 // cells per block edge
  const int* idx;        // [B][27] neighbour blocks, or null: one periodic block
};

// A CTA's tile: block b, its 27 neighbours in shared memory, origin (x, y, z).
template <int E>
struct Tile {
  int b, x, y, z;
};

template <int E>
__device__ __forceinline__ Tile<E> tile_of(const TileLevel& L, int* s_nb) {
  const int per = L.n / E;
  unsigned t = blockIdx.x;
  Tile<E> w;
  w.x = (int)(t % per) * E; t /= per;
  w.y = (int)(t % per) * E; t /= per;
  w.z = (int)(t % per) * E; t /= per;
  w.b = (int)t;
  if (threadIdx.x < 27) s_nb[threadIdx.x] = L.idx ? L.idx[(long)w.b * 27 + threadIdx.x] : 0;
  __syncthreads();
  return w;
}

// Offset of the cell (x, y, z) of a block of n cells per edge, each coordinate
// in [-n, 2n), in the array of its level.
__device__ __forceinline__ long cell_at(int n, const int* s_nb, int x, int y, int z) {
  int e = 13;
  if (x < 0) { e -= 1; x += n; } else if (x >= n) { e += 1; x -= n; }
  if (y < 0) { e -= 3; y += n; } else if (y >= n) { e += 3; y -= n; }
  if (z < 0) { e -= 9; z += n; } else if (z >= n) { e += 9; z -= n; }
  return (((long)s_nb[e] * n + z) * n + y) * n + x;
}

// A thread works on columns along z of the cube of E + 2 H cells per edge around
// a tile: where a column lies is found once (the neighbour lookup and the index
// divisions took two thirds of the instructions of a cell-by-cell form), its
// loads are independent, and a stencil keeps the column's own values in registers.
template <int E, int H> constexpr int kColumns = (E + 2 * H) * (E + 2 * H);
template <int E, int H> constexpr int kCube = kColumns<E, H> * (E + 2 * H);
// Threads per CTA: one column each at the widest halo.
template <int E> constexpr int kTileThreads = E == 16 ? 416 : (E == 8 ? 160 : 64);

template <int E>
struct Column {
  long lo, mid, hi, plane;   // of the cells below, in and above the tile

  // (x, y): offsets from the tile's origin
  __device__ __forceinline__ Column(int n, const int* s_nb, const Tile<E>& w, int x, int y) {
    plane = (long)n * n;
    mid = cell_at(n, s_nb, w.x + x, w.y + y, w.z);
    lo = w.z == 0 ? cell_at(n, s_nb, w.x + x, w.y + y, -1) + plane : mid;
    hi = w.z + E == n ? cell_at(n, s_nb, w.x + x, w.y + y, n) - E * plane : mid;
  }
  __device__ __forceinline__ long at(int z) const { return (z < 0 ? lo : (z < E ? mid : hi)) + z * plane; }
};

template <int E, int H>
__device__ __forceinline__ void column_xy(int c, int& x, int& y) {
  x = c % (E + 2 * H) - H;
  y = c / (E + 2 * H) - H;
}
template <int E, int H>
__device__ __forceinline__ int cube_at(int x, int y, int z) {
  constexpr int W = E + 2 * H;
  return ((z + H) * W + (y + H)) * W + x + H;
}

// The neighbour sum of the cell at p, its column's neighbours in registers.
template <typename T, int W>
__device__ __forceinline__ T cross_sum(const T* p, T below, T above) {
  return ((((p[-1] + p[1]) + p[-W]) + p[W]) + below) + above;
}

// Where the restricted residual goes: the blocks of the next level ([B][(n/2)^3]),
// or, leaf given, one periodic array of Mg cells per edge.
struct Coarse {
  const int4* leaf;
  int Mg;
};
__device__ __forceinline__ long coarse_at(const Coarse& c, int nc, int b, int X, int Y, int Z) {
  if (c.leaf) {
    const int4 lf = c.leaf[b];
    return gidx(lf.y * nc + X, lf.z * nc + Y, lf.w * nc + Z, c.Mg);
  }
  return (((long)b * nc + Z) * nc + Y) * nc + X;
}

// Mean of the 8 children of each coarse cell of the tile, in (dz, dy, dx)
// order; r: residuals in a cube with halo H.
template <typename T, int E, int H>
__device__ __forceinline__ void restrict_tile(const T* r, const TileLevel& L, const Tile<E>& w, const Coarse& to,
                                              T* fc) {
  constexpr int W = E + 2 * H, EC = E / 2;
  for (int i = threadIdx.x; i < EC * EC * EC; i += kTileThreads<E>) {
    const int X = i % EC, Y = (i / EC) % EC, Z = i / (EC * EC);
    const T* p = r + cube_at<E, H>(2 * X, 2 * Y, 2 * Z);
    T s = p[0];
    s = s + p[1];
    s = s + p[W];
    s = s + p[W + 1];
    s = s + p[W * W];
    s = s + p[W * W + 1];
    s = s + p[W * W + W];
    s = s + p[W * W + W + 1];
    fc[coarse_at(to, L.n / 2, w.b, w.x / 2 + X, w.y / 2 + Y, w.z / 2 + Z)] = s * T(0.125);
  }
}

// Down leg of a cycle in float32: two sweeps from zero, the residual and its
// restriction, reading f once and writing phi once.
template <typename T, int E>
__global__ void __launch_bounds__(kTileThreads<E>)
tile_down_kernel(TileLevel L, const T* __restrict__ f, T* __restrict__ phi, Coarse to, T* __restrict__ fc, T h2,
                 T ih2) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  T* sF = reinterpret_cast<T*>(tile_raw);         // f, halo 2; then the residuals of the tile
  T* sP = sF + kCube<E, 2>;                        // phi after two sweeps, halo 1
  __shared__ int s_nb[27];
  const Tile<E> w = tile_of<E>(L, s_nb);
  constexpr int W2 = E + 4, W1 = E + 2;
  int x, y;
  for (int c = threadIdx.x; c < kColumns<E, 2>; c += kTileThreads<E>) {
    column_xy<E, 2>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
#pragma unroll
    for (int z = -2; z < E + 2; ++z) sF[(z + 2) * W2 * W2 + c] = f[col.at(z)];
  }
  __syncthreads();
  for (int c = threadIdx.x; c < kColumns<E, 1>; c += kTileThreads<E>) {
    column_xy<E, 1>(c, x, y);
    const T* p = sF + cube_at<E, 2>(x, y, -1);
    T g = p[0];
    T below = relax_zero(p[-W2 * W2], h2), own = relax_zero(g, h2);
#pragma unroll
    for (int z = -1; z < E + 1; ++z, p += W2 * W2) {
      const T gn = p[W2 * W2], above = relax_zero(gn, h2);
      const T s = ((((relax_zero(p[-1], h2) + relax_zero(p[1], h2)) + relax_zero(p[-W2], h2)) +
                    relax_zero(p[W2], h2)) + below) + above;
      sP[(z + 1) * W1 * W1 + c] = relax(own, s, g, h2);
      below = own;
      own = above;
      g = gn;
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < kColumns<E, 0>; c += kTileThreads<E>) {
    column_xy<E, 0>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
    const T* p = sP + cube_at<E, 1>(x, y, 0);
    T* q = sF + cube_at<E, 2>(x, y, 0);
    T below = p[-W1 * W1], own = p[0];
#pragma unroll
    for (int z = 0; z < E; ++z, p += W1 * W1, q += W2 * W2) {
      const T above = p[W1 * W1];
      phi[col.at(z)] = own;
      *q = residual_of(own, cross_sum<T, W1>(p, below, above), *q, ih2);
      below = own;
      own = above;
    }
  }
  __syncthreads();
  restrict_tile<T, E, 2>(sF, L, w, to, fc);
}

// The coarse error around a tile (halo 2 in coarse cells) into shared memory:
// from the next level's blocks, or from one periodic array of Mg cells per edge.
template <typename T, int E>
__device__ __forceinline__ void load_coarse(const TileLevel& L, const Tile<E>& w, const int* s_nb, const Coarse& from,
                                            const T* __restrict__ ec, T* sC) {
  constexpr int EC = E / 2, WC = EC + 4;
  const int nc = L.n / 2;
  for (int i = threadIdx.x; i < kCube<EC, 2>; i += kTileThreads<E>) {
    int x = i % WC - 2, y = (i / WC) % WC - 2, z = i / (WC * WC) - 2;
    x += w.x / 2;
    y += w.y / 2;
    z += w.z / 2;
    if (from.leaf) {
      const int4 lf = from.leaf[w.b];
      const int M = from.Mg;   // >= 2: an offset of two cells wraps at most once
      sC[i] = ec[gidx(wrapm(lf.y * nc + x, M), wrapm(lf.z * nc + y, M), wrapm(lf.w * nc + z, M), M)];
    } else {
      sC[i] = ec[cell_at(nc, s_nb, x, y, z)];
    }
  }
}

// Trilinear interpolation of the coarse error to the fine cells of the tile and
// its halo of H cells, one axis at a time, so that each one-axis value is formed
// once (2 instructions) instead of once per fine cell that uses it (14 a cell):
// along x for the coarse rows into shared memory, along y for the coarse planes
// into a column's registers, along z as the column is walked.
template <int E, int H> constexpr int kInterpX = (E + 2 * H) * (E / 2 + 4) * (E / 2 + 4);

template <typename T, int E, int H>
__device__ __forceinline__ void interpolate_x(const T* sC, T* sX) {
  constexpr int W = E + 2 * H, WC = E / 2 + 4;
  for (int i = threadIdx.x; i < kInterpX<E, H>; i += kTileThreads<E>) {
    const int x = i % W - H, row = i / W;
    const T* p = sC + row * WC + (x >> 1) + 2;   // arithmetic shift: floor for the halo
    sX[i] = quarter(p[0], p[(x & 1) ? 1 : -1]);
  }
}
// The fine values of the column (x, y) from below the tile up: out(z, value).
template <typename T, int E, int H, typename Out>
__device__ __forceinline__ void interpolate_column(const T* sX, int x, int y, Out out) {
  constexpr int W = E + 2 * H, WC = E / 2 + 4;
  const T* p = sX + ((y >> 1) + 2) * W + x + H;
  const int dy = (y & 1) ? W : -W;
  T v[WC];
#pragma unroll
  for (int k = 0; k < WC; ++k) v[k] = quarter(p[k * WC * W], p[k * WC * W + dy]);
#pragma unroll
  for (int z = -H; z < E + H; ++z) {
    const int k = (z + 4) / 2;   // floor(z / 2) + 2
    out(z, quarter(v[k], v[(z & 1) ? k + 1 : k - 1]));
  }
}

// Up leg in float32: the interpolated coarse error added to phi, then two
// sweeps.  OUT: 0 the result to out; on the finest level of a mixed-precision
// cycle it goes straight to the float64 potential, 1 added, 2 as its first value.
template <typename T, int E, int OUT>
__global__ void __launch_bounds__(kTileThreads<E>)
tile_up_kernel(TileLevel L, const T* __restrict__ f, const T* __restrict__ phi, Coarse from,
               const T* __restrict__ ec, T* __restrict__ out, double* __restrict__ phi64, T h2) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  T* sQ = reinterpret_cast<T*>(tile_raw);         // phi plus the interpolated error, halo 2
  T* sC = sQ + kCube<E, 2>;                        // the coarse error, halo 2
  T* sX = sC + kCube<E / 2, 2>;                    // its interpolation along x
  T* sR = sC;                                      // then the field after the first sweep, halo 1
  __shared__ int s_nb[27];
  const Tile<E> w = tile_of<E>(L, s_nb);
  constexpr int W2 = E + 4, W1 = E + 2;
  int x, y;
  load_coarse<T, E>(L, w, s_nb, from, ec, sC);
  __syncthreads();
  interpolate_x<T, E, 2>(sC, sX);
  __syncthreads();
  for (int c = threadIdx.x; c < kColumns<E, 2>; c += kTileThreads<E>) {
    column_xy<E, 2>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
    interpolate_column<T, E, 2>(sX, x, y, [&](int z, T e) { sQ[(z + 2) * W2 * W2 + c] = phi[col.at(z)] + e; });
  }
  __syncthreads();
  for (int c = threadIdx.x; c < kColumns<E, 1>; c += kTileThreads<E>) {
    column_xy<E, 1>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
    const T* p = sQ + cube_at<E, 2>(x, y, -1);
    T below = p[-W2 * W2], own = p[0];
#pragma unroll
    for (int z = -1; z < E + 1; ++z, p += W2 * W2) {
      const T above = p[W2 * W2];
      sR[(z + 1) * W1 * W1 + c] = relax(own, cross_sum<T, W2>(p, below, above), f[col.at(z)], h2);
      below = own;
      own = above;
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < kColumns<E, 0>; c += kTileThreads<E>) {
    column_xy<E, 0>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
    const T* p = sR + cube_at<E, 1>(x, y, 0);
    T below = p[-W1 * W1], own = p[0];
#pragma unroll
    for (int z = 0; z < E; ++z, p += W1 * W1) {
      const T above = p[W1 * W1];
      const long o = col.at(z);
      const T v = relax(own, cross_sum<T, W1>(p, below, above), f[o], h2);
      if (OUT == 0) out[o] = v;
      else if (OUT == 1) phi64[o] = phi64[o] + widen(v);
      else phi64[o] = widen(v);
      below = own;
      own = above;
    }
  }
}

// Float64 cycles are bound by the float64 pipe (1.6 lanes per SM and clock
// measured), so nothing is evaluated twice that costs more than a pointwise
// product: the legs are split into passes with a halo of one cell.
enum TilePass : int { kSmoothZero = 0, kSweep = 1, kUpSweep = 2, kRestrict = 3 };

// kSmoothZero: out = two sweeps from zero.  kSweep: out = one sweep of phi.
// kUpSweep: out = one sweep of phi plus the interpolated coarse error.
// kRestrict: fc = restricted residual of phi.
template <typename T, int E, int PASS>
__global__ void __launch_bounds__(kTileThreads<E>)
tile_pass_kernel(TileLevel L, const T* __restrict__ f, const T* __restrict__ phi, Coarse other,
                 const T* __restrict__ ec, T* __restrict__ out, T* __restrict__ fc, T h2, T ih2) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  T* sP = reinterpret_cast<T*>(tile_raw);          // the field being swept, halo 1
  T* sC = sP + kCube<E, 1>;                         // kUpSweep: the coarse error; kRestrict: the residuals
  T* sX = sC + kCube<E / 2, 2>;                     // kUpSweep: its interpolation along x
  __shared__ int s_nb[27];
  const Tile<E> w = tile_of<E>(L, s_nb);
  constexpr int W1 = E + 2;
  int x, y;
  if (PASS == kUpSweep) {
    load_coarse<T, E>(L, w, s_nb, other, ec, sC);
    __syncthreads();
    interpolate_x<T, E, 1>(sC, sX);
    __syncthreads();
  }
  for (int c = threadIdx.x; c < kColumns<E, 1>; c += kTileThreads<E>) {
    column_xy<E, 1>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
    T* q = sP + c + W1 * W1;
    if constexpr (PASS == kUpSweep) {
      interpolate_column<T, E, 1>(sX, x, y, [&](int z, T e) { q[z * W1 * W1] = phi[col.at(z)] + e; });
    } else {
#pragma unroll
      for (int z = -1; z < E + 1; ++z)
        q[z * W1 * W1] = PASS == kSmoothZero ? relax_zero(f[col.at(z)], h2) : phi[col.at(z)];
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < kColumns<E, 0>; c += kTileThreads<E>) {
    column_xy<E, 0>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
    const T* p = sP + cube_at<E, 1>(x, y, 0);
    T below = p[-W1 * W1], own = p[0];
#pragma unroll
    for (int z = 0; z < E; ++z, p += W1 * W1) {
      const T above = p[W1 * W1];
      const long o = col.at(z);
      const T s = cross_sum<T, W1>(p, below, above);
      if (PASS == kRestrict) sC[z * E * E + c] = residual_of(own, s, f[o], ih2);
      else out[o] = relax(own, s, f[o], h2);
      below = own;
      own = above;
    }
  }
  if (PASS == kRestrict) {
    __syncthreads();
    restrict_tile<T, E, 0>(sC, L, w, other, fc);
  }
}

// Float64 residual on the finest level: rounded to float32 (the right-hand side
// of a mixed-precision cycle), or its largest magnitude per CTA.
template <int E, bool MAX>
__global__ void __launch_bounds__(kTileThreads<E>)
tile_residual_kernel(TileLevel L, const double* __restrict__ f, const double* __restrict__ phi,
                     float* __restrict__ r, double* __restrict__ partial, double ih2) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  double* sP = reinterpret_cast<double*>(tile_raw);
  __shared__ int s_nb[27];
  const Tile<E> w = tile_of<E>(L, s_nb);
  constexpr int W1 = E + 2;
  int x, y;
  for (int c = threadIdx.x; c < kColumns<E, 1>; c += kTileThreads<E>) {
    column_xy<E, 1>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
#pragma unroll
    for (int z = -1; z < E + 1; ++z) sP[(z + 1) * W1 * W1 + c] = phi[col.at(z)];
  }
  __syncthreads();
  double worst = 0.0;
  for (int c = threadIdx.x; c < kColumns<E, 0>; c += kTileThreads<E>) {
    column_xy<E, 0>(c, x, y);
    const Column<E> col(L.n, s_nb, w, x, y);
    const double* p = sP + cube_at<E, 1>(x, y, 0);
    double below = p[-W1 * W1], own = p[0];
#pragma unroll
    for (int z = 0; z < E; ++z, p += W1 * W1) {
      const double above = p[W1 * W1];
      const long o = col.at(z);
      const double v = residual_of(own, cross_sum<double, W1>(p, below, above), f[o], ih2);
      if (MAX) worst = fabs(v) > worst ? fabs(v) : worst;
      else r[o] = (float)v;
      below = own;
      own = above;
    }
  }
  if (MAX) {
    for (int k = 16; k > 0; k >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, k));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sP[threadIdx.x >> 5] = worst;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 1; k < kTileThreads<E> / 32; ++k) worst = fmax(worst, sP[k]);
      partial[blockIdx.x] = worst;
    }
  }
}

// f without its mean, in float64 and, for a mixed-precision solve, rounded to
// float32: the residual of phi = 0 is f itself.
__global__ void shift_kernel(const double* __restrict__ src, double* __restrict__ dst, float* __restrict__ r,
                             long count, const double* shift) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const double v = src[i] - *shift;
  dst[i] = v;
  if (r) r[i] = (float)v;
}

// ---------------------------------------------------------------------------
// The bottom of the cycle in one CTA: every level from M cells per edge down,
// phi, a second field and f of each in shared memory.
__host__ __device__ inline long bottom_cells(int M) {
  long c = 0;
  for (int m = M;; m /= 2) {
    c += (long)m * m * m;
    if (m == 1 || m % 2 == 1) break;
  }
  return c;
}

template <typename T>
__device__ void bottom_sweep(const T* in, T* out, const T* f, int M, T h2) {
  for (int i = threadIdx.x; i < M * M * M; i += blockDim.x) {
    const int x = i % M, y = (i / M) % M, z = i / (M * M);
    out[i] = relax(in[i], nbsum(in, x, y, z, M), f[i], h2);
  }
  __syncthreads();
}

constexpr int kBottomThreads = 512;

template <typename T>
__global__ void __launch_bounds__(kBottomThreads)
bottom_kernel(const T* __restrict__ f, T* __restrict__ out, int M0, double h0) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  T* base = reinterpret_cast<T*>(tile_raw);
  for (int i = threadIdx.x; i < M0 * M0 * M0; i += blockDim.x) base[2 * M0 * M0 * M0 + i] = f[i];
  __syncthreads();
  // level of M cells: [phi, second field, f]; the coarser levels follow it
  int M = M0, depth = 0;
  double h = h0;
  T* lv = base;
  while (M > 1 && M % 2 == 0) {
    const int c = M * M * M, Mc = M / 2, cc = Mc * Mc * Mc;
    T *phi = lv, *tmp = lv + c, *g = lv + 2 * c, *gc = lv + 3 * c + 2 * cc;
    const T h2 = T(h * h), ih2 = T(1.0 / (h * h));
    for (int i = threadIdx.x; i < c; i += blockDim.x) tmp[i] = relax_zero(g[i], h2);
    __syncthreads();
    bottom_sweep(tmp, phi, g, M, h2);
    for (int i = threadIdx.x; i < c; i += blockDim.x) {
      const int x = i % M, y = (i / M) % M, z = i / (M * M);
      tmp[i] = residual_of(phi[i], nbsum(phi, x, y, z, M), g[i], ih2);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cc; i += blockDim.x) {
      const T* p = tmp + gidx(2 * (i % Mc), 2 * ((i / Mc) % Mc), 2 * (i / (Mc * Mc)), M);
      T s = p[0];
      s = s + p[1];
      s = s + p[M];
      s = s + p[M + 1];
      s = s + p[M * M];
      s = s + p[M * M + 1];
      s = s + p[M * M + M];
      s = s + p[M * M + M + 1];
      gc[i] = s * T(0.125);
    }
    __syncthreads();
    lv += 3 * c;
    M = Mc;
    h *= 2.0;
    ++depth;
  }
  {
    const int c = M * M * M;
    for (int i = threadIdx.x; i < c; i += blockDim.x) lv[i] = T(0);
    __syncthreads();
    if (M > 1) {   // odd coarsest grid (an even number of sweeps: the result is in phi)
      const T h2 = T(h * h);
      for (int k = 0; k < kCoarseSweeps; k += 2) {
        bottom_sweep(lv, lv + c, lv + 2 * c, M, h2);
        bottom_sweep(lv + c, lv, lv + 2 * c, M, h2);
      }
    }
  }
  while (depth > 0) {
    const int Mc = M;
    const T* ec = lv;
    M *= 2;
    h *= 0.5;
    --depth;
    const int c = M * M * M;
    lv -= 3 * c;
    T *phi = lv, *tmp = lv + c, *g = lv + 2 * c;
    const T h2 = T(h * h);
    for (int i = threadIdx.x; i < c; i += blockDim.x) {
      const int x = i % M, y = (i / M) % M, z = i / (M * M);
      phi[i] = phi[i] + prolonged(ec, x, y, z, Mc);
    }
    __syncthreads();
    bottom_sweep(phi, tmp, g, M, h2);
    bottom_sweep(tmp, phi, g, M, h2);
  }
  for (int i = threadIdx.x; i < M0 * M0 * M0; i += blockDim.x) out[i] = base[i];
}

unsigned blocks_for(long count) { return (unsigned)((count + 255) / 256); }

// How a level runs: on tiles, in the one-CTA bottom (with every level below it),
// or on the single-array kernels (an edge that is no multiple of 4, too large
// for the bottom).
enum LevelKind { kTiles, kBottom, kArray };

template <typename T>
struct Level {
  LevelKind kind;
  int n;             // cells per block edge, or per edge of the single array
  int blocks;
  const int* idx;    // neighbour blocks, null for a single array
  double h;
  T *phi, *tmp, *f;

  long cells() const { return (long)blocks * n * n * n; }
};

// Largest edge of a grid the one-CTA bottom takes.  Float32: 16 (16^3 cells and
// the levels below take 56 KB and ~10 us; two tile launches per level cost as
// much).  Float64: 10, one SM's float64 pipe (two lanes a clock) needs 13 us for
// 10^3 cells and 52 us for 16^3, where the launches of a tile level take ~10.
template <typename T> constexpr int kBottomMax = sizeof(T) == 4 ? 16 : 10;

// Tile edge of a level: 16 where that leaves at least two CTAs per SM, else 8, 4
// where the edge asks for it.
inline int tile_edge(int n, int blocks) {
  if (n % 16 == 0 && (long)blocks * (n / 16) * (n / 16) * (n / 16) >= 304) return 16;
  return n % 8 == 0 ? 8 : 4;
}

// Shared memory of the up leg: the float32 kernel reuses the interpolation's
// arrays for its second field.
template <typename T, int E>
constexpr size_t up_smem() {
  constexpr int H = sizeof(T) == 4 ? 2 : 1;
  constexpr int interp = kCube<E / 2, 2> + kInterpX<E, H>;
  constexpr int second = sizeof(T) == 4 ? kCube<E, 1> : 0;
  return sizeof(T) * (kCube<E, H> + (interp > second ? interp : second));
}

template <typename T>
struct Cycle {
  std::vector<Level<T>> lv;
  const int4* leaf;     // of the mesh: where a block's cells lie in the first single array
  cudaStream_t s;

  // ---- single arrays, one pass per launch
  void sweeps(Level<T>& L, int count) {
    for (int k = 0; k < count; ++k) {
      jacobi_kernel<T><<<grid_zc(L.n), kBlock3, 0, s>>>(L.phi, L.tmp, L.f, L.n, T(L.h * L.h));
      std::swap(L.phi, L.tmp);
    }
  }
  void array_level(int l) {
    Level<T>& L = lv[l];
    fill_kernel<T><<<blocks_for(L.cells()), 256, 0, s>>>(L.phi, L.cells(), T(0));
    if (L.n % 2 == 1) {
      sweeps(L, kCoarseSweeps);
      return;
    }
    sweeps(L, kNu);
    Level<T>& C = lv[l + 1];
    residual_restrict_kernel<T><<<grid3(C.n), kBlock3, 0, s>>>(L.phi, L.f, C.f, L.n, T(1.0 / (L.h * L.h)));
    solve(l + 1);
    prolong_add_kernel<T><<<grid3(L.n), kBlock3, 0, s>>>(C.phi, L.phi, L.n);
    sweeps(L, kNu);
  }

  // ---- tiles
  template <int E>
  void tile_level(int l, double* phi64, bool add, bool zero) {
    Level<T>& L = lv[l];
    Level<T>& C = lv[l + 1];
    const unsigned grid = (unsigned)((long)L.blocks * (L.n / E) * (L.n / E) * (L.n / E));
    constexpr int TH = kTileThreads<E>;
    const TileLevel t{L.n, L.idx};
    const Coarse c{L.idx && !C.idx ? leaf : nullptr, C.n};   // blocks above a single array
    const T h2 = T(L.h * L.h), ih2 = T(1.0 / (L.h * L.h));
    if constexpr (sizeof(T) == 4) {
      constexpr size_t down = sizeof(T) * (kCube<E, 2> + kCube<E, 1>);
      constexpr size_t up = up_smem<T, E>();
      tile_down_kernel<T, E><<<grid, TH, down, s>>>(t, L.f, L.phi, c, C.f, h2, ih2);
      solve(l + 1);
      if (!phi64) {
        tile_up_kernel<T, E, 0><<<grid, TH, up, s>>>(t, L.f, L.phi, c, C.phi, L.tmp, nullptr, h2);
        std::swap(L.phi, L.tmp);
      } else if (add) {
        tile_up_kernel<T, E, 1><<<grid, TH, up, s>>>(t, L.f, L.phi, c, C.phi, nullptr, phi64, h2);
      } else {
        tile_up_kernel<T, E, 2><<<grid, TH, up, s>>>(t, L.f, L.phi, c, C.phi, nullptr, phi64, h2);
      }
    } else {
      constexpr size_t one = sizeof(T) * kCube<E, 1>;
      constexpr size_t up = up_smem<T, E>(), rr = one + sizeof(T) * E * E * E;
      if (zero) {
        tile_pass_kernel<T, E, kSmoothZero><<<grid, TH, one, s>>>(t, L.f, nullptr, c, nullptr, L.phi, nullptr, h2,
                                                                  ih2);
      } else {
        tile_pass_kernel<T, E, kSweep><<<grid, TH, one, s>>>(t, L.f, L.phi, c, nullptr, L.tmp, nullptr, h2, ih2);
        tile_pass_kernel<T, E, kSweep><<<grid, TH, one, s>>>(t, L.f, L.tmp, c, nullptr, L.phi, nullptr, h2, ih2);
      }
      tile_pass_kernel<T, E, kRestrict><<<grid, TH, rr, s>>>(t, L.f, L.phi, c, nullptr, nullptr, C.f, h2, ih2);
      solve(l + 1);
      tile_pass_kernel<T, E, kUpSweep><<<grid, TH, up, s>>>(t, L.f, L.phi, c, C.phi, L.tmp, nullptr, h2, ih2);
      tile_pass_kernel<T, E, kSweep><<<grid, TH, one, s>>>(t, L.f, L.tmp, c, nullptr, L.phi, nullptr, h2, ih2);
    }
  }

  // One V-cycle on level l, its result in lv[l].phi, or (finest level of a
  // mixed-precision cycle) in, or added to, phi64.  It starts from zero, or
  // (finest level of a float64 cycle) from lv[l].phi.
  void solve(int l, double* phi64 = nullptr, bool add = false, bool zero = true) {
    Level<T>& L = lv[l];
    if (L.kind == kBottom) {
      const size_t sh = sizeof(T) * 3 * bottom_cells(L.n);
      bottom_kernel<T><<<1, kBottomThreads, sh, s>>>(L.f, L.phi, L.n, L.h);
    } else if (L.kind == kArray) {
      array_level(l);
    } else {
      switch (tile_edge(L.n, L.blocks)) {
        case 16: tile_level<16>(l, phi64, add, zero); break;
        case 8: tile_level<8>(l, phi64, add, zero); break;
        default: tile_level<4>(l, phi64, add, zero); break;
      }
    }
  }
};

}  // namespace

// Scratch of the solver for one mesh: the level arrays (float64 and, for
// mixed precision, float32), the reduction partials.  Allocated on the
// first solve of each kind, freed with the mesh.
struct PoissonScratch {
  std::vector<void*> d64, d32;
  double* f64 = nullptr;   // mixed precision: f without its mean
  double* red = nullptr;   // 1024 partials + 2 scalars
  double* top = nullptr;   // residual maxima per tile of the finest level
  ~PoissonScratch() {
    for (void* p : d64) cudaFree(p);
    for (void* p : d32) cudaFree(p);
    if (f64) cudaFree(f64);
    if (red) cudaFree(red);
    if (top) cudaFree(top);
  }
};

void poisson_free(PoissonScratch* p) { delete p; }

namespace {

// Three arrays per level (cells per array given), for the levels not yet
// allocated.
cudaError_t alloc_levels(std::vector<void*>& bufs, const std::vector<long>& cells, size_t elem) {
  for (size_t l = bufs.size() / 3; l < cells.size(); ++l)
    for (int k = 0; k < 3; ++k) {
      void* d = nullptr;
      cudaError_t e = cudaMalloc(&d, elem * (size_t)cells[l]);
      if (e != cudaSuccess) {
        for (; k > 0; --k) {   // a level has all three arrays or none
          cudaFree(bufs.back());
          bufs.pop_back();
        }
        return e;
      }
      bufs.push_back(d);
    }
  return cudaSuccess;
}

// The level structure: block levels n, n/2, ..., 4, then single arrays of
// M = root 2^L 2 cells per axis, halved while even and above 1.
template <typename T>
std::vector<Level<T>> plan_levels(const DevMesh& m, int Mblocks, double h) {
  std::vector<Level<T>> lv;
  for (int nl = m.n; nl >= 4; nl /= 2, h *= 2.0) lv.push_back(Level<T>{kTiles, nl, m.B, m.idx, h, nullptr, nullptr, nullptr});
  for (int Ml = Mblocks * 2;; Ml /= 2, h *= 2.0) {
    const LevelKind k = Ml <= kBottomMax<T> ? kBottom : (Ml % 4 == 0 ? kTiles : kArray);
    lv.push_back(Level<T>{k, Ml, 1, nullptr, h, nullptr, nullptr, nullptr});
    if (k == kBottom || Ml % 2 == 1) break;
  }
  return lv;
}

template <typename T>
cudaError_t make_cycle(Cycle<T>& C, const DevMesh& m, int Mblocks, double h, std::vector<void*>& bufs,
                       cudaStream_t s) {
  C.lv = plan_levels<T>(m, Mblocks, h);
  C.leaf = m.leaf;
  C.s = s;
  std::vector<long> cells;
  for (const Level<T>& L : C.lv) cells.push_back(L.cells());
  const cudaError_t e = alloc_levels(bufs, cells, sizeof(T));
  if (e != cudaSuccess) return e;
  for (size_t k = 0; k < C.lv.size(); ++k) {
    C.lv[k].phi = static_cast<T*>(bufs[3 * k]);
    C.lv[k].tmp = static_cast<T*>(bufs[3 * k + 1]);
    C.lv[k].f = static_cast<T*>(bufs[3 * k + 2]);
  }
  return cudaSuccess;
}

template <typename K>
void allow_smem(K kernel, size_t bytes) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int E>
void prepare_tiles() {
  constexpr size_t f2 = sizeof(float) * (kCube<E, 2> + kCube<E, 1>), fu = up_smem<float, E>();
  allow_smem(tile_down_kernel<float, E>, f2);
  allow_smem(tile_up_kernel<float, E, 0>, fu);
  allow_smem(tile_up_kernel<float, E, 1>, fu);
  allow_smem(tile_up_kernel<float, E, 2>, fu);
  constexpr size_t d1 = sizeof(double) * kCube<E, 1>;
  allow_smem(tile_pass_kernel<double, E, kSmoothZero>, d1);
  allow_smem(tile_pass_kernel<double, E, kSweep>, d1);
  allow_smem(tile_pass_kernel<double, E, kUpSweep>, up_smem<double, E>());
  allow_smem(tile_pass_kernel<double, E, kRestrict>, d1 + sizeof(double) * E * E * E);
  allow_smem(tile_residual_kernel<E, false>, d1);
  allow_smem(tile_residual_kernel<E, true>, d1);
}

void prepare_poisson() {
  prepare_tiles<16>();
  prepare_tiles<8>();
  prepare_tiles<4>();
  allow_smem(bottom_kernel<float>, sizeof(float) * 3 * bottom_cells(kBottomMax<float>));
  allow_smem(bottom_kernel<double>, sizeof(double) * 3 * bottom_cells(kBottomMax<double>));
}

// mean of a compact array (count doubles) into *out
void mean_of(const double* a, long count, double* red, double* out, cudaStream_t s) {
  reduce_kernel<<<1024, kRedThreads, 0, s>>>(a, count, red);
  fold_kernel<<<1, kRedThreads, 0, s>>>(red, 1024, 0, 1.0 / (double)count, out);
}

template <int E>
void residual_pass(const DevMesh& m, const double* f, const double* phi, float* r, double* partial, double ih2,
                   cudaStream_t s) {
  const unsigned grid = (unsigned)((long)m.B * (m.n / E) * (m.n / E) * (m.n / E));
  const TileLevel t{m.n, m.idx};
  constexpr size_t sh = sizeof(double) * kCube<E, 1>;
  if (r) tile_residual_kernel<E, false><<<grid, kTileThreads<E>, sh, s>>>(t, f, phi, r, nullptr, ih2);
  else tile_residual_kernel<E, true><<<grid, kTileThreads<E>, sh, s>>>(t, f, phi, nullptr, partial, ih2);
}

// The finest level's float64 residual: rounded into r, or its maxima per tile.
void residual(const DevMesh& m, const double* f, const double* phi, float* r, double* partial, double ih2,
              cudaStream_t s) {
  if (tile_edge(m.n, m.B) == 16) residual_pass<16>(m, f, phi, r, partial, ih2, s);
  else residual_pass<8>(m, f, phi, r, partial, ih2, s);
}

}  // namespace

cudaError_t poisson_solve(PoissonScratch** scratch, const DevMesh& m, int M, double h, const double* f_leaves,
                          double* phi_leaves, int cycles, int inner, double* resid_host, cudaStream_t s) {
  const int n = m.n, B = m.B;
  static OncePerDevice once;
  int dev = 0;
  const cudaError_t found = cudaGetDevice(&dev);
  if (found != cudaSuccess) return found;
  once.run(dev, prepare_poisson);
  if (!*scratch) *scratch = new PoissonScratch();
  PoissonScratch* S = *scratch;
  const long nl = (long)B * n * n * n;
  Cycle<double> C64;
  Cycle<float> C32;
  cudaError_t e = inner == 8 ? make_cycle(C64, m, M / n, h, S->d64, s) : make_cycle(C32, m, M / n, h, S->d32, s);
  if (e == cudaSuccess && inner == 4 && !S->f64) e = cudaMalloc(&S->f64, sizeof(double) * (size_t)nl);
  if (e == cudaSuccess && !S->red) e = cudaMalloc(&S->red, sizeof(double) * (1024 + 2));
  const int edge = tile_edge(n, B);
  const long tiles = (long)B * (n / edge) * (n / edge) * (n / edge);
  if (e == cudaSuccess && resid_host && !S->top) e = cudaMalloc(&S->top, sizeof(double) * (size_t)tiles);
  if (e != cudaSuccess) return e;
  double* scalar = S->red + 1024;
  const double ih2 = 1.0 / (h * h);
  // f without its mean; phi starts at 0
  double* f0 = inner == 8 ? C64.lv[0].f : S->f64;
  mean_of(f_leaves, nl, S->red, scalar, s);
  shift_kernel<<<blocks_for(nl), 256, 0, s>>>(f_leaves, f0, inner == 4 ? C32.lv[0].f : nullptr, nl, scalar);
  double* phi = inner == 4 ? phi_leaves : nullptr;
  for (int k = 0; k < cycles; ++k) {
    if (inner == 4) {
      if (k > 0) residual(m, f0, phi, C32.lv[0].f, nullptr, ih2, s);   // of phi = 0: f, already there
      C32.solve(0, phi, k > 0);
    } else {
      C64.solve(0, nullptr, false, k == 0);
      phi = C64.lv[0].phi;
    }
    if (resid_host) {
      residual(m, f0, phi, nullptr, S->top, ih2, s);
      fold_kernel<<<1, kRedThreads, 0, s>>>(S->top, tiles, 1, 1.0, scalar + 1);
      e = cudaMemcpyAsync(resid_host + k, scalar + 1, sizeof(double), cudaMemcpyDeviceToHost, s);
      if (e != cudaSuccess) return e;
    }
  }
  mean_of(phi, nl, S->red, scalar, s);
  if (inner == 8) shift_kernel<<<blocks_for(nl), 256, 0, s>>>(phi, phi_leaves, nullptr, nl, scalar);
  else add_kernel<<<blocks_for(nl), 256, 0, s>>>(phi_leaves, nl, scalar, 1.0);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (resid_host) e = cudaStreamSynchronize(s);
  return e;
}

}  // namespace cello
