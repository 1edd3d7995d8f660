// Adjoint of one directional PPM sweep and of the periodic same-level ghost
// copy, with dt held fixed.  Included by the per-precision translation units.
#pragma once

#include "adjoint.cuh"
#include "cello_internal.h"

namespace cello {

// ---------------------------------------------------------------------
// Adjoint sweep.  The forward sweep maps U to U' with
//   U'_j = U_j - (dt/dx) (F_{j+1/2} - F_{j-1/2})  for updated cells j.
// Given lam' (adjoint of U'), the flux at interface c|c+1 gets the adjoint
// mu_c = (dt/dx)(m_{c+1} lam'_{c+1} - m_c lam'_c), m = 1 on updated cells, and
// lam = lam' + (dF/dU)^T mu is the sweep in reverse.  One CTA item = P
// pencils, one thread per cell and pencil, the pencils of a cell in one warp;
// the sweep's phases run forward (primitives, slopes and shock detector,
// interface values, edge values and tracing) and then backward (Riemann
// problem, tracing and edge values, interface values, slopes and shock
// detector, primitives), each quantity and its adjoint evaluated once per cell
// or interface and handed to the neighbours through shared memory.
//
// The float64 kernel is bound by the float64 pipe (1.6 lanes per SM and clock
// measured).  Evaluating each interface's whole eight-cell stencil in its own
// thread ran every primitive, slope and edge value up to eight times: three
// steps of a gradient on 64 leaves of 16^3 took 99.9 ms; with reciprocals shared
// per divisor and the Newton reverse from the stored history 69.1 ms; each
// quantity once, as here, 38.2 ms; with the short float64 forms of ppm64.cuh 28.0 ms,
// of which the float64 forward sweeps then lost another 1.3 ms.
// The cells without an edge state (three at each end) come last in the CTA, so
// that they leave whole warps idle rather than lanes (26.7 -> 26.4 ms; 8^3 blocks 7.3 ->
// 7.15 ms); P: see adj_pencils.
// ---------------------------------------------------------------------
template <typename T, int NB>
constexpr size_t adjoint_smem() {
  constexpr int A = (NB + 2 * kGhosts) * adj_pencils(NB, (int)sizeof(T));
  return (sizeof(T) * 33 + sizeof(int)) * A;
}

template <typename T, int NB>
__global__ void __launch_bounds__((NB + 8) * adj_pencils(NB, (int)sizeof(T)))
adjoint_sweep_kernel(DevMesh m, AdjSweepParams prm) {
  constexpr int G = kGhosts, N = NB + 2 * G, P = adj_pencils(NB, (int)sizeof(T)), A = N * P;
  constexpr long SLAB = (long)N * N * N;
  constexpr bool k64 = std::is_same<T, double>::value;   // ppm64.cuh: the same values
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sW = reinterpret_cast<T*>(smem_raw);   // primitives
  T* sLam = sW + 5 * A;                      // lam', then lam
  T* sD = sLam + 5 * A;                      // slopes, then adjoints they give cell j-1
  T* sI = sD + 5 * A;                        // interface values j+1/2, then slope adjoints for cell j+1
  T* sL = sI + 5 * A;                        // left edge states, their adjoints, adjoints of interface j-1/2
  T* sR = sL + 5 * A;                        // right edge states, their adjoints, adjoints of interface j+1/2
  T* sFT = sR + 5 * A;                       // shock detector, then its adjoint for p of cells j+-1
  T* sF2 = sFT + A;                          // its adjoint for p of cells j+-2
  T* sFb = sF2 + A;                          // adjoint of the flattening coefficient
  int* sSel = reinterpret_cast<int*>(sFb + A);   // which detector it was taken from (-1, 0, 1)

  const Gas<T> gs = Gas<T>::make(m.gamma);
  const T* U = static_cast<const T*>(prm.U);
  T* lam = static_cast<T*>(prm.lam);
  const int axis = prm.axis;
  const int cA = prm.a1 - prm.a0, cB = prm.b1 - prm.b0;
  const long sAx = axis == 0 ? 1 : (axis == 1 ? N : (long)N * N);
  const long sTA = axis == 2 ? N : (long)N * N;
  const long sTB = axis == 0 ? N : 1;
  int comp[5];
  comp[0] = 0; comp[1] = 1 + axis; comp[4] = 4;
  comp[2] = axis == 0 ? 2 : 1;
  comp[3] = axis == 2 ? 2 : 3;
  const int t = threadIdx.x;
  // cell and pencil moved to and from memory (along x first on the x sweep), and computed
  const int mc = axis == 0 ? t % N : t / P, mp = axis == 0 ? t / N : t % P;
  // cells from the first one with an edge state on, the three before it last: those
  // without one (three at each end) are whole warps
  const int j = t / P + 3 < N ? t / P + 3 : t / P + 3 - N, p = t % P, at = j * P + p;
  __shared__ T s_dtdx[16];
  if (t <= m.max_level) s_dtdx[t] = T(*prm.dt / ldexp(m.dx0, -t));
  __syncthreads();

  for (int item = blockIdx.x; item < prm.n_items; item += gridDim.x) {
    const int leaf = prm.leaf0 + item / prm.tiles_per_leaf;
    const int tile = item % prm.tiles_per_leaf;
    const T dtdx = s_dtdx[m.leaf[leaf].x];
    const int mq = tile * P + mp;
    const bool moves = mq < cA * cB;
    const int ma = prm.a0 + (moves ? mq / cB : 0), mb = prm.b0 + (moves ? mq % cB : 0);
    const long off = (long)leaf * 5 * SLAB + ma * sTA + mb * sTB + mc * sAx;
    {
      T Us[5], W[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) Us[k] = moves ? U[off + comp[k] * SLAB] : T(1);
      if constexpr (k64) q64::primitives<5>(Us, gs, W);
      else to_primitive(Us, gs, W);
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        sW[k * A + mc * P + mp] = W[k];
        sLam[k * A + mc * P + mp] = moves ? lam[off + comp[k] * SLAB] : T(0);
      }
    }
    __syncthreads();
    // ---- forward: slopes and shock detector, interface values, edge states
    T ft = T(0);
    if (j >= 2 && j <= N - 3) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const T* a = sW + k * A + at;
        if constexpr (k64) sD[k * A + at] = q64::slope(a[-P], a[0], a[P]);
        else sD[k * A + at] = limited_slope(a[-P], a[0], a[P]);
      }
      const T *pr = sW + 4 * A + at, *un = sW + A + at;
      if constexpr (k64) ft = q64::detector(pr[-2 * P], pr[-P], pr[P], pr[2 * P], un[-P], un[P]);
      else ft = flatten_tilde(pr[-2 * P], pr[-P], pr[P], pr[2 * P], un[-P], un[P]);
    }
    sFT[at] = ft;
    __syncthreads();
    if (j >= 2 && j <= N - 4) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const T a0 = sW[k * A + at], a1 = sW[k * A + at + P], d0 = sD[k * A + at], d1 = sD[k * A + at + P];
        if constexpr (k64) sI[k * A + at] = q64::interface_val(a0, a1, d0, d1);
        else sI[k * A + at] = interface_value(a0, a1, d0, d1);
      }
    }
    __syncthreads();
    const bool traced = j >= 3 && j <= N - 4;
    T f = T(0), aL[5], aR[5];
    int sel = 0;
    if (traced) {
      const T* pr = sW + 4 * A + at;
      const T s = pr[P] - pr[-P];
      const T fm = sFT[at - P], fp = sFT[at + P];
      f = ft;
      if (s > T(0)) {
        if (!(ft > fm)) { f = fm; sel = -1; }
      } else if (s < T(0)) {
        if (!(ft > fp)) { f = fp; sel = 1; }
      }
      T W[5], Wm[5], Wp[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        W[k] = sW[k * A + at];
        aL[k] = sI[k * A + at - P];
        aR[k] = sI[k * A + at];
        if constexpr (!k64) flatten_monotone(W[k], f, aL[k], aR[k]);
      }
      if constexpr (k64) q64::edge_states<5>(W, f, aL, aR, dtdx, gs, Wm, Wp);
      else trace(W, aL, aR, dtdx, gs, Wm, Wp);
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        sL[k * A + at] = Wm[k];
        sR[k * A + at] = Wp[k];
      }
    }
    __syncthreads();
    // ---- backward: the Riemann problem at j+1/2 turns the states beside it into their adjoints
    if (j >= 3 && j <= N - 5) {
      const T m0 = (j >= G) ? T(1) : T(0);
      const T m1 = (j + 1 < G + NB) ? T(1) : T(0);
      T mu[5], Lb[5], Rb[5];
      bool any = false;
#pragma unroll
      for (int k = 0; k < 5; ++k) mu[k] = dtdx * (m1 * sLam[k * A + at + P] - m0 * sLam[k * A + at]);
      if (prm.regb && (j == G - 1 || j == G + NB - 1)) {   // flux kept for the coarse-fine correction
        const int q = tile * P + p;
        if (q < cA * cB) {
          const int ca = prm.a0 + q / cB, cb = prm.b0 + q % cB;
          if (ca >= G && ca < G + NB && cb >= G && cb < G + NB) {
            const int slot = m.face_slot[leaf * 6 + 2 * axis + (j == G - 1 ? 0 : 1)];
            if (slot >= 0) {
              const double* r = prm.regb + (long)slot * 5 * NB * NB + (ca - G) * NB + (cb - G);
#pragma unroll
              for (int k = 0; k < 5; ++k) mu[k] += T(r[(long)comp[k] * NB * NB]);
            }
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        any = any || (mu[k] != T(0));
        Lb[k] = Rb[k] = T(0);
      }
      if (any) {
        T L[5], R[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          L[k] = sR[k * A + at];
          R[k] = sL[k * A + at + P];
        }
        riemann_flux_bwd(L, R, gs, mu, Lb, Rb);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        sR[k * A + at] = Lb[k];
        sL[k * A + at + P] = Rb[k];
      }
    }
    // the first traced cell has no interface on its left, the last none on its right
    if (j == 3)
#pragma unroll
      for (int k = 0; k < 5; ++k) sL[k * A + at] = T(0);
    if (j == N - 4)
#pragma unroll
      for (int k = 0; k < 5; ++k) sR[k * A + at] = T(0);
    __syncthreads();
    // ---- tracing and the edge values
    T Wb[5] = {0, 0, 0, 0, 0};
    T fb = T(0);
    if (traced) {
      T Wmb[5], Wpb[5];
      bool any = false;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        Wmb[k] = sL[k * A + at];
        Wpb[k] = sR[k * A + at];
        any = any || Wmb[k] != T(0) || Wpb[k] != T(0);
      }
      if (any) {
        T W[5], aLb[5] = {0, 0, 0, 0, 0}, aRb[5] = {0, 0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < 5; ++k) W[k] = sW[k * A + at];
        trace_bwd(W, aL, aR, dtdx, gs, Wmb, Wpb, Wb, aLb, aRb);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          T lb = T(0), rb = T(0);
          flatten_monotone_bwd(W[k], f, sI[k * A + at - P], sI[k * A + at], aLb[k], aRb[k], Wb[k], fb, lb, rb);
          sL[k * A + at] = lb;
          sR[k * A + at] = rb;
        }
      }
    } else {
#pragma unroll
      for (int k = 0; k < 5; ++k) sL[k * A + at] = sR[k * A + at] = T(0);
    }
    sFb[at] = fb;
    sSel[at] = sel;
    __syncthreads();
    // ---- interface values, slopes, shock detector: cell j's share, the neighbours' left in shared memory
    T d1 = T(0), d2 = T(0);
    if (j >= 2 && j <= N - 3) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const T im = sR[k * A + at - P] + sL[k * A + at], ip = sR[k * A + at] + sL[k * A + at + P];
        const T* a = sW + k * A + at;
        T lo = T(0), own = T(0.5) * (im + ip), hi = T(0);
        limited_slope_bwd(a[-P], a[0], a[P], (ip - im) * T(1.0 / 6.0), lo, own, hi);
        Wb[k] += own;
        sD[k * A + at] = lo;
        sI[k * A + at] = hi;
      }
      T ftb = (sSel[at] == 0) ? fb : T(0);
      if (sSel[at - P] == 1) ftb += sFb[at - P];
      if (sSel[at + P] == -1) ftb += sFb[at + P];
      if (ftb != T(0)) {
        const T *pr = sW + 4 * A + at, *un = sW + A + at;
        T m2 = T(0), m1 = T(0);
        flatten_tilde_bwd(pr[-2 * P], pr[-P], pr[P], pr[2 * P], un[-P], un[P], ftb, m2, m1, d1, d2);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 5; ++k) sD[k * A + at] = sI[k * A + at] = T(0);
    }
    sFT[at] = d1;
    sF2[at] = d2;
    __syncthreads();
    // ---- primitives
    {
      T W[5], Ub[5] = {0, 0, 0, 0, 0};
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        W[k] = sW[k * A + at];
        if (j >= 1) Wb[k] += sI[k * A + at - P];
        if (j <= N - 2) Wb[k] += sD[k * A + at + P];
      }
      if (j >= 1) Wb[4] += sFT[at - P];
      if (j <= N - 2) Wb[4] -= sFT[at + P];
      if (j >= 2) Wb[4] += sF2[at - 2 * P];
      if (j <= N - 3) Wb[4] -= sF2[at + 2 * P];
      to_primitive_bwd(W, gs, Wb, Ub);
#pragma unroll
      for (int k = 0; k < 5; ++k) sLam[k * A + at] += Ub[k];
    }
    __syncthreads();
    if (moves) {
#pragma unroll
      for (int k = 0; k < 5; ++k) lam[off + comp[k] * SLAB] = sLam[k * A + mc * P + mp];
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------
// Transposed periodic same-level ghost copy: every interior cell gathers the
// adjoints of the ghost cells copied from it (directions in table order),
// then all ghost adjoints are cleared.
// ---------------------------------------------------------------------
template <typename T, int NB>
__global__ void __launch_bounds__(256) adjoint_refresh_gather_kernel(DevMesh m, T* lam) {
  constexpr int G = kGhosts, N = NB + 2 * G;
  constexpr long SLAB = (long)N * N * N;
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long)m.B * NB * NB * NB) return;
  const int leaf = (int)(gid / (NB * NB * NB));
  const int i = (int)(gid % (NB * NB * NB));
  const int s[3] = {i % NB + G, (i / NB) % NB + G, i / (NB * NB) + G};
  T acc[5];
  const long own = (long)leaf * 5 * SLAB + ((long)s[2] * N + s[1]) * N + s[0];
#pragma unroll
  for (int f = 0; f < 5; ++f) acc[f] = lam[own + f * SLAB];
  for (int e = 0; e < 27; ++e) {
    if (e == 13) continue;
    const int d[3] = {e % 3 - 1, (e / 3) % 3 - 1, e / 9 - 1};
    int c[3];
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      c[a] = s[a] + d[a] * NB;
      ok = ok && c[a] >= 0 && c[a] < N;
    }
    if (!ok) continue;
    const int back = (-d[2] + 1) * 9 + (-d[1] + 1) * 3 + (-d[0] + 1);
    const int src = m.idx[leaf * 27 + back];   // the leaf whose ghost in direction d copies this cell
    const long o = (long)src * 5 * SLAB + ((long)c[2] * N + c[1]) * N + c[0];
#pragma unroll
    for (int f = 0; f < 5; ++f) acc[f] += lam[o + f * SLAB];
  }
#pragma unroll
  for (int f = 0; f < 5; ++f) lam[own + f * SLAB] = acc[f];
}

// ---------------------------------------------------------------------
// AMR transpose of the ghost refresh.  Each ghost cell's adjoint is added to
// the cells its forward value was made from, with the forward's weights:
// copy 1; restriction 0.125 on each of 8 cells; prolongation U_C + 0.25
// sum_d s_d D_d with D_d = minmod(U_C - U_m, U_p - U_C) differentiated along
// the branch the forward took (per field), the neighbour values U_m, U_p
// being copies, restrictions or injections of further cells.  Sources are
// leaf interiors, ghosts are only read, so atomic adds suffice.
// ---------------------------------------------------------------------
template <typename T, int NB>
__device__ __forceinline__ void add5(T* lam, int leaf, int x, int y, int z, const T w[5]) {
  constexpr int N = NB + 2 * kGhosts;
  constexpr long SLAB = (long)N * N * N;
  T* b = lam + (long)leaf * 5 * SLAB + ((long)z * N + y) * N + x;
#pragma unroll
  for (int f = 0; f < 5; ++f)
    if (w[f] != T(0)) atomicAdd(b + f * SLAB, w[f]);
}

template <typename T, int NB>
__device__ __forceinline__ void add_restrict8(T* lam, int leaf, int fx, int fy, int fz, const T w[5]) {
  T w8[5];
#pragma unroll
  for (int f = 0; f < 5; ++f) w8[f] = w[f] * T(0.125);
  for (int dz = 0; dz < 2; ++dz)
    for (int dy = 0; dy < 2; ++dy)
      for (int dx = 0; dx < 2; ++dx) add5<T, NB>(lam, leaf, fx + dx, fy + dy, fz + dz, w8);
}

// Adjoint of slope_neighbour: w onto the sources of that neighbour value.
template <typename T, int NB>
__device__ void slope_neighbour_bwd(const DevMesh& m, T* lam, int C, const int rc[3], int a, int side, const T w[5]) {
  constexpr int G = kGhosts, H = NB / 2;
  const int e = C * 27 + face_dir(a, side);
  const int8_t k = m.kind[e];
  if (k == kBoundary) {
    add5<T, NB>(lam, C, rc[0] + G, rc[1] + G, rc[2] + G, w);
    return;
  }
  int r2[3] = {rc[0], rc[1], rc[2]};
  r2[a] = side < 0 ? NB - 1 : 0;
  if (k == kSame) {
    add5<T, NB>(lam, m.idx[e], r2[0] + G, r2[1] + G, r2[2] + G, w);
  } else if (k == kFine) {
    const int o0 = r2[0] / H, o1 = r2[1] / H, o2 = r2[2] / H;
    const int child = m.fine8[e * 8 + o2 * 4 + o1 * 2 + o0];
    add_restrict8<T, NB>(lam, child, 2 * r2[0] - o0 * NB + G, 2 * r2[1] - o1 * NB + G, 2 * r2[2] - o2 * NB + G, w);
  } else {
    const int4 cl = m.leaf[C];
    const int K = m.idx[e];
    const int4 kl = m.leaf[K];
    int g[3] = {cl.y * NB + rc[0], cl.z * NB + rc[1], cl.w * NB + rc[2]};
    g[a] += side;
    g[a] = wrap_mod(g[a], (m.root[a] << cl.x) * NB);
    add5<T, NB>(lam, K, (g[0] >> 1) - kl.y * NB + G, (g[1] >> 1) - kl.z * NB + G, (g[2] >> 1) - kl.w * NB + G, w);
  }
}

template <typename T, int NB>
__global__ void __launch_bounds__(256) adjoint_refresh_scatter_kernel(DevMesh m, const T* U, T* lam) {
  constexpr int G = kGhosts, N = NB + 2 * G, NG = N * N * N - NB * NB * NB, H = NB / 2;
  constexpr long SLAB = (long)N * N * N;
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long)m.B * NG) return;
  const int leaf = (int)(gid / NG);
  int c[3];
  ghost_coord<NB>((int)(gid % NG), c[0], c[1], c[2]);
  const long own = (long)leaf * 5 * SLAB + ((long)c[2] * N + c[1]) * N + c[0];
  T lg[5];
  bool any = false;
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    lg[f] = lam[own + f * SLAB];
    any = any || lg[f] != T(0);
  }
  if (!any) return;
  int d[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    d[a] = c[a] < G ? -1 : (c[a] >= G + NB ? 1 : 0);
    if (d[a] != 0 && m.kind[leaf * 27 + face_dir(a, d[a])] == kBoundary) {
      c[a] = d[a] < 0 ? G : G + NB - 1;
      d[a] = 0;
    }
  }
  const int e = leaf * 27 + (d[2] + 1) * 9 + (d[1] + 1) * 3 + (d[0] + 1);
  const int8_t k = m.kind[e];
  if (k == kSame) {
    add5<T, NB>(lam, m.idx[e], c[0] - d[0] * NB, c[1] - d[1] * NB, c[2] - d[2] * NB, lg);
    return;
  }
  if (k == kFine) {
    int r[3], o[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      r[a] = c[a] - G - d[a] * NB;
      o[a] = r[a] / H;
    }
    const int child = m.fine8[e * 8 + o[2] * 4 + o[1] * 2 + o[0]];
    add_restrict8<T, NB>(lam, child, 2 * r[0] - o[0] * NB + G, 2 * r[1] - o[1] * NB + G, 2 * r[2] - o[2] * NB + G, lg);
    return;
  }
  // prolongation from the coarser leaf C, differentiated along the forward's branches
  const int4 lf = m.leaf[leaf];
  const int C = m.idx[e];
  const int4 cl = m.leaf[C];
  const int L = lf.x;
  const int lij[3] = {lf.y, lf.z, lf.w}, cij[3] = {cl.y, cl.z, cl.w};
  int rc[3];
  T sgn[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int ncell = (m.root[a] << L) * NB;
    const int gl = wrap_mod(lij[a] * NB + (c[a] - G), ncell);
    rc[a] = (gl >> 1) - cij[a] * NB;
    sgn[a] = (gl & 1) ? T(1) : T(-1);
  }
  T Uc[5];
  load5<T, NB>(U, C, rc[0] + G, rc[1] + G, rc[2] + G, Uc);
  T wc[5];
#pragma unroll
  for (int f = 0; f < 5; ++f) wc[f] = lg[f];
  for (int a = 0; a < 3; ++a) {
    T Um[5], Up[5];
    int rm[3] = {rc[0], rc[1], rc[2]}, rp[3] = {rc[0], rc[1], rc[2]};
    rm[a] -= 1;
    rp[a] += 1;
    if (rm[a] >= 0) load5<T, NB>(U, C, rm[0] + G, rm[1] + G, rm[2] + G, Um);
    else slope_neighbour<T, NB>(m, U, C, rc, a, -1, Uc, Um);
    if (rp[a] < NB) load5<T, NB>(U, C, rp[0] + G, rp[1] + G, rp[2] + G, Up);
    else slope_neighbour<T, NB>(m, U, C, rc, a, 1, Uc, Up);
    T wm[5], wp[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      const T lo = Uc[f] - Um[f], hi = Up[f] - Uc[f];
      const T gD = T(0.25) * sgn[a] * lg[f];   // adjoint of D_a
      wm[f] = T(0);
      wp[f] = T(0);
      if (lo * hi > T(0)) {
        if (vabs(lo) <= vabs(hi)) {   // D = U_C - U_m
          wc[f] += gD;
          wm[f] = -gD;
        } else {                      // D = U_p - U_C
          wc[f] -= gD;
          wp[f] = gD;
        }
      }
    }
    if (rm[a] >= 0) add5<T, NB>(lam, C, rm[0] + G, rm[1] + G, rm[2] + G, wm);
    else slope_neighbour_bwd<T, NB>(m, lam, C, rc, a, -1, wm);
    if (rp[a] < NB) add5<T, NB>(lam, C, rp[0] + G, rp[1] + G, rp[2] + G, wp);
    else slope_neighbour_bwd<T, NB>(m, lam, C, rc, a, 1, wp);
  }
  add5<T, NB>(lam, C, rc[0] + G, rc[1] + G, rc[2] + G, wc);
}

// Adjoint of the coarse-fine flux correction: with lam the adjoint after the
// step, d/dF_c = s (dt/dx_c) lam_c and each of the four fine fluxes gets
// -0.25 s (dt/dx_c) lam_c.  One thread per coarse face cell.
template <typename T, int NB>
__global__ void __launch_bounds__(256) fluxcorr_adjoint_kernel(DevMesh m, const T* lam, const CoarseFace* faces,
                                                               int nfaces, double* regb, const double* dt) {
  constexpr int G = kGhosts, N = NB + 2 * G, H = NB / 2;
  constexpr long SLAB = (long)N * N * N;
  constexpr long FS = (long)NB * NB;
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long)nfaces * NB * NB) return;
  const CoarseFace cf = faces[gid / (NB * NB)];
  const int i = (int)(gid % (NB * NB));
  const int t1 = i % NB, t2 = i / NB;
  const int4 cl = m.leaf[cf.leaf];
  const double coef = (*dt / ldexp(m.dx0, -cl.x)) * double(cf.side);
  const int t1a = cf.axis == 0 ? 1 : 0, t2a = cf.axis == 2 ? 1 : 2;
  int cc[3];
  cc[cf.axis] = cf.side > 0 ? G + NB - 1 : G;
  cc[t1a] = G + t1;
  cc[t2a] = G + t2;
  const T* cell = lam + (long)cf.leaf * 5 * SLAB + ((long)cc[2] * N + cc[1]) * N + cc[0];
  const int o1 = t1 / H, o2 = t2 / H, b1 = t1 - o1 * H, b2 = t2 - o2 * H;
  double* Rc = regb + (long)cf.cslot * 5 * FS + t2 * NB + t1;
  double* Rf = regb + (long)cf.fslot[o2 * 2 + o1] * 5 * FS + (2 * b2) * NB + 2 * b1;
#pragma unroll
  for (int f = 0; f < 5; ++f) {
    const double g = coef * double(cell[f * SLAB]);
    Rc[f * FS] = g;
    const double gf = -0.25 * g;
    double* r = Rf + f * FS;
    r[0] = gf;
    r[1] = gf;
    r[NB] = gf;
    r[NB + 1] = gf;
  }
}

template <typename T, int NB>
__global__ void __launch_bounds__(256) zero_ghosts_kernel(T* lam, int B) {
  constexpr int G = kGhosts, N = NB + 2 * G, NG = N * N * N - NB * NB * NB;
  constexpr long SLAB = (long)N * N * N;
  const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= (long)B * NG) return;
  const int leaf = (int)(gid / NG);
  int x, y, z;
  ghost_coord<NB>((int)(gid % NG), x, y, z);
  const long o = (long)leaf * 5 * SLAB + ((long)z * N + y) * N + x;
#pragma unroll
  for (int f = 0; f < 5; ++f) lam[o + f * SLAB] = T(0);
}

}  // namespace cello
