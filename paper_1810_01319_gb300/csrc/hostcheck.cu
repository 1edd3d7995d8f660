// Host-compiled entry points of the per-interface PPM arithmetic and its
// hand-written adjoint, and of the host operation count of a leaf's sweep,
// for CPU unit tests of the device math (the same CELLO_HD functions the
// kernels run).  Built into a separate test library; the product library
// does not contain it.
#include <thread>

#include "adjoint.cuh"
#include "opcount.cu"
#include "per_device.h"
#include "ppm64.cuh"

using namespace cello;

// The flux at the interface between cells 3 and 4 of an 8-cell window of
// conserved states (sweep component order), and its vector-Jacobian
// product: Ub[c][k] += sum_q Fb[q] dF_q/dU[c][k].  The pieces are those of the
// kernels, put together here interface by interface; the kernels evaluate each once
// per cell and hand it to the neighbours through shared memory.
template <typename T>
CELLO_HD void window_flux(const T U[8][5], T dtdx, const Gas<T>& gs, T F[5]) {
  T W[8][5];
  for (int c = 0; c < 8; ++c) to_primitive(U[c], gs, W[c]);
  T dm[8][5];
  for (int c = 1; c < 7; ++c)
    for (int q = 0; q < 5; ++q) dm[c][q] = limited_slope(W[c - 1][q], W[c][q], W[c + 1][q]);
  T ai[8][5];  // ai[c] = interface c|c+1, c = 2, 3, 4
  for (int c = 2; c < 5; ++c)
    for (int q = 0; q < 5; ++q) ai[c][q] = interface_value(W[c][q], W[c + 1][q], dm[c][q], dm[c + 1][q]);
  T ft[8];
  for (int c = 2; c < 6; ++c)
    ft[c] = flatten_tilde(W[c - 2][4], W[c - 1][4], W[c + 1][4], W[c + 2][4], W[c - 1][1], W[c + 1][1]);
  T edge[2][5];
  for (int side = 0; side < 2; ++side) {
    const int j = 3 + side;
    const T s = W[j + 1][4] - W[j - 1][4];
    const T f = (s > T(0)) ? vmax(ft[j], ft[j - 1]) : ((s < T(0)) ? vmax(ft[j], ft[j + 1]) : ft[j]);
    T aL[5], aR[5], Wm[5], Wp[5];
    for (int q = 0; q < 5; ++q) {
      aL[q] = ai[j - 1][q];
      aR[q] = ai[j][q];
      flatten_monotone(W[j][q], f, aL[q], aR[q]);
    }
    trace(W[j], aL, aR, dtdx, gs, Wm, Wp);
    for (int q = 0; q < 5; ++q) edge[side][q] = side == 0 ? Wp[q] : Wm[q];
  }
  riemann_flux(edge[0], edge[1], gs, F);
}

template <typename T>
CELLO_HD void window_flux_vjp(const T U[8][5], T dtdx, const Gas<T>& gs, const T Fb[5], T Ub[8][5]) {
  T W[8][5];
  for (int c = 0; c < 8; ++c) to_primitive(U[c], gs, W[c]);
  T dm[8][5];
  for (int c = 1; c < 7; ++c)
    for (int q = 0; q < 5; ++q) dm[c][q] = limited_slope(W[c - 1][q], W[c][q], W[c + 1][q]);
  T ai[8][5];
  for (int c = 2; c < 5; ++c)
    for (int q = 0; q < 5; ++q) ai[c][q] = interface_value(W[c][q], W[c + 1][q], dm[c][q], dm[c + 1][q]);
  T ft[8];
  for (int c = 2; c < 6; ++c)
    ft[c] = flatten_tilde(W[c - 2][4], W[c - 1][4], W[c + 1][4], W[c + 2][4], W[c - 1][1], W[c + 1][1]);
  T fval[2], aLm[2][5], aRm[2][5], edge[2][5];
  int fsel[2];  // -1: f = ft[j-1], 0: ft[j], +1: ft[j+1]
  for (int side = 0; side < 2; ++side) {
    const int j = 3 + side;
    const T s = W[j + 1][4] - W[j - 1][4];
    T f;
    if (s > T(0)) {
      f = vmax(ft[j], ft[j - 1]);
      fsel[side] = (ft[j] > ft[j - 1]) ? 0 : -1;
    } else if (s < T(0)) {
      f = vmax(ft[j], ft[j + 1]);
      fsel[side] = (ft[j] > ft[j + 1]) ? 0 : 1;
    } else {
      f = ft[j];
      fsel[side] = 0;
    }
    fval[side] = f;
    T Wm[5], Wp[5];
    for (int q = 0; q < 5; ++q) {
      aLm[side][q] = ai[j - 1][q];
      aRm[side][q] = ai[j][q];
      flatten_monotone(W[j][q], f, aLm[side][q], aRm[side][q]);
    }
    trace(W[j], aLm[side], aRm[side], dtdx, gs, Wm, Wp);
    for (int q = 0; q < 5; ++q) edge[side][q] = side == 0 ? Wp[q] : Wm[q];
  }
  // ---- reverse
  T eb[2][5] = {{0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}};
  riemann_flux_bwd(edge[0], edge[1], gs, Fb, eb[0], eb[1]);
  T Wb[8][5], aib[8][5], dmb[8][5], ftb[8];
  for (int c = 0; c < 8; ++c) {
    ftb[c] = T(0);
    for (int q = 0; q < 5; ++q) Wb[c][q] = aib[c][q] = dmb[c][q] = T(0);
  }
  for (int side = 0; side < 2; ++side) {
    const int j = 3 + side;
    const T zero5[5] = {0, 0, 0, 0, 0};
    T aLb[5] = {0, 0, 0, 0, 0}, aRb[5] = {0, 0, 0, 0, 0};
    trace_bwd(W[j], aLm[side], aRm[side], dtdx, gs, side == 0 ? zero5 : eb[1], side == 0 ? eb[0] : zero5, Wb[j],
              aLb, aRb);
    T fb = T(0);
    for (int q = 0; q < 5; ++q)
      flatten_monotone_bwd(W[j][q], fval[side], ai[j - 1][q], ai[j][q], aLb[q], aRb[q], Wb[j][q], fb, aib[j - 1][q],
                           aib[j][q]);
    ftb[j + fsel[side]] += fb;
  }
  for (int c = 5; c >= 2; --c)
    flatten_tilde_bwd(W[c - 2][4], W[c - 1][4], W[c + 1][4], W[c + 2][4], W[c - 1][1], W[c + 1][1], ftb[c], Wb[c - 2][4],
                      Wb[c - 1][4], Wb[c + 1][4], Wb[c + 2][4]);
  for (int c = 4; c >= 2; --c)
    for (int q = 0; q < 5; ++q) interface_value_bwd(aib[c][q], Wb[c][q], Wb[c + 1][q], dmb[c][q], dmb[c + 1][q]);
  for (int c = 6; c >= 1; --c)
    for (int q = 0; q < 5; ++q) limited_slope_bwd(W[c - 1][q], W[c][q], W[c + 1][q], dmb[c][q], Wb[c - 1][q], Wb[c][q],
                                                  Wb[c + 1][q]);
  for (int c = 0; c < 8; ++c) to_primitive_bwd(W[c], gs, Wb[c], Ub[c]);
}

template <typename T>
static void flux_t(const double* U, double dtdx, double gamma, double* F) {
  T u[8][5], f[5];
  for (int c = 0; c < 8; ++c)
    for (int k = 0; k < 5; ++k) u[c][k] = T(U[c * 5 + k]);
  window_flux(u, T(dtdx), Gas<T>::make(gamma), f);
  for (int k = 0; k < 5; ++k) F[k] = double(f[k]);
}

template <typename T>
static void vjp_t(const double* U, double dtdx, double gamma, const double* Fb, double* Ub) {
  T u[8][5], fb[5], ub[8][5];
  for (int c = 0; c < 8; ++c)
    for (int k = 0; k < 5; ++k) {
      u[c][k] = T(U[c * 5 + k]);
      ub[c][k] = T(0);
    }
  for (int k = 0; k < 5; ++k) fb[k] = T(Fb[k]);
  window_flux_vjp(u, T(dtdx), Gas<T>::make(gamma), fb, ub);
  for (int c = 0; c < 8; ++c)
    for (int k = 0; k < 5; ++k) Ub[c * 5 + k] = double(ub[c][k]);
}

extern "C" {
void cello_hc_window_flux(const double* U, double dtdx, double gamma, int precision, double* F) {
  if (precision == 4) flux_t<float>(U, dtdx, gamma, F);
  else flux_t<double>(U, dtdx, gamma, F);
}
void cello_hc_window_flux_vjp(const double* U, double dtdx, double gamma, int precision, const double* Fb,
                              double* Ub) {
  if (precision == 4) vjp_t<float>(U, dtdx, gamma, Fb, Ub);
  else vjp_t<double>(U, dtdx, gamma, Fb, Ub);
}
// One set-up asked for on each of the listed devices in turn, each by two threads at
// once; calls[d] counts its runs on device d.
void cello_hc_once_per_device(const int* devices, int count, int* calls) {
  OncePerDevice once;
  for (int i = 0; i < count; ++i) {
    const int d = devices[i];
    auto ask = [&] { once.run(d, [&] { ++calls[d]; }); };
    std::thread other(ask);
    ask();
    other.join();
  }
}
int cello_hc_corner_index(int v, int g, int N) { return corner_index(v, g, N); }
// One leaf's sweep through the counting scalar (float32 arithmetic), its
// update written back into slab [fields][N^3]; counts[6] per phase.
void cello_hc_opcount_leaf(float* slab, int n, int g, int axis, int a0, int a1, int b0, int b1, double dtdx,
                           double gamma, int riemann, int steepen, int dual, unsigned long long* counts) {
  opcount_leaf(slab, n, g, axis, a0, a1, b0, b1, dtdx, gamma, riemann, steepen, dual, counts);
}
// The float64 sweep's functions (ppm64.cuh) and their namesakes of ppm.cuh on
// count argument lists of `stride` values; results of both, out values each.
// what: 0 a / b, 1 sqrt, 2 primitives, 3 slope, 4 interface value, 5 detector,
// 6 edge states, 7 two-shock flux; 12, 16, 17 the six-field forms of 2, 6, 7.
void cello_hc_q64(int what, long count, int stride, const double* in, double gamma, int out, double* fast,
                  double* plain) {
  const Gas<double> gs = Gas<double>::make(gamma);
  auto states = [&](auto nq, const double* x, double* y, double* z) {
    constexpr int NQ = decltype(nq)::value;
    for (int form = 0; form < 2; ++form) {
      double* o = form ? z : y;
      double aL[NQ], aR[NQ], F[6], uf = 0.0;
      for (int q = 0; q < NQ; ++q) {
        aL[q] = x[NQ + q];
        aR[q] = x[2 * NQ + q];
      }
      if (what % 10 == 2) {
        if (!form) q64::primitives<NQ>(x, gs, o);
        else if constexpr (NQ == 6) to_primitive_de(x, gs, o);
        else to_primitive(x, gs, o);
      } else if (what % 10 == 6) {
        if (!form) {
          q64::edge_states<NQ>(x, x[3 * NQ], aL, aR, x[3 * NQ + 1], gs, o, o + NQ);
        } else {
          for (int q = 0; q < NQ; ++q) flatten_monotone(x[q], x[3 * NQ], aL[q], aR[q]);
          trace<double, NQ>(x, aL, aR, x[3 * NQ + 1], gs, o, o + NQ);
        }
      } else {
        if (!form) q64::two_shock_flux<NQ>(x, x + NQ, gs, F, &uf);
        else riemann_flux<double, NQ>(x, x + NQ, gs, F, &uf);
        for (int q = 0; q < NQ; ++q) o[q] = F[q];
        if (NQ == 6) o[6] = uf;
      }
    }
  };
  for (long i = 0; i < count; ++i) {
    const double* x = in + i * stride;
    double *y = fast + i * out, *z = plain + i * out;
    double inv;
    switch (what) {
      case 0: *y = q64::quot_any(x[0], x[1], q64::rcp(x[1])); *z = x[0] / x[1]; break;
      case 1: *y = q64::root(x[0], inv); *z = sqrt(x[0]); break;
      case 3: *y = q64::slope(x[0], x[1], x[2]); *z = limited_slope(x[0], x[1], x[2]); break;
      case 4: *y = q64::interface_val(x[0], x[1], x[2], x[3]); *z = interface_value(x[0], x[1], x[2], x[3]); break;
      case 5:
        *y = q64::detector(x[0], x[1], x[2], x[3], x[4], x[5]);
        *z = flatten_tilde(x[0], x[1], x[2], x[3], x[4], x[5]);
        break;
      default:
        if (what >= 10) states(std::integral_constant<int, 6>{}, x, y, z);
        else states(std::integral_constant<int, 5>{}, x, y, z);
    }
  }
}
}
