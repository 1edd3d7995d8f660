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
