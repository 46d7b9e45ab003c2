// Host build of the fixed-point kernels' integer arithmetic (fixed_int.cuh) and of
// the integer primitives (soft64.cuh) for tests/test_fixed_int_host.py.
#include "device_host.h"

#include <cstdlib>

// the FP32 reciprocal with an error of its own, in units of 2^-23
static float rcp_error = 0.0f;
static float rcp_approx(float d) { return (float)(1.0 / (double)d + (double)rcp_error * 0x1p-23); }

#include "fixed_int.cuh"
#include "numa_internal.h"
#include "soft64.cuh"

using namespace numa;

namespace {

struct Node {
  double U[3], u[3], th, pp;
};

template <int N>
void lines(const int2* F, const int2* D, long long* out) {
  long long o[N + 1];
  fx_line<N>(F, 1, D, o);
  for (int m = 0; m <= N; ++m) out[m] = o[m];
}

}  // namespace

// The flux fields of one node (U, u, theta, p') as the kernels stage them for an
// element whose nodes all hold it, with the directions scaled by 2^-s: the 15 of
// the rectilinear form, or (shared) the 12 of the per-node form; false if the
// element is out of range.  f: (low, high) per field; e: the exponents of U, the
// three momentum equations and theta U.
extern "C" int fluxes_of(const double* z, const int* s, int shared, int* f, int* e) {
  Node n;
  std::memcpy(&n, z, sizeof n);
  FxScale w;
  FxKeys k = FxKeys();
  for (int c = 0; c < 3; ++c) {
    w.s[c] = s[c];
    k.u[c] = fx_key(n.u[c]);
  }
  k.U = fx_key_scaled(n.U, w);
  k.th = fx_key(n.th);
  k.pp = fx_key(n.pp);
  const FxExp x = fx_exps(k, w);
  if (!x.ok) return 0;
  auto put = [&](int slot, int2 v) {
    f[2 * slot] = v.x;
    f[2 * slot + 1] = v.y;
  };
  if (shared) fx_fluxes_shared(n, x, w, put);
  else fx_fluxes(n, x, w, put);
  e[0] = x.U;
  for (int v = 0; v < 3; ++v) e[1 + v] = x.m[v];
  e[4] = x.t;
  return 1;
}

// fx_pair of the equations' exponents m and the scale s.
extern "C" int pair_of(const int* m, const int* s, int a, int b) {
  FxExp e = {};
  FxScale w;
  for (int c = 0; c < 3; ++c) {
    e.m[c] = m[c];
    w.s[c] = s[c];
  }
  return fx_pair(e, w, a, b);
}
// A derivative as the first (second = 0) or second of the pair's equations takes it.
extern "C" long long value_of(long long x, int pair, int second) {
  return fx_shift(x, second ? -pair : pair);
}

// fx_line of order N over the line's fields (low, high), with the table of
// 2^(60 - e) D, the largest row sum of |D| below 2^e.
extern "C" void line_of(int N, const int* f, int e, long long* out) {
  int2 D[kFxEntries], F[kMaxN + 1];
  fx_table_host(N + 1, nullptr, 1.0, 1.0, 1.0, 60 - e, 0, D);
  for (int m = 0; m <= N; ++m) F[m] = make_int2(f[2 * m], f[2 * m + 1]);
  switch (N) {
    case 1: lines<1>(F, D, out); break;
    case 2: lines<2>(F, D, out); break;
    case 3: lines<3>(F, D, out); break;
    case 4: lines<4>(F, D, out); break;
    case 5: lines<5>(F, D, out); break;
    case 6: lines<6>(F, D, out); break;
    case 7: lines<7>(F, D, out); break;
    case 8: lines<8>(F, D, out); break;
  }
}

// x / rho as the update's primitive pass forms it, with a reciprocal seed that is
// off by `error` units of 2^-23.
extern "C" double div_of(double x, double rho, float error) {
  rcp_error = error;
  return soft_div(x, rcp58(rho), soft_exp(rho));
}
