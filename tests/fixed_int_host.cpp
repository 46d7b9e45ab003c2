// Host build of the fixed-point kernels' integer arithmetic (fixed_int.cuh) and of
// the integer primitives (soft64.cuh) for tests/test_fixed_int_host.py.
#include "device_host.h"

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

unsigned key1(double x) { return fx_group_key(&x, 1); }

template <int N>
void lines(const int2* F, const int2* D, long long* out) {
  long long o[N + 1];
  fx_line<N>(F, 1, D, o);
  for (int m = 0; m <= N; ++m) out[m] = o[m];
}

}  // namespace

// The 12 flux fields of one node (U, u, theta, p') as the kernels stage them for
// an element whose nodes all hold it; false if the element is out of range.
// f: (low, high) per slot; e: the exponents of U, the momentum fluxes and theta U.
extern "C" int fluxes_of(const double* z, int pipe, int* f, int* e) {
  Node n;
  std::memcpy(&n, z, sizeof n);
  const uint4 k = make_uint4(fx_group_key(n.U, 3), fx_group_key(n.u, 3), key1(n.th), key1(n.pp));
  if (!fx_in_range(k)) return 0;
  const FxExp x = fx_exps(k);
  auto put = [&](int slot, int2 v) {
    f[2 * slot] = v.x;
    f[2 * slot + 1] = v.y;
  };
  if (pipe) fx_fluxes<true>(n, x, k.z, put);
  else fx_fluxes<false>(n, x, k.z, put);
  e[0] = x.U;
  e[1] = x.m;
  e[2] = x.t;
  return 1;
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
