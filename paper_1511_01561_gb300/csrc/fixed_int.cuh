// Integer arithmetic of the fixed-point FP64 kernels (fixed64.cuh, imex.cu):
// conversions, equation-group exponents, products and lines of D.  Plain
// functions of their arguments, so that a host build can run them too, given
// the device intrinsics they use.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace numa {
namespace {

constexpr int kFxBits = 29;                       // bits of a low part
constexpr unsigned kFxMask = (1u << kFxBits) - 1;
constexpr long long kFxHalf = 1ll << (kFxBits - 1);  // half a unit of the high part: where a middle accumulator starts
// biased exponents of a group's largest value, and of a metric row's
constexpr unsigned kFxMinExp = 400, kFxMaxExp = 1600;
constexpr int kFxMetMin = 1023 - 200, kFxMetMax = 1023 + 200;

// Entry i of a table of small integers, 4 bits per point of a line.
__device__ __forceinline__ int fx_nibble(unsigned long long t, int i) { return (int)((t >> (4 * i)) & 15ull); }

// The power of two taken out of node (i, j, k)'s quadrature weight: the sum of
// its three points' exponents (negated in fxw).
__device__ __forceinline__ int fx_weight_exp(unsigned long long fxw, int i, int j, int k) {
  return -(fx_nibble(fxw, i) + fx_nibble(fxw, j) + fx_nibble(fxw, k));
}

// x as a 58-bit integer in units of 2^(E - 1022 - 58), |x| < 2^(E - 1022).
// Exact for values within 2^5 of that; below, truncated towards zero.
__device__ __forceinline__ long long fx_of(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = (hi & 0xfffffu) | 0x100000u;
  const int e = (int)((hi >> 20) & 0x7ffu);
  const int sh = min(E - e + 5, 63);  // (a zero or subnormal: e = 0, all bits shifted out)
  unsigned long long q = ((unsigned long long)__funnelshift_l(lo, m, 10) << 32) | (lo << 10);
  q >>= sh;
  const long long sg = (long long)((int)hi >> 31);
  return (long long)(q ^ (unsigned long long)sg) - sg;
}

// s as l + 2^29 h, l from -2^28 to 2^28 - 1: signed, so that the products of low
// parts that fx_mac leaves out have no mean (with l from 0 their mean, the
// same at every node of a row of D, is half a unit of a derivative).
__device__ __forceinline__ int2 fx_split(long long s) {
  s += kFxHalf;
  return make_int2((int)((unsigned)s & kFxMask) - (int)kFxHalf, (int)(s >> kFxBits));
}

// S 2^(kexp - 1086) rounded to nearest (kexp - 63 within an FP64's biased
// exponents: the host's bounds on the tables' and fx_in_range's on the groups'), and fx_of by the FP64 pipe: a conversion
// and an exact product each, 32 cycles of a pipe that is otherwise idle in
// place of 24 and 15 integer instructions.  Measured on 32^3 elements, N = 4
// (rectilinear) and the 6x30x30x8 shell (per-node): all five results so, 0.183
// -> 0.174 and 0.540 -> 0.526 ms; U and p' of the eight inputs too, 0.183 and
// 0.519 ms (so in the per-node form only); all eight, 0.213 and 0.520 ms.
__device__ __forceinline__ double fx_to_double(long long S, int kexp) {
  return __ll2double_rn(S) * __hiloint2double((kexp - 63) << 20, 0);
}
__device__ __forceinline__ long long fx_of_pipe(double x, int E) {
  return __double2ll_rn(x * __hiloint2double((2103 - E) << 20, 0));
}

// Magnitude key of a group of values: the largest of their high words without
// the sign (monotonic in |x|); at least 1 if any value is nonzero.
__device__ __forceinline__ unsigned fx_group_key(const double* x, int n) {
  unsigned k = 0, low = 0;
#pragma unroll
  for (int t = 0; t < n; ++t) {
    k = max(k, (unsigned)__double2hiint(x[t]) & 0x7fffffffu);
    low |= (unsigned)__double2loint(x[t]);
  }
  return max(k, low ? 1u : 0u);
}

// The biased exponents of an element's equation groups, |field| <
// 2^(exponent - 1022), from the magnitude keys of U, u, theta and p' (x, y, z,
// w): mass: U; momentum: U u + p' I; theta: theta U.  A group of zeros has the
// exponent of 1, so that its zero sums meet a finite factor in fx_to_double.
struct FxExp {
  int U, m, t;
};
constexpr int kFxZero = 1023;
constexpr int kFxLeast = 100;  // at this exponent and above fx_of shifts every bit of a zero out
// U u and p' each stay below 2^(m - 1022).  Where their exponents are equal m is
// one above them, so their sum stays below 1.5 2^(m - 1022): 1.5 2^58 as an
// integer, whose high part is at most 1.5 2^29, so that fx_line's sums of two
// of them fit 32 bits.
__device__ __forceinline__ FxExp fx_exps(uint4 k) {
  const int U = k.x ? (int)(k.x >> 20) : kFxZero, p = (int)(k.w >> 20);
  // whether the product of the largest U and u carries into the next power of two
  const unsigned mU = (k.x & 0xfffffu) + 0x100001u, mu = (k.y & 0xfffffu) + 0x100001u;
  const int Uu = U + (int)(k.y >> 20) - 1023 + ((unsigned long long)mU * mu > (1ull << 41));
  const int m = k.x && k.y ? max(Uu, p) + (Uu == p) : k.w ? p : kFxZero;
  return {U, m, k.x && k.z ? U + (int)(k.z >> 20) - 1022 : kFxZero};
}

// Whether the fixed-point form holds an element with these keys: every field
// and every group.
__device__ __forceinline__ bool fx_in_range(uint4 k) {
  auto in = [](int E) { return (unsigned)E - kFxMinExp <= kFxMaxExp - kFxMinExp; };
  auto ok = [&](unsigned key) { return key == 0u || in((int)(key >> 20)); };
  const FxExp e = fx_exps(k);
  return ok(k.x) && ok(k.y) && ok(k.z) && ok(k.w) && in(e.m) && in(e.t);
}

// (high, middle) accumulators += D * f, D = Dh 2^29 + Dl, f = fh 2^29 + fl;
// the product of the low parts (below half a unit of the high one) is left out.  The
// middle accumulator starts at half a unit of the high one, so that
// h + (m >> 29) is rounded, not cut: a cut would leave every derivative half a
// unit low, an error that does not average out over a mesh.
__device__ __forceinline__ void fx_mac(long long& h, long long& m, int2 D, int fl, int fh) {
  h += (long long)D.y * fh;
  m += (long long)D.y * fl;
  m += (long long)D.x * fh;
}

// h + (m >> 29).  (With m's high word as one more multiply-add, h + 8 m.hi + ...:
// 5% slower.)
__device__ __forceinline__ long long fx_sum(long long h, long long m) {
  return h + (m >> kFxBits);
}

// a b 2^-58, rounded but for the product of the low parts.
__device__ __forceinline__ long long fx_mul(int2 a, int2 b) {
  long long h = 0, m = kFxHalf;
  fx_mac(h, m, a, b.x, b.y);
  return fx_sum(h, m);
}

// Shared-memory slots of the 12 flux fields: the five fields differentiated
// along x in the order of the equations, so that the x lines of all five are
// one run of memory (no bank conflicts), then the rest.
enum : int { sUx = 0, sTxx, sTxy, sTxz, sHx, sUy, sTyy, sTyz, sHy, sUz, sTzz, sHz };
// The 12 flux fields of a node (U, u, theta, p' in z) as integers of their
// groups: put(slot, value).  thkey: the magnitude key of theta.
template <bool PIPE, typename Z, typename Put>
__device__ __forceinline__ void fx_fluxes(const Z& z, FxExp e, unsigned thkey, Put put) {
  // u in the unit that makes U u one of the momentum group's, p' in the group's own
  int2 U[3], u[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    U[c] = fx_split((PIPE ? fx_of_pipe : fx_of)(z.U[c], e.U));
    u[c] = fx_split(fx_of(z.u[c], max(e.m - e.U + 1022, kFxLeast)));
  }
  const int2 th = fx_split(fx_of(z.th, max((int)(thkey >> 20), kFxLeast)));
  const long long p = (PIPE ? fx_of_pipe : fx_of)(z.pp, e.m);
  put(sUx, U[0]);
  put(sUy, U[1]);
  put(sUz, U[2]);
  put(sTxx, fx_split(fx_mul(U[0], u[0]) + p));
  put(sTyy, fx_split(fx_mul(U[1], u[1]) + p));
  put(sTzz, fx_split(fx_mul(U[2], u[2]) + p));
  put(sTxy, fx_split(fx_mul(U[0], u[1])));
  put(sTxz, fx_split(fx_mul(U[0], u[2])));
  put(sTyz, fx_split(fx_mul(U[1], u[2])));
  put(sHx, fx_split(fx_mul(U[0], th)));
  put(sHy, fx_split(fx_mul(U[1], th)));
  put(sHz, fx_split(fx_mul(U[2], th)));
}

// Entries of a direction's even/odd table (see fx_line).
template <int N>
__host__ __device__ constexpr int fx_table_entries() {
  constexpr int P = N + 1, H = P / 2, O = P % 2;
  return H * (H + O) + H * H + O * H;
}

// out = D F along one line, with the even/odd split of D: the Lobatto points
// are symmetric, so D_{N-i,N-j} = -D_ij and with e_j = F_j + F_{N-j},
// o_j = F_j - F_{N-j} (j < P/2),
//   A_i = sum_j (D_ij + D_{i,N-j})/2 e_j + D_{i,mid} F_mid,
//   B_i = sum_j (D_ij - D_{i,N-j})/2 o_j,
//   out_i = A_i + B_i, out_{N-i} = B_i - A_i, out_mid = sum_j D_{mid,j} o_j:
// 12 products per line of 5 nodes instead of 25.  D points at the direction's
// table (A's rows, B's rows, then the middle row), in the kernel parameters or
// in shared memory: operands of the multiply-adds, no register each.  Fields
// below 1.5 2^58, so that the high parts of e and o stay within 1.5 2^30.
template <int N>
__device__ __forceinline__ void fx_line(const int2* __restrict__ F, int stride, const int2* D,
                                        long long (&out)[N + 1]) {
  constexpr int P = N + 1, H = P / 2, O = P % 2;
  int el[H + 1], eh[H + 1], ol[H], oh[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const int2 a = F[j * stride], b = F[(N - j) * stride];
    el[j] = a.x + b.x;
    eh[j] = a.y + b.y;
    ol[j] = a.x - b.x;
    oh[j] = a.y - b.y;
  }
  if constexpr (O) {
    const int2 c = F[H * stride];
    el[H] = c.x;
    eh[H] = c.y;
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    long long ah = 0, am = kFxHalf, bh = 0, bm = kFxHalf;
#pragma unroll
    for (int j = 0; j < H + O; ++j) fx_mac(ah, am, D[i * (H + O) + j], el[j], eh[j]);
#pragma unroll
    for (int j = 0; j < H; ++j) fx_mac(bh, bm, D[H * (H + O) + i * H + j], ol[j], oh[j]);
    const long long A = fx_sum(ah, am), B = fx_sum(bh, bm);
    out[i] = B + A;
    out[N - i] = B - A;
  }
  if constexpr (O) {
    long long h = 0, m = kFxHalf;
#pragma unroll
    for (int j = 0; j < H; ++j) fx_mac(h, m, D[H * (H + O) + H * H + j], ol[j], oh[j]);
    out[H] = fx_sum(h, m);
  }
}

}  // namespace
}  // namespace numa
