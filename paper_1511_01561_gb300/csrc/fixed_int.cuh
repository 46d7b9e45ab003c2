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

// S 2^(kexp - 1086) rounded to nearest, and fx_of by the FP64 pipe: a conversion
// and an exact product each, 32 cycles of a pipe that is otherwise idle in
// place of 24 and 15 integer instructions.  The host's bounds on the tables and
// fx_exps' on the groups keep kexp - 63 within an FP64's biased exponents.
// Measured with one momentum unit on 32^3 elements, N = 4 (rectilinear) and the
// 6x30x30x8 shell (per-node): all five results so, 0.183 -> 0.174 and 0.540 ->
// 0.526 ms; U and p' of the eight inputs too, 0.183 and 0.519 ms (so in the
// per-node form only); all eight, 0.213 and 0.520 ms.
__device__ __forceinline__ double fx_to_double(long long S, int kexp) {
  return __ll2double_rn(S) * __hiloint2double((kexp - 63) << 20, 0);
}
__device__ __forceinline__ long long fx_of_pipe(double x, int E) {
  return __double2ll_rn(x * __hiloint2double((2103 - E) << 20, 0));
}

// Magnitude key of a value: its high word without the sign (monotonic in |x|);
// at least 1 unless the value is zero.
__device__ __forceinline__ unsigned fx_key(double x) {
  return max((unsigned)__double2hiint(x) & 0x7fffffffu, min((unsigned)__double2loint(x), 1u));
}

// Powers of two (s_x, s_y, s_z >= 0) taken out of the three directions of a
// flux, one of them zero: 2^-s_c F_c are of a size with the terms K_c dF_c / dx_c of
// Eq. 4 that they lead to (K_c: the size of the metric terms that multiply
// F_c).  On an element a hundred times wider than high U_z is a hundredth of U_x
// and K_z a hundred times K_x: with one unit for both, the integers lost a
// hundred times as much as FP64 sums, whose error follows max_c K_c |F_c|: on smooth
// flow over elements of 500 to 1 the tendencies of mass and theta were 20 to 40 times
// as far off as FP64's.  In these units the integers' error follows the same bound.
struct FxScale {
  int s[3];
};

// The same without a look at the low word: 0 for values below 2^-1042 too.  (With
// the low words of a node's eight values the kernels take 1% longer at N = 4.)
__device__ __forceinline__ unsigned fx_high(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// The key of the vector 2^-s_c x_c from its high words; 0 where those of all components
// are below 2^(s_c - 1022).
__device__ __forceinline__ unsigned fx_high_scaled(const double (&x)[3], const FxScale& w) {
  int k = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) k = max(k, (int)fx_high(x[c]) - (w.s[c] << 20));
  return (unsigned)k;
}
// The key of the vector; at least 1 unless it is zero.
__device__ __forceinline__ unsigned fx_key_scaled(const double (&x)[3], const FxScale& w) {
  return max(fx_high_scaled(x, w), min(fx_key(x[0]) | fx_key(x[1]) | fx_key(x[2]), 1u));
}

// Magnitude keys of an element: of 2^-s_c U_c, theta, p' and each component of u.
struct alignas(16) FxKeys {
  unsigned U, th, pp, unused;
  unsigned u[3], unused2;
};

// The biased exponents of an element's equation groups, |field| <
// 2^(exponent - 1022): mass: 2^-s_c U_c; momentum equation v: 2^-s_c (U_c u_v +
// p' I); theta: 2^-s_c theta U_c; and of theta and p' themselves.  A group of zeros has the
// exponent of 1, so that its zero sums meet a finite factor in fx_to_double.
struct alignas(16) FxExp {
  int U, m[3];
  int t, th, pp;
  int ok;  // the integers hold the element
};
constexpr int kFxZero = 1023;
constexpr int kFxLeast = 100;  // at this exponent and above fx_of shifts every bit of a zero out

__device__ __forceinline__ bool fx_in(int E) { return (unsigned)E - kFxMinExp <= kFxMaxExp - kFxMinExp; }
__device__ __forceinline__ bool fx_ok(unsigned key) { return key == 0u || fx_in((int)(key >> 20)); }

// The exponent of momentum equation v from the keys of U, u_v and p', s = s_v;
// ok: whether u_v and the group are in range.  U_c u_v and p' each stay below
// 2^(m - 1022).  Where their exponents are equal m is one above them, so their
// sum stays below 1.5 2^(m - 1022): 1.5 2^58 as an integer, whose high part is at
// most 1.5 2^29, so that fx_line's sums of two of them fit 32 bits.
__device__ __forceinline__ int fx_momentum_exp(unsigned U, unsigned u, unsigned pp, int s, bool& ok) {
  // whether the product of the largest U and u carries into the next power of two
  const unsigned mU = (U & 0xfffffu) + 0x100001u, mu = (u & 0xfffffu) + 0x100001u;
  const int Uu = (int)(U >> 20) + (int)(u >> 20) - 1023 + ((unsigned long long)mU * mu > (1ull << 41));
  const int p = (int)(pp >> 20) - s;
  const int m = U && u ? max(Uu, p) + (Uu == p) : pp ? p : kFxZero;
  ok = fx_ok(u) && fx_in(m);
  return m;
}
// The other exponents of e; ok: whether they and the keys of U, theta and p' are in range.
__device__ __forceinline__ bool fx_scalar_exps(FxExp& e, unsigned U, unsigned th, unsigned pp) {
  e.U = U ? (int)(U >> 20) : kFxZero;
  e.t = U && th ? (int)(U >> 20) + (int)(th >> 20) - 1022 : kFxZero;
  e.th = max((int)(th >> 20), kFxLeast);
  e.pp = max((int)(pp >> 20), kFxLeast);
  return fx_ok(U) && fx_ok(th) && fx_ok(pp) && fx_in(e.t);
}
// One unit for U_a u_b in both its equations (fx_pair = 0) where that makes no
// equation's unit larger than four times its own: the 58 bits of a group then
// keep 56 of the largest of its equation, FP64 sums 53.
__device__ __forceinline__ void fx_join(FxExp& e, const FxScale& w) {
  const int m = max(e.m[0] - w.s[0], max(e.m[1] - w.s[1], e.m[2] - w.s[2]));
  const int least = min(e.m[0] - w.s[0], min(e.m[1] - w.s[1], e.m[2] - w.s[2]));
  if (m - least <= 2) {
#pragma unroll
    for (int v = 0; v < 3; ++v) e.m[v] = m + w.s[v];
  }
}
__device__ __forceinline__ FxExp fx_exps(const FxKeys& k, const FxScale& w) {
  FxExp e = FxExp();
  bool ok = fx_scalar_exps(e, k.U, k.th, k.pp);
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    bool in;
    e.m[v] = fx_momentum_exp(k.U, k.u[v], k.pp, w.s[v], in);
    ok &= in;
  }
  e.ok = ok;
  fx_join(e, w);
  return e;
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

// a b 2^-58 + c, rounded but for the product of the low parts, split as by fx_split.
__device__ __forceinline__ int2 fx_mul_split(int2 a, int2 b, long long c = 0) {
  long long h = c + kFxHalf, m = kFxHalf;
  fx_mac(h, m, a, b.x, b.y);
  const long long s = fx_sum(h, m);
  return make_int2((int)((unsigned)s & kFxMask) - (int)kFxHalf, (int)(s >> kFxBits));
}

// The integers of a node (U, u, theta, p' in z): U_c in the unit of the mass
// group, u_v in the unit that makes U_c u_v one of momentum equation v, theta and
// p' in their own.
struct FxNode {
  int2 U[3], u[3], th;
  long long pp;
};
template <bool PIPE, typename Z>
__device__ __forceinline__ FxNode fx_node(const Z& z, const FxExp& e, const FxScale& w) {
  FxNode n;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    n.U[c] = fx_split((PIPE ? fx_of_pipe : fx_of)(z.U[c], e.U + w.s[c]));
    n.u[c] = fx_split(fx_of(z.u[c], max(e.m[c] - e.U + 1022, kFxLeast)));
  }
  n.th = fx_split(fx_of(z.th, e.th));
  n.pp = (PIPE ? fx_of_pipe : fx_of)(z.pp, e.pp);
  return n;
}
// p' in momentum equation v along v, in the equation's unit (cut: the derivative of a
// constant is exactly zero).
__device__ __forceinline__ long long fx_pressure(const FxNode& n, const FxExp& e, const FxScale& w, int v) {
  return n.pp >> min(e.m[v] + w.s[v] - e.pp, 63);
}

// The 15 flux fields of a node for the rectilinear form: put(5 c + v, value) of
// the flux of equation v along direction c, scaled by 2^-s_c, in equation v's
// unit.  With one scale and one unit for all (elements of three like edges) U_a u_b
// serves as the flux of a along b and of b along a, and p' is shifted once.
template <typename Z, typename Put>
__device__ __forceinline__ void fx_fluxes(const Z& z, const FxExp& e, const FxScale& w, Put put) {
  const FxNode n = fx_node<false>(z, e, w);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    put(5 * c, n.U[c]);
    put(5 * c + 4, fx_mul_split(n.U[c], n.th));
  }
  if (((e.m[0] ^ e.m[1]) | (e.m[0] ^ e.m[2]) | w.s[0] | w.s[1] | w.s[2]) == 0) {
    const long long p = fx_pressure(n, e, w, 0);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      put(5 * c + 1 + c, fx_mul_split(n.U[c], n.u[c], p));
#pragma unroll
      for (int v = c + 1; v < 3; ++v) {
        const int2 T = fx_mul_split(n.U[c], n.u[v]);
        put(5 * c + 1 + v, T);
        put(5 * v + 1 + c, T);
      }
    }
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int v = 0; v < 3; ++v)
        put(5 * c + 1 + v, fx_mul_split(n.U[c], n.u[v], v == c ? fx_pressure(n, e, w, v) : 0));
  }
}

// Slots of the 12 flux fields of the per-node form, in which U_a u_b stands for the
// flux of momentum a along b and of b along a.
enum : int { sUx = 0, sTxx, sTxy, sTxz, sHx, sUy, sTyy, sTyz, sHy, sUz, sTzz, sHz };

// The two equations' exponents of U_a u_b (a != b), their difference: equation a takes it along b, in the
// unit m_a + s_b, equation b along a, in m_b + s_a.  The field is held in the
// smaller unit; the equation of the other shifts its derivative right (fx_shift).
__device__ __forceinline__ int fx_pair(const FxExp& e, const FxScale& w, int a, int b) {
  return (e.m[a] + w.s[b]) - (e.m[b] + w.s[a]);
}
// x 2^-sh rounded for sh > 0, else x.
__device__ __forceinline__ long long fx_shift(long long x, int sh) {
  if (sh > 0) {
    sh = min(sh, 62);
    x = (x + (1ll << (sh - 1))) >> sh;
  }
  return x;
}

// The 12 flux fields of a node for the per-node form: put(slot, value).
template <typename Z, typename Put>
__device__ __forceinline__ void fx_fluxes_shared(const Z& z, const FxExp& e, const FxScale& w, Put put) {
  const FxNode n = fx_node<true>(z, e, w);
  auto diag = [&](int c) { return fx_mul_split(n.U[c], n.u[c], fx_pressure(n, e, w, c)); };
  auto off = [&](int a, int b) {
    const bool in_a = fx_pair(e, w, a, b) <= 0;
    return fx_mul_split(in_a ? n.U[b] : n.U[a], in_a ? n.u[a] : n.u[b]);
  };
  put(sUx, n.U[0]);
  put(sUy, n.U[1]);
  put(sUz, n.U[2]);
  put(sTxx, diag(0));
  put(sTyy, diag(1));
  put(sTzz, diag(2));
  put(sTxy, off(0, 1));
  put(sTxz, off(0, 2));
  put(sTyz, off(1, 2));
  put(sHx, fx_mul_split(n.U[0], n.th));
  put(sHy, fx_mul_split(n.U[1], n.th));
  put(sHz, fx_mul_split(n.U[2], n.th));
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
