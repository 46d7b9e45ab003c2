// The primitive fields of a node in FP64 accuracy on the integer pipe
// (sm_103a): 1/rho, u = U / rho, theta = Theta / rho and p' as products of
// 58-bit mantissas.
//
// The update's FP64 operations bound it (2 per SM per clock: 16 cycles of an
// SM per warp instruction), while 83% of its issue slots are empty.  A
// product of two 58-bit mantissas is three IMAD.WIDE (one cycle of an SM each)
// and about 20 instructions with its normalisation and rounding, 5 cycles.
// Every result is rounded once: u and theta from 57 bits, p' from a product of
// 56 to 58 bits that is short by up to a unit and a half per factor.  Against 113
// bits u and theta are within 0.56 ulp and p' within 0.81: below the error of the
// FP64 sequence (a reciprocal, then a product).  The update went
// from 0.169 to 0.133 ms a stage on 32^3 elements at N = 4 and from 0.294 to
// 0.215 ms on the 6x30x30x8 shell.
//
// Values outside the exponent range below, or |Theta'/Theta0| > 2^-5, take
// the FP64 sequence (write_prim).
#pragma once

#include <cstdint>

#include "numa_internal.h"

namespace numa {
namespace {

constexpr int kSoftLo = 1023 - 400, kSoftHi = 1023 + 400;  // biased exponents taken

__device__ __forceinline__ int soft_exp(double x) { return (int)(((unsigned)__double2hiint(x) >> 20) & 0x7ffu); }
__device__ __forceinline__ bool soft_zero(double x) {
  return (((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x)) == 0u;
}
__device__ __forceinline__ bool soft_in(double x) { return (unsigned)(soft_exp(x) - kSoftLo) <= (unsigned)(kSoftHi - kSoftLo); }

// 58 bits as h 2^29 + l.
struct M58 {
  unsigned l, h;
};

// The mantissa of a normal x, 1.f 2^57 (in [2^57, 2^58)).
__device__ __forceinline__ M58 mant58(double x) {
  const unsigned lo = (unsigned)__double2loint(x), hi = ((unsigned)__double2hiint(x) & 0xfffffu) | 0x100000u;
  return {(lo << 5) & 0x1fffffffu, __funnelshift_r(lo, hi, 24)};
}
__device__ __forceinline__ M58 split58(unsigned long long v) {
  return {(unsigned)v & 0x1fffffffu, (unsigned)(v >> 29)};
}

// a b 2^-58, short by less than one unit and a half (the low parts' product).
__device__ __forceinline__ unsigned long long mul58(M58 a, M58 b) {
  unsigned long long m = 1ull << 28;
  m += (unsigned long long)a.l * b.h;
  m += (unsigned long long)a.h * b.l;
  return (unsigned long long)a.h * b.h + (m >> 29);
}

#ifdef __CUDACC__
// 1/d in FP32, d in [1, 2): within 2^-23.
__device__ __forceinline__ float rcp_approx(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}
#endif

// 1/d 2^58 for d = m 2^-52 in [1, 2): the FP32 reciprocal r0, then
// r0 (1 + e + e^2) with e = 1 - d r0 formed exactly (its leading bits cancel).
// The approximation may fall on either side of [1/2, 1), whose exponent R0
// relies on: next to d = 1 and d = 2 r0 is that interval's end (|e| < 2^-22).
__device__ __forceinline__ M58 rcp58(double x) {
  const unsigned lo = (unsigned)__double2loint(x), hi = ((unsigned)__double2hiint(x) & 0xfffffu) | 0x100000u;
  const float df = __uint_as_float(0x3f800000u | __funnelshift_l(lo, hi & 0xfffffu, 3));
  const float r = fmaxf(fminf(rcp_approx(df), 0.99999994f), 0.5f);
  const unsigned R0 = (__float_as_uint(r) & 0x7fffffu) | 0x800000u;  // r0 2^24
  // e 2^76 = 2^76 - m R0, exact in the low 64 bits (|e| < 2^-21)
  const long long E = -(long long)((unsigned long long)lo * R0 + ((unsigned long long)(hi * R0) << 32));
  const long long e1 = E >> 16;          // e 2^60
  const int es = (int)(E >> 32);         // e 2^44
  const long long t1 = ((long long)(unsigned)e1 * R0 + (((long long)((int)(e1 >> 32) * (int)R0)) << 32)) >> 24;
  const unsigned e2 = (unsigned)(((long long)es * es) >> 20);               // e^2 2^68
  const unsigned t2 = (unsigned)(((unsigned long long)e2 * R0) >> 32);      // r0 e^2 2^60
  const unsigned long long R = ((unsigned long long)R0 << 36) + (unsigned long long)t1 + t2;  // 2^60 / d
  return split58((R + 2) >> 2);
}

// P 2^-57 (in [1/2, 2)) times 2^(e - 1023), with x's sign; zero for x = 0.
__device__ __forceinline__ double pack57(unsigned long long P, int e, double x) {
  const unsigned top = (unsigned)(P >> 57);  // whether P >= 2^57
  const unsigned long long mant = (P + (8u << top)) >> (4 + top);  // 53 bits, or 2^53 (then the exponent carries)
  const unsigned long long b = mant + ((unsigned long long)(unsigned)(e + (int)top - 2) << 52);
  const unsigned sign = (unsigned)__double2hiint(x) & 0x80000000u;
  const bool zero = soft_zero(x);
  return __hiloint2double(zero ? (int)sign : (int)((unsigned)(b >> 32) | sign), zero ? 0 : (int)(unsigned)b);
}

// p' = p0 ((1 + x)^gamma - 1), x = T iT, by the binomial series
// x (c1 + x (c2 + ...)) with the term counts of eos_ratio: x in units of
// 2^-63, the coefficients in units of 2^-58.  Terms whose power of x is below
// 2^-29 of the first are summed in units of 2^-29 (32 bits), the first n64 in
// 2^-58.
__device__ __forceinline__ double soft_pressure(const PrimArgs& a, double p0, double T, double iT) {
  const int eT = soft_exp(T), eI = soft_exp(iT), eP = soft_exp(p0);
  const unsigned long long X = mul58(mant58(T), mant58(iT));  // |x| 2^(2102 - eT - eI)
  const unsigned long long xf = soft_zero(T) ? 0ull : X >> min(2039 - (eT + eI), 63);
  const long long xs = __double2hiint(T) < 0 ? -(long long)xf : (long long)xf;
  const int xl = (int)((unsigned)xs & 0x1fffffffu), xh = (int)(xs >> 29);
  const unsigned hx = (unsigned)(xf >> 26);  // |x| 2^37
  const int K = hx <= 1u << 7 ? 2 : hx <= 1u << 17 ? 3 : hx <= 1u << 22 ? 4 : hx <= 1u << 25 ? 5 : hx <= 1u << 27 ? 6 : kEosTerms;
  const int n64 = hx <= 1u << 8 ? 1 : hx <= 1u << 22 ? 2 : hx <= 1u << 27 ? 3 : hx <= 1u << 29 ? 4 : kEosFull;
  int acc = a.eosH[K - 1];
  for (int k = K - 2; k >= n64; --k) acc = a.eosH[k] + (int)(((long long)acc * xh) >> 34);
  long long A = (long long)acc << 29;
  for (int k = n64 - 1; k >= 0; --k) {
    const int al = (int)((unsigned)A & 0x1fffffffu), ah = (int)(A >> 29);
    long long m = 1ll << 28;
    m += (long long)ah * xl;
    m += (long long)al * xh;
    A = a.eosI[k] + (((long long)ah * xh + (m >> 29)) >> 5);
  }
  // p0 |x| A: P1 in [2^55, 2^58), then up to sqrt(2) times that
  const unsigned long long P = mul58(split58(mul58(split58(X), mant58(p0))), split58((unsigned long long)A));
  const int lz = __clzll((long long)P);
  const unsigned long long n = P << lz;
  const unsigned long long b = (n >> 11) + ((n >> 10) & 1ull) +
                               ((unsigned long long)(unsigned)(eP + eT + eI - 2039 - lz) << 52);
  const unsigned sign = (unsigned)__double2hiint(T) & 0x80000000u;
  const bool zero = soft_zero(T);
  return __hiloint2double(zero ? (int)sign : (int)((unsigned)(b >> 32) | sign), zero ? 0 : (int)(unsigned)b);
}

// Whether the integer form takes these values: rho > 0, Theta, U and Theta' zero or
// normal and not extreme, |Theta'/Theta0| below 2^-5.
__device__ __forceinline__ bool soft_ok(const PrimArgs& a, double rho, double Ux, double Uy, double Uz, double Th,
                                        double Tp, double p0, double iTh0) {
  auto in0 = [](double x) { return soft_in(x) || soft_zero(x); };
  return a.eos_soft && __double2hiint(rho) > 0 && soft_in(rho) && in0(Ux) && in0(Uy) && in0(Uz) && in0(Th) &&
         soft_in(p0) && soft_in(iTh0) && __double2hiint(p0) > 0 && __double2hiint(iTh0) > 0 &&
         (soft_zero(Tp) || (soft_in(Tp) && soft_exp(Tp) + soft_exp(iTh0) <= 2039));
}

// x / rho with r = rcp58(rho).
__device__ __forceinline__ double soft_div(double x, M58 r, int erho) {
  return pack57(mul58(mant58(x), r), soft_exp(x) - erho + 1023, x);
}

}  // namespace
}  // namespace numa
