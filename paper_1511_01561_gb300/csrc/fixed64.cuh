// FP64 element kernels with their contractions in 64-bit fixed point on the
// integer pipe (sm_103a).
//
// GB300 issues 2 FP64 operations per SM per clock and 32 32x32+64-bit integer
// multiply-adds (IMAD.WIDE), so a product of two 58-bit numbers in three of
// them costs 3 cycles of the SM per warp against 16 for an FP64 FMA.  Every
// field of an element is written as a 58-bit integer relative to the largest
// magnitude of its equation group in the element (a power of two), D as a
// 60-bit integer relative to its largest row sum, and their products are
// summed exactly in 64-bit accumulators.  What is dropped is below 2^-58 of
// (largest field) x (row sum of |D|), the size whose 2^-53 an FP64 chain
// loses at every step.
//
// Elements whose values the integers cannot hold (an infinity or a NaN, or
// magnitudes near the ends of the FP64 range) go through a plain FP64 form,
// one element at a time, with the same results as ordinary arithmetic.
#pragma once

#include "kernels_common.cuh"

namespace numa {
namespace {

constexpr int kFxBits = 29;                       // bits of a low part
constexpr unsigned kFxMask = (1u << kFxBits) - 1;
constexpr unsigned kFxMinExp = 400, kFxMaxExp = 1600;  // biased exponents of a group's largest value

// x as a 58-bit integer in units of 2^(E - 1022 - 58), E the biased exponent
// of the group's largest magnitude: (low 29 bits, signed rest).  Exact for
// values within 2^5 of the largest; below, truncated towards zero.
__device__ __forceinline__ int2 fx_of(double x, int E) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = (hi & 0xfffffu) | 0x100000u;
  const int e = (int)((hi >> 20) & 0x7ffu);
  const int sh = min(E - e + 5, 63);  // (a zero or subnormal: e = 0, all bits shifted out)
  unsigned long long q = ((unsigned long long)__funnelshift_l(lo, m, 10) << 32) | (lo << 10);
  q >>= sh;
  const long long sg = (long long)((int)hi >> 31);
  const long long s = (long long)(q ^ (unsigned long long)sg) - sg;
  return make_int2((int)((unsigned)s & kFxMask), (int)(s >> kFxBits));
}

// S 2^(kexp - 1086) rounded to nearest: the double whose biased exponent is
// kexp less the leading zeros of |S|.
__device__ __forceinline__ double fx_to_double(long long S, int kexp) {
  const unsigned sg = (unsigned)((unsigned long long)S >> 32) & 0x80000000u;
  const unsigned long long u = (unsigned long long)(S < 0 ? -S : S);
  const int lz = __clzll((long long)u);
  const unsigned long long n = u << lz;  // (u = 0: lz = 64, selected away below)
  const unsigned long long mant = (n >> 11) + ((n >> 10) & 1ull);  // carries into the exponent
  const unsigned long long b = mant + ((unsigned long long)(unsigned)(kexp - lz - 1) << 52);
  return __hiloint2double(u ? (int)((unsigned)(b >> 32) | sg) : 0, u ? (int)(unsigned)b : 0);
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

// Whether the fixed-point form holds a CTA's groups (keys x, y, z).
__device__ __forceinline__ bool fx_in_range(uint4 k) {
  auto ok = [](unsigned key) { return key == 0u || ((key >> 20) - kFxMinExp <= kFxMaxExp - kFxMinExp); };
  return ok(k.x) && ok(k.y) && ok(k.z);
}

// (high, middle) accumulators += D * f, D = Dh 2^29 + Dl, f = fh 2^29 + fl;
// the product of the low parts (2^-58 of the full scale) is left out.
__device__ __forceinline__ void fx_mac(long long& h, long long& m, int2 D, int fl, int fh) {
  h += (long long)D.y * fh;
  m += (long long)D.y * fl;
  m += (long long)D.x * fh;
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
// in shared memory: operands of the multiply-adds, no register each.
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
    long long ah = 0, am = 0, bh = 0, bm = 0;
#pragma unroll
    for (int j = 0; j < H + O; ++j) fx_mac(ah, am, D[i * (H + O) + j], el[j], eh[j]);
#pragma unroll
    for (int j = 0; j < H; ++j) fx_mac(bh, bm, D[H * (H + O) + i * H + j], ol[j], oh[j]);
    const long long A = ah + (am >> kFxBits), B = bh + (bm >> kFxBits);
    out[i] = B + A;
    out[N - i] = B - A;
  }
  if constexpr (O) {
    long long h = 0, m = 0;
#pragma unroll
    for (int j = 0; j < H; ++j) fx_mac(h, m, D[H * (H + O) + H * H + j], ol[j], oh[j]);
    out[H] = h + (m >> kFxBits);
  }
}

// Elements per CTA and threads: the contractions of the rectilinear form are
// 5 (N+1)^2 lines per direction and element, one per thread and direction.
// At N = 4 an element's 125 lines and 125 nodes fill 128 threads; the small
// orders take several elements so that their lines fill whole warps.
template <int N>
__host__ __device__ constexpr int fx_rect_epb() {
  return N == 1 ? 8 : N == 2 ? 2 : N == 3 ? 2 : 1;
}
template <int N>
__host__ __device__ constexpr int fx_rect_threads() {
  return (fx_rect_epb<N>() * 5 * (N + 1) * (N + 1) + 31) / 32 * 32;
}
template <int N>
constexpr size_t fx_rect_smem() {
  constexpr int NN = fx_rect_epb<N>() * (N + 1) * (N + 1) * (N + 1);
  return 8 * (size_t)(kLF + 10) * NN + 16 * (size_t)(fx_rect_epb<N>() == 1 ? fx_rect_threads<N>() / 32 : fx_rect_epb<N>());
}

// The three directions' tables of one mesh.
template <int N>
struct FxTables {
  int2 d[3 * fx_table_entries<N>()];
};

// The rectilinear residual of one element by plain FP64 arithmetic, nothing
// staged: for elements the fixed-point form cannot hold.
template <int N>
__device__ __noinline__ void rect_plain(const VolumeArgs& a, long long e) {
  constexpr int P = N + 1, NP = P * P * P;
  const long long Nl = a.Nl, Ng = a.Ng;
  const double* w = static_cast<const double*>(a.prim);
  double* re = static_cast<double*>(a.re);
  for (int l = threadIdx.x; l < NP; l += blockDim.x) {
    const int i = l % P, j = (l / P) % P, k = l / (P * P);
#pragma unroll 1
    for (int v = 0; v < 5; ++v) {
      double t = 0.0;
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int row = d == 0 ? i : d == 1 ? j : k, st = d == 0 ? 1 : d == 1 ? P : P * P;
        const double K = a.affk[d * (long long)a.Ne + e];
        // the field of equation v along d: U, the symmetric U u + p' I, theta U
        const int s = v == 0 ? -1 - d : v == 4 ? 6 + d : v - 1 == d ? d : (v - 1) + d + 2;
        const double* f = s < 0 ? a.q + (1 + d) * Ng : w + s * Ng;
#pragma unroll 1
        for (int m = 0; m < P; ++m)
          t = fma(K * a.D64[row * P + m], f[a.l2g[e * NP + l + (m - row) * st]], t);
      }
      re[v * Nl + e * NP + l] = t;
    }
  }
}

// Shared-memory slots of the 12 flux fields: the five fields differentiated
// along x in the order of the equations, so that the x lines of all five are
// one run of memory (no bank conflicts), then the rest.
enum : int { sUx = 0, sTxx, sTxy, sTxz, sHx, sUy, sTyy, sTyz, sHy, sUz, sTzz, sHz };
__host__ __device__ constexpr int fx_slot(int f) {
  return f == lUx ? sUx : f == lUy ? sUy : f == lUz ? sUz : f == lTxx ? sTxx : f == lTyy ? sTyy : f == lTzz ? sTzz
       : f == lTxy ? sTxy : f == lTxz ? sTxz : f == lTyz ? sTyz : f == lHx ? sHx : f == lHy ? sHy : sHz;
}

// create_rhs of up to fx_rect_epb<N>() rectilinear elements e0 .. e0 + ne - 1
// in fixed point: the residual sum_d K_d (D F_d) without its weight
// w_i w_j w_k (which the update applies with the inverse mass).
//   1. one thread per element node gathers the 12 flux fields; the largest
//      magnitude of each equation group (mass: U; momentum: U u + p' I;
//      theta: theta U) gives the group's exponent;
//   2. the fields go to shared memory as fixed-point pairs;
//   3. thread t takes line t of the 5 (N+1)^2 lines along x (equation
//      v = t / (N+1)^2), then along y (fx_line), and leaves the derivatives in
//      shared memory;
//   4. it then takes its line along z, adds the x and y derivatives at the
//      line's nodes as integers and converts the sums to FP64, rounded once.
// On 32^3 elements at N = 4: 0.529 ms as FP64 (its pipe 97% busy: 75
// operations a node at 16 cycles a warp), 0.216 ms here; 19x23x17 at N = 6:
// 0.460 -> 0.148 ms.  108 integer multiply-adds a thread keep their pipe 21%
// busy; shared memory and the scattered gather (54% of the load/store unit's
// wavefronts) and the 845 instructions a warp are what is left.  D in the
// kernel parameters instead of global memory: 0.256 -> 0.226 ms; the z lines
// finishing the nodes (10 shared accesses a node fewer, ten CTAs an SM
// instead of eight): 0.226 -> 0.216 ms.
template <int N>
__device__ __forceinline__ void volume_fx_rect(const VolumeArgs& a, const int2* T, long long e0, int ne,
                                               unsigned char* smem_raw) {
  constexpr int P = N + 1, PP = P * P, NP = PP * P, EPB = fx_rect_epb<N>(), NN = EPB * NP;
  constexpr int NT = fx_rect_threads<N>(), IT = (NN + NT - 1) / NT;
  // the largest magnitudes of the three groups: one slot per warp (EPB = 1), or per element
  constexpr int SLOTS = EPB == 1 ? NT / 32 : EPB;
  uint4* gmax = reinterpret_cast<uint4*>(smem_raw);              // [SLOTS] (first: 16-byte aligned)
  int2* F = reinterpret_cast<int2*>(gmax + SLOTS);               // [kLF][NN]
  long long* part = reinterpret_cast<long long*>(F + kLF * NN);  // [2][5][NN]
  const int tid = threadIdx.x;
  const long long Nl = a.Nl, n0 = e0 * NP;
  const int nn = ne * NP;
  if constexpr (EPB > 1) {
    if (tid < EPB) gmax[tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
  }
  uint4 gw = make_uint4(0u, 0u, 0u, 0u);
  FluxState64 z[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int l = tid + it * NT;
    unsigned g0 = 0, g1 = 0, g2 = 0;
    if (l < nn) {
      z[it] = gather_fluxes64(a, n0 + l);
      g0 = fx_group_key(z[it].f + lUx, 3);
      g1 = fx_group_key(z[it].f + lTxx, 6);
      g2 = fx_group_key(z[it].f + lHx, 3);
    }
    if constexpr (EPB == 1) {
      gw = make_uint4(max(gw.x, g0), max(gw.y, g1), max(gw.z, g2), 0u);
    } else if (l < nn) {
      unsigned* gm = reinterpret_cast<unsigned*>(gmax + l / NP);
      atomicMax(&gm[0], g0);
      atomicMax(&gm[1], g1);
      atomicMax(&gm[2], g2);
    }
  }
  if constexpr (EPB == 1) {
    gw.x = __reduce_max_sync(0xffffffffu, gw.x);
    gw.y = __reduce_max_sync(0xffffffffu, gw.y);
    gw.z = __reduce_max_sync(0xffffffffu, gw.z);
    if ((tid & 31) == 0) gmax[tid >> 5] = gw;
  }
  __syncthreads();
  // biased exponents of the groups; (uniform over the CTA) any group outside
  // the range: every element plain
  bool plain = a.fxD == nullptr;
  uint4 gm = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int t = 0; t < SLOTS; ++t) {
    const uint4 w = gmax[t];
    if constexpr (EPB == 1) gm = make_uint4(max(gm.x, w.x), max(gm.y, w.y), max(gm.z, w.z), 0u);
    else plain |= !fx_in_range(w);
  }
  if constexpr (EPB == 1) plain |= !fx_in_range(gm);
  if (plain) {
    for (int t = 0; t < ne; ++t) rect_plain<N>(a, e0 + t);
    return;
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int l = tid + it * NT;
    if (l < nn) {
      if constexpr (EPB > 1) gm = gmax[l / NP];
      const int E0 = (int)(gm.x >> 20), E1 = (int)(gm.y >> 20), E2 = (int)(gm.z >> 20);
#pragma unroll
      for (int f = 0; f < kLF; ++f) F[fx_slot(f) * NN + l] = fx_of(z[it].f[f], f <= lUz ? E0 : f <= lTyz ? E1 : E2);
    }
  }
  __syncthreads();
  const bool act = tid < ne * 5 * PP;
  const int el = EPB == 1 ? 0 : tid / (5 * PP), tt = tid - el * 5 * PP;
  const int v = tt / PP, r = tt - v * PP;
  constexpr int M = fx_table_entries<N>();
  if (act) {
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      // the field of equation v along x, y (four bits each)
      constexpr unsigned fy = sUy | sTxy << 4 | sTyy << 8 | sTyz << 12 | sHy << 16;
      const int f = d == 0 ? v : (int)((fy >> (4 * v)) & 15u);
      const int base = el * NP + (d == 0 ? P * r : r % P + PP * (r / P)), st = d == 0 ? 1 : P;
      long long out[P];
      fx_line<N>(F + f * NN + base, st, T + d * M, out);
      long long* o = part + (d * 5 + v) * NN + base;
#pragma unroll
      for (int m = 0; m < P; ++m) o[m * st] = out[m];
    }
  }
  __syncthreads();
  if (act) {
    constexpr unsigned fz = sUz | sTxz << 4 | sTyz << 8 | sTzz << 12 | sHz << 16;
    const int f = (int)((fz >> (4 * v)) & 15u), base = el * NP + r;
    long long out[P];
    fx_line<N>(F + f * NN + base, PP, T + 2 * M, out);
    const long long* o = part + v * NN + base;
    if constexpr (EPB > 1) gm = gmax[el];
    const int kexp = (int)((v == 0 ? gm.x : v == 4 ? gm.z : gm.y) >> 20) + a.fxexp;
    double* re = static_cast<double*>(a.re) + v * Nl + n0 + base;
#pragma unroll
    for (int m = 0; m < P; ++m) re[m * PP] = fx_to_double(out[m] + o[m * PP] + o[5 * NN + m * PP], kexp);
  }
}

template <int N>
__global__ void __launch_bounds__(fx_rect_threads<N>())
    volume_fx_rect_kernel(const __grid_constant__ VolumeArgs a, const __grid_constant__ FxTables<N> T) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int EPB = fx_rect_epb<N>();
  const int e = (int)blockIdx.x * EPB;
  volume_fx_rect<N>(a, T.d, a.ebeg + (long long)e, min(EPB, a.ecnt - e), smem_raw);
}

// Ragged form: positions of the group are chunks of fx_rect_epb<N>() elements
// of one member.
template <int N>
__global__ void __launch_bounds__(fx_rect_threads<N>())
    volume_fx_rect_ragged(const MemberDesc* __restrict__ d, const RaggedGroup* __restrict__ g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_m;
  __shared__ long long s_e;
  __shared__ int2 s_T[3 * fx_table_entries<N>()];
  constexpr int EPB = fx_rect_epb<N>();
  const int n = g->n;
  const long long total = n > 0 ? g->elem_prefix[n] : 0;
  for (long long w = blockIdx.x; w < total; w += gridDim.x) {
    if (threadIdx.x == 0) {
      const int m = ragged_find(g->elem_prefix, n, w);
      s_m = g->member[m];
      s_e = (w - g->elem_prefix[m]) * EPB;
    }
    __syncthreads();
    // (uniform across the CTA) guard against a table that disagrees with the member
    if (s_m >= 0 && s_m < kMaxMembers && s_e >= 0 && s_e < d[s_m].va.Ne) {
      const VolumeArgs& a = d[s_m].va;
      if (a.fxD)  // (read after the barriers of volume_fx_rect)
        for (int t = threadIdx.x; t < 3 * fx_table_entries<N>(); t += blockDim.x) s_T[t] = a.fxD[t];
      volume_fx_rect<N>(a, s_T, s_e, (int)min((long long)EPB, a.Ne - s_e), smem_raw);
    }
    __syncthreads();
  }
}

}  // namespace
}  // namespace numa
