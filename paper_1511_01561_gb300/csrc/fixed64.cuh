// FP64 element kernels with their contractions in 64-bit fixed point on the
// integer pipe (sm_103a).
//
// GB300 issues 2 FP64 operations per SM per clock and 32 32x32+64-bit integer
// multiply-adds (IMAD.WIDE), so a product of two 58-bit numbers in three of
// them costs 3 cycles of the SM per warp against 16 for an FP64 FMA.  Every
// field of an element is a 58- or 59-bit integer relative to the largest magnitude
// of its equation group in the element (a power of two), D as a
// 60-bit integer relative to its largest row sum, and their products are
// summed exactly in 64-bit accumulators.  What is dropped is below 2^-58 of
// (largest field) x (row sum of |D|), the size whose 2^-53 an FP64 chain
// loses at every step.
//
// Elements whose values the integers cannot hold (an infinity or a NaN, or
// magnitudes near the ends of the FP64 range) go through a plain FP64 form,
// one element at a time, whichever elements share their CTA.
#pragma once

#include "fixed_int.cuh"
#include "kernels_common.cuh"

namespace numa {
namespace {

// Shared-memory layout of an element's nodes: node (i, j, k) at i + A j + B k.
// The lines of a direction are read one per lane; at N = 3 and N = 7 the
// natural pitches put whole warps on a few banks (a direction's reads take 2.3
// and 2.8 times the wavefronts), so the planes and rows are padded there.
template <int N>
__host__ __device__ constexpr int fx_row() {
  return N == 7 ? 9 : N + 1;
}
template <int N>
__host__ __device__ constexpr int fx_plane() {
  return N == 3 ? 19 : fx_row<N>() * (N + 1);
}
template <int N>
__host__ __device__ constexpr int fx_pitch() {  // one element
  return fx_plane<N>() * (N + 1);
}
// Shared index of node l of the CTA's elements.
template <int N>
__device__ __forceinline__ int fx_index(int l) {
  constexpr int P = N + 1, PP = P * P, NP = PP * P;
  if constexpr (fx_pitch<N>() == NP) return l;
  else {
    const int el = l / NP, m = l - el * NP;
    return el * fx_pitch<N>() + m % P + fx_row<N>() * ((m / P) % P) + fx_plane<N>() * (m / PP);
  }
}
// First node and stride of line r along direction d.
template <int N>
__device__ __forceinline__ int fx_line_base(int d, int r) {
  constexpr int P = N + 1, A = fx_row<N>(), B = fx_plane<N>();
  const int lo = r % P, hi = r / P;
  return d == 0 ? A * lo + B * hi : d == 1 ? lo + B * hi : lo + A * hi;
}
template <int N>
__device__ __forceinline__ constexpr int fx_line_stride(int d) {
  return d == 0 ? 1 : d == 1 ? fx_row<N>() : fx_plane<N>();
}

// Elements per CTA and threads of the rectilinear form: 5 (N+1)^2 lines per
// direction and element, one per thread.  At N = 4 an element's 125 lines and
// 125 nodes fill 128 threads; the small orders take several elements so that
// their lines fill whole warps.
template <int N>
__host__ __device__ constexpr int fx_rect_epb() {
  return N == 1 ? 8 : N == 2 ? 2 : N == 3 ? 2 : 1;
}
template <int N>
__host__ __device__ constexpr int fx_rect_threads() {
  return (fx_rect_epb<N>() * 5 * (N + 1) * (N + 1) + 31) / 32 * 32;
}
// Slots of the groups' magnitudes: one per warp of a CTA with one element, or one per element.
template <int EPB, int NT>
__host__ __device__ constexpr int fx_slots() {
  return EPB == 1 ? NT / 32 : EPB;
}
template <int N>
constexpr size_t fx_rect_smem() {
  constexpr int EPB = fx_rect_epb<N>();
  return 8 * (size_t)(kLF + 10) * EPB * fx_pitch<N>() + 16 * fx_slots<EPB, fx_rect_threads<N>()>();
}

// The per-node form: one thread per node, several elements for the small
// orders (their 12 (N+1)^2 lines per direction go round the threads).
template <int N>
__host__ __device__ constexpr int fx_nodal_epb() {
  return N == 1 ? 16 : N == 2 ? 4 : N == 3 ? 2 : 1;
}
template <int N>
__host__ __device__ constexpr int fx_nodal_threads() {
  return (fx_nodal_epb<N>() * (N + 1) * (N + 1) * (N + 1) + 31) / 32 * 32;
}
template <int N>
constexpr size_t fx_nodal_smem() {
  constexpr int EPB = fx_nodal_epb<N>();
  return 8 * (size_t)(2 * kLF) * EPB * fx_pitch<N>() + 16 * fx_slots<EPB, fx_nodal_threads<N>()>();
}

// A mesh's tables as a kernel parameter: K_d D for the three directions
// (rectilinear form), or D alone (per-node form).
template <int N, int DIRS>
struct FxTables {
  int2 d[DIRS * fx_table_entries<N>()];
};

// The flux of equation v along c at global node g, plain FP64: U, the
// symmetric U u + p' I, theta U.
__device__ __forceinline__ double plain_flux(const VolumeArgs& a, int v, int c, int g) {
  const double* U = a.q + a.Ng + g;
  const double* w = static_cast<const double*>(a.prim) + g;
  if (v == 0) return U[c * a.Ng];
  if (v == 4) return w[3 * a.Ng] * U[c * a.Ng];
  const int lo = min(v - 1, c), hi = max(v - 1, c);
  return fma(U[lo * a.Ng], w[hi * a.Ng], lo == hi ? w[4 * a.Ng] : 0.0);
}

// The rectilinear residual of one element by plain FP64 arithmetic, nothing
// staged: for elements the fixed-point form cannot hold.
template <int N>
__device__ __forceinline__ void rect_plain(const VolumeArgs& a, long long e) {
  constexpr int P = N + 1, NP = P * P * P;
  const long long Nl = a.Nl;
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
#pragma unroll 1
        for (int m = 0; m < P; ++m)
          t = fma(K * a.D64[row * P + m], plain_flux(a, v, d, a.l2g[e * NP + l + (m - row) * st]), t);
      }
      re[v * Nl + e * NP + l] = t;
    }
  }
}

// Gathers U, u, theta and p' at the nn element nodes from n0, one thread per
// element node, and leaves the 12 flux fields in F as fixed-point integers.
// The largest magnitudes in an element give its groups' exponents: left as
// keys per element in gmax (EPB > 1), or returned in ge (EPB = 1).  False
// (uniform over the CTA) if the integers cannot hold its one element; with
// several, the fields of an element they cannot hold (fx_in_range of its key)
// are left unset, so that no element's result depends on which others share
// its CTA (a slab launch groups them otherwise).
template <int N, int EPB, int NT, bool PIPE>
__device__ __forceinline__ bool fx_stage(const VolumeArgs& a, long long n0, int nn, uint4* gmax, int2* F, FxExp& ge) {
  constexpr int NP = (N + 1) * (N + 1) * (N + 1), NN = EPB * NP, IT = (NN + NT - 1) / NT;
  constexpr int FP = EPB * fx_pitch<N>(), SLOTS = fx_slots<EPB, NT>();
  const int tid = threadIdx.x;
  if constexpr (EPB > 1) {
    if (tid < EPB) gmax[tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
  }
  uint4 gw = make_uint4(0u, 0u, 0u, 0u);
  NodeState64 z[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int l = tid + it * NT;
    if (l < nn) {
      z[it] = gather_node64(a, n0 + l);
      const uint4 k = make_uint4(fx_group_key(z[it].U, 3), fx_group_key(z[it].u, 3), fx_group_key(&z[it].th, 1),
                                 fx_group_key(&z[it].pp, 1));
      if constexpr (EPB == 1) {
        gw = make_uint4(max(gw.x, k.x), max(gw.y, k.y), max(gw.z, k.z), max(gw.w, k.w));
      } else {
        unsigned* g = reinterpret_cast<unsigned*>(gmax + l / NP);
        atomicMax(&g[0], k.x);
        atomicMax(&g[1], k.y);
        atomicMax(&g[2], k.z);
        atomicMax(&g[3], k.w);
      }
    }
  }
  if constexpr (EPB == 1) {
    gw.x = __reduce_max_sync(0xffffffffu, gw.x);
    gw.y = __reduce_max_sync(0xffffffffu, gw.y);
    gw.z = __reduce_max_sync(0xffffffffu, gw.z);
    gw.w = __reduce_max_sync(0xffffffffu, gw.w);
    if ((tid & 31) == 0) gmax[tid >> 5] = gw;
  }
  grid_wait();  // (threads without a node; before any write of the kernel)
  __syncthreads();
  uint4 gm = make_uint4(0u, 0u, 0u, 0u);
  if constexpr (EPB == 1) {
#pragma unroll
    for (int t = 0; t < SLOTS; ++t) {
      const uint4 w = gmax[t];
      gm = make_uint4(max(gm.x, w.x), max(gm.y, w.y), max(gm.z, w.z), max(gm.w, w.w));
    }
    if (!fx_in_range(gm)) return false;
    ge = fx_exps(gm);
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int l = tid + it * NT;
    if (l < nn) {
      if constexpr (EPB > 1) {
        gm = gmax[l / NP];
        if (!fx_in_range(gm)) continue;
      }
      const FxExp e = fx_exps(gm);
      int2* f = F + fx_index<N>(l);
      fx_fluxes<PIPE>(z[it], e, gm.z, [&](int slot, int2 x) { f[slot * FP] = x; });
    }
  }
  return true;
}

// create_rhs of up to fx_rect_epb<N>() rectilinear elements e0 .. e0 + ne - 1
// in fixed point: the residual sum_d K_d (D F_d) without its weight
// w_i w_j w_k (which the update applies with the inverse mass).
//   1. the 12 flux fields go to shared memory (fx_stage);
//   2. thread t takes line t of the 5 (N+1)^2 lines along x (equation
//      v = t / (N+1)^2), then along y (fx_line), and leaves the derivatives in
//      shared memory;
//   3. it then takes its line along z, adds the x and y derivatives at the
//      line's nodes as integers and converts the sums to FP64, rounded once.
// On 32^3 elements at N = 4: 0.529 ms as FP64 (its pipe 97% busy: 75
// operations a node at 16 cycles a warp), 0.156 ms here; 19x23x17 at N = 6:
// 0.460 -> 0.135 ms.  135 integer multiply-adds a thread keep their pipe a
// quarter busy; shared memory, the scattered gather and the instructions
// beside the products are what is left.  D in the kernel parameters instead
// of global memory: 0.256 -> 0.226 ms; the z lines finishing the nodes (10
// shared accesses a node fewer, ten CTAs an SM instead of eight): 0.226 ->
// 0.216 ms; the products formed here from 8 gathered fields instead of 12
// gathered fluxes: 0.216 -> 0.186 ms (and the update 0.199 -> 0.169 ms); the
// results converted by the FP64 pipe and 64 registers: 0.186 -> 0.156 ms.
template <int N>
__device__ __forceinline__ void volume_fx_rect(const VolumeArgs& a, const int2* T, long long e0, int ne,
                                               unsigned char* smem_raw) {
  constexpr int P = N + 1, PP = P * P, NP = PP * P, EPB = fx_rect_epb<N>(), NT = fx_rect_threads<N>();
  constexpr int EP = fx_pitch<N>(), FP = EPB * EP, M = fx_table_entries<N>(), B = fx_plane<N>();
  uint4* gmax = reinterpret_cast<uint4*>(smem_raw);                // (first: 16-byte aligned)
  int2* F = reinterpret_cast<int2*>(gmax + fx_slots<EPB, NT>());  // [kLF][FP]
  long long* part = reinterpret_cast<long long*>(F + kLF * FP);    // [2][5][FP]
  const int tid = threadIdx.x;
  const long long n0 = e0 * NP;
  FxExp ge;
  if (a.fxD == nullptr || !fx_stage<N, EPB, NT, false>(a, n0, ne * NP, gmax, F, ge)) {  // uniform over the CTA
    for (int t = 0; t < ne; ++t) rect_plain<N>(a, e0 + t);
    return;
  }
  __syncthreads();
  const bool act = tid < ne * 5 * PP;
  const int el = EPB == 1 ? 0 : tid / (5 * PP), tt = tid - el * 5 * PP;
  const int v = tt / PP, r = tt - v * PP;
  if (act) {
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      // the field of equation v along x, y (four bits each)
      constexpr unsigned fy = sUy | sTxy << 4 | sTyy << 8 | sTyz << 12 | sHy << 16;
      const int f = d == 0 ? v : (int)((fy >> (4 * v)) & 15u);
      const int base = el * EP + fx_line_base<N>(d, r), st = fx_line_stride<N>(d);
      long long out[P];
      fx_line<N>(F + f * FP + base, st, T + d * M, out);
      long long* o = part + (d * 5 + v) * FP + base;
#pragma unroll
      for (int m = 0; m < P; ++m) o[m * st] = out[m];
    }
  }
  __syncthreads();
  if (act) {
    constexpr unsigned fz = sUz | sTxz << 4 | sTyz << 8 | sTzz << 12 | sHz << 16;
    const int f = (int)((fz >> (4 * v)) & 15u), base = el * EP + fx_line_base<N>(2, r);
    long long out[P];
    fx_line<N>(F + f * FP + base, B, T + 2 * M, out);
    const long long* o = part + v * FP + base;
    bool ok = true;
    if constexpr (EPB > 1) {
      ok = fx_in_range(gmax[el]);
      ge = fx_exps(gmax[el]);
    }
    if (ok) {
      const int kexp = (v == 0 ? ge.U : v == 4 ? ge.t : ge.m) + a.fxexp;
      double* re = static_cast<double*>(a.re) + v * a.Nl + n0 + el * NP + r;
#pragma unroll
      for (int m = 0; m < P; ++m) re[m * PP] = fx_to_double(out[m] + o[m * B] + o[5 * FP + m * B], kexp);
    }
  }
  if constexpr (EPB > 1) {
    for (int t = 0; t < ne; ++t)  // (uniform over the CTA)
      if (!fx_in_range(gmax[t])) rect_plain<N>(a, e0 + t);
  }
}

// The per-node residual of one element by plain FP64 arithmetic (see
// rect_plain), with the metric terms read back from their integers.
template <int N>
__device__ __forceinline__ void nodal_plain(const VolumeArgs& a, long long e) {
  constexpr int P = N + 1, PP = P * P, NP = PP * P;
  const long long Nl = a.Nl;
  double* re = static_cast<double*>(a.re);
  const int4 eb = a.fxE[e];
  for (int l = threadIdx.x; l < NP; l += blockDim.x) {
    const int i = l % P, j = (l / P) % P, k = l / PP;
#pragma unroll 1
    for (int v = 0; v < 5; ++v) {
      double t = 0.0;
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int row = d == 0 ? i : d == 1 ? j : k, st = d == 0 ? 1 : d == 1 ? P : PP;
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
          double x = 0.0;
#pragma unroll 1
          for (int m = 0; m < P; ++m)
            x = fma(a.D64[row * P + m], plain_flux(a, v, c, a.l2g[e * NP + l + (m - row) * st]), x);
          // eb.w: the metric terms of this element stayed doubles
          const long long at = (3 * d + c) * Nl + e * NP + l;
          double b = a.met64[at];
          if (!eb.w) {
            const int2 h = reinterpret_cast<const int2*>(a.met64)[at];
            const int E = d == 0 ? eb.x : d == 1 ? eb.y : eb.z;
            b = scalbn((double)(((long long)h.y << kFxBits) + h.x), E - 1022 - 2 * kFxBits + fx_weight_exp(a.fxw, i, j, k));
          }
          t = fma(b, x, t);
        }
      }
      re[v * Nl + e * NP + l] = t;
    }
  }
}

// create_rhs of up to fx_nodal_epb<N>() elements of any shape in fixed point,
// the per-node form of Eq. 5.  Per reference direction d:
//   1. each thread takes one line and every G-th field on it (fx_line) and
//      leaves the derivatives in shared memory;
//   2. one thread per node multiplies the 12 derivatives by the direction's
//      row of -Jw dxi_d/dx_c (58-bit integers relative to the row's largest
//      value in the element, fx_metric_kernel) into the five equations.
// Every row of D is scaled to its own row sum (an end row's is up to 16 times
// an inner one's).  The directions' sums are aligned by the exponents of their
// rows, added as integers and rounded once.
// On the 6x30x30x8 shell at N = 4: 2.068 ms as FP64 (225 operations a node, its
// pipe 96% busy), 0.520 ms here; 21x17x13 at N = 3: 0.105 -> 0.039 ms.  The 430
// integer multiply-adds a thread keep their pipe 40% busy and the 2300
// instructions a warp 60% of the issue slots, at 8 CTAs an SM (64 registers).
// With the fluxes formed in the update it took 0.505 ms, and the update 0.335
// instead of 0.294 ms.  Going round all lines of a direction with a division per line
// instead of one line per thread: 0.570 against 0.505 ms.
template <int N>
__device__ __forceinline__ void volume_fx_nodal(const VolumeArgs& a, const int2* T, long long e0, int ne,
                                                unsigned char* smem_raw) {
  constexpr int P = N + 1, PP = P * P, NP = PP * P, EPB = fx_nodal_epb<N>(), NT = fx_nodal_threads<N>();
  constexpr int EP = fx_pitch<N>(), FP = EPB * EP;
  uint4* gmax = reinterpret_cast<uint4*>(smem_raw);                // (first: 16-byte aligned)
  int2* F = reinterpret_cast<int2*>(gmax + fx_slots<EPB, NT>());  // [kLF][FP]
  long long* S = reinterpret_cast<long long*>(F + kLF * FP);       // [kLF][FP]: the direction's derivatives
  const int tid = threadIdx.x, nn = ne * NP;
  const long long Nl = a.Nl, n0 = e0 * NP;
  const bool node = tid < nn;
  const int nel = EPB == 1 ? 0 : tid / NP;
  // the elements' metric exponents (w: the element takes plain FP64)
  const int4 eb = a.fxE[e0 + (node ? nel : 0)];
  FxExp ge;
  bool ok = fx_stage<N, EPB, NT, true>(a, n0, nn, gmax, F, ge) && !eb.w;
  if constexpr (EPB == 1) {  // (uniform over the CTA)
    if (!ok) {
      nodal_plain<N>(a, e0);
      return;
    }
  } else {
    ok = ok && fx_in_range(gmax[nel]);
  }
  __syncthreads();
  const int at = fx_index<N>(tid);
  const int2* met = reinterpret_cast<const int2*>(a.met64) + n0 + tid;
  // the exponents of the node's three directions: the metric row's less that
  // taken out of its row of D; the sums are kept in units of the largest
  const int l = tid - nel * NP;
  const int x0 = eb.x - fx_nibble(a.fxr, l % P), x1 = eb.y - fx_nibble(a.fxr, (l / P) % P);
  const int x2 = eb.z - fx_nibble(a.fxr, l / PP), xm = max(x0, max(x1, x2));
  long long sum[5] = {0, 0, 0, 0, 0};
  // thread's line of every direction, and its first field; the threads of a
  // line's group take every G-th field
  constexpr int LN = EPB * PP, G = NT / LN;
  static_assert(G >= 1, "a thread per line");
  const int g = tid / LN, q = tid - g * LN, lel = EPB == 1 ? 0 : q / PP, r = q - lel * PP;
  const int f0 = g < G && lel < ne ? g : kLF;
  auto direction = [&](auto dir) {
    constexpr int d = decltype(dir)::value, st = fx_line_stride<N>(d);
    int2 B[3];
    if (node) {
#pragma unroll
      for (int c = 0; c < 3; ++c) B[c] = met[(3 * d + c) * Nl];
    }
    const int base = lel * EP + fx_line_base<N>(d, r);
    for (int f = f0; f < kLF; f += G) {
      long long out[P];
      fx_line<N>(F + f * FP + base, st, T, out);
#pragma unroll
      for (int m = 0; m < P; ++m) S[f * FP + base + m * st] = out[m];
    }
    __syncthreads();
    if (node) {
      const int sh = min(xm + 1 - (d == 0 ? x0 : d == 1 ? x1 : x2), 62);
      const long long half = 1ll << (sh - 1);  // the shift below rounds
      auto use = [&](long long& h, long long& m, int slot, int c) {
        const long long x = S[slot * FP + at];  // (its low part from 0: the metric's has no mean)
        fx_mac(h, m, B[c], (int)((unsigned)x & kFxMask), (int)(x >> kFxBits));
      };
      auto eq = [&](int v, int s0, int s1, int s2) {
        long long h = half, m = kFxHalf;
        use(h, m, s0, 0);
        use(h, m, s1, 1);
        use(h, m, s2, 2);
        sum[v] += fx_sum(h, m) >> sh;  // (nine products below 2^60, halved: below 2^63)
      };
      eq(0, sUx, sUy, sUz);
      eq(1, sTxx, sTxy, sTxz);
      eq(2, sTxy, sTyy, sTyz);
      eq(3, sTxz, sTyz, sTzz);
      eq(4, sHx, sHy, sHz);
    }
    if (d < 2) __syncthreads();
  };
  direction(std::integral_constant<int, 0>());
  direction(std::integral_constant<int, 1>());
  direction(std::integral_constant<int, 2>());
  if (node && ok) {
    if constexpr (EPB > 1) ge = fx_exps(gmax[nel]);
    const int kx = xm + 1 + a.fxexp + fx_weight_exp(a.fxw, l % P, (l / P) % P, l / PP);
    double* re = static_cast<double*>(a.re) + n0 + tid;
#pragma unroll
    for (int v = 0; v < 5; ++v)
      re[v * Nl] = fx_to_double(sum[v], kx + (v == 0 ? ge.U : v == 4 ? ge.t : ge.m));
  }
  if constexpr (EPB > 1) {
    for (int t = 0; t < ne; ++t)  // (uniform over the CTA)
      if (a.fxE[e0 + t].w || !fx_in_range(gmax[t])) nodal_plain<N>(a, e0 + t);
  }
}

// CTAs an SM holds at r registers a thread.  64 registers for both forms: the
// rectilinear one at N = 4 took 0.188, 0.177, 0.182 and 0.156 ms with 40, 48, 56
// and 64 (12 to 8 CTAs an SM); the per-node one 0.531, 0.520, 0.531 and 0.554 ms
// with 56, 64, 72 and 80 (at N = 3 80 are 4% better).
__host__ __device__ constexpr int fx_blocks(int threads, int r) { return 65536 / (threads * r); }

template <int N>
__global__ void __launch_bounds__(fx_rect_threads<N>(), fx_blocks(fx_rect_threads<N>(), 64))
    volume_fx_rect_kernel(const __grid_constant__ VolumeArgs a, const __grid_constant__ FxTables<N, 3> T) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int EPB = fx_rect_epb<N>();
  const int e = (int)blockIdx.x * EPB;
  if (a.fxD == nullptr) grid_wait();
  volume_fx_rect<N>(a, T.d, a.ebeg + (long long)e, min(EPB, a.ecnt - e), smem_raw);
}

template <int N>
__global__ void __launch_bounds__(fx_nodal_threads<N>(), fx_blocks(fx_nodal_threads<N>(), N == 3 ? 80 : 64))
    volume_fx_nodal_kernel(const __grid_constant__ VolumeArgs a, const __grid_constant__ FxTables<N, 1> T) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int EPB = fx_nodal_epb<N>();
  const int e = (int)blockIdx.x * EPB;
  volume_fx_nodal<N>(a, T.d, a.ebeg + (long long)e, min(EPB, a.ecnt - e), smem_raw);
}

// Ragged forms: positions of the group are chunks of EPB elements of one
// member, whose tables are copied to shared memory.
template <int N, bool RECT>
__global__ void __launch_bounds__(RECT ? fx_rect_threads<N>() : fx_nodal_threads<N>(),
                                  fx_blocks(RECT ? fx_rect_threads<N>() : fx_nodal_threads<N>(), 64))
    volume_fx_ragged(const MemberDesc* __restrict__ d, const RaggedGroup* __restrict__ g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int EPB = RECT ? fx_rect_epb<N>() : fx_nodal_epb<N>(), ENT = (RECT ? 3 : 1) * fx_table_entries<N>();
  __shared__ int s_m;
  __shared__ long long s_e;
  __shared__ int2 s_T[ENT];
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
      if (a.fxD)  // (read after the barriers of the gather)
        for (int t = threadIdx.x; t < ENT; t += blockDim.x) s_T[t] = a.fxD[t];
      const int ne = (int)min((long long)EPB, a.Ne - s_e);
      if constexpr (RECT) volume_fx_rect<N>(a, s_T, s_e, ne, smem_raw);
      else volume_fx_nodal<N>(a, s_T, s_e, ne, smem_raw);
    }
    __syncthreads();
  }
}

// At bind: rows 0..8 of one element's metric array, dxi_d/dx_c, become
// -Jw dxi_d/dx_c as 58-bit integers (fx_of) relative to the largest of their
// direction in the element, after division by the power of two
// fx_weight_exp of the node's quadrature weight (the weights of a corner and
// of the centre differ by up to 2^13 at N = 8); their biased exponents go to
// fxE.  Elements whose values the integers cannot hold keep doubles (w = 1).
template <int UNUSED = 0>
__global__ void __launch_bounds__(128)
    fx_metric_kernel(double* met, int4* fxE, long long Nl, int P, unsigned long long fxw) {
  __shared__ unsigned s_key[3];
  const int NP = P * P * P;
  const long long n0 = (long long)blockIdx.x * NP;
  if (threadIdx.x < 3) s_key[threadIdx.x] = 0u;
  __syncthreads();
  for (int l = threadIdx.x; l < NP; l += blockDim.x) {
    const double jw = -met[9 * Nl + n0 + l];
    const int we = fx_weight_exp(fxw, l % P, (l / P) % P, l / (P * P));
    for (int t = 0; t < 9; ++t) {
      const double b = met[t * Nl + n0 + l] * jw;
      met[t * Nl + n0 + l] = b;
      const double x = scalbn(b, -we);
      atomicMax(&s_key[t / 3], (unsigned)__double2hiint(x) & 0x7fffffffu);
    }
  }
  __syncthreads();
  const int E[3] = {(int)(s_key[0] >> 20), (int)(s_key[1] >> 20), (int)(s_key[2] >> 20)};
  bool ok = true;
  for (int d = 0; d < 3; ++d) ok &= E[d] >= kFxMetMin && E[d] <= kFxMetMax;
  if (threadIdx.x == 0) fxE[blockIdx.x] = make_int4(E[0], E[1], E[2], ok ? 0 : 1);
  if (!ok) return;
  for (int l = threadIdx.x; l < NP; l += blockDim.x) {
    const int we = fx_weight_exp(fxw, l % P, (l / P) % P, l / (P * P));
    for (int t = 0; t < 9; ++t) {
      double* m = met + t * Nl + n0 + l;
      *reinterpret_cast<int2*>(m) = fx_split(fx_of(scalbn(*m, -we), E[t / 3]));
    }
  }
}

}  // namespace
}  // namespace numa
