// FP64 element kernels with their contractions in 64-bit fixed point on the
// integer pipe (sm_103a).
//
// GB300 issues 2 FP64 operations per SM per clock and 32 32x32+64-bit integer
// multiply-adds (IMAD.WIDE), so a product of two 58-bit numbers in three of
// them costs 3 cycles of the SM per warp against 16 for an FP64 FMA.  The flux
// fields of an element are 58- or 59-bit integers relative to the largest value of
// their equation in the element (a power of two), with the directions scaled by
// the size of their metric terms (FxScale); D is a 59- or 60-bit integer relative to
// its largest row sum, and their products are summed exactly in 64-bit
// accumulators.  What is dropped is a few units of 2^-58 (2^-56 where equations
// share a unit, fx_join) of max_c K_c |F_vc| x (row sum of |D|), K_c the metric
// terms' size along c: the size whose 2^-53 an FP64 chain loses at every step, on
// elements of any aspect.
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
  return 8 * (size_t)15 * EPB * fx_pitch<N>() + sizeof(FxKeys) * fx_slots<EPB, fx_rect_threads<N>()>();
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
  return 8 * (size_t)(2 * kLF) * EPB * fx_pitch<N>() + sizeof(FxKeys) * fx_slots<EPB, fx_nodal_threads<N>()>();
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

// An element's scale, ten bits a direction, in the last word of its metric exponents.
__device__ __forceinline__ FxScale fx_scale_of(int packed) {
  return {{packed & 1023, (packed >> 10) & 1023, (packed >> 20) & 1023}};
}
// The exponents of element t of the CTA (EPB > 1: they take its keys' place).
__device__ __forceinline__ const FxExp& fx_slot(const FxKeys* keys, int t) {
  return reinterpret_cast<const FxExp*>(keys)[t];
}

// The largest of a warp's keys, in every lane; keys raised to at least k's.
__device__ __forceinline__ FxKeys fx_warp_max(FxKeys k) {
  k.U = __reduce_max_sync(0xffffffffu, k.U);
  k.th = __reduce_max_sync(0xffffffffu, k.th);
  k.pp = __reduce_max_sync(0xffffffffu, k.pp);
#pragma unroll
  for (int c = 0; c < 3; ++c) k.u[c] = __reduce_max_sync(0xffffffffu, k.u[c]);
  return k;
}
__device__ __forceinline__ void fx_raise(FxKeys* keys, const FxKeys& k) {
  atomicMax(&keys->U, k.U);
  atomicMax(&keys->th, k.th);
  atomicMax(&keys->pp, k.pp);
#pragma unroll
  for (int c = 0; c < 3; ++c) atomicMax(&keys->u[c], k.u[c]);
}
// The most elements (of NP nodes each, NN in all) that the nodes of one warp belong to.
template <int NP, int NN>
__host__ __device__ constexpr int fx_warp_elements() {
  int most = 0;
  for (int l = 0; l < NN; l += 32) {
    const int last = l + 31 < NN ? l + 31 : NN - 1, n = last / NP - l / NP + 1;
    if (n > most) most = n;
  }
  return most;
}

// Gathers U, u, theta and p' at the nodes of the ne elements from e0, one thread per
// element node, and leaves their flux fields in F as fixed-point integers (15
// for the rectilinear form, 12 for the per-node form).  The largest magnitudes
// in an element give its groups' exponents: returned in ge for the thread's own
// element node, and with several elements left in shared memory (fx_slot) for
// every element.  The fields of an element that the integers cannot hold (ok = 0)
// are left unset: no element's result depends on which others share its CTA (a
// slab launch groups them otherwise).  w: the scale of the thread's element.
template <int N, int EPB, int NT, bool RECT>
__device__ __forceinline__ void fx_stage(const VolumeArgs& a, long long e0, int ne, FxKeys* keys, int2* F,
                                         const FxScale& w, FxExp& ge) {
  constexpr int NP = (N + 1) * (N + 1) * (N + 1), NN = EPB * NP, IT = (NN + NT - 1) / NT;
  constexpr int FP = EPB * fx_pitch<N>(), SLOTS = fx_slots<EPB, NT>();
  static_assert((RECT && EPB == 1) || IT == 1, "one node per thread");
  const int tid = threadIdx.x, nn = ne * NP;
  int packed = 0;  // of the element whose exponents the thread forms below
  if constexpr (EPB > 1) {
    if (!RECT && tid < ne) packed = a.fxE[e0 + tid].w;
    if (tid < EPB) keys[tid] = FxKeys();
    __syncthreads();
  }
  FxKeys g = FxKeys();
  NodeState64 z[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int l = tid + it * NT;
    if (l < nn) {
      z[it] = gather_node64(a, e0 * NP + l);
      if constexpr (EPB == 1) {  // (without the low words: see below)
        g.U = max(g.U, fx_high_scaled(z[it].U, w));
#pragma unroll
        for (int c = 0; c < 3; ++c) g.u[c] = max(g.u[c], fx_high(z[it].u[c]));
        g.th = max(g.th, fx_high(z[it].th));
        g.pp = max(g.pp, fx_high(z[it].pp));
      } else {
        g.U = fx_key_scaled(z[it].U, w);
#pragma unroll
        for (int c = 0; c < 3; ++c) g.u[c] = fx_key(z[it].u[c]);
        g.th = fx_key(z[it].th);
        g.pp = fx_key(z[it].pp);
      }
    }
  }
  if constexpr (EPB == 1) {
    g = fx_warp_max(g);
    if ((tid & 31) == 0) keys[tid >> 5] = g;
  } else if constexpr (fx_warp_elements<NP, NN>() <= 2) {
    // the warp's elements one after the other (an atomic per lane, 27 to 32 of them in
    // turn on one address: 0.211 ms instead of 0.179 on 50^3 elements at N = 2, 0.228
    // instead of 0.186 on 40^3 at N = 3)
#pragma unroll
    for (int j = 0; j < fx_warp_elements<NP, NN>(); ++j) {
      const int t = (tid & ~31) / NP + j;
      const FxKeys k = fx_warp_max(tid < nn && tid / NP == t ? g : FxKeys());
      if ((tid & 31) == 0 && t < ne) fx_raise(keys + t, k);
    }
  } else {
    if (tid < nn) fx_raise(keys + tid / NP, g);
  }
  grid_wait();  // (threads without a node; before any write of the kernel)
  __syncthreads();
  if constexpr (EPB == 1) {
    // every warp by itself: lane j (of eight) the largest of key j; lanes 4 to 6 the
    // exponents of the three momentum equations
    const int lane = tid & 7;
    const unsigned* q = reinterpret_cast<const unsigned*>(keys) + lane;
    unsigned k = 0;
#pragma unroll
    for (int t = 0; t < SLOTS; ++t) k = max(k, q[8 * t]);
    const unsigned U = __shfl_sync(0xffffffffu, k, 0), th = __shfl_sync(0xffffffffu, k, 1);
    const unsigned pp = __shfl_sync(0xffffffffu, k, 2);
    bool in;
    const int m = fx_momentum_exp(U, k, pp, lane == 4 ? w.s[0] : lane == 5 ? w.s[1] : w.s[2], in);
    const bool ok = fx_scalar_exps(ge, U, th, pp);
    ge.ok = __all_sync(0xffffffffu, ok && (in || lane < 4 || lane == 7));
#pragma unroll
    for (int c = 0; c < 3; ++c) ge.m[c] = __shfl_sync(0xffffffffu, m, 4 + c);
    fx_join(ge, w);
    if (__any_sync(0xffffffffu, k == 0 && lane != 3 && lane != 7)) {  // (uniform over the CTA)
      // a group that is zero, or whose values lie below 2^-1042 (plain FP64 then)
      bool zero[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) zero[c] = __shfl_sync(0xffffffffu, k, 4 + c) == 0;
      unsigned low = 0;
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        if (tid + it * NT < nn) {
          if (U == 0) low |= fx_key(z[it].U[0]) | fx_key(z[it].U[1]) | fx_key(z[it].U[2]);
#pragma unroll
          for (int c = 0; c < 3; ++c)
            if (zero[c]) low |= fx_key(z[it].u[c]);
          if (th == 0) low |= fx_key(z[it].th);
          if (pp == 0) low |= fx_key(z[it].pp);
        }
      }
      if (__syncthreads_or(low != 0)) ge.ok = 0;
    }
  } else {
    if (tid < ne) {
      FxExp e = fx_exps(keys[tid], RECT ? w : fx_scale_of(packed));
      if (packed < 0) e.ok = 0;
      *reinterpret_cast<FxExp*>(keys + tid) = e;
    }
    __syncthreads();
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int l = tid + it * NT;
    if (l < nn) {
      if constexpr (EPB > 1) ge = fx_slot(keys, l / NP);
      if (ge.ok) {
        int2* f = F + fx_index<N>(l);
        auto put = [&](int slot, int2 x) { f[slot * FP] = x; };
        if constexpr (RECT) fx_fluxes(z[it], ge, w, put);
        else fx_fluxes_shared(z[it], ge, w, put);
      }
    }
  }
}

// create_rhs of up to fx_rect_epb<N>() rectilinear elements e0 .. e0 + ne - 1
// in fixed point: the residual sum_d K_d (D F_d) without its weight
// w_i w_j w_k (which the update applies with the inverse mass).
//   1. the 15 flux fields (of equation v along direction d: 5 d + v) go to
//      shared memory (fx_stage);
//   2. thread t takes line t of the 5 (N+1)^2 lines along x (equation
//      v = t / (N+1)^2), then along y (fx_line), and leaves the derivatives in
//      the line's place: each line of a field is read by one thread only;
//   3. it then takes its line along z, adds the x and y derivatives at the
//      line's nodes as integers and converts the sums to FP64, rounded once.
// On 32^3 elements at N = 4: 0.529 ms as FP64 (its pipe 97% busy: 75 operations
// a node at 16 cycles a warp), 0.164 ms here on the rising bubble (0.172 where the
// momentum equations' units differ); 19x23x17 at N = 6: 0.460 -> 0.132 ms, 12^3 at
// N = 8 0.090 ms.  135 to 144 integer multiply-adds a thread; the instructions beside
// them (1030 a warp) and shared memory are what is left.  One unit for
// all of momentum and one scale took 0.154 ms, with an error that grew with an
// element's aspect.  D in the kernel parameters instead of global memory: 0.256 ->
// 0.226 ms; the z lines finishing the nodes (10 shared accesses a node fewer):
// 0.226 -> 0.216; the products formed here from 8 gathered fields instead of 12
// gathered fluxes: 0.216 -> 0.186 (and the update 0.199 -> 0.169 ms); the results
// converted by the FP64 pipe and 64 registers: 0.186 -> 0.156.  Derivatives in the
// lines' place (15 fields of shared memory, not 22): N = 8 0.132 -> 0.090 ms.
template <int N>
__device__ __forceinline__ void volume_fx_rect(const VolumeArgs& a, const int2* T, long long e0, int ne,
                                               unsigned char* smem_raw) {
  constexpr int P = N + 1, PP = P * P, NP = PP * P, EPB = fx_rect_epb<N>(), NT = fx_rect_threads<N>();
  constexpr int EP = fx_pitch<N>(), FP = EPB * EP, M = fx_table_entries<N>(), B = fx_plane<N>();
  FxKeys* keys = reinterpret_cast<FxKeys*>(smem_raw);              // (first: 16-byte aligned)
  int2* F = reinterpret_cast<int2*>(keys + fx_slots<EPB, NT>());  // [15][FP]
  const int tid = threadIdx.x;
  const long long n0 = e0 * NP;
  const FxScale w = {{a.fxs[0], a.fxs[1], a.fxs[2]}};
  FxExp ge;
  if (a.fxD == nullptr) {
    for (int t = 0; t < ne; ++t) rect_plain<N>(a, e0 + t);
    return;
  }
  fx_stage<N, EPB, NT, true>(a, e0, ne, keys, F, w, ge);
  if (EPB == 1 && !ge.ok) {  // (uniform over the CTA)
    rect_plain<N>(a, e0);
    return;
  }
  __syncthreads();
  const bool act = tid < ne * 5 * PP;
  const int el = EPB == 1 ? 0 : tid / (5 * PP), tt = tid - el * 5 * PP;
  const int v = tt / PP, r = tt - v * PP;
  if (act) {
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      int2* f = F + (5 * d + v) * FP + el * EP + fx_line_base<N>(d, r);
      const int st = fx_line_stride<N>(d);
      long long out[P];
      fx_line<N>(f, st, T + d * M, out);
#pragma unroll
      for (int m = 0; m < P; ++m) f[m * st] = make_int2((int)out[m], (int)(out[m] >> 32));
    }
  }
  __syncthreads();
  if (act) {
    const int2* o = F + v * FP + el * EP + fx_line_base<N>(2, r);
    long long out[P];
    fx_line<N>(o + 10 * FP, B, T + 2 * M, out);
    if constexpr (EPB > 1) ge = fx_slot(keys, el);
    if (ge.ok) {
      const int kexp = (v == 0 ? ge.U : v == 4 ? ge.t : ge.m[v == 1 ? 0 : v == 2 ? 1 : 2]) + a.fxexp;
      double* re = static_cast<double*>(a.re) + v * a.Nl + n0 + el * NP + r;
      auto value = [&](int2 x) { return (long long)x.y << 32 | (unsigned)x.x; };
#pragma unroll
      for (int m = 0; m < P; ++m) re[m * PP] = fx_to_double(out[m] + value(o[m * B]) + value(o[5 * FP + m * B]), kexp);
    }
  }
  if constexpr (EPB > 1) {
    if (__syncthreads_or(act && !ge.ok)) {
      for (int t = 0; t < ne; ++t)
        if (!fx_slot(keys, t).ok) rect_plain<N>(a, e0 + t);
    }
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
          // eb.w < 0: the metric terms of this element stayed doubles
          const long long at = (3 * d + c) * Nl + e * NP + l;
          double b = a.met64[at];
          if (eb.w >= 0) {
            const int2 h = reinterpret_cast<const int2*>(a.met64)[at];
            const int E = (d == 0 ? eb.x : d == 1 ? eb.y : eb.z) - fx_scale_of(eb.w).s[c];
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
//      row of -Jw dxi_d/dx_c (58-bit integers, fx_metric_kernel) into the five
//      equations, those of U_a u_b aligned to the equation's unit (fx_pair).
// Every row of D is scaled to its own row sum (an end row's is up to 16 times
// an inner one's).  The directions' sums are aligned by the exponents of their
// rows, added as integers and rounded once.
// On the 6x30x30x8 shell at N = 4: 2.068 ms as FP64 (225 operations a node, its
// pipe 96% busy), 0.580 ms here; 21x17x13 at N = 3: 0.105 -> 0.039 ms.  The 421
// integer multiply-adds a thread keep their pipe 40% busy and the 2515
// instructions a warp 60% of the issue slots.  One unit for all of momentum and one
// scale for the directions took 0.517 and 0.039 ms, with the error stated at
// FxScale; of the difference on the shell, the exponents and keys are 0.017 ms, the
// alignment 0.011, the choice between U_a u_b and U_b u_a 0.020.  With the fluxes formed in the
// update the kernel was 0.035 ms shorter, and the update 0.041 longer.  Going round
// all lines of a direction with a division per line instead of one line per
// thread: 0.065 ms more.
template <int N>
__device__ __forceinline__ void volume_fx_nodal(const VolumeArgs& a, const int2* T, long long e0, int ne,
                                                unsigned char* smem_raw) {
  constexpr int P = N + 1, PP = P * P, NP = PP * P, EPB = fx_nodal_epb<N>(), NT = fx_nodal_threads<N>();
  constexpr int EP = fx_pitch<N>(), FP = EPB * EP;
  FxKeys* keys = reinterpret_cast<FxKeys*>(smem_raw);              // (first: 16-byte aligned)
  int2* F = reinterpret_cast<int2*>(keys + fx_slots<EPB, NT>());  // [kLF][FP]
  long long* S = reinterpret_cast<long long*>(F + kLF * FP);       // [kLF][FP]: the direction's derivatives
  const int tid = threadIdx.x, nn = ne * NP;
  const long long Nl = a.Nl, n0 = e0 * NP;
  const bool node = tid < nn;
  const int nel = EPB == 1 ? 0 : tid / NP;
  // the elements' metric exponents and scale (w < 0: the element takes plain FP64)
  const int4 eb = a.fxE[e0 + (node ? nel : 0)];
  const FxScale w = fx_scale_of(eb.w);
  FxExp ge;
  fx_stage<N, EPB, NT, false>(a, e0, ne, keys, F, w, ge);
  const bool ok = ge.ok && (EPB > 1 || eb.w >= 0);
  if (EPB == 1 && !ok) {  // (uniform over the CTA)
    nodal_plain<N>(a, e0);
    return;
  }
  __syncthreads();
  // (positive: equation a shifts the derivative of U_a u_b, negative: equation b)
  const int xy = fx_pair(ge, w, 0, 1), xz = fx_pair(ge, w, 0, 2), yz = fx_pair(ge, w, 1, 2);
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
      auto use = [&](long long& h, long long& m, int slot, int c, int by) {
        const long long x = fx_shift(S[slot * FP + at], by);  // (its low part from 0: the metric's has no mean)
        fx_mac(h, m, B[c], (int)((unsigned)x & kFxMask), (int)(x >> kFxBits));
      };
      auto eq = [&](int v, int s0, int b0, int s1, int b1, int s2, int b2) {
        long long h = half, m = kFxHalf;
        use(h, m, s0, 0, b0);
        use(h, m, s1, 1, b1);
        use(h, m, s2, 2, b2);
        sum[v] += fx_sum(h, m) >> sh;  // (nine products below 1.5 2^59, halved: below 2^63)
      };
      eq(0, sUx, 0, sUy, 0, sUz, 0);
      eq(1, sTxx, 0, sTxy, xy, sTxz, xz);
      eq(2, sTxy, -xy, sTyy, 0, sTyz, yz);
      eq(3, sTxz, -xz, sTyz, -yz, sTzz, 0);
      eq(4, sHx, 0, sHy, 0, sHz, 0);
    }
    if (d < 2) __syncthreads();
  };
  direction(std::integral_constant<int, 0>());
  direction(std::integral_constant<int, 1>());
  direction(std::integral_constant<int, 2>());
  if (node && ok) {
    const int kx = xm + 1 + a.fxexp + fx_weight_exp(a.fxw, l % P, (l / P) % P, l / PP);
    double* re = static_cast<double*>(a.re) + n0 + tid;
#pragma unroll
    for (int v = 0; v < 5; ++v)
      re[v * Nl] = fx_to_double(sum[v], kx + (v == 0 ? ge.U : v == 4 ? ge.t : ge.m[(v + 2) % 3]));
  }
  if constexpr (EPB > 1) {
    if (__syncthreads_or(node && !ok)) {
      for (int t = 0; t < ne; ++t)
        if (!fx_slot(keys, t).ok) nodal_plain<N>(a, e0 + t);
    }
  }
}

// CTAs an SM holds at r registers a thread.  64 registers: the rectilinear form
// at N = 4 took 0.188, 0.177, 0.182 and 0.156 ms with 40, 48, 56 and 64 (12 to 8
// CTAs an SM; measured with one momentum unit).  The per-node form takes 72 at N = 4 (0.588 ->
// 0.578 ms on the shell) and 80 at N = 3 (4% better than 64).
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
__global__ void __launch_bounds__(fx_nodal_threads<N>(), fx_blocks(fx_nodal_threads<N>(), N == 3 ? 80 : N == 4 ? 72 : 64))
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
// -Jw dxi_d/dx_c as 58-bit integers, after division by the power of two
// fx_weight_exp of the node's quadrature weight (the weights of a corner and
// of the centre differ by up to 2^13 at N = 8) and multiplication by 2^s_c, which
// makes the largest of the three terms of each c equal to within a factor of
// two (FxScale): fx_of relative to the largest of their direction d in the element.
// The three biased exponents and the scale go to fxE.  Elements whose values the
// integers cannot hold keep doubles (w = -1).
template <int UNUSED = 0>
__global__ void __launch_bounds__(128)
    fx_metric_kernel(double* met, int4* fxE, long long Nl, int P, unsigned long long fxw) {
  __shared__ unsigned s_key[9];
  const int NP = P * P * P;
  const long long n0 = (long long)blockIdx.x * NP;
  if (threadIdx.x < 9) s_key[threadIdx.x] = 0u;
  __syncthreads();
  for (int l = threadIdx.x; l < NP; l += blockDim.x) {
    const double jw = -met[9 * Nl + n0 + l];
    const int we = fx_weight_exp(fxw, l % P, (l / P) % P, l / (P * P));
    for (int t = 0; t < 9; ++t) {
      const double b = met[t * Nl + n0 + l] * jw;
      met[t * Nl + n0 + l] = b;
      const double x = scalbn(b, -we);
      atomicMax(&s_key[t], (unsigned)__double2hiint(x) & 0x7fffffffu);
    }
  }
  __syncthreads();
  int k[9], col[3], E[3] = {0, 0, 0};
  bool ok = true;
  for (int t = 0; t < 9; ++t) {
    k[t] = (int)(s_key[t] >> 20);
    ok &= k[t] <= kFxMetMax;  // (no infinity, no NaN)
  }
  for (int c = 0; c < 3; ++c) col[c] = max(k[c], max(k[3 + c], k[6 + c]));
  const int top = max(col[0], max(col[1], col[2]));
  // (columns within a factor of four of each other: one scale, see fx_join)
  if (top - min(col[0], min(col[1], col[2])) <= 1) col[0] = col[1] = col[2] = top;
  for (int c = 0; c < 3; ++c) {
    ok &= top - col[c] <= kFxMaxScale;
    for (int d = 0; d < 3; ++d) E[d] = max(E[d], k[3 * d + c] + top - col[c]);
  }
  for (int d = 0; d < 3; ++d) ok &= E[d] >= kFxMetMin && E[d] <= kFxMetMax;
  const int w = (top - col[0]) | (top - col[1]) << 10 | (top - col[2]) << 20;
  if (threadIdx.x == 0) fxE[blockIdx.x] = make_int4(E[0], E[1], E[2], ok ? w : -1);
  if (!ok) return;
  for (int l = threadIdx.x; l < NP; l += blockDim.x) {
    const int we = fx_weight_exp(fxw, l % P, (l / P) % P, l / (P * P));
    for (int t = 0; t < 9; ++t) {
      double* m = met + t * Nl + n0 + l;
      *reinterpret_cast<int2*>(m) = fx_split(fx_of(scalbn(*m, -we), E[t / 3] - (top - col[t % 3])));
    }
  }
}

}  // namespace
}  // namespace numa
