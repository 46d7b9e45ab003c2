// Column part of the 1D-IMEX leapfrog step (Sec. 2.2: an explicit leapfrog
// step, then implicit corrections along each vertical column of grid points;
// the IMEX line of the time loop in Sec. 7), for the z-columns of a box and
// the radial columns of the cubed-sphere shell.
//
// With the explicit tendency R = R(q^n) already in memory, per column:
//   q*  = qprev + cR R                      (cR = 2 dt; dt on the start step)
//   s   = 2 q^n - qprev                     (q^0 on the start step)
//   solve (I - tau L) x = q* - tau L s for rho', W, Theta'; U, V take q*.
// L couples rho', W (the momentum along the column) and Theta' through the
// column derivative Dz and the divergence G = Dz + 2/r (G = Dz in the box);
// eliminating rho' and Theta' leaves the Schur system H x_W = f in W,
//   H = I - tau^2 (Dz C2 G T0 + g G)        (identity rows at the walls),
// which in the increment y = x_W - s reads
//   H y = q*_W - s_W - tau g (q*_rho - s_rho) + tau Dz(c2 (s_Theta - q*_Theta))
// (q*_W - s_W at the walls), after which
//   x_W = s_W + y,  x_rho = q*_rho - tau G y,  x_Theta = q*_Theta - tau G(theta0 y).
// The Robert-Asselin filter gives qbar^n = q^n + nu (qprev - 2 q^n + x).
//
// One block holds cols_per_block consecutive columns.  Shared memory keeps
// the two vectors whose neighbours the column derivative reads ([2][nz][cols]
// doubles) and, in the integer form, six values that the same thread needs
// again at the end (q*_rho, s_W, q*_Theta and the filter's first part); the LU
// form leaves those in R and qbar^n.  The derivative applications run over
// all (level, column) pairs of the block.
//
// Columns of up to kImexDense levels (DENSE): y = H^-1 r with the inverse as
// fixed-point integers, and its derivatives likewise (fixed64.cuh), r in 56
// bits relative to the largest value of its column.  A level is nz products
// of three integer multiply-adds, all levels at once, against the 16 to 24
// FP64 operations of the LU sweeps (16 cycles of an SM a warp each, one thread
// per column level by level): at 33 levels 99 cycles against 320.  The inverse
// is refined beyond FP64 on the host.  On the thin box of 64x64x8 elements at
// N = 4 the DSS and this kernel went from 0.398 to 0.348 ms a step.  All loads
// of a phase before its first store (0.348 -> 0.322 ms with 128 threads, 0.313
// with 256), and the six values in shared memory instead of global memory with
// up to 384 threads, three blocks an SM (0.309 ms; the shell 0.551 -> 0.509);
// two blocks an SM and no spills: 0.325.  The FP64 operations of the explicit
// step, the first derivative and the filter (0.154 ms of their pipe) bound it
// now.  Taller columns take the LU factors, one thread per column running the
// banded sweeps.
#include "fixed64.cuh"

namespace numa {
namespace {

constexpr int kImexThreads = 128, kImexDenseThreads = 384;
constexpr size_t kImexSmemMax = 200 * 1024;
constexpr int kImexMinExp = 200, kImexMaxExp = 1800;  // biased exponents of a column's r taken as they are

// Band entries [j0, j1] of row k of Dz that can be nonzero: the row of a node
// inside element e couples to that element's N+1 nodes; a node shared by two
// elements (k a multiple of N) to both elements' nodes.
__device__ __forceinline__ void dz_row_range(int k, int N, int nz, int& j0, int& j1) {
  const int i = k % N;
  if (i == 0) {
    j0 = max(0, N - k);
    j1 = min(2 * N, nz - 1 - k + N);
  } else {
    j0 = N - i;  // column k - i, the element's first node
    j1 = 2 * N - i;
  }
}

// Column c, level k is global node c + ncol k.  RADIAL = false: z-columns of
// the box (W = U_z); RADIAL = true: radial columns of the shell (W = U . r_hat,
// U^{n+1} = U* + (x_W - W*) r_hat).
template <bool RADIAL, bool DENSE>
__global__ void __launch_bounds__(DENSE ? kImexDenseThreads : kImexThreads, DENSE ? 3 : 4) imex_column_kernel(ImexArgs a) {
  extern __shared__ __align__(16) double sm[];
  const int nz = a.nz, CPB = a.cols_per_block, N = a.N, W2 = 2 * a.N + 1, kl = a.kl, US = 1 + 4 * a.N;
  const long long Ng = a.Ng, ncol = a.ncol;
  const size_t plane = (size_t)nz * CPB;
  double* UT = sm;          // c2 (s_Theta - q*_Theta), then theta0 y
  double* EY = sm + plane;  // e, then r (right-hand side of H y = r), then y
  // the factors, read on the serial path of the sweeps, staged once per block
  double* Ls = EY + plane;                   // [nz][kl]
  double* Us = Ls + (size_t)nz * kl;         // [nz][1 + 4N]
  int* Ps = reinterpret_cast<int*>(Us + (size_t)nz * US);  // [nz][3]
  // DENSE: q*_rho, s_W, q*_Theta and qbar^n of rho', W, Theta' without x, [6][nz][cols],
  // then [CPB] largest |r| of each column (high word)
  double* PK = EY + plane;
  unsigned* key = reinterpret_cast<unsigned*>(PK + 6 * plane);
  if constexpr (DENSE) {
    if (threadIdx.x < CPB) key[threadIdx.x] = 0u;
  } else {
    for (int t = threadIdx.x; t < nz * kl; t += blockDim.x) Ls[t] = a.Lf[t];
    for (int t = threadIdx.x; t < nz * US; t += blockDim.x) Us[t] = a.Uf[t];
    for (int t = threadIdx.x; t < 3 * nz; t += blockDim.x) Ps[t] = a.piv[t];
  }
  double* R = a.R;
  const long long col0 = (long long)blockIdx.x * CPB;
  const double nu = a.nu, tau = a.tau;
  const int items = nz * CPB;
  auto node = [&](long long col, int k) -> long long { return col + ncol * k; };

  // explicit step, the filter's first part; U and V finished in the box,
  // U* parked in q on the shell
  for (int t = threadIdx.x; t < items; t += blockDim.x) {
    const int k = t / CPB, cl = t - k * CPB;
    const long long col = col0 + cl;
    if (col >= ncol) continue;
    const long long g = node(col, k);
    // (all loads before the first store, which the compiler cannot move them over)
    double qst[5], sv[5], qn[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      qn[v] = a.q[v * Ng + g];
      sv[v] = a.qprev[v * Ng + g];
      qst[v] = R[v * Ng + g];
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const double qp = sv[v];
      qst[v] = fma(a.cR, qst[v], qp);
      sv[v] = fma(2.0, qn[v], -qp);  // s = 2 q^n - qprev, so qprev - 2 q^n = -s
      if (!RADIAL && (v == 1 || v == 2)) {
        a.q[v * Ng + g] = qst[v];
        a.qs[v * Ng + g] = fma(nu, qst[v] - sv[v], qn[v]);  // x = q* for U and V
      } else {
        if (RADIAL && v >= 1 && v <= 3) a.q[v * Ng + g] = qst[v];
        const double b = fma(-nu, sv[v], qn[v]);  // q^n + nu (qprev - 2 q^n)
        if (DENSE && (v == 0 || v >= 3)) PK[(v == 0 ? 3 : v + 1) * plane + t] = b;
        else a.qs[v * Ng + g] = b;
      }
    }
    double wst = qst[3], swv = sv[3];
    if constexpr (RADIAL) {
      const double nx = a.nrm[g], ny = a.nrm[Ng + g], nz_ = a.nrm[2 * Ng + g];
      wst = fma(qst[1], nx, fma(qst[2], ny, qst[3] * nz_));
      swv = fma(sv[1], nx, fma(sv[2], ny, sv[3] * nz_));
      R[Ng + g] = wst;
    }
    if constexpr (DENSE) {
      PK[t] = qst[0];
      PK[plane + t] = swv;
      PK[2 * plane + t] = qst[4];
    } else {
      R[g] = qst[0];
      R[3 * Ng + g] = swv;
      R[4 * Ng + g] = qst[4];
    }
    const size_t o = (size_t)k * CPB + cl;
    UT[o] = a.c2[k] * (sv[4] - qst[4]);
    const double e = wst - swv;
    EY[o] = (k == 0 || k == nz - 1) ? e : fma(-tau * a.gl[k], qst[0] - sv[0], e);
  }
  __syncthreads();

  // r = e + tau Dz(c2 (s_Theta - q*_Theta)) on the interior rows
  for (int t = threadIdx.x; t < items; t += blockDim.x) {
    const int k = t / CPB, cl = t - k * CPB;
    if (k > 0 && k < nz - 1) {
      int j0, j1;
      dz_row_range(k, N, nz, j0, j1);
      double acc = 0.0;
      for (int j = j0; j <= j1; ++j) acc = fma(a.Dz[k * W2 + j], UT[(size_t)(k - N + j) * CPB + cl], acc);
      EY[(size_t)k * CPB + cl] = fma(tau, acc, EY[(size_t)k * CPB + cl]);
    }
    if constexpr (DENSE)
      if (col0 + cl < ncol) atomicMax(&key[cl], (unsigned)__double2hiint(EY[(size_t)k * CPB + cl]) & 0x7fffffffu);
  }
  __syncthreads();

  // exponent of a column's r; above kImexMaxExp (infinities and NaN too) the
  // column's y is NaN, as the sweeps would make it
  auto col_exp = [&](int cl) { return key[cl] ? max((int)(key[cl] >> 20), kImexMinExp) : 1023; };
  int2* Ri = reinterpret_cast<int2*>(EY);           // DENSE: r, then
  long long* Yi = reinterpret_cast<long long*>(UT);  // y
  if constexpr (DENSE) {
    for (int t = threadIdx.x; t < items; t += blockDim.x) {
      const int cl = t % CPB, E = col_exp(cl);
      Ri[t] = col0 + cl < ncol && E <= kImexMaxExp ? fx_split(fx_of(EY[t], E + 2)) : make_int2(0, 0);
    }
    __syncthreads();
    // three levels of one column per thread (a warp's lanes are columns)
    for (int t = threadIdx.x; t < (nz + 2) / 3 * CPB; t += blockDim.x) {
      const int k = t / CPB * 3, cl = t % CPB;
      const int2* H0 = a.Hi + (size_t)k * nz;
      const int2* H1 = k + 1 < nz ? H0 + nz : H0;
      const int2* H2 = k + 2 < nz ? H0 + 2 * nz : H0;
      long long h0 = 0, m0 = kFxHalf, h1 = 0, m1 = kFxHalf, h2 = 0, m2 = kFxHalf;
      for (int j = 0; j < nz; ++j) {
        const int2 r = Ri[j * CPB + cl];
        fx_mac(h0, m0, __ldg(H0 + j), r.x, r.y);
        fx_mac(h1, m1, __ldg(H1 + j), r.x, r.y);
        fx_mac(h2, m2, __ldg(H2 + j), r.x, r.y);
      }
      Yi[k * CPB + cl] = fx_sum(h0, m0);
      if (k + 1 < nz) Yi[(k + 1) * CPB + cl] = fx_sum(h1, m1);
      if (k + 2 < nz) Yi[(k + 2) * CPB + cl] = fx_sum(h2, m2);
    }
  } else {
  // H y = r: forward elimination with the recorded row swaps, back substitution
  for (int cl = threadIdx.x; cl < CPB; cl += blockDim.x) {
    if (col0 + cl >= ncol) break;
    for (int k = 0; k < nz; ++k) {
      const int p = Ps[3 * k];
      double yk = EY[(size_t)k * CPB + cl];
      if (p != k) {
        const double yp = EY[(size_t)p * CPB + cl];
        EY[(size_t)p * CPB + cl] = yk;
        EY[(size_t)k * CPB + cl] = yp;
        yk = yp;
      }
      const int imax = Ps[3 * k + 1];
      for (int i = 1; i <= imax; ++i)
        EY[(size_t)(k + i) * CPB + cl] = fma(-Ls[k * kl + i - 1], yk, EY[(size_t)(k + i) * CPB + cl]);
    }
    for (int k = nz - 1; k >= 0; --k) {
      double acc = EY[(size_t)k * CPB + cl];
      const int jmax = Ps[3 * k + 2];
      for (int j = 1; j <= jmax; ++j) acc = fma(-Us[k * US + j], EY[(size_t)(k + j) * CPB + cl], acc);
      EY[(size_t)k * CPB + cl] = acc * Us[k * US];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < items; t += blockDim.x) UT[t] = a.th0[t / CPB] * EY[t];
  }
  __syncthreads();

  // x_rho = q*_rho - tau G y, x_Theta = q*_Theta - tau G(theta0 y), x_W = s_W + y
  // (G = Dz + 2/r); q^{n+1}, the filtered q^n and the primitive fields of q^{n+1}
  for (int t = threadIdx.x; t < items; t += blockDim.x) {
    const int k = t / CPB, c = t - k * CPB;
    const long long col = col0 + c;
    if (col >= ncol) continue;
    const long long g = node(col, k);
    // (loads first, as above)
    const double R0 = DENSE ? PK[t] : R[g], R3 = DENSE ? PK[plane + t] : R[3 * Ng + g];
    const double R4 = DENSE ? PK[2 * plane + t] : R[4 * Ng + g];
    const double s0 = DENSE ? PK[3 * plane + t] : a.qs[g], s3 = DENSE ? PK[4 * plane + t] : a.qs[3 * Ng + g];
    const double s4 = DENSE ? PK[5 * plane + t] : a.qs[4 * Ng + g];
    const double q1 = a.q[Ng + g], q2 = a.q[2 * Ng + g];
    int j0, j1;
    dz_row_range(k, N, nz, j0, j1);
    const size_t o = (size_t)k * CPB + c;
    double dy = 0.0, dty = 0.0, yk, tyk = 0.0;
    if constexpr (DENSE) {
      long long h = 0, m = kFxHalf, th = 0, tm = kFxHalf;
      for (int j = j0; j <= j1; ++j) {
        const long long y = Yi[(k - N + j) * CPB + c];
        const int yl = (int)((unsigned)y & kFxMask), yh = (int)(y >> kFxBits);
        fx_mac(h, m, __ldg(a.DzI + k * W2 + j), yl, yh);
        fx_mac(th, tm, __ldg(a.DtI + k * W2 + j), yl, yh);
      }
      const int E = col_exp(c);
      const bool bad = E > kImexMaxExp;
      const int Eu = bad ? 1023 : E;
      yk = bad ? __hiloint2double(0x7ff80000, 0) : fx_to_double(Yi[o], Eu + a.y_exp);
      dy = fx_to_double(fx_sum(h, m), Eu + a.d_exp);
      dty = fx_to_double(fx_sum(th, tm), Eu + a.t_exp);
      if (bad) dy = dty = yk;
      if constexpr (RADIAL) tyk = a.th0[k] * yk;
    } else {
      for (int j = j0; j <= j1; ++j) {
        const double d = a.Dz[k * W2 + j];
        const size_t oj = (size_t)(k - N + j) * CPB + c;
        dy = fma(d, EY[oj], dy);
        dty = fma(d, UT[oj], dty);
      }
      yk = EY[o];
      if constexpr (RADIAL) tyk = UT[o];
    }
    if constexpr (RADIAL) {
      dy = fma(a.r2[k], yk, dy);
      dty = fma(a.r2[k], tyk, dty);
    }
    const double xr = fma(-tau, dy, R0);
    const double xw = R3 + yk;
    const double xt = fma(-tau, dty, R4);
    double xu = q1, xv = q2, xz = xw;
    if constexpr (RADIAL) {
      const double dw = xw - R[Ng + g];  // x_W - W*
      xu = fma(dw, a.nrm[g], q1);
      xv = fma(dw, a.nrm[Ng + g], q2);
      xz = fma(dw, a.nrm[2 * Ng + g], a.q[3 * Ng + g]);
      const double s1 = a.qs[Ng + g], s2 = a.qs[2 * Ng + g];
      a.q[Ng + g] = xu;
      a.q[2 * Ng + g] = xv;
      a.qs[Ng + g] = fma(nu, xu, s1);
      a.qs[2 * Ng + g] = fma(nu, xv, s2);
    }
    write_prim<false>(a.pa, g, xr, xu, xv, xz, xt);
    a.q[g] = xr;
    a.q[3 * Ng + g] = xz;
    a.q[4 * Ng + g] = xt;
    a.qs[g] = fma(nu, xr, s0);
    a.qs[3 * Ng + g] = fma(nu, xz, s3);
    a.qs[4 * Ng + g] = fma(nu, xt, s4);
    if (nonfinite(xr) | nonfinite(xu) | nonfinite(xv) | nonfinite(xz) | nonfinite(xt)) atomicOr(a.flag, 1);
  }
}

DeviceFlags imex_attr;

template <bool RADIAL>
cudaError_t set_imex_attr() {
  cudaError_t e = cudaFuncSetAttribute(imex_column_kernel<RADIAL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kImexSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(imex_column_kernel<RADIAL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kImexSmemMax);
  return e;
}

}  // namespace

// Columns per block: kImexColsTarget while a block's shared memory stays
// under kImexSmemMax / 2, fewer for tall columns.
constexpr int kImexColsTarget = 32;
// Levels up to which the integer form takes 32 columns a block (72 KB), 16 above.
constexpr int kImexWide = 36;

int imex_cols_per_block(int nz, int N) {
  for (int c = kImexColsTarget; c >= 32; c /= 2)
    if (imex_smem_bytes(nz, N, c) <= kImexSmemMax / 2) return c;
  for (int c = 16; c >= 1; c /= 2)
    if (imex_smem_bytes(nz, N, c) <= kImexSmemMax) return c;
  return 0;
}

// Two column vectors per column, the factors of one Schur matrix (rows of
// 2N multipliers and 1 + 4N U entries) and the pivot rows.
size_t imex_smem_bytes(int nz, int N, int cols_per_block) {
  return sizeof(double) * (size_t)nz * (2 * (size_t)cols_per_block + 2 * N + 1 + 4 * N) + 3 * sizeof(int) * (size_t)nz;
}

// The integer form: eight vectors per column and a key.
static size_t imex_dense_smem(int nz, int cols) {
  return sizeof(double) * 8 * (size_t)nz * cols + sizeof(unsigned) * cols;
}

cudaError_t imex_kernel_setup() {
  if (imex_attr.has()) return cudaSuccess;
  cudaError_t e = set_imex_attr<false>();
  if (e == cudaSuccess) e = set_imex_attr<true>();
  if (e == cudaSuccess) imex_attr.set();
  return e;
}

cudaError_t launch_imex(const ImexArgs& a, cudaStream_t s) {
  if (a.cols_per_block < 1 || a.cols_per_block > kImexThreads || a.nz < 2 || a.N < 1 || a.kl > 2 * a.N ||
      a.ku > 4 * a.N)
    return cudaErrorInvalidValue;
  const size_t smem = imex_smem_bytes(a.nz, a.N, a.cols_per_block);
  if (smem > kImexSmemMax || !imex_attr.has()) return cudaErrorInvalidValue;
  if (a.ncol == 0) return cudaSuccess;
  const long long blocks = (a.ncol + a.cols_per_block - 1) / a.cols_per_block;
  if (a.Hi && a.nz <= kImexDense) {
    ImexArgs d = a;
    d.cols_per_block = a.nz <= kImexWide ? 32 : 16;
    const long long items = (long long)a.nz * d.cols_per_block;
    int warps = 8;  // the count that leaves the fewest lanes idle in the last of its rounds
    for (int w = 9; w <= kImexDenseThreads / 32; ++w)
      if ((items + 32 * w - 1) / (32 * w) * w <= (items + 32 * warps - 1) / (32 * warps) * warps) warps = w;
    const unsigned nb = (unsigned)((a.ncol + d.cols_per_block - 1) / d.cols_per_block);
    const size_t dense = imex_dense_smem(a.nz, d.cols_per_block);
    if (a.nrm) imex_column_kernel<true, true><<<nb, 32 * warps, dense, s>>>(d);
    else imex_column_kernel<false, true><<<nb, 32 * warps, dense, s>>>(d);
  } else if (a.nrm) {
    imex_column_kernel<true, false><<<(unsigned)blocks, kImexThreads, smem, s>>>(a);
  } else {
    imex_column_kernel<false, false><<<(unsigned)blocks, kImexThreads, smem, s>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace numa
