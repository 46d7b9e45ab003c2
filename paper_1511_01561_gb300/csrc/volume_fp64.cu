// Element kernels (Eq. 4 / Eq. 5) in FP64, in fixed point (fixed64.cuh): the
// rectilinear and the per-node form, single-mesh and ragged multi-member
// launches, and the metric terms' conversion at bind.
#include "fixed64.cuh"

namespace numa {
namespace {

template <int N, bool RECT>
cudaError_t launch_fx_t(const VolumeArgs& a, cudaStream_t s) {
  constexpr int EPB = RECT ? fx_rect_epb<N>() : fx_nodal_epb<N>(), DIRS = RECT ? 3 : 1;
  constexpr int NT = RECT ? fx_rect_threads<N>() : fx_nodal_threads<N>();
  constexpr size_t smem = RECT ? fx_rect_smem<N>() : fx_nodal_smem<N>();
  static DeviceFlags attr_set;
  if (!attr_set.has()) {
    cudaError_t e;
    if constexpr (RECT)
      e = cudaFuncSetAttribute(volume_fx_rect_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    else e = cudaFuncSetAttribute(volume_fx_nodal_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set.set();
  }
  if (a.ecnt <= 0) return cudaSuccess;
  FxTables<N, DIRS> T = {};
  if (a.fxD_host)
    for (int t = 0; t < DIRS * fx_table_entries<N>(); ++t) T.d[t] = a.fxD_host[t];
  const unsigned nb = (unsigned)((a.ecnt + EPB - 1) / EPB);
  if constexpr (RECT) return launch_kernel(volume_fx_rect_kernel<N>, nb, NT, smem, s, a.early != 0, a, T);
  else return launch_kernel(volume_fx_nodal_kernel<N>, nb, NT, smem, s, a.early != 0, a, T);
}

template <int N, bool RECT>
cudaError_t launch_fx_ragged_t(const MemberDesc* d, const RaggedGroup* g, cudaStream_t s) {
  static DeviceInts grids;  // per device, set up at its first launch there
  return launch_persistent(volume_fx_ragged<N, RECT>, RECT ? fx_rect_threads<N>() : fx_nodal_threads<N>(),
                           RECT ? fx_rect_smem<N>() : fx_nodal_smem<N>(), grids, d, g, s);
}

// f<N>() for the run-time order N = 1..8
template <typename F>
cudaError_t for_order(int N, F f) {
  switch (N) {
    case 1: return f(std::integral_constant<int, 1>());
    case 2: return f(std::integral_constant<int, 2>());
    case 3: return f(std::integral_constant<int, 3>());
    case 4: return f(std::integral_constant<int, 4>());
    case 5: return f(std::integral_constant<int, 5>());
    case 6: return f(std::integral_constant<int, 6>());
    case 7: return f(std::integral_constant<int, 7>());
    case 8: return f(std::integral_constant<int, 8>());
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_volume_fp64(int N, bool rect, const VolumeArgs& a, cudaStream_t s) {
  return for_order(N, [&](auto n) {
    constexpr int K = decltype(n)::value;
    return rect ? launch_fx_t<K, true>(a, s) : launch_fx_t<K, false>(a, s);
  });
}

cudaError_t launch_volume_ragged_fp64(int N, bool rect, const MemberDesc* d, const RaggedGroup* g, cudaStream_t s) {
  return for_order(N, [&](auto n) {
    constexpr int K = decltype(n)::value;
    return rect ? launch_fx_ragged_t<K, true>(d, g, s) : launch_fx_ragged_t<K, false>(d, g, s);
  });
}

int volume_chunk(int N, int precision, int form) {
  if (precision != NUMA_FP64) return 1;
  int c = 1;
  for_order(N, [&](auto n) {
    c = form == 2 ? fx_rect_epb<decltype(n)::value>() : fx_nodal_epb<decltype(n)::value>();
    return cudaSuccess;
  });
  return c;
}

cudaError_t launch_fx_metric(double* met, int4* fxE, long long Ne, int N, unsigned long long fxw, cudaStream_t s) {
  if (Ne == 0) return cudaSuccess;
  fx_metric_kernel<<<(unsigned)Ne, 128, 0, s>>>(met, fxE, Ne * (N + 1) * (N + 1) * (N + 1), N + 1, fxw);
  return cudaGetLastError();
}

}  // namespace numa
