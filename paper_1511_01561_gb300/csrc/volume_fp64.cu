// Element kernels (Eq. 4 / Eq. 5) in FP64: the per-node form, and the
// rectilinear form in fixed point (fixed64.cuh), single-mesh and ragged
// multi-member launches.
#include "fixed64.cuh"

namespace numa {
namespace {

template <int N>
cudaError_t launch_fx_rect_t(const VolumeArgs& a, cudaStream_t s) {
  constexpr int EPB = fx_rect_epb<N>();
  constexpr size_t smem = fx_rect_smem<N>();
  static DeviceFlags attr_set;
  if (!attr_set.has()) {
    cudaError_t e =
        cudaFuncSetAttribute(volume_fx_rect_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_set.set();
  }
  if (a.ecnt <= 0) return cudaSuccess;
  FxTables<N> T = {};
  if (a.fxD_host)
    for (int t = 0; t < 3 * fx_table_entries<N>(); ++t) T.d[t] = a.fxD_host[t];
  volume_fx_rect_kernel<N><<<(a.ecnt + EPB - 1) / EPB, fx_rect_threads<N>(), smem, s>>>(a, T);
  return cudaGetLastError();
}

template <int N>
cudaError_t launch_fx_rect_ragged_t(const MemberDesc* d, const RaggedGroup* g, cudaStream_t s) {
  static DeviceInts grids;  // per device, set up at its first launch there
  return launch_persistent(volume_fx_rect_ragged<N>, fx_rect_threads<N>(), fx_rect_smem<N>(), grids, d, g, s);
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

cudaError_t launch_volume_fp64(int N, bool affine, const VolumeArgs& a, cudaStream_t s) {
  if (!affine) return launch_volume_p<double, false>(N, a, s);
  return for_order(N, [&](auto n) { return launch_fx_rect_t<decltype(n)::value>(a, s); });
}

cudaError_t launch_volume_ragged_fp64(int N, bool affine, const MemberDesc* d, const RaggedGroup* g, cudaStream_t s) {
  if (!affine) return launch_volume_ragged_p<double, false>(N, d, g, s);
  return for_order(N, [&](auto n) { return launch_fx_rect_ragged_t<decltype(n)::value>(d, g, s); });
}

int volume_chunk(int N, int precision, int form) {
  if (precision != NUMA_FP64 || form != 2) return 1;
  int c = 1;
  for_order(N, [&](auto n) { c = fx_rect_epb<decltype(n)::value>(); return cudaSuccess; });
  return c;
}

}  // namespace numa
