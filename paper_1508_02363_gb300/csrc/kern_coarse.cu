// Launchers of the coarse-grid correction (coarse.cuh).
#include "coarse.cuh"
#include "launch.cuh"

namespace dbar {

template <typename T>
cudaError_t launch_coarse_start(const CoarseArgs& a, const cx<T>* V, long long vss, const CycleState& f, int nslots,
                                cudaStream_t s) {
  if (nslots <= 0) return cudaSuccess;
  k_coarse_norms<T><<<dim3(kCoarseBlocks, nslots), 256, 0, s>>>(a, V, vss, f);
  k_coarse_start<<<nslots, 256, 0, s>>>(a, f);
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_coarse_restrict(const CoarseArgs& a, int l, const cx<T>* V, long long vss, cx<T>* Vc, long long vcss,
                                   void* xc, int x_f64, int nslots, cudaStream_t s) {
  if (nslots <= 0) return cudaSuccess;
  const dim3 grid(64, nslots);
  if constexpr (std::is_same<T, float>::value)
    if (!x_f64) {
      k_coarse_restrict<T, dd><<<grid, 256, 0, s>>>(a, l, V, vss, Vc, vcss, reinterpret_cast<cx<dd>*>(xc));
      return cudaGetLastError();
    }
  k_coarse_restrict<T, double><<<grid, 256, 0, s>>>(a, l, V, vss, Vc, vcss, reinterpret_cast<cx<double>*>(xc));
  return cudaGetLastError();
}
cudaError_t launch_coarse_count(const CycleState& f, const CycleState& c, int nslots, cudaStream_t s) {
  if (nslots <= 0) return cudaSuccess;
  k_coarse_count<<<(nslots + 127) / 128, 128, 0, s>>>(f, c, nslots);
  return cudaGetLastError();
}
#define CO_INST(T)                                                                                                  \
  template cudaError_t launch_coarse_start<T>(const CoarseArgs&, const cx<T>*, long long, const CycleState&, int, \
                                              cudaStream_t);                                                        \
  template cudaError_t launch_coarse_restrict<T>(const CoarseArgs&, int, const cx<T>*, long long, cx<T>*, long long, \
                                                 void*, int, int, cudaStream_t);
CO_INST(float)
CO_INST(double)

}  // namespace dbar
