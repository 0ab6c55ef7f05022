// Line passes (lines.cuh): the x passes, FP32
#include "lines.cuh"

namespace okmc {

template <class T, class Q>
cudaError_t launch_x_fwd(const Q* eps, C2<T>* spec, const PassCfg& c, cudaStream_t st) {
  const dim3 grid(c.ny / x_rows<T>(), c.ncomp * c.nzin);
  switch (c.H) {
#define OKMC_CASE(h) \
  case h: return launch_lines(k_x_fwd<T, Q, h>, grid, x_threads<T, h>(), x_smem<T, h>(), st, eps, spec, c);
    OKMC_HALF_EDGES(OKMC_CASE)
#undef OKMC_CASE
    default: return cudaErrorInvalidConfiguration;
  }
}
template <class T>
cudaError_t launch_x_inv(const C2<T>* spec, T* sig, const PassCfg& c, cudaStream_t st) {
  const dim3 grid(c.ny / x_rows<T>(), c.ncomp * c.nzout);
  switch (c.H) {
#define OKMC_CASE(h) \
  case h: return launch_lines(k_x_inv<T, h>, grid, x_threads<T, h>(), x_smem<T, h>(), st, spec, sig, c);
    OKMC_HALF_EDGES(OKMC_CASE)
#undef OKMC_CASE
    default: return cudaErrorInvalidConfiguration;
  }
}
template cudaError_t launch_x_fwd<float, int32_t>(const int32_t*, C2<float>*, const PassCfg&, cudaStream_t);
template cudaError_t launch_x_fwd<float, float>(const float*, C2<float>*, const PassCfg&, cudaStream_t);
template cudaError_t launch_x_inv<float>(const C2<float>*, float*, const PassCfg&, cudaStream_t);

}  // namespace okmc
