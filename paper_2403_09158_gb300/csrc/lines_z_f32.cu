// Line passes (lines.cuh): the pencil pass, FP32
#include "lines.cuh"

namespace okmc {

template <class T>
cudaError_t launch_z(const C2<T>* in, C2<T>* out, const PassCfg& c, cudaStream_t st) {
  const unsigned P = (unsigned)(c.H + 1) * c.ny;
  switch (c.nz) {
#define OKMC_CASE(n) \
  case n: return launch_lines(k_z<T, n>, dim3(P / z_tw<T, n>()), kZThreads, z_smem<T, n>(), st, in, out, c);
    OKMC_EDGES(OKMC_CASE)
#undef OKMC_CASE
    default: return cudaErrorInvalidConfiguration;
  }
}
template cudaError_t launch_z<float>(const C2<float>*, C2<float>*, const PassCfg&, cudaStream_t);

}  // namespace okmc
