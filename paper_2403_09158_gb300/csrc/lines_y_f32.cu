// Line passes (lines.cuh): the y pass, FP32
#include "lines.cuh"

namespace okmc {

template <class T>
cudaError_t launch_y(bool inverse, C2<T>* spec, const PassCfg& c, cudaStream_t st) {
  const int nlines = c.ncomp * (inverse ? c.nzout : c.nzin) * (c.H + 1);
  switch (c.ny) {
#define OKMC_CASE(n)                                                                                                  \
  case n: {                                                                                                           \
    const dim3 grid((nlines + y_lines<T, n>() - 1) / y_lines<T, n>());                                                \
    return inverse ? launch_lines(k_y<T, n, true>, grid, y_threads<T, n>(), y_smem<T, n>(), st, spec, c, nlines)      \
                   : launch_lines(k_y<T, n, false>, grid, y_threads<T, n>(), y_smem<T, n>(), st, spec, c, nlines);    \
  }
    OKMC_EDGES(OKMC_CASE)
#undef OKMC_CASE
    default: return cudaErrorInvalidConfiguration;
  }
}
template cudaError_t launch_y<float>(bool, C2<float>*, const PassCfg&, cudaStream_t);

}  // namespace okmc
