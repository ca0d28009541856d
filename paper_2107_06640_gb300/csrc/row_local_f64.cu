// Row form of the local kernel, double.
#include "row_local.cuh"

namespace adg {
int launch_local_row_f64(int N, const StepArgs& a, const Segs& g, int threads, bool spec, void* stream) {
  return row::launch_local_row_n<double>(N, a, g, threads, spec, (cudaStream_t)stream);
}
int launch_local_fluid_f64(int N, const StepArgs& a, const Segs& g, int threads, void* stream) {
  return row::launch_local_fluid_n<double>(N, a, g, threads, (cudaStream_t)stream);
}
}  // namespace adg
