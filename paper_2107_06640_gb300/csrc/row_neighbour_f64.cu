// Row form of the neighbour kernel, double.
#include "row_neighbour.cuh"

namespace adg {
int launch_neighbour_row_f64(int N, const StepArgs& a, const Segs& g, int threads, bool spec, void* stream) {
  return row::launch_neighbour_row_n<double>(N, a, g, threads, spec, (cudaStream_t)stream);
}
}  // namespace adg
