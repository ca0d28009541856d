// Row form of the neighbour kernel, float.
#include "row_neighbour.cuh"

namespace adg {
int launch_neighbour_row_f32(int N, const StepArgs& a, const Segs& g, int threads, bool spec, void* stream) {
  return row::launch_neighbour_row_n<float>(N, a, g, threads, spec, (cudaStream_t)stream);
}
}  // namespace adg
