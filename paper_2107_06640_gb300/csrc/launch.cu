// Launchers shared by the kernel kinds.
#include "kernels.cuh"

namespace adg {

int launch_local_row_f32(int N, const StepArgs& a, const Segs& g, int threads, bool spec, void* stream);
int launch_local_row_f64(int N, const StepArgs& a, const Segs& g, int threads, bool spec, void* stream);
int launch_neighbour_row_f32(int N, const StepArgs& a, const Segs& g, int threads, bool spec, void* stream);
int launch_neighbour_row_f64(int N, const StepArgs& a, const Segs& g, int threads, bool spec, void* stream);
int launch_local_fluid_f32(int N, const StepArgs& a, const Segs& g, int threads, void* stream);
int launch_local_fluid_f64(int N, const StepArgs& a, const Segs& g, int threads, void* stream);

int launch_local_row(int fp64, int N, const StepArgs& a, const Segs& g, void* stream, int threads, bool spec) {
  return fp64 ? launch_local_row_f64(N, a, g, threads, spec, stream)
              : launch_local_row_f32(N, a, g, threads, spec, stream);
}
int launch_neighbour_row(int fp64, int N, const StepArgs& a, const Segs& g, void* stream, int threads, bool spec) {
  return fp64 ? launch_neighbour_row_f64(N, a, g, threads, spec, stream)
              : launch_neighbour_row_f32(N, a, g, threads, spec, stream);
}
int launch_local_fluid(int fp64, int N, const StepArgs& a, const Segs& g, void* stream, int threads) {
  return fp64 ? launch_local_fluid_f64(N, a, g, threads, stream) : launch_local_fluid_f32(N, a, g, threads, stream);
}

Segs make_segs(const Seg* s, int n, int unit, int chunk) {
  Segs g{};
  g.chunk = chunk < 1 ? 1 : chunk;
  int64_t u = 0;
  for (int i = 0; i < n && g.n < kMaxSeg; ++i) {
    if (s[i].n <= 0) continue;
    g.s[g.n] = s[i];
    for (int k = 0; k < 8; ++k) {
      g.s[g.n].tcoef32[k] = (float)s[i].tcoef[k];
      g.s[g.n].ccoef32[k] = (float)s[i].ccoef[k];
    }
    g.first[g.n] = u;
    u += (s[i].n + unit - 1) / unit;
    g.n++;
  }
  g.first[g.n] = u;
  return g;
}
}  // namespace adg
