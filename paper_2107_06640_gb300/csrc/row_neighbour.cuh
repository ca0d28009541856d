// Row form of the neighbour kernel (Sec. 4.2; see row_common.cuh for the
// layout): Godunov fluxes of the four faces in modal form (row_flux.cuh) and
// their lift with the sparse transposed face projections (faces 0 and 1 share
// theirs through sum and difference), three elements per warp.  kSpec: as in
// row_local.cuh.
#pragma once
#include "row_common.cuh"
#include "row_flux.cuh"

namespace adg {
namespace row {

// shared memory (values of T): the re-orientation table, then per warp two
// stage buffers and the flux rows; the lifted rows take the second stage
// buffer and the flux rows at the end
template <class T, int N>
struct NbrSmem {
  using S = Shape<T, N>;
  using F = FaceSmem<T, N>;
  static constexpr int nP = (F::table + 3) / 4 * 4;
  static constexpr int tail = F::stage + F::rows > 27 * S::SB ? F::stage + F::rows : 27 * S::SB;
  static constexpr int warp = (F::stage + tail + 3) / 4 * 4;
  static constexpr int bytes(int threads) { return (nP + warp * (threads / 32)) * (int)sizeof(T); }
};

template <class T, int N, bool kSpec>
__global__ void __launch_bounds__(kMaxThreads, sizeof(T) == 4 ? 2 : 1) neighbour_row_kernel(StepArgs a, const __grid_constant__ Segs g) {
  using S = Shape<T, N>;
  using M = NbrSmem<T, N>;
  using F = FaceSmem<T, N>;
  constexpr int B = S::B, Bf = S::Bf;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* const sP = reinterpret_cast<T*>(smem_raw);
  const int lane = threadIdx.x & 31;
  T* const sSt = sP + M::nP + (threadIdx.x >> 5) * M::warp;
  T* const sG = sSt + 2 * F::stage;
  T* const sA = sSt + F::stage;  // the lifted rows
  const Unit u = unit_of(g);
  const Seg& sg = g.s[u.seg];
  // lane 4 j + f (< 12): face f of element j, its neighbour and what it is
  int info = 0, nbr = -1;
  if (lane < 4 * u.nE) {
    const int64_t ef = elem_of(u.v0 + (lane >> 2), a.S) * 4 + (lane & 3);
    info = a.ninfo[ef];
    nbr = a.nbr[ef];
  }
  reorient_table<T, N>(sP, reinterpret_cast<const T*>(a.reorient), threadIdx.x, blockDim.x);
  __syncthreads();
  if (u.nE == 0) return;
  const bool one = a.S == 1;
  auto stage = [&](int f) {
    if (one)
      face_stage<T, N, true>(a, sSt + (f & 1) * F::stage, u.v0, u.nE, info, nbr, f, lane);
    else
      face_stage<T, N, false>(a, sSt + (f & 1) * F::stage, u.v0, u.nE, info, nbr, f, lane);
  };
  stage(0);
  const int j = lane < 27 ? lane / 9 : 0;
  const bool valid = lane < 9 * u.nE;
  T acc[B];
#pragma unroll
  for (int m = 0; m < B; ++m) acc[m] = T(0);

  // flux row of face f (of this lane's element and quantity) -> gr
  auto face = [&](const int f, T(&gr)[Bf]) {
    T* const st = sSt + (f & 1) * F::stage;
    tc::cp_async_wait<0>();
    __syncwarp();
    if (f < 3) stage(f + 1);
    if constexpr (kSpec) {
      face_lts<T, N>(a, sg, st, u.v0, u.nE, info, nbr, f, lane);
      __syncwarp();
    }
    face_items<T, N, kSpec>(a, st, sP, sG, u.v0, u.nE, info, f, lane);
    __syncwarp();
    face_row<T, N>(sG, valid ? lane : 0, gr);
    if constexpr (kSpec) {
      // a fault's flux comes from the friction solve, at the face nodes
      const int in = __shfl_sync(0xffffffffu, info, 4 * j + f);
      if (valid && ((in >> 5) & 7) == NK_FAULT) {
        const int64_t v = u.v0 + j, e = elem_of(v, a.S);
        const int fsl = a.fslot[e * 4 + f];
        const T* const src = reinterpret_cast<const T*>(a.drout) +
                             ((((int64_t)(fsl >> 1) * a.S + (v - e * a.S)) * 2 + (fsl & 1)) * 9 + (lane - 9 * j)) * Bf;
        const T sc = reinterpret_cast<const T*>(a.par)[e * PAR + 12 + f];
        const T* const mn = reinterpret_cast<const T*>(a.modalT);
#pragma unroll
        for (int r = 0; r < Bf; ++r) gr[r] = T(0);
        for (int n = 0; n < Bf; ++n) {
          const T x = sc * src[n];
#pragma unroll
          for (int r = 0; r < Bf; ++r) gr[r] = fma(mn[n * Bf + r], x, gr[r]);
        }
      }
    }
    __syncwarp();  // the next face refills the rows
  };
  {
    T g0[Bf], g1[Bf];
    face(0, g0);
    face(1, g1);
#pragma unroll
    for (int r = 0; r < Bf; ++r) {
      const T s = g0[r] + g1[r];
      g1[r] = g0[r] - g1[r];
      g0[r] = s;
    }
    sp::each<B>([&](auto mc) {
      constexpr int m = decltype(mc)::value;
      acc[m] = sp::dot<sp::R0t, m, Bf>(acc[m], sp::parity(m) ? g1 : g0);
    });
  }
  {
    T g2[Bf];
    face(2, g2);
    sp::each<B>([&](auto mc) {
      constexpr int m = decltype(mc)::value;
      acc[m] = sp::dot<sp::R2t, m, Bf>(acc[m], g2);
    });
    face(3, g2);
    sp::each<B>([&](auto mc) {
      constexpr int m = decltype(mc)::value;
      acc[m] = sp::dot<sp::R3t, m, Bf>(acc[m], g2);
    });
  }
  // ---- Q -= lift, the rows through shared memory
  __syncwarp();
  constexpr int VW = S::VW, C = B / VW;
  using V = Vec<T, VW>;
  if (valid) {
#pragma unroll
    for (int c = 0; c < C; ++c) {
      V x;
#pragma unroll
      for (int k = 0; k < VW; ++k) x.x[k] = acc[c * VW + k];
      *reinterpret_cast<V*>(sA + lane * S::SB + c * VW) = x;
    }
  }
  __syncwarp();
  T* const Q = reinterpret_cast<T*>(a.Q) + u.v0 * 9 * B;
  T bad = T(0);  // stays 0 while every updated dof is finite (x * 0 is NaN for x = inf, NaN)
  auto update = [&](auto wc) {
    constexpr int W = decltype(wc)::value;
    using U = Vec<T, W>;
    each_chunk<T, N, W>(u.nE, lane, [&](int r, int c, int i) {
      const U x = *reinterpret_cast<const U*>(sA + r * S::SB + c);
      U q = reinterpret_cast<const U*>(Q)[i];
#pragma unroll
      for (int k = 0; k < W; ++k) {
        q.x[k] -= x.x[k];
        if constexpr (sizeof(T) == 4)
          bad = fmaf(q.x[k], 0.f, bad);
        else
          bad = isfinite(q.x[k]) ? bad : T(1);
      }
      reinterpret_cast<U*>(Q)[i] = q;
    });
  };
  if (vector_rows<T, N>(Q))
    update(std::integral_constant<int, VW>{});
  else
    update(std::integral_constant<int, 1>{});
  if (__any_sync(0xffffffffu, bad != T(0)) && lane == 0) atomicOr(a.err, ERR_NAN);
}

template <class T, int N>
int launch_neighbour_row_t(const StepArgs& a, const Segs& g, int threads, bool spec, cudaStream_t st) {
  const int rc = configure_on_device((const void*)neighbour_row_kernel<T, N, false>, [] {
    cudaError_t ce = cudaFuncSetAttribute(neighbour_row_kernel<T, N, false>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, NbrSmem<T, N>::bytes(kMaxThreads));
    if (ce == cudaSuccess)
      ce = cudaFuncSetAttribute(neighbour_row_kernel<T, N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                NbrSmem<T, N>::bytes(kMaxThreads));
    return ce;
  });
  if (rc) return rc;
  const int64_t units = g.n ? g.first[g.n] : 0;
  if (units <= 0) return 0;
  threads = block_threads<T, N>(threads, units, a.n_sms);
  if (threads < 32 || threads > kMaxThreads || threads % 32) return (int)cudaErrorInvalidValue;
  const int w = threads / 32;
  const unsigned blocks = (unsigned)((units + w - 1) / w);
  if (spec)
    neighbour_row_kernel<T, N, true><<<blocks, threads, NbrSmem<T, N>::bytes(threads), st>>>(a, g);
  else
    neighbour_row_kernel<T, N, false><<<blocks, threads, NbrSmem<T, N>::bytes(threads), st>>>(a, g);
  return (int)cudaGetLastError();
}

template <class T>
int launch_neighbour_row_n(int N, const StepArgs& a, const Segs& g, int th, bool spec, cudaStream_t st) {
  switch (N) {
    case 1: return launch_neighbour_row_t<T, 1>(a, g, th, spec, st);
    case 2: return launch_neighbour_row_t<T, 2>(a, g, th, spec, st);
    case 3: return launch_neighbour_row_t<T, 3>(a, g, th, spec, st);
    case 4: return launch_neighbour_row_t<T, 4>(a, g, th, spec, st);
    case 5: return launch_neighbour_row_t<T, 5>(a, g, th, spec, st);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace row
}  // namespace adg
