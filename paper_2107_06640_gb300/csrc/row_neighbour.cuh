// Row form of the neighbour kernel (Sec. 4.2; see row_common.cuh for the
// layout): Godunov fluxes of the four faces in modal form and their lift, three
// elements per warp.  Per face:
//   1. work item (element, mode), 3 Bf per warp: the own part of the scaled
//      flux from the own traction and velocity, and the neighbour's part from
//      the neighbour's, both frame-free with the face's coefficients
//      (crec_face): t^b = s_tt t + s_tv v + (normal part) n, and so on;
//   2. lane (element, quantity): the neighbour's part re-oriented to this
//      side's modes (block-diagonal, coefficients in shared memory), added to
//      the own part, and lifted with the sparse transposed face projections
//      (faces 0 and 1 share theirs through sum and difference).
// kSpec: as in row_local.cuh.
#pragma once
#include "row_common.cuh"

namespace adg {
namespace row {

template <class T, int N>
struct NbrSmem {
  using S = Shape<T, N>;
  // the two parts of one face's flux rows, or the lifted rows
  static constexpr int nG = (2 * 9 * EW * S::Bf + 3) / 4 * 4, nQ = (9 * EW * S::SB + 3) / 4 * 4;
  static constexpr int warp = nG > nQ ? nG : nQ;
  static constexpr int nP = (6 * sp::blk(N + 1) + 3) / 4 * 4;  // re-orientation entries (block)
  static constexpr int bytes(int threads) { return (nP + warp * (threads / 32)) * (int)sizeof(T); }
};

// one side's part of the scaled flux: traction t and velocity v of that side,
// the side's four tangential and four normal coefficients, normal source terms
template <class T>
__device__ __forceinline__ void flux_part(const T* n, const T* ct, const T* cn, const T* cm, const T t[3], const T v[3],
                                          T st, T sv, T g[9]) {
  const T tn = fma(t[2], n[2], fma(t[1], n[1], t[0] * n[0]));
  const T vn = fma(v[2], n[2], fma(v[1], n[1], v[0] * n[0]));
  const T an = fma(cn[0], tn, fma(cn[1], vn, st)), bn = fma(cn[2], tn, fma(cn[3], vn, sv));
  T tb[3], vb[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    tb[i] = fma(an, n[i], fma(ct[0], t[i], ct[1] * v[i]));
    vb[i] = fma(bn, n[i], fma(ct[2], t[i], ct[3] * v[i]));
  }
  const T l = cm[0] * fma(vb[2], n[2], fma(vb[1], n[1], vb[0] * n[0]));
  const T m[3] = {cm[1] * vb[0], cm[1] * vb[1], cm[1] * vb[2]};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    g[i] = fma(T(2) * n[i], m[i], l);
    g[6 + i] = cm[2] * tb[i];
  }
  g[3] = fma(n[0], m[1], n[1] * m[0]);
  g[4] = fma(n[1], m[2], n[2] * m[1]);
  g[5] = fma(n[0], m[2], n[2] * m[0]);
}

template <class T, int N, bool kSpec>
__global__ void __launch_bounds__(kMaxThreads, sizeof(T) == 4 ? 2 : 1) neighbour_row_kernel(StepArgs a, const __grid_constant__ Segs g) {
  using S = Shape<T, N>;
  using M = NbrSmem<T, N>;
  constexpr int B = S::B, Bf = S::Bf, FS = S::FS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* const sP = reinterpret_cast<T*>(smem_raw);
  const int lane = threadIdx.x & 31;
  T* const sA = sP + M::nP + (threadIdx.x >> 5) * M::warp;  // own part [row][Bf], then the neighbours'
  T* const sB = sA + 9 * EW * Bf;
  constexpr int nPV = sp::blk(N + 1);
  for (int i = threadIdx.x; i < 6 * nPV; i += blockDim.x) sP[i] = reinterpret_cast<const T*>(a.reorient)[i];
  __syncthreads();
  const Unit u = unit_of(g);
  if (u.nE == 0) return;
  const Seg& sg = g.s[u.seg];
  // lane 4 j + f (< 12): face f of element j, its neighbour and what it is
  int my_info = 0, my_nbr = -1;
  if (lane < 4 * u.nE) {
    const int64_t ef = (u.v0 + (lane >> 2)) / a.S * 4 + (lane & 3);
    my_info = a.ninfo[ef];
    my_nbr = a.nbr[ef];
  }
  const T* const trace = reinterpret_cast<const T*>(a.trace);
  const int j = lane < 27 ? lane / 9 : 0;
  const bool valid = lane < 9 * u.nE;
  T acc[B];
#pragma unroll
  for (int m = 0; m < B; ++m) acc[m] = T(0);

  // flux rows of face f (of this lane's element and quantity) -> gr
  auto face = [&](const int f, T(&gr)[Bf]) {
    __syncwarp();
#pragma unroll
    for (int it = 0; it < (EW * Bf + 31) / 32; ++it) {
      const int i = lane + 32 * it;
      const int je = i < EW * Bf ? i / Bf : 0, n = i - je * Bf;
      const int info = __shfl_sync(0xffffffffu, my_info, 4 * je + f), nb = __shfl_sync(0xffffffffu, my_nbr, 4 * je + f);
      if (i >= u.nE * Bf) continue;
      const int64_t v = u.v0 + je, e = v / a.S;
      const int s = (int)(v - e * a.S);
      const int kind = (info >> 5) & 7;
      const T* const cp = reinterpret_cast<const T*>(a.crec) + (e * 4 + f) * CREC;
      T c[CREC];
#pragma unroll
      for (int k = 0; k < CREC / S::V16; ++k) {
        const Vec<T, S::V16> x = reinterpret_cast<const Vec<T, S::V16>*>(cp)[k];
#pragma unroll
        for (int t = 0; t < S::V16; ++t) c[k * S::V16 + t] = x.x[t];
      }
      T q[6], ga[9], gb[9];
      const T* const own = trace + (v * 4 + f) * FS + n;
#pragma unroll
      for (int k = 0; k < 6; ++k) q[k] = own[k * Bf];
      T w[6];
#pragma unroll
      for (int k = 0; k < 6; ++k) w[k] = T(0);
      T st = T(0), sv = T(0);
      if (!kSpec || kind == NK_SAME) {
        if (kind == NK_SAME) {
          const T* const src = trace + (((int64_t)nb * a.S + s) * 4 + (info & 3)) * FS + n;
#pragma unroll
          for (int k = 0; k < 6; ++k) w[k] = src[k * Bf];
        }
      } else if (kind == NK_FINE) {  // the integral of the finer neighbour's traces over this step
        const double* const src = a.btrace + (((int64_t)a.bslot[nb] * a.S + s) * 4 + (info & 3)) * FS + n;
#pragma unroll
        for (int k = 0; k < 6; ++k) w[k] = (T)src[k * Bf];
      } else if (kind == NK_COARSE) {  // the coarser neighbour's expansion over this sub-interval
        const T* const src = reinterpret_cast<const T*>(a.dtrace) +
                             ((int64_t)a.dslot[(int64_t)nb * 4 + (info & 3)] * a.S + s) * (N + 1) * 9 * Bf + n;
#pragma unroll
        for (int d = 0; d <= N; ++d) {
          const T cc = (T)sg.ccoef[d];
#pragma unroll
          for (int k = 0; k < 6; ++k) w[k] = fma(cc, src[d * FS + k * Bf], w[k]);
        }
      } else if (kind == NK_NONE && a.gslot) {  // a gravitational surface's traction and normal velocity
        const int gs = a.gslot[e * 4 + f];
        if (gs >= 0) {
          const T* const src = reinterpret_cast<const T*>(a.gflux) + ((int64_t)gs * a.S + s) * 9 * Bf + n;
          st = src[0];
          sv = src[Bf];
        }
      }
      flux_part(c, c + 3, c + 11, c + 19, q, q + 3, st, sv, ga);
      flux_part(c, c + 7, c + 15, c + 19, w, w + 3, T(0), T(0), gb);
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        sA[(9 * je + k) * Bf + n] = ga[k];
        sB[(9 * je + k) * Bf + n] = gb[k];
      }
    }
    __syncwarp();
    const int info = __shfl_sync(0xffffffffu, my_info, 4 * j + f);
    const T* const P = sP + ((info >> 2) & 7) * nPV;
    const T *const ra = sA + (valid ? lane : 0) * Bf, *const rb = sB + (valid ? lane : 0) * Bf;
#pragma unroll
    for (int n = 0; n <= N; ++n) {
      constexpr int W = N + 1;
      T b[W];
#pragma unroll
      for (int s = 0; s < W; ++s)
        if (s <= n) b[s] = rb[n * (n + 1) / 2 + s];
#pragma unroll
      for (int r = 0; r < W; ++r) {
        if (r > n) continue;
        T x = ra[n * (n + 1) / 2 + r];
#pragma unroll
        for (int s = 0; s < W; ++s)
          if (s <= n) x = fma(P[sp::blk(n) + r * (n + 1) + s], b[s], x);
        gr[n * (n + 1) / 2 + r] = x;
      }
    }
    if constexpr (kSpec) {
      // a fault's flux comes from the friction solve, at the face nodes
      if (valid && ((info >> 5) & 7) == NK_FAULT) {
        const int64_t v = u.v0 + j, e = v / a.S;
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
