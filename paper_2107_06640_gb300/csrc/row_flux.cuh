// Modal face fluxes of a warp's three elements, shared by the row and the
// tensor-core neighbour kernel.  Per face:
//   face_stage  the own blocks, the neighbours' and the coefficients of one
//               face, requested with 16-byte cp.async into one of two buffers
//               while the face before is worked on;
//   face_items  work item (element, mode), 3 Bf per warp: the neighbour's six
//               quantities re-oriented to this side's modes (block diagonal in
//               the modes' degree: at most N + 1 products each, the entries of
//               the item's row in a shared table), the middle state, and the
//               nine scaled flux components, written as rows [quantity][mode]
//               for the lift.
// Re-orienting the six quantities by items needs 6 (N + 1) products per item;
// re-orienting the nine flux rows of the neighbour's part by (element,
// quantity) lanes, with their second flux evaluation and the table read as 16
// bytes per lane, took a third more instructions and shared-memory wavefronts.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.cuh"
#include "sparse_ops.cuh"
#include "tc_common.cuh"

namespace adg {

template <class T, int N>
struct FaceSmem {
  static constexpr int BF = nb2(N), FS = face_block(N), V = 16 / (int)sizeof(T);
  static constexpr int stage = 6 * FS + 3 * CREC;  // own blocks, the neighbours', coefficients
  // flux row: whole 16-byte units, an odd number of them (the rows of a quarter warp on distinct banks)
  static constexpr int gu = (BF + V - 1) / V, GS = (gu % 2 ? gu : gu + 1) * V;
  static constexpr int rows = 27 * GS;
  static constexpr int BP = BF + (BF & 1);          // re-orientation table [6][N + 1][BP]: entry s of row n
  static constexpr int table = 6 * (N + 1) * BP;
};

// thread `t` of `nt` fills the re-orientation table from StepArgs::reorient (blocks by degree)
template <class T, int N>
__device__ __forceinline__ void reorient_table(T* sP, const T* blocks, int t, int nt) {
  using F = FaceSmem<T, N>;
  for (int i = t; i < F::table; i += nt) {
    const int p = i / ((N + 1) * F::BP), s = i / F::BP % (N + 1), n = i % F::BP;
    int d = 0;
    while ((d + 1) * (d + 2) / 2 <= n) ++d;
    sP[i] = n < F::BF && s <= d ? blocks[p * sp::blk(N + 1) + sp::blk(d) + (n - d * (d + 1) / 2) * (d + 1) + s] : T(0);
  }
}

// info, nbr: of face f of element j in lane 4 j + f; kOne: one scenario
template <class T, int N, bool kOne>
__device__ __forceinline__ void face_stage(const StepArgs& a, T* st, int64_t v0, int nE, int info, int nbr, int f,
                                           int lane) {
  using F = FaceSmem<T, N>;
  constexpr int C = F::FS / F::V, CC = CREC / F::V;
  const T* const trace = reinterpret_cast<const T*>(a.trace);
  const T* const crec = reinterpret_cast<const T*>(a.crec);
#pragma unroll
  for (int k = 0; k < (3 * C + 31) / 32; ++k) {
    const int i = lane + 32 * k, j = i < 3 * C ? i / C : 0, c = i - j * C;
    const int in = __shfl_sync(0xffffffffu, info, 4 * j + f), nb = __shfl_sync(0xffffffffu, nbr, 4 * j + f);
    if (i >= nE * C) continue;
    const int64_t v = v0 + j;
    tc::cp_async16(st + i * F::V, trace + (v * 4 + f) * F::FS + c * F::V);
    if (((in >> 5) & 7) == NK_SAME) {
      const int64_t vn = kOne ? (int64_t)nb : (int64_t)nb * a.S + (v - elem_of(v, a.S) * a.S);
      tc::cp_async16(st + 3 * F::FS + i * F::V, trace + (vn * 4 + (in & 3)) * F::FS + c * F::V);
    }
  }
#pragma unroll
  for (int k = 0; k < (3 * CC + 31) / 32; ++k) {
    const int i = lane + 32 * k, j = i / CC, c = i - j * CC;
    if (i >= nE * CC) continue;
    const int64_t v = v0 + j, e = kOne ? v : elem_of(v, a.S);
    tc::cp_async16(st + 6 * F::FS + i * F::V, crec + (e * 4 + f) * CREC + c * F::V);
  }
  tc::cp_async_commit();
}

// the neighbours' blocks of face f that are not in the trace array: a finer
// LTS neighbour's buffer (the integral of its traces over this step), a
// coarser one's expansion over this sub-interval
template <class T, int N>
__device__ void face_lts(const StepArgs& a, const Seg& sg, T* st, int64_t v0, int nE, int info, int nbr, int f,
                         int lane) {
  using F = FaceSmem<T, N>;
  for (int j = 0; j < nE; ++j) {
    const int in = __shfl_sync(0xffffffffu, info, 4 * j + f), nb = __shfl_sync(0xffffffffu, nbr, 4 * j + f);
    const int kind = (in >> 5) & 7;
    const int s = (int)(v0 + j - elem_of(v0 + j, a.S) * a.S);
    T* const out = st + (3 + j) * F::FS;
    if (kind == NK_FINE) {
      const double* const src = a.btrace + (((int64_t)a.bslot[nb] * a.S + s) * 4 + (in & 3)) * F::FS;
      for (int i = lane; i < 6 * F::BF; i += 32) out[i] = (T)src[i];
    } else if (kind == NK_COARSE) {
      const T* const src = reinterpret_cast<const T*>(a.dtrace) +
                           ((int64_t)a.dslot[(int64_t)nb * 4 + (in & 3)] * a.S + s) * (N + 1) * 9 * F::BF;
      for (int i = lane; i < 6 * F::BF; i += 32) {
        T x = T(0);
#pragma unroll
        for (int d = 0; d <= N; ++d) x = fma(seg_ccoef<T>(sg, d), src[d * F::FS + i], x);
        out[i] = x;
      }
    }
  }
}

// flux rows of face f; sP: the re-orientation table, sG: [27] rows of GS
template <class T, int N, bool kLts>
__device__ __forceinline__ void face_items(const StepArgs& a, const T* st, const T* sP, T* sG, int64_t v0, int nE,
                                           int info, int f, int lane) {
  using F = FaceSmem<T, N>;
  constexpr int BF = F::BF, FS = F::FS;
#pragma unroll
  for (int k = 0; k < (3 * BF + 31) / 32; ++k) {
    const int i = lane + 32 * k, je = i < 3 * BF ? i / BF : 0, n = i - je * BF;
    const int in = __shfl_sync(0xffffffffu, info, 4 * je + f);
    if (i >= nE * BF) continue;
    const int kind = (in >> 5) & 7;
    struct alignas(2 * sizeof(T)) V2 {
      T x, y;
    };
    T q[6], w[6];
#pragma unroll
    for (int d = 0; d < 6; d += 2) {
      const V2 x = *reinterpret_cast<const V2*>(st + je * FS + 6 * n + d);
      q[d] = x.x; q[d + 1] = x.y;
      w[d] = w[d + 1] = T(0);
    }
    T srt = T(0), srv = T(0);
    if (kind != NK_NONE) {
      int first = 0;  // of the modes of n's degree
#pragma unroll
      for (int d = 1; d <= N; ++d) first = n >= d * (d + 1) / 2 ? d * (d + 1) / 2 : first;
      const T* const u = st + (3 + je) * FS + 6 * first;
      const T* const p = sP + ((in >> 2) & 7) * ((N + 1) * F::BP) + n;
#pragma unroll
      for (int s = 0; s <= N; ++s) {
        const T x = p[s * F::BP];  // (zero past the degree's modes)
#pragma unroll
        for (int d = 0; d < 6; d += 2) {
          const V2 y = *reinterpret_cast<const V2*>(u + 6 * s + d);
          w[d] = fma(x, y.x, w[d]);
          w[d + 1] = fma(x, y.y, w[d + 1]);
        }
      }
    } else if (kLts && a.gslot) {
      // a gravitational surface's normal traction and velocity
      const int64_t v = v0 + je, e = elem_of(v, a.S);
      const int gs = a.gslot[e * 4 + f];
      if (gs >= 0) {
        const T* const src = reinterpret_cast<const T*>(a.gflux) + ((int64_t)gs * a.S + (v - e * a.S)) * 9 * BF + n;
        srt = src[0];
        srv = src[BF];
      }
    }
    T c[CREC];
#pragma unroll
    for (int d = 0; d < CREC / F::V; ++d) {
      struct alignas(16) V16 {
        T x[F::V];
      };
      const V16 x = reinterpret_cast<const V16*>(st + 6 * FS + je * CREC)[d];
#pragma unroll
      for (int t = 0; t < F::V; ++t) c[d * F::V + t] = x.x[t];
    }
    T r[9];
    face_flux_state(c, q, w, srt, srv, r);
    T* const g = sG + 9 * je * F::GS + n;
#pragma unroll
    for (int p = 0; p < 9; ++p) g[p * F::GS] = r[p];
  }
}

// this lane's flux row (lanes past the warp's rows: row 0)
template <class T, int N>
__device__ __forceinline__ void face_row(const T* sG, int row, T (&x)[nb2(N)]) {
  using F = FaceSmem<T, N>;
  struct alignas(16) V16 {
    T x[F::V];
  };
#pragma unroll
  for (int c = 0; c < F::gu; ++c) {
    const V16 u = reinterpret_cast<const V16*>(sG + row * F::GS)[c];
#pragma unroll
    for (int t = 0; t < F::V; ++t)
      if (c * F::V + t < F::BF) x[c * F::V + t] = u.x[t];
  }
}

}  // namespace adg
