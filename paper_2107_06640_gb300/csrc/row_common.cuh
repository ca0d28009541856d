// What the two row kernels (row_local.cuh, row_neighbour.cuh) share.
//
// They are the CUDA-core form of the element update, in both precisions and at
// every degree (in a tensor-core context for its fault elements): one warp works
// on three (virtual) elements, lane 9 j + p holds
// the row of quantity p of element j in registers (lanes 27..31 idle; plain
// acoustic elements in the local phase: eight elements, lane 4 j + p, all lanes
// busy), the operators are straight-line sparse code (sparse_ops.cuh), the quantities of
// an element meet in warp shuffles, and no block barrier is needed.
//
// Face data are modal: a face block holds traction sigma n (n the owner's
// outward normal) and velocity, the six quantities that the Godunov flux
// reads, in the face's orthonormal Dubiner modes: [Bf][6], padded to
// face_block(N) values.  An element's four blocks follow one another in the
// trace array.  LTS buffers ([slot*S][4] blocks, FP64) and the derivative
// traces of faces with a finer neighbour ([slot*S][N+1] blocks in the space of
// [N+1][9][Bf]) are modal as well; those of fault faces stay
// nodal in all nine quantities ([N+1][9][Bf]), as the friction solve reads them.
//
// What bounds them: FP64, the 2 FMA per clock and SM (the sparse form has 3.4
// to 4 times fewer of them than dense nodal products, and no lane waits on an
// operand; 87 % of the FP64 pipe busy at degree 5); FP32, instruction issue and
// the latency of the copies (50 to 58 % of issue slots at degree 3).  Against one block per element with dense
// operands in global memory and block barriers between the levels: degree 3
// FP64, 3,072 tets, 366 -> 110 us per step; degree 5 FP64, 33,696 tets, 17.0 ->
// 4.4 ms; degree 3 FP32, 13,182 tets, 130 -> 30 us; 102,258 tets, 1.13 -> 0.22
// ms.
#pragma once
#include <cuda_runtime.h>

#include "func_attr.hpp"
#include "kernels.cuh"
#include "sparse_ops.cuh"

namespace adg {
namespace row {

constexpr int EW = kRowElems;  // elements per warp
constexpr int kMaxThreads = 256;

// Shapes of degree N in type T: vector width VW of the copies between global
// and shared memory (16 bytes where a row allows it), and the row stride SB
// in shared memory, padded so that the vector accesses of a quarter warp's
// eight rows fall on distinct banks.
template <class T, int N>
struct Shape {
  static constexpr int B = nb3(N), Bf = nb2(N), B1 = nb3(N - 1);
  static constexpr int V16 = 16 / (int)sizeof(T);
  static constexpr int VW = B % V16 == 0 ? V16 : 1;
  // 16-byte accesses: the stride in 16-byte units must be odd
  static constexpr int SB = VW == 1 ? (sizeof(T) == 4 ? (B | 1) : B) : (B / VW % 2 ? B : B + VW);
  static constexpr int FS = face_block(N);     // values of a face block
};
template <class T, int VW>
struct alignas(VW * sizeof(T)) Vec {
  T x[VW];
};

// f(row, column, offset) for every VW values of nE elements' rows, offset the place in global memory
template <class T, int N, int VW, class F>
__device__ __forceinline__ void each_chunk(int nE, int lane, F&& f) {
  constexpr int C = Shape<T, N>::B / VW;
  for (int i = lane; i < nE * 9 * C; i += 32) f(i / C, (i % C) * VW, i);
}
// adg_step_noalloc's caller may pass dofs on any multiple of sizeof(T)
template <class T, int N>
__device__ __forceinline__ bool vector_rows(const T* Q) {
  return Shape<T, N>::VW > 1 && (reinterpret_cast<uintptr_t>(Q) & 15) == 0;
}
template <class T, int N, int VW>
__device__ __forceinline__ void rows_in_v(T* sQ, const T* Q, int nE, int lane) {
  using V = Vec<T, VW>;
  each_chunk<T, N, VW>(nE, lane, [&](int r, int c, int i) {
    *reinterpret_cast<V*>(sQ + r * Shape<T, N>::SB + c) = reinterpret_cast<const V*>(Q)[i];
  });
}
template <class T, int N, int VW>
__device__ __forceinline__ void rows_out_v(const T* sQ, T* Q, int nE, int lane) {
  using V = Vec<T, VW>;
  each_chunk<T, N, VW>(nE, lane, [&](int r, int c, int i) {
    reinterpret_cast<V*>(Q)[i] = *reinterpret_cast<const V*>(sQ + r * Shape<T, N>::SB + c);
  });
}
// the warp's nE elements' dofs rows, global <-> shared (row stride SB)
template <class T, int N>
__device__ __forceinline__ void rows_in(T* sQ, const T* Q, int nE, int lane) {
  if (vector_rows<T, N>(Q))
    rows_in_v<T, N, Shape<T, N>::VW>(sQ, Q, nE, lane);
  else
    rows_in_v<T, N, 1>(sQ, Q, nE, lane);
}
template <class T, int N>
__device__ __forceinline__ void rows_out(const T* sQ, T* Q, int nE, int lane) {
  if (vector_rows<T, N>(Q))
    rows_out_v<T, N, Shape<T, N>::VW>(sQ, Q, nE, lane);
  else
    rows_out_v<T, N, 1>(sQ, Q, nE, lane);
}

// Threads per block; `threads` (0: none) is the choice of adg_autotune for launches
// above eight warps per SM.  The warps of a block share nothing but, in the neighbour kernel, the re-orientation
// table, so blocks are as small as that allows: with at most eight warps per SM
// single warps spread best (degree 3 FP64, 3,072 tets: 110 us per step with 32
// threads, 120 with 128), above that 128 (13,182 tets, FP32: 29.7 with 128,
// 32.6 with 32).  FP32 at degrees 4 and 5 gains more from filling the table once
// for eight warps instead of four (183,456 tets: degree 5 1106 -> 1028 us, degree 4
// 782 -> 759 us) than degree 3 does (102,258 tets: 225 -> 231).  FP32 kernels are
// held to 128 registers (two blocks of 256 per SM): at degree 4 the local ones
// spill 288 to 400 bytes for it, at degree 5 20 to 304, below that nothing; FP64 at
// degree 5 (255 registers) spills 250 to 500 bytes.
template <class T, int N>
inline int block_threads(int threads, int64_t units, int n_sms) {
  if (units <= (int64_t)kSmallLaunchWarps * n_sms) return 32;
  if (threads) return threads;
  return sizeof(T) == 4 && N >= 4 ? 256 : 128;
}

// this warp's work unit: its segment, first virtual element and element count (0: none)
struct Unit {
  int seg, nE;
  int64_t v0;
};
template <int EW = kRowElems>
__device__ __forceinline__ Unit unit_of(const Segs& g) {
  const int64_t u = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (u >= g.first[g.n]) return {0, 0, 0};
  const int i = seg_find(g, u);
  const int64_t o = (u - g.first[i]) * EW, left = g.s[i].n - o;
  return {i, (int)(left < EW ? left : EW), g.s[i].v_begin + o};
}

}  // namespace row
}  // namespace adg
