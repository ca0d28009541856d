// The reference operators as compile-time lists of their nonzero entries.
//
// In the Dubiner basis the stiffness matrices and the projections of a
// polynomial onto a face's own orthonormal Dubiner modes are sparse: at degree
// 5 the three derivatives of a row hold 924 of 5,880 entries (written in
// directions that respect the basis' parity in i, see gen_sparse_ops.py) and
// the four face projections 966 multiplications (face 1 is face 0 with the
// odd-i columns negated, so the two share their sums) against 4,704 entries of
// nodal face values.  The operators are applied row by row in straight-line
// code: the entries are literals of the instructions, a zero costs nothing and
// no operand is loaded.  The basis is hierarchical, so degree N uses the
// leading block of the degree-5 tables.
#pragma once
#include <utility>

#include "kernels.cuh"

namespace adg {
namespace sp {

struct Entry {
  int r, c;
  double v;
};
#include "sparse_ops.inc"

// entries grouped by row (kT: by column, r and c exchanged)
template <int NE, int NR>
struct Csr {
  int ptr[NR + 1] = {};
  int col[NE] = {};
  double val[NE] = {};
};
template <int NR, bool kT, int NE>
constexpr Csr<NE, NR> csr(const Entry (&e)[NE]) {
  Csr<NE, NR> m{};
  int k = 0;
  for (int r = 0; r < NR; ++r) {
    m.ptr[r] = k;
    for (int i = 0; i < NE; ++i)
      if ((kT ? e[i].c : e[i].r) == r) {
        m.col[k] = kT ? e[i].r : e[i].c;
        m.val[k] = e[i].v;
        ++k;
      }
  }
  m.ptr[NR] = k;
  return m;
}

// parity of i in phi_ijk for mode l (order: total degree, then i, then j)
__host__ __device__ constexpr int parity(int l) {
  int k = 0;
  for (int n = 0; n <= 5; ++n)
    for (int i = 0; i <= n; ++i)
      for (int j = 0; j <= n - i; ++j, ++k)
        if (k == l) return i & 1;
  return 0;
}

// ... and of i in psi_ij for mode r of a face (order: degree, then i)
__host__ __device__ constexpr int fparity(int r) {
  int n = 0;
  while ((n + 1) * (n + 2) / 2 <= r) ++n;
  return (r - n * (n + 1) / 2) & 1;
}
// how many of the first n modes have parity p, and the place of a mode among those of its parity
__host__ __device__ constexpr int count_par(int n, int p) {
  int c = 0;
  for (int l = 0; l < n; ++l) c += parity(l) == p;
  return c;
}
__host__ __device__ constexpr int count_fpar(int n, int p) {
  int c = 0;
  for (int r = 0; r < n; ++r) c += fparity(r) == p;
  return c;
}
__host__ __device__ constexpr int par_index(int l) { return count_par(l, parity(l)); }
__host__ __device__ constexpr int fpar_index(int r) { return count_fpar(r, fparity(r)); }
// the i-th mode of parity p
__host__ __device__ constexpr int par_mode(int p, int i) {
  int l = 0;
  while (parity(l) != p || par_index(l) != i) ++l;
  return l;
}

#define ADG_SPARSE_OP(name, NR, kT, table)                                                     \
  struct name {                                                                                \
    static constexpr auto m = csr<NR, kT>(table);                                              \
    __host__ __device__ static constexpr int begin(int r) { return m.ptr[r]; }                 \
    __host__ __device__ static constexpr int end(int r) { return m.ptr[r + 1]; }               \
    __host__ __device__ static constexpr int col(int i) { return m.col[i]; }                   \
    __host__ __device__ static constexpr double val(int i) { return m.val[i]; }                \
  };
ADG_SPARSE_OP(KX, 35, false, kKX)   // predictor: rows of D^{k+1}
ADG_SPARSE_OP(KY, 35, false, kKY)
ADG_SPARSE_OP(KZ, 35, false, kKZ)
ADG_SPARSE_OP(KXt, 56, true, kKX)   // volume: the transposes
ADG_SPARSE_OP(KYt, 56, true, kKY)
ADG_SPARSE_OP(KZt, 56, true, kKZ)
ADG_SPARSE_OP(R0, 21, false, kR0)   // traces: modes of a face
ADG_SPARSE_OP(R2, 21, false, kR2)
ADG_SPARSE_OP(R3, 21, false, kR3)
ADG_SPARSE_OP(R0t, 56, true, kR0)   // lift: the transposes
ADG_SPARSE_OP(R2t, 56, true, kR2)
ADG_SPARSE_OP(R3t, 56, true, kR3)
#undef ADG_SPARSE_OP

// one entry: acc + v x[c] for columns c < LIM, and only those of parity PAR (0, 1; -1: both)
template <class Op, int I, int LIM, int PAR, class T>
__device__ __forceinline__ T term(T acc, const T* x) {
  constexpr int c = Op::col(I);
  if constexpr (c < LIM && (PAR < 0 || parity(c) == PAR)) {
    constexpr T v = (T)Op::val(I);
    return fma(v, x[c], acc);
  } else {
    return acc;
  }
}
template <class Op, int B0, int LIM, int PAR, class T, int... I>
__device__ __forceinline__ T dot_seq(T acc, const T* x, std::integer_sequence<int, I...>) {
  ((acc = term<Op, B0 + I, LIM, PAR>(acc, x)), ...);
  return acc;
}
// acc + sum_c Op[R][c] x[c]
template <class Op, int R, int LIM, int PAR = -1, class T>
__device__ __forceinline__ T dot(T acc, const T* x) {
  return dot_seq<Op, Op::begin(R), LIM, PAR>(acc, x, std::make_integer_sequence<int, Op::end(R) - Op::begin(R)>{});
}

// f(std::integral_constant<int, i>) for i = 0 .. N-1, unrolled
template <class F, int... I>
__device__ __forceinline__ void each_seq(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void each(F&& f) {
  each_seq(f, std::make_integer_sequence<int, N>{});
}

// the re-orientation of a face's modes: entries of one permutation, block n at blk(n)
__host__ __device__ constexpr int blk(int n) { return n * (n + 1) * (2 * n + 1) / 6; }

}  // namespace sp
}  // namespace adg
