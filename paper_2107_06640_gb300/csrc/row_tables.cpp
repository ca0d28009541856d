// Host tables of the row kernels (row_common.cuh) from the nonzero entries of
// the reference operators.
#include <algorithm>
#include <cmath>

#include "adg_internal.hpp"

namespace adg {

namespace {
struct Entry {
  int r, c;
  double v;
};
#include "sparse_ops.inc"

template <int n>
void add(const Entry (&e)[n], int rows, int cols, double s, std::vector<double>& m) {
  for (const Entry& x : e)
    if (x.r < rows && x.c < cols) m[(size_t)x.r * cols + x.c] += s * x.v;
}
}  // namespace

RowTables make_row_tables(const RefOps& o) {
  const int N = o.N, B = o.B, B1 = o.B1, Bf = nface(N);
  RowTables t;
  // the lists against the operators of this run
  for (int a = 0; a < 3; ++a) {
    std::vector<double> m((size_t)B1 * B, 0.0);
    add(kKX, B1, B, a == 0 ? 1.0 : 0.5, m);
    if (a) add(kKY, B1, B, 1.0, m);
    if (a == 2) add(kKZ, B1, B, 1.0, m);
    for (int r = 0; r < B1; ++r)
      for (int l = 0; l < B; ++l)
        t.max_err = std::max(t.max_err, std::fabs(m[(size_t)r * B + l] - o.kt[((size_t)a * B + r) * B + l]));
  }
  t.rfcT.assign((size_t)4 * B * Bf, 0.0);
  int l = 0;
  std::vector<int> odd(B);
  for (int n = 0; n <= N; ++n)
    for (int i = 0; i <= n; ++i)
      for (int j = 0; j <= n - i; ++j) odd[l++] = i & 1;
  for (int f = 0; f < 4; ++f) {
    std::vector<double> m((size_t)Bf * B, 0.0);
    if (f < 2) add(kR0, Bf, B, 1.0, m);
    if (f == 2) add(kR2, Bf, B, 1.0, m);
    if (f == 3) add(kR3, Bf, B, 1.0, m);
    for (int r = 0; r < Bf; ++r)
      for (int k = 0; k < B; ++k)
        t.rfcT[((size_t)f * B + k) * Bf + r] = (f == 1 && odd[k] ? -1.0 : 1.0) * m[(size_t)r * B + k];
  }
  // nodes to modes, int psi_r ell_n: on face 3 every phi_l is a multiple v of one
  // mode r, and lift[3][l][n] = v int psi_r ell_n
  t.modalT.assign((size_t)Bf * Bf, 0.0);
  for (const Entry& x : kR3)
    if (x.r < Bf && x.c < B)
      for (int n = 0; n < Bf; ++n) t.modalT[(size_t)n * Bf + x.r] = o.lift[((size_t)3 * B + x.c) * Bf + n] / x.v;
  // modes at the nodes, from the same multiples: efc[3][n][l] = v psi_r(n)
  t.nodalT.assign((size_t)Bf * Bf, 0.0);
  for (const Entry& x : kR3)
    if (x.r < Bf && x.c < B)
      for (int n = 0; n < Bf; ++n) t.nodalT[(size_t)x.r * Bf + n] = o.efc[((size_t)3 * Bf + n) * B + x.c] / x.v;
  // both ways of lifting a node: over the modes, and the nodal lift
  for (int f = 0; f < 4; ++f)
    for (int m = 0; m < B; ++m)
      for (int n = 0; n < Bf; ++n) {
        double s = 0;
        for (int r = 0; r < Bf; ++r) s += t.rfcT[((size_t)f * B + m) * Bf + r] * t.modalT[(size_t)n * Bf + r];
        t.max_err = std::max(t.max_err, std::fabs(s - o.lift[((size_t)f * B + m) * Bf + n]));
      }
  const int np = (N + 1) * (N + 2) * (2 * N + 3) / 6;
  for (int p = 0; p < 6; ++p) t.reorient.insert(t.reorient.end(), kPV[p], kPV[p] + np);
  return t;
}

}  // namespace adg
