// Row form of the local kernel (Sec. 4.1; see row_common.cuh for the layout):
// Cauchy-Kovalewski predictor, time integral, modal face traces and volume
// term of three elements per warp.  kSpec: the launch's elements may have
// gravitational faces (Sec. 4.3), fault faces or neighbours in another LTS
// cluster (Sec. 4.4).
#pragma once
#include "row_common.cuh"
#include "tc_common.cuh"

#include <type_traits>

namespace adg {
namespace row {

// two FP32 values in a register pair, and their packed multiply and fused multiply-add
struct F2 {
  uint64_t v;
};
__device__ __forceinline__ F2 f2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_get(F2 x, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// Star product of this lane's quantity: D[p] = sum_d c_d X_d[src_d] with
// X_d = sum_b G_b,d Y_b over the three parity-respecting directions b of
// sparse_ops.inc (Jacobian form of -sum_a A*_a Y_a), for two basis functions at
// a time.
// FP32: X_d here, one shuffle per direction and function, the arithmetic
// packed in pairs (18 instructions for two functions, 30 without: the kernels
// are bound by instruction issue).  FP64: the arithmetic is what counts (2 FMA
// per clock and SM), so the Y_b travel and the products c_d G_b,d are formed
// once: 9 FMAs per function instead of 12 operations.
template <class T>
struct RowStar {
  static constexpr bool f32 = sizeof(T) == 4;
  using W = std::conditional_t<f32, F2, T>;
  W w[9];      // FP32: G_b,d at 3 b + d, twice; FP64: c_d G_b,d
  W c[3];
  int src[3];
  __device__ __forceinline__ void set(const T (&G)[9], const T (&cc)[3]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      if constexpr (f32) w[k] = f2(G[k], G[k]);
      else w[k] = G[k] * cc[k % 3];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if constexpr (f32) c[d] = f2(cc[d], cc[d]);
      else c[d] = cc[d];
    }
  }
  __device__ __forceinline__ void metric(bool valid, const T* par, T (&G)[9]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T gx = valid ? par[d] : T(0), gy = valid ? par[3 + d] : T(0), gz = valid ? par[6 + d] : T(0);
      G[d] = gx + T(0.5) * (gy + gz);
      G[3 + d] = gy + gz;
      G[6 + d] = gz;
    }
  }
  __device__ __forceinline__ void setup(int lane, bool valid, const T* par) {
    const int j = lane / 9, p = lane - 9 * j, base = 9 * j;
    T lam = 0, mu = 0, irho = 0, G[9];
    metric(valid, par, G);
    if (valid) {
      irho = T(1) / par[9];
      lam = par[10];
      mu = par[11];
    }
    const T l2m = lam + T(2) * mu;
    int q0 = p, q1 = p, q2 = p;
    T c0 = 0, c1 = 0, c2 = 0;
    switch (p) {
      case 0: q0 = 6; c0 = l2m; q1 = 7; c1 = lam; q2 = 8; c2 = lam; break;
      case 1: q0 = 6; c0 = lam; q1 = 7; c1 = l2m; q2 = 8; c2 = lam; break;
      case 2: q0 = 6; c0 = lam; q1 = 7; c1 = lam; q2 = 8; c2 = l2m; break;
      case 3: q0 = 7; c0 = mu; q1 = 6; c1 = mu; break;
      case 4: q1 = 8; c1 = mu; q2 = 7; c2 = mu; break;
      case 5: q0 = 8; c0 = mu; q2 = 6; c2 = mu; break;
      case 6: q0 = 0; c0 = irho; q1 = 3; c1 = irho; q2 = 5; c2 = irho; break;
      case 7: q0 = 3; c0 = irho; q1 = 1; c1 = irho; q2 = 4; c2 = irho; break;
      default: q0 = 5; c0 = irho; q1 = 4; c1 = irho; q2 = 2; c2 = irho; break;
    }
    const bool on = lane < 27;
    src[0] = on ? base + q0 : lane;
    src[1] = on ? base + q1 : lane;
    src[2] = on ? base + q2 : lane;
    const T cc[3] = {c0, c1, c2};
    set(G, cc);
  }
  // the acoustic rows of lane 4 j + p (p = 0: sigma_xx, p = 1..3: v_x, v_y, v_z): the
  // normal stress reads the velocities with lambda, a velocity the normal stress with 1 / rho
  __device__ __forceinline__ void setup_acoustic(int lane, bool valid, const T* par) {
    const int p = lane & 3, base = lane & ~3;
    T lam = 0, irho = 0, G[9], cc[3];
    metric(valid, par, G);
    if (valid) {
      irho = T(1) / par[9];
      lam = par[10];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      cc[d] = p == 0 ? lam : (p == d + 1 ? irho : T(0));
      src[d] = p == 0 ? base + 1 + d : (p == d + 1 ? base : lane);
    }
    set(G, cc);
  }
  // y[b][k]: the directions' values of the functions k = 0, 1
  __device__ __forceinline__ void apply(const T (&y)[3][2], T& o0, T& o1) const {
    if constexpr (f32) {
      const F2 y0 = f2(y[0][0], y[0][1]), y1 = f2(y[1][0], y[1][1]), y2 = f2(y[2][0], y[2][1]);
      F2 s;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        float a, b;
        f2_get(f2_fma(w[6 + d], y2, f2_fma(w[3 + d], y1, f2_mul(w[d], y0))), a, b);
        const F2 x = f2(__shfl_sync(0xffffffffu, a, src[d]), __shfl_sync(0xffffffffu, b, src[d]));
        s = d == 0 ? f2_mul(c[0], x) : f2_fma(c[d], x, s);
      }
      f2_get(s, o0, o1);
    } else {
      T s[2] = {T(0), T(0)};
#pragma unroll
      for (int k = 0; k < 2; ++k) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          s[k] = fma(w[d], __shfl_sync(0xffffffffu, y[0][k], src[d]), s[k]);
          s[k] = fma(w[3 + d], __shfl_sync(0xffffffffu, y[1][k], src[d]), s[k]);
          s[k] = fma(w[6 + d], __shfl_sync(0xffffffffu, y[2][k], src[d]), s[k]);
        }
      }
      o0 = s[0];
      o1 = s[1];
    }
  }
  // one function
  __device__ __forceinline__ T apply1(T y0, T y1, T y2) const {
    if constexpr (f32) {
      const T y[3][2] = {{y0, T(0)}, {y1, T(0)}, {y2, T(0)}};
      T a, b;
      apply(y, a, b);
      return a;
    } else {
      T s = T(0);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        s = fma(w[d], __shfl_sync(0xffffffffu, y0, src[d]), s);
        s = fma(w[3 + d], __shfl_sync(0xffffffffu, y1, src[d]), s);
        s = fma(w[6 + d], __shfl_sync(0xffffffffu, y2, src[d]), s);
      }
      return s;
    }
  }
};
// out[m] for m < M from the directions' values y(b, integral_constant<m>), two functions at a time
template <int M, class T, class Y>
__device__ __forceinline__ void star_rows(const RowStar<T>& st, T* out, Y&& yf) {
  sp::each<M / 2>([&](auto hc) {
    constexpr int m = 2 * decltype(hc)::value;
    using A = std::integral_constant<int, m>;
    using C = std::integral_constant<int, m + 1>;
    const T y[3][2] = {{yf(std::integral_constant<int, 0>{}, A{}), yf(std::integral_constant<int, 0>{}, C{})},
                       {yf(std::integral_constant<int, 1>{}, A{}), yf(std::integral_constant<int, 1>{}, C{})},
                       {yf(std::integral_constant<int, 2>{}, A{}), yf(std::integral_constant<int, 2>{}, C{})}};
    st.apply(y, out[m], out[m + 1]);
  });
  if constexpr (M % 2) {
    using A = std::integral_constant<int, M - 1>;
    out[M - 1] = st.apply1(yf(std::integral_constant<int, 0>{}, A{}), yf(std::integral_constant<int, 1>{}, A{}),
                           yf(std::integral_constant<int, 2>{}, A{}));
  }
}

// shared memory of one warp (values of T): dofs rows, the nine-quantity modes
// of two faces, and with kSpec the modes of the gravitational faces
template <class T, int N, bool kSpec>
struct LocalSmem {
  using S = Shape<T, N>;
  static constexpr int nQ = (9 * EW * S::SB + 3) / 4 * 4, nT = (2 * 9 * EW * S::Bf + 3) / 4 * 4;
  static constexpr int nD = kSpec ? 4 * EW * (N + 1) * S::Bf : 0;
  static constexpr int nN = 16 * EW;  // the faces' normals
  static constexpr int warp = (nQ + nN + nT + nD + 3) / 4 * 4;
  static constexpr int bytes(int threads) { return warp * (int)sizeof(T) * (threads / 32); }
};

static __constant__ double kRowRcp[48] = {
    0.0, 1.0 / 1, 1.0 / 2, 1.0 / 3, 1.0 / 4, 1.0 / 5, 1.0 / 6, 1.0 / 7, 1.0 / 8, 1.0 / 9, 1.0 / 10, 1.0 / 11,
    1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16, 1.0 / 17, 1.0 / 18, 1.0 / 19, 1.0 / 20, 1.0 / 21, 1.0 / 22,
    1.0 / 23, 1.0 / 24, 1.0 / 25, 1.0 / 26, 1.0 / 27, 1.0 / 28, 1.0 / 29, 1.0 / 30, 1.0 / 31, 1.0 / 32, 1.0 / 33,
    1.0 / 34, 1.0 / 35, 1.0 / 36, 1.0 / 37, 1.0 / 38, 1.0 / 39, 1.0 / 40, 1.0 / 41, 1.0 / 42, 1.0 / 43, 1.0 / 44,
    1.0 / 45, 1.0 / 46, 1.0 / 47};
static __constant__ double kRowRcpFact[6] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120};

// D^{K+1} rows from D^K, then the next levels; I accumulates the time
// integral; lev(integral_constant<k>, D^k) sees every new level
template <class T, int N, int K, class Lev>
__device__ __forceinline__ void predict(const T* D, T* I, const RowStar<T>& st, const Seg& sg, Lev&& lev) {
  constexpr int L = nb3(N - K), M = nb3(N - K - 1);
  T Dn[M];
  star_rows<M>(st, Dn, [&](auto bc, auto mc) {
    constexpr int b = decltype(bc)::value, m = decltype(mc)::value;
    if constexpr (b == 0) return sp::dot<sp::KX, m, L>(T(0), D);
    else if constexpr (b == 1) return sp::dot<sp::KY, m, L>(T(0), D);
    else return sp::dot<sp::KZ, m, L>(T(0), D);
  });
  if constexpr (K == 0) {  // D^0 is not needed any more: its registers become I
    const T c0 = seg_tcoef<T>(sg, 0);
#pragma unroll
    for (int l = 0; l < L; ++l) I[l] = c0 * D[l];
  }
  const T ck = seg_tcoef<T>(sg, K + 1);
#pragma unroll
  for (int m = 0; m < M; ++m) I[m] = fma(ck, Dn[m], I[m]);
  lev(std::integral_constant<int, K + 1>{}, Dn);
  if constexpr (K + 1 < N) predict<T, N, K + 1>(Dn, I, st, sg, lev);
}

// the outward normals of the warp's faces into sN[4 j + f][4] (asynchronously)
template <class T>
__device__ __forceinline__ void normals_request(const StepArgs& a, T* sN, int64_t v0, int nE, int lane) {
  constexpr int V = 16 / (int)sizeof(T), C = 4 / V;
  for (int i = lane; i < nE * 4 * C; i += 32) {
    const int jf = i / C, c = (i % C) * V;
    tc::cp_async16(sN + jf * 4 + c, reinterpret_cast<const T*>(a.crec) +
                                        (elem_of(v0 + (jf >> 2), a.S) * 4 + (jf & 3)) * CREC + c);
  }
}
// the faces F0, F0 + 1 of the warp's elements: staged modes -> traction and
// velocity blocks of the trace array (and the LTS buffers, in FP64)
template <class T, int N, bool kSpec>
__device__ __forceinline__ void faces_out(const StepArgs& a, const Seg& sg, int64_t v0, int nE, int f0, const T* sT,
                                          const T* sN, int lane) {
  using S = Shape<T, N>;
  constexpr int Bf = S::Bf;
  T* const trace = reinterpret_cast<T*>(a.trace);
#pragma unroll(sizeof(T) == 4 ? 8 : 1)
  for (int it = 0; it < (2 * EW * Bf + 31) / 32; ++it) {
    const int i = lane + 32 * it, jf = i / Bf, n = i - jf * Bf, j = jf >> 1, f = f0 + (jf & 1);
    if (i >= nE * 2 * Bf) continue;
    const int64_t v = v0 + j;
    const T* const s = sT + ((jf & 1) * 9 * EW + 9 * j) * Bf + n;
    T q[9];
#pragma unroll
    for (int p = 0; p < 9; ++p) q[p] = s[p * Bf];
    const T* const c = sN + (4 * j + f) * 4;
    const T nx = c[0], ny = c[1], nz = c[2];
    const T o[6] = {fma(q[5], nz, fma(q[3], ny, q[0] * nx)), fma(q[4], nz, fma(q[1], ny, q[3] * nx)),
                    fma(q[2], nz, fma(q[4], ny, q[5] * nx)), q[6], q[7], q[8]};
    Vec<T, 2>* const out = reinterpret_cast<Vec<T, 2>*>(trace + (v * 4 + f) * S::FS + 6 * n);
#pragma unroll
    for (int k = 0; k < 3; ++k) out[k] = {o[2 * k], o[2 * k + 1]};
    if constexpr (kSpec) {
      if (sg.btrace_mode && a.bslot) {
        const int64_t e = elem_of(v, a.S);
        const int bs = a.bslot[e];
        if (bs >= 0) {
          double* const b = a.btrace + (((int64_t)bs * a.S + (v - e * a.S)) * 4 + f) * S::FS + 6 * n;
#pragma unroll
          for (int k = 0; k < 6; ++k) b[k] = (sg.btrace_mode == 1 ? 0.0 : b[k]) + (double)o[k];
        }
      }
    }
  }
}

// Acoustic elements (mu = 0, stress -p I; kept so by the solver when it runs with
// acoustic media): lane 4 j + p holds sigma_xx (p = 0) or a velocity of element j
// of eight; sigma_yy = sigma_zz = sigma_xx, no shear.
constexpr int EWF = kRowElemsFluid;
__device__ __forceinline__ int fluid_row(int r) { return 9 * (r >> 2) + ((r & 3) ? 5 + (r & 3) : 0); }  // of the dofs

// the warp's rows from shared memory to the dofs: the normal stress three times, the velocities
template <class T, int N>
__device__ __forceinline__ void fluid_rows_out(const T* sQ, T* Q, int nE, int lane) {
  using S = Shape<T, N>;
  using V = Vec<T, S::VW>;
  constexpr int C = S::B / S::VW;
#pragma unroll 4
  for (int i = lane; i < nE * 6 * C; i += 32) {
    const int r = i / C, c = (i - r * C) * S::VW, e = r / 6, q = r - e * 6;  // q = 0..2 the stresses, 3..5 the velocities
    const int sr = 4 * e + (q < 3 ? 0 : q - 2), gr = 9 * e + (q < 3 ? q : q + 3);
    *reinterpret_cast<V*>(Q + gr * S::B + c) = *reinterpret_cast<const V*>(sQ + sr * S::SB + c);
  }
}
// the normal of face f of element j, in lane 4 j + f (nE may be 0: nothing is read)
template <class T>
__device__ __forceinline__ void fluid_normal(const StepArgs& a, int64_t v0, int nE, int lane, T (&n)[3]) {
  const int64_t face = lane_face(v0, nE, lane, a.S);
  n[0] = n[1] = n[2] = T(0);
  if (face >= 0) {
    const T* const c = reinterpret_cast<const T*>(a.crec) + face * CREC;
#pragma unroll
    for (int d = 0; d < 3; ++d) n[d] = c[d];
  }
}
// Face f of the warp's elements, staged (sigma, v) modes -> face blocks; nrm: of
// fluid_normal.  (Read from global memory here, each of the four faces waits for
// its normals with every 32 modes: 40 % of the tensor-core kernel's time.)
template <class T, int N>
__device__ __forceinline__ void fluid_face_out(const StepArgs& a, int64_t v0, int nE, int f, const T* sT,
                                               const T (&nrm)[3], int lane) {
  constexpr int Bf = Shape<T, N>::Bf;
#pragma unroll(sizeof(T) == 4 ? 8 : 1)
  for (int it = 0; it < (EWF * Bf + 31) / 32; ++it) {
    const int i = lane + 32 * it, j = i / Bf, n = i - j * Bf;
    T c[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) c[d] = __shfl_sync(0xffffffffu, nrm[d], (4 * j + f) & 31);
    if (i >= nE * Bf) continue;
    const int64_t v = v0 + j;
    const T* const s = sT + 4 * j * Bf + n;
    Vec<T, 2>* const out =
        reinterpret_cast<Vec<T, 2>*>(reinterpret_cast<T*>(a.trace) + (v * 4 + f) * Shape<T, N>::FS + 6 * n);
    const T x = s[0];
    out[0] = {x * c[0], x * c[1]};
    out[1] = {x * c[2], s[Bf]};
    out[2] = {s[2 * Bf], s[3 * Bf]};
  }
}

// Faces that need more than their traces (kSpec): a finer neighbour integrates
// this element's Taylor expansion over its sub-steps, a fault's friction solve
// evaluates it at its time points, and a gravitational surface's ODE (Sec. 4.3)
// is driven by it.  All three read the derivatives' traces, formed level by
// level from the rows in registers with the sparse face projections (faces 0, 1
// and 2, 3 together, only where some element of the warp has such a face):
//   finer neighbour  the modal blocks of every level, to the derivative traces
//   fault            nine quantities at the face nodes (as the solve reads them)
//   gravity          the modes of v_n - sigma_nn / Z, kept in shared memory for
//                    surface() at the end
// No level outlives its registers.  kOneGrav: at most one gravitational face
// per element (the tensor-core kernels).
// A surface's forcing is a difference that cancels for incoming waves: 1 / Z is
// held in two values of T, so that the difference of the traces is exact to one
// rounding of the result, as if formed in FP64 (with 1 / Z rounded to FP32 it was
// 6e-3 off where the parts cancel to four millionths).  Its series is FP64.  (FP64
// differences and sums for FP32 dofs made steps of small FP32 meshes with a sea
// surface 2 to 9 % longer.  Error of eta against FP64 dofs, coupled boxes of 864
// and 648 tets, degrees 3 to 5, FP32 and 3xTF32: 1.0e-5 to 1.4e-5 after 1,500 steps,
// 0.7 to 1.03 times that of nodal traces with FP64 differences.)
template <class T, int N, bool kOneGrav>
struct SpecLevels {
  using S = Shape<T, N>;
  enum { NONE = 0, FINE = 1, GRAVITY = 2, FAULT = 3 };
  static constexpr int values = (kOneGrav ? 1 : 4) * EW * (N + 1) * S::Bf;  // of sF
  const StepArgs& a;
  bool on;            // this lane holds a row
  T *sT, *sF;         // staging as in faces_out; the surfaces' modes [face][level][Bf]
  const T* sN;
  int64_t v0;
  int nE, lane;
  int what, slot;     // lane 4 j + f: of face f of element j
  T iz, iz2;          // 1 / Z (gravity) rounded to T and what that leaves
  unsigned mask, surf;  // faces f to project; bit 4 j + f: a gravitational face
  __device__ __forceinline__ SpecLevels(const StepArgs& args, bool row, T* t, T* sf, const T* n, int64_t v, int e, int l)
      : a(args), on(row), sT(t), sF(sf), sN(n), v0(v), nE(e), lane(l), what(NONE), slot(-1), iz(T(0)),
        iz2(T(0)) {
    if (lane < 4 * nE) {
      const int64_t ef = elem_of(v0 + (lane >> 2), a.S) * 4 + (lane & 3);
      const int kind = (a.ninfo[ef] >> 5) & 7;
      if (kind == NK_FINE || kind == NK_FAULT) {
        what = kind == NK_FINE ? FINE : FAULT;
        slot = a.dslot[ef];
      } else if (a.gslot) {
        slot = a.gslot[ef];
        if (slot >= 0) {
          what = GRAVITY;
          const double r = 1.0 / a.gpar[(size_t)slot * GPAR + 3];
          iz = (T)r;
          iz2 = (T)(r - (double)iz);
        }
      }
    }
    const unsigned b = __ballot_sync(0xffffffffu, what != NONE);
    mask = (b | b >> 4 | b >> 8) & 15u;
    surf = __ballot_sync(0xffffffffu, what == GRAVITY);
  }
  __device__ __forceinline__ int scenario(int j) const {
    return a.S == 1 ? 0 : (int)(v0 + j - elem_of(v0 + j, a.S) * a.S);
  }
  // the surface modes of face f of element j
  __device__ __forceinline__ T* face_modes(int j, int f) const {
    return sF + (kOneGrav ? j : 4 * j + f) * (N + 1) * S::Bf;
  }
  template <int K, int F0>
  __device__ __forceinline__ void pair(const T* D) const {
    constexpr int L = nb3(N - K), Bk = nb2(N - K), Bf = S::Bf;  // (degree N - K: no higher modes)
    if (on) {
      T* const s0 = sT + lane * Bf;
      sp::each<Bk>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        if constexpr (F0 == 0) {
          const T ev = sp::dot<sp::R0, r, L, 0>(T(0), D), od = sp::dot<sp::R0, r, L, 1>(T(0), D);
          s0[r] = ev + od;
          s0[9 * EW * Bf + r] = ev - od;
        } else {
          s0[r] = sp::dot<sp::R2, r, L>(T(0), D);
          s0[9 * EW * Bf + r] = sp::dot<sp::R3, r, L>(T(0), D);
        }
      });
    }
    __syncwarp();
#pragma unroll 1
    for (int i = lane; i < (2 * EW * Bf + 31) / 32 * 32; i += 32) {
      const int jf = i / Bf, n = i - jf * Bf, j = jf >> 1, f = F0 + (jf & 1);
      const int w = __shfl_sync(0xffffffffu, what, (4 * j + f) & 31), sl = __shfl_sync(0xffffffffu, slot, (4 * j + f) & 31);
      const T z = __shfl_sync(0xffffffffu, iz, (4 * j + f) & 31), z2 = __shfl_sync(0xffffffffu, iz2, (4 * j + f) & 31);
      if (j >= nE || w == NONE) continue;
      const T* const s = sT + ((jf & 1) * 9 * EW + 9 * j) * Bf;
      T* const d = reinterpret_cast<T*>(a.dtrace) + ((int64_t)sl * a.S + scenario(j)) * (N + 1) * 9 * Bf;
      T q[9];
      if (w == FAULT) {
#pragma unroll
        for (int p = 0; p < 9; ++p) q[p] = T(0);
        const T* const nd = reinterpret_cast<const T*>(a.nodalT) + n;
#pragma unroll 3
        for (int r = 0; r < Bk; ++r) {
          const T x = nd[r * Bf];
#pragma unroll
          for (int p = 0; p < 9; ++p) q[p] = fma(x, s[p * Bf + r], q[p]);
        }
#pragma unroll
        for (int p = 0; p < 9; ++p) d[(K * 9 + p) * Bf + n] = q[p];
        continue;
      }
      const T* const c = sN + (4 * j + f) * 4;
#pragma unroll
      for (int p = 0; p < 9; ++p) q[p] = n < Bk ? s[p * Bf + n] : T(0);
      const T o[6] = {fma(q[5], c[2], fma(q[3], c[1], q[0] * c[0])), fma(q[4], c[2], fma(q[1], c[1], q[3] * c[0])),
                      fma(q[2], c[2], fma(q[4], c[1], q[5] * c[0])), q[6], q[7], q[8]};
      if (w == FINE) {
#pragma unroll
        for (int k = 0; k < 6; ++k) d[K * S::FS + 6 * n + k] = o[k];
      } else {
        const T vn = fma(o[5], c[2], fma(o[4], c[1], o[3] * c[0])), tn = fma(o[2], c[2], fma(o[1], c[1], o[0] * c[0]));
        face_modes(j, f)[K * Bf + n] = fma(-tn, z2, fma(-tn, z, vn));
      }
    }
    __syncwarp();
  }
  template <int K>
  __device__ __forceinline__ void operator()(std::integral_constant<int, K>, const T* D) const {
    if (mask & 3u) pair<K, 0>(D);
    if (mask & 12u) pair<K, 2>(D);
  }
  // The gravitational surfaces over the step, up to three faces at a time, one
  // (face, node) per lane: f_m = modes of level m at the node / m!, the (eta, H)
  // series in FP64, then the modes of -rho g H and eta^{n+1} - eta^n.
  __device__ void surface(const Seg& sg) const {
    constexpr int Bf = S::Bf;
    unsigned left = surf;
    while (left) {
      int face[EW];  // 4 j + f, or -1
#pragma unroll
      for (int c = 0; c < EW; ++c) {
        face[c] = __ffs(left) - 1;
        left &= left - 1;
      }
      auto which = [&](int c) { return c == 0 ? face[0] : c == 1 ? face[1] : face[2]; };
#pragma unroll 1
      for (int it = 0; it < (EW * Bf + 31) / 32; ++it) {
        const int i = lane + 32 * it, c = i < EW * Bf ? i / Bf : 0, n = i - c * Bf, jf = which(c);
        const int gs = __shfl_sync(0xffffffffu, slot, jf & 31);
        if (i >= EW * Bf || jf < 0) continue;
        const T* const F = face_modes(jf >> 2, jf & 3);
        const double* const gp = a.gpar + (size_t)gs * GPAR;
        double* const eta = a.eta + ((int64_t)gs * a.S + scenario(jf >> 2)) * Bf + n;
        const double kappa = gp[4], rg = gp[5], dt = sg.dt, eta0 = *eta;
        const T* const nd = reinterpret_cast<const T*>(a.nodalT) + n;
        T acc[N + 1];
#pragma unroll
        for (int m = 0; m <= N; ++m) acc[m] = T(0);
#pragma unroll
        for (int r = 0; r < Bf; ++r) {
          const T w = nd[r * Bf];
#pragma unroll
          for (int m = 0; m <= N; ++m)
            if (r < nb2(N - m)) acc[m] = fma(w, F[m * Bf + r], acc[m]);
        }
        double cm = eta0, e1 = eta0, H = eta0 * dt, pw = 1.0;
        auto term = [&](int m, double fv) {
          cm = (fv - kappa * cm) * kRowRcp[m + 1];
          pw *= dt;
          const double t = cm * pw;
          e1 += t;
          H += t * dt * kRowRcp[m + 2];
          return t;
        };
#pragma unroll
        for (int m = 0; m <= N; ++m) term(m, (double)acc[m] * kRowRcpFact[m]);
#pragma unroll 1
        for (int m = N + 1; m < N + 40; ++m)
          if (fabs(term(m, 0.0)) <= 1e-17 * fabs(e1)) break;
        *eta = e1;
        sT[c * 2 * Bf + n] = (T)(-rg * H);
        sT[(c * 2 + 1) * Bf + n] = (T)(e1 - eta0);
      }
      __syncwarp();
#pragma unroll 1
      for (int it = 0; it < (EW * Bf + 31) / 32; ++it) {
        const int i = lane + 32 * it, c = i < EW * Bf ? i / Bf : 0, r = i - c * Bf, jf = which(c);
        const int gs = __shfl_sync(0xffffffffu, slot, jf & 31);
        if (i >= EW * Bf || jf < 0) continue;
        const T* const mn = reinterpret_cast<const T*>(a.modalT) + r;
        T h = T(0), d = T(0);
#pragma unroll
        for (int n = 0; n < Bf; ++n) {
          const T w = mn[n * Bf];
          h = fma(w, sT[c * 2 * Bf + n], h);
          d = fma(w, sT[(c * 2 + 1) * Bf + n], d);
        }
        T* const out = reinterpret_cast<T*>(a.gflux) + ((int64_t)gs * a.S + scenario(jf >> 2)) * 9 * Bf + r;
        out[0] = h;
        out[Bf] = d;
      }
      __syncwarp();
    }
  }
};
struct NoLevels {
  template <int K, class T>
  __device__ __forceinline__ void operator()(std::integral_constant<int, K>, const T*) const {}
};

// row -= this lane's row of the volume term sum_a A*_a K_a I
template <class T, int N>
__device__ __forceinline__ void volume_row(const RowStar<T>& st, const T* I, bool valid, T* row) {
  using S = Shape<T, N>;
  constexpr int VW = S::VW;
  sp::each<S::B / VW>([&](auto cc) {
    constexpr int m0 = decltype(cc)::value * VW;
    T x[VW];
    star_rows<VW>(st, x, [&](auto bc, auto kc) {
      constexpr int b = decltype(bc)::value, m = m0 + decltype(kc)::value;
      if constexpr (b == 0) return sp::dot<sp::KXt, m, S::B1>(T(0), I);
      else if constexpr (b == 1) return sp::dot<sp::KYt, m, S::B1>(T(0), I);
      else return sp::dot<sp::KZt, m, S::B1>(T(0), I);
    });
    if (valid) {
      Vec<T, VW> q = *reinterpret_cast<const Vec<T, VW>*>(row + m0);
#pragma unroll
      for (int k = 0; k < VW; ++k) q.x[k] -= x[k];
      *reinterpret_cast<Vec<T, VW>*>(row + m0) = q;
    }
  });
}

template <class T, int N, bool kSpec>
__global__ void __launch_bounds__(kMaxThreads, sizeof(T) == 4 ? 2 : 1) local_row_kernel(StepArgs a, const __grid_constant__ Segs g) {
  using S = Shape<T, N>;
  using M = LocalSmem<T, N, kSpec>;
  constexpr int B = S::B, Bf = S::Bf, VW = S::VW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  T* const sQ = reinterpret_cast<T*>(smem_raw) + (threadIdx.x >> 5) * M::warp;
  T* const sN = sQ + M::nQ;
  T* const sT = sN + M::nN;
  const Unit u = unit_of(g);
  if (u.nE == 0) return;
  const Seg& sg = g.s[u.seg];
  T* const Q = reinterpret_cast<T*>(a.Q) + u.v0 * 9 * B;
  normals_request(a, sN, u.v0, u.nE, lane);
  tc::cp_async_commit();
  rows_in<T, N>(sQ, Q, u.nE, lane);
  const int j = lane / 9;
  const bool valid = lane < 9 * u.nE;
  RowStar<T> st;
  st.setup(lane, valid, reinterpret_cast<const T*>(a.par) + elem_of(u.v0 + (valid ? j : 0), a.S) * PAR);
  T* const row = sQ + (valid ? lane : 0) * S::SB;
  __syncwarp();

  // ---- D^0, the predictor levels and the time integral
  T I[B];
#pragma unroll
  for (int c = 0; c < B / VW; ++c) {
    const Vec<T, VW> x = *reinterpret_cast<const Vec<T, VW>*>(row + c * VW);
#pragma unroll
    for (int k = 0; k < VW; ++k) I[c * VW + k] = valid ? x.x[k] : T(0);
  }
  if constexpr (kSpec) {
    tc::cp_async_wait<0>();
    __syncwarp();  // the normals
  }
  std::conditional_t<kSpec, SpecLevels<T, N, false>, NoLevels> lev = [&] {
    if constexpr (kSpec) return SpecLevels<T, N, false>(a, valid, sT, sT + M::nT, sN, u.v0, u.nE, lane);
    else return NoLevels{};
  }();
  lev(std::integral_constant<int, 0>{}, I);
  predict<T, N, 0>(I, I, st, sg, lev);

  // ---- modal face traces, two faces at a time through shared memory
  {
    T* const s0 = sT + lane * Bf;
    if (valid) {
      sp::each<Bf>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        const T ev = sp::dot<sp::R0, r, B, 0>(T(0), I), od = sp::dot<sp::R0, r, B, 1>(T(0), I);
        s0[r] = ev + od;
        s0[9 * EW * Bf + r] = ev - od;
      });
    }
    tc::cp_async_wait<0>();
    __syncwarp();
    faces_out<T, N, kSpec>(a, sg, u.v0, u.nE, 0, sT, sN, lane);
    __syncwarp();
    if (valid) {
      sp::each<Bf>([&](auto rc) {
        constexpr int r = decltype(rc)::value;
        s0[r] = sp::dot<sp::R2, r, B>(T(0), I);
        s0[9 * EW * Bf + r] = sp::dot<sp::R3, r, B>(T(0), I);
      });
    }
    __syncwarp();
    faces_out<T, N, kSpec>(a, sg, u.v0, u.nE, 2, sT, sN, lane);
  }

  // ---- volume term (face terms follow in the neighbour kernel)
  volume_row<T, N>(st, I, valid, row);
  __syncwarp();
  rows_out<T, N>(sQ, Q, u.nE, lane);
  if constexpr (kSpec) lev.surface(sg);
}

// Acoustic elements without any special face: four rows instead of nine, eight
// elements per warp, otherwise as local_row_kernel.  What bounds it and where
// the rows wait is the same; the work is 4 / 9.
template <class T, int N>
struct FluidSmem {
  using S = Shape<T, N>;
  static constexpr int nQ = (32 * S::SB + 3) / 4 * 4, warp = (nQ + 2 * 32 * S::Bf + 3) / 4 * 4;
  static constexpr int bytes(int threads) { return warp * (int)sizeof(T) * (threads / 32); }
  static_assert(bytes(kMaxThreads) <= 232448, "acoustic row kernel exceeds the shared memory of one block");
};
template <class T, int N>
__global__ void __launch_bounds__(kMaxThreads, sizeof(T) == 4 ? 2 : 1) local_fluid_kernel(StepArgs a, const __grid_constant__ Segs g) {
  using S = Shape<T, N>;
  using M = FluidSmem<T, N>;
  constexpr int B = S::B, Bf = S::Bf, VW = S::VW, C = B / VW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31;
  T* const sQ = reinterpret_cast<T*>(smem_raw) + (threadIdx.x >> 5) * M::warp;
  T* const sT = sQ + M::nQ;
  const Unit u = unit_of<EWF>(g);
  if (u.nE == 0) return;
  T* const Q = reinterpret_cast<T*>(a.Q) + u.v0 * 9 * B;
  for (int i = lane; i < 4 * u.nE * C; i += 32) {
    const int r = i / C, c = (i - r * C) * VW;
    *reinterpret_cast<Vec<T, VW>*>(sQ + r * S::SB + c) =
        *reinterpret_cast<const Vec<T, VW>*>(Q + fluid_row(r) * B + c);
  }
  const bool valid = lane < 4 * u.nE;
  RowStar<T> st;
  st.setup_acoustic(lane, valid, reinterpret_cast<const T*>(a.par) + elem_of(u.v0 + (valid ? lane >> 2 : 0), a.S) * PAR);
  T* const row = sQ + (valid ? lane : 0) * S::SB;
  __syncwarp();
  T I[B];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const Vec<T, VW> x = *reinterpret_cast<const Vec<T, VW>*>(row + c * VW);
#pragma unroll
    for (int k = 0; k < VW; ++k) I[c * VW + k] = valid ? x.x[k] : T(0);
  }
  predict<T, N, 0>(I, I, st, g.s[u.seg], NoLevels{});
  T nrm[3];
  fluid_normal(a, u.v0, u.nE, lane, nrm);
  T* const s0 = sT + lane * Bf;
  if (valid) {
    sp::each<Bf>([&](auto rc) {
      constexpr int r = decltype(rc)::value;
      const T ev = sp::dot<sp::R0, r, B, 0>(T(0), I), od = sp::dot<sp::R0, r, B, 1>(T(0), I);
      s0[r] = ev + od;
      s0[32 * Bf + r] = ev - od;
    });
  }
  __syncwarp();
  fluid_face_out<T, N>(a, u.v0, u.nE, 0, sT, nrm, lane);
  fluid_face_out<T, N>(a, u.v0, u.nE, 1, sT + 32 * Bf, nrm, lane);
  __syncwarp();
  if (valid) {
    sp::each<Bf>([&](auto rc) {
      constexpr int r = decltype(rc)::value;
      s0[r] = sp::dot<sp::R2, r, B>(T(0), I);
      s0[32 * Bf + r] = sp::dot<sp::R3, r, B>(T(0), I);
    });
  }
  __syncwarp();
  fluid_face_out<T, N>(a, u.v0, u.nE, 2, sT, nrm, lane);
  fluid_face_out<T, N>(a, u.v0, u.nE, 3, sT + 32 * Bf, nrm, lane);
  volume_row<T, N>(st, I, valid, row);
  __syncwarp();
  fluid_rows_out<T, N>(sQ, Q, u.nE, lane);
}

template <class T, int N>
int launch_local_fluid_t(const StepArgs& a, const Segs& g, int threads, cudaStream_t st) {
  using M = FluidSmem<T, N>;
  const int rc = configure_on_device((const void*)local_fluid_kernel<T, N>, [] {
    return cudaFuncSetAttribute(local_fluid_kernel<T, N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                M::bytes(kMaxThreads));
  });
  if (rc) return rc;
  const int64_t units = g.n ? g.first[g.n] : 0;
  if (units <= 0) return 0;
  threads = block_threads<T, N>(threads, units, a.n_sms);
  if (threads < 32 || threads > kMaxThreads || threads % 32) return (int)cudaErrorInvalidValue;
  const int w = threads / 32;
  local_fluid_kernel<T, N><<<(unsigned)((units + w - 1) / w), threads, M::bytes(threads), st>>>(a, g);
  return (int)cudaGetLastError();
}

template <class T, int N>
int launch_local_row_t(const StepArgs& a, const Segs& g, int threads, bool spec, cudaStream_t st) {
  const int rc = configure_on_device((const void*)local_row_kernel<T, N, false>, [] {
    cudaError_t ce = cudaFuncSetAttribute(local_row_kernel<T, N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          LocalSmem<T, N, false>::bytes(kMaxThreads));
    if (ce == cudaSuccess)
      ce = cudaFuncSetAttribute(local_row_kernel<T, N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                LocalSmem<T, N, true>::bytes(128));
    return ce;
  });
  if (rc) return rc;
  const int64_t units = g.n ? g.first[g.n] : 0;
  if (units <= 0) return 0;
  threads = block_threads<T, N>(threads, units, a.n_sms);
  if (threads < 32 || threads > kMaxThreads || threads % 32) return (int)cudaErrorInvalidValue;
  if (spec && threads > 128) threads = 128;  // (shared memory)
  const int w = threads / 32;
  const unsigned blocks = (unsigned)((units + w - 1) / w);
  if (spec)
    local_row_kernel<T, N, true><<<blocks, threads, LocalSmem<T, N, true>::bytes(threads), st>>>(a, g);
  else
    local_row_kernel<T, N, false><<<blocks, threads, LocalSmem<T, N, false>::bytes(threads), st>>>(a, g);
  return (int)cudaGetLastError();
}

template <class T>
int launch_local_fluid_n(int N, const StepArgs& a, const Segs& g, int th, cudaStream_t st) {
  switch (N) {
    case 1: return launch_local_fluid_t<T, 1>(a, g, th, st);
    case 2: return launch_local_fluid_t<T, 2>(a, g, th, st);
    case 3: return launch_local_fluid_t<T, 3>(a, g, th, st);
    case 4: return launch_local_fluid_t<T, 4>(a, g, th, st);
    case 5: return launch_local_fluid_t<T, 5>(a, g, th, st);
  }
  return (int)cudaErrorInvalidValue;
}

template <class T>
int launch_local_row_n(int N, const StepArgs& a, const Segs& g, int th, bool spec, cudaStream_t st) {
  switch (N) {
    case 1: return launch_local_row_t<T, 1>(a, g, th, spec, st);
    case 2: return launch_local_row_t<T, 2>(a, g, th, spec, st);
    case 3: return launch_local_row_t<T, 3>(a, g, th, spec, st);
    case 4: return launch_local_row_t<T, 4>(a, g, th, spec, st);
    case 5: return launch_local_row_t<T, 5>(a, g, th, spec, st);
  }
  return (int)cudaErrorInvalidValue;
}

}  // namespace row
}  // namespace adg
