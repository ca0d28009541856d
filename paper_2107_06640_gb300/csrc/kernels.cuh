// ADER-DG element-update kernels: what they compute, their arguments and launchers.
//
// Per element v (virtual index; ensembles stack S scenarios per element) over
// one own step:
//   local kernel      Sec. 4.1: Cauchy-Kovalewski predictor
//                       D^{k+1} = -sum_a KT_a D^k A*_a^T,  KT_a[m][l] = int phi_m dphi_l/dxi_a,
//                     time integral I = sum_k dt^{k+1}/(k+1)! D^k (Eq. taylor),
//                     volume sum_a K_a I A*_a^T, traction and velocity of its
//                     faces in the faces' modes (and LTS buffers / derivative
//                     traces); gravitational faces (Sec. 4.3): exact (eta, H)
//                     Taylor recursion in FP64 at the face nodes, driven by the
//                     derivatives' traces, and the modes of the integrated
//                     normal state int w1^b = -rho g H, int w7^b = eta^{n+1} - eta^n.
//   neighbour kernel  Godunov fluxes of all four faces (Sec. 4.2, Eq.
//                     numerical-flux) mode by mode: the neighbour's modes
//                     re-oriented to this side's, one middle state from the
//                     face's coefficients (face_flux_state), gravitational
//                     surfaces' normal states and fault fluxes added; one lift.
// Dofs layout: Q[v][9][B] (basis fastest).  Face data: modal, see row_common.cuh.
#pragma once
#include <cmath>
#include <cstdint>

namespace adg {

__host__ __device__ constexpr int nb3(int n) { return n < 0 ? 0 : (n + 1) * (n + 2) * (n + 3) / 6; }
__host__ __device__ constexpr int nb2(int n) { return (n + 1) * (n + 2) / 2; }
// values of one face in the trace array: traction and velocity in the face's
// modes, [Bf][6], padded to a multiple of 4 so that a block starts on 16 bytes
__host__ __device__ constexpr int face_block(int n) { return (6 * nb2(n) + 3) / 4 * 4; }
// values that the trace array (also the scratch of the FP32 dofs transfers) holds per face
__host__ __device__ constexpr int face_stride(int n) { return (9 * nb2(n) + 3) / 4 * 4; }

// neighbour-face kinds (ninfo bits 5..7)
enum { NK_NONE = 0, NK_SAME = 1, NK_COARSE = 2, NK_FINE = 3, NK_FAULT = 4 };

// per-element parameters (stride PAR): Jinv[9] (d xi_a/d x_d, row a), rho, lam, mu, scale[4]
constexpr int PAR = 16;
// per-gravity-face parameters (double, stride GPAR):
//   n[3], Z, kappa = rho g / Z, rho*g
constexpr int GPAR = 6;

// the tensor-core kernels that have a tile counter of their own
enum { TILES_ELASTIC = 0, TILES_BUFFER, TILES_FLUID, TILES_SPECIAL, TILES_NEIGHBOUR, kTileKinds };

struct StepArgs {
  void* Q;              // T [V][9][B]
  void* trace;          // T [V][4][face_block(N)]
  double* btrace;       // [nbslot*S][4][face_block(N)]  (LTS buffer, FP64)
  void* dtrace;         // T [ndslot*S][N+1][9][Bf] (derivative traces; modal blocks, at fault faces nodal)
  double* eta;          // [ngslot*S][Bf]
  const void* par;      // T [E][PAR]
  const int* nbr;       // [E][4] internal neighbour element or -1
  const int* ninfo;     // [E][4] j | perm<<2 | kind<<5
  const int* gslot;     // [E][4] gravity slot or -1
  const int* bslot;     // [E]    LTS buffer slot or -1
  const int* dslot;     // [E][4] LTS derivative-trace slot or -1
  const double* gpar;   // [ngslot][GPAR]
  int S;                // ensemble size
  unsigned int* err;    // device error word
  const int* fslot;     // [E][4] 2*fault + side for fault faces, else -1
  const void* drout;    // T [nff*S][2][9][Bf] time-integrated fault flux per side
  void* gflux;          // T [ngslot*S][9][Bf], the first two rows: the modes of the time-integrated normal
                        // traction -rho g H and normal velocity of gravitational faces
  int* tiles;            // [kTileKinds][2] tile counters of the tensor-core kernels (tc::TileFeed)
  const float* tc_local; // tensor-core operands of the local kernel (hi/lo, canonical layout), degree 5 or 4
  const float* tc_lift;  // tensor-core lift operand of the neighbour kernel (hi/lo, canonical layout), degree 5 or 4
  const void* crec;      // T [E][4][CREC] face coefficients
  const void* nodalT;    // T [Bf(r)][Bf(n)]    face modes at the face nodes, r-major
  const void* modalT;    // T [Bf(n)][Bf(r)]    face nodes to face modes, n-major
  int n_sms;             // of the context's GPU (read by the launchers)
  const void* reorient;  // T [6][sum (n+1)^2]  a neighbour's face modes in this side's, blocks by degree
};
// Element of a virtual element, S scenarios per element: the 64-bit division
// (some 100 instructions) only where it is needed.
__host__ __device__ inline int64_t elem_of(int64_t v, int S) {
  if (S == 1) return v;
  if ((v >> 32) == 0) return (int64_t)((uint32_t)v / (uint32_t)S);
  return v / S;
}
// Virtual elements per warp of the row kernels
constexpr int kRowElems = 3;
constexpr int kRowElemsFluid = 8;  // of its acoustic form
constexpr int kSmallLaunchWarps = 8;  // warps per SM of a row launch that counts as small
// Face coefficients: outward normal n[3]; the middle
// state's tangential coefficients of the own and of the neighbour's side (t^b
// from t and v, v^b from t and v) and of both sides' normal components (t^b: what
// they add to the tangential product, v^b: the normal velocity itself), the
// neighbour's traction taken with its own normal; then
// -s_f lambda, -s_f mu, -s_f / rho of the element (s_f = 2|S_f|/|J|); padding.
constexpr int CREC = 24;
// The scaled flux s_f T A^- w^b of one mode (or point) of a face: c the face's
// coefficients, q and w the own and the neighbour's traction and velocity (each
// traction with its owner's outward normal), srt and srv a gravitational surface's
// normal traction and velocity.
// The normal velocity state vs is formed by itself and goes into the lambda
// rows directly.  The tangential velocity coefficients hold 1 / Z_s: in a soft
// solid (Z_s << Z_p) the normal part of their product is large, and what is left
// of it in vb.n after the subtraction is rounding of that size, which the mu rows
// bear (mu / Z_s is small) and the lambda rows do not (FP32, v_s 50 m/s beside
// water: 3e-6 of the row where this form has 8e-8).
template <class T>
__host__ __device__ __forceinline__ void face_flux_state(const T* c, const T* q, const T* w, T srt, T srv, T* g) {
  const T tn = fma(q[2], c[2], fma(q[1], c[1], q[0] * c[0])), vn = fma(q[5], c[2], fma(q[4], c[1], q[3] * c[0]));
  const T tm = fma(w[2], c[2], fma(w[1], c[1], w[0] * c[0])), vm = fma(w[5], c[2], fma(w[4], c[1], w[3] * c[0]));
  const T an = fma(c[11], tn, fma(c[12], vn, fma(c[15], tm, fma(c[16], vm, srt))));
  const T vs = fma(c[13], tn, fma(c[14], vn, fma(c[17], tm, fma(c[18], vm, srv))));
  const T bn = vs - fma(c[5], tn, fma(c[6], vn, fma(c[9], tm, c[10] * vm)));
  T tb[3], vb[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    tb[d] = fma(an, c[d], fma(c[3], q[d], fma(c[4], q[3 + d], fma(c[7], w[d], c[8] * w[3 + d]))));
    vb[d] = fma(bn, c[d], fma(c[5], q[d], fma(c[6], q[3 + d], fma(c[9], w[d], c[10] * w[3 + d]))));
  }
  const T l = c[19] * vs;
  const T m[3] = {c[20] * vb[0], c[20] * vb[1], c[20] * vb[2]};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    g[d] = fma(T(2) * c[d], m[d], l);
    g[6 + d] = c[21] * tb[d];
  }
  g[3] = fma(c[0], m[1], c[1] * m[0]);
  g[4] = fma(c[1], m[2], c[2] * m[1]);
  g[5] = fma(c[0], m[2], c[2] * m[0]);
}
// The clusters of one LTS phase (Sec. 4.4) in a single launch: segment i
// covers the virtual elements [v_begin, v_begin + n) of one cluster with that
// cluster's time coefficients, and the launch's work units (tiles of the
// tensor-core kernels, warps of the row kernels) [first[i], first[i+1]).
// The launch takes the table by value (kernel parameter space), so a CUDA
// graph keeps it and no device buffer is involved.
constexpr int kMaxSeg = 16;
// virtual elements per tile of the tensor-core kernels (12 x 9 quantities =
// the 128 rows of one MMA)
constexpr int kTileElems = 12;
// ... and of the acoustic (4-quantity, ocean) instantiation of the local one
constexpr int kTileElemsFluid = 32;
struct Seg {
  int64_t v_begin, n;
  double tcoef[8];   // dt^{k+1}/(k+1)!, k = 0..N (the cluster's own step)
  double ccoef[8];   // (tb^{k+1}-ta^{k+1})/(k+1)! on a coarser neighbour's expansion
  float tcoef32[8], ccoef32[8];  // the same in FP32 (make_segs): a conversion in the kernel would run on the FP64 pipe
  double dt;         // the cluster's step (gravity ODE)
  int btrace_mode;   // 0 none, 1 overwrite, 2 accumulate (LTS buffers)
};
template <class T>
__host__ __device__ inline T seg_tcoef(const Seg& s, int k) {
  if constexpr (sizeof(T) == 4) return s.tcoef32[k]; else return s.tcoef[k];
}
template <class T>
__host__ __device__ inline T seg_ccoef(const Seg& s, int k) {
  if constexpr (sizeof(T) == 4) return s.ccoef32[k]; else return s.ccoef[k];
}
struct Segs {
  int n;                        // segments
  int chunk;                    // tensor-core kernels: consecutive tiles a CTA slot takes at a time
  int64_t first[kMaxSeg + 1];   // first work unit of each segment; first[n] = all units
  Seg s[kMaxSeg];
};
// segment of work unit u (segments are few: a linear scan)
__host__ __device__ inline int seg_find(const Segs& g, int64_t u) {
  int i = 0;
  while (i + 1 < g.n && u >= g.first[i + 1]) ++i;
  return i;
}
// The part of tile `tl` (TE virtual elements) that warp `w` of a slot works on, EW
// elements each: first virtual element, elements, segment.  Warps past a segment's
// end have nE = 0 and a v0 that is no element of the launch: nothing may be read there.
struct TilePart {
  int64_t v0;
  int nE, seg;
};
template <int TE, int EW>
__host__ __device__ inline TilePart tile_part(const Segs& g, int64_t tl, int w) {
  const int i = seg_find(g, tl);
  const int64_t o = (tl - g.first[i]) * TE + EW * w, left = g.s[i].n - o;
  return {g.s[i].v_begin + o, (int)(left < 0 ? 0 : left < EW ? left : EW), i};
}
// Face 4 element + f that lane 4 j + f of a warp with elements v0 .. v0 + nE - 1 stands for; -1: none
__host__ __device__ inline int64_t lane_face(int64_t v0, int nE, int lane, int S) {
  return lane < 4 * nE ? elem_of(v0 + (lane >> 2), S) * 4 + (lane & 3) : -1;
}
// Segs of the given segments with `unit` virtual elements per work unit
Segs make_segs(const Seg* s, int n, int unit, int chunk = 1);

// tensor-core (tcgen05, 3xTF32) local kernel, degree 5 or 4, FP32 dofs
// (local_tc.cuh; one translation unit per degree), for elements without fault
// faces or two or more gravitational faces
// buffers: the launch's elements include some with an LTS buffer (a coarser neighbour)
// acoustic: the launch's elements are fluid (mu = 0) without LTS buffer, on the
// 4-quantity (p, v) instantiation; their stress must be isotropic (-p I)
// (other degrees: cudaErrorInvalidValue)
// grav: the launch's elements have one gravitational face or a finer LTS
// neighbour (elastic instantiation; the face's (eta, H) update in FP64 and
// the derivative traces of every level on faces with a finer neighbour)
int launch_local_tc(int degree, const StepArgs& a, const Segs& g, int n_sms, void* stream, bool buffers,
                    bool acoustic = false, bool grav = false);
void pack_local_tc(int degree, const double* kt, const double* kvol, const double* rfc, float* out);
int local_tc_floats(int degree);
// tensor-core (tcgen05, 3xTF32) neighbour kernel, degree 5 or 4, FP32 dofs
// (neighbour_tc.cuh), for the same elements
// lts: the launch's elements include some with a neighbour in another cluster or a gravitational face
int launch_neighbour_tc(int degree, const StepArgs& a, const Segs& g, int n_sms, void* stream, bool lts);
void pack_lift_tc(int degree, const double* rfc, float* out);
int lift_tc_floats(int degree);

// ---- dynamic rupture (rupture.cu) ----
// per-node fault parameters (double, stride FPAR), in this order:
//   a, b, L, f0, V0, f_w, V_w, sigma_n0, tau0_x, tau0_y, tau0_z, psi_init, V_init
// (linear slip weakening: mu_s, mu_d, D_c, cohesion in the first four slots)
constexpr int FPAR = 13;
// per-node fault state (double, stride FSTATE): |V|, psi, slip_xyz, traction_xyz
constexpr int FSTATE = 8;
// per-fault-face geometry (double, stride FGEO): n (minus outward), rho-, lam-, mu-, rho+, lam+, mu+
constexpr int FGEO = 9;
// friction-guess network: inputs, hidden width (two tanh layers), parameters
constexpr int MLP_IN = 6, MLP_H = 32;
constexpr int MLP_NPARAM = MLP_IN * MLP_H + MLP_H + MLP_H * MLP_H + MLP_H + MLP_H + 1 + 2 * MLP_IN + 2;

struct DRArgs {
  const void* dtrace;   // derivative traces of both sides (see StepArgs)
  const int* dslot;
  const int* fface;     // [nff][5] minus elem, minus face, plus elem, plus face, perm
  const double* fgeo;   // [nff][FGEO]
  const double* fpar;   // [nff*S][Bf][FPAR]
  double* fstate;       // [nff*S][Bf][FSTATE]
  void* drout;          // T [nff*S][2][9][Bf]
  const int* perm;      // [6][Bf]
  int64_t f_begin, n_faces;
  int S;
  double dt;
  double tp[8], tw[8];  // Gauss-Legendre time points / weights on [0, dt]
  double tk[6][6];      // Taylor weights of the time points, tp[j]^k / k!
  unsigned long long* newton;  // [0] solves, [1] iterations
  unsigned int* err;
  const float* mlp;     // network parameters (or null: plain start)
  float* capture;       // training samples [cap][MLP_IN + 1] (or null)
  unsigned long long* cap_count;
  int64_t cap_capacity;
  int law;              // FRIC_RS or FRIC_LSW
};

enum { FRIC_RS = 0, FRIC_LSW = 1 };  // the ADG_FRICTION_* values of adg.h

// (no faces: the kernels are configured on the current device, nothing is launched)
int launch_rupture(int fp64, int N, const DRArgs& a, void* stream);

enum { ERR_NAN = 1u, ERR_TIMEOUT = 2u, ERR_NEWTON = 4u };

// host-side launchers; return cudaError_t as int
// (threads: per block, a multiple of 32 up to 256; 0: by row::block_threads)
// row kernels (row_local.cuh, row_neighbour.cuh): both precisions, every degree;
// spec: the launch's elements may have gravitational or fault faces or
// neighbours in another cluster
int launch_local_row(int fp64, int N, const StepArgs& a, const Segs& g, void* stream, int threads, bool spec);
int launch_neighbour_row(int fp64, int N, const StepArgs& a, const Segs& g, void* stream, int threads, bool spec);
// the local row kernel of plain acoustic elements (adg_set_acoustic_ocean)
int launch_local_fluid(int fp64, int N, const StepArgs& a, const Segs& g, void* stream, int threads);

}  // namespace adg
