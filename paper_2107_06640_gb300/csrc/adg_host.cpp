// Host side of the C ABI (include/adg.h): mesh set-up, geometry, clustering,
// coefficients of the face fluxes, device memory, the rate-2 LTS tick schedule and the
// per-macro-step CUDA graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <functional>
#include <map>
#include <stdexcept>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/adg.h"
#include "kernels.cuh"
#include "refmat.hpp"
#include "adg_internal.hpp"

using namespace adg;

namespace {

const int kFaceV[4][3] = {{1, 2, 3}, {0, 2, 3}, {0, 1, 3}, {0, 1, 2}};

using Err = adg::AdgError;

#define CK(call)                                                                          \
  do {                                                                                    \
    cudaError_t _e = (call);                                                              \
    if (_e != cudaSuccess) throw Err(ADG_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(_e)); \
  } while (0)

// ---------------- 9x9 matrices (row-major) ----------------
typedef std::array<double, 81> M9;

// x-Jacobian of Eq. (elasticity-pde) (the rotated 1-D problem uses A only)
M9 jac_x(double rho, double lam, double mu) {
  M9 A{};
  A[0 * 9 + 6] = -(lam + 2 * mu);
  A[1 * 9 + 6] = -lam;
  A[2 * 9 + 6] = -lam;
  A[3 * 9 + 7] = -mu;
  A[5 * 9 + 8] = -mu;
  A[6 * 9 + 0] = -1.0 / rho;
  A[7 * 9 + 3] = -1.0 / rho;
  A[8 * 9 + 5] = -1.0 / rho;
  return A;
}

// Middle state w^b = Mm w^- + Mp w^+ (Sec. 4.2, Eq. boundary-state; solid-solid
// shear with the same welded form using Z_s).
void middle_state(double Zpm, double Zpp, double Zsm, double Zsp, M9& Mm, M9& Mp) {
  Mm.fill(0);
  Mp.fill(0);
  const double c = Zpm * Zpp / (Zpm + Zpp);
  Mm[0 * 9 + 0] = 1 - c / Zpp; Mm[0 * 9 + 6] = -c;
  Mp[0 * 9 + 0] = c / Zpp;     Mp[0 * 9 + 6] = c;
  Mm[6 * 9 + 0] = -c / (Zpp * Zpm); Mm[6 * 9 + 6] = 1 - c / Zpm;
  Mp[6 * 9 + 0] = c / (Zpp * Zpm);  Mp[6 * 9 + 6] = c / Zpm;
  for (int r : {1, 2, 4}) Mm[r * 9 + r] = 1;  // irrelevant components (zero columns of A)
  const int pairs[2][2] = {{3, 7}, {5, 8}};
  for (auto& pr : pairs) {
    const int ts = pr[0], tv = pr[1];
    if (Zsm > 0 && Zsp > 0) {
      const double cs = Zsm * Zsp / (Zsm + Zsp);
      Mm[ts * 9 + ts] = 1 - cs / Zsp; Mm[ts * 9 + tv] = -cs;
      Mp[ts * 9 + ts] = cs / Zsp;     Mp[ts * 9 + tv] = cs;
      Mm[tv * 9 + ts] = -cs / (Zsp * Zsm); Mm[tv * 9 + tv] = 1 - cs / Zsm;
      Mp[tv * 9 + ts] = cs / (Zsp * Zsm);  Mp[tv * 9 + tv] = cs / Zsm;
    } else {
      Mm[tv * 9 + tv] = 1;
      if (Zsm > 0) Mm[tv * 9 + ts] = -1.0 / Zsm;
    }
  }
}

M9 diag9(std::initializer_list<double> d) {
  M9 r{};
  int i = 0;
  for (double v : d) { r[i * 9 + i] = v; ++i; }
  return r;
}

// Ghost state w^+ = G w^- of a linear boundary (Sec. 4.3), with the minus
// material: free surface, traction w1, w4, w6 mirrored; rigid wall, w7, w4, w6
// mirrored; absorbing, zero.
M9 ghost(int tag) {
  M9 G{};
  if (tag == ADG_TAG_FREE) G = diag9({-1, 1, 1, -1, 1, -1, 1, 1, 1});
  else if (tag == ADG_TAG_RIGID) G = diag9({1, 1, 1, -1, 1, -1, -1, 1, 1});
  return G;
}

// Coefficients of one face for the kernels (kernels.cuh, CREC) from the middle
// state of Sec. 4.2 (Eq. boundary-state), a linear boundary's ghost folded into
// the own side.  A gravitational face keeps the own tangential velocity and takes
// its normal state from the (eta, H) ODE; a fault face's flux is the friction
// solve's.
void face_coefficients(const double n[3], int tag, double Zp, double Zs, double Zpp, double Zsp, double rho, double lam,
                       double mu, double sf, double* c) {
  for (int d = 0; d < 3; ++d) c[d] = n[d];
  if (tag == ADG_TAG_FAULT) return;
  const bool nb = tag == ADG_TAG_INTERIOR || tag == ADG_TAG_PERIODIC;
  M9 Mm, Mp;
  middle_state(Zp, nb ? Zpp : Zp, Zs, nb ? Zsp : Zs, Mm, Mp);
  if (tag == ADG_TAG_GRAVITY) {
    for (int r : {0, 6}) Mm[r * 9 + 0] = Mm[r * 9 + 6] = 0;
    Mm[3 * 9 + 3] = Mm[3 * 9 + 7] = 0;
    Mm[7 * 9 + 3] = Zs > 0 ? -1 / Zs : 0.0;
    Mm[7 * 9 + 7] = 1;
  } else if (!nb) {
    const M9 G = ghost(tag);  // diagonal
    for (int r : {0, 3, 6, 7})
      for (int k : {0, 3, 6, 7}) Mm[r * 9 + k] += Mp[r * 9 + k] * G[k * 9 + k];
  }
  // normal pair (w1, w7) and tangential pair (w4, w8; w6, w9 alike): the rows of
  // traction and velocity, each from traction and velocity
  for (int k = 0; k < 4; ++k) {
    const int rn = k < 2 ? 0 : 6, cn = k % 2 ? 6 : 0, rt = k < 2 ? 3 : 7, ct = k % 2 ? 7 : 3;
    const double an = Mm[rn * 9 + cn], at = Mm[rt * 9 + ct];
    const double s = nb ? (k % 2 ? 1.0 : -1.0) : 0.0;  // the neighbour's traction has the opposite normal
    const double bn = s * Mp[rn * 9 + cn], bt = s * Mp[rt * 9 + ct];
    c[3 + k] = at;
    c[7 + k] = bt;
    // (traction: what the normal part adds to the tangential coefficients' product;
    // velocity: the normal state itself, see face_flux_state)
    c[11 + k] = k < 2 ? an - at : an;
    c[15 + k] = k < 2 ? bn - bt : bn;
  }
  const M9 A = jac_x(rho, lam, mu);
  c[19] = sf * (A[0 * 9 + 6] - 2 * A[3 * 9 + 7]);  // (A holds -(lam + 2 mu), -mu, -1 / rho)
  c[20] = sf * A[3 * 9 + 7];
  c[21] = sf * A[6 * 9 + 0];
}

// ---------------- Gauss-Legendre on [0,1] (Newton on P_n) ----------------
void gauss01(int n, std::vector<double>& x, std::vector<double>& w) {
  x.resize(n);
  w.resize(n);
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5)), pp = 0;
    for (int it = 0; it < 100; ++it) {
      double p1 = 1, p2 = 0;
      for (int j = 1; j <= n; ++j) { double p3 = p2; p2 = p1; p1 = ((2 * j - 1) * z * p2 - (j - 1) * p3) / j; }
      pp = n * (z * p1 - p2) / (z * z - 1);
      double dz = p1 / pp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    x[i] = 0.5 * (1 - z);
    w[i] = 1.0 / ((1 - z * z) * pp * pp);  // = 0.5 * 2/((1-z^2) P'^2)
  }
}

}  // namespace

// ======================================================================
namespace adg {

[[noreturn]] void throw_err(int code, const std::string& m) { throw Err(code, m); }

template <typename T>
static void* upload_vec(const std::vector<double>& h, std::vector<void*>& owned, int64_t& bytes) {
  std::vector<T> t(h.begin(), h.end());
  void* d = nullptr;
  if (t.empty()) return nullptr;
  CK(cudaMalloc(&d, t.size() * sizeof(T)));
  owned.push_back(d);
  bytes += t.size() * sizeof(T);
  CK(cudaMemcpy(d, t.data(), t.size() * sizeof(T), cudaMemcpyHostToDevice));
  return d;
}
template <typename T>
static T* upload_raw(const std::vector<T>& h, std::vector<void*>& owned, int64_t& bytes) {
  if (h.empty()) return nullptr;
  void* d = nullptr;
  CK(cudaMalloc(&d, h.size() * sizeof(T)));
  owned.push_back(d);
  bytes += h.size() * sizeof(T);
  CK(cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
  return (T*)d;
}
static void* dalloc(size_t n, std::vector<void*>& owned, int64_t& bytes) {
  if (n == 0) return nullptr;
  void* d = nullptr;
  CK(cudaMalloc(&d, n));
  owned.push_back(d);
  bytes += n;
  CK(cudaMemset(d, 0, n));
  return d;
}

// Host-side plan of the mesh in the caller's element order: geometry, face
// connectivity with node permutations, CFL time steps and rate-2 clusters
// (Sec. 4.4).  Needs no device; adg_init and adg_plan both use it.
void Ctx::plan_mesh(const RefOps& o, int degree, MeshPlan& plan) const {
  const int64_t E = nt;
  // ---- geometry (user order)
  plan.Jinv.assign(9 * E, 0.0); plan.detJ.assign(E, 0.0); plan.area.assign(4 * E, 0.0); plan.nrm.assign(12 * E, 0.0);
  plan.fcen.assign(12 * E, 0.0); plan.h.assign(E, 0.0);
  std::vector<double>&Jinv = plan.Jinv, &detJ = plan.detJ, &area = plan.area, &nrm = plan.nrm, &fcen = plan.fcen, &h = plan.h;
  for (int64_t e = 0; e < E; ++e) {
    const double* P[4];
    for (int k = 0; k < 4; ++k) {
      int64_t vid = tets[4 * e + k];
      if (vid < 0 || vid >= nv) throw Err(ADG_E_MESH, "vertex index out of range");
      P[k] = &xyz[3 * vid];
    }
    double J[3][3];
    for (int d = 0; d < 3; ++d)
      for (int c = 0; c < 3; ++c) J[d][c] = P[c + 1][d] - P[0][d];
    double det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                 J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                 J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
    if (!(det > 0)) throw Err(ADG_E_MESH, "inverted or degenerate tetrahedron " + std::to_string(e));
    detJ[e] = det;
    // inverse: Jinv[a][d] = d xi_a / d x_d
    double Ji[3][3];
    Ji[0][0] = (J[1][1] * J[2][2] - J[1][2] * J[2][1]) / det;
    Ji[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) / det;
    Ji[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) / det;
    Ji[1][0] = (J[1][2] * J[2][0] - J[1][0] * J[2][2]) / det;
    Ji[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) / det;
    Ji[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) / det;
    Ji[2][0] = (J[1][0] * J[2][1] - J[1][1] * J[2][0]) / det;
    Ji[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) / det;
    Ji[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) / det;
    for (int a = 0; a < 3; ++a)
      for (int d = 0; d < 3; ++d) Jinv[9 * e + 3 * a + d] = Ji[a][d];
    double asum = 0;
    for (int f = 0; f < 4; ++f) {
      const double* A = P[kFaceV[f][0]];
      const double* Bv = P[kFaceV[f][1]];
      const double* C = P[kFaceV[f][2]];
      double u[3], w[3], cr[3];
      for (int d = 0; d < 3; ++d) { u[d] = Bv[d] - A[d]; w[d] = C[d] - A[d]; }
      cr[0] = u[1] * w[2] - u[2] * w[1];
      cr[1] = u[2] * w[0] - u[0] * w[2];
      cr[2] = u[0] * w[1] - u[1] * w[0];
      double ar = std::sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]);
      double out = 0;
      for (int d = 0; d < 3; ++d) out += cr[d] * (A[d] - P[f][d]);
      double sg = out > 0 ? 1.0 : -1.0;
      for (int d = 0; d < 3; ++d) {
        nrm[12 * e + 3 * f + d] = sg * cr[d] / ar;
        fcen[12 * e + 3 * f + d] = (A[d] + Bv[d] + C[d]) / 3.0;
      }
      area[4 * e + f] = 0.5 * ar;
      asum += 0.5 * ar;
    }
    h[e] = 6.0 * (det / 6.0) / asum;  // insphere diameter 2 r_in = 6 V / sum(A)
  }

  // ---- face connectivity: interior/fault by vertex triples, periodic by partner
  plan.nbr.assign(4 * E, -1); plan.nface.assign(4 * E, -1); plan.nperm.assign(4 * E, -1);
  std::vector<int64_t>& nbr_u = plan.nbr;
  std::vector<int>&nface_u = plan.nface, &nperm_u = plan.nperm;
  {
    // match interior/fault faces by their sorted vertex triples: sort all
    // triples, then equal neighbours in the sorted list are the two sides
    struct FK {
      int64_t v0, v1, v2, id;
    };
    std::vector<FK> keys;
    keys.reserve((size_t)(4 * E));
    for (int64_t e = 0; e < E; ++e)
      for (int f = 0; f < 4; ++f) {
        int tg = tag[4 * e + f];
        if (tg < 0 || tg > 6) throw Err(ADG_E_MESH, "unknown face tag");
        if (tg != ADG_TAG_INTERIOR && tg != ADG_TAG_FAULT) continue;
        int64_t v[3] = {tets[4 * e + kFaceV[f][0]], tets[4 * e + kFaceV[f][1]], tets[4 * e + kFaceV[f][2]]};
        std::sort(v, v + 3);
        keys.push_back({v[0], v[1], v[2], 4 * e + f});
      }
    auto less = [](const FK& a, const FK& b) {
      if (a.v0 != b.v0) return a.v0 < b.v0;
      if (a.v1 != b.v1) return a.v1 < b.v1;
      if (a.v2 != b.v2) return a.v2 < b.v2;
      return a.id < b.id;
    };
    std::sort(keys.begin(), keys.end(), less);
    auto same = [](const FK& a, const FK& b) { return a.v0 == b.v0 && a.v1 == b.v1 && a.v2 == b.v2; };
    for (size_t k = 0; k < keys.size();) {
      if (k + 1 >= keys.size() || !same(keys[k], keys[k + 1]))
        throw Err(ADG_E_MESH, "interior face without a matching neighbour (tet " + std::to_string(keys[k].id / 4) + ")");
      if (k + 2 < keys.size() && same(keys[k], keys[k + 2])) throw Err(ADG_E_MESH, "face shared by more than two tets");
      const int64_t e = keys[k].id / 4, e2 = keys[k + 1].id / 4;
      const int f = (int)(keys[k].id % 4), f2 = (int)(keys[k + 1].id % 4);
      if (tag[4 * e2 + f2] != tag[4 * e + f]) throw Err(ADG_E_MESH, "fault face tagged on one side only");
      nbr_u[4 * e + f] = e2; nface_u[4 * e + f] = f2;
      nbr_u[4 * e2 + f2] = e; nface_u[4 * e2 + f2] = f;
      k += 2;
    }
    for (int64_t e = 0; e < E; ++e)
      for (int f = 0; f < 4; ++f) {
        if (tag[4 * e + f] != ADG_TAG_PERIODIC) continue;
        if (partner.empty()) throw Err(ADG_E_MESH, "periodic face without partner array");
        int64_t p = partner[4 * e + f];
        if (p < 0 || p >= 4 * E || tag[p] != ADG_TAG_PERIODIC) throw Err(ADG_E_MESH, "bad periodic partner");
        nbr_u[4 * e + f] = p / 4;
        nface_u[4 * e + f] = (int)(p % 4);
      }
    // orientation: node permutation so that my node n sits on the neighbour's node perm[n]
    for (int64_t e = 0; e < E; ++e)
      for (int f = 0; f < 4; ++f) {
        int64_t e2 = nbr_u[4 * e + f];
        if (e2 < 0) continue;
        int f2 = nface_u[4 * e + f];
        int sig[3];
        for (int s = 0; s < 3; ++s) {
          int64_t gv = tets[4 * e + kFaceV[f][s]];
          sig[s] = -1;
          if (tag[4 * e + f] == ADG_TAG_PERIODIC) {
            double sh[3];
            for (int d = 0; d < 3; ++d) sh[d] = fcen[12 * e2 + 3 * f2 + d] - fcen[12 * e + 3 * f + d];
            double best = 1e300;
            for (int s2 = 0; s2 < 3; ++s2) {
              const double* X = &xyz[3 * tets[4 * e2 + kFaceV[f2][s2]]];
              double dd = 0;
              for (int d = 0; d < 3; ++d) { double df = X[d] - (xyz[3 * gv + d] + sh[d]); dd += df * df; }
              if (dd < best) { best = dd; sig[s] = s2; }
            }
          } else {
            for (int s2 = 0; s2 < 3; ++s2)
              if (tets[4 * e2 + kFaceV[f2][s2]] == gv) sig[s] = s2;
          }
        }
        int pid = -1;
        for (int p = 0; p < 6; ++p)
          if (o.vperm[3 * p] == sig[0] && o.vperm[3 * p + 1] == sig[1] && o.vperm[3 * p + 2] == sig[2]) pid = p;
        if (pid < 0) throw Err(ADG_E_MESH, "could not orient a face pair");
        nperm_u[4 * e + f] = pid;
      }
  }

  // ---- CFL time steps and rate-2 clusters (Sec. 4.4)
  plan.dte.assign(E, 0.0);
  std::vector<double>& dte = plan.dte;
  double& dt_min = plan.dtmin;
  dt_min = 1e300;
  for (int64_t e = 0; e < E; ++e) {
    double cp = std::sqrt((lam[e] + 2 * mu[e]) / rho[e]);
    if (!(cp > 0) || !(rho[e] > 0) || mu[e] < 0) throw Err(ADG_E_INVALID, "bad material");
    dte[e] = cfg.cfl / (2 * degree + 1) * h[e] / cp;
    dt_min = std::min(dt_min, dte[e]);
  }
  plan.cl.assign(E, 0);
  std::vector<int>& cl = plan.cl;
  const int cmaxcap = std::max(1, std::min(cfg.max_clusters, 16)) - 1;
  for (int64_t e = 0; e < E; ++e) {
    int c = (int)std::floor(std::log2(dte[e] / dt_min) + 1e-12);
    cl[e] = std::max(0, std::min(c, cmaxcap));
  }
  for (bool changed = true; changed;) {
    changed = false;
    for (int64_t e = 0; e < E; ++e)
      for (int f = 0; f < 4; ++f) {
        int64_t e2 = nbr_u[4 * e + f];
        if (e2 < 0) continue;
        int lim = tag[4 * e + f] == ADG_TAG_FAULT ? cl[e2] : cl[e2] + 1;
        if (cl[e] > lim) { cl[e] = lim; changed = true; }
      }
  }
  plan.ncl = 0;
  for (int64_t e = 0; e < E; ++e) plan.ncl = std::max(plan.ncl, cl[e] + 1);
}

// The flux through face f of user tet eu as matrices (global frame, row-major):
// the kernels' face_flux_state with the coefficients that setup() gives them, on
// unit states.  Interior and periodic faces Fm, Fp; free, rigid and absorbing
// faces Fm (Fp zero); gravitational and fault faces zero (their fluxes come
// from the (eta, H) ODE and the friction solve).
void Ctx::face_flux(const MeshPlan& pl, int64_t eu, int f, double* Fm, double* Fp) const {
  const int tg = tag[4 * eu + f];
  for (double* F : {Fm, Fp})
    if (F) std::fill(F, F + 81, 0.0);
  if (tg == ADG_TAG_GRAVITY || tg == ADG_TAG_FAULT) return;
  const double* n = &pl.nrm[12 * eu + 3 * f];
  const int64_t e2 = pl.nbr[4 * eu + f] < 0 ? eu : pl.nbr[4 * eu + f];
  double c[CREC] = {0};
  face_coefficients(n, tg, std::sqrt(rho[eu] * (lam[eu] + 2 * mu[eu])), std::sqrt(rho[eu] * mu[eu]),
                    std::sqrt(rho[e2] * (lam[e2] + 2 * mu[e2])), std::sqrt(rho[e2] * mu[e2]), rho[eu], lam[eu], mu[eu],
                    1.0, c);
  const int vo[3][3] = {{0, 3, 5}, {3, 1, 4}, {5, 4, 2}};  // the stress tensor's entries
  const double zero[6] = {0};
  for (int side = 0; side < 2; ++side) {
    double* const F = side ? Fp : Fm;
    if (!F) continue;
    for (int k = 0; k < 9; ++k) {
      double q[6] = {0}, g[9];  // a trace: traction with the owner's outward normal, velocity
      for (int d = 0; d < 3; ++d)
        for (int x = 0; x < 3; ++x)
          if (vo[d][x] == k) q[d] += side ? -n[x] : n[x];
      if (k >= 6) q[k - 3] = 1;
      face_flux_state(c, side ? zero : q, side ? q : zero, 0.0, 0.0, g);
      for (int r = 0; r < 9; ++r) F[r * 9 + k] = g[r];
    }
  }
}

// Face f of user tet eu seen from its neighbour (interior, periodic and fault
// faces): the neighbour tet and local face, and node_map[n] = the neighbour's
// face node at the place of my face node n (the friction solve's; the neighbour
// kernels re-orient modes by the same vertex permutation); nb = -1 for faces
// without one.
void Ctx::face_neighbour(const MeshPlan& pl, const RefOps& o, int64_t eu, int f, int64_t* nb, int* nf,
                         int32_t* node_map) const {
  const int64_t e2 = pl.nbr[4 * eu + f];
  if (nb) *nb = e2;
  if (nf) *nf = e2 < 0 ? -1 : pl.nface[4 * eu + f];
  if (e2 < 0 || !node_map) return;
  const int pid = pl.nperm[4 * eu + f];
  for (int n = 0; n < o.Bf; ++n) node_map[n] = o.perm[(size_t)pid * o.Bf + n];
}

void Ctx::setup() {
  if (!has_mesh || !has_mat) throw Err(ADG_E_STATE, "upload mesh and material before adg_init");
  CK(cudaSetDevice(cfg.device));
  const int64_t E = nt;
  N = cfg.degree;
  S = cfg.ensemble;
  fp64 = cfg.precision == ADG_FP64;
  tc = cfg.precision == ADG_3XTF32 && (cfg.degree == 5 || cfg.degree == 4);
  ops = make_ref_ops(N);
  if (ops.max_orth_err > 1e-12) throw Err(ADG_E_INVALID, "reference basis not orthonormal");
  B = ops.B; Bf = ops.Bf; B1 = ops.B1;

  MeshPlan pl;
  plan_mesh(ops, N, pl);
  const std::vector<double>&Jinv = pl.Jinv, &detJ = pl.detJ, &area = pl.area, &nrm = pl.nrm;
  const std::vector<int64_t>& nbr_u = pl.nbr;
  const std::vector<int>&nface_u = pl.nface, &nperm_u = pl.nperm, &cl = pl.cl;
  dtmin = pl.dtmin;
  ncl = pl.ncl;
  // ---- internal order: by cluster, then by kernel kind, stable: plain elements
  // first (acoustic ones apart), those that a kernel handles at some extra cost
  // at the end, so that they fill few tiles and warps
  // (special: 1 a coarser neighbour, 3 one gravitational face or a finer
  // neighbour (both on the tensor-core kernels, 3 on their special local
  // instantiation), 2 the row kernels: a fault face or more than one
  // gravitational face; without the tensor-core kernels any of these)
  std::vector<char> special(E, 0);
  for (int64_t e = 0; e < E; ++e) {
    int ng_e = 0;
    bool cc = false, coarser = false, finer = false;
    for (int f = 0; f < 4; ++f) {
      const int tg = tag[4 * e + f];
      const int64_t e2 = nbr_u[4 * e + f];
      ng_e += tg == ADG_TAG_GRAVITY;
      cc = cc || tg == ADG_TAG_FAULT;
      coarser = coarser || (e2 >= 0 && cl[e2] > cl[e]);
      finer = finer || (e2 >= 0 && cl[e2] < cl[e]);
    }
    if (tc)
      special[e] = (cc || ng_e > 1) ? 2 : ((ng_e == 1 || finer) ? 3 : (coarser ? 1 : 0));
    else  // the row kernels: their special instantiation takes all of these
      special[e] = cc || ng_e || coarser || finer ? 2 : 0;
  }
  // order key within a cluster: 0 plain elastic, 1 plain fluid on an
  // acoustic local kernel, 2 with a coarser neighbour, 3 with a gravitational
  // face or a finer neighbour (with the tensor-core kernels all four on them),
  // 4 the rest
  // (contexts without the tensor-core kernels that adg_step_noalloc takes keep the
  // caller's order, which its dofs are in; those with them get tables in that order)
  bool sort_fluid = acoustic;
  if (!tc && ncl == 1 && S == 1) {
    sort_fluid = false;
    for (int64_t i = 0; i < 4 * E; ++i)
      sort_fluid = sort_fluid || (acoustic && (tag[i] == ADG_TAG_GRAVITY || tag[i] == ADG_TAG_FAULT));
  }
  std::vector<char> key(E, 0);
  for (int64_t e = 0; e < E; ++e)
    key[e] = special[e] == 1 ? 2 : special[e] == 3 ? 3 : special[e] == 2 ? 4
                                 : (char)(sort_fluid && mu[e] == 0.0 ? 1 : 0);
  order.resize(E);
  for (int64_t e = 0; e < E; ++e) order[e] = e;
  std::stable_sort(order.begin(), order.end(), [&](int64_t a, int64_t b) {
    return cl[a] != cl[b] ? cl[a] < cl[b] : key[a] < key[b];
  });
  inv.assign(E, 0);
  for (int64_t i = 0; i < E; ++i) inv[order[i]] = i;
  cl_begin.assign(ncl + 1, 0);
  cl_plain.assign(ncl, 0);
  cl_row.assign(ncl, 0);
  cl_row_fluid.assign(ncl, 0);
  cl_elastic.assign(ncl, 0);
  cl_fluid.assign(ncl, 0);
  cl_grav.assign(ncl, 0);
  cl_tc_lts.assign(ncl, 0);
  for (int64_t i = 0; i < E; ++i) {
    const int k = key[order[i]], c = cl[order[i]];
    cl_begin[c + 1]++;
    if (tc && k < 4) cl_plain[c]++;
    if (!tc && k <= 1) cl_row[c]++;
    if (!tc && k == 1) cl_row_fluid[c]++;
    if (tc && k == 0) cl_elastic[c]++;
    if (tc && k == 1) cl_fluid[c]++;
    if (tc && k == 3) cl_grav[c]++;
    if (tc && (k == 2 || k == 3)) cl_tc_lts[c] = 1;
  }
  for (int c = 0; c < ncl; ++c) cl_begin[c + 1] += cl_begin[c];
  cluster.resize(E);
  for (int64_t i = 0; i < E; ++i) cluster[i] = cl[order[i]];

  // ---- per-element / per-face device data (internal order)
  std::vector<double> par((size_t)E * PAR), crec((size_t)E * 4 * CREC, 0.0);
  std::vector<int> nbr((size_t)E * 4, -1), ninfo((size_t)E * 4, 0), gslot((size_t)E * 4, -1),
      bslot(E, -1), dslot((size_t)E * 4, -1);
  std::vector<double> gpar;
  gfaces.clear();
  int nb_slots = 0, nd_slots = 0, ng = 0;
  // gravity faces in increasing user (tet*4+face) order
  for (int64_t eu = 0; eu < E; ++eu)
    for (int f = 0; f < 4; ++f)
      if (tag[4 * eu + f] == ADG_TAG_GRAVITY) gfaces.push_back(4 * eu + f);
  for (size_t g = 0; g < gfaces.size(); ++g) {
    int64_t eu = gfaces[g] / 4;
    gslot[inv[eu] * 4 + gfaces[g] % 4] = (int)g;
  }
  ng = (int)gfaces.size();
  gpar.assign((size_t)ng * GPAR, 0.0);
  // per element in parallel; LTS/fault slots are flagged here and numbered in
  // element order afterwards
#pragma omp parallel for schedule(dynamic, 256)
  for (int64_t i = 0; i < E; ++i) {
    const int64_t eu = order[i];
    for (int k = 0; k < 9; ++k) par[i * PAR + k] = Jinv[9 * eu + k];
    par[i * PAR + 9] = rho[eu];
    par[i * PAR + 10] = lam[eu];
    par[i * PAR + 11] = mu[eu];
    for (int f = 0; f < 4; ++f) par[i * PAR + 12 + f] = 2.0 * area[4 * eu + f] / detJ[eu];
    const double Zpm = std::sqrt(rho[eu] * (lam[eu] + 2 * mu[eu])), Zsm = std::sqrt(rho[eu] * mu[eu]);
    bool has_coarse = false;
    for (int f = 0; f < 4; ++f) {
      const double* n = &nrm[12 * eu + 3 * f];
      const int tg = tag[4 * eu + f];
      const int64_t e2u = nbr_u[4 * eu + f];
      double Zpp = Zpm, Zsp = Zsm;
      if (tg == ADG_TAG_INTERIOR || tg == ADG_TAG_PERIODIC || tg == ADG_TAG_FAULT) {
        Zpp = std::sqrt(rho[e2u] * (lam[e2u] + 2 * mu[e2u]));
        Zsp = std::sqrt(rho[e2u] * mu[e2u]);
        const int64_t e2 = inv[e2u];
        const int c1 = cluster[i], c2 = cluster[e2];
        // (a fault face's flux is supplied by the rupture solver from both sides' derivative traces)
        const int kind = tg == ADG_TAG_FAULT ? NK_FAULT : c1 == c2 ? NK_SAME : (c2 > c1 ? NK_COARSE : NK_FINE);
        if (kind == NK_COARSE) has_coarse = true;
        if (kind == NK_FINE || kind == NK_FAULT) dslot[i * 4 + f] = 1;
        nbr[i * 4 + f] = (int)e2;
        ninfo[i * 4 + f] = nface_u[4 * eu + f] | (nperm_u[4 * eu + f] << 2) | (kind << 5);
      } else if (tg == ADG_TAG_GRAVITY) {
        double* gp = &gpar[(size_t)gslot[i * 4 + f] * GPAR];
        gp[0] = n[0]; gp[1] = n[1]; gp[2] = n[2];
        gp[3] = Zpm;
        gp[4] = rho[eu] * cfg.gravity / Zpm;
        gp[5] = rho[eu] * cfg.gravity;
      }
      face_coefficients(n, tg, Zpm, Zsm, Zpp, Zsp, rho[eu], lam[eu], mu[eu], par[i * PAR + 12 + f],
                        &crec[((size_t)i * 4 + f) * CREC]);
    }
    if (has_coarse) bslot[i] = 1;
  }
  for (int64_t i = 0; i < E; ++i) {
    if (bslot[i] == 1) bslot[i] = nb_slots++;
    for (int f = 0; f < 4; ++f)
      if (dslot[i * 4 + f] == 1) dslot[i * 4 + f] = nd_slots++;
  }
  n_bslots = nb_slots;
  n_dslots = nd_slots;
  n_gslots = ng;
  // the tensor-core kernels handle same-cluster and coarser neighbours and
  // linear boundaries: check that the ordering gave them nothing else
  if (tc)
    for (int c = 0; c < ncl; ++c)
      for (int64_t i = cl_begin[c]; i < cl_begin[c] + cl_plain[c]; ++i) {
        // (the last cl_grav[c] of them may have one gravitational face and faces
        // with a finer neighbour)
        const bool spec = i >= cl_begin[c] + cl_plain[c] - cl_grav[c];
        bool ok = true;
        int ngf = 0;
        for (int f = 0; f < 4; ++f) {
          const int kind = (ninfo[i * 4 + f] >> 5) & 7;
          ngf += gslot[i * 4 + f] >= 0;
          ok = ok && (kind == NK_SAME || kind == NK_NONE || kind == NK_COARSE || (spec && kind == NK_FINE)) &&
               (dslot[i * 4 + f] < 0 || (spec && kind == NK_FINE));
        }
        ok = ok && ngf <= (spec ? 1 : 0);
        if (!ok) throw Err(ADG_E_STATE, "internal: element order for the tensor-core kernels is inconsistent");
      }
  // ---- fault faces: one entry per tet pair, minus side = lower user tet index,
  // listed in internal (cluster) order; both sides share a cluster by construction
  fface.clear(); fgeo.clear(); fminus_user.clear(); fplus_user.clear();
  std::vector<int> fslot((size_t)E * 4, -1);
  fcl_begin.assign(ncl + 1, 0);
  for (int64_t i = 0; i < E; ++i) {
    const int64_t eu = order[i];
    for (int f = 0; f < 4; ++f) {
      if (tag[4 * eu + f] != ADG_TAG_FAULT) continue;
      const int64_t e2u = nbr_u[4 * eu + f];
      if (e2u < eu) continue;  // listed from the minus side
      const int f2 = nface_u[4 * eu + f];
      const int64_t e2 = inv[e2u];
      const int64_t fi = (int64_t)fface.size() / 5;
      fface.insert(fface.end(), {(int)i, f, (int)e2, f2, nperm_u[4 * eu + f]});
      fslot[i * 4 + f] = (int)(2 * fi);
      fslot[e2 * 4 + f2] = (int)(2 * fi + 1);
      fminus_user.push_back(4 * eu + f);
      fplus_user.push_back(4 * e2u + f2);
      const double* n = &nrm[12 * eu + 3 * f];
      fgeo.insert(fgeo.end(), {n[0], n[1], n[2], rho[eu], lam[eu], mu[eu], rho[e2u], lam[e2u], mu[e2u]});
      if (!(mu[eu] > 0 && mu[e2u] > 0)) throw Err(ADG_E_MESH, "fault faces must separate two solids");
      fcl_begin[cluster[i] + 1]++;
    }
  }
  nff = (int64_t)fface.size() / 5;
  for (int c = 0; c < ncl; ++c) fcl_begin[c + 1] += fcl_begin[c];
  n_fault_faces = nff;
  fault_set = false;

  // ---- reference operators in device layouts (l-major / n-major)
  const RowTables rt = make_row_tables(ops);
  if (rt.max_err > 1e-10) throw Err(ADG_E_STATE, "internal: the sparse operators do not match the basis");

  // ---- device allocations
  if (cfg.cuda_stream) {
    stream = (cudaStream_t)cfg.cuda_stream;
  } else {
    CK(cudaStreamCreateWithFlags(&own_stream, cudaStreamNonBlocking));
    stream = own_stream;
  }
  const size_t ts = fp64 ? 8 : 4;
  const int64_t V = E * S;
  dQ = dalloc((size_t)V * 9 * B * ts, owned, dev_bytes);
  dTrace = dalloc((size_t)V * 4 * face_stride(N) * ts, owned, dev_bytes);
  dOrder = upload_raw(order, owned, dev_bytes);
  dBtrace = (double*)dalloc((size_t)nb_slots * S * 36 * Bf * 8, owned, dev_bytes);
  dDtrace = dalloc((size_t)nd_slots * S * (N + 1) * 9 * Bf * ts, owned, dev_bytes);
  dEta = (double*)dalloc((size_t)ng * S * Bf * 8, owned, dev_bytes);
  dGflux = dalloc((size_t)ng * S * 9 * Bf * ts, owned, dev_bytes);
  if (fp64) {
    dPar = upload_vec<double>(par, owned, dev_bytes);
    dCrec = upload_vec<double>(crec, owned, dev_bytes);
    dNodal = upload_vec<double>(rt.nodalT, owned, dev_bytes);
    dModal = upload_vec<double>(rt.modalT, owned, dev_bytes);
    dReorient = upload_vec<double>(rt.reorient, owned, dev_bytes);
  } else {
    dPar = upload_vec<float>(par, owned, dev_bytes);
    dCrec = upload_vec<float>(crec, owned, dev_bytes);
    dNodal = upload_vec<float>(rt.nodalT, owned, dev_bytes);
    dModal = upload_vec<float>(rt.modalT, owned, dev_bytes);
    dReorient = upload_vec<float>(rt.reorient, owned, dev_bytes);
  }
  if (takes_noalloc() && noalloc_scratch() <= kNoallocScratch && !std::is_sorted(order.begin(), order.end())) {
    std::vector<double> par_u(par.size()), crec_u(crec.size());
    std::vector<int> nbr_u2(nbr.size()), ninfo_u(ninfo.size());
    for (int64_t i = 0; i < E; ++i) {
      const int64_t eu = order[i];
      std::copy_n(&par[i * PAR], PAR, &par_u[eu * PAR]);
      std::copy_n(&crec[i * 4 * CREC], 4 * CREC, &crec_u[eu * 4 * CREC]);
      for (int f = 0; f < 4; ++f) {
        nbr_u2[eu * 4 + f] = nbr[i * 4 + f] < 0 ? -1 : (int)order[nbr[i * 4 + f]];
        ninfo_u[eu * 4 + f] = ninfo[i * 4 + f];
      }
    }
    dParUser = fp64 ? upload_vec<double>(par_u, owned, dev_bytes) : upload_vec<float>(par_u, owned, dev_bytes);
    dCrecUser = fp64 ? upload_vec<double>(crec_u, owned, dev_bytes) : upload_vec<float>(crec_u, owned, dev_bytes);
    dNbrUser = upload_raw<int>(nbr_u2, owned, dev_bytes);
    dNinfoUser = upload_raw<int>(ninfo_u, owned, dev_bytes);
  }
  dNbr = upload_raw<int>(nbr, owned, dev_bytes);
  dNinfo = upload_raw<int>(ninfo, owned, dev_bytes);
  dGslot = ng ? upload_raw<int>(gslot, owned, dev_bytes) : nullptr;
  dBslot = nb_slots ? upload_raw<int>(bslot, owned, dev_bytes) : nullptr;
  dDslot = nd_slots ? upload_raw<int>(dslot, owned, dev_bytes) : nullptr;
  dGpar = ng ? upload_raw<double>(gpar, owned, dev_bytes) : nullptr;
  dPerm = upload_raw<int>(ops.perm, owned, dev_bytes);
  CK(cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, cfg.device));
  if (tc) {
    std::vector<float> tl(local_tc_floats(N));
    pack_local_tc(N, ops.kt.data(), ops.kvol.data(), rt.rfcT.data(), tl.data());
    dTcLocal = upload_raw<float>(tl, owned, dev_bytes);
    std::vector<float> tf(lift_tc_floats(N));
    pack_lift_tc(N, rt.rfcT.data(), tf.data());
    dTcLift = upload_raw<float>(tf, owned, dev_bytes);
  }
  dErr = (unsigned int*)dalloc(sizeof(unsigned int), owned, dev_bytes);
  dTiles = (int*)dalloc(2 * kTileKinds * sizeof(int), owned, dev_bytes);
  if (acoustic) {
    std::vector<int64_t> fl;
    for (int64_t i = 0; i < E; ++i)
      if (mu[order[i]] == 0.0) fl.push_back(i);
    n_fluid = (int64_t)fl.size();
    dFluid = n_fluid ? upload_raw<int64_t>(fl, owned, dev_bytes) : nullptr;
  }
  if (nff) {
    dFface = upload_raw<int>(fface, owned, dev_bytes);
    dFslot = upload_raw<int>(fslot, owned, dev_bytes);
    dFgeo = upload_raw<double>(fgeo, owned, dev_bytes);
    dFpar = (double*)dalloc((size_t)nff * S * Bf * FPAR * 8, owned, dev_bytes);
    dFstate = (double*)dalloc((size_t)nff * S * Bf * FSTATE * 8, owned, dev_bytes);
    dDrout = dalloc((size_t)nff * S * 2 * 9 * Bf * ts, owned, dev_bytes);
    dNewton = (unsigned long long*)dalloc(2 * sizeof(unsigned long long), owned, dev_bytes);
    dMlp = (float*)dalloc(MLP_NPARAM * sizeof(float), owned, dev_bytes);
    dCapCount = (unsigned long long*)dalloc(sizeof(unsigned long long), owned, dev_bytes);
  }
  int prio_low = 0, prio_high = 0;
  CK(cudaDeviceGetStreamPriorityRange(&prio_low, &prio_high));
  for (int i = 0; i < kSide; ++i) {
    CK(cudaStreamCreateWithPriority(&side[i], cudaStreamNonBlocking, prio_high));
    CK(cudaEventCreateWithFlags(&side_done[i], cudaEventDisableTiming));
  }
  CK(cudaEventCreateWithFlags(&side_fork, cudaEventDisableTiming));
  // configure every kernel that a step of this context may launch (outside any stream capture)
  StepArgs a0 = base_args();
  const Segs none = make_segs(nullptr, 0, 1);
  int rc = launch_local_row(fp64, N, a0, none, stream, 128, false);
  if (!rc) rc = launch_neighbour_row(fp64, N, a0, none, stream, 128, false);
  if (!rc && acoustic && !tc) rc = launch_local_fluid(fp64, N, a0, none, stream, 128);
  if (!rc && nff) rc = launch_rupture(fp64, N, DRArgs{}, stream);
  if (!rc && tc) rc = launch_local_tc(N, a0, none, n_sms, stream, false);
  if (!rc && tc) rc = launch_neighbour_tc(N, a0, none, n_sms, stream, false);
  if (rc) throw Err(ADG_E_CUDA, std::string("kernel configuration: ") + cudaGetErrorString((cudaError_t)rc));
  tick = 0;
  time = 0.0;
  inited = true;
}

bool Ctx::takes_noalloc() const { return ncl == 1 && S == 1 && gfaces.empty() && n_fault_faces == 0; }
size_t Ctx::noalloc_scratch() const { return (size_t)nt * 4 * face_stride(N) * (fp64 ? 8 : 4); }

StepArgs Ctx::base_args() const {
  StepArgs a{};
  a.Q = dQ; a.trace = dTrace; a.btrace = dBtrace; a.dtrace = dDtrace; a.eta = dEta;
  a.par = dPar; a.nbr = dNbr; a.ninfo = dNinfo;
  a.gslot = dGslot; a.bslot = dBslot; a.dslot = dDslot;
  a.gpar = dGpar;
  a.S = S; a.err = dErr; a.n_sms = n_sms;
  a.fslot = dFslot; a.drout = dDrout; a.gflux = dGflux; a.tc_local = dTcLocal; a.tc_lift = dTcLift;
  a.tiles = dTiles;
  a.crec = dCrec; a.nodalT = dNodal; a.modalT = dModal; a.reorient = dReorient;
  return a;
}

static void taylor_int(int N, double ta, double tb, double* out) {
  double fa = ta, fb = tb, fac = 1;
  for (int k = 0; k <= N; ++k) {
    fac *= (k + 1);
    out[k] = (fb - fa) / fac;
    fa *= ta;
    fb *= tb;
  }
}

// Launch the work of tick s of the rate-2 schedule with fine step dtm (Sec.
// 4.4): first the local phase of every cluster that starts a step at this
// tick, then the friction solves and the neighbour phase of every cluster
// that ends one.  Each phase is one launch per kernel kind covering all its
// clusters (a segment per cluster with that cluster's step and coefficients):
// the tensor-core kernels take what they can, the row kernels the rest (all
// elements without the tensor-core form).
void Ctx::launch_tick(int s, double dtm) {
  StepArgs a = base_args();
  for (int phase = 0; phase < 2; ++phase) {
    // per kernel kind the clusters' segments: tensor-core elastic, tensor-core
    // acoustic and gravitational-face (local phase only), the row kernels' plain,
    // acoustic (local phase) and special elements
    // (tcb: the local phase's elements with a coarser neighbour outside the
    // special range, on the instantiation with the LTS-buffer code)
    std::vector<Seg> tcs, tcb, fls, grs, rws, rfs, rss;
    bool ltsf = false;
    for (int c = 0; c < ncl; ++c) {
      const bool active = phase == 0 ? s % (1 << c) == 0 : (s + 1) % (1 << c) == 0;
      const int64_t n = cl_begin[c + 1] - cl_begin[c];
      if (!active || !n) continue;
      const double dt = (double)(1 << c) * dtm;
      Seg sg{};
      sg.dt = dt;
      if (phase == 0) {
        taylor_int(N, 0.0, dt, sg.tcoef);
        sg.btrace_mode = (s % (1 << (c + 1)) == 0) ? 1 : 2;
      } else {
        // position of this step inside the coarser neighbour's (2x longer) step
        const int half = ((s + 1) / (1 << c) - 1) % 2;
        taylor_int(N, half * dt, (half + 1) * dt, sg.ccoef);
        if (fcl_begin.size() > (size_t)c + 1 && fcl_begin[c + 1] > fcl_begin[c]) launch_rupture_cluster(c, dt);
      }
      auto seg = [&](int64_t first, int64_t count) {
        Seg t = sg;
        t.v_begin = first * S;
        t.n = count * S;
        return t;
      };
      const int64_t np = tc ? cl_plain[c] : 0;
      if (np > 0) {
        ltsf = ltsf || cl_tc_lts[c] != 0;
        const int64_t n0 = cl_elastic[c], n1 = cl_fluid[c], ng_c = cl_grav[c], n2 = np - ng_c - n0 - n1;
        if (phase == 0) {
          // plain elastic, acoustic, coarser-neighbour and special ranges, each on
          // its own kernel
          if (n0 > 0) tcs.push_back(seg(cl_begin[c], n0));
          if (n1 > 0) fls.push_back(seg(cl_begin[c] + n0, n1));
          if (n2 > 0) tcb.push_back(seg(cl_begin[c] + n0 + n1, n2));
          if (ng_c > 0) grs.push_back(seg(cl_begin[c] + np - ng_c, ng_c));
        } else {
          tcs.push_back(seg(cl_begin[c], np));
        }
      }
      if (tc) {
        if (n > np) rss.push_back(seg(cl_begin[c] + np, n - np));
      } else {
        const int64_t plain = row_plain(c), nf = phase == 0 ? std::min(plain, cl_row_fluid[c]) : 0, nr = plain - nf;
        if (nr > 0) rws.push_back(seg(cl_begin[c], nr));
        if (nf > 0) rfs.push_back(seg(cl_begin[c] + nr, nf));
        if (n > plain) rss.push_back(seg(cl_begin[c] + plain, n - plain));
      }
    }
    if (tcs.empty() && tcb.empty() && fls.empty() && grs.empty() && rws.empty() && rfs.empty() && rss.empty()) continue;
    ProfEv ev{phase, nullptr, nullptr, 0};
    if (prof) {
      CK(cudaEventCreate(&ev.a));
      CK(cudaEventCreate(&ev.b));
      CK(cudaEventRecord(ev.a, stream));
    }
    // The launches of a phase, the tensor-core kinds first.  They work on
    // different elements and run side by side, the special kernel (the longest
    // tiles) first: a tensor-core kernel keeps a CTA on every SM that it gets, but
    // its tiles go to whoever is free (tc::TileFeed), so the kernels' last tiles
    // overlap.  adg_profile measures the kinds one after the other.
    struct Launch {
      const std::vector<Seg>* v;
      int unit;  // virtual elements of a work unit
      bool tc;
      std::function<int(const Segs&, void*)> fn;
    };
    const Launch all[] = {
        {&grs, kTileElems, true,
         [&](const Segs& g, void* st) { return launch_local_tc(N, a, g, n_sms, st, true, false, true); }},
        {&fls, kTileElemsFluid, true,
         [&](const Segs& g, void* st) { return launch_local_tc(N, a, g, n_sms, st, false, true); }},
        {&tcb, kTileElems, true,
         [&](const Segs& g, void* st) { return launch_local_tc(N, a, g, n_sms, st, true); }},
        {&tcs, kTileElems, true,
         [&](const Segs& g, void* st) {
           return phase == 0 ? launch_local_tc(N, a, g, n_sms, st, false) : launch_neighbour_tc(N, a, g, n_sms, st, ltsf);
         }},
        {&rss, kRowElems, false,
         [&](const Segs& g, void* st) {
           return phase == 0 ? launch_local_row(fp64, N, a, g, st, cc_threads[0], true)
                             : launch_neighbour_row(fp64, N, a, g, st, cc_threads[1], true);
         }},
        {&rfs, kRowElemsFluid, false,
         [&](const Segs& g, void* st) { return launch_local_fluid(fp64, N, a, g, st, cc_threads[0]); }},
        {&rws, kRowElems, false,
         [&](const Segs& g, void* st) {
           return phase == 0 ? launch_local_row(fp64, N, a, g, st, cc_threads[0], false)
                             : launch_neighbour_row(fp64, N, a, g, st, cc_threads[1], false);
         }}};
    constexpr int kKinds = (int)(sizeof(all) / sizeof(all[0]));
    int kinds = 0, last = -1;
    bool any_tc = false;
    for (int k = 0; k < kKinds; ++k) {
      if (all[k].v->empty()) continue;
      ++kinds;
      last = k;
      any_tc = any_tc || all[k].tc;
    }
    const bool fork = kinds > 1 && !prof;
    int rc = 0, side_used = 0;
    bool tc_open = prof != nullptr;
    if (fork) CK(cudaEventRecord(side_fork, stream));
    for (int k = 0; k < kKinds && !rc; ++k) {
      if (tc_open && !all[k].tc && any_tc) {  // (adg_profile: the tensor-core launches alone)
        CK(cudaEventCreate(&ev.m));
        CK(cudaEventRecord(ev.m, stream));
        tc_open = false;
      }
      if (all[k].v->empty()) continue;
      cudaStream_t st = stream;
      if (fork && k != last) {
        st = side[side_used];
        CK(cudaStreamWaitEvent(st, side_fork, 0));
      }
      // one launch per kind and at most kMaxSeg segments
      const std::vector<Seg>& v = *all[k].v;
      for (size_t i = 0; i < v.size() && !rc; i += kMaxSeg) {
        const int n = (int)std::min<size_t>(kMaxSeg, v.size() - i);
        rc = all[k].fn(make_segs(v.data() + i, n, all[k].unit, all[k].tc ? tc_chunk[phase] : 1), st);
        ev.launches++;
      }
      if (st != stream) CK(cudaEventRecord(side_done[side_used++], st));
    }
    for (int i = 0; i < side_used; ++i) CK(cudaStreamWaitEvent(stream, side_done[i], 0));
    if (prof) { CK(cudaEventRecord(ev.b, stream)); prof->push_back(ev); }
    if (rc)
      throw Err(ADG_E_CUDA, std::string(phase == 0 ? "local kernel: " : "neighbour kernel: ") +
                                cudaGetErrorString((cudaError_t)rc));
  }
}

// Friction solve on the fault faces of cluster c over its step dt (before the
// neighbour kernel of that cluster, which lifts the fault fluxes).
void Ctx::launch_rupture_cluster(int c, double dt) {
  if (!fault_set) throw Err(ADG_E_STATE, "fault faces present: call adg_set_fault before stepping");
  DRArgs d{};
  d.dtrace = dDtrace; d.dslot = dDslot; d.fface = dFface; d.fgeo = dFgeo; d.fpar = dFpar;
  d.fstate = dFstate; d.drout = dDrout; d.perm = dPerm;
  d.f_begin = fcl_begin[c];
  d.n_faces = fcl_begin[c + 1] - fcl_begin[c];
  d.S = S;
  d.dt = dt;
  std::vector<double> x, w;
  gauss01(N + 1, x, w);
  for (int j = 0; j <= N; ++j) {
    d.tp[j] = dt * x[j];
    d.tw[j] = dt * w[j];
    d.tk[j][0] = 1.0;
    for (int k = 1; k <= N; ++k) d.tk[j][k] = d.tk[j][k - 1] * d.tp[j] / k;
  }
  d.newton = dNewton; d.err = dErr;
  d.mlp = mlp_on ? dMlp : nullptr;
  d.capture = cap_on ? dCapture : nullptr;
  d.cap_count = dCapCount;
  d.cap_capacity = cap_capacity;
  d.law = fric_law;
  ProfEv ev{2, nullptr, nullptr, 1};
  if (prof) {
    CK(cudaEventCreate(&ev.a));
    CK(cudaEventCreate(&ev.b));
    CK(cudaEventRecord(ev.a, stream));
  }
  int rc = launch_rupture(fp64, N, d, stream);
  if (prof) { CK(cudaEventRecord(ev.b, stream)); prof->push_back(ev); }
  if (rc) throw Err(ADG_E_CUDA, std::string("rupture kernel: ") + cudaGetErrorString((cudaError_t)rc));
}

// Elements of cluster c that take the plain row kernels (contexts without the
// tensor-core kernels).  In a cluster that a launch cannot fill the GPU with,
// none if some are special: the special kernels then take all of them, one
// launch a phase instead of two or three (2,688 tets, degree 3 FP32, ten steps
// 493 -> 375 us; 1,050 tets, degree 5 FP64, 4.43 -> 3.67 ms).  At 11,232 tets
// that costs more than it saves (degree 2 FP64 2.36 -> 2.57 ms).
int64_t Ctx::row_plain(int c) const {
  const int64_t n = cl_begin[c + 1] - cl_begin[c];
  return n > cl_row[c] && n * S <= (int64_t)kSmallLaunchWarps * n_sms * kRowElems ? 0 : cl_row[c];
}

int64_t Ctx::launches_per_macro() const {
  int64_t L = 0;
  const int ticks = 1 << (ncl - 1);
  for (int s = 0; s < ticks; ++s)
    for (int phase = 0; phase < 2; ++phase) {
      bool tcl = false, tbl = false, fll = false, grl = false, ccl = false, rwl = false, rfl = false;
      for (int c = 0; c < ncl; ++c) {
        const int64_t n = cl_begin[c + 1] - cl_begin[c];
        if (!n || (phase == 0 ? s % (1 << c) : (s + 1) % (1 << c))) continue;
        if (phase == 1 && fcl_begin[c + 1] > fcl_begin[c]) L += 1;  // friction solve per cluster
        const int64_t np = tc ? cl_plain[c] : 0;
        if (phase == 0 && np > 0) {
          const int64_t n0 = cl_elastic[c], nf = cl_fluid[c], ngr = cl_grav[c];
          tcl = tcl || n0 > 0;
          fll = fll || nf > 0;
          tbl = tbl || np - ngr - n0 - nf > 0;
          grl = grl || ngr > 0;
        } else {
          tcl = tcl || np > 0;
        }
        const int64_t plain = tc ? 0 : row_plain(c), rf = tc || phase ? 0 : std::min(plain, cl_row_fluid[c]);
        ccl = ccl || n > (tc ? np : plain);
        rfl = rfl || rf > 0;
        rwl = rwl || plain > rf;
      }
      L += tcl + tbl + fll + grl + ccl + rwl + rfl;
    }
  return L;
}

// Place of every element in a saved state: the tensor-core contexts' own order,
// else by cluster and the caller's numbering alone (empty: nothing to move).
std::vector<int64_t> Ctx::state_places() const {
  std::vector<int64_t> p;
  if (tc) return p;
  bool moved = false;
  for (int c = 0; c < ncl; ++c) {
    std::vector<int64_t> user(order.begin() + cl_begin[c], order.begin() + cl_begin[c + 1]);
    std::sort(user.begin(), user.end());
    for (int64_t i = cl_begin[c]; i < cl_begin[c + 1]; ++i) {
      p.push_back(cl_begin[c] + (std::lower_bound(user.begin(), user.end(), order[i]) - user.begin()));
      moved = moved || p.back() != i;
    }
  }
  if (!moved) p.clear();
  return p;
}

void Ctx::project_fluid(bool sync) {
  if (!acoustic || !n_fluid) return;
  const int rc = launch_isotropic_fluid(fp64, dQ, dFluid, n_fluid, S * B, B, stream);
  if (rc) throw Err(ADG_E_CUDA, std::string("fluid projection: ") + cudaGetErrorString((cudaError_t)rc));
  if (sync) CK(cudaStreamSynchronize(stream));
}

void Ctx::aio_setup() {
  if (aio.in) return;  // (created last: everything else is in place)
  const size_t bytes = (size_t)nt * S * 9 * B * sizeof(float);
  for (int b = 0; b < 2; ++b) {
    if (!aio.dIn[b]) aio.dIn[b] = static_cast<float*>(dalloc(bytes, owned, dev_bytes));
    if (!aio.dOut[b]) aio.dOut[b] = static_cast<float*>(dalloc(bytes, owned, dev_bytes));
    for (cudaEvent_t* e : {&aio.in_copied[b], &aio.in_used[b], &aio.out_made[b], &aio.out_copied[b]})
      if (!*e) CK(cudaEventCreateWithFlags(e, cudaEventDisableTiming));
  }
  if (!aio.out) CK(cudaStreamCreateWithFlags(&aio.out, cudaStreamNonBlocking));
  CK(cudaStreamCreateWithFlags(&aio.in, cudaStreamNonBlocking));
}

void Ctx::aio_sync() {
  if (aio.in) CK(cudaStreamSynchronize(aio.in));
  if (aio.out) CK(cudaStreamSynchronize(aio.out));
}

void Ctx::aio_free() {
  for (cudaStream_t st : {aio.in, aio.out})
    if (st) {
      cudaStreamSynchronize(st);
      cudaStreamDestroy(st);
    }
  for (int b = 0; b < 2; ++b)
    for (cudaEvent_t e : {aio.in_copied[b], aio.in_used[b], aio.out_made[b], aio.out_copied[b]})
      if (e) cudaEventDestroy(e);
  aio = AsyncIo{};  // (the staging buffers are among the owned allocations)
}

void Ctx::run_macro(double scale) {
  const int ticks = 1 << (ncl - 1);
  const double dtm = dtmin * scale;
  if (scale == 1.0 && use_graph) {
    if (!graph_exec) {
      cudaGraph_t g;
      CK(cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal));
      try {
        for (int s = 0; s < ticks; ++s) launch_tick(s, dtm);
      } catch (...) {
        cudaStreamEndCapture(stream, &g);
        throw;
      }
      CK(cudaStreamEndCapture(stream, &g));
      CK(cudaGraphInstantiate(&graph_exec, g, 0));
      CK(cudaGraphDestroy(g));
    }
    CK(cudaGraphLaunch(graph_exec, stream));
  } else {
    for (int s = 0; s < ticks; ++s) launch_tick(s, dtm);
  }
  time += ticks * dtm;
}

// Cadence recording: after a macro step of adg_advance / adg_advance_to, take
// the samples that are due into their device ring slots on the library stream
// and queue each slot's copy to the pinned host ring on the recording stream.
void Ctx::record_after_macro() {
  for (int k = 0; k < 2; ++k) {
    Recorder& r = rec[k];
    if (!r.every || ++r.macro % r.every) continue;
    const int64_t slot = r.count % r.cap;
    if (r.count - r.read >= r.cap) {  // the oldest unread sample is overwritten
      r.read++;
      r.dropped++;
    }
    CK(cudaStreamWaitEvent(stream, r.copied[slot], 0));  // the slot's previous copy is done
    double* d = r.dRing + slot * r.sample;
    if (k == 0) {
      const int rc = launch_receivers(fp64, B, dQ, S, n_rec, dRecElem, dRecPhi, d, stream);
      if (rc) throw Err(ADG_E_CUDA, std::string("receiver kernel: ") + cudaGetErrorString((cudaError_t)rc));
    } else {
      CK(cudaMemcpyAsync(d, dEta, r.sample * 8, cudaMemcpyDeviceToDevice, stream));
    }
    CK(cudaEventRecord(r.taken[slot], stream));
    CK(cudaStreamWaitEvent(rec_stream, r.taken[slot], 0));
    CK(cudaMemcpyAsync(r.hRing + slot * r.sample, d, r.sample * 8, cudaMemcpyDeviceToHost, rec_stream));
    CK(cudaEventRecord(r.copied[slot], rec_stream));
    r.t[slot] = time;
    r.count++;
  }
}

void Ctx::record_free(int kind) {
  Recorder& r = rec[kind];
  if (rec_stream) cudaStreamSynchronize(rec_stream);
  if (r.dRing) cudaFree(r.dRing);
  if (r.hRing) cudaFreeHost(r.hRing);
  for (cudaEvent_t e : r.taken) cudaEventDestroy(e);
  for (cudaEvent_t e : r.copied) cudaEventDestroy(e);
  r = Recorder();
}

void Ctx::check_err() {
  CK(cudaStreamSynchronize(stream));
  unsigned int h = 0;
  CK(cudaMemcpy(&h, dErr, sizeof(h), cudaMemcpyDeviceToHost));
  if (h) {
    CK(cudaMemset(dErr, 0, sizeof(unsigned int)));
    if (h & ERR_NAN) throw Err(ADG_E_NAN, "non-finite dofs detected");
    if (h & ERR_NEWTON) throw Err(ADG_E_NEWTON, "friction Newton solve did not converge");
    if (h & ERR_TIMEOUT) throw Err(ADG_E_TIMEOUT, "bounded device wait ran out");
  }
}

Ctx::~Ctx() {
  record_free(0);
  record_free(1);
  aio_free();
  if (rec_stream) cudaStreamDestroy(rec_stream);
  if (graph_exec) cudaGraphExecDestroy(graph_exec);
  for (int i = 0; i < kSide; ++i) {
    if (side[i]) cudaStreamDestroy(side[i]);
    if (side_done[i]) cudaEventDestroy(side_done[i]);
  }
  if (side_fork) cudaEventDestroy(side_fork);
  for (void* p : owned) cudaFree(p);
  if (hstage) cudaFreeHost(hstage);
  if (own_stream) cudaStreamDestroy(own_stream);
}

// Volume quadrature for projections: collapsed Gauss-Legendre, exact for degree deg.
void tet_rule(int deg, std::vector<double>& pts, std::vector<double>& w) {
  int n = std::max(1, (deg + 4) / 2);
  std::vector<double> x, wx;
  gauss01(n, x, wx);
  pts.clear();
  w.clear();
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < n; ++j)
      for (int k = 0; k < n; ++k) {
        double u = x[i], v = x[j], s = x[k];
        pts.push_back(u * (1 - v) * (1 - s));
        pts.push_back(v * (1 - s));
        pts.push_back(s);
        w.push_back(wx[i] * wx[j] * wx[k] * (1 - v) * (1 - s) * (1 - s));
      }
}

}  // namespace adg
