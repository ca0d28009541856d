"""Writes sparse_ops.inc: the reference operators of degree 5 as lists of their
nonzero entries, from 40-digit quadrature.  The basis is hierarchical, so the
operators of degree N < 5 are the leading blocks.  Run by hand when the basis
changes (python gen_sparse_ops.py > sparse_ops.inc); tests compare the tables
with the operators the library computes at run time.

  KX  int phi_m dphi_l/dxi
  KY  int phi_m (d/deta - 1/2 d/dxi) phi_l
  KZ  int phi_m (d/dzeta - 1/2 d/dxi - (d/deta - 1/2 d/dxi)) phi_l
      The reflection xi -> 1 - xi - eta - zeta maps phi_ijk to (-1)^i phi_ijk
      and commutes with the derivatives of KY and KZ, which therefore couple
      modes of equal parity in i only; KZ is moreover the direction in which
      the products in eta and zeta cancel most entries.
  R0, R2, R3  int_f psi_r phi_l over faces 0, 2, 3 with the orthonormal Dubiner
      modes psi_r of the reference triangle; by the same reflection face 1 is
      R1[r][l] = (-1)^i R0[r][l].
  PV  [6][Bf][Bf] blocks: modes of a face seen through the six vertex
      permutations (block diagonal in the degree n of the modes, blocks of
      n + 1 rows; block entries row by row).
"""
import itertools
from math import comb

import mpmath as mp

mp.mp.dps = 40
N = 5
FACE_VERTS = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))
# the library's order of the vertex permutations
PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))


def jacobi(n, a, x, t):
    """t^n P_n^(a,0)(2x/t - 1) and its derivatives by x and t (homogeneous form)."""
    v = dx = dt = mp.mpf(0)
    for s in range(n + 1):
        w = comb(n + a, n - s) * comb(n, s)
        p, q = (x - t) ** s, x ** (n - s)
        dp = s * (x - t) ** (s - 1) if s else mp.mpf(0)
        dq = (n - s) * x ** (n - s - 1) if n > s else mp.mpf(0)
        v += w * p * q
        dx += w * (dp * q + p * dq)
        dt -= w * dp * q
    return v, dx, dt


TRI3 = [(i, j, n - i - j) for n in range(N + 1) for i in range(n + 1) for j in range(n - i + 1)]
TRI2 = [(i, n - i) for n in range(N + 1) for i in range(n + 1)]


def phi(x, y, z, grad=False):
    s, t, one = 1 - y - z, 1 - z, mp.mpf(1)
    out = []
    for i, j, k in TRI3:
        a, ax, as_ = jacobi(i, 0, x, s)
        b, by, bt = jacobi(j, 2 * i + 1, y, t)
        d, dz, _ = jacobi(k, 2 * i + 2 * j + 2, z, one)
        if grad:
            out.append((a * b * d, (ax * b * d, (a * by - as_ * b) * d, -as_ * b * d - a * bt * d + a * b * dz)))
        else:
            out.append(a * b * d)
    return out


def psi(x, y):
    return [jacobi(i, 0, x, 1 - y)[0] * jacobi(j, 2 * i + 1, y, mp.mpf(1))[0] for i, j in TRI2]


def gauss(n):
    x, w = [], []
    for k in range(n):
        t = mp.cos(mp.pi * (k + mp.mpf(3) / 4) / (n + mp.mpf(1) / 2))
        for _ in range(60):
            slope = n * (t * mp.legendre(n, t) - mp.legendre(n - 1, t)) / (t * t - 1)
            t -= mp.legendre(n, t) / slope
        x.append((1 + t) / 2)
        w.append(1 / ((1 - t * t) * slope ** 2))
    return x, w


def operators():
    p, w = gauss(N + 3)
    B, Bf = len(TRI3), len(TRI2)
    pts = [(x * (1 - y) * (1 - z), y * (1 - z), z, wx * wy * wz * (1 - y) * (1 - z) ** 2)
           for x, wx in zip(p, w) for y, wy in zip(p, w) for z, wz in zip(p, w)]
    vals = [phi(x, y, z, True) for x, y, z, _ in pts]
    norm = [1 / mp.sqrt(mp.fsum(q[3] * v[l][0] ** 2 for q, v in zip(pts, vals))) for l in range(B)]
    kt = [[[norm[m] * norm[l] * mp.fsum(q[3] * v[m][0] * v[l][1][a] for q, v in zip(pts, vals)) for l in range(B)]
           for m in range(B)] for a in range(3)]
    half = mp.mpf(1) / 2
    ky = [[kt[1][m][l] - half * kt[0][m][l] for l in range(B)] for m in range(B)]
    kz = [[kt[2][m][l] - half * kt[0][m][l] - ky[m][l] for l in range(B)] for m in range(B)]
    tri = [(x * (1 - y), y, wx * wy * (1 - y)) for x, wx in zip(p, w) for y, wy in zip(p, w)]
    pv = [psi(x, y) for x, y, _ in tri]
    pn = [1 / mp.sqrt(mp.fsum(q[2] * v[r] ** 2 for q, v in zip(tri, pv))) for r in range(Bf)]
    ref = ((0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1))
    R = []
    for f in range(4):
        a, b, c = (ref[v] for v in FACE_VERTS[f])
        fv = [phi(*(a[d] + x * (b[d] - a[d]) + y * (c[d] - a[d]) for d in range(3))) for x, y, _ in tri]
        R.append([[pn[r] * norm[l] * mp.fsum(q[2] * v[r] * u[l] for q, v, u in zip(tri, pv, fv)) for l in range(B)]
                  for r in range(Bf)])
    # my vertex s is the neighbour's vertex sig[s]: mine psi_r = sum_s P[r][s] theirs psi_s as functions on the face
    corner = ((0, 0), (1, 0), (0, 1))
    P = []
    for sig in PERMS:
        a, b, c = (corner[s] for s in sig)
        their = [psi(a[0] + x * (b[0] - a[0]) + y * (c[0] - a[0]), a[1] + x * (b[1] - a[1]) + y * (c[1] - a[1]))
                 for x, y, _ in tri]
        P.append([[pn[r] * pn[s] * mp.fsum(q[2] * v[r] * u[s] for q, v, u in zip(tri, pv, their)) for s in range(Bf)]
                  for r in range(Bf)])
    return kt[0], ky, kz, R, P


def num(x):
    return mp.nstr(x, 19, strip_zeros=True)


def table(name, M, rows):
    e = [(r, l, M[r][l]) for r in range(rows) for l in range(len(M[r])) if abs(M[r][l]) > mp.mpf(10) ** -25]
    print("constexpr Entry k%s[] = {" % name)
    line = ""
    for r, l, v in e:
        item = "{%d, %d, %s}, " % (r, l, num(v))
        if len(line) + len(item) > 118:
            print(line.rstrip())
            line = ""
        line += item
    print(line.rstrip())
    print("};")


def main():
    kx, ky, kz, R, P = operators()
    par = [(-1) ** i for i, _, _ in TRI3]
    assert all(abs(R[1][r][l] - par[l] * R[0][r][l]) < mp.mpf(10) ** -25 for r in range(21) for l in range(56))
    print("// written by gen_sparse_ops.py")
    for name, M in (("KX", kx), ("KY", ky), ("KZ", kz)):
        table(name, M, 35)
    for name, M in (("R0", R[0]), ("R2", R[2]), ("R3", R[3])):
        table(name, M, 21)
    print("constexpr double kPV[6][%d] = {" % sum((n + 1) ** 2 for n in range(N + 1)))
    for M in P:
        vals = [M[r][s] for n in range(N + 1) for r in range(n * (n + 1) // 2, (n + 1) * (n + 2) // 2)
                for s in range(n * (n + 1) // 2, (n + 1) * (n + 2) // 2)]
        off = max(abs(M[r][s]) for r in range(21) for s in range(21)
                  if sum(TRI2[r]) != sum(TRI2[s]))
        assert off < mp.mpf(10) ** -25
        print("{" + ",\n".join(", ".join(num(v) if abs(v) > mp.mpf(10) ** -25 else "0" for v in vals[i:i + 5])
                               for i in range(0, len(vals), 5)) + "},")
    print("};")


if __name__ == "__main__":
    main()
