"""The compiled-in nonzero entries of the reference operators (sparse_ops.inc)
against the oracle's basis: stiffness in the parity-respecting directions, face
projections onto orthonormal face modes, re-orientation of face modes."""

import os
import re

import numpy as np
import pytest

from oracle import basis as ob
from oracle.quadrature import tri_rule

INC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_06640_gb300", "csrc",
                   "sparse_ops.inc")
TOL = 1e-11  # quadrature of degree-10 integrands with entries up to 40 in float64


def _tables():
    text = open(INC).read()
    out = {}
    for name, body in re.findall(r"constexpr Entry k(\w+)\[\] = \{(.*?)\};", text, re.S):
        e = np.array([[float(x) for x in t.split(",")] for t in re.findall(r"\{(.*?)\}", body)])
        m = np.zeros((35 if name[0] == "K" else 21, 56))
        m[e[:, 0].astype(int), e[:, 1].astype(int)] = e[:, 2]
        out[name] = m
    body = re.search(r"kPV\[6\]\[91\] = \{(.*)\};", text, re.S).group(1)
    out["PV"] = np.array([[float(x) for x in t.split(",")] for t in re.findall(r"\{(.*?)\}", body, re.S)])
    return out


T = _tables()


def _face_modes(chi):
    """The oracle's tetrahedral modes phi_ij0 on face 3 (zeta = 0) are multiples of the face's Dubiner modes."""
    w_chi, w = tri_rule(12)
    order = {t: l for l, t in enumerate(ob.triples(5))}
    cols = [order[(i, n - i, 0)] for n in range(6) for i in range(n + 1)]
    on = lambda c: ob.eval_basis(5, ob.face_to_ref(3, c))[:, cols]  # noqa: E731
    norm = 1 / np.sqrt(np.einsum("q,qr->r", w, on(w_chi) ** 2))
    sign = np.sign(T["R3"][np.arange(21), cols])
    return on(chi) * norm * sign


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_stiffness(axis):
    kt = ob.stiffness(5)[axis].T[:35]  # kt[m][l] = int phi_m dphi_l
    got = T["KX"] if axis == 0 else 0.5 * T["KX"] + T["KY"] + (T["KZ"] if axis == 2 else 0)
    assert np.abs(got - kt).max() <= TOL


@pytest.mark.parametrize("face", [0, 1, 2, 3])
def test_face_projection(face):
    chi, w = tri_rule(12)
    ref = np.einsum("q,qr,ql->rl", w, _face_modes(chi), ob.eval_basis(5, ob.face_to_ref(face, chi)))
    odd = np.array([t[0] % 2 for t in ob.triples(5)])
    got = T["R%d" % face] if face != 1 else T["R0"] * (1 - 2 * odd)
    assert np.abs(got - ref).max() <= TOL


@pytest.mark.parametrize("p", range(6))
def test_reorientation(p):
    sig = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)][p]
    chi, w = tri_rule(12)
    corner = np.array([[0.0, 0], [1, 0], [0, 1]])[list(sig)]
    theirs = corner[0] + chi[:, :1] * (corner[1] - corner[0]) + chi[:, 1:] * (corner[2] - corner[0])
    ref = np.einsum("q,qr,qs->rs", w, _face_modes(chi), _face_modes(theirs))
    got, k = np.zeros((21, 21)), 0
    for n in range(6):
        b = slice(n * (n + 1) // 2, (n + 1) * (n + 2) // 2)
        got[b, b] = T["PV"][p, k:k + (n + 1) ** 2].reshape(n + 1, n + 1)
        k += (n + 1) ** 2
    assert np.abs(got - ref).max() <= TOL
