"""The host checks of adg_face_flux catch mistakes in the face coefficients that the
kernels read: one mistake planted in a copy of csrc/adg_host.cpp per case, built
and run as in test_host_mutations.py."""

import pytest

from test_host_mutations import _nvcc, _run, objects  # noqa: F401

CASES = [
    ("neighbour-traction-sign", "const double s = nb ? (k % 2 ? 1.0 : -1.0) : 0.0;", "const double s = nb ? 1.0 : 0.0;",
     "face_flux"),
    ("normal-velocity-as-difference", "c[11 + k] = k < 2 ? an - at : an;", "c[11 + k] = an - at;", "face_flux"),
    ("boundary-without-ghost", "Mm[r * 9 + k] += Mp[r * 9 + k] * G[k * 9 + k];", ";", "face_flux"),
    ("density-twice", "c[21] = sf * A[6 * 9 + 0];", "c[21] = sf * A[6 * 9 + 0] / rho;", "face_flux"),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_planted_mistake_in_the_coefficients_fails_the_host_checks(case, objects, tmp_path):  # noqa: F811
    if _nvcc() is None:
        pytest.skip("nvcc not available")
    rc, out = _run(case, objects, str(tmp_path))
    assert rc == 1, out
