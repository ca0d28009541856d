"""The forcing of the gravitational surface, v_n - sigma_nn / Z, where the two parts
cancel to a millionth: FP32 dofs whose traces are in an exact ratio of 2^20 and an
impedance a few millionths above it.  The difference keeps what FP64 would keep."""

import numpy as np
import pytest

from _cases import make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,N", [(1, 1), (1, 2), (1, 3), (1, 4), (1, 5), (2, 4), (2, 5)])
def test_forcing_of_the_surface_keeps_what_does_not_cancel(precision, N):
    from synthetic.workloads import coupled_box
    m, _ = coupled_box(nxy=2, n_water=1, n_crust=1, L=4096.0, depth=2048.0, water=1024.0, rigid_bottom=True)
    rho, c = 1024.0, 1024.0 * (1 + 3.9e-6)
    Z = rho * c
    one = np.ones(m.nt)
    _, s = make_pair(m, (rho * one, rho * c * c * one, 0 * one), N, precision=precision)
    Q = np.zeros((m.nt, 9, s.B))
    Q[:, 0:3, 0], Q[:, 8, 0] = 2.0 ** 10, 2.0 ** -10  # constant: mode 0 is sqrt(6)
    s.set_dofs(Q)
    s.set_eta(np.zeros((int(s.info.n_gravity_faces), 1, s.Bf)))
    s.advance(1)
    f = 2.0 ** -10 * 6 ** 0.5 * (1 - 2.0 ** 20 / Z)
    kappa = 9.81 / c
    want = -f / kappa * np.expm1(-kappa * s.time)
    # traces, node values and eta each within an FP32 rounding of a table entry or product; half an
    # FP32 unit of 1 / Z alone would be 1e-2 here
    assert np.abs(s.read_ssh() / want - 1).max() <= 2e-6
