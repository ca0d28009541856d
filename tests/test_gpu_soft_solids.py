"""Fluxes of soft solids in single precision: sediment with a shear speed far below
its compressional speed under water, over a rigid and beside absorbing walls."""

import numpy as np
import pytest

from _cases import make_pair, rel_l2, to_gpu_layout, to_oracle_layout

pytestmark = pytest.mark.gpu

VP, RHO = 1600.0, 2000.0


def _errors(precision, N, vs):
    """Relative errors of stress and velocity after two steps against the oracle."""
    from synthetic.workloads import coupled_box, random_dofs
    m, mat = coupled_box(nxy=3, n_water=1, n_crust=2, L=6e3, depth=3e3, water=1e3, rigid_bottom=True)
    rho, lam, mu = (x.copy() for x in mat)
    soft = mu > 0
    rho[soft], mu[soft] = RHO, RHO * vs ** 2
    lam[soft] = RHO * (VP ** 2 - 2 * vs ** 2)
    o, s = make_pair(m, (rho, lam, mu), N, precision=precision)
    Q0 = random_dofs((m.nt, s.B, 9), 23, N=N)
    p = Q0[..., 0:3].mean(axis=-1, keepdims=True)
    dev = np.where(soft, vs / VP, 0.0)[:, None, None]  # deviatoric stress as a wave of the medium has it
    Q0[..., 0:3] = p + dev * (Q0[..., 0:3] - p)
    Q0[..., 3:6] *= dev
    o.Q, o._D, o.t = Q0.copy(), None, 0.0
    o.eta[:] = 0
    s.set_dofs(to_gpu_layout(Q0))
    s.set_eta(np.zeros((int(s.info.n_gravity_faces), 1, s.Bf)))
    s.advance(2)
    for _ in range(2):
        o.advance_macro()
    got = to_oracle_layout(s.get_dofs())
    return np.array([rel_l2(got[..., :6], o.Q[..., :6]), rel_l2(got[..., 6:], o.Q[..., 6:])])


@pytest.mark.parametrize("precision,N", [(1, 2), (1, 3), (2, 4), (2, 5)])
def test_soft_solids_are_as_exact_as_stiff_ones(precision, N):
    """The error of one flux row in FP32, emulated against float64 for all neighbours and boundaries,
    is at v_s 50 and 0.5 m/s at most 2.5 times that at v_p / sqrt(3); twice that is allowed for the rest of a step."""
    stiff = _errors(precision, N, VP / 3 ** 0.5)
    for vs in (50.0, 0.5):
        assert np.all(_errors(precision, N, vs) <= 5 * stiff), (vs, stiff)
