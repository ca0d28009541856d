"""The tensor-core kernels against the oracle where tiles are cut: element counts
of every kind (plain, acoustic, coarser neighbour, special) that are no multiple
of a tile, more tiles than one segment, scenarios that share a tile."""

import numpy as np
import pytest

from _cases import make_pair, rel_l2, to_gpu_layout, to_oracle_layout

pytestmark = pytest.mark.gpu

TOL = 2e-5  # the repository's parity tolerance of ADG_3XTF32


@pytest.mark.parametrize("acoustic", [False, True])
@pytest.mark.parametrize("N,S,nxy,clusters", [(5, 1, 1, 1), (5, 3, 5, 3), (4, 1, 5, 3), (4, 5, 3, 1)])
def test_partial_tiles(N, S, nxy, clusters, acoustic):
    from synthetic.workloads import coupled_box, random_dofs
    grading = 6.0 if clusters > 1 else 1.0
    m, mat = coupled_box(nxy=nxy, n_water=2, n_crust=2, L=20e3, depth=6e3, water=1e3, grading=grading, rigid_bottom=True)
    o, s = make_pair(m, mat, N, precision=2, max_clusters=clusters, ensemble=S, acoustic_ocean=acoustic)
    assert s.info.n_clusters > 1 or clusters == 1
    Q0 = random_dofs((S, m.nt, s.B, 9), 13, N=N)
    fluid = mat[2] == 0
    Q0[:, fluid, :, 0:3] = Q0[:, fluid, :, 0:3].mean(axis=-1, keepdims=True)
    Q0[:, fluid, :, 3:6] = 0
    s.set_dofs(np.ascontiguousarray(np.stack([to_gpu_layout(q) for q in Q0], axis=1)))
    s.set_eta(np.zeros((int(s.info.n_gravity_faces), S, s.Bf)))
    s.advance(2)
    got = s.get_dofs().reshape(m.nt, S, 9, s.B)
    for k in range(S):
        o.Q, o._D, o.t = Q0[k].copy(), None, 0.0
        o.eta[:] = 0
        for _ in range(2):
            o.advance_macro()
        assert rel_l2(to_oracle_layout(got[:, k]), o.Q) <= TOL
