"""A saved state lists the dofs of a context without the tensor-core kernels by
cluster and the caller's element numbers, whatever order the library works in."""

import numpy as np
import pytest

from _cases import make_pair, small_coupled, to_gpu_layout

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,acoustic", [(0, False), (1, True)])
def test_state_lists_elements_in_the_callers_order(precision, acoustic):
    from synthetic.workloads import random_dofs
    m, mat = small_coupled()
    _, s = make_pair(m, mat, 3, precision=precision, acoustic_ocean=acoustic)
    assert s.info.n_gravity_faces > 0
    s.set_dofs(to_gpu_layout(random_dofs((m.nt, s.B, 9), 11, N=3)))
    dofs = np.asarray(s.get_dofs()).reshape(m.nt, -1)
    state = s.save_state()
    buf = bytes(state)
    ts = 8 if precision == 0 else 4
    at = len(buf) - dofs.size * ts - int(s.info.n_gravity_faces) * s.Bf * 8  # past the header
    body = np.frombuffer(buf, np.float64 if precision == 0 else np.float32, dofs.size, at).reshape(dofs.shape)
    assert np.array_equal(body, dofs)
    s.set_dofs(np.zeros_like(to_gpu_layout(random_dofs((m.nt, s.B, 9), 11, N=3))))
    s.load_state(state)
    assert np.array_equal(np.asarray(s.get_dofs()).reshape(m.nt, -1), dofs)
