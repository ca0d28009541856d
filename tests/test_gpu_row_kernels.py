"""The row kernels (CUDA cores, three elements per warp) against the oracle at
every degree: boxes with all face kinds and LTS neighbours whose plain and
special element ranges are not multiples of three, ensembles whose warps mix
scenarios and elements, and a caller's dofs that are not 16-byte aligned."""

import numpy as np
import pytest

from _cases import make_pair, rel_l2, to_gpu_layout, to_oracle_layout

pytestmark = pytest.mark.gpu

TOL = {0: 1e-10, 1: 2e-5}  # the repository's parity tolerances of ADG_FP64 and ADG_FP32


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N,S", [(1, 1), (2, 5), (3, 2), (4, 1), (5, 2)])
def test_lts_box_every_degree(N, S, precision):
    from synthetic.workloads import coupled_box, random_dofs
    m, mat = coupled_box(nxy=5, n_water=1, n_crust=2, L=20e3, depth=6e3, water=1e3, grading=6.0, rigid_bottom=True)
    m.face_tag[(m.face_tag == 3) & (np.arange(m.nt)[:, None] % 2 == 0)] = 1  # some free surfaces among the absorbing
    o, s = make_pair(m, mat, N, precision=precision, max_clusters=3, ensemble=S)
    info = s.info
    assert info.n_clusters > 1
    Q0 = random_dofs((S, m.nt, s.B, 9), 5, N=N)
    s.set_dofs(np.ascontiguousarray(np.stack([to_gpu_layout(q) for q in Q0], axis=1)))
    s.set_eta(np.zeros((int(info.n_gravity_faces), S, s.Bf)))
    s.advance(2)
    got = s.get_dofs().reshape(m.nt, S, 9, s.B)
    for k in range(S):
        o.Q, o._D, o.t = Q0[k].copy(), None, 0.0
        o.eta[:] = 0
        for _ in range(2):
            o.advance_macro()
        assert rel_l2(to_oracle_layout(got[:, k]), o.Q) <= TOL[precision]


@pytest.mark.parametrize("precision,N", [(0, 3), (1, 3), (1, 5), (0, 2)])
def test_noalloc_dofs_at_any_element_alignment(precision, N):
    import torch
    from paper_2107_06640_gb300 import _lib
    from synthetic.workloads import plane_wave_case, random_dofs
    m, mat = plane_wave_case(2)
    _, s = make_pair(m, mat, N, precision=precision)
    Q0 = torch.from_numpy(random_dofs((m.nt, 9, s.B), 3, N=N)).to(torch.float64 if precision == 0 else torch.float32)
    out = []
    for off in (0, 1):
        buf = torch.zeros(Q0.numel() + 4, dtype=Q0.dtype, device="cuda")
        d = buf[off:off + Q0.numel()]
        d.copy_(Q0.reshape(-1))
        _lib.adg_step_noalloc(s.ctx, d.data_ptr(), 2, torch.cuda.current_stream().cuda_stream)
        out.append(d.cpu().numpy())
        assert float(buf[:off].abs().sum()) == 0 and float(buf[off + Q0.numel():].abs().sum()) == 0
    s.sync()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N,S,nxy", [(1, 1, 3), (2, 3, 3), (3, 1, 4), (4, 1, 2), (5, 2, 3)])
def test_acoustic_rows(N, S, nxy, precision):
    """The acoustic local kernel (eight elements per warp) on element counts that are no multiple of eight."""
    from synthetic.workloads import coupled_box, random_dofs
    m, mat = coupled_box(nxy=nxy, n_water=3, n_crust=1, L=6e3, depth=4e3, water=2e3, rigid_bottom=True)
    o, s = make_pair(m, mat, N, precision=precision, ensemble=S, acoustic_ocean=True)
    Q0 = random_dofs((S, m.nt, s.B, 9), 7, N=N)
    fluid = mat[2] == 0
    Q0[:, fluid, :, 0:3] = Q0[:, fluid, :, 0:3].mean(axis=-1, keepdims=True)
    Q0[:, fluid, :, 3:6] = 0
    s.set_dofs(np.ascontiguousarray(np.stack([to_gpu_layout(q) for q in Q0], axis=1)))
    s.set_eta(np.zeros((int(s.info.n_gravity_faces), S, s.Bf)))
    s.advance(2)
    got = s.get_dofs().reshape(m.nt, S, 9, s.B)
    assert np.array_equal(got[fluid][:, :, 0], got[fluid][:, :, 2]) and not got[fluid][:, :, 3:6].any()
    for k in range(S):
        o.Q, o._D, o.t = Q0[k].copy(), None, 0.0
        o.eta[:] = 0
        for _ in range(2):
            o.advance_macro()
        assert rel_l2(to_oracle_layout(got[:, k]), o.Q) <= TOL[precision]


@pytest.mark.parametrize("precision", [0, 1])
def test_noalloc_on_an_acoustic_context_without_gravity(precision):
    """Its dofs are in the caller's order, also where fluid and solid elements alternate."""
    import torch
    from paper_2107_06640_gb300 import _lib
    from synthetic.workloads import coupled_box, random_dofs
    m, mat = coupled_box(nxy=2, n_water=1, n_crust=2, L=6e3, depth=4e3, water=2e3)
    m.face_tag[m.face_tag == 2] = 1  # no gravitational surface
    mat = [x.copy() for x in mat]
    for x, solid in zip(mat, (2700.0, 3e10, 3e10)):  # a solid tet between fluid ones
        x[-2] = solid
    N = 3
    o, s = make_pair(m, mat, N, precision=precision, acoustic_ocean=True)
    assert s.info.n_gravity_faces == 0
    Q0 = random_dofs((m.nt, s.B, 9), 17, N=N)
    fluid = mat[2] == 0
    Q0[fluid, :, 0:3] = Q0[fluid, :, 0:3].mean(axis=-1, keepdims=True)
    Q0[fluid, :, 3:6] = 0
    o.Q, o._D, o.t = Q0.copy(), None, 0.0
    d = torch.from_numpy(to_gpu_layout(Q0).copy()).to("cuda", torch.float64 if precision == 0 else torch.float32)
    _lib.adg_step_noalloc(s.ctx, d.data_ptr(), 2, torch.cuda.current_stream().cuda_stream)
    s.sync()
    for _ in range(2):
        o.advance_macro()
    assert rel_l2(to_oracle_layout(d.cpu().numpy().reshape(m.nt, 9, s.B)), o.Q) <= TOL[precision]


@pytest.mark.parametrize("N", [4, 5])
def test_noalloc_on_an_acoustic_tensor_core_context(N):
    """There the library sorts the fluid elements behind the solid ones; the caller's dofs keep the caller's order."""
    import torch
    from paper_2107_06640_gb300 import _lib
    from synthetic.workloads import coupled_box, random_dofs
    m, mat = coupled_box(nxy=2, n_water=1, n_crust=2, L=6e3, depth=4e3, water=2e3)
    m.face_tag[m.face_tag == 2] = 1  # no gravitational surface
    mat = [x.copy() for x in mat]
    for x, water, rock in zip(mat, (1000.0, 2.25e9, 0.0), (2700.0, 3e10, 3e10)):
        x[:] = np.where(np.arange(m.nt) % 3 == 1, rock, water)  # fluid and solid tets alternate
    o, s = make_pair(m, mat, N, precision=2, acoustic_ocean=True)
    fluid = mat[2] == 0
    assert s.info.n_gravity_faces == 0 and s.info.acoustic_updates_per_macro == fluid.sum()
    Q0 = random_dofs((m.nt, s.B, 9), 17, N=N)
    Q0[fluid, :, 0:3] = Q0[fluid, :, 0:3].mean(axis=-1, keepdims=True)
    Q0[fluid, :, 3:6] = 0
    o.Q, o._D, o.t = Q0.copy(), None, 0.0
    s.set_dofs(to_gpu_layout(Q0))
    d = torch.from_numpy(to_gpu_layout(Q0).copy()).to("cuda", torch.float32)
    _lib.adg_step_noalloc(s.ctx, d.data_ptr(), 2, torch.cuda.current_stream().cuda_stream)
    s.sync()
    s.advance(2)
    for _ in range(2):
        o.advance_macro()
    for got in (d.cpu().numpy().reshape(m.nt, 9, s.B), s.get_dofs()):
        assert rel_l2(to_oracle_layout(got), o.Q) <= TOL[1]
