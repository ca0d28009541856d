"""The work that users of the solver have it do, as measurable cases.

A pass is one call sequence of a user's program on a context that it keeps: the
initial state of a scenario is uploaded, the solver advances it through a number
of macro steps, and the whole state is read back (dofs, sea-surface height, fault
state, recorded samples).  The initial state is uploaded on every pass, so that
every pass does the same work.  The host arrays are pinned, as adg.h recommends.

Meshes are Kuhn-split boxes in the shapes of the repository's own workloads: the
periodic unit cube of the plane wave, the ocean over crust with a gravitational
sea surface (flat, or graded with a sea floor of +-500 m for local time stepping)
and the 15-degree megathrust under an ocean.

In the single-precision contexts (ADG_FP32, ADG_3XTF32) the library hands out the
sea surface, the fault state and the receivers as float64 arrays, but what drives
them is the single-precision dofs; they are returned in the dofs' precision.

exact() is the same scheme in plain torch in float64: element by element the
Cauchy-Kovalewski predictor, the Godunov fluxes at the face nodes, rate-2 local
time stepping, the gravitational surface's ODE and the friction laws.
"""

import math
from functools import lru_cache
from itertools import permutations

import numpy as np
import torch

import paper_2107_06640_gb300 as adg
from paper_2107_06640_gb300 import Solver, _lib

PRECISION = {"fp64": adg.ADG_FP64, "fp32": adg.ADG_FP32, "3xtf32": adg.ADG_3XTF32}
INTERIOR, FREE, GRAVITY, ABSORB, PERIODIC, FAULT, RIGID = range(7)
WATER = (1000.0, 1000.0 * 1500.0 ** 2, 0.0)
CRUST = (2700.0, 2700.0 * (6000.0 ** 2 - 2 * 3464.0 ** 2), 2700.0 * 3464.0 ** 2)
UNIT = (1.0, 2.0, 1.0)
FACE_VERTS = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))

#: Every case has all of these keys.
DEFAULT = dict(mesh="ocean", nx=8, ny=8, water=4, crust=35, graded=False, degree=5, precision="3xtf32", acoustic=True,
               clusters=1, ensemble=1, law="", call="advance", steps=8)


def listed():
    return [dict(DEFAULT, **c) for c in (
        # The convergence study: 3,072 tets of the periodic unit cube, degree 3 in double precision, 100 short steps.
        dict(name="plane_wave_p3_fp64", mesh="cube", nx=8, degree=3, precision="fp64", acoustic=False, steps=100),
        # A host application's own device array stepped in place without allocations (adg_step_noalloc), an odd size.
        dict(name="plugin_p3_fp32", mesh="cube", nx=13, degree=3, precision="fp32", acoustic=False, call="noalloc", steps=20),
        # A regional test box of 1,512 tets: one step is a few tiles per SM, launches and latency count.
        dict(name="small_coupled_p5", nx=6, ny=6, crust=3, steps=100),
        # The headline workload, ocean over crust at order 6 on the tensor cores, with global steps.
        dict(name="coupled_p5", nx=28, ny=28, steps=16),
        # The same box in double precision: the runs that the reduced precision is judged against.
        dict(name="coupled_p5_fp64", nx=12, ny=12, precision="fp64", steps=6),
        # Order 4, below the tensor-core degrees: the single-precision CUDA-core kernels, a ragged box.
        dict(name="coupled_p3_fp32", nx=23, ny=19, degree=3, precision="fp32", steps=10),
        # Tsunami generation in a deep ocean at order 5, receivers and sea surface recorded on every step.
        dict(name="ocean_record_p4", nx=20, ny=20, water=34, crust=5, degree=4, call="record", steps=20),
        # A graded mesh with bathymetry and local time steps: four clusters of uneven size, a macro step is 8 ticks.
        dict(name="lts_p5", nx=24, ny=24, graded=True, clusters=6, steps=3),
        # The megathrust with rate-and-state friction, order 5 on the tensor cores.
        dict(name="megathrust_rs_p4", mesh="fault", nx=32, ny=40, water=2, crust=16, degree=4, law="rs", steps=10),
        # A smaller one with linear slip weakening, order 4 in double precision.
        dict(name="megathrust_lsw_p3_fp64", mesh="fault", nx=16, ny=20, water=2, crust=8, degree=3, precision="fp64",
             acoustic=False, law="lsw", steps=10),
        # Sixteen scenarios on one mesh.
        dict(name="ensemble_p5", nx=8, ny=8, ensemble=16, steps=8),
        # States streamed through the GPU, one step each, copies and compute overlapped (the pipelined calls).
        dict(name="stream_p5", nx=16, ny=16, call="stream", steps=6),
    )]


def draw(rng):
    """One more case of these kinds: any degree and precision, sizes spread over their logarithm."""
    kind = rng.choice(("cube", "plugin", "coupled", "coupled", "ocean", "lts", "fault", "ensemble", "stream"))
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    c = dict(DEFAULT, degree=rng.choice((2, 3, 4, 4, 5, 5, 5)), precision=rng.choice(("3xtf32", "3xtf32", "3xtf32", "fp32", "fp64")))
    if kind in ("cube", "plugin"):
        c.update(mesh="cube", nx=log(3, 13), acoustic=False, precision=rng.choice(("fp32", "fp64")))
        c["degree"] = rng.choice((1, 2, 3))
        if kind == "plugin":
            c["call"] = "noalloc"
            c["nx"] = min(c["nx"], 10)
    elif kind == "fault":
        n = log(4, 26)
        c.update(mesh="fault", nx=n, ny=log(4, 36), crust=max(2, n // 2), water=rng.choice((1, 2)), law=rng.choice(("rs", "lsw")))
        c["degree"] = rng.choice((3, 4))
    else:
        c.update(nx=log(3, 24), ny=log(3, 24), water=rng.choice((2, 4)), crust=rng.choice((3, 9, 35)), acoustic=rng.choice((True, True, False)))
        if kind == "ocean":
            c.update(water=rng.choice((12, 34)), crust=5, call="record")
        elif kind == "lts":
            c.update(graded=True, clusters=rng.choice((3, 6)), nx=max(8, c["nx"]), ny=max(8, c["ny"]))
        elif kind == "ensemble":
            c.update(ensemble=rng.choice((2, 5, 16)), nx=min(c["nx"], 8), ny=min(c["ny"], 8))
        elif kind == "stream":
            c.update(call="stream", precision=rng.choice(("3xtf32", "fp32")))
    most = 2e5 if c["precision"] == "fp64" else 2.5e6  # element updates of a pass
    per_step = _tets(c) * c["ensemble"] * (12 if c["graded"] else 1)
    c["steps"] = max(1, min(rng.choice((4, 10, 30)), int(most / per_step)))
    return c


# ---- meshes ---------------------------------------------------------------------------------------------------------


def _tets(c):
    return 6 * c["nx"] * (c["nx"] ** 2 if c["mesh"] == "cube" else c["ny"] * (c["water"] + c["crust"]))


def _graded(length, n, ratio):
    """n + 1 coordinates on [0, length], cells smallest in the middle by `ratio`."""
    half = n // 2
    w = [r ** (k / max(1, m - 1)) for r, m in ((1 / ratio, half), (ratio, n - half)) for k in range(m)]
    w = np.concatenate([np.array(w[:half]) / sum(w[:half]), np.array(w[half:]) / sum(w[half:])]) * length / 2
    return np.concatenate([[0.0], np.cumsum(w)])


@lru_cache(maxsize=2)
def _mesh(key):
    """Vertices, tets, face tags, periodic partners and material of a case's box; `key`: its items."""
    c = dict(key)
    wet = c["water"]
    if c["mesh"] == "cube":
        axes = [np.linspace(0.0, 1.0, c["nx"] + 1)] * 3
        wet = 0
    elif c["mesh"] == "fault":
        dz = 16e3 / c["crust"]
        dx = dz / math.tan(math.radians(15.0))
        axes = [np.arange(c["nx"] + 1) * dx, np.arange(c["ny"] + 1) * dx,
                np.concatenate([np.linspace(-18e3, -2e3, c["crust"] + 1), np.linspace(-2e3, 0.0, wet + 1)[1:]])]
    else:
        sea = -500.0 * wet
        z = np.concatenate([np.linspace(sea - 38e3 / 35 * c["crust"], sea, c["crust"] + 1), np.linspace(sea, 0.0, wet + 1)[1:]])
        axes = [_graded(100e3, n, 32.0) if c["graded"] else 1250.0 * np.arange(n + 1) for n in (c["nx"], c["ny"])] + [z]
    n = [len(a) - 1 for a in axes]
    k, j, i = np.meshgrid(*(np.arange(m + 1) for m in n[::-1]), indexing="ij")
    ijk = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    xyz = np.stack([axes[a][ijk[:, a]] for a in range(3)], 1)
    if c["graded"]:  # the sea floor lifted by up to 500 m, the layers above and below stretched with it
        bottom, sea = axes[2][0], axes[2][c["crust"]]
        floor = sea + 0.25 * -sea * np.sin(2 * np.pi * xyz[:, 0] / 100e3) * np.sin(2 * np.pi * xyz[:, 1] / 100e3)
        z = xyz[:, 2]
        xyz[:, 2] = np.where(z <= sea, bottom + (z - bottom) * (floor - bottom) / (sea - bottom), floor * z / sea)
    k, j, i = np.meshgrid(*(np.arange(m) for m in n[::-1]), indexing="ij")
    hexes = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    vid = lambda p: p[..., 0] + (n[0] + 1) * (p[..., 1] + (n[1] + 1) * p[..., 2])  # noqa: E731
    unit = np.eye(3, dtype=np.int64)
    corners = np.array([[0 * unit[0], unit[p[0]], unit[p[0]] + unit[p[1]], unit.sum(0)] for p in permutations(range(3))])
    tets = vid(hexes[:, None, None, :] + corners[None]).reshape(-1, 4)
    layer = np.repeat(hexes[:, 2], 6)
    p = xyz[tets]
    det = np.einsum("ij,ij->i", np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), p[:, 3] - p[:, 0])
    tets[det < 0] = tets[det < 0][:, [0, 2, 1, 3]]
    tag = np.zeros((len(tets), 4), np.int32)
    partner = np.full((len(tets), 4), -1, np.int64)
    at = ijk[tets][:, np.array(FACE_VERTS)]  # [tet][face][vertex][axis], grid indices
    for a in range(3):
        sides = [np.all(at[..., a] == end, 2) for end in (0, n[a])]
        for up, on in enumerate(sides):
            tag[on] = PERIODIC if c["mesh"] == "cube" else GRAVITY if a == 2 and up else ABSORB
        if c["mesh"] == "cube":
            others = [b for b in range(3) if b != a]
            ids, keys = [], []
            for on in sides:
                t, f = np.nonzero(on)
                code = np.sort(at[t, f][:, :, others] @ np.array([1, n[0] + 1]), 1)
                ids.append(t * 4 + f)
                keys.append(np.lexsort(code.T))
            lo, hi = ids[0][keys[0]], ids[1][keys[1]]
            partner.ravel()[lo], partner.ravel()[hi] = hi, lo
    if c["mesh"] == "fault":  # the index diagonal i = k of the crust dips by 15 degrees
        on = np.all(at[..., 0] == at[..., 2], 2) & np.all(at[..., 2] <= c["crust"], 2) & (tag == INTERIOR)
        tag[on] = FAULT
    solid = UNIT if c["mesh"] == "cube" else CRUST
    in_water = layer >= n[2] - wet if wet else np.zeros(len(tets), bool)
    mat = [np.where(in_water, w, s) for w, s in zip(WATER, solid)]
    return xyz, tets, tag, partner, mat


def _key(c):
    return tuple((k, c[k]) for k in ("mesh", "nx", "ny", "water", "crust", "graded"))


def _cfl(c):
    return 0.5 if c["mesh"] == "cube" else 0.35


# ---- inputs ---------------------------------------------------------------------------------------------------------


def _state(c, seed, count=1):
    """`count` initial states [nt][S][9][B]: a seafloor velocity pulse (the fault boxes: at rest) and small noise in all
    modes, larger modes smaller; stresses in proportion to density and wave speed.  float32 values in every precision."""
    xyz, tets, _, _, (rho, lam, mu) = _mesh(_key(c))
    B = (c["degree"] + 1) * (c["degree"] + 2) * (c["degree"] + 3) // 6
    g = torch.Generator("cuda").manual_seed(seed)
    mid = torch.from_numpy(xyz[tets].mean(1)).cuda()
    lo, hi = mid.min(0).values, mid.max(0).values
    z = torch.from_numpy(np.sqrt(rho * (lam + 2 * mu))).cuda().float()
    decay = (1.0 + torch.arange(B, device="cuda")) ** -1.0
    out = []
    for _ in range(count):
        q = torch.randn((len(tets), c["ensemble"], 9, B), device="cuda", generator=g)
        q *= decay * (1e-6 if c["law"] else 1e-2)
        if not c["law"]:
            for s in range(c["ensemble"]):
                at = lo + (hi - lo) * (0.2 + 0.6 * torch.rand(3, device="cuda", generator=g))
                r2 = (((mid - at) / (0.15 * (hi - lo))) ** 2).sum(1)
                q[:, s, 8, 0] += torch.exp(-0.5 * r2).float() / math.sqrt(6.0)
        q[:, :, :6] *= z[:, None, None, None]
        if c["acoustic"]:  # what the acoustic ocean makes of an upload
            wet = torch.from_numpy(mu == 0).cuda()
            q[wet, :, :3] = q[wet, :, :3].mean(2, keepdim=True)
            q[wet, :, 3:6] = 0
        out.append(q)
    return out


def _surface(c, seed, xy):
    """Sea-surface height [face][S][node]: a few broad bumps for each scenario."""
    rng = np.random.default_rng(seed)
    size = xy.reshape(-1, 2).max(0) - xy.reshape(-1, 2).min(0)
    eta = np.zeros((xy.shape[0], c["ensemble"], xy.shape[1]))
    for s in range(c["ensemble"]):
        for _ in range(4):
            at, w = xy.reshape(-1, 2).min(0) + rng.uniform(0.1, 0.9, 2) * size, rng.uniform(0.1, 0.3) * size.max()
            eta[:, s] += rng.uniform(0.1, 2.0) * np.exp(-((xy - at) ** 2).sum(-1) / (2 * w * w))
    return eta


def _friction(c, seed, xyz, normal):
    """Parameters [face][1][node][13] of the two laws: +-5 % noise, an overstressed patch in the middle."""
    rng = np.random.default_rng(seed)
    out = np.zeros(xyz.shape[:2] + (13,))
    rs = c["law"] == "rs"
    for k, v in enumerate((0.01, 0.014, 0.2, 0.6, 1e-6) if rs else (0.6, 0.4, 0.5)):
        out[..., k] = v * (1.0 + 0.05 * rng.uniform(-1.0, 1.0, xyz.shape[:2]))
    if rs:
        out[..., 5:7] = 0.1
        out[..., 11], out[..., 12] = 0.6, 1e-12
    else:
        out[..., 3] = 2e6 * np.clip(1.0 - (xyz[..., 2].max() - xyz[..., 2]) / 10e3, 0.0, 1.0)
    out[..., 7] = -40e6
    up = np.array([0.0, 0.0, 1.0]) - normal[:, 2:] * normal
    up /= np.linalg.norm(up, axis=1, keepdims=True)
    near = np.linalg.norm(xyz - xyz.reshape(-1, 3).mean(0), axis=2) < 8.01e3
    mag = 40e6 * np.where(near, 0.85 if rs else 0.62, 0.55 if rs else 0.48)
    out[..., 8:11] = mag[..., None] * up[:, None]
    return out[:, None]


def _receivers(c, seed):
    """Elements and reference coordinates of up to 1,000 receivers."""
    rng = np.random.default_rng(seed + 1)
    e = rng.choice(_tets(c), min(1000, _tets(c)), replace=False)
    return e, 0.25 + rng.uniform(-0.08, 0.08, (len(e), 3))


def prepare(case, seed):
    xyz, tets, tag, partner, mat = _mesh(_key(case))
    N, S = case["degree"], case["ensemble"]
    st = {"case": case, "f64": case["precision"] == "fp64"}
    sol = st["sol"] = Solver(xyz, tets, tag, *mat, face_partner=partner, degree=N, precision=PRECISION[case["precision"]],
                             cfl=_cfl(case), max_clusters=case["clusters"], ensemble=S, acoustic_ocean=case["acoustic"])
    states = _state(case, seed, case["steps"] if case["call"] == "stream" else 1)
    if case["call"] == "noalloc":
        st["q0"] = states[0].reshape(len(tets), 9, -1).to(torch.float64 if st["f64"] else torch.float32)
        st["q"] = torch.empty_like(st["q0"])
        return st
    if st["f64"]:
        st["in"] = [q.cpu().numpy().astype(np.float64) for q in states]
    else:
        st["in"] = [torch.empty(q.shape, dtype=torch.float32, pin_memory=True).copy_(q).numpy() for q in states]
        st["out"] = [torch.empty(q.shape, dtype=torch.float32, pin_memory=True).numpy() for q in states]
    if int(sol.info.n_gravity_faces):
        st["eta"] = _surface(case, seed, sol.gravity_faces()[1][..., :2])
    if case["law"]:
        nff = st["faults"] = int(sol.info.n_fault_faces)
        _, _, node, normal = _lib.adg_fault_faces(sol.ctx, nff, sol.Bf)
        if case["law"] == "lsw":
            _lib.adg_set_friction_law(sol.ctx, _lib.ADG_FRICTION_LSW)
        st["par"] = _friction(case, seed, node, normal)
    if case["call"] == "record":
        e, xi = _receivers(case, seed)
        p = xyz[tets[e]]
        sol.add_receivers(p[:, 0] + np.einsum("na,nad->nd", xi, p[:, 1:] - p[:, :1]))
        sol.record(_lib.ADG_RECORD_RECEIVERS, 1, case["steps"])
        sol.record(_lib.ADG_RECORD_SSH, 1, case["steps"])
    return st


def run(st):
    case, sol = st["case"], st["sol"]
    n = case["steps"]
    if case["call"] == "noalloc":
        st["q"].copy_(st["q0"])
        _lib.adg_step_noalloc(sol.ctx, st["q"].data_ptr(), n, torch.cuda.current_stream().cuda_stream)
        return {"dofs": st["q"]}
    real = np.float64 if st["f64"] else np.float32
    got = {}
    if "eta" in st:
        sol.set_eta(st["eta"])
    if "par" in st:
        _lib.adg_set_fault(sol.ctx, st["par"])
    if case["call"] == "stream":
        for q, o in zip(st["in"], st["out"]):
            sol.set_dofs_f32_async(q)
            sol.advance_async(1)
            sol.get_dofs_f32_async(o)
        sol.sync()
        got["dofs"] = st["out"]
    elif st["f64"]:
        sol.set_dofs(st["in"][0])
        sol.advance(n)
        got["dofs"] = sol.get_dofs()
    else:
        sol.set_dofs_f32(st["in"][0])
        sol.advance(n)
        got["dofs"] = sol.get_dofs_f32(st["out"][0])
    if "eta" in st:
        got["eta"] = sol.read_ssh().astype(real)
    if "par" in st:
        got["fault"] = _lib.adg_read_fault(sol.ctx, np.empty((st["faults"], 1, sol.Bf, 8))).astype(real)
    if case["call"] == "record":
        got["receivers"] = sol.read_record(_lib.ADG_RECORD_RECEIVERS)[1].astype(real)
        got["surface"] = sol.read_record(_lib.ADG_RECORD_SSH)[1].astype(real)
    return got


# ---- reference operators --------------------------------------------------------------------------------------------


def _jacobi(n, a, x, t):
    """t^n P_n^(a,0)(2 x / t - 1) and its derivatives by x and t, from the sum over (x - t)^s x^(n - s)."""
    v, dx, dt = (np.zeros_like(x) for _ in range(3))
    for s in range(n + 1):
        w = math.comb(n + a, n - s) * math.comb(n, s)
        p, q = (x - t) ** s, x ** (n - s)
        dp = s * (x - t) ** (s - 1) if s else 0.0 * x
        dq = (n - s) * x ** (n - s - 1) if n > s else 0.0 * x
        v, dx, dt = v + w * p * q, dx + w * (dp * q + p * dq), dt - w * dp * q
    return v, dx, dt


def _basis(N, x):
    """The Dubiner products at points x (n, 3), not normalised, and their gradients (n, B, 3)."""
    xi, eta, zeta = x.T
    s, t, one = 1 - eta - zeta, 1 - zeta, np.ones_like(xi)
    val, grad = [], []
    for n in range(N + 1):
        for i in range(n + 1):
            for j in range(n - i + 1):
                a, ax, as_ = _jacobi(i, 0, xi, s)
                b, by, bt = _jacobi(j, 2 * i + 1, eta, t)
                d, dz, _ = _jacobi(n - i - j, 2 * i + 2 * j + 2, zeta, one)
                val.append(a * b * d)
                grad.append(np.stack([ax * b * d, (a * by - as_ * b) * d, -as_ * b * d - a * bt * d + a * b * dz], 1))
    return np.stack(val, 1), np.stack(grad, 1)


def _face_points(f, chi):
    v = np.array([[0.0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]])[list(FACE_VERTS[f])]
    return v[0] + chi[:, :1] * (v[1] - v[0]) + chi[:, 1:] * (v[2] - v[0])


@lru_cache(maxsize=None)
def _reference(N):
    """kt[a][m][l] = int phi_m dphi_l/dxi_a, face values [f][n][l], lift [f][m][n], barycentric face nodes, basis norms."""
    p, w = np.polynomial.legendre.leggauss(N + 4)
    p, w = (p + 1) / 2, w / 2
    z, y, x = (a.ravel() for a in np.meshgrid(p, p, p, indexing="ij"))
    wz, wy, wx = (a.ravel() for a in np.meshgrid(w, w, w, indexing="ij"))
    pts, wt = np.stack([x * (1 - y) * (1 - z), y * (1 - z), z], 1), wx * wy * (1 - y) * wz * (1 - z) ** 2
    v, g = _basis(N, pts)
    norm = 1 / np.sqrt(np.einsum("q,ql,ql->l", wt, v, v))
    kt = np.einsum("q,qm,qla->aml", wt, v * norm, g * norm[:, None])
    kt[np.abs(kt) < 1e-11] = 0
    b, a = (q.ravel() for q in np.meshgrid(p, p, indexing="ij"))
    wb, wa = (q.ravel() for q in np.meshgrid(w, w, indexing="ij"))
    chi, wc = np.stack([a * (1 - b), b], 1), wa * wb * (1 - b)
    ij = np.array([(i, j) for j in range(N + 1) for i in range(N + 1 - j)])
    powers = [(i, j) for i in range(N + 1) for j in range(N + 1 - i)]
    mono = lambda c: np.stack([c[:, 0] ** i * c[:, 1] ** j for i, j in powers], 1)  # noqa: E731
    nodal = mono(chi) @ np.linalg.inv(mono(ij / N))
    face = np.stack([_basis(N, _face_points(f, ij / N))[0] * norm for f in range(4)])
    lift = np.stack([np.einsum("q,qm,qn->mn", wc, _basis(N, _face_points(f, chi))[0] * norm, nodal) for f in range(4)])
    return kt, face, lift, np.column_stack([N - ij.sum(1), ij]), norm


# ---- the scheme in float64 ------------------------------------------------------------------------------------------


class _Exact:
    """The scheme on a case's mesh for one scenario; dofs Q [element][basis][quantity]."""

    def __init__(self, c):
        xyz, tets, tag, partner, mat = _mesh(_key(c))
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev)  # noqa: E731
        N = self.N = c["degree"]
        kt, face, lift, bary, self.norm = _reference(N)
        self.kt, self.face, self.lift = t(kt), t(face), t(lift)
        E = self.E = len(tets)
        P = xyz[tets]
        J = np.stack([P[:, k] - P[:, 0] for k in (1, 2, 3)], 2)
        det, Ji = np.linalg.det(J), np.linalg.inv(J)
        V = P[:, np.array(FACE_VERTS)]  # [e][f][vertex][3]
        cr = np.cross(V[:, :, 1] - V[:, :, 0], V[:, :, 2] - V[:, :, 0])
        area = np.linalg.norm(cr, axis=2)  # twice the face's
        out = np.sign(np.einsum("efd,efd->ef", cr, V[:, :, 0] - P))
        self.normal = t(cr / area[..., None] * out[..., None])
        self.scale = t(area / det[:, None])
        self.tag = t(tag)
        # neighbours: interior and fault faces by their vertices, periodic ones by their partners
        nb = partner.copy()
        ids = np.flatnonzero((tag == INTERIOR) | (tag == FAULT))
        tri = np.sort(tets[:, np.array(FACE_VERTS)].reshape(-1, 3)[ids], 1)
        key = (tri[:, 0] * len(xyz) + tri[:, 1]) * len(xyz) + tri[:, 2]
        pairs = ids[np.argsort(key, kind="stable")].reshape(-1, 2)
        nb.ravel()[pairs[:, 0]], nb.ravel()[pairs[:, 1]] = pairs[:, 1], pairs[:, 0]
        # my face node n is the neighbour's node: its weights on my vertices, taken to the neighbour's
        rel = (V - V.mean(2, keepdims=True)).reshape(-1, 3, 3)
        has = np.flatnonzero(nb.ravel() >= 0)
        d = np.linalg.norm(rel[has][:, :, None] - rel[nb.ravel()[has]][:, None], axis=3)
        sig = np.argmin(d, 2)
        theirs = np.zeros((len(has), len(bary), 3), np.int64)
        np.put_along_axis(theirs, np.broadcast_to(sig[:, None], theirs.shape), np.broadcast_to(bary, theirs.shape), 2)
        at = np.zeros((N + 1, N + 1), np.int64)
        at[bary[:, 1], bary[:, 2]] = np.arange(len(bary))
        perm = np.zeros((4 * E, len(bary)), np.int64)
        perm[has] = at[theirs[..., 1], theirs[..., 2]]
        self.nb, self.perm = t(nb), t(perm.reshape(E, 4, -1))
        self.bary, self.V = bary, V
        rho, lam, mu = mat
        cp = np.sqrt((lam + 2 * mu) / rho)
        dt = _cfl(c) / (2 * N + 1) * 2 * det / area.sum(1) / cp
        self.dt = dt.min()
        cl = np.clip(np.floor(np.log2(dt / self.dt) + 1e-12).astype(np.int64), 0, c["clusters"] - 1)
        while True:
            old = cl
            beside = np.where(nb >= 0, cl[nb // 4], 99) + np.where(tag == FAULT, 0, 1)
            cl = np.minimum(cl, beside.min(1))
            if np.array_equal(cl, old):
                break
        self.cl = t(cl)
        self.rho, self.lam, self.mu = (t(m) for m in mat)
        self.Zp, self.Zs = torch.sqrt(self.rho * (self.lam + 2 * self.mu)), torch.sqrt(self.rho * self.mu)
        A = torch.zeros((3, E, 9, 9), dtype=torch.float64, device=dev)  # of the x, y and z directions
        for d in range(3):
            for i in range(3):
                A[d, :, i, 6 + d] -= self.lam
            for row, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2))):
                if j == d:
                    A[d, :, row, 6 + i] -= self.mu
                if i == d:
                    A[d, :, row, 6 + j] -= self.mu
            for i, row in enumerate(((0, 3, 5), (3, 1, 4), (5, 4, 2))[d]):
                A[d, :, 6 + i, row] = -1 / self.rho
        self.star = torch.einsum("ead,depq->aepq", t(Ji), A)
        self.g = 9.81
        self.gravity = torch.nonzero(self.tag == GRAVITY)  # in the caller's order
        fe, ff = np.nonzero((tag == FAULT) & (nb // 4 > np.arange(E)[:, None]))
        order = np.lexsort((ff, fe, cl[fe]))
        self.fault = t(np.stack([fe[order], ff[order]], 1))
        self.Q = self.eta = self.par = None
        self.flux_of = {}

    def nodes(self, ef):
        """Physical face nodes of the faces ef (n, 2)."""
        return np.einsum("nv,xvd->xnd", self.bary / self.N, self.V[ef[:, 0], ef[:, 1]])

    def derivatives(self, idx):
        D = [self.Q[idx]]
        for _ in range(self.N):
            D.append(-sum(torch.matmul(torch.matmul(self.kt[a], D[-1]), self.star[a, idx].transpose(1, 2)) for a in range(3)))
        return D

    @staticmethod
    def integral(D, ta, tb):
        return sum((tb ** (k + 1) - ta ** (k + 1)) / math.factorial(k + 1) * d for k, d in enumerate(D))

    @staticmethod
    def traction(q, n):
        s = lambda *i: q[..., i[0]] * n[..., 0] + q[..., i[1]] * n[..., 1] + q[..., i[2]] * n[..., 2]  # noqa: E731
        return torch.stack([s(0, 3, 5), s(3, 1, 4), s(5, 4, 2)], -1)

    @staticmethod
    def split(x, n):
        xn = (x * n).sum(-1, keepdim=True)
        return xn, x - xn * n

    @staticmethod
    def normal_flux(n, tb, vb, rho, lam, mu):
        """n . (A, B, C) on a state of traction tb and velocity vb."""
        lam, mu, rho = (a[:, None] for a in (lam, mu, rho))
        nv = (n * vb).sum(-1)
        rows = [-mu * (n[..., j] * vb[..., i] + n[..., i] * vb[..., j]) - (lam * nv if i == j else 0)
                for i, j in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2))]
        return torch.stack(rows + [-tb[..., i] / rho for i in range(3)], -1)

    def flux(self, idx, f, qm, qp, D, dt, k):
        """Time-integrated flux [x][node][9] through face f of the elements idx; qp: the neighbours' values."""
        n = self.normal[idx, f][:, None]
        tag = self.tag[idx, f]
        nb = torch.where(self.nb[idx, f] >= 0, self.nb[idx, f] // 4, idx)
        col = lambda a: a[:, None, None]  # noqa: E731
        Zp, Zs, Zpp, Zsp = col(self.Zp[idx]), col(self.Zs[idx]), col(self.Zp[nb]), col(self.Zs[nb])
        tn, ts = self.split(self.traction(qm, n), n)
        vn, vs = self.split(qm[..., 6:], n)
        tnp, tsp = self.split(self.traction(qp, n), n)
        vnp, vsp = self.split(qp[..., 6:], n)
        for bt, (a, b, d, e) in {FREE: (-1, -1, 1, 1), ABSORB: (0, 0, 0, 0), RIGID: (1, -1, -1, 1), GRAVITY: (-1, -1, 1, 1)}.items():
            on = col(tag == bt)
            tnp, tsp, vnp, vsp = (torch.where(on, s * own, x) for s, own, x in ((a, tn, tnp), (b, ts, tsp), (d, vn, vnp), (e, vs, vsp)))
        a1 = Zp * Zpp / (Zp + Zpp) * ((tn - tnp) / Zpp + vn - vnp)
        tnb, vnb = tn - a1, vn - a1 / Zp
        one = torch.ones_like(Zs)
        solid, fluid = (Zs > 0) & (Zsp > 0), Zs == 0
        cs = Zs * Zsp / torch.where(solid, Zs + Zsp, one)
        a2 = cs * ((ts - tsp) / torch.where(solid, Zsp, one) + vs - vsp)
        tsb = torch.where(solid, ts - a2, 0 * ts)
        vsb = torch.where(fluid, vs, vs - torch.where(solid, a2, ts) / torch.where(fluid, one, Zs))
        g = torch.nonzero(tag == GRAVITY)[:, 0]
        if len(g):
            e, ng = idx[g], n[g]
            fm = []
            for m, d in enumerate(D):
                q = torch.matmul(self.face[f], d[g])
                fm.append((self.split(q[..., 6:], ng)[0] - self.split(self.traction(q, ng), ng)[0] / Zp[g])[..., 0] / math.factorial(m))
            kappa = (self.rho[e] * self.g / self.Zp[e])[:, None]
            a = e0 = self.eta[e, f]
            e1, H = e0.clone(), e0 * dt
            for m in range(self.N + 30):
                a = ((fm[m] if m <= self.N else 0.0) - kappa * a) / (m + 1)
                e1 = e1 + a * dt ** (m + 1)
                H = H + a * dt ** (m + 2) / (m + 2)
            self.eta[e, f] = e1
            tnb[g], vnb[g] = (-self.rho[e] * self.g)[:, None, None] * H[..., None], (e1 - e0)[..., None]
            tsb[g], vsb[g] = 0.0, torch.where(fluid[g], vs[g], vs[g] - ts[g] / torch.where(fluid, one, Zs)[g])
        F = self.normal_flux(n, tnb * n + tsb, vnb * n + vsb, self.rho[idx], self.lam[idx], self.mu[idx])
        if k in self.flux_of:
            Fm, Fp, sel = self.flux_of[k]
            where = torch.full((self.E,), -1, device=idx.device)
            where[idx] = torch.arange(len(idx), device=idx.device)
            e, fm = self.fault[sel].T
            on = fm == f
            F[where[e[on]]] = Fm[on]
            other = self.nb[e, fm]
            on = other % 4 == f
            F[where[other[on] // 4]] = Fp[on]
        return F

    def slide(self, k, D, dt):
        """The friction solves of cluster k over its step from the expansions D of all elements."""
        sel = torch.nonzero(self.cl[self.fault[:, 0]] == k)[:, 0]
        if not len(sel):
            return
        e, f = self.fault[sel].T
        e2, f2 = self.nb[e, f] // 4, self.nb[e, f] % 4
        perm = self.perm[e, f]
        n = self.normal[e, f][:, None].expand(-1, perm.shape[1], -1)
        col = lambda a: a[:, None, None]  # noqa: E731
        Zp, Zs, Zpp, Zsp = col(self.Zp[e]), col(self.Zs[e]), col(self.Zp[e2]), col(self.Zs[e2])
        eta = Zs * Zsp / (Zs + Zsp)
        Dm = [torch.matmul(self.face[f], d[e]) for d in D]
        Dp = [torch.gather(torch.matmul(self.face[f2], d[e2]), 1, perm[..., None].expand(-1, -1, 9)) for d in D]
        par = self.par[sel, 0]
        t0 = self.split(par[..., 8:11], n)[1]
        V, psi = self.V_[sel], self.psi[sel]
        x, w = np.polynomial.legendre.leggauss(self.N + 1)
        Gm = Gp = 0.0
        last, et = 0.0, eta[..., 0]
        slip = self.slip[sel]
        for xj, wj in zip((x + 1) / 2 * dt, w / 2 * dt):
            qm, qp = (sum(xj ** m / math.factorial(m) * d for m, d in enumerate(S)) for S in (Dm, Dp))
            tn, ts = self.split(self.traction(qm, n), n)
            vn, vs = self.split(qm[..., 6:], n)
            tnp, tsp = self.split(self.traction(qp, n), n)
            vnp, vsp = self.split(qp[..., 6:], n)
            a1 = Zp * Zpp / (Zp + Zpp) * ((tn - tnp) / Zpp + vn - vnp)
            theta = t0 + eta * (vsp - vs + tsp / Zsp + ts / Zs)
            th = theta.norm(dim=-1)
            S = torch.clamp(-(par[..., 7] + (tn - a1)[..., 0]), min=0.0)
            old, h = V, xj - last
            for again in (False, True):
                mid = 0.5 * (old + V) if again else old
                if self.law == "lsw":
                    new = psi + mid * h
                    fr = par[..., 0] - (par[..., 0] - par[..., 1]) * torch.clamp(new / par[..., 2], max=1.0)
                    V = torch.clamp(th - (par[..., 3] + fr * S), min=0.0) / et
                else:
                    new = self.relax(psi, mid, h, par)
                    V = self.slip_rate(th, S, et, new, V, par)
            psi, last = new, xj
            d = theta / torch.where(th > 0, th, torch.ones_like(th))[..., None]
            tau = (th - et * V)[..., None] * d
            dv = tau - t0
            slip = slip + wj * V[..., None] * d
            tb, vb = (tn - a1) * n + dv, (vn - a1 / Zp) * n
            Gm = Gm + wj * self.normal_flux(n, tb, vb + vs + (dv - ts) / Zs, self.rho[e], self.lam[e], self.mu[e])
            Gp = Gp - wj * self.normal_flux(n, tb, vb + vsp - (dv - tsp) / Zsp, self.rho[e2], self.lam[e2], self.mu[e2])
        self.psi[sel] = psi + V * (dt - last) if self.law == "lsw" else self.relax(psi, V, dt - last, par)
        self.V_[sel], self.slip[sel], self.tau[sel] = V, slip, tau
        self.flux_of[k] = (Gm, torch.zeros_like(Gp).scatter(1, perm[..., None].expand(-1, -1, 9), Gp), sel)

    @staticmethod
    def relax(psi, V, h, par):
        a, b, L, f0, V0, fw, Vw = (par[..., i] for i in range(7))
        V = torch.clamp(V, min=1e-300)
        fss = fw + (f0 - (b - a) * torch.log(V / V0) - fw) / (1 + (V / Vw) ** 8) ** 0.125
        x = fss / a
        ss = a * (torch.log(2 * V0 / V) + x + torch.log1p(-torch.exp(-2 * x)) - math.log(2.0))
        return ss + (psi - ss) * torch.exp(-V * h / L)

    @staticmethod
    def slip_rate(th, S, eta, psi, V, par):
        """The root of Theta - eta V = S a asinh(V / (2 V0) e^(psi / a)), by Newton in ln V."""
        a, lc = par[..., 0], psi / par[..., 0] - torch.log(2 * par[..., 4])
        hi = torch.log(th / eta)
        x = torch.minimum(torch.log(torch.clamp(V, min=1e-300)), hi)
        for _ in range(100):
            v, cv = torch.exp(x), torch.exp(lc + x)
            step = (th - eta * v - S * a * torch.asinh(cv)) / (-eta * v - S * a * cv / torch.sqrt(1 + cv * cv))
            new = torch.minimum(torch.clamp(x - step, min=-700.0), hi)
            done = float((new - x).abs().max()) < 1e-13
            x = new
            if done:
                break
        return torch.exp(x)

    def macro(self):
        """One macro step of rate-2 local time stepping."""
        kmax = int(self.cl.max())
        sets = [torch.nonzero(self.cl == k)[:, 0] for k in range(kmax + 1)]
        D = [torch.zeros_like(self.Q) for _ in range(self.N + 1)]
        own, buf = torch.zeros_like(self.Q), torch.zeros_like(self.Q)
        for s in range(1 << kmax):
            for k, idx in enumerate(sets):
                if s % (1 << k) == 0 and len(idx):
                    for m, d in enumerate(self.derivatives(idx)):
                        D[m][idx] = d
                    own[idx] = self.integral([d[idx] for d in D], 0.0, (1 << k) * self.dt)
                    buf[idx] = own[idx] + (0.0 if s % (2 << k) == 0 else buf[idx])
            for k, idx in enumerate(sets):
                if (s + 1) % (1 << k) or not len(idx):
                    continue
                dt = (1 << k) * self.dt
                self.slide(k, D, dt)
                I = own[idx]
                Dk = [d[idx] for d in D]
                dQ = sum(torch.matmul(torch.matmul(self.kt[a].T, I), self.star[a, idx].transpose(1, 2)) for a in range(3))
                second = float(((s + 1) // (1 << k) - 1) % 2)
                for f in range(4):
                    nb = self.nb[idx, f]
                    e2, f2 = torch.clamp(nb, min=0) // 4, torch.clamp(nb, min=0) % 4
                    J = torch.where((self.cl[e2] < k)[:, None, None], buf[e2], own[e2])
                    far = torch.nonzero(self.cl[e2] > k)[:, 0]
                    if len(far):
                        J[far] = self.integral([d[e2[far]] for d in D], second * dt, (second + 1) * dt)
                    qp = torch.zeros(len(idx), self.face.shape[1], 9, dtype=I.dtype, device=I.device)
                    for g in range(4):
                        on = f2 == g
                        qp[on] = torch.matmul(self.face[g], J[on])
                    qp = torch.gather(qp, 1, self.perm[idx, f][..., None].expand(-1, -1, 9))
                    F = self.flux(idx, f, torch.matmul(self.face[f], I), qp, Dk, dt, k)
                    dQ -= self.scale[idx, f][:, None, None] * torch.matmul(self.lift[f], F)
                self.Q[idx] += dQ


def exact(case, seed):
    sim = _Exact(case)
    dev, S, n = sim.kt.device, case["ensemble"], case["steps"]
    if case["law"]:
        ef = sim.fault.cpu().numpy()
        sim.law = case["law"]
        sim.par = torch.from_numpy(_friction(case, seed, sim.nodes(ef), sim.normal[ef[:, 0], ef[:, 1]].cpu().numpy())).to(dev)
        sim.psi, sim.V_ = sim.par[:, 0, :, 11].clone(), sim.par[:, 0, :, 12].clone()
        sim.slip, sim.tau = (torch.zeros(sim.psi.shape + (3,), dtype=torch.float64, device=dev) for _ in range(2))
    grav = sim.gravity
    if len(grav):
        eta0 = torch.from_numpy(_surface(case, seed, sim.nodes(grav.cpu().numpy())[..., :2])).to(dev)
    stream = case["call"] == "stream"
    states = [q.double() for q in _state(case, seed, n if stream else 1)]
    dofs, eta, receivers, surface = [[] for _ in range(n if stream else 1)], [], [], []
    if case["call"] == "record":
        e, xi = _receivers(case, seed)
        phi, e = torch.from_numpy(_basis(sim.N, xi)[0] * sim.norm).to(dev), torch.from_numpy(e).to(dev)
    for s in range(S):
        if len(grav):
            sim.eta = torch.zeros((sim.E, 4, len(sim.bary)), dtype=torch.float64, device=dev)
            sim.eta[grav[:, 0], grav[:, 1]] = eta0[:, s]
        for k, q in enumerate(states):
            sim.Q = q[:, s].transpose(1, 2).contiguous()
            for _ in range(1 if stream else n):
                sim.macro()
                if case["call"] == "record":
                    receivers.append(torch.einsum("nl,nlp->np", phi, sim.Q[e])[:, None])
                    surface.append(sim.eta[grav[:, 0], grav[:, 1]][:, None])
            dofs[k].append(sim.Q.transpose(1, 2))
        if len(grav):
            eta.append(sim.eta[grav[:, 0], grav[:, 1]])
    dofs = [torch.stack(q, 1) for q in dofs]
    got = {"dofs": dofs if stream else dofs[0]}
    if len(grav):
        got["eta"] = torch.stack(eta, 1)
    if case["law"]:
        got["fault"] = torch.cat([sim.V_[..., None], sim.psi[..., None], sim.slip, sim.tau], -1)[:, None]
    if case["call"] == "record":
        got["receivers"], got["surface"] = torch.stack(receivers), torch.stack(surface)
    return got


@lru_cache(maxsize=None)
def _updates(key, degree, clusters, cfl):
    """Element updates of one macro step."""
    sim = _Exact(dict(DEFAULT, **dict(key), degree=degree, clusters=clusters))
    counts = torch.bincount(sim.cl).tolist()
    return sum(n << (len(counts) - 1 - k) for k, n in enumerate(counts))


def work(case):
    """Of one pass: every element update reads and writes its dofs and passes its face traces on once, and the nonzero
    entries of the reference matrices, the star products and the fluxes are what it computes; plus the transfers."""
    kt, face, lift, bary, _ = _reference(case["degree"])
    N, B, Bf = case["degree"], face.shape[2], len(bary)
    size = 8 if case["precision"] == "fp64" else 4
    per = _tets(case) if not case["graded"] else _updates(_key(case), N, case["clusters"], _cfl(case))
    updates = per * case["steps"] * case["ensemble"]
    rows = lambda k: (N - k + 1) * (N - k + 2) * (N - k + 3) // 6  # noqa: E731
    flops = sum(18 * np.count_nonzero(kt[:, : rows(k + 1), : rows(k)]) + 75 * rows(k + 1) for k in range(N))
    flops += 18 * (np.count_nonzero(kt) + np.count_nonzero(np.abs(face) > 1e-11) + np.count_nonzero(np.abs(lift) > 1e-13))
    flops += 75 * B + 18 * sum(rows(k) for k in range(N + 1)) + 4 * Bf * 110
    states = case["steps"] if case["call"] == "stream" else 1
    moved = 2 * states * _tets(case) * case["ensemble"] * 9 * B * size
    return {"bytes": updates * size * 9 * (2 * B + 8 * Bf) + moved, "flops": updates * int(flops)}
