"""FP64 operator on LGL nodes: block fixed point against the oracle where its
range and its branches end -- densities varying by more than the series of the
logarithmic means take (ratio 1.13 and 1.67), by about the admitted factor of
8 to 16 and beyond it (those elements run in FP64), blocks that hold elements
of both kinds, velocities of zero and of Mach 17, low Mach numbers and states
of far-off scales.

Bar: R(U) within 1e-12 of max |R| per variable and ten RK steps within 1e-10,
as for the parity tests.  The momentum of R comes from the variation of the
pressure while the rounding of the metric terms (1e-13 between the two codes)
multiplies its mean, so the bar grows with their quotient (2.5 for the ranges
0.8 to 1.2, 5.5 for the low Mach number).  Meshes above the node count of the
latency kernels, with ragged last blocks."""
import numpy as np
import pytest

from workloads import box_mesh, random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZE = {1: 13, 2: 9, 3: 7, 4: 3, 5: 3, 7: 2, 8: 2}


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _err(got, ref):
    d = np.abs(got - ref).reshape(ref.shape[0], 5, -1).max(axis=(0, 2))
    return d / np.abs(ref).reshape(ref.shape[0], 5, -1).max(axis=(0, 2))


STATES = {
    "means by long series": dict(rho=(0.75, 1.0), p=(0.75, 1.0)),
    "means by logarithm": dict(rho=(0.3, 1.0), p=(0.4, 1.0)),
    "edge of the range": dict(rho=(0.08, 1.0), p=(0.8, 1.0)),
    "FP64 elements": dict(rho=(0.03, 1.0), p=(0.8, 1.2)),
    "at rest": dict(vel=0.0),
    "Mach 17": dict(vel=20.0),
    "low Mach": dict(vel=0.5, p=(1.0e5, 1.2e5)),
    "far-off scales": dict(rho=(0.8e-9, 1.2e-9), vel=1e8, p=(0.8e7, 1.2e7)),
}


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 7, 8])
@pytest.mark.parametrize("kind", list(STATES))
def test_time_derivative(orc, N, kind):
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(SIZE[N], min(N, 4), deform="sinprod", rotate_seed=400 + N)
    mu = 0.02 * (STATES[kind].get("rho", (1, 1))[1] * STATES[kind].get("vel", 0.5) if kind == "far-off scales" else 1.0)
    o, s = orc.Oracle(mesh, N, mu=mu), dg.Solver(mesh, N, mu=mu)
    U = random_state(mesh.n_elems, N, seed=500 + N, **STATES[kind])
    err = _err(s.time_derivative(_cuda(U)).cpu().numpy(), o.time_derivative(U))
    p = STATES[kind].get("p", (0.8, 1.2))
    assert (err < 1e-12 * max(1.0, 0.5 * (p[0] + p[1]) / (p[1] - p[0]))).all(), err


@pytest.mark.parametrize("N", [1, 3, 4, 7])
def test_blocks_of_both_kinds(orc, N):
    """Every third element outside the fixed-point range, R(U) and RK steps in
    place (each element is written by one of the two bodies)."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(SIZE[N], min(N, 4), deform="sinprod", rotate_seed=420 + N)
    o, s = orc.Oracle(mesh, N, mu=0.01), dg.Solver(mesh, N, mu=0.01)
    U = random_state(mesh.n_elems, N, seed=520 + N)
    W = random_state(mesh.n_elems, N, seed=521 + N, rho=(0.03, 1.0))
    U[::3] = W[::3]
    err = _err(s.time_derivative(_cuda(U)).cpu().numpy(), o.time_derivative(U))
    assert (err < 1e-12).all(), err
    Ud = _cuda(U)
    s.rk_step(Ud, torch.empty_like(Ud), 0.0, 2e-5, 10)
    ref = o.rk_steps(U, 0.0, 2e-5, 10)
    assert np.abs(Ud.cpu().numpy() - ref).max() / np.abs(ref).max() < 1e-10


@pytest.mark.parametrize("N,K", [(1, 2), (1, 5), (2, 3), (3, 2), (3, 5)])
@pytest.mark.parametrize("kind", list(STATES) + ["both"])
def test_latency_kernels(orc, N, K, kind):
    """The same on meshes of the latency kernels (three threads per node, one
    element per block): R(U), and three RK steps in place."""
    import paper_2605_28627_gb300 as dg
    kw = STATES["FP64 elements"] if kind == "both" else STATES[kind]
    mesh = box_mesh(K, min(N, 4), deform="sinprod", rotate_seed=460 + N)
    mu = 0.02 * (kw.get("rho", (1, 1))[1] * kw.get("vel", 0.5) if kind == "far-off scales" else 1.0)
    o, s = orc.Oracle(mesh, N, mu=mu), dg.Solver(mesh, N, mu=mu)
    U = random_state(mesh.n_elems, N, seed=560 + N, **kw)
    if kind == "both":
        U[1::2] = random_state(mesh.n_elems, N, seed=570 + N)[1::2]
    err = _err(s.time_derivative(_cuda(U)).cpu().numpy(), o.time_derivative(U))
    p = kw.get("p", (0.8, 1.2))
    assert (err < 1e-12 * max(1.0, 0.5 * (p[0] + p[1]) / (p[1] - p[0]))).all(), err
    dt = 2e-5 / (1e3 if kind in ("low Mach",) else 1e9 if kind == "far-off scales" else 1.0)
    Ud = _cuda(U)
    s.rk_step(Ud, torch.empty_like(Ud), 0.0, dt, 3)
    ref = o.rk_steps(U, 0.0, dt, 3)
    assert (np.abs(Ud.cpu().numpy() - ref).max(axis=(0, 2, 3, 4)) <= 1e-11 * np.abs(ref).max(axis=(0, 2, 3, 4))).all()


def test_non_finite_state_stays_local():
    """A NaN gives NaN in its element and leaves elements that do not touch it
    as they are, bit for bit; so does an infinity."""
    import paper_2605_28627_gb300 as dg
    N = 3
    mesh = box_mesh(7, 3, deform="sinprod", rotate_seed=430)
    s = dg.Solver(mesh, N, mu=0.01)
    U = _cuda(random_state(mesh.n_elems, N, seed=530))
    R = s.time_derivative(U)
    e = 100
    near = {e} | set(int(x) for x in mesh.face_nbr[e, :, 0])
    near |= {int(x) for a in list(near) for x in mesh.face_nbr[a, :, 0]}
    far = [x for x in range(mesh.n_elems) if x not in near]
    for bad in (float("nan"), float("inf")):
        V = U.clone()
        V[e, 4, 1, 2, 1] = bad
        Rv = s.time_derivative(V)
        assert not bool(torch.isfinite(Rv[e]).all())
        assert torch.equal(Rv[far], R[far])


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 7])
@pytest.mark.parametrize("kind,scale", [("means by long series", 1.0), ("means by logarithm", 1.0),
                                        ("edge of the range", 1e3), ("FP64 elements", 1.0), ("at rest", 1.0),
                                        ("Mach 17", 1e-3), ("low Mach", 1e4)])
def test_vjp(orc, N, kind, scale):
    """<(dR/dU)^T v, w> against <v, (dR/dU) w> of the oracle's tangent-linear,
    as in the adjoint's dot-product tests (bar 1e-11 of the terms' sum), with
    the components of v of different sizes (mass scale^2, momentum scale,
    energy 1) and every fifth element's v zero."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(2, min(N, 4), deform="sinprod", rotate_seed=440 + N)
    o, s = orc.Oracle(mesh, N, mu=0.02), dg.Solver(mesh, N, mu=0.02)
    U = random_state(mesh.n_elems, N, seed=540 + N, **STATES[kind])
    rng = np.random.default_rng(640 + N)
    w, v = rng.normal(size=U.shape), rng.normal(size=U.shape)
    v[:, 0] *= scale ** 2
    v[:, 1:4] *= scale
    v[::5] = 0.0
    _, Jw = o.time_derivative_tl(U, w, 0.0)
    JTv = s.time_derivative_vjp(_cuda(U), _cuda(v)).cpu().numpy()
    lhs, rhs = float((JTv * w).sum()), float((v * Jw).sum())
    assert abs(lhs - rhs) <= 1e-11 * float(np.abs(JTv * w).sum()), (lhs, rhs)


@pytest.mark.parametrize("N", [1, 2, 3, 4, 7, 8])
@pytest.mark.parametrize("scale", [1.0, 1e30])
def test_gauss_nodes(orc, N, scale):
    """The weak form on Gauss nodes in range, and with density and pressure
    scaled out of the fixed-point range (2^90), which all runs in FP64.  The
    pressure's mean is 10 times its variation (see the bar above)."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(SIZE[N], min(N, 4), deform="sinprod", rotate_seed=450 + N)
    o, s = orc.Oracle(mesh, N, mu=0.01 * scale, nodes=1), dg.Solver(mesh, N, mu=0.01 * scale, nodes=dg.NODES_LG)
    U = random_state(mesh.n_elems, N, seed=550 + N, rho=(0.95, 1.05), vel=0.2, p=(0.95, 1.05)) * scale
    err = _err(s.time_derivative(_cuda(U)).cpu().numpy(), o.time_derivative(U))
    assert (err < 1e-11).all(), err


def _stretched(K, N, sizes, seed):
    """Cartesian box of K^3 cells of the given sizes, frames turned at random."""
    mesh = box_mesh(K, 1, rotate_seed=seed)
    mesh.xgeo *= np.array(sizes)[None, :, None, None, None] * K / 2.0
    return mesh


def _axis_flow(s, mesh, N, L, ax, comp):
    """Density, velocity component comp and pressure vary along axis ax only; the
    same to the last bit at the nodes of different elements that coincide."""
    X = s.node_coords().cpu().numpy().reshape(mesh.n_elems, 3, N + 1, N + 1, N + 1)
    y = 2.0 * np.pi * np.round(X[:, ax] / L * 2.0 ** 36) * 2.0 ** -36
    rho, vel, p = 1.0 + 0.2 * np.sin(y), 0.5 + 0.3 * np.cos(y), 1.0 + 0.2 * np.sin(y + 1.0)
    U = np.zeros((mesh.n_elems, 5, N + 1, N + 1, N + 1))
    U[:, 0], U[:, 1 + comp], U[:, 4] = rho, rho * vel, p / 0.4 + 0.5 * rho * vel ** 2
    return U


# in fixed point with two directions shifted, and in FP64
CELLS = [(3.0, 1.2, 3.5), (3.0, 1.0, 24.0), (1.0, 10.0, 1000.0)]


LGL = [(1, 3, 0), (1, 13, 0), (2, 3, 0), (3, 3, 0), (3, 7, 0), (4, 3, 0), (5, 3, 0), (7, 2, 0), (8, 2, 0)]
LG = [(1, 3, 1), (3, 3, 1), (4, 2, 1), (6, 2, 1)]


@pytest.mark.parametrize("N,K,nodes,k", [c + (k,) for c in LGL + LG for k in (1, 2, 5, 20) if not c[2] or k <= 5])
def test_flow_along_stretched_cells(N, K, nodes, k):
    """Cells 2^k times as long along an axis as across it and an inviscid flow
    that varies along this axis: every term of the mass, energy and axis momentum
    equations is 2^-k times that on cubic cells, and so is its rounding, as there
    is no flow in the directions with the larger metric terms.  Bar 1e-13 of max
    |R|: the rounding of both evaluations.  On Gauss nodes 3e-13 and k up to 5: the
    face values are rounded sums, whose jumps at the long faces enter 2^k times."""
    import paper_2605_28627_gb300 as dg
    ax = (N + k) % 3
    R = []
    for long in (1.0, 2.0 ** k):
        mesh = _stretched(K, N, [long if a == ax else 1.0 for a in range(3)], 470 + N)
        s = dg.Solver(mesh, N, mu=0.0, nodes=nodes)
        if long == 1.0:
            U = _axis_flow(s, mesh, N, K, ax, ax)
        R.append(long * s.time_derivative(_cuda(U)).cpu().numpy()[:, [0, 1 + ax, 4]])
    d = np.abs(R[1] - R[0]).max(axis=(0, 2, 3, 4)) / np.abs(R[0]).max(axis=(0, 2, 3, 4))
    assert (d < (3e-13 if nodes else 1e-13)).all(), d


@pytest.mark.parametrize("N,K,nodes", LGL + [(9, 2, 0)] + LG)
@pytest.mark.parametrize("k", [1, 2, 5, 20])
def test_gradients_along_stretched_cells(orc, N, K, nodes, k):
    """The same cells with a transverse velocity that varies along the axis:
    the dissipation is a sum of squares of its lifted gradient, which the rounding
    in the other directions enters as a square.  Bar 2e-13."""
    import paper_2605_28627_gb300 as dg
    ax = (N + k) % 3
    mesh = _stretched(K, N, [2.0 ** k if a == ax else 1.0 for a in range(3)], 470 + N)
    o, s = orc.Oracle(mesh, N, mu=0.01, nodes=nodes), dg.Solver(mesh, N, mu=0.01, nodes=nodes)
    U = _axis_flow(s, mesh, N, K * 2.0 ** k, ax, (ax + 1) % 3)
    got, ref = s.integrals(_cuda(U))[6], o.integrals(U)[6]
    assert abs(got - ref) <= 2e-13 * ref, (got, ref)


@pytest.mark.parametrize("N,K,nodes", LGL + LG)
@pytest.mark.parametrize("cells", CELLS)
def test_stretched_cells(orc, N, K, nodes, cells):
    """A random state on stretched cells."""
    import paper_2605_28627_gb300 as dg
    mesh = _stretched(K, N, cells, 475 + N)
    kw = dict(mu=0.02, nodes=nodes)
    o, s = orc.Oracle(mesh, N, **kw), dg.Solver(mesh, N, **kw)
    mild = dict(rho=(0.95, 1.05), vel=0.2, p=(0.95, 1.05)) if nodes else {}   # admissible at the face points too
    U = random_state(mesh.n_elems, N, seed=580 + N, **mild)
    err = _err(s.time_derivative(_cuda(U)).cpu().numpy(), o.time_derivative(U))
    assert (err < 1e-11).all() if nodes else (err < 1e-12).all(), err


@pytest.mark.parametrize("N", [1, 3, 5, 7])
@pytest.mark.parametrize("cells", CELLS)
def test_vjp_on_stretched_cells(orc, N, cells):
    """As test_vjp."""
    import paper_2605_28627_gb300 as dg
    mesh = _stretched(2, N, cells, 480 + N)
    o, s = orc.Oracle(mesh, N, mu=0.02), dg.Solver(mesh, N, mu=0.02)
    U = random_state(mesh.n_elems, N, seed=590 + N)
    rng = np.random.default_rng(690 + N)
    w, v = rng.normal(size=U.shape), rng.normal(size=U.shape)
    _, Jw = o.time_derivative_tl(U, w, 0.0)
    JTv = s.time_derivative_vjp(_cuda(U), _cuda(v)).cpu().numpy()
    lhs, rhs = float((JTv * w).sum()), float((v * Jw).sum())
    assert abs(lhs - rhs) <= 1e-11 * float(np.abs(JTv * w).sum()), (lhs, rhs)


@pytest.mark.parametrize("N", [1, 3, 4])
def test_ensemble_with_stretched_member(N):
    """An FP64 ensemble of a cubic and a stretched mesh: the tile-table kernels
    against each member stepped alone."""
    import paper_2605_28627_gb300 as dg
    meshes = [box_mesh(4, 1), _stretched(3, N, CELLS[0], 490 + N)]
    solvers = [dg.Solver(m, N, mu=0.01) for m in meshes]
    U = [_cuda(random_state(m.n_elems, N, seed=600 + i)) for i, m in enumerate(meshes)]
    ref = [u.clone() for u in U]
    dt = 1e-3 / (N + 1) ** 2
    for s, u in zip(solvers, ref):
        s.rk_step(u, torch.empty_like(u), 0.0, dt, 2)
    dg.Ensemble(solvers).step(U, [torch.empty_like(u) for u in U], [0.0] * 2, [dt] * 2, 2)
    for a, b in zip(U, ref):
        assert float((a - b).abs().max()) <= 1e-13 * float(b.abs().max())


@pytest.mark.parametrize("N", [1, 3, 4, 7])
@pytest.mark.parametrize("k", [-100, -150, -400, 100])
def test_vjp_scales_with_the_cotangent(N, k):
    """The VJP is linear in the cotangent: scaled by a power of two it scales to
    the last bit where the exponents move with it, and to rounding (1e-12) where
    they leave the fixed-point range and FP64 takes over."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(2, min(N, 4), deform="sinprod", rotate_seed=600 + N)
    s = dg.Solver(mesh, N, mu=0.02)
    U = _cuda(random_state(mesh.n_elems, N, seed=610 + N))
    v = _cuda(np.random.default_rng(620 + N).normal(size=tuple(U.shape)))
    dm = [torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2)]
    ref = s.time_derivative_vjp(U, v, None, dm[0])
    got = s.time_derivative_vjp(U, v * 2.0 ** k, None, dm[1]) * 2.0 ** -k
    assert float((got - ref).abs().max()) <= (0.0 if k < 0 and k > -180 else 1e-12) * float(ref.abs().max())
    assert abs(float(dm[1]) * 2.0 ** -k - float(dm[0])) <= 1e-10 * abs(float(dm[0]))


@pytest.mark.parametrize("N", [1, 3, 5])
def test_vjp_at_low_speed(orc, N):
    """Velocities of 1e-22 of the sound speed and a cotangent of the mass equation
    alone, equal at every node of an element face's both sides: the adjoint of the
    density is proportional to the velocity."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(2, 1)
    o, s = orc.Oracle(mesh, N), dg.Solver(mesh, N)
    U = random_state(mesh.n_elems, N, seed=630 + N, rho=(1.0, 1.0), p=(1.0, 1.0), vel=1e-22)
    X = s.node_coords().cpu().numpy().reshape(mesh.n_elems, 3, N + 1, N + 1, N + 1)
    v, w = np.zeros_like(U), np.zeros_like(U)
    v[:, 0] = np.sin(np.pi * np.round(X[:, 0] * 2.0 ** 40) * 2.0 ** -40)
    w[:, 0] = np.random.default_rng(640 + N).normal(size=w[:, 0].shape)
    w[:, 0, [0, -1]] = w[:, 0, :, [0, -1]] = w[:, 0, :, :, [0, -1]] = 0.0   # interior nodes (none at N = 1)
    JTv = s.time_derivative_vjp(_cuda(U), _cuda(v)).cpu().numpy()
    _, Jw = o.time_derivative_tl(U, w, 0.0)
    lhs, rhs = float((JTv * w).sum()), float((v * Jw).sum())
    assert abs(lhs - rhs) <= 1e-11 * float(np.abs(JTv * w).sum()), (lhs, rhs)


@pytest.mark.parametrize("N,K,nodes", [(1, 3, 0), (3, 3, 0), (3, 7, 0), (5, 3, 0), (7, 2, 0), (1, 3, 1), (3, 3, 1), (6, 2, 1)])
@pytest.mark.parametrize("vel", [1e-12, 1e-22, 1e-40, 1e-80])
def test_low_speed(orc, N, K, nodes, vel):
    """Uniform density and pressure, velocities far below the sound speed: mass
    and energy of R(U) and the dissipation follow the velocity down to any size."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(K, min(N, 4), deform="sinprod", rotate_seed=650 + N)
    U = random_state(mesh.n_elems, N, seed=660 + N, rho=(1.0, 1.0), p=(1.0, 1.0), vel=vel)
    U[:, 4] = 2.5   # the kinetic energy is below the rounding of p / 0.4
    if not nodes:
        # inviscid, as the conduction of the temperature's rounding is larger; on Gauss
        # nodes the face values of density and energy are rounded sums, whose jumps
        # LLF multiplies by the sound speed
        o, s = orc.Oracle(mesh, N), dg.Solver(mesh, N)
        err = _err(s.time_derivative(_cuda(U)).cpu().numpy(), o.time_derivative(U))
        assert (err[[0, 4]] < 1e-12).all(), err
    kw = dict(mu=0.01, nodes=nodes)
    got, ref = dg.Solver(mesh, N, **kw).integrals(_cuda(U))[6], orc.Oracle(mesh, N, **kw).integrals(U)[6]
    assert abs(got - ref) <= 1e-12 * ref, (got, ref)


@pytest.mark.parametrize("N,K,nodes", [(1, 3, 0), (3, 3, 0), (3, 7, 0), (5, 3, 0), (1, 3, 1), (3, 3, 1), (6, 2, 1)])
@pytest.mark.parametrize("k", [-120, -240])
def test_cold_gas_at_rest(orc, N, K, nodes, k):
    """Pressure and temperature scaled by 2^k at unit density, no flow: the energy
    equation is heat conduction alone, in proportion."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(K, 1, rotate_seed=670 + N)
    kw = dict(mu=1.0, nodes=nodes)
    o, s = orc.Oracle(mesh, N, **kw), dg.Solver(mesh, N, **kw)
    U = random_state(mesh.n_elems, N, seed=680 + N, rho=(1.0, 1.0), p=(0.95, 1.05), vel=0.0)
    U[:, 4] *= 2.0 ** k
    R, ref = s.time_derivative(_cuda(U)).cpu().numpy()[:, 4], o.time_derivative(U)[:, 4]
    assert np.abs(R - ref).max() < (1e-11 if nodes else 1e-12) * np.abs(ref).max()


@pytest.mark.parametrize("N", [1, 3, 6])
@pytest.mark.parametrize("k", [-100, -150, -250])
def test_gauss_nodes_scaled_down(N, k):
    """Density, pressure and viscosity scaled by 2^k: R(U) scales to the last bit
    where the exponents move with it, and to rounding in FP64."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(3, min(N, 4), deform="sinprod", rotate_seed=690 + N)
    U = _cuda(random_state(mesh.n_elems, N, seed=700 + N, rho=(0.95, 1.05), vel=0.2, p=(0.95, 1.05)))
    R = [dg.Solver(mesh, N, mu=0.01 * 2.0 ** x, nodes=dg.NODES_LG).time_derivative(U * 2.0 ** x) * 2.0 ** -x for x in (0, k)]
    assert float((R[1] - R[0]).abs().max()) <= (0.0 if k > -180 else 1e-12) * float(R[0].abs().max())


@pytest.mark.parametrize("N", [1, 3, 6])
def test_gas_without_pressure(orc, N):
    """No pressure, no flow: the sound speed is 0 and so is R(U) on Gauss nodes
    (the split form on LGL nodes divides by the pressure)."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(3, min(N, 4), deform="sinprod", rotate_seed=710 + N)
    o, s = orc.Oracle(mesh, N, mu=0.01, nodes=1), dg.Solver(mesh, N, mu=0.01, nodes=dg.NODES_LG)
    U = random_state(mesh.n_elems, N, seed=720 + N, rho=(0.95, 1.05), vel=0.0)
    U[:, 4] = 0.0
    assert not o.time_derivative(U).any()
    assert not bool(s.time_derivative(_cuda(U)).any())


def test_sound_speed_in_the_lax_friedrichs_flux():
    """Densities that jump at the faces, no flow, uniform pressure: R of the mass is
    sound speed times jump over the face weight.  One plane of faces of cubic cells,
    N = 1 (w_0 = 1, J = 1/8): bar 6 ulp, the roundings of the terms around sqrt."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(8, 1)
    s = dg.Solver(mesh, 1, mu=0.0)
    rng = np.random.default_rng(730)
    r = np.exp(rng.uniform(np.log(0.25), np.log(4.0), mesh.n_elems // 64))       # per plane of constant x
    plane = np.arange(mesh.n_elems) % 8
    rho = np.empty((mesh.n_elems, 2, 2, 2))
    rho[:] = r[plane][:, None, None, None]
    p = 2.0 ** rng.integers(-8, 8) * 1.3
    U = np.zeros((mesh.n_elems, 5, 2, 2, 2))
    U[:, 0], U[:, 4] = rho, p / 0.4
    R = s.time_derivative(_cuda(U)).cpu().numpy()[:, 0]
    L = np.longdouble
    gm1 = L(1.4 - 1.0)
    c = np.sqrt(L(1.4) * (gm1 * L(U[0, 4, 0, 0, 0])) / r.astype(L))
    left = np.maximum(c, np.roll(c, 1)) * (np.roll(r, 1) - r)                    # at the faces of smaller x
    scale = 0.5 * 8.0                                                            # lambda/2 and sJ / (J w_0)
    assert np.abs(R[:, :, :, 0] / (scale * left[plane])[:, None, None] - 1).max() < 6 * 2.0 ** -52


@pytest.mark.parametrize("N,K,nodes", [(3, 40, 0), (2, 44, 1)])
def test_mesh_that_leaves_no_room_for_fixed_point(N, K, nodes):
    """With the device memory filled so that the fixed-point copy of the metric
    terms (80 B per node) does not fit, a context runs in FP64 instead of failing."""
    import paper_2605_28627_gb300 as dg
    mesh = box_mesh(K, 1)
    n = mesh.n_elems * (N + 1) ** 3
    U = _cuda(random_state(mesh.n_elems, N, seed=740, rho=(0.95, 1.05), vel=0.2, p=(0.95, 1.05)))
    out, G = torch.empty_like(U), torch.empty_like(U)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    s = dg.Solver(mesh, N, mu=0.01, nodes=nodes)
    used = free0 - torch.cuda.mem_get_info()[0]
    ref = s.time_derivative(U).clone()
    s.close()
    torch.cuda.synchronize()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - used + 40 * n, dtype=torch.uint8, device="cuda")
    s = dg.Solver(mesh, N, mu=0.01, nodes=nodes)
    left = torch.cuda.mem_get_info()[0]
    del filler
    torch.cuda.empty_cache()
    assert left > 20 * n          # of 40 B per node, less the allocator's granularity
    s.time_derivative(U, out)
    assert float((out - ref).abs().max()) <= 1e-12 * float(ref.abs().max())
    s.rk_step(U, G, 0.0, 1e-6, 1)
    assert bool(torch.isfinite(s.time_derivative_vjp(U, ref, out)).all())
