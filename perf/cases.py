"""The calls that a user of the framework makes, as cases to be timed and compared.

Every case goes through the public Python entry points (``Solver``,
``Ensemble``).  The meshes are periodic boxes of hexahedra, Cartesian or
curved with every element's frame turned at random, the flows a Taylor-Green
vortex or a density wave with seeded smooth disturbances: what the paper's
verification and performance runs compute.

``exact`` evaluates the same scheme in plain torch, in 64 bits, on arrays
[E, ..., k, j, i]; it uses none of the framework's code.
"""
import math

import numpy as np
import torch

DEV = "cuda"
LSERK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
           -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
LSERK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
           1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
           2277821191437.0 / 14882151754819.0)
LSERK_C = (0.0, 1432997174477.0 / 9575080441755.0, 2526269341429.0 / 6820363962896.0,
           2006345519317.0 / 3224310063776.0, 2802321613138.0 / 2924317926251.0)
GAMMA, RGAS, PR, MMS_AMP = 1.4, 1.0, 0.72, 0.1


def _case(name, do, dims, N, flow="tgv", curved=False, fp32=False, gauss=False, flux="llf", suth=False, mach=0.1,
          re=1600.0, steps=1):
    c = {"do": do, "kx": dims[0], "ky": dims[1], "kz": dims[2], "N": N, "flow": flow, "curved": curved, "fp32": fp32,
         "gauss": gauss, "flux": flux, "suth": suth, "mach": mach, "re": re, "steps": steps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest verification run: 4^3 elements, ten steps per call
        _case("tgv4_n3_10steps", "step", (4, 4, 4), 3, steps=10),
        # one R(U) on a small odd mesh with turned frames, as an own time loop calls it
        _case("rhs_5x6x7_n2_ec", "rhs", (5, 6, 7), 2, curved=True, flux="ec", mach=0.3),
        # the convergence study's finest run: curved, unstructured, manufactured source
        _case("mms16_n7", "step", (16, 16, 16), 7, flow="mms", curved=True),
        # a compressible run on a ragged mesh: Roe faces, Sutherland's law, larger density ratios
        _case("comp_15x13x11_n4_roe", "step", (15, 13, 11), 4, curved=True, flux="roe", suth=True, mach=0.8, re=400.0),
        # a Cartesian turbulence run of ordinary size and degree
        _case("tgv20_n5", "step", (20, 20, 20), 5, mach=0.2, re=800.0),
        # the same study with the FP32 operator, and the largest run with it
        _case("mms16_n7_fp32", "step", (16, 16, 16), 7, flow="mms", curved=True, fp32=True),
        _case("tgv32_n7_fp32", "step", (32, 32, 32), 7, fp32=True),
        # Legendre-Gauss nodes (the node set of the paper's PID runs), both operators
        _case("tgv32_n3_gauss", "step", (32, 32, 32), 3, gauss=True),
        _case("tgv16_n6_gauss_fp32", "step", (16, 16, 16), 6, gauss=True, curved=True, fp32=True, mach=0.3),
        # the adjoint: one vector-Jacobian product of R(U), and one step backwards on Gauss nodes
        _case("vjp16_n5", "vjp", (16, 16, 16), 5, mach=0.2, re=800.0),
        _case("adjstep12_n3_gauss", "adjstep", (12, 12, 12), 3, gauss=True, curved=True, mach=0.2, re=800.0),
        # uneven small runs advanced together
        _case("ensemble8_fp32", "ensemble", (5, 5, 5), 7, fp32=True, mach=0.3, re=1000.0, steps=2),
    ]


def draw(rng):
    do = rng.choice(["step", "step", "step", "rhs", "vjp", "adjstep"])
    N = rng.randint(1, 9)
    # nodes: log-uniform over the listed range of the kind
    top = 2.2e6 if do in ("step", "rhs") else 8e5
    nodes = math.exp(rng.uniform(math.log(4e3), math.log(top)))
    k = max(2.0, (nodes / (N + 1) ** 3) ** (1.0 / 3.0))
    dims = [max(2, int(round(k * rng.uniform(0.75, 1.15)))) for _ in range(3)]
    fp32 = do in ("step", "rhs") and rng.random() < 0.35
    return _case(None, do, dims, N, flow=rng.choice(["tgv", "tgv", "mms"]), curved=rng.random() < 0.6, fp32=fp32,
                 gauss=rng.random() < 0.3, flux=rng.choice(["llf", "llf", "ec", "roe"]), suth=rng.random() < 0.2,
                 mach=round(rng.uniform(0.1, 0.9), 2), re=round(rng.uniform(400.0, 1600.0), 1),
                 steps=rng.choice([1, 2]) if do == "step" else 1)


# ---------------------------------------------------------------- meshes
def _rotations():
    out = []
    for p in ((0, 1, 2), (1, 2, 0), (2, 0, 1), (0, 2, 1), (2, 1, 0), (1, 0, 2)):
        for s in range(8):
            sg = [1 - 2 * ((s >> a) & 1) for a in range(3)]
            even = p in ((0, 1, 2), (1, 2, 0), (2, 0, 1))
            if sg[0] * sg[1] * sg[2] == (1 if even else -1):
                out.append((p, sg))
    return out


class Mesh:
    """Periodic box of hexahedra: xgeo [E, 3, m, m, m] (k, j, i) and face_nbr [E, 6, 3]."""

    def __init__(self, dims, ngeo, lo, hi, curved, seed):
        K = np.array(dims)
        E = int(K.prod())
        e = np.arange(E)
        cell = np.stack([e % K[0], (e // K[0]) % K[1], e // (K[0] * K[1])], 1)
        m = ngeo + 1
        lat = np.empty((E, 3, m, m, m), dtype=np.int64)
        t = np.arange(m)
        lat[:, 0] = cell[:, 0, None, None, None] * ngeo + t[None, None, None, :]
        lat[:, 1] = cell[:, 1, None, None, None] * ngeo + t[None, None, :, None]
        lat[:, 2] = cell[:, 2, None, None, None] * ngeo + t[None, :, None, None]
        L = (K * ngeo)[None, :, None, None, None]
        x = lo + (hi - lo) * (lat / L)
        if curved:   # x_i += 0.1 prod_j sin(pi s_j), s in [-1, 1]; zero on the box faces
            s = np.sin(np.pi * (-1.0 + 2.0 * lat / L))
            s[(lat == 0) | (lat == L)] = 0.0
            x = x + 0.05 * (hi - lo) * s.prod(1, keepdims=True)
        g = np.tile(np.arange(3), (E, 1))     # global axis of each local axis
        sg = np.ones((E, 3), dtype=np.int64)  # and its sense
        if curved:
            rots = _rotations()
            pick = np.random.default_rng(seed).integers(0, 24, E)
            for r, (p, s) in enumerate(rots):
                sel = np.nonzero(pick == r)[0]
                if not len(sel):
                    continue
                g[sel], sg[sel] = p, s
                y = x[sel]
                # array axes of x: 2, 3, 4 = global z, y, x; of the result: local 2, 1, 0
                y = y.transpose(0, 1, 4 - p[2], 4 - p[1], 4 - p[0])
                for a in range(3):
                    if s[a] < 0:
                        y = np.flip(y, 4 - a)
                x[sel] = y
        self.xgeo = np.ascontiguousarray(x)
        nbr = np.empty((E, 6, 3), dtype=np.int32)
        stride = np.array([1, K[0], K[0] * K[1]])
        inv = np.argsort(g, 1)                # local axis of each global axis
        for f in range(6):
            d, s = divmod(f, 2)
            G = g[:, d]
            sense = sg[e, d] * (2 * s - 1)
            c2 = cell.copy()
            c2[e, G] = (c2[e, G] + sense) % K[G]
            e2 = (c2 * stride).sum(1)
            d2 = inv[e2, G]
            f2 = 2 * d2 + np.where(sg[e2, d2] * -sense > 0, 1, 0)
            tan = [a for a in range(3) if a != d]
            b0 = np.where(d2 == 0, 1, 0)
            b1 = np.where(d2 == 2, 1, 2)
            g0, g1 = g[e2, b0], g[e2, b1]
            swap = g0 != g[:, tan[0]]
            r0 = sg[e2, b0] != sg[e, inv[e, g0]]
            r1 = sg[e2, b1] != sg[e, inv[e, g1]]
            nbr[:, f, 0], nbr[:, f, 1] = e2, f2
            nbr[:, f, 2] = swap * 1 + r0 * 2 + r1 * 4
        self.face_nbr = nbr


# ---------------------------------------------------------------- bases
def _legendre(N, x):
    return np.polynomial.legendre.legval(x, [0.0] * N + [1.0])


def _lgl(N):
    """Legendre-Gauss-Lobatto nodes and weights, Newton's method on (1 - x^2) P_N'."""
    x = -np.cos(np.pi * np.arange(N + 1) / N)
    for _ in range(60):
        p, p1 = _legendre(N, x), _legendre(N - 1, x)
        x = x - (x * p - p1) / ((N + 1) * p)
    x = (x - x[::-1]) / 2
    x[0], x[-1] = -1.0, 1.0
    return x, 2.0 / (N * (N + 1) * _legendre(N, x) ** 2)


def _lagrange(x, y):
    """Matrix [len(y), len(x)] of the Lagrange polynomials on x at the points y."""
    V = np.ones((len(y), len(x)))
    for a in range(len(x)):
        for b in range(len(x)):
            if a != b:
                V[:, a] *= (y - x[b]) / (x[a] - x[b])
    return V


def _diff(x):
    n = len(x)
    c = np.array([np.prod([x[i] - x[j] for j in range(n) if j != i]) for i in range(n)])
    D = np.zeros((n, n))
    for i in range(n):
        for j in range(n):
            if i != j:
                D[i, j] = c[i] / (c[j] * (x[i] - x[j]))
        D[i, i] = -D[i].sum()
    return D


def _nodes(N, gauss):
    return np.polynomial.legendre.leggauss(N + 1) if gauss else _lgl(N)


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _ap(M, f, d):
    """M applied along reference direction d of f [..., k, j, i]."""
    return torch.movedim(torch.movedim(f, -1 - d, -1) @ M.T, -1, -1 - d)


def _coords(mesh, N, gauss):
    m = mesh.xgeo.shape[-1]
    x = _t(mesh.xgeo)
    V = _t(_lagrange(np.linspace(-1.0, 1.0, m), _lgl(N)[0]))
    for d in range(3):
        x = _ap(V, x, d)
    if gauss:
        V = _t(_lagrange(_lgl(N)[0], _nodes(N, True)[0]))
        for d in range(3):
            x = _ap(V, x, d)
    return x


# ---------------------------------------------------------------- inputs
def _box(c):
    return (-1.0, 1.0) if c["flow"] == "mms" else (0.0, 2.0 * math.pi)


def _mesh(c, dims=None, N=None):
    lo, hi = _box(c)
    n = N or c["N"]
    return Mesh(dims or (c["kx"], c["ky"], c["kz"]), min(n, 4) if c["curved"] else 1, lo, hi, c["curved"], 20260528)


def _flow(c, x, seed, mach=None):
    """Conserved state at the points x [E, 3, k, j, i]: the flow with seeded smooth disturbances."""
    lo, hi = _box(c)
    r = np.random.default_rng(seed)
    k0 = 2.0 * math.pi / (hi - lo)

    def modes(amp):
        s = 0.0
        for _ in range(4):
            k, ph = r.integers(-2, 3, 3), r.uniform(0.0, 2.0 * math.pi)
            s = s + amp * r.uniform(0.3, 1.0) * torch.sin(
                k0 * (int(k[0]) * x[:, 0] + int(k[1]) * x[:, 1] + int(k[2]) * x[:, 2]) + ph)
        return s

    mach = mach or c["mach"]
    if c["flow"] == "mms":
        rho = 2.0 + MMS_AMP * torch.sin(math.pi * (x[:, 0] + x[:, 1] + x[:, 2])) + modes(0.005)
        vel = [1.0 + modes(0.005) for _ in range(3)]
        p = 1.0 + modes(0.005)
    else:
        p0 = 1.0 / (GAMMA * mach ** 2)
        sh = [float(v) for v in r.uniform(0.0, 2.0 * math.pi, 3)]
        X, Y, Z = x[:, 0] + sh[0], x[:, 1] + sh[1], x[:, 2] + sh[2]
        vel = [torch.sin(X) * torch.cos(Y) * torch.cos(Z) + modes(0.02),
               -torch.cos(X) * torch.sin(Y) * torch.cos(Z) + modes(0.02), modes(0.02)]
        p = p0 + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
        p = p * (1.0 + modes(0.1 * mach ** 2))
        rho = (1.0 + modes(0.25 * mach ** 2)) * (p / p0)
    e = p / (GAMMA - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho, *[rho * v for v in vel], e], 1).contiguous()


def _mu(c):
    return 0.001 if c["flow"] == "mms" else 1.0 / c["re"]


def _tref(c):
    return 1.0 / (GAMMA * c["mach"] ** 2) if c["flow"] == "tgv" else 0.5


def _dt(c, N=None, dims=None, mach=None):
    """A stable step, about half of the CFL bound of the largest signal speed."""
    lo, hi = _box(c)
    N = N or c["N"]
    K = max(dims or (c["kx"], c["ky"], c["kz"]))
    h = (hi - lo) / K * (0.6 if c["curved"] else 1.0)
    lam = 3.0 + 1.0 / (mach or c["mach"]) if c["flow"] == "tgv" else 6.0
    return (0.2 if c["gauss"] else 0.5) * h / ((2 * N + 1) * lam)


def _solver(c, mesh, N=None, **more):
    import paper_2605_28627_gb300 as dg
    kw = dict(gamma=GAMMA, R=RGAS, Pr=PR, mu=_mu(c), precision=dg.FP32OP if c["fp32"] else dg.FP64,
              surf_flux={"llf": dg.FLUX_LLF, "ec": dg.FLUX_EC, "roe": dg.FLUX_ROE}[c["flux"]],
              nodes=dg.NODES_LG if c["gauss"] else dg.NODES_LGL)
    if c["flow"] == "mms" and c["do"] in ("step", "rhs"):
        kw.update(source=dg.SOURCE_MMS, mms_amp=MMS_AMP)
    if c["flow"] == "tgv" and c["fp32"]:
        kw.update(p_ref=1.0 / (GAMMA * c["mach"] ** 2))
    if c["suth"]:
        kw.update(visc_law=dg.VISC_SUTHERLAND, T_ref=_tref(c), S_suth=0.4 * _tref(c))
    kw.update(more)
    return dg.Solver(mesh, N or c["N"], **kw)


def _members(c, seed):
    r = np.random.default_rng(20260529)
    out = []
    for i in range(8):
        K, N = int(r.integers(2, 7)), int(r.integers(3, 8))
        out.append((K, N, float(r.uniform(0.1, 0.5)), float(r.uniform(400.0, 1600.0)), seed * 8 + i))
    return out


def _lambda(U, seed):
    g = torch.Generator(device=DEV).manual_seed(seed + 77)
    return torch.randn(U.shape, dtype=torch.float64, device=DEV, generator=g)


def prepare(case, seed):
    c = case
    if c["do"] == "ensemble":
        import paper_2605_28627_gb300 as dg
        s, U, dt = [], [], []
        for K, N, ma, re, sd in _members(c, seed):
            m = _mesh(c, (K, K, K), N)
            s.append(_solver(c, m, N, mu=1.0 / re, p_ref=0.0))
            U.append(_flow(c, _coords(m, N, False), sd, ma))
            dt.append(_dt(c, N, (K, K, K), ma))
        return {"c": c, "s": s, "e": dg.Ensemble(s), "U": U, "G": [torch.zeros_like(u) for u in U], "t": [0.0] * 8,
                "dt": dt}
    mesh = _mesh(c)
    U = _flow(c, _coords(mesh, c["N"], c["gauss"]), seed)
    st = {"c": c, "s": _solver(c, mesh), "U": U, "t": 0.0, "dt": _dt(c)}
    if c["do"] == "step":
        st["G"] = torch.zeros_like(U)
    else:
        st["out"] = torch.empty_like(U)
    if c["do"] in ("vjp", "adjstep"):
        st["lam"] = _lambda(U, seed)
        st["dmu"] = torch.zeros(1, dtype=torch.float64, device=DEV)
    return st


def run(state):
    c, s = state["c"], state["s"]
    if c["do"] == "ensemble":
        state["e"].step(state["U"], state["G"], state["t"], state["dt"], c["steps"])
        state["t"] = [t + c["steps"] * d for t, d in zip(state["t"], state["dt"])]
        return state["U"]
    if c["do"] == "step":
        s.rk_step(state["U"], state["G"], state["t"], state["dt"], c["steps"])
        state["t"] += c["steps"] * state["dt"]
        return state["U"]
    if c["do"] == "rhs":
        return s.time_derivative(state["U"], state["out"], state["t"])
    state["dmu"].zero_()
    if c["do"] == "vjp":
        s.time_derivative_vjp(state["U"], state["lam"], state["out"], state["dmu"])
    else:
        s.adjoint_step(state["U"], state["lam"], state["out"], state["dmu"], 0.0, state["dt"])
    return [state["out"], state["dmu"]]


# ---------------------------------------------------------------- work and tolerance
def _flops(N, gauss):
    """Operations per node of one R(U), counted from the formulas (an FMA is two, a division one): lifting, face
    flux, volume integral with each pair of the split form taken once (Gauss nodes: the weak form's line sums)."""
    n = N + 1
    lift = 14 + 132.0 / n + 24 * n + 72
    face = 600.0 / n
    vol = 91 + 24 * n + 150.0 / n + (60 + 24 * n if gauss else 145.5 * N + 30)
    return lift + face + vol + (60.0 * 17 / n if gauss else 0.0)


def work(case):
    c = case
    b = 4 if c["fp32"] else 8
    # per evaluation and node: state in, metric terms and 1/J, result out
    rhs = 40 + 10 * b + 40
    if c["do"] == "ensemble":
        nodes = [(K ** 3 * (N + 1) ** 3, N) for K, N, _, _, _ in _members(c, 0)]
        return {"bytes": sum(p for p, _ in nodes) * 5.0 * c["steps"] * (160 + 10 * b),
                "flops": sum(p * _flops(N, False) for p, N in nodes) * 5.0 * c["steps"]}
    nodes = float(c["kx"] * c["ky"] * c["kz"] * (c["N"] + 1) ** 3)
    f = nodes * _flops(c["N"], c["gauss"])
    if c["do"] == "rhs":
        return {"bytes": nodes * rhs, "flops": f}
    if c["do"] == "step":   # five stages, each reading and writing state and register
        return {"bytes": nodes * 5.0 * c["steps"] * (160 + 10 * b), "flops": 5.0 * c["steps"] * f}
    # a vector-Jacobian product: about twice the operations of the function, after its gradients
    if c["do"] == "vjp":
        return {"bytes": nodes * (rhs + 40), "flops": 3.0 * f}
    return {"bytes": nodes * 5.0 * (rhs + 160 + 40), "flops": 5.0 * 4.0 * f}


def tolerance(case):
    """About four times what the path differs by from ``exact`` (measured over listed and drawn cases)."""
    c = case
    if c["fp32"]:
        # the state is 64 bits wide and takes dt R(U) with R in 32 bits; R(U) itself shows 32-bit sums
        return {"rel": 2e-4, "max": 2e-2} if c["do"] == "rhs" else {"rel": 4e-7, "max": 4e-5}
    if c["do"] == "step":   # rounding of dt R(U), which grows with the degree as the metric terms' does
        return {"rel": 4e-14, "max": 4e-12} if c["N"] <= 7 else {"rel": 4e-13, "max": 4e-11}
    # R(U) and products with its Jacobian are differences of terms that are larger by a factor of about 1e3,
    # on metric terms that carry rounding amplified by the differentiation; d/dmu is one sum with cancellation
    return {"rel": 1e-10, "max": 1e-8} if c["do"] == "rhs" else {"rel": 4e-10, "max": 4e-8}


# ---------------------------------------------------------------- the scheme in plain torch, 64 bits
class Plain:
    def __init__(self, c, mesh, N):
        self.c, self.N, self.n, self.gauss = c, N, N + 1, c["gauss"]
        xl, wl = _lgl(N)
        Dl = _t(_diff(xl))
        x = _t(mesh.xgeo)
        x = x - x[:, :, :1, :1, :1]
        V = _t(_lagrange(np.linspace(-1.0, 1.0, mesh.xgeo.shape[-1]), xl))
        for d in range(3):
            x = _ap(V, x, d)
        dx = torch.stack([_ap(Dl, x, d) for d in range(3)], 2)      # [E, c, d, ...]
        Ja = torch.empty_like(dx)                                   # [E, d, c, ...]
        for a in range(3):                                          # curl form: -curl(x_l grad x_m)
            m, l = (a + 1) % 3, (a + 2) % 3
            v = [x[:, l] * dx[:, m, r] for r in range(3)]
            Ja[:, 0, a] = -(_ap(Dl, v[2], 1) - _ap(Dl, v[1], 2))
            Ja[:, 1, a] = -(_ap(Dl, v[0], 2) - _ap(Dl, v[2], 0))
            Ja[:, 2, a] = -(_ap(Dl, v[1], 0) - _ap(Dl, v[0], 1))
        if self.gauss:
            xg, wg = _nodes(N, True)
            G = _t(_lagrange(xl, xg))
            fJa = [self._tangent(G, self._end(Ja[:, f // 2], f), f) for f in range(6)]
            for d in range(3):
                Ja, dx = _ap(G, Ja, d), _ap(G, dx, d)
            self.D, self.w = _t(_diff(xg)), _t(wg)
            self.lend = [_t(_lagrange(xg, np.array([e]))[0]) for e in (-1.0, 1.0)]
        else:
            fJa = [self._end(Ja[:, f // 2], f) for f in range(6)]
            self.D, self.w = Dl, _t(wl)
        J = (dx[:, 0, 0] * (dx[:, 1, 1] * dx[:, 2, 2] - dx[:, 1, 2] * dx[:, 2, 1])
             - dx[:, 0, 1] * (dx[:, 1, 0] * dx[:, 2, 2] - dx[:, 1, 2] * dx[:, 2, 0])
             + dx[:, 0, 2] * (dx[:, 1, 0] * dx[:, 2, 1] - dx[:, 1, 1] * dx[:, 2, 0]))
        self.Ja, self.J = Ja, J
        # outward n sJ of every face point [E, 6, 3, q, p]
        self.ns = torch.stack([(2 * (f % 2) - 1) * fJa[f] for f in range(6)], 1)
        self.sJ = self.ns.square().sum(2).sqrt()
        self.nv = self.ns / self.sJ[:, :, None]
        # the neighbour's face point: flat index over [E, 6, q, p]
        n = self.n
        nb = torch.as_tensor(mesh.face_nbr.astype(np.int64), device=DEV)
        p = torch.arange(n, device=DEV)[None, None, None, :]
        q = torch.arange(n, device=DEV)[None, None, :, None]
        e2, f2, fl = (nb[..., i, None, None] for i in range(3))
        a, b = torch.where((fl & 1) > 0, q, p), torch.where((fl & 1) > 0, p, q)
        p2, q2 = torch.where((fl & 2) > 0, n - 1 - a, a), torch.where((fl & 4) > 0, n - 1 - b, b)
        self.nbr = (((e2 * 6 + f2) * n + q2) * n + p2).reshape(-1)
        if c["flow"] == "mms" and c["do"] in ("step", "rhs"):
            self.ph = math.pi * _coords(mesh, N, self.gauss).sum(1)

    @staticmethod
    def _end(f, face):
        return torch.select(f, f.dim() - 1 - face // 2, -1 if face % 2 else 0)

    @staticmethod
    def _tangent(G, f, face):   # along both directions of a face field [..., q, p]
        return _ap(G, _ap(G, f, 0), 1)

    def faces(self, f):
        """Face values [E, 6, v, q, p] of f [E, v, k, j, i]."""
        if not self.gauss:
            return torch.stack([self._end(f, a) for a in range(6)], 1)
        return torch.stack([torch.movedim(f, -1 - a // 2, -1) @ self.lend[a % 2] for a in range(6)], 1)

    def other(self, f):
        v = f.shape[2]
        return torch.movedim(f, 2, 0).reshape(v, -1)[:, self.nbr].reshape(v, f.shape[0], 6, self.n, self.n).movedim(0, 2)

    def visc(self, T, mu):
        if not self.c["suth"]:
            return mu
        T0 = _tref(self.c)
        return mu * (T / T0) ** 1.5 * (1.4 * T0) / (T + 0.4 * T0)

    def fvisc(self, g, v, mu, nn):
        """Viscous flux . n: momentum and energy; g[phi][l], n of 3."""
        div = (2.0 / 3.0) * (g[0][0] + g[1][1] + g[2][2])
        f = []
        for a in range(3):
            s = 0.0
            for l in range(3):
                tau = g[a][l] + g[l][a]
                s = s + (tau - div if a == l else tau) * nn[l]
            f.append(mu * s)
        kap = GAMMA * RGAS / (GAMMA - 1.0) / PR
        e = f[0] * v[0] + f[1] * v[1] + f[2] * v[2] + mu * kap * (g[3][0] * nn[0] + g[3][1] * nn[1] + g[3][2] * nn[2])
        return f + [e]

    @staticmethod
    def logmean(a, b):
        """(a - b) / ln(a / b), through the series near a = b."""
        z = (a - b) / (a + b)
        u = z * z
        near = u < 1e-4
        ser = 1.0 + u * (1.0 / 3.0 + u * (1.0 / 5.0 + u * (1.0 / 7.0 + u / 9.0)))
        zz = torch.where(near, torch.full_like(z, 0.5), z)
        return (a + b) / (2.0 * torch.where(near, ser, torch.atanh(zz) / zz))

    def pair(self, A, B, nn):
        """Chandrashekar's two-point flux of the primitives A, B = (rho, v, p) in direction nn."""
        ba, bb = 0.5 * A[0] / A[2], 0.5 * B[0] / B[2]
        v = [0.5 * (x + y) for x, y in zip(A[1], B[1])]
        ph = 0.5 * (A[0] + B[0]) / (ba + bb)
        ke = 0.25 * sum(x * x + y * y for x, y in zip(A[1], B[1]))
        fr = self.logmean(A[0], B[0]) * (v[0] * nn[0] + v[1] * nn[1] + v[2] * nn[2])
        m = [fr * v[a] + ph * nn[a] for a in range(3)]
        e = fr * (0.5 / ((GAMMA - 1.0) * self.logmean(ba, bb)) - ke) + sum(v[a] * m[a] for a in range(3))
        return [fr, *m, e]

    @staticmethod
    def euler(q, v, p, nn):
        un = v[0] * nn[0] + v[1] * nn[1] + v[2] * nn[2]
        return [q[0] * un, *[q[1 + a] * un + p * nn[a] for a in range(3)], (q[4] + p) * un]

    def riemann(self, L, R, nn):
        (qL, rL, vL, pL), (qR, rR, vR, pR) = L, R
        if self.c["flux"] == "ec":
            return self.pair((rL, vL, pL), (rR, vR, pR), nn)
        fL, fR = self.euler(qL, vL, pL, nn), self.euler(qR, vR, pR, nn)
        uL, uR = (sum(v[a] * nn[a] for a in range(3)) for v in (vL, vR))
        cL, cR = torch.sqrt(GAMMA * pL / rL), torch.sqrt(GAMMA * pR / rR)
        if self.c["flux"] == "llf":
            lam = torch.maximum(uL.abs() + cL, uR.abs() + cR)
            return [0.5 * (fL[i] + fR[i]) - 0.5 * lam * (qR[i] - qL[i]) for i in range(5)]
        # Roe's solver, Harten-Hyman fix on the acoustic waves
        sL, sR = torch.sqrt(rL), torch.sqrt(rR)
        wl, wr = sL / (sL + sR), sR / (sL + sR)
        v = [wl * vL[a] + wr * vR[a] for a in range(3)]
        H = wl * (qL[4] + pL) / rL + wr * (qR[4] + pR) / rR
        q2 = sum(x * x for x in v)
        c = torch.sqrt((GAMMA - 1.0) * (H - 0.5 * q2))
        rho, un = sL * sR, sum(v[a] * nn[a] for a in range(3))
        dp, dr, dv = pR - pL, rR - rL, [vR[a] - vL[a] for a in range(3)]
        dn = uR - uL
        a1, a5, a2 = 0.5 * (dp - rho * c * dn) / c ** 2, 0.5 * (dp + rho * c * dn) / c ** 2, dr - dp / c ** 2

        def fixed(l, lL, lR):
            d = torch.maximum(torch.clamp(l - lL, min=0.0), lR - l)
            return torch.maximum(l.abs(), d)

        A1, A5 = fixed(un - c, uL - cL, uR - cR) * a1, fixed(un + c, uL + cL, uR + cR) * a5
        l2 = un.abs()
        D = [A1 + l2 * a2 + A5]
        D += [A1 * (v[a] - c * nn[a]) + l2 * (a2 * v[a] + rho * (dv[a] - dn * nn[a])) + A5 * (v[a] + c * nn[a])
              for a in range(3)]
        vdv = sum(v[a] * dv[a] for a in range(3))
        D += [A1 * (H - un * c) + l2 * (0.5 * a2 * q2 + rho * (vdv - un * dn)) + A5 * (H + un * c)]
        return [0.5 * (fL[i] + fR[i] - D[i]) for i in range(5)]

    def source(self, t, mu):
        if not hasattr(self, "ph"):
            return None
        ph = self.ph - math.pi * t
        A, s, co = MMS_AMP, torch.sin(ph), torch.cos(ph)
        r, rp = 2.0 + A * s, math.pi * A * co
        lap = 3.0 / RGAS * (math.pi ** 2 * A * s / r ** 2 + 2.0 * rp ** 2 / r ** 3)
        kap = GAMMA * RGAS / (GAMMA - 1.0) / PR
        return torch.stack([2.0 * rp] * 4 + [3.0 * rp - mu * kap * lap], 1)

    def rhs(self, U, t, mu):
        n, D, Ja = self.n, self.D, self.Ja
        q = U.unbind(1)
        v = [q[a] / q[0] for a in (1, 2, 3)]
        p = (GAMMA - 1.0) * (q[4] - 0.5 * (q[1] * v[0] + q[2] * v[1] + q[3] * v[2]))
        phi = torch.stack([*v, p / (q[0] * RGAS)], 1)
        # faces: states of both sides, lifted variables
        Uf = self.faces(U)
        qf = Uf.unbind(2)
        vf = [qf[a] / qf[0] for a in (1, 2, 3)]
        pf = (GAMMA - 1.0) * (qf[4] - 0.5 * (qf[1] * vf[0] + qf[2] * vf[1] + qf[3] * vf[2]))
        phf = torch.stack([*vf, pf / (qf[0] * RGAS)], 2)
        pho = self.other(phf)
        # weak and strong form of the lifting
        g = [[0.0] * 3 for _ in range(4)]
        Dw = (self.w[None, :] / self.w[:, None]) * D.T            # (w_m / w_r) D_mr
        star = 0.5 * (phf + pho) if self.gauss else 0.5 * (pho - phf)
        for a in range(4):
            for l in range(3):
                s = 0.0
                for d in range(3):
                    s = s - _ap(Dw, phi[:, a] * Ja[:, d, l], d) if self.gauss else s + _ap(D, phi[:, a], d) * Ja[:, d, l]
                g[a][l] = (s + self.lift_faces(star[:, :, a] * self.ns[:, :, l])) / self.J
        gf = self.faces(torch.stack([g[a][l] for a in range(4) for l in range(3)], 1))
        # face fluxes, each element's outward view
        other = self.other(Uf).unbind(2)
        vo = [other[a] / other[0] for a in (1, 2, 3)]
        po = (GAMMA - 1.0) * (other[4] - 0.5 * (other[1] * vo[0] + other[2] * vo[1] + other[3] * vo[2]))
        nn = self.nv.unbind(2)
        F = self.riemann((qf, qf[0], vf, pf), (other, other[0], vo, po), nn)
        go = self.other(gf)
        fv = self.fvisc(self.g43(gf, 2), vf, self.visc(pf / (qf[0] * RGAS), mu), nn)
        fo = self.fvisc(self.g43(go, 2), vo, self.visc(po / (other[0] * RGAS), mu), nn)
        for a in range(4):
            F[a + 1] = F[a + 1] - 0.5 * (fv[a] + fo[a])
        F = [f * self.sJ for f in F]
        muv = self.visc(p / (q[0] * RGAS), mu)
        if not self.gauss:
            # the strong form: the inner flux is taken off at the faces
            fin = self.euler(qf, vf, pf, self.ns.unbind(2))
            fvi = self.fvisc(self.g43(gf, 2), vf, self.visc(pf / (qf[0] * RGAS), mu), self.ns.unbind(2))
            F = [F[0] - fin[0]] + [F[a + 1] - fin[a + 1] + fvi[a] for a in range(4)]
        acc = [self.lift_faces(f) for f in F]
        for d in range(3):
            nn = Ja[:, d].unbind(1)
            ft = [None, *self.fvisc(g, v, muv, nn)]
            if self.gauss:
                fe = self.euler(q, v, p, nn)
                for a in range(5):
                    acc[a] = acc[a] - _ap(Dw, fe[a] - ft[a] if a else fe[a], d)
                continue
            for a in range(1, 5):
                acc[a] = acc[a] - _ap(D, ft[a], d)
            ax = -1 - d
            for s in range(n):   # every pair (r, r + s) of the lines of direction d
                roll = [torch.roll(y, -s, ax) for y in (q[0], *v, p, *nn)]
                B = (roll[0], roll[1:4], roll[4])
                f = self.pair((q[0], v, p), B, [0.5 * (x + y) for x, y in zip(nn, roll[5:])])
                i = torch.arange(n, device=DEV)
                sh = [1, 1, 1, 1]
                sh[ax] = n
                w = 2.0 * D[i, (i + s) % n].reshape(sh)
                for a in range(5):
                    acc[a] = acc[a] + w * f[a]
        out = -torch.stack(acc, 1) / self.J[:, None]
        src = self.source(t, mu)
        return out if src is None else out + src

    @staticmethod
    def g43(gf, ax):
        g = gf.unbind(ax)
        return [[g[a * 3 + l] for l in range(3)] for a in range(4)]

    def lift_faces(self, s):
        """sum over the faces of s [E, 6, q, p] l(+-1)/w, at the nodes [E, k, j, i]."""
        out = 0.0
        for f in range(6):
            if self.gauss:
                l = self.lend[f % 2] / self.w
            else:
                l = torch.zeros(self.n, dtype=torch.float64, device=DEV)
                l[-1 if f % 2 else 0] = 1.0 / self.w[0]
            sh = [1, 1, 1, 1]
            sh[3 - f // 2] = self.n
            out = out + s[:, f].unsqueeze(3 - f // 2) * l.reshape(sh)
        return out

    def steps(self, U, t, dt, count, mu):
        for _ in range(count):
            G = torch.zeros_like(U)
            for a, b, c in zip(LSERK_A, LSERK_B, LSERK_C):
                G = a * G + dt * self.rhs(U, t + c * dt, mu)
                U = U + b * G
            t += dt
        return U


def exact(case, seed):
    c = case
    if c["do"] == "ensemble":
        out = []
        for K, N, ma, re, sd in _members(c, seed):
            m = _mesh(c, (K, K, K), N)
            with torch.no_grad():
                out.append(Plain(c, m, N).steps(_flow(c, _coords(m, N, False), sd, ma), 0.0, _dt(c, N, (K, K, K), ma),
                                                c["steps"], 1.0 / re))
        return out
    mesh = _mesh(c)
    U = _flow(c, _coords(mesh, c["N"], c["gauss"]), seed)
    P, mu = Plain(c, mesh, c["N"]), _mu(c)
    if c["do"] in ("step", "rhs"):
        with torch.no_grad():
            return P.rhs(U, 0.0, mu) if c["do"] == "rhs" else P.steps(U, 0.0, _dt(c), c["steps"], mu)
    U.requires_grad_(True)
    m = torch.tensor(mu, dtype=torch.float64, device=DEV, requires_grad=True)
    lam = _lambda(U, seed)
    f = P.rhs(U, 0.0, m) if c["do"] == "vjp" else P.steps(U, 0.0, _dt(c), 1, m)
    gU, gm = torch.autograd.grad(f, (U, m), lam)
    return [gU, gm.reshape(1)]
