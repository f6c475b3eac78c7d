"""Performance cases: the calls that a user of the solver makes, at the sizes they are made.

``listed()`` gives the fixed cases, ``draw(rng)`` one more case of the same ranges,
``prepare(case, seed)`` the mesh, bias and tensors a program holds before the call, ``run(state)``
one pass through the public entry points, ``work(case)`` the bytes and operations a pass cannot do
without, and ``exact(case, seed)`` what ``run`` returns, from plain torch in 64 bits.

Devices are the five-gate Si/SiO2 double-dot stack and the MOS capacitor of the repository's
workloads, on meshes from 16 x 16 x 12 to 256 x 256 x 128 elements, at 0.5 K, 4 K and 300 K. The gate
voltages are drawn from the seed in the range where the plungers fill the dots and the barriers
separate them.
"""
import math
import random

import numpy as np
import torch

import paper_1403_7561_gb300 as q

F64 = torch.float64
LX = LY = 200.0
T_SI, T_OX = 90.0, 10.0
GATES_X = [(25.0, 45.0), (50.0, 90.0), (95.0, 105.0), (110.0, 150.0), (155.0, 175.0)]
GATES_Y = (30.0, 170.0)
DOTS_X = [(50.0, 90.0), (110.0, 150.0)]
DOTS_Y = (70.0, 130.0)
SI = dict(eps_r=11.7, chi=4.05, Eg=1.12, semiconductor=1, m_l=0.98, m_t=0.19, m_hh=0.49, m_lh=0.16,
          N_A=1e-6, N_D=0.0, E_a=0.044, E_d=0.046, g_A=4.0, g_D=2.0)
SIO2 = dict(eps_r=3.9, chi=0.95, Eg=9.0, semiconductor=0, m_l=0.5, m_t=0.5, m_hh=0.5, m_lh=0.5,
            N_A=0.0, N_D=0.0, E_a=0.0, E_d=0.0, g_A=4.0, g_D=2.0)
M_EFF = (0.19, 0.19, 0.19)


# ---------------------------------------------------------------------------
# The cases
def listed():
    return [
        # one residual of a laboratory-size MOS capacitor: the smallest call, where launches count
        dict(name="residual_mos", kind="residual", device="mos", nx=16, ny=16, nz=32, T=300.0, theta=False),
        # the line search and the Newton step of the largest device evaluate this
        dict(name="residual_large", kind="residual", device="dqd", nx=256, ny=256, nz=128, T=0.5, theta=False),
        # residual with the interface fixed charge on a mesh whose sizes fit no tile
        dict(name="residual_ragged", kind="residual", device="dqd", nx=101, ny=93, nz=61, T=4.0, theta=True),
        # FP64 Jacobian-vector products, as an outer Krylov method of a user calls them
        dict(name="jv_double", kind="jv", device="dqd", nx=128, ny=128, nz=96, T=4.0),
        # H and M applied to a block of states (a user's own eigensolver, expectation values)
        dict(name="hm_block", kind="hm", device="dqd", nx=128, ny=128, nz=96, T=4.0, nvec=10),
        # the library's defaults (FP64, Jacobi) on the small capacitor: a first program
        dict(name="solve_default", kind="solve", device="mos", nx=16, ny=16, nz=32, T=300.0, precision=0, cheb=1),
        # mixed solve of a small device of odd size, as in a parameter scan
        dict(name="solve_mixed_odd", kind="solve", device="dqd", nx=61, ny=62, nz=40, T=4.0, precision=1, cheb=-1),
        # plain FP64 solve of the 1.6M-node device
        dict(name="solve_double", kind="solve", device="dqd", nx=128, ny=128, nz=96, T=4.0, precision=0, cheb=-1),
        # forward and backward of the differentiable dot charge (gate voltages and every element's charge)
        dict(name="charge_gradient", kind="gradient", device="dqd", nx=128, ny=128, nz=96, T=4.0),
        # the lowest ten levels of the double dot
        dict(name="levels", kind="levels", device="dqd", nx=128, ny=128, nz=96, T=4.0, nev=10),
        # eight devices of different sizes solved and differentiated together
        dict(name="batch", kind="batch", T=4.0, count=8, n_min=48, n_max=112, n_seed=4),
        # the whole path on the largest device: solve, counts, capacitances and levels
        dict(name="device_large", kind="device", device="dqd", nx=256, ny=256, nz=128, T=0.5, nev=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh_sizes(rng, lo, hi_xy, hi_z):
    return dict(nx=_log_int(rng, lo, hi_xy), ny=_log_int(rng, lo, hi_xy), nz=_log_int(rng, 3 * lo // 4, hi_z))


def draw(rng):
    kind = rng.choice(["residual", "residual", "jv", "hm", "solve", "solve", "gradient", "levels", "batch", "device"])
    if kind == "batch":
        lo = rng.randrange(24, 65)
        return dict(kind=kind, T=rng.choice([0.5, 4.0]), count=rng.randrange(3, 9), n_min=lo,
                    n_max=rng.randrange(lo, 113), n_seed=rng.randrange(1000))
    small = kind in ("solve", "gradient", "levels", "device")
    # the dots and the subdomain need a few elements across
    lo = 32 if kind in ("levels", "device") else 24 if kind == "gradient" else 16
    c = dict(kind=kind, device="dqd", **_mesh_sizes(rng, lo, 160 if small else 256, 96 if small else 128))
    c["T"] = rng.choice([0.5, 4.0])
    if kind == "residual":
        c["device"] = rng.choice(["dqd", "dqd", "mos"])
        c["theta"] = c["device"] == "dqd" and rng.random() < 0.5
        if c["device"] == "mos":
            c["T"] = 300.0
    elif kind == "hm":
        c["nvec"] = rng.randrange(1, 17)
    elif kind == "solve":
        c["precision"] = rng.choice([0, 1, 1])
        c["cheb"] = -1
        if rng.random() < 0.3:  # defaults on a capacitor of moderate size
            c.update(device="mos", T=300.0, precision=0, cheb=1, nx=min(c["nx"], 48), ny=min(c["ny"], 48),
                     nz=min(max(c["nz"], 12), 48))
    elif kind in ("levels", "device"):
        c["nev"] = rng.randrange(4, 11)
    return c


# ---------------------------------------------------------------------------
# Devices
def _device(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["device"] == "mos":
        n_ox = max(1, round(nz * 10.0 / 60.0))
        return dict(Lx=100.0, Ly=100.0, nx=nx, ny=ny,
                    layers=[dict(material=0, thickness=50.0, n=nz - n_ox), dict(material=1, thickness=10.0, n=n_ox)],
                    materials=[dict(SI), dict(SIO2)], gates=[dict(x0=0.0, x1=100.0, y0=0.0, y1=100.0)],
                    gate_work_function=None, bottom_ohmic=1, dots=[], subdomain=None)
    n_ox = max(1, round(nz * T_OX / (T_SI + T_OX)))
    n_si = nz - n_ox
    kz = round(n_si * 32.0 / 86.0)
    return dict(Lx=LX, Ly=LY, nx=nx, ny=ny,
                layers=[dict(material=0, thickness=T_SI, n=n_si), dict(material=1, thickness=T_OX, n=n_ox)],
                materials=[dict(SI), dict(SIO2)],
                gates=[dict(x0=a, x1=b, y0=GATES_Y[0], y1=GATES_Y[1]) for a, b in GATES_X],
                gate_work_function=SI["chi"], bottom_ohmic=1,
                dots=[dict(x0=a, x1=b, y0=DOTS_Y[0], y1=DOTS_Y[1], z0=T_SI - 15.0, z1=T_SI) for a, b in DOTS_X],
                subdomain=dict(i0=nx // 4, i1=3 * nx // 4, j0=ny // 4, j1=3 * ny // 4, k0=n_si - kz, k1=n_si))


def _bias(case, device, rng):
    if device == "mos":
        V = [rng.uniform(0.3, 0.8)]
    else:
        V = [rng.uniform(0.66, 0.76) if g in (1, 3) else rng.uniform(0.15, 0.4) for g in range(5)]
    return dict(T=case["T"], V_gate=V, V_sub=0.0, statistics=1, incomplete_ionization=1)


def _charge(dev, seed):
    """Fixed charge of the element layer under the interface: N(0, 1e-4 nm^-2) sheets over the layer height."""
    n_si, per = dev["layers"][0]["n"], dev["nx"] * dev["ny"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    theta = torch.zeros(per * sum(l["n"] for l in dev["layers"]), dtype=F64, device="cuda")
    theta[per * (n_si - 1):per * n_si] = torch.randn(per, generator=g, dtype=F64, device="cuda") * (1e-4 * n_si / T_SI)
    return theta


def _gate_field(dev, values, bulk):
    """Potential of rectangular surface gates at the given values over a surface at `bulk`, by the closed
    form of Davies, Larkin and Sukhorukov (J. Appl. Phys. 77, 4504, 1995): the unscreened field under the
    gates, which is what a Newton iteration starts from."""
    x, y, z = _axes(dev)
    X, Y = x[None, None, :], y[None, :, None]
    d = (z[-1] - z)[:, None, None]
    phi = torch.full((z.numel(), y.numel(), x.numel()), bulk, dtype=F64, device="cuda")
    for G, v in zip(dev["gates"], values):
        for u in (X - G["x0"], G["x1"] - X):
            for w in (Y - G["y0"], G["y1"] - Y):
                phi += (v - bulk) / (2 * math.pi) * torch.atan2(u * w, d * torch.sqrt(u * u + w * w + d * d))
    return phi.reshape(-1)


def _axes(dev):
    x = torch.arange(dev["nx"] + 1, dtype=F64, device="cuda") * dev["Lx"] / dev["nx"]
    y = torch.arange(dev["ny"] + 1, dtype=F64, device="cuda") * dev["Ly"] / dev["ny"]
    z, z0 = [0.0], 0.0
    for l in dev["layers"]:
        z += [z0 + (k + 1) * l["thickness"] / l["n"] for k in range(l["n"])]
        z0 = z[-1]
    return x, y, torch.tensor(z, dtype=F64, device="cuda")


def _gates(dev):
    """Gate of every node (-1: none), and one more than the gates at the Ohmic contact below."""
    x, y, z = _axes(dev)
    gate = torch.full((z.numel(), y.numel(), x.numel()), -1, dtype=torch.int64, device="cuda")
    for k, G in enumerate(dev["gates"]):
        inside = ((x >= G["x0"]) & (x <= G["x1"]))[None, :] & ((y >= G["y0"]) & (y <= G["y1"]))[:, None]
        gate[-1][inside & (gate[-1] < 0)] = k
    gate[0] = len(dev["gates"])
    return gate


def _inputs(case, seed):
    """Everything that the seed decides, without the library: device, bias, potential, charge, vectors."""
    rng = random.Random(seed)
    if case["kind"] == "batch":
        sizes = random.Random(case["n_seed"])
        devs = []
        for _ in range(case["count"]):
            n = sizes.randint(case["n_min"], case["n_max"])
            devs.append(_device(dict(case, device="dqd", nx=n, ny=n, nz=n)))
            devs[-1]["subdomain"] = None
        return dict(devs=devs, biases=[_bias(case, "dqd", rng) for _ in devs])
    dev = _device(case)
    s = dict(dev=dev, bias=_bias(case, case["device"], rng))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n_nodes = (dev["nx"] + 1) * (dev["ny"] + 1) * (sum(l["n"] for l in dev["layers"]) + 1)
    if case["kind"] in ("residual", "jv", "hm", "levels"):
        # levels a few tens to a few hundred meV above the Fermi level; carriers under the plungers elsewhere
        off = -0.15 if case["kind"] in ("hm", "levels") else 0.1 if case["device"] == "dqd" else 0.0
        s["phi"] = _gate_field(dev, [v + off for v in s["bias"]["V_gate"]], -0.5)
    if case["kind"] == "jv":
        # a search direction: zero where the potential is prescribed
        v = torch.randn(n_nodes, generator=gen, dtype=F64, device="cuda")
        s["v"] = v.masked_fill_(_gates(dev).reshape(-1) >= 0, 0.0)
    if case["kind"] == "hm":
        S = dev["subdomain"]
        ns = (S["i1"] - S["i0"] - 1) * (S["j1"] - S["j0"] - 1) * (S["k1"] - S["k0"] - 1)
        s["X"] = torch.randn(case["nvec"], ns, generator=gen, dtype=F64, device="cuda")
    s["theta"] = _charge(dev, seed) if case.get("theta") or case["kind"] == "gradient" else None
    if case["kind"] == "gradient":
        s["weight"] = torch.tensor([rng.uniform(0.5, 1.5) for _ in dev["dots"]], dtype=F64)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"] = case["kind"]
    new = lambda n: torch.zeros(n, dtype=F64, device="cuda")  # noqa: E731
    if case["kind"] == "batch":
        s["meshes"] = [q.qcad_mesh_create(d) for d in s["devs"]]
        s["phis"] = [new(m.n_nodes) for m in s["meshes"]]
        s["opts"] = q.make_opts(precision=1, cheb_degree=-1)
        return s
    m = s["mesh"] = q.qcad_mesh_create(s["dev"])
    if case["kind"] == "residual":
        s["R"], s["diag"] = new(m.n_nodes), new(m.n_nodes)
    elif case["kind"] == "jv":
        s["y"] = new(m.n_nodes)
    elif case["kind"] == "hm":
        s["HX"], s["MX"] = torch.empty_like(s["X"]), torch.empty_like(s["X"])
    elif case["kind"] == "levels":
        s["nev"] = case["nev"]
    else:
        s["phi"] = new(m.n_nodes)
        s["opts"] = q.make_opts(precision=case.get("precision", 1), cheb_degree=case.get("cheb", -1))
        s["nev"] = case.get("nev")
    if case["kind"] == "gradient":
        s["V"] = torch.tensor(s["bias"]["V_gate"], dtype=F64)
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        q.qcad_poisson_solve_batch(s["meshes"], s["biases"], s["opts"], s["phis"])
        dN = q.qcad_adjoint_batch(s["meshes"], s["biases"], s["opts"], s["phis"])
        return {"phi": s["phis"], "dN_dV": np.array(dN)}
    m, b = s["mesh"], s["bias"]
    if kind == "residual":
        st = q.qcad_poisson_residual(m, b, s["phi"], s["R"], diag=s["diag"], fixed_charge=s["theta"])
        return {"R": s["R"], "diag": s["diag"], "norms": np.array(st)}
    if kind == "jv":
        q.qcad_poisson_jv(m, b, s["phi"], s["v"], s["y"])
        return s["y"]
    if kind == "hm":
        q.qcad_schrodinger_apply(m, b, s["phi"], M_EFF, s["X"], HX=s["HX"], MX=s["MX"])
        return {"HX": s["HX"], "MX": s["MX"]}
    if kind == "solve":
        q.qcad_poisson_solve(m, b, s["opts"], s["phi"])
        return s["phi"]
    if kind == "gradient":
        V, theta = s["V"].requires_grad_(), s["theta"].requires_grad_()
        N = q.QcadDotCharge.apply(V, theta, m, b, s["opts"])
        gV, gt = torch.autograd.grad(N, (V, theta), s["weight"])
        return {"N": N.detach(), "dV": gV, "dtheta": gt}
    if kind == "levels":
        E, _ = q.qcad_schrodinger_eigs(m, b, s["phi"], nev=s["nev"], m_eff=M_EFF, tol=1e-8)
        return np.array(E)
    q.qcad_poisson_solve(m, b, s["opts"], s["phi"])
    N = q.qcad_electron_counts(m, b, s["phi"])
    dN, E, _ = q.qcad_adjoint_eigs(m, b, s["phi"], s["opts"], nev=s["nev"], m_eff=M_EFF, tol=1e-8)
    return {"phi": s["phi"], "N": np.array(N), "dN_dV": np.array(dN), "E": np.array(E)}


def work(case):
    """Inputs read once and outputs written once; operations of one evaluation of the operators involved
    (the 27-point stiffness and the 2 x 2 x 2 quadrature), since how often a solver applies them is its own."""
    if case["kind"] == "batch":
        sizes = random.Random(case["n_seed"])
        n3 = [sizes.randint(case["n_min"], case["n_max"]) for _ in range(case["count"])]
        return {"bytes": 8.0 * sum((n + 1) ** 3 for n in n3), "flops": 150.0 * sum(n ** 3 for n in n3)}
    nodes = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    elems = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] in ("hm", "levels"):
        S = _device(case)["subdomain"]
        ns = (S["i1"] - S["i0"] - 1) * (S["j1"] - S["j0"] - 1) * (S["k1"] - S["k0"] - 1)
        box = (S["i1"] - S["i0"] + 1) * (S["j1"] - S["j0"] + 1) * (S["k1"] - S["k0"] + 1)
        nv = case.get("nvec", case.get("nev"))
        return {"bytes": 8.0 * box + (24.0 * ns * nv if case["kind"] == "hm" else 0.0), "flops": 130.0 * ns * nv}
    per_node = {"residual": 24, "jv": 24, "solve": 8, "gradient": 0, "device": 8}[case["kind"]]
    per_elem = 16 if case["kind"] == "gradient" else 8 if case.get("theta") else 0
    return {"bytes": float(per_node * nodes + per_elem * elems), "flops": 42.0 * nodes + 100.0 * elems}


# ---------------------------------------------------------------------------
# The same results from plain torch in 64 bits (2 x 2 x 2 Gauss points, Q1 hexahedra on tensor grids)
Q_E, K_B, HBAR, M0, EPS0 = 1.602176634e-19, 1.380649e-23, 1.054571817e-34, 9.1093837015e-31, 8.8541878128e-12
QE = Q_E / EPS0 * 1e9
H2M0 = HBAR * HBAR / (2.0 * M0) / Q_E * 1e18
G0, G1 = 0.5 + 0.5 / math.sqrt(3.0), 0.5 - 0.5 / math.sqrt(3.0)


def _line(v, w, dim, stiff):
    """The 1D element matrices w/h [1 -1; -1 1] or w h/6 [2 1; 1 2], given per element in w, along one axis."""
    n = v.shape[dim] - 1
    shape = [1] * v.dim()
    shape[dim] = n
    w = w.view(shape)
    a, b = v.narrow(dim, 0, n), v.narrow(dim, 1, n)
    out = torch.zeros_like(v)
    if stiff:
        t = (b - a) * w
        out.narrow(dim, 0, n).sub_(t)
        out.narrow(dim, 1, n).add_(t)
    else:
        s = (a + b) * (w / 6)
        out.narrow(dim, 0, n).add_(s + a * (w / 6))
        out.narrow(dim, 1, n).add_(s + b * (w / 6))
    return out


def _to_gauss(v):
    """Values at the Gauss points of every element, the points' z, y, x indices leading."""
    for dim in (-1, -2, -3):
        n = v.shape[dim] - 1
        a, b = v.narrow(dim, 0, n), v.narrow(dim, 1, n)
        v = torch.stack([G0 * a + G1 * b, G1 * a + G0 * b])
    return v


def _from_gauss(u):
    """The transpose of _to_gauss."""
    for dim in (-3, -2, -1):
        shape = list(u.shape[1:])
        n = shape[dim]
        shape[dim] = n + 1
        v = torch.zeros(shape, dtype=F64, device=u.device)
        v.narrow(dim, 0, n).add_(G0 * u[0] + G1 * u[1])
        v.narrow(dim, 1, n).add_(G1 * u[0] + G0 * u[1])
        u = v
    return u


class _Operator:
    """K + (mass with coefficients c at the Gauss points) on a tensor grid; kappa: conductivity per axis and layer."""

    def __init__(self, x, y, z, kappa):
        self.h = [z.diff(), y.diff(), x.diff()]
        self.kappa = kappa  # [axis z, y, x][layer]
        self.wdet = (self.h[0][:, None, None] * self.h[1][None, :, None] * self.h[2][None, None, :]) / 8

    def stiff(self, v):
        (hz, hy, hx), (kz, ky, kx) = self.h, self.kappa
        mx = _line(v, hx, -1, False)
        kxv = _line(_line(_line(v, 1 / hx, -1, True), hy, -2, False), hz * kx, -3, False)
        kyv = _line(_line(mx, 1 / hy, -2, True), hz * ky, -3, False)
        return kxv + kyv + _line(_line(mx, hy, -2, False), kz / hz, -3, True)

    def mass(self, v, c):
        return _from_gauss(_to_gauss(v) * c)

    def diagonal(self, c):
        """Diagonal of the whole operator."""
        (hz, hy, hx), (kz, ky, kx) = self.h, self.kappa

        def d(w):
            out = torch.zeros(w.numel() + 1, dtype=F64, device=w.device)
            out[:-1] += w
            out[1:] += w
            return out

        def p(a, b, e):
            return a[:, None, None] * b[None, :, None] * e[None, None, :]

        out = p(d(hz * kx / 3), d(hy / 3), d(1 / hx)) + p(d(hz * ky / 3), d(1 / hy), d(hx / 3)) \
            + p(d(kz / hz), d(hy / 3), d(hx / 3))
        for dim in (-3, -2, -1):  # the transpose of _to_gauss with squared weights
            shape = list(c.shape[1:])
            n = shape[dim]
            shape[dim] = n + 1
            v = torch.zeros(shape, dtype=F64, device=c.device)
            v.narrow(dim, 0, n).add_(G0 * G0 * c[0] + G1 * G1 * c[1])
            v.narrow(dim, 1, n).add_(G1 * G1 * c[0] + G0 * G0 * c[1])
            c = v
        return out + c


class _Poisson:
    """The nonlinear Poisson problem of a device at a bias, matrix-free."""

    def __init__(self, dev, bias, theta=None):
        self.dev, x, y, z = dev, *_axes(dev)
        self.n_si = dev["layers"][0]["n"]
        eps = torch.cat([torch.full((l["n"],), dev["materials"][l["material"]]["eps_r"], dtype=F64, device="cuda")
                         for l in dev["layers"]])
        self.op = _Operator(x, y, z, [eps, eps, eps])
        self.shape = (z.numel(), y.numel(), x.numel())
        self.eshape = (z.numel() - 1, y.numel() - 1, x.numel() - 1)
        self.theta = None if theta is None else theta.view(self.eshape)
        T = bias["T"]
        self.kT = kT = K_B * T / Q_E
        mn = 6.0 ** (2.0 / 3.0) * (SI["m_l"] * SI["m_t"] ** 2) ** (1.0 / 3.0)
        mp = (SI["m_hh"] ** 1.5 + SI["m_lh"] ** 1.5) ** (2.0 / 3.0)
        dos = lambda m: 2.0 * (m * M0 * K_B * T / (2.0 * math.pi * HBAR * HBAR) * 1e-18) ** 1.5  # noqa: E731
        self.NC, self.NV = dos(mn), dos(mp)
        self.ref = SI["chi"] + 0.5 * SI["Eg"] + 0.5 * kT * math.log(self.NC / self.NV)
        if T < 50.0:
            ln_y = 0.5 * math.log(SI["N_A"] / (4.0 * self.NV)) + SI["E_a"] / (2.0 * kT)
        else:
            ln_y = math.log(-0.125 + 0.125 * math.sqrt(1.0 + 16.0 * SI["N_A"] / self.NV * math.exp(SI["E_a"] / kT)))
        ohmic = SI["E_a"] + self.ref - SI["chi"] - SI["Eg"] - kT * ln_y
        self.gate = _gates(dev)
        self.fixed = self.gate >= 0
        wf = dev["gate_work_function"]
        self.values = torch.zeros(self.shape, dtype=F64, device="cuda")
        for k, V in enumerate(bias["V_gate"]):
            self.values[self.gate == k] = V if wf is None else V - (wf - self.ref)
        self.values[0] = ohmic

    def density(self, phi):
        """rho, rho', n, n' at the Gauss points of the silicon elements."""
        kT, u = self.kT, _to_gauss(phi[:self.n_si + 1])

        def fermi(t):
            s = t.clamp(min=-50.0)
            g = torch.exp(-0.17 * (s + 1.0) ** 2)
            v = s ** 4 + 50.0 + 33.6 * s * (1.0 - 0.68 * g)
            dv = 4.0 * s ** 3 + 33.6 * (1.0 - 0.68 * g) + 33.6 * 0.68 * 0.34 * s * (s + 1.0) * g
            c, e = 0.75 * math.sqrt(math.pi), torch.exp(-s)
            D = e + c * v ** -0.375
            low, mb = t < -50.0, torch.exp(t.clamp(max=0.0))
            return torch.where(low, mb, 1 / D), torch.where(low, mb, (e + 0.375 * c * v ** -1.375 * dv) / (D * D))

        n, dn = fermi((u - self.ref + SI["chi"]) / kT)
        p, dp = fermi((self.ref - SI["chi"] - SI["Eg"] - u) / kT)
        n, dn, p, dp = n * self.NC, dn * (self.NC / kT), p * self.NV, dp * (-self.NV / kT)
        t = (SI["E_a"] + self.ref - SI["chi"] - SI["Eg"] - u) / kT
        s = torch.sigmoid(-(t + math.log(SI["g_A"])))
        na, dna = SI["N_A"] * s, SI["N_A"] / kT * s * torch.sigmoid(t + math.log(SI["g_A"]))
        return p - n - na, dp - dn - dna, n, dn

    def all_elements(self, v):
        out = torch.zeros((2, 2, 2) + self.eshape, dtype=F64, device="cuda")
        out[:, :, :, :self.n_si] = v
        return out

    def residual(self, phi, rho):
        rho = self.all_elements(rho)
        if self.theta is not None:
            rho = rho + self.theta
        R = self.op.stiff(phi) - QE * _from_gauss(rho * self.op.wdet)
        return R.masked_fill_(self.fixed, 0.0)

    def coefficients(self, drho):
        return self.all_elements(-QE * drho) * self.op.wdet

    def jv(self, v, c):
        return self.op.stiff(v) + self.op.mass(v, c)

    def pcg(self, c, b, rtol):
        d = self.op.diagonal(c)
        x, r = torch.zeros_like(b), b.clone()
        z = r / d
        p, rz = z.clone(), (r * z).sum()
        stop = (rtol * b.norm()) ** 2
        for it in range(20000):
            Ap = self.jv(p, c).masked_fill_(self.fixed, 0.0)
            a = rz / (p * Ap).sum()
            x += a * p
            r -= a * Ap
            if it % 16 == 15 and bool((r * r).sum() <= stop):
                break
            z = r / d
            rz, old = (r * z).sum(), rz
            p = z + (rz / old) * p
        return x

    def solve(self):
        zero = torch.zeros((2, 2, 2) + self.eshape, dtype=F64, device="cuda")
        phi = self.values.clone()
        phi += self.pcg(zero, -self.op.stiff(phi).masked_fill_(self.fixed, 0.0), 1e-3)
        rho, drho, _, _ = self.density(phi)
        R = self.residual(phi, rho)
        first = R.norm()
        for _ in range(100):
            rtol = max(1e-8, min(1e-2, float(R.norm() / first)))
            step, a = self.pcg(self.coefficients(drho), -R, rtol), 1.0
            for _ in range(31):
                t = phi + a * step
                rho, drho, _, _ = self.density(t)
                Rt = self.residual(t, rho)
                if bool(Rt.norm() <= (1 - 1e-4 * a) * R.norm()):
                    break
                a *= 0.5
            if float(a * step.abs().max()) < 1e-11 and float(Rt.abs().max()) < 1e-10:
                return t
            phi, R = t, Rt
        return phi

    def dots(self):
        out = []
        x, y, z = _axes(self.dev)
        xc, yc, zc = ((v[1:] + v[:-1]) / 2 for v in (x, y, z[:self.n_si + 1]))
        for D in self.dev["dots"]:
            out.append(((zc >= D["z0"]) & (zc <= D["z1"]))[:, None, None]
                       & ((yc >= D["y0"]) & (yc <= D["y1"]))[None, :, None]
                       & ((xc >= D["x0"]) & (xc <= D["x1"]))[None, None, :])
        return out

    def counts(self, phi):
        n = self.density(phi)[2]
        return torch.stack([(n * self.op.wdet[:self.n_si] * m).sum() for m in self.dots()])

    def gradients(self, phi, weights):
        """d(sum_d weights[d] N_d) by gate voltage, and by each element's fixed charge."""
        _, drho, _, dn = self.density(phi)
        c = self.coefficients(drho)
        g = torch.zeros(self.shape, dtype=F64, device="cuda")
        for w, m in zip(weights, self.dots()):
            g[:self.n_si + 1] += _from_gauss(dn * self.op.wdet[:self.n_si] * m * w)
        lam = self.pcg(c, g.masked_fill(self.fixed, 0.0), 1e-13)
        out = []
        for k in range(len(self.dev["gates"])):
            e = (self.gate == k).to(F64)
            out.append((g * e).sum() - (lam * self.jv(e, c)).sum())
        one = torch.ones((2, 2, 2) + (1, 1, 1), dtype=F64, device="cuda")
        return torch.stack(out), (QE * (_to_gauss(lam) * one).sum((0, 1, 2)) * self.op.wdet).reshape(-1)


class _Dot:
    """H and M on the interior nodes of the quantum subdomain."""

    def __init__(self, dev, ref, phi):
        S, (x, y, z) = dev["subdomain"], _axes(dev)
        x, y, z = x[S["i0"]:S["i1"] + 1], y[S["j0"]:S["j1"] + 1], z[S["k0"]:S["k1"] + 1]
        k = [torch.full((z.numel() - 1,), H2M0 / m, dtype=F64, device="cuda") for m in reversed(M_EFF)]
        self.op = _Operator(x, y, z, k)
        box = phi[S["k0"]:S["k1"] + 1, S["j0"]:S["j1"] + 1, S["i0"]:S["i1"] + 1]
        self.c = ((ref - SI["chi"]) - _to_gauss(box)) * self.op.wdet
        self.shape = (z.numel() - 2, y.numel() - 2, x.numel() - 2)

    def _pad(self, X):
        return torch.nn.functional.pad(X.view((-1,) + self.shape), (1, 1, 1, 1, 1, 1))

    def _cut(self, Y):
        return Y[:, 1:-1, 1:-1, 1:-1].reshape(Y.shape[0], -1)

    def H(self, X):
        v = self._pad(X)
        return self._cut(self.op.stiff(v) + self.op.mass(v, self.c[:, :, :, None]))

    def M(self, X):
        v = self._pad(X)
        for dim, h in zip((-3, -2, -1), self.op.h):
            v = _line(v, h, dim, False)
        return self._cut(v)

    def levels(self, nev):
        """Chebyshev-filtered subspace iteration of M^-1 H (M inverted axis by axis)."""
        inv = [torch.linalg.inv(_line(torch.eye(h.numel() + 1, dtype=F64, device="cuda"), h, 0, False)[1:-1, 1:-1])
               for h in self.op.h]

        def B(X):
            v = self.H(X).view((-1,) + self.shape)
            v = v @ inv[2]
            v = inv[1] @ v
            return torch.einsum("ab,nbyx->nayx", inv[0], v).reshape(X.shape)

        gen = torch.Generator(device="cuda").manual_seed(1)
        n = self.shape[0] * self.shape[1] * self.shape[2]
        X = torch.randn(min(n, 2 * nev + 4), n, generator=gen, dtype=F64, device="cuda")
        top = X[:1]
        for _ in range(40):
            top = B(top / top.norm())
        hi, lo, last = 1.3 * float(top.norm()), None, None
        for it in range(60):
            if lo is not None:  # the Chebyshev polynomial that is small on [lo, hi]
                mid, half = (hi + lo) / 2, (hi - lo) / 2
                s = half / (last[0] - mid)
                sigma, Y = s, (B(X) - mid * X) * (s / half)
                for _ in range(79):
                    t = 1 / (2 / sigma - s)
                    Y, X, s = (B(Y) - mid * Y) * (2 * t / half) - (s * t) * X, Y, t
                X = Y
            X = X / X.norm(dim=1, keepdim=True)
            L = torch.linalg.inv(torch.linalg.cholesky(X @ self.M(X).T))
            E, C = torch.linalg.eigh(L @ (X @ self.H(X).T) @ L.T)
            X = (C.T @ L) @ X
            E = E.tolist()
            if last is not None and max(abs(a - b) for a, b in zip(E[:nev], last)) < 1e-13 * abs(E[nev - 1]):
                break
            last, lo = E, E[-1]
        return E[:nev]


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "batch":
        if sum(d["nx"] ** 3 for d in s["devs"]) > 2e6:
            return None
        problems = [_Poisson(d, b) for d, b in zip(s["devs"], s["biases"])]
        phis = [p.solve() for p in problems]
        dN = [[p.gradients(f, [d == 0, d == 1])[0].tolist() for d in (0, 1)] for p, f in zip(problems, phis)]
        return {"phi": [f.reshape(-1) for f in phis], "dN_dV": np.array(dN)}
    P = _Poisson(s["dev"], s["bias"], s["theta"])
    if case["kind"] in ("residual", "jv", "hm", "levels"):
        phi = s["phi"].view(P.shape)
        if case["kind"] == "residual":
            rho, drho, _, _ = P.density(phi)
            R = P.residual(phi, rho)
            diag = P.op.diagonal(P.coefficients(drho)).masked_fill_(P.fixed, 1.0)
            return {"R": R.reshape(-1), "diag": diag.reshape(-1),
                    "norms": np.array([float(R.abs().max()), float((R * R).sum())])}
        if case["kind"] == "jv":
            v = s["v"].view(P.shape)
            y = P.jv(v.masked_fill(P.fixed, 0.0), P.coefficients(P.density(phi)[1]))
            return torch.where(P.fixed, v, y).reshape(-1)
        D = _Dot(s["dev"], P.ref, phi)
        if case["kind"] == "hm":
            return {"HX": D.H(s["X"]), "MX": D.M(s["X"])}
        return np.array(D.levels(case["nev"])) if math.prod(D.shape) <= 1.5e5 else None
    if math.prod(P.eshape) > 2e6:
        return None
    phi = P.solve()
    if case["kind"] == "solve":
        return phi.reshape(-1)
    if case["kind"] == "gradient":
        gV, gt = P.gradients(phi, s["weight"].tolist())
        return {"N": P.counts(phi), "dV": gV, "dtheta": gt}
    dN = [P.gradients(phi, [d == 0, d == 1])[0].tolist() for d in (0, 1)]
    D = _Dot(s["dev"], P.ref, phi)
    E = np.array(D.levels(case["nev"])) if math.prod(D.shape) <= 1.5e5 else None
    return {"phi": phi.reshape(-1), "N": P.counts(phi), "dN_dV": np.array(dN), "E": E}
