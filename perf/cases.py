"""The timed cases: the work that a user of the library has it do, through its public entry points.

A case is a mesh, an order, a precision form and a kind of call:

  rhs       dg_rhs, one evaluation of the right-hand side
  steps     dg_set_state, dg_step_async over some steps, dg_get_state
  host      the same from and to pinned host memory (dg_set_state, dg_step_to_host)
  adjoint   dg_adjoint_step, one time step reversed
  ensemble  dg_ensemble_step_async over members of uneven sizes and orders

listed() holds the sizes that the repository's workloads, tests and benchmark
use, and odd ones; draw() gives more of the same ranges.  prepare() makes a
moist hydrostatic column, a warm bubble with smooth momentum perturbations and
a rain shaft on the GPU, from the seed alone.  exact() evaluates the same
discretisation with plain float64 torch operations (and torch's automatic
differentiation for the adjoint), without the library.
"""
import functools
import math

import numpy as np
import torch

from paper_2305_13847_gb300 import dgmoist as dm

TOP, WIDTH = 10.0e3, 20.0e3           # the column's height and the horizontal extent, m
SIGMA = 10.0                          # interior penalty of the artificial diffusion
SPONGE = (0.75 * TOP, 0.1)            # sponge layer: lower edge and strength
FORMS = {"fp64": dm.DG_FP64, "bulk": dm.DG_FP32_BULK, "pert": dm.DG_FP32_PERT, "ffc": dm.DG_FP64_FFC}


def _case(kind, n, order, rain=1, form="fp64", steps=1, walls=0, gamma=0.0, name=None):
    """walls: 1 puts slip walls in y too (3-D) or in x (2-D) instead of periodic sides."""
    c = dict(kind=kind, dim=len(n), n0=n[0], n1=n[1], n2=n[2] if len(n) == 3 else 1, order=order,
             rain=rain, form=form, steps=steps, walls=walls, gamma=gamma)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one right-hand side of the smallest workload, as an outside integrator calls it: latency
        _case("rhs", (20, 10), 3, rain=0, name="rhs_2d_q3"),
        # the 2-D bubble workload without rain, stepped in one call: launches
        _case("steps", (20, 10), 3, rain=0, steps=10, name="steps_2d_q3"),
        # the forward run of the 2-D adjoint workload: a mesh of a few waves
        _case("steps", (128, 64), 4, steps=4, name="steps_2d_q4_rain"),
        # a small 3-D run at low order, ragged sizes, walls on two directions
        _case("steps", (21, 17, 13), 2, steps=4, walls=1, name="steps_3d_q2_ragged"),
        # the headline workload: 3-D warm rain in float64 at full size
        _case("steps", (64, 64, 32), 4, steps=2, name="steps_3d_q4"),
        # the float32 workload at full size: single-precision fluxes, float64 split
        _case("steps", (128, 128, 64), 3, form="bulk", steps=2, name="bulk_3d_q3"),
        # the float32 perturbation form at a middling, odd size
        _case("steps", (61, 47, 29), 3, form="pert", steps=4, name="pert_3d_q3_ragged"),
        # float64 with float-float contractions at the profiles' size
        _case("steps", (32, 32, 16), 4, form="ffc", steps=2, name="ffc_3d_q4"),
        # a stabilised run: artificial diffusion and the sponge layer
        _case("steps", (24, 24, 16), 4, steps=2, gamma=0.06, name="stabilised_3d_q4"),
        # one reversed step of the adjoint workload
        _case("adjoint", (128, 64), 4, name="adjoint_2d_q4"),
        # a batch of independent 2-D runs, float32
        dict(kind="ensemble", dim=2, members=32, steps=2, form="bulk", name="ensemble_32"),
        # a coupled host program: state up, one step, state down
        _case("host", (48, 48, 24), 4, name="host_3d_q4"),
    ]


def draw(rng):
    kind = rng.choice(["rhs", "steps", "steps", "steps", "steps", "host", "adjoint", "ensemble"])
    if kind == "ensemble":
        return dict(kind=kind, dim=2, members=rng.randint(4, 40), steps=rng.randint(1, 3),
                    form=rng.choice(["bulk", "pert"]))
    form = "fp64" if kind in ("adjoint", "host") else rng.choice(["fp64", "fp64", "bulk", "pert", "ffc"])
    dim = 2 if kind == "adjoint" else rng.choice([2, 3, 3])
    order = rng.randint(1, 5)
    gamma = 0.06 if kind == "steps" and form == "fp64" and rng.random() < 0.2 else 0.0
    # the nodes over the range of the listed cases (logarithm), then uneven sides
    top = {2: 4.0e5, 3: 3.0e7 if form in ("bulk", "pert") else 4.0e6}[dim] / (4.0 if gamma else 1.0)
    elements = max(8.0, math.exp(rng.uniform(math.log(3.0e3), math.log(top))) / (order + 1) ** dim)
    side = elements ** (1.0 / dim)
    n = tuple(max(2, round(side * rng.uniform(0.6, 1.4))) for _ in range(dim))
    return _case(kind, n, order, rain=rng.choice([0, 1, 1]), form=form, steps=rng.randint(1, 4),
                 walls=rng.choice([0, 0, 1]), gamma=gamma)


# ---------------------------------------------------------------------------
# the physics, for the inputs and for exact()
# ---------------------------------------------------------------------------
CL, CVD, CVV, RD, RV, TREF, PREF, G = 4218.0, 718.0, 1390.0, 287.05, 461.51, 273.15, 1.0e5, 9.81
ES_A = (1850.0 - CL) / RV
ES_B = (2.835e6 - (1850.0 - CL) * TREF) / RV
LAT = 2.835e6 - RV * TREF
FLOOR = 1e-12                         # rain density below which the adjoint freezes fractional powers
VR0 = 130.0 * math.gamma(4.5) / 6.0 * (math.pi * 8.0e6) ** -0.125


def _rho_vs(T):
    return 610.7 / (RV * TREF) * torch.exp((ES_A - 1.0) * torch.log(T / TREF) + ES_B * (1.0 / TREF - 1.0 / T))


def _moist(p, T, qt):
    """rho_d, rho_m and the internal energy of moist air at rest at pressure p, temperature T."""
    rvs = _rho_vs(T)
    rd = p / (T * (RD + qt * RV))
    sat = qt * rd > rvs
    rd = torch.where(sat, (p - rvs * RV * T) / (RD * T), rd)
    rm = qt * rd
    rv = torch.where(sat, rvs, rm)
    return rd, rm, (CVD * rd + CVV * rv + CL * (rm - rv)) * (T - TREF) + rv * LAT


@functools.lru_cache(None)
def _log_pressure(h=5.0):
    """ln p on a grid of h metres, hydrostatic by RK4: 300 K dry potential temperature, total water
    0.015 (1 - z/TOP)."""
    def dp(zz, p):
        T, qt = 300.0 * (p / PREF) ** (RD / 1005.0), 0.015 * (1.0 - zz / TOP)
        rvs = 610.7 / (RV * T) * (T / TREF) ** ES_A * math.exp(ES_B * (1.0 / TREF - 1.0 / T))
        rd = p / (T * (RD + qt * RV))
        if qt * rd > rvs:
            rd = (p - rvs * RV * T) / (RD * T)
        return -(1.0 + qt) * rd * G

    p, grid = PREF, [PREF]
    for i in range(int(TOP / h)):
        zz = i * h
        k1 = dp(zz, p)
        k2 = dp(zz + 0.5 * h, p + 0.5 * h * k1)
        k3 = dp(zz + 0.5 * h, p + 0.5 * h * k2)
        k4 = dp(zz + h, p + h * k3)
        p += h * (k1 + 2.0 * k2 + 2.0 * k3 + k4) / 6.0
        grid.append(p)
    return h * np.arange(len(grid)), np.log(grid)


def _column(z):
    """Base state [rho_d, rho_m, E, p] at the levels z (numpy)."""
    p = np.exp(np.interp(z, *_log_pressure()))
    t = torch.from_numpy(p)
    rd, rm, E = _moist(t, 300.0 * (t / PREF) ** (RD / 1005.0), torch.from_numpy(0.015 * (1.0 - z / TOP)))
    return np.stack([rd.numpy(), rm.numpy(), E.numpy(), p])


class _Mesh:
    """Gauss-Legendre tables, z-levels and the base state of one mesh."""

    def __init__(self, dim, n, order, rain, walls):
        self.dim, self.n, self.k, self.p1, self.rain = dim, tuple(n[:dim]), order, order + 1, bool(rain)
        self.L = (WIDTH,) * (dim - 1) + (TOP,)
        self.h = [a / b for a, b in zip(self.L, self.n)]
        self.periodic = [True] * (dim - 1) + [False]
        if walls:
            self.periodic[dim - 2] = False
        self.im = 3 if rain else 2
        self.nf = self.im + dim + 1
        x, w = np.polynomial.legendre.leggauss(self.p1)
        c = np.array([np.prod([x[a] - x[i] for i in range(self.p1) if i != a]) for a in range(self.p1)])
        D = np.array([[(c[i] / c[a]) / (x[i] - x[a]) if a != i else 0.0 for a in range(self.p1)]
                      for i in range(self.p1)])                      # D[i, a] = l_a'(x_i)
        D -= np.diag(D.sum(axis=1))
        at = lambda s: np.array([np.prod([(s - x[i]) / (x[a] - x[i]) for i in range(self.p1) if i != a])  # noqa: E731
                                 for a in range(self.p1)])
        dat = lambda s: np.array([sum(np.prod([s - x[i] for i in range(self.p1) if i not in (a, b)])  # noqa: E731
                                      for b in range(self.p1) if b != a) / c[a] for a in range(self.p1)])
        self.x, self.w = x, w
        self.dhat = (w[None, :] / w[:, None]) * D.T
        self.D, self.lm, self.lp, self.dlm, self.dlp = D, at(-1.0), at(1.0), dat(-1.0), dat(1.0)
        nv, hz = self.n[-1], self.h[-1]
        self.zn = (np.arange(nv)[:, None] * hz + (1.0 + x)[None, :] * hz * 0.5).reshape(-1)
        self.zf = np.arange(nv + 1) * hz
        tab = _column(np.concatenate([self.zn, self.zf]))
        self.node, self.face = np.ascontiguousarray(tab[:, :self.zn.size]), np.ascontiguousarray(tab[:, self.zn.size:])
        self.shape = (self.nf,) + self.n[::-1] + (self.p1,) * dim   # fields, elements (z, y, x), nodes (z, y, x)
        self.nodes = int(np.prod(self.shape[1:]))
        self.dt = 0.05 * min(self.h) / 380.0

    def config(self, form):
        mask = sum(1 << j for j in range(self.dim - 1) if self.periodic[j])
        return dm.make_config(self.dim, self.n, self.L, self.k, mask, self.rain, FORMS[form], G)

    # element axis and node axis of direction j in a field of shape[1:], and one with the vertical levels
    def ea(self, j):
        return self.dim - 1 - j

    def na(self, j):
        return 2 * self.dim - 1 - j

    def levels(self, tab, dev):
        s = [1] * (2 * self.dim)
        s[0], s[self.dim] = self.n[-1], self.p1
        return torch.from_numpy(tab).to(dev).reshape(s)

    def coords(self, j, dev):
        s = [1] * (2 * self.dim)
        s[self.ea(j)], s[self.na(j)] = self.n[j], self.p1
        c = (np.arange(self.n[j])[:, None] + 0.5 * (1.0 + self.x)[None, :]) * self.h[j]
        return torch.from_numpy(c).to(dev).reshape(s)

    def initial(self, seed, dev):
        """Warm bubble, smooth winds of a few m/s, temperature noise of 0.1 K, a rain shaft under the bubble."""
        g = torch.Generator(device=dev).manual_seed(seed)
        r = torch.rand(16, generator=g, device=dev, dtype=torch.float64).tolist()
        U = torch.zeros(self.shape, dtype=torch.float64, device=dev)
        xs = [self.coords(j, dev) for j in range(self.dim)]
        p, z = self.levels(self.node[3], dev), xs[-1]
        centre = [WIDTH * (0.3 + 0.4 * r[j]) for j in range(self.dim - 1)] + [2.0e3 + 500.0 * r[2]]
        rad = [max(2.0e3, 2.0 * h) for h in self.h]
        far = sum(((x - c) / a) ** 2 for x, c, a in zip(xs, centre, rad)).sqrt().clamp(max=1.0)
        ex = (p / PREF) ** (RD / 1005.0)
        T = (300.0 + (1.5 + r[3]) * torch.cos(0.5 * math.pi * far) ** 2) * ex
        T = T + 0.2 * (torch.rand(self.shape[1:], generator=g, device=dev, dtype=torch.float64) - 0.5)
        rd, rm, E = _moist(p, T, 0.015 * (1.0 - z / TOP))
        U[0] = rd - self.levels(self.node[0], dev)
        U[1] = rm - self.levels(self.node[1], dev)
        U[-1] = E - self.levels(self.node[2], dev)
        for j in range(self.dim):
            wave = 1.0 + r[4 + j]
            for i, x in enumerate(xs):
                wave = wave * torch.sin(2.0 * math.pi * (x / self.L[i] * (1 + (i + j) % 2) + r[7 + i + j]) + 0.3)
            U[self.im + j] = 2.0 * wave
        if self.rain:
            off = sum(((x - c) / (1.2 * a)) ** 2 for x, c, a in zip(xs[:-1], centre, rad)) + ((z - 2.5e3) / 3.0e3) ** 2
            U[2] = 1.0e-4 * torch.cos(0.5 * math.pi * off.sqrt().clamp(max=1.0)) ** 2
        return U


def _mesh(c):
    return _Mesh(c["dim"], (c["n0"], c["n1"], c["n2"]), c["order"], c["rain"], c["walls"])


def _members(c):
    """Ensemble members: sides 32 to 256, orders 2 to 5, rain on, as one list of meshes per case."""
    r = np.random.RandomState(5000 + c["members"]).rand(c["members"], 2)
    out = []
    for a, b in r:
        nx = 32 + int(a * 225)
        out.append(_Mesh(2, (nx, nx // 2), 2 + int(b * 4), 1, 0))
    return out


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
class _State:
    """A context (or an ensemble) with its inputs and output buffers; freed with the object."""
    ctx = ens = None

    def __del__(self):
        if self.ctx is not None:
            dm.dg_free(self.ctx)
        if self.ens is not None:
            dm.dg_ensemble_free(self.ens)


def prepare(case, seed):
    s = _State()
    s.case = case
    real = torch.float32 if case["form"] in ("bulk", "pert") else torch.float64
    if case["kind"] == "ensemble":
        s.stream = torch.cuda.Stream()
        meshes = _members(case)
        b = dm.dg_bubble()
        b.theta, b.p_s, b.qt0, b.H, b.amplitude = 300.0, 1.0e5, 0.015, TOP, 2.0
        for j in range(3):
            b.centre[j], b.radius[j] = 2.0e3, 2.0e3
        s.ens = dm.dg_ensemble_create([m.config(case["form"]) for m in meshes], [b] * len(meshes), s.stream)
        s.member = [dm.dg_ensemble_member(s.ens, i) for i in range(len(meshes))]
        s.out = []
        for i, m in enumerate(meshes):
            U = m.initial(seed * 64 + i, "cuda").to(real)
            torch.cuda.current_stream().synchronize()
            dm.dg_set_base_state(s.member[i], m.node, m.face)
            dm.dg_set_state(s.member[i], U, dm.DG_DEVICE)
            s.out.append(torch.empty_like(U))
        dm.dg_ensemble_configure_branches(s.ens, [m.dt for m in meshes], 64)
        return s
    m = _mesh(case)
    s.dt = m.dt
    s.ctx = dm.dg_init_mesh(m.config(case["form"]), torch.cuda.current_stream())
    dm.dg_set_base_state(s.ctx, m.node, m.face)
    if case["gamma"]:
        dm.dg_set_stabilisation(s.ctx, case["gamma"], SIGMA, *SPONGE)
    s.U = m.initial(seed, "cuda").to(real)
    if case["kind"] == "host":
        s.U = s.U.cpu().pin_memory()
        s.out = torch.empty_like(s.U).pin_memory()
    else:
        s.out = torch.empty_like(s.U)
    if case["kind"] == "adjoint":
        s.lam = _adjoint_input(m, seed, "cuda")
    return s


def _adjoint_input(m, seed, dev):
    """A smooth functional's gradient with every field's own scale."""
    g = torch.Generator(device=dev).manual_seed(seed + 77)
    lam = torch.randn(m.shape, generator=g, device=dev, dtype=torch.float64)
    scale = torch.tensor([1.0] * m.im + [1.0e-1] * m.dim + [1.0e-5], dtype=torch.float64, device=dev)
    return lam * scale.reshape((-1,) + (1,) * (2 * m.dim))


def run(s):
    kind = s.case["kind"]
    if kind == "rhs":
        dm.dg_rhs(s.ctx, s.U, s.out)
    elif kind == "steps":
        dm.dg_set_state(s.ctx, s.U, dm.DG_DEVICE)
        dm.dg_step_async(s.ctx, s.dt, s.case["steps"])
        dm.dg_get_state(s.ctx, s.out, dm.DG_DEVICE)
    elif kind == "host":
        dm.dg_set_state(s.ctx, s.U.numpy(), dm.DG_HOST)
        dm.dg_step_to_host(s.ctx, s.dt, s.case["steps"], s.out.numpy())
    elif kind == "adjoint":
        dm.dg_adjoint_step(s.ctx, s.dt, s.U, s.lam, s.out)
    else:
        s.stream.wait_stream(torch.cuda.current_stream())
        dm.dg_ensemble_step_async(s.ens, s.case["steps"])
        for ctx, out in zip(s.member, s.out):
            dm.dg_get_state(ctx, out, dm.DG_DEVICE)
        torch.cuda.current_stream().wait_stream(s.stream)
    return s.out


def work(case):
    """A stage reads and writes the state once and reads U^n once in four; its operations are those of
    the discretisation: sum-factorised volume term, lift, traces, fluxes, sources, split and update.
    The reversed step is three stages and four transposed right-hand sides of twice a stage's work."""
    if case["kind"] == "ensemble":
        each = [(m, case["steps"]) for m in _members(case)]
    else:
        each = [(_mesh(case), case["steps"])]
    size = 4.0 if case["form"] in ("bulk", "pert") else 8.0
    stages = {"rhs": 1.0, "adjoint": 11.0}.get(case["kind"])
    got = {"bytes": 0.0, "flops": 0.0}
    for m, steps in each:
        d, nf, p1 = m.dim, m.nf, m.p1
        flops = 2 * d * nf * p1 + 4 * d * nf + 4 * (d * (nf + 2) + 1) + (6 + d) + d * (5 + d) + (8 + 4 * d) + 30
        flops += 2 * d + 49 + (2 * (31 + 2 * d) + 1 + 5 * nf + 2 * (8 + 4 * d) / d) * d / p1 + 3.5 * nf
        k = 4.0 * steps if stages is None else stages
        got["flops"] += k * flops * m.nodes
        got["bytes"] += k * 2.25 * nf * size * m.nodes
    return got


# ---------------------------------------------------------------------------
# exact: the same discretisation in plain float64 torch
# ---------------------------------------------------------------------------
def _root(r, n):
    """max(r, 0)^(1/n), differentiated at max(r, FLOOR)."""
    pos = r.detach().clamp(min=0.0)
    der = torch.where(r.detach() > 0.0, pos.clamp(min=FLOOR) ** (1.0 / n - 1.0) / n, torch.zeros_like(pos))
    return pos ** (1.0 / n) + der * (r - r.detach())


def _fall_speed(rm, rr):
    """Terminal speed of rain; 0 where there is no rain or no water."""
    rw = rm + rr
    return torch.where(rw > 0.0, VR0 * rw.clamp(min=1e-300) ** -0.125 * _root(rr, 8), torch.zeros_like(rw))


def _split(m, U, base):
    """T, rho_v, p' of the implicit condensation at the nodes."""
    rd, rm, rr = base[0] + U[0], base[1] + U[1], U[2] if m.rain else torch.zeros_like(U[0])
    re = base[2] + U[-1] - sum(U[m.im + j] ** 2 for j in range(m.dim)) / (2.0 * (rd + rm + rr))
    Tu = TREF + (re - rm * LAT) / (CVD * rd + CVV * rm + CL * rr)
    sat = rm > _rho_vs(Tu)

    def H(T, d, e, q, f):
        rvs = _rho_vs(T)
        return (CVD * d + CVV * rvs + CL * (q - rvs + f)) * (T - TREF) + rvs * LAT - e, rvs

    args = [v.detach() for v in (rd, re, rm, rr)]
    T = Tu.detach().clone()
    for _ in range(8):                     # increasing and convex: Newton from the left of the root
        h, rvs = H(T, *args)
        dr = rvs * ((ES_A - 1.0) / T + ES_B / T ** 2)
        dh = CVD * args[0] + CVV * rvs + CL * (args[2] - rvs + args[3]) + ((CVV - CL) * (T - TREF) + LAT) * dr
        T = T - h / dh
    T = torch.where(sat, T - H(T, rd, re, rm, rr)[0] / dh, Tu)   # the last step carries the derivative
    rv = torch.where(sat, _rho_vs(T), rm)
    return T, rv, (rd * RD + rv * RV) * T - base[3], sat


def _flux(m, j, U, b, T, rv, pp):
    """Flux along e_j and the wave speed of states U with base b = [rho_d, rho_m, E, p]."""
    vert = j == m.dim - 1
    rd, rm = b[0] + U[0], b[1] + U[1]
    rr = U[2] if m.rain else torch.zeros_like(rd)
    rho = rd + rm + rr
    u = [U[m.im + i] / rho for i in range(m.dim)]
    F = [rd * u[j], rm * u[j]] + ([rr * u[j]] if m.rain else [])
    F += [U[m.im + i] * u[j] + (pp if i == j else 0.0) for i in range(m.dim)]
    F.append((b[2] + U[-1] + b[3] + pp) * u[j])
    cv = CVD * rd + CVV * rv + CL * (rm - rv + rr)
    lam = u[j].abs() + torch.sqrt((cv + RD * rd + RV * rv) / cv * (b[3] + pp) / rho)
    if m.rain and vert:
        vr = _fall_speed(rm, rr)
        q = rr * vr
        F[2] = F[2] - q
        for i in range(m.dim):
            F[m.im + i] = F[m.im + i] - q * u[i]
        F[-1] = F[-1] - (CL * (T - TREF) + 0.5 * sum(v * v for v in u)) * q
        lam = lam + vr.abs()
    return F, lam


def _rhs(m, U, gamma=0.0):
    dev = U.device
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    base = [m.levels(b, dev) for b in m.node]
    T, rv, pp, sat = _split(m, U, base)
    R = [torch.zeros_like(T) for _ in range(m.nf)]

    def along(M, v, j):                    # a matrix or a row applied along the nodes of direction j
        v = torch.movedim(v, m.na(j), -1) @ M.T
        return torch.movedim(v, -1, m.na(j)) if M.dim() == 2 else v

    def trace(row, v, j):                  # nodal field -> value on the face, the node axis kept with size 1
        return (torch.movedim(v, m.na(j), -1) @ row).unsqueeze(m.na(j))

    alpha = _alpha(m, U, base, gamma) if gamma else None
    for j in range(m.dim):
        s, ea = 2.0 / m.h[j], m.ea(j)
        F, _ = _flux(m, j, U, base, T, rv, pp)
        if gamma:
            F = [f - alpha.nodes(i) * s * along(t(m.D), U[i], j) for i, f in enumerate(F)]
        lo = [trace(t(m.lm), v, j) for v in list(U) + [T, rv, pp]]
        hi = [trace(t(m.lp), v, j) for v in list(U) + [T, rv, pp]]
        first, last = (lambda v: v.narrow(ea, 0, 1)), (lambda v: v.narrow(ea, m.n[j] - 1, 1))
        sign = [(-1.0 if i == m.im + j else 1.0) for i in range(len(lo))]
        if m.periodic[j]:
            left = [torch.cat([last(b), b], ea) for b in hi]
            right = [torch.cat([a, first(a)], ea) for a in lo]
        else:
            left = [torch.cat([g * first(a), b], ea) for g, a, b in zip(sign, lo, hi)]
            right = [torch.cat([a, g * last(b)], ea) for g, a, b in zip(sign, lo, hi)]
        fb = base
        if j == m.dim - 1:
            shape = [1] * (2 * m.dim)
            shape[0] = m.n[j] + 1
            fb = [t(b).reshape(shape) for b in m.face]
        Fl, ll = _flux(m, j, left[:m.nf], fb, *left[m.nf:])
        Fr, lr = _flux(m, j, right[:m.nf], fb, *right[m.nf:])
        lam = torch.where(ll > lr, ll, lr)
        Gf = [0.5 * (a + b) + 0.5 * lam * (x - y) for a, b, x, y in zip(Fl, Fr, left, right)]
        Sf = None
        if gamma:
            # interior penalty on interior faces; walls carry no diffusive flux
            sig = SIGMA * m.k ** 2 / m.h[j]
            inner = torch.ones(m.n[j] + 1, dtype=torch.float64, device=dev)
            if not m.periodic[j]:
                inner[0] = inner[-1] = 0.0
            shape = [1] * (2 * m.dim)
            shape[ea] = m.n[j] + 1
            Sf = []
            for i in range(m.nf):
                dl, dh = s * trace(t(m.dlm), U[i], j), s * trace(t(m.dlp), U[i], j)
                dl, dh = torch.cat([dl, first(dl)], ea), torch.cat([last(dh), dh], ea)
                al = alpha.faces(i, j) * inner.reshape(shape)
                jump = left[i] - right[i]
                Gf[i] = Gf[i] + al * (sig * jump - 0.5 * (dl + dh))
                Sf.append(0.5 * al * jump)
        node = [1] * (2 * m.dim)
        node[m.na(j)] = m.p1
        row = lambda a: t(a).reshape(node)  # noqa: E731
        for i in range(m.nf):
            below, above = Gf[i].narrow(ea, 0, m.n[j]), Gf[i].narrow(ea, 1, m.n[j])
            R[i] = R[i] + s * (along(t(m.dhat), F[i], j) + row(m.lm / m.w) * below - row(m.lp / m.w) * above)
            if gamma:
                below, above = Sf[i].narrow(ea, 0, m.n[j]), Sf[i].narrow(ea, 1, m.n[j])
                R[i] = R[i] + s * s * (row(m.dlm / m.w) * below + row(m.dlp / m.w) * above)
    rp = U[0] + U[1]
    if m.rain:
        x = _root(U[2], 16)
        rc = base[1] + U[1] - rv
        deficit = _rho_vs(T) - rv
        deficit = torch.where(sat, deficit - deficit.detach(), deficit)
        gm = (3.86e-3 - 9.41e-5 * (T - TREF)) * (1.0 + 9.1 * x ** 3) * deficit * x ** 8
        gm = gm - 1.0e-3 * rc.clamp(min=0.0) - 1.72 * rc * x ** 14
        R[1], R[2], rp = R[1] + gm, R[2] - gm, rp + U[2]
    vert = m.im + m.dim - 1
    R[vert] = R[vert] - G * rp
    R[-1] = R[-1] - G * U[vert]
    return torch.stack(R)


class _alpha:
    """The continuous diffusion coefficients: element values gamma h/2 rms|w|, the mean over the elements
    at each vertex, the multilinear interpolant in the element."""

    def __init__(self, m, U, base, gamma):
        self.m, dev = m, U.device
        rr = U[2] if m.rain else 0.0
        rho = base[0] + U[0] + base[1] + U[1] + rr
        u = [U[m.im + j] / rho for j in range(m.dim)]
        ur = list(u)
        if m.rain:
            ur[-1] = ur[-1] - _fall_speed(base[1] + U[1], rr)
        h = float(np.prod(m.h)) ** (1.0 / m.dim)
        wt = torch.ones((), dtype=torch.float64, device=dev)
        for j in range(m.dim):
            s = [1] * (2 * m.dim)
            s[m.na(j)] = m.p1
            wt = wt * torch.from_numpy(0.5 * m.w).to(dev).reshape(s)
        nodes = tuple(range(m.dim, 2 * m.dim))
        self.v = []
        for w in (u, ur):
            a = 0.5 * gamma * h * torch.sqrt((wt * sum(x * x for x in w)).sum(nodes))
            cnt = torch.ones_like(a)
            for j in range(m.dim):
                ea = m.ea(j)
                if m.periodic[j]:
                    lo = lambda y: torch.cat([y.narrow(ea, m.n[j] - 1, 1), y], ea)  # noqa: E731
                    hi = lambda y: torch.cat([y, y.narrow(ea, 0, 1)], ea)  # noqa: E731
                else:
                    zero = lambda y: torch.zeros_like(y.narrow(ea, 0, 1))  # noqa: E731
                    lo, hi = (lambda y: torch.cat([zero(y), y], ea)), (lambda y: torch.cat([y, zero(y)], ea))
                a, cnt = lo(a) + hi(a), lo(cnt) + hi(cnt)
            self.v.append(a / cnt)         # n_j + 1 vertices per direction, the last a copy if periodic
        self.t = torch.from_numpy(0.5 * (1.0 + m.x)).to(dev)

    def interp(self, i, skip):
        m = self.m
        a = self.v[1 if m.rain and i == 2 else 0]
        a = a.reshape(tuple(a.shape) + (1,) * m.dim)
        for j in range(m.dim):
            if j == skip:
                continue
            s = [1] * (2 * m.dim)
            s[m.na(j)] = m.p1
            t, ea = self.t.reshape(s), m.ea(j)
            a = (1.0 - t) * a.narrow(ea, 0, m.n[j]) + t * a.narrow(ea, 1, m.n[j])
        return a

    def nodes(self, i):
        return self.interp(i, None)

    def faces(self, i, j):
        return self.interp(i, j)


def _step(m, U, gamma=0.0):
    dt = m.dt
    u1 = U + 0.5 * dt * _rhs(m, U, gamma)
    u2 = u1 + 0.5 * dt * _rhs(m, u1, gamma)
    u3 = (2.0 / 3.0) * U + (1.0 / 3.0) * u2 + (dt / 6.0) * _rhs(m, u2, gamma)
    U = u3 + 0.5 * dt * _rhs(m, u3, gamma)
    if gamma:
        z = m.coords(m.dim - 1, U.device)
        dl = 0.5 * SPONGE[1] * (1.0 - torch.cos(math.pi * (z - SPONGE[0]) / (TOP - SPONGE[0])))
        dl = torch.where(z >= SPONGE[0], dl, torch.zeros_like(dl))
        moved = dl * U[1] + (dl * U[2] if m.rain else 0.0)
        U = torch.cat([(U[0] + moved)[None], (1.0 - dl) * U[1:]])
    return U


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    real = torch.float32 if case["form"] in ("bulk", "pert") else torch.float64
    if case["kind"] == "ensemble":
        out = []
        for i, m in enumerate(_members(case)):
            U = m.initial(seed * 64 + i, dev).to(real).double()
            for _ in range(case["steps"]):
                U = _step(m, U)
            out.append(U)
        return out
    m = _mesh(case)
    U = m.initial(seed, dev).to(real).double()
    if case["kind"] == "rhs":
        return _rhs(m, U)
    if case["kind"] == "adjoint":
        U.requires_grad_(True)
        return torch.autograd.grad(_step(m, U), U, _adjoint_input(m, seed, dev))[0]
    for _ in range(case["steps"]):
        U = _step(m, U, case["gamma"])
    return U
