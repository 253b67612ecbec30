"""The work a user of this framework has it do, as cases to be timed and compared.

A case is one call (or the two or three calls that a program makes together)
through the Python entry points, on one of the meshes this repository solves:

  solve     residual, linearization and FGMRES solve: one Newton linear system
            (the README's example), at a seeded linearization state
  step      one backward-Euler step by Newton, in place on the state (the
            transient of bench.py)
  adjoint   linearization, transposed solve, parameter gradient and the
            coupling to the previous time level: one step of the reverse sweep
  operator  residual, J x and J^T x on given vectors: what a caller with its
            own Krylov method uses
  gradient  terminal voltage after a few steps and its gradient through
            torch.autograd, the handle's setup included
  batch     one Newton linear system in each of several gyroid cells of uneven
            sizes, solved in lockstep

`exact` states the discrete equations once more in plain torch, in 64 bits
(element matrices, Butler-Volmer kinetics, radial finite differences) and
solves them with dense factorizations where the cell is small enough.
"""
import math

import numpy as np
import torch

from p4d_inputs import make_box_case, make_gyroid_cell, make_slab_case, make_tpms_cell
from paper_2602_07225_gb300 import BatchSolver, P4DSolver, terminal_voltage

LAYERS_M = (100e-6, 25e-6, 100e-6)   # anode, separator, cathode thickness
NEWTON = dict(rtol=1e-8, maxit=20)
FIELDS = ("phis", "phie", "ce", "cs")


def listed():
    return [
        # the smallest cell in use (smoke test, unit tests): launches and latency
        dict(name="solve_cube8", kind="solve", nx=8, ny=8, na=10, ns=4, nr=10, hetero=False, precision=1, mode=1,
             combine=0, rtol=1e-8),
        # one time step of a small cell with odd sizes under the paper's material laws
        dict(name="step_laws_small", kind="step", nx=13, ny=11, na=7, ns=3, nr=8, hetero=True, laws=1, precision=1),
        # gradient of the terminal voltage through autograd, setup included
        dict(name="gradient_small", kind="gradient", nx=21, ny=18, na=8, ns=3, nr=8, steps=3),
        # the precision study's middle size: heterogeneous porosity and particle radii
        dict(name="solve_hetero64", kind="solve", nx=64, ny=64, na=20, ns=8, nr=10, hetero=True, precision=1, mode=1,
             combine=0, rtol=1e-8),
        # the FP64 preconditioner with Krylov vectors over every unknown (reference accuracy)
        dict(name="solve_fp64_full", kind="solve", nx=40, ny=36, na=15, ns=6, nr=12, hetero=False, precision=0, mode=0,
             combine=0, rtol=1e-10),
        # block Gauss-Seidel with BF16 coarse-level stencils, ragged sizes
        dict(name="solve_bgs_bf16", kind="solve", nx=73, ny=57, na=22, ns=9, nr=12, hetero=True, precision=2, mode=1,
             combine=1, rtol=1e-8),
        # the paper's interpenetrating gyroid electrodes (Case IV), N_c = 6
        dict(name="solve_tpms", kind="solve", tpms=True, nx=64, ny=64, na=32, ns=0, nr=6, hetero=False, precision=1,
             mode=1, combine=0, rtol=1e-8),
        # a batch of gyroid cells of uneven sizes (a slice of the 64-cell batch)
        dict(name="batch_gyroid", kind="batch", cells=10, nmax=48),
        # one step of the reverse sweep on the jelly-roll slab with tabs
        dict(name="adjoint_slab", kind="adjoint", nx=512, ny=16, na=20, ns=8, nr=15),
        # a time step of a middle-sized cell with odd sizes under the paper's material laws
        dict(name="step_laws", kind="step", nx=75, ny=61, na=27, ns=11, nr=15, hetero=True, laws=1, precision=1),
        # the bare operator at the profiling size
        dict(name="operator_cube96", kind="operator", nx=96, ny=96, na=30, ns=12, nr=20),
        # the headline workload: one backward-Euler step of the 128 x 128 x 96 cube, 32.1M unknowns
        dict(name="step_cube128", kind="step", nx=128, ny=128, na=40, ns=16, nr=20, hetero=False, laws=0, precision=1),
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    kind = rng.choice(("solve", "solve", "solve", "step", "step", "adjoint", "operator", "batch", "gradient"))
    if kind == "batch":
        return dict(kind="batch", cells=rng.randint(3, 12), nmax=rng.choice((24, 32, 40, 48)))
    if kind == "gradient":
        nx = log_int(8, 40)
        return dict(kind="gradient", nx=nx, ny=max(6, nx - rng.randint(0, nx // 3)), na=max(5, nx // 3),
                    ns=rng.randint(2, 5), nr=rng.randint(5, 12), steps=rng.randint(2, 4))
    if kind == "adjoint":
        return dict(kind="adjoint", nx=log_int(48, 640), ny=rng.randint(5, 18), na=rng.randint(8, 20),
                    ns=rng.randint(3, 8), nr=rng.randint(6, 18))
    if kind == "solve" and rng.random() < 0.2:
        n = log_int(24, 72)
        return dict(kind="solve", tpms=True, nx=n, ny=n, na=n // 2, ns=0, nr=rng.randint(5, 8), hetero=False,
                    precision=rng.choice((1, 1, 2)), mode=1, combine=0, rtol=1e-8)
    nx = log_int(8, 104)
    size = dict(nx=nx, ny=max(6, nx - rng.randint(0, nx // 3)), na=max(5, int(0.33 * nx) + rng.randint(-2, 3)),
                ns=max(2, int(0.13 * nx) + rng.randint(-1, 2)), nr=rng.randint(5, 20))
    if kind == "operator":
        return dict(kind="operator", **size)
    if kind == "step":
        return dict(kind="step", hetero=rng.random() < 0.5, laws=rng.choice((0, 1)), precision=rng.choice((1, 1, 2)),
                    **size)
    precision = rng.choice((0, 1, 1, 1, 2))
    return dict(kind="solve", hetero=rng.random() < 0.5, precision=precision, mode=rng.choice((0, 1, 1)),
                combine=rng.choice((0, 0, 1)), rtol=1e-8 if precision else 1e-10, **size)


# ------------------------------------------------------------------ inputs
def _box(case, seed, state):
    return make_box_case(case["nx"], case["ny"], (case["na"], case["ns"], case["na"]), 100e-6, LAYERS_M, case["nr"],
                         seed, hetero=bool(case.get("hetero")), rs_cv=0.3 if case.get("hetero") else 0.0, state=state)


def _in_discharge(cell, rng):
    """A cell somewhere in a discharge: seeded rate and stoichiometries, smooth
    concentration profiles, open-circuit potentials of the mean composition."""
    m, p, st = cell["mesh"], cell["params"], cell["state"]
    nn = st["phis"].size
    dims = (m["nz"] + 1, m["ny"] + 1, m["nx"] + 1)
    z, y, x = (np.linspace(0.0, 1.0, n) for n in dims)
    a = rng.uniform(0.0, 2.0 * np.pi, 3)
    wave = (np.cos(np.pi * z + a[0])[:, None, None] * np.cos(2 * np.pi * y + a[1])[None, :, None]
            * np.cos(2 * np.pi * x + a[2])[None, None, :]).ravel()
    p["i_app"] *= rng.uniform(0.7, 1.5)
    th_n, th_p = rng.uniform(0.65, 0.8), rng.uniform(0.45, 0.6)
    anode = st["phis"] == 0.0      # the generator's anode (and separator) potential
    st["cs_node"] = np.where(anode, th_n * p["cmax_n"], th_p * p["cmax_p"])[:, None] * (1 + 2e-3 * wave)[:, None] \
        * np.ones(m["nc"])
    u_n = p["ocp_n"][0] + p["ocp_n"][1] * th_n
    u_p = p["ocp_p"][0] + p["ocp_p"][1] * th_p
    st["ce"] = 1000.0 * (1 + 2e-2 * wave)
    st["phie"] = np.full(nn, -u_n) + 1e-3 * wave
    st["phis"] = np.where(anode, 0.0, u_p - u_n)
    st["ce_prev"], st["cs_prev_node"] = st["ce"].copy(), st["cs_node"].copy()
    return cell


def _cell(case, seed):
    """The cell of a case (mesh, parameters, state), from the seed alone."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "adjoint":
        cell = make_slab_case(nx=case["nx"], ny=case["ny"], layers=(case["na"], case["ns"], case["na"]), nc=case["nr"],
                              seed=seed, tab=max(4, case["nx"] // 32))
        return _in_discharge(cell, rng)
    if case["kind"] in ("step", "gradient"):
        return _in_discharge(_box(case, seed, "initial"), rng)
    if case.get("tpms"):
        return make_tpms_cell(case["nx"], case["ny"], case["na"], nc=case["nr"], seed=seed)
    return _box(case, seed, "seeded")


def _options(case):
    if case["kind"] == "step":
        return dict(precision=case["precision"], mode=1, combine=0, rtol=1e-8, restart=30, maxit=600, cgs_refine=0,
                    ocp_model=case["laws"], transport_model=case["laws"])
    if case["kind"] == "adjoint":
        return dict(precision=1, mode=1, combine=0, rtol=1e-10, restart=100, maxit=1500)
    if case["kind"] == "operator":
        return dict(precision=1)
    return dict(precision=case["precision"], mode=case["mode"], combine=case["combine"], rtol=case["rtol"], maxit=600)


def _materials(cell):
    """Per-element bulk conductivity, solid diffusivity and porosity of a cell
    with poorly conducting electrodes: at the default conductivities the
    voltage's sensitivity to sigma lies at the rounding of the time steps."""
    m, p = cell["mesh"], cell["params"]
    sig = 1e-2 * np.where(m["region"] == 0, p["sigma_n"], np.where(m["region"] == 2, p["sigma_p"], 0.0))
    return sig, np.full(sig.size, float(m["Ds"][0])), np.asarray(m["eps"], float)


def _vectors(case, seed, ndof, nn, device):
    """Two vectors of the size of a Newton step and of an adjoint."""
    g = torch.Generator(device=device).manual_seed(seed)
    x, lam = (torch.randn(ndof, generator=g, device=device, dtype=torch.float64) for _ in range(2))
    x[: 2 * nn] *= 1e-3
    x[2 * nn:3 * nn] *= 10.0
    x[3 * nn:] *= 100.0
    return x, lam


def _split(v, nn):
    """The fields of a vector in the full layout (views)."""
    return dict(phis=v[:nn], phie=v[nn:2 * nn], ce=v[2 * nn:3 * nn], cs=v[3 * nn:])


def _gyroids(case, seed):
    rng = np.random.default_rng(seed)
    sizes = [n for n in (16, 24, 32, 40, 48) if n <= case["nmax"]]
    # the sizes and level sets in turn, so that neither work nor shapes depend on the seed
    return [make_gyroid_cell(sizes[i % len(sizes)], (i % 7 - 3) / 10, 1 + i % 3, 10 + (3 * i) % 11,
                             int(rng.integers(1 << 30))) for i in range(case["cells"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(kind=kind, batch=BatchSolver(_gyroids(case, seed), threads=16, autotune=False, precision=1, mode=1,
                                                 rtol=1e-8, maxit=600))
    cell = _cell(case, seed)
    if kind == "gradient":
        leaves = [torch.tensor(a, device="cuda", requires_grad=True) for a in _materials(cell)]
        return dict(kind=kind, cell=cell, leaves=leaves, steps=case["steps"])
    s = P4DSolver(cell, **_options(case))
    st = s.state_tensors(cell["state"])
    out = dict(kind=kind, solver=s, state=st)
    if kind == "step":
        out["start"] = {k: v.clone() for k, v in st.items()}
    if kind == "adjoint":
        g = torch.Generator(device="cuda").manual_seed(seed)
        st["phis"] += 1e-2 * torch.randn(s.nn, generator=g, device="cuda", dtype=torch.float64)
        out["rhs"] = s.voltage_weights()
    if kind == "operator":
        out["x"], out["lam"] = _vectors(case, seed, s.ndof, s.nn, "cuda")
        s.jacobian_update(st)
    return out


# ------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind == "batch":
        return [x for x, _ in state["batch"].solve_all()]
    if kind == "gradient":
        for t in state["leaves"]:
            t.grad = None
        v = terminal_voltage(*state["leaves"], state["cell"], state["steps"], checkpoint=2)
        v.backward()
        sigma, Ds, eps = (t.grad for t in state["leaves"])
        return dict(v=v.detach(), sigma=sigma, Ds=Ds, eps=eps)
    s, st = state["solver"], state["state"]
    if kind == "solve":
        b = s.residual(st).neg_()
        s.jacobian_update(st)
        x, _ = s.solve(b)
        return _split(x, s.nn)
    if kind == "step":
        for k, v in state["start"].items():
            st[k].copy_(v)
        s.newton(st, **NEWTON)
        return {k: st[k] for k in FIELDS}
    if kind == "adjoint":
        s.jacobian_update(st)
        lam, _ = s.solve(state["rhs"], adjoint=True)
        g = [torch.zeros(s._nelem, dtype=torch.float64, device="cuda") for _ in range(3)]
        s.param_grad(st, lam, *g)
        prev = s.adjoint_prev(lam)
        return dict(lam=_split(lam, s.nn), sigma=g[0], Ds=g[1], eps=g[2], prev_ce=prev[2 * s.nn:3 * s.nn],
                    prev_cs=prev[3 * s.nn:])
    r = s.residual(st)
    y, yt = s.jvp(state["x"]), s.jvp(state["lam"], transpose=True)
    return dict(r=_split(r, s.nn), y=_split(y, s.nn), yt=_split(yt, s.nn))


def work(case):
    """Inputs read once, outputs written once: the state's vectors in, the
    result's out, the mesh's element data; flops of one operator application
    (27-point stencils of three fields, five operations per radial node)."""
    if case["kind"] == "batch":
        sizes = [n for n in (16, 24, 32, 40, 48) if n <= case["nmax"]]
        cells = [(sizes[i % len(sizes)], 10 + (3 * i) % 11) for i in range(case["cells"])]
        dims = [(n, n, 3 * n // 2, 20 * (3 * n // 2) // 24, nr) for n, nr in cells]
    elif case.get("tpms"):
        dims = [(case["nx"], case["ny"], case["na"], case["na"] // 2, case["nr"])]
    else:
        dims = [(case["nx"], case["ny"], 2 * case["na"] + case["ns"], 2 * case["na"], case["nr"])]
    nbytes = flops = 0.0
    for nx, ny, nz, nz_el, nr in dims:
        nn, ncs = (nx + 1) * (ny + 1) * (nz + 1), (nx + 1) * (ny + 1) * (nz_el + 1) * nr
        vec = 8.0 * (3 * nn + ncs)
        vectors = dict(solve=2.2, step=2.2, adjoint=3.5, operator=6.2, gradient=2.2, batch=2.2)[case["kind"]]
        nbytes += vectors * vec + 26.0 * nx * ny * nz
        flops += (162.0 * nn + 10.0 * ncs) * dict(operator=3, gradient=2 * case.get("steps", 1)).get(case["kind"], 1)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64 bits
class _Exact:
    """The discrete equations in plain torch: all arrays (nz, ny, nx) or
    (nz + 1, ny + 1, nx + 1), one particle per electrode node."""

    def __init__(self, cell, laws, device):
        m, p = cell["mesh"], cell["params"]
        self.p, self.laws, self.dev = p, laws, device
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device=device)
        nx, ny, nz = m["nx"], m["ny"], m["nz"]
        self.ne, self.nd = (nz, ny, nx), (nz + 1, ny + 1, nx + 1)
        self.nn = (nz + 1) * (ny + 1) * (nx + 1)
        hx, hy, hz = t(m["hx"])[None, None, :], t(m["hy"])[None, :, None], t(m["hz"])[:, None, None]
        one = torch.ones(self.ne, dtype=torch.float64, device=device)
        self.vol = hx * hy * hz * one
        self.geo = torch.stack([hy * hz / hx * one, hx * hz / hy * one, hx * hy / hz * one])
        # 8 x 8 element matrices of the three stiffness directions and the mass
        k1 = torch.tensor([[1.0, -1.0], [-1.0, 1.0]], dtype=torch.float64)
        m1 = torch.tensor([[1 / 3, 1 / 6], [1 / 6, 1 / 3]], dtype=torch.float64)
        kron = lambda c, b, a: torch.kron(c, torch.kron(b, a)).to(device)
        self.S = torch.stack([kron(m1, m1, k1), kron(m1, k1, m1), kron(k1, m1, m1)])
        self.M = kron(m1, m1, m1)
        region = torch.as_tensor(np.asarray(m["region"]).astype(np.int64), device=device).view(self.ne)
        self.eps, eps_s = t(m["eps"]).view(self.ne), t(m["eps_s"]).view(self.ne)
        el = (region == 0) | (region == 2)
        two = lambda flag, a, b: torch.where(flag, t(a), t(b))
        sig = two(region == 0, p["sigma_n"], p["sigma_p"])
        if m.get("sigma_e") is not None:
            sig = t(m["sigma_e"]).view(self.ne)
        self.csig = torch.where(el, eps_s ** p["brug"] * sig, torch.zeros_like(sig))
        self.epb = self.eps ** p["brug"]
        node = lambda e: self._gather((e.double() * one)[None].expand(8, *self.ne)) > 0
        self.anode, cathode = node(region == 0), node(region == 2)
        self.el = self.anode | cathode
        ground = torch.zeros(self.nd, dtype=torch.bool, device=device)
        gn = torch.as_tensor(np.asarray(m["gamma_n"]).astype(bool), device=device).view(ny, nx)
        gp = torch.as_tensor(np.asarray(m["gamma_p"]).astype(np.float64), device=device).view(ny, nx)
        self.gpw = torch.zeros(self.nd, dtype=torch.float64, device=device)
        a4 = gp * hx[0] * hy[0] / 4
        for b in (0, 1):
            for a in (0, 1):
                ground[0, b:b + ny, a:a + nx] |= gn
                self.gpw[nz, b:b + ny, a:a + nx] += a4
        self.act = self.el & ~ground
        v8 = torch.where(el, self.vol / 8, torch.zeros_like(self.vol))[None].expand(8, *self.ne)
        Mn, Sn = self._gather(v8), self._gather(v8 * eps_s)
        self.enodes = torch.nonzero(self.el.reshape(-1)).view(-1)
        pick = lambda a: a.reshape(-1)[self.enodes]
        R, D = pick(t(m["Rs"])), pick(t(m["Ds"]))
        if m.get("Ds_e") is not None:
            D = pick(self._gather(v8 * t(m["Ds_e"]).view(self.ne))) / pick(Mn)
        self.Mj, self.kap = pick(Mn), D / (R * R)
        self.Aj = 3 * pick(Sn) / R
        self.an_j = pick(self.anode)
        self.k = two(self.an_j, p["k_n"], p["k_p"])
        self.cmax = two(self.an_j, p["cmax_n"], p["cmax_p"])
        r, nc = t(m["rgrid"]), m["nc"]
        L = torch.zeros(nc, nc, dtype=torch.float64, device=device)
        L[0, 0], L[0, 1] = -6 / r[1] ** 2, 6 / r[1] ** 2
        for i in range(1, nc - 1):
            dp, dm = r[i + 1] - r[i], r[i] - r[i - 1]
            th = dp / dm
            c1, c2 = 2 / (r[i] * dp * (1 + th)), 2 / (dp * dm * (1 + th))
            L[i, i - 1], L[i, i], L[i, i + 1] = -c1 * th ** 2 + c2 * th, -c1 * (1 - th ** 2) - c2 * (1 + th), c1 + c2
        dr = r[nc - 1] - r[nc - 2]
        L[nc - 1, nc - 2], L[nc - 1, nc - 1] = 2 / dr ** 2, -2 / dr ** 2
        self.L, self.nc = L, nc
        self.beta = 2 * (1 + dr) / (p["F"] * dr) / R
        self.gamma = p["diffpot_sign"] * 2 * p["R"] * p["T"] * (1 - p["tplus"]) / p["F"]
        self.tau = (1 - p["tplus"]) / p["F"]

    # element corner views of a node field, and the sum of corner values into nodes
    def _corners(self, u):
        nz, ny, nx = self.ne
        return torch.stack([u[c:c + nz, b:b + ny, a:a + nx] for c in (0, 1) for b in (0, 1) for a in (0, 1)])

    def _gather(self, v):
        pad = torch.nn.functional.pad
        return sum(pad(v[a + 2 * b + 4 * c], (a, 1 - a, b, 1 - b, c, 1 - c))
                   for c in (0, 1) for b in (0, 1) for a in (0, 1))

    def _stiff(self, coef, u):
        v = self._corners(u)
        w = sum(self.geo[d] * torch.einsum("lm,mzyx->lzyx", self.S[d], v) for d in range(3))
        return self._gather(coef * w)

    def _ocp(self, th):
        p = self.p
        if not self.laws:
            lin = lambda c: c[0] + c[1] * th
            return torch.where(self.an_j, lin(p["ocp_n"]), lin(p["ocp_p"]))
        q, tanh = 1.062 * th, torch.tanh
        up = (2.16216 + 0.07645 * tanh(30.834 - 54.4806 * q) + 2.1581 * tanh(52.294 - 50.294 * q)
              - 0.14169 * tanh(11.0923 - 19.8543 * q) + 0.2051 * tanh(1.4684 - 5.4888 * q)
              + 0.2531 * tanh((-q + 0.56478) / 0.1316) - 0.02167 * tanh((q - 0.525) / 0.006))
        un = (0.194 + 1.5 * torch.exp(-120.0 * th) + 0.0351 * tanh((th - 0.286) / 0.083)
              - 0.0045 * tanh((th - 0.849) / 0.119) - 0.035 * tanh((th - 0.9233) / 0.05)
              - 0.0147 * tanh((th - 0.5) / 0.034) - 0.102 * tanh((th - 0.194) / 0.142)
              - 0.022 * tanh((th - 0.9) / 0.0164) - 0.011 * tanh((th - 0.124) / 0.0226)
              + 0.0155 * tanh((th - 0.105) / 0.029))
        return torch.where(self.an_j, un, up)

    def _transport(self, ce):
        p = self.p
        if not self.laws:
            return self.epb * p["kappa"], self.epb * p["De"]
        c = self._corners(ce).mean(0) / 1000
        dT = (1 / 298.15 - 1 / p["T"]) / p["R"]
        return (self.epb * math.exp(34700 * dT) * (0.0911 + 1.9101 * c - 1.052 * c ** 2 + 0.1554 * c ** 3),
                self.epb * math.exp(37040 * dT) * 5.34e-10 * torch.exp(-0.65 * c))

    def residual(self, u, prev):
        """R(u), u and the previous level's (c_e, c_s) in the full layout's pieces."""
        phis, phie, ce = (v.view(self.nd) for v in u[:3])
        cs, (ce0, cs0), p = u[3], prev, self.p
        e = self.enodes
        pick = lambda a: a.reshape(-1)[e]
        ph = torch.where(self.act, phis, torch.zeros_like(phis))
        cmax, s, c, f, al = self.cmax, cs[:, -1], pick(ce), p["F"] / (p["R"] * p["T"]), p["alpha"]
        eta = pick(ph) - pick(phie) - self._ocp(s / cmax)
        i0 = self.k * c ** al * (cmax - s) ** al * s ** (1 - al)
        i_n = i0 * (torch.exp(al * f * eta) - torch.exp((al - 1) * f * eta))
        ain = torch.zeros(self.nn, dtype=torch.float64, device=self.dev).index_put((e,), self.Aj * i_n).view(self.nd)
        kap, De = self._transport(ce)
        rs = torch.where(self.act, self._stiff(self.csig, ph) + ain - p["i_app"] * self.gpw, phis)
        re = self._stiff(kap, phie + self.gamma * torch.log(ce)) - ain
        mass = self._gather(self.eps * self.vol / p["dt"]
                            * torch.einsum("lm,mzyx->lzyx", self.M, self._corners(ce - ce0.view(self.nd))))
        rc = mass + self._stiff(De, ce) - self.tau * ain
        rp = self.Mj[:, None] * ((cs - cs0) / p["dt"] - self.kap[:, None] * (cs @ self.L.T))
        last = torch.zeros(self.nc, dtype=torch.float64, device=self.dev)
        last[-1] = 1.0
        rp = rp + (self.Mj * self.beta * i_n)[:, None] * last
        return rs.reshape(-1), re.reshape(-1), rc.reshape(-1), rp

    def state(self, st):
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device=self.dev)
        cs, cs0 = t(st["cs_node"])[self.enodes], t(st["cs_prev_node"])[self.enodes]
        return (t(st["phis"]), t(st["phie"]), t(st["ce"]), cs), (t(st["ce_prev"]), cs0)

    def jvp(self, u, prev, x):
        return torch.func.jvp(lambda *v: self.residual(v, prev), u, x)[1]

    def vjp(self, u, prev, y):
        return torch.func.vjp(lambda *v: self.residual(v, prev), *u)[1](y)

    def pieces(self, v):
        nn = self.nn
        return v[:nn], v[nn:2 * nn], v[2 * nn:3 * nn], v[3 * nn:].view(-1, self.nc)

    def jacobian(self, u, prev):
        """Dense macro block, and the node-local particle blocks: columns by
        products with one vector per colour of the 3 x 3 x 3 node colouring."""
        nn, nd, dev = self.nn, self.nd, self.dev
        idx = torch.arange(nn, device=dev)
        ijk = (idx // (nd[1] * nd[2]), idx // nd[2] % nd[1], idx % nd[2])
        colour = (ijk[0] % 3) * 9 + (ijk[1] % 3) * 3 + ijk[2] % 3
        zero = [torch.zeros_like(v) for v in u]
        A = torch.zeros(3 * nn, 3 * nn, dtype=torch.float64, device=dev)
        E = self.enodes.numel()
        acm = torch.zeros(E, 3, dtype=torch.float64, device=dev)
        for f in range(3):
            x = list(zero)
            x[f] = torch.ones_like(u[f])
            acm[:, f] = self.jvp(u, prev, tuple(x))[3][:, -1]
            for col in range(27):
                x[f] = (colour == col).double()
                y = self.jvp(u, prev, tuple(x))
                # the one node of this colour within reach of each node
                src = [((c - i % 3 + 1) % 3 - 1 + i) for i, c in zip(ijk, (col // 9, col // 3 % 3, col % 3))]
                ok = torch.ones(nn, dtype=torch.bool, device=dev)
                for s_, n_ in zip(src, nd):
                    ok &= (s_ >= 0) & (s_ < n_)
                col_of = (src[0] * nd[1] + src[1]) * nd[2] + src[2]
                for g in range(3):
                    A[g * nn + idx[ok], f * nn + col_of[ok]] = y[g][ok]
        x = list(zero)
        x[3] = torch.zeros_like(u[3])
        x[3][:, -1] = 1.0
        y = self.jvp(u, prev, tuple(x))
        amc = torch.stack([v[self.enodes] for v in y[:3]], 1)
        T = torch.zeros(E, self.nc, self.nc, dtype=torch.float64, device=dev)
        for i in range(self.nc):
            x[3] = torch.zeros_like(u[3])
            x[3][:, i] = 1.0
            T[:, :, i] = self.jvp(u, prev, tuple(x))[3]
        return A, amc, acm, T

    def solve(self, u, prev, b, trans=False, refine=2):
        """x with J x = b (J^T x = b): particles eliminated, dense LU of the
        equilibrated Schur complement, iterative refinement."""
        A, amc, acm, T = self.jacobian(u, prev)
        if trans:
            A, (amc, acm), T = A.T.contiguous(), (acm, amc), T.transpose(1, 2).contiguous()
        nn, e = self.nn, self.enodes
        d = T.diagonal(dim1=1, dim2=2).abs().sqrt()
        lu_t = torch.linalg.lu_factor(T / (d[:, :, None] * d[:, None, :]))
        tsolve = lambda r: torch.linalg.lu_solve(*lu_t, (r / d)[:, :, None])[:, :, 0] / d
        last = torch.zeros(e.numel(), self.nc, dtype=torch.float64, device=self.dev)
        last[:, -1] = 1.0
        z = tsolve(last)[:, -1]
        for f in range(3):
            for g in range(3):
                A[f * nn + e, g * nn + e] -= z * amc[:, f] * acm[:, g]
        dm = A.diagonal().abs().sqrt()
        lu = torch.linalg.lu_factor(A / (dm[:, None] * dm[None, :]))
        del A
        x = [torch.zeros_like(v) for v in b]
        r = list(b)
        for _ in range(1 + refine):
            yc = tsolve(r[3])
            rm = [v.clone() for v in r[:3]]
            for f in range(3):
                rm[f][e] -= amc[:, f] * yc[:, -1]
            zm = (torch.linalg.lu_solve(*lu, (torch.cat(rm) / dm)[:, None])[:, 0] / dm).split(nn)
            tN = sum(acm[:, f] * zm[f][e] for f in range(3))
            zc = yc - tsolve(last * tN[:, None])
            x = [a + v for a, v in zip(x, (*zm, zc))]
            jx = (self.vjp if trans else self.jvp)(u, prev, tuple(x))
            r = [v - w for v, w in zip(b, jx)]
        return x

    def newton(self, u, prev):
        for _ in range(7):
            d = self.solve(u, prev, self.residual(u, prev), refine=1)
            u = tuple(a - v for a, v in zip(u, d))
        return u


def _named(pieces):
    return dict(zip(FIELDS, (v.reshape(-1) for v in pieces)))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "gradient"):
        return None     # several cells, or several time steps and their reverse sweep
    nn = (case["nx"] + 1) * (case["ny"] + 1) * ((case["na"] if case.get("tpms") else 2 * case["na"] + case["ns"]) + 1)
    if kind != "operator" and nn > 4000:
        return None     # dense factorization of 3 nn unknowns
    dev = "cuda"
    cell = _cell(case, seed)
    E = _Exact(cell, case.get("laws", 0), dev)
    u, prev = E.state(cell["state"])
    if kind == "operator":
        ndof = 3 * E.nn + E.enodes.numel() * E.nc
        x, lam = _vectors(case, seed, ndof, E.nn, dev)
        return dict(r=_named(E.residual(u, prev)), y=_named(E.jvp(u, prev, E.pieces(x))),
                    yt=_named(E.vjp(u, prev, E.pieces(lam))))
    if kind == "solve":
        b = tuple(-v for v in E.residual(u, prev))
        return _named(E.solve(u, prev, b))
    if kind == "step":
        u = list(E.newton(u, prev))
        u[3] = u[3].reshape(-1, E.nc)
        return dict(zip(FIELDS, u))
    g = torch.Generator(device=dev).manual_seed(seed)
    u = (u[0] + 1e-2 * torch.randn(E.nn, generator=g, device=dev, dtype=torch.float64), *u[1:])
    q = (E.gpw / E.gpw.sum()).reshape(-1)
    b = (q, torch.zeros_like(q), torch.zeros_like(q), torch.zeros_like(u[3]))
    lam = E.solve(u, prev, b, trans=True)
    return dict(lam=_named(lam), sigma=None, Ds=None, eps=None, prev_ce=None,
                prev_cs=(lam[3] * E.Mj[:, None] / cell["params"]["dt"]).reshape(-1))
