"""The calls whose speed matters to a user of this library, each as a case that can be timed and
checked: a dictionary of plain values (``listed``, ``draw``), the state a program holds before the
call (``prepare``), one pass through the public binding (``run``), the work no implementation can
avoid (``work``) and the result in 64 bits from plain torch (``exact``).

Operations:

* ``rhs``    one ``hyp_rhs`` of a grid: what a caller with its own time integrator calls.
* ``step``   one RK3 step (three ``hyp_rk_stage``, the state filter included where the case sets
  it): the inner loop of every solve. The state advances from pass to pass, as in a solve.
* ``batch``  one step of a batch of independent solves, as the server runs between admissions.
* ``thermo`` one ``hyp_thermo_eval`` of independent states: table generation, post-processing,
  coupling to another solver. The smallest is a probe line, the largest a volume.
"""
import math

import numpy as np
import torch

from paper_2210_05547_gb300 import abi as A
from paper_2210_05547_gb300 import inputs as I

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64


def _grid(name, op, flow, nx, ny, nz=1, gas="air5", kind="cneq", precision="fp64"):
    return dict(name=name, op=op, flow=flow, nx=nx, ny=ny, nz=nz, gas=gas, kind=kind,
                precision=precision)


def _thermo(name, n, gas="air5", precision="fp64"):
    return dict(name=name, op="thermo", n=n, gas=gas, precision=precision)


def _batch(name, stream, members, precision="mixed"):
    return dict(name=name, op="batch", stream=stream, members=members, gas="air5",
                precision=precision)


def listed():
    return [
        # the smallest useful grid (the size of the smoke test): a real-time or unit-cell solve,
        # all latency and launches
        _grid("rhs_bl_32x16", "rhs", "bl", 32, 16),
        # the boundary-layer case at its own size, stepped in FP64
        _grid("step_bl_256x64", "step", "bl", 256, 64),
        # a ragged interaction grid, right-hand side for a caller's own integrator
        _grid("rhs_sbli_515x131", "rhs", "sbli", 515, 131),
        # the headline workload: the shock / boundary-layer interaction at full size
        _grid("step_sbli_2048x256", "step", "sbli", 2048, 256),
        # the same in the mixed precision that production runs use
        _grid("step_sbli_2048x256_mixed", "step", "sbli", 2048, 256, precision="mixed"),
        # ionised air: eleven species, 49 reactions
        _grid("rhs_sbli_air11_512x128", "rhs", "sbli", 512, 128, gas="air11"),
        # local thermodynamic equilibrium at the boundary-layer size
        _grid("rhs_bl_lte_256x64", "rhs", "bl", 256, 64, kind="lte"),
        # the three-dimensional jet in crossflow, half the full resolution per direction (its
        # right-hand side: at this resolution the jet cannot be stepped for long)
        _grid("rhs_jet_256x128x64", "rhs", "jet", 256, 128, 64),
        # members of the serving stream (grids 128 x 32 to 1024 x 256) stepped together
        _batch("batch_6_mixed", 100, 6),
        # closures of independent states: a probe line, a volume, ionised air
        _thermo("thermo_1200", 1200),
        _thermo("thermo_4000037", 4000037),
        _thermo("thermo_air11_300007_mixed", 300007, gas="air11", precision="mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["rhs", "rhs", "step", "thermo", "batch", "jet"])
    if op == "thermo":
        gas = rng.choice(["air5", "air5", "air11"])
        top = 4_000_000 if gas == "air5" else 1_500_000
        return dict(op="thermo", n=_log_int(rng, 1000, top), gas=gas,
                    precision=rng.choice(["fp64", "fp64", "mixed"]))
    if op == "batch":
        return dict(op="batch", stream=rng.randrange(1000), members=rng.randint(2, 8), gas="air5",
                    precision=rng.choice(["mixed", "fp64"]))
    if op == "jet":
        nz = _log_int(rng, 12, 64)
        return dict(op="rhs", flow="jet", nx=_log_int(rng, 64, 256), ny=_log_int(rng, 48, 128),
                    nz=nz, gas="air5", kind="cneq", precision="fp64")
    if op == "step":
        # the sizes of the serving stream, on which 500-2000 steps are known to stay clean
        flow = rng.choice(["bl", "sbli"])
        ny = _log_int(rng, 32, 256) if flow == "bl" else _log_int(rng, 128, 256)
        return dict(op="step", flow=flow, nx=_log_int(rng, 128, 1024), ny=ny, nz=1, gas="air5",
                    kind="cneq", precision=rng.choice(["fp64", "mixed"]))
    # right-hand sides: any size, any gas
    gas, kind = rng.choice([("air5", "cneq")] * 4 + [("air11", "cneq"), ("air5", "lte")])
    top = 2048 if (gas, kind) == ("air5", "cneq") else 640
    return dict(op="rhs", flow=rng.choice(["bl", "sbli"]), nx=_log_int(rng, 24, top),
                ny=_log_int(rng, 16, 256), nz=1, gas=gas, kind=kind, precision="fp64")


# ---------------------------------------------------------------------------------------------
# States and passes
# ---------------------------------------------------------------------------------------------

PRECISION = {"fp64": A.FP64, "mixed": A.MIXED}


def _config(case):
    """The case dictionary of a single-grid case."""
    kind = case["kind"]
    if case["flow"] == "jet":
        cfg = I.jet_case(case["nx"], case["ny"], case["nz"], 0, kind)
    elif case["flow"] == "sbli":
        cfg = I.sbli_case(case["nx"], case["ny"], 0, kind)
        if case["op"] == "step" and case["nx"] < 2048:
            cfg["dt"] = 5.0e-4                     # the time step of the serving stream's grids
    else:
        cfg = I.bl_case(case["nx"], case["ny"], 0, kind)
    return I.with_species(cfg, "air11") if case["gas"] == "air11" else cfg


def _batch_configs(case):
    return [c for c, _, _ in I.serving_requests(case["members"], seed=case["stream"])]


def _noise(n, seed):
    return np.random.default_rng([seed, n]).uniform(-1.0, 1.0, n)


def _open_state(cfg, seed):
    gas = A.gas_model_load(cfg)
    n = A.state_size(gas, cfg)
    U = torch.empty(n, dtype=F64, device=DEV)
    dQ = torch.empty_like(U)
    return gas, A.state_init(gas, cfg, U, dQ, _noise(n, seed))


def _thermo_inputs(case, seed, tab):
    """T log-uniform in [300, 15000] K, rho log-uniform in [1e-4, 1] kg/m^3, mass fractions
    Dirichlet(1) over the heavy species, electrons to neutrality; e from T in binary64."""
    n = case["n"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    T = 300.0 * torch.exp(torch.rand(n, generator=g, dtype=F64, device=DEV) * math.log(50.0))
    rho = 1e-4 * torch.exp(torch.rand(n, generator=g, dtype=F64, device=DEV) * math.log(1e4))
    Y = -torch.log1p(-torch.rand(tab.ns, n, generator=g, dtype=F64, device=DEV))
    if tab.ie is not None:
        Y[tab.ie] = tab.M[tab.ie] * sum(Y[s] / tab.M[s] for s in range(tab.ns) if tab.q[s] > 0)
    Y /= Y.sum(0)
    e = (Y * tab.energy(T)).sum(0)
    return T, rho, e, Y


def prepare(case, seed):
    if case["op"] == "thermo":
        cfg = I.with_species(I.bl_case()) if case["gas"] == "air11" else I.bl_case()
        tab = Table(A.table_path(cfg))
        _, rho, e, Y = _thermo_inputs(case, seed, tab)
        one, per = torch.empty_like(rho), torch.empty_like(Y)
        out = dict(T=one, p=one.clone(), wdot=per, mu=one.clone(), k=one.clone(), D=per.clone(),
                   status=torch.empty(case["n"], dtype=torch.uint8, device=DEV))
        return dict(op="thermo", gas=A.gas_model_load(cfg), rho=rho, e=e, Y=Y, out=out,
                    precision=PRECISION[case["precision"]])
    if case["op"] == "batch":
        batch = A.Batch(PRECISION[case["precision"]], use_graph=True)
        states = []
        for k, cfg in enumerate(_batch_configs(case)):
            states.append(_open_state(cfg, seed + 1000003 * k))
            batch.add(states[-1][1], cfg["dt"])
        return dict(op="batch", batch=batch, states=states)
    cfg = _config(case)
    gas, st = _open_state(cfg, seed)
    return dict(op=case["op"], gas=gas, st=st, dt=cfg["dt"], R=torch.empty_like(st.U),
                precision=PRECISION[case["precision"]])


def run(s):
    if s["op"] == "thermo":
        A.thermo_eval(s["gas"], s["rho"], s["e"], s["Y"], precision=s["precision"], **s["out"])
        return s["out"]
    if s["op"] == "batch":
        s["batch"].step(1)
        return [st.U for _, st in s["states"]]
    if s["op"] == "rhs":
        A.rhs(s["gas"], s["st"].grid, s["st"].U, s["R"], precision=s["precision"])
        return {"dUdt": s["R"]}
    for stage in range(3):
        A.rk_stage(s["st"], stage, s["dt"], precision=s["precision"])
    return {"U": s["st"].U}


# ---------------------------------------------------------------------------------------------
# Work: what no implementation of the same method can do without
# ---------------------------------------------------------------------------------------------

# Floating-point operations per state or cell (a fused multiply-add counts two, an exponential or
# logarithm 15, a quotient or root 8), from the formulas: one evaluation of the species energies,
# the rate groups, the transport and the diffusion coefficients; 10 operations per point and
# compact operator (four inputs, two recurrences); the pointwise fluxes, sensors and filters.
CLOSURE = {"air5": 1500.0, "air11": 5000.0}


def _grid_work(cfg, stages):
    ns = I.TABLE_SPECIES[cfg["table"]]
    nz = cfg.get("nz", 1)
    cells = cfg["nx"] * cfg["ny"] * max(nz, 1)
    dims = 3 if nz > 1 else 2
    closure = CLOSURE[cfg["table"]] * (2.0 if cfg["kind"] == "lte" else 1.0)
    operators = (9 * ns + 42) if dims == 2 else (15 * ns + 90)
    points = 100.0 * dims + (40.0 * (ns + 3) if cfg["artificial_diffusivity"] else 0.0)
    flops = cells * stages * (closure + 10.0 * operators + points)
    if stages == 3 and cfg["filter_sigma"] > 0:
        flops += cells * 2 * 21.0 * (ns + 3)
    # the state is read and its derivative or successor written
    return {"bytes": 16.0 * cells * (ns + 1 + dims), "flops": flops}


def work(case):
    if case["op"] == "thermo":
        ns = I.TABLE_SPECIES[case["gas"]]
        return {"bytes": case["n"] * (8.0 * (2 + ns) + 8.0 * (4 + 2 * ns) + 1.0),
                "flops": case["n"] * CLOSURE[case["gas"]]}
    if case["op"] == "batch":
        parts = [_grid_work(c, 3) for c in _batch_configs(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    return _grid_work(_config(case), 3 if case["op"] == "step" else 1)


# ---------------------------------------------------------------------------------------------
# The same results in 64 bits from plain torch: the closure from statistical mechanics, every
# compact operator as a dense matrix, the right-hand side term by term (two-dimensional grids in
# chemical nonequilibrium)
# ---------------------------------------------------------------------------------------------

KB, NA, HP = 1.380649e-23, 6.02214076e23, 6.62607015e-34
RU, P0 = KB * NA, 1.0e5
NEUFELD = ((0.19300, 0.47635), (1.03587, 1.52996), (1.76474, 3.89411))


class Table:
    """A gas table (SPECIES / LEVEL / REACTION lines) and the closure it defines, in SI units.
    States are vectors of n points, per-species arrays (ns, n)."""

    def __init__(self, path):
        self.names, self.sp, self.levels, self.reactions = [], [], {}, []
        for line in open(path):
            tok = line.split("#", 1)[0].split()
            if tok[:1] == ["SPECIES"]:
                self.names.append(tok[1])
                self.sp.append([float(v) for v in tok[2:]] + [0.0] * (14 - len(tok[2:])))
            elif tok[:1] == ["LEVEL"]:
                self.levels.setdefault(tok[1], []).append((float(tok[2]), float(tok[3])))
            elif tok[:1] == ["REACTION"]:
                arrow = tok.index("=>")
                lhs = [self.names.index(v) for v in tok[5:arrow]]
                rhs = [self.names.index(v) for v in tok[arrow + 1:]]
                C = float(tok[1]) * 1e-6 ** (len(lhs) - 1)
                self.reactions.append((C, float(tok[2]), float(tok[3]), lhs, rhs))
        self.ns = len(self.sp)
        self.M = [s[0] for s in self.sp]
        self.q = [int(s[13]) for s in self.sp]
        self.ie = next((i for i, q in enumerate(self.q) if q < 0), None)
        self.heavy = [i for i in range(self.ns) if self.q[i] >= 0]
        at298 = torch.tensor([298.15], dtype=F64)
        self.e0 = [s[1] - float(self._sensible(i, at298)[0]) - RU * 298.15
                   for i, s in enumerate(self.sp)]

    def _electronic(self, i, T):
        Q = m1 = m2 = 0.0
        for g, th in self.levels[self.names[i]]:
            w = g * torch.exp(-th / T)
            Q, m1, m2 = Q + w, m1 + w * th, m2 + w * th * th
        return Q, m1 / Q, m2 / Q

    def _sensible(self, i, T):
        """Molar internal energy above 0 K."""
        _, m1, _ = self._electronic(i, T)
        x = 1.5 * T + m1
        if self.sp[i][2]:
            x = x + T + self.sp[i][3] / torch.expm1(self.sp[i][3] / T)
        return RU * x

    def energy(self, T):
        return torch.stack([(self.e0[i] + self._sensible(i, T)) / self.M[i] for i in range(self.ns)])

    def cv(self, T):
        out = []
        for i in range(self.ns):
            _, m1, m2 = self._electronic(i, T)
            c = 1.5 + (m2 - m1 * m1) / (T * T)
            if self.sp[i][2]:
                x = self.sp[i][3] / T
                c = c + 1.0 + x * x * torch.exp(-x) / torch.expm1(-x) ** 2
            out.append(RU * c / self.M[i])
        return torch.stack(out)

    def temperature(self, e, Y):
        """Bisection of sum Y e(T) = e in ln T, then Newton steps."""
        lo, hi = torch.full_like(e, math.log(50.0)), torch.full_like(e, math.log(1e5))
        for _ in range(24):
            mid = 0.5 * (lo + hi)
            up = (Y * self.energy(torch.exp(mid))).sum(0) <= e
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        T = torch.exp(0.5 * (lo + hi))
        for _ in range(4):
            T = T - ((Y * self.energy(T)).sum(0) - e) / (Y * self.cv(T)).sum(0)
        return T

    def _log_r(self, i, T):
        """ln of the molar partition function per unit volume over its ground-state energy."""
        s = self.sp[i]
        q = 1.5 * torch.log(2.0 * math.pi * s[0] / NA * KB * T / HP ** 2) - math.log(NA)
        Q, _, _ = self._electronic(i, T)
        q = q + torch.log(Q)
        if s[2]:
            q = q + torch.log(T / (s[5] * s[4])) - torch.log(-torch.expm1(-s[3] / T))
        return q - self.e0[i] / (RU * T)

    def rates(self, T, rho, Y):
        c = [rho * Y[i] / self.M[i] for i in range(self.ns)]
        lr = [self._log_r(i, T) for i in range(self.ns)]
        w = [torch.zeros_like(T) for _ in range(self.ns)]
        for C, n, Ta, lhs, rhs in self.reactions:
            kf = math.log(C) + n * torch.log(T) - Ta / T
            kb = kf - (sum(lr[i] for i in rhs) - sum(lr[i] for i in lhs))
            f, b = torch.exp(kf), torch.exp(kb)
            for i in lhs:
                f = f * c[i]
            for i in rhs:
                b = b * c[i]
            r = f - b
            for i in set(lhs + rhs):
                if lhs.count(i) != rhs.count(i):
                    w[i] = w[i] + (rhs.count(i) - lhs.count(i)) * r
        return torch.stack([self.M[i] * w[i] for i in range(self.ns)])

    def transport(self, T, p, X, cv):
        """Mixture viscosity, frozen conductivity and averaged diffusion coefficients."""
        lnT = torch.log(T)
        mu = [0.1 * torch.exp((s[6] * lnT + s[7]) * lnT + s[8]) for s in self.sp]
        k = [mu[i] * (3.75 * RU / self.M[i] + cv[i] - 1.5 * RU / self.M[i]) for i in range(self.ns)]
        mix_mu = mix_k = 0.0
        for i in self.heavy:
            phi = 0.0
            for r in self.heavy:
                t = 1.0 + torch.sqrt(mu[i] / mu[r]) * (self.M[r] / self.M[i]) ** 0.25
                phi = phi + X[r] * t * t / math.sqrt(8.0 * (1.0 + self.M[i] / self.M[r]))
            mix_mu, mix_k = mix_mu + X[i] * mu[i] / phi, mix_k + X[i] * k[i] / phi
        D = torch.zeros_like(X)
        for i in self.heavy:
            den = torch.zeros_like(T)
            for r in self.heavy:
                if r == i:
                    continue
                a, b = self.sp[i], self.sp[r]
                m = a[0] * b[0] / (a[0] + b[0]) / NA
                sig = 0.5 * (a[9] + b[9]) * 1e-10
                ts = T / math.sqrt(a[10] * b[10])
                om = 1.06036 / ts ** 0.15610 + sum(c * torch.exp(-d * ts) for c, d in NEUFELD)
                Dir = 0.1875 * torch.sqrt(2.0 * math.pi * (KB * T) ** 3 / m) / (p * math.pi * sig ** 2 * om)
                den = den + X[r] / Dir
            D[i] = torch.where(den != 0, (1.0 - X[i]) / den, torch.zeros_like(den))
            D[i] *= 2.0 if self.q[i] > 0 else 1.0
        return mix_mu, mix_k, D

    def closure(self, rho, e, Y):
        T = self.temperature(e, Y)
        M = torch.tensor(self.M, dtype=F64, device=T.device)[:, None]
        ym = (Y / M).sum(0)
        p = rho * RU * ym * T
        cvs = self.cv(T)
        cv = (Y * cvs).sum(0)
        X = Y / M / ym
        mu, k, D = self.transport(T, p, X, cvs)
        return dict(T=T, p=p, X=X, mu=mu, k=k, D=D, wdot=self.rates(T, rho, Y),
                    h=self.energy(T) + RU / M * T, Mmix=1.0 / ym,
                    a=torch.sqrt((cv + RU * ym) / cv * p / rho))


def _lagrange(nodes, x, deriv):
    w = []
    for k, xk in enumerate(nodes):
        rest = [v for m, v in enumerate(nodes) if m != k]
        den = math.prod(xk - v for v in rest)
        if deriv:
            num = sum(math.prod(x - v for m, v in enumerate(rest) if m != s) for s in range(len(rest)))
        else:
            num = math.prod(x - v for v in rest)
        w.append(num / den)
    return w


class Operators:
    """The sixth-order compact staggered interpolation ("I") and derivative ("D") between n
    centres and n + 1 faces of a line ("cf", "fc"), as dense matrices; with a wall value at
    position 0 the closure rows at that end use it ("w")."""

    def __init__(self, n):
        self.m = {}
        for what in ("I", "D"):
            for way, wall in (("cf", ""), ("fc", ""), ("cf", "w")):
                self.m[what + way + wall] = self._dense(n, what == "D", way, bool(wall))

    @staticmethod
    def _dense(n, deriv, way, wall):
        al, a, b = (9 / 62, 63 / 62, 17 / 62) if deriv else (3 / 10, 3 / 2, 1 / 10)
        centres, faces = [k + 0.5 for k in range(n)], [float(k) for k in range(n + 1)]
        src, dst = (centres, faces) if way == "cf" else (faces, centres)
        if wall:
            src = [0.0] + src
        o = int(wall)
        first, last = (2, n - 2) if way == "cf" else (1, n - 2)
        L, B = np.eye(len(dst)), np.zeros((len(dst), len(src)))
        for r, x in enumerate(dst):
            if first <= r <= last:
                L[r, r - 1] = L[r, r + 1] = al
                c = r - 2 + o if way == "cf" else r - 1
                B[r, c:c + 4] = [-b / 3, -a, a, b / 3] if deriv else [b / 2, a / 2, a / 2, b / 2]
            else:
                c = 0 if r < first else len(src) - 5
                B[r, c:c + 5] = _lagrange(src[c:c + 5], x, deriv)
        return torch.linalg.solve(torch.tensor(L, device=DEV), torch.tensor(B, device=DEV))

    def x(self, name, f):
        return f @ self.m[name].T

    def y(self, name, f, wall=None):
        if wall is None:
            return self.m[name] @ f
        M = self.m[name + "w"]
        return M[:, 1:] @ f + M[:, :1] * wall


class Flow:
    """Right-hand side, RK3 step and filter of one two-dimensional case in chemical
    nonequilibrium, on the state vector of the library's layout."""

    def __init__(self, cfg, tab):
        self.c, self.t = cfg, tab
        self.nx, self.ny = cfg["nx"], cfg["ny"]
        one = lambda v: torch.tensor([v], dtype=F64, device=DEV)  # noqa: E731
        Yi = torch.tensor(cfg["Y_inf"], dtype=F64, device=DEV)[:, None]
        M = torch.tensor(tab.M, dtype=F64, device=DEV)[:, None]
        Ti = one(cfg["T_inf"])
        cvs = tab.cv(Ti)
        R, cv = RU * float((Yi / M).sum()), float((Yi * cvs).sum())
        self.gam, cp = (cv + R) / cv, cv + R
        self.rho0, self.a0 = cfg["p_inf"] / (R * cfg["T_inf"]), math.sqrt(self.gam * R * cfg["T_inf"])
        X = Yi / M / (Yi / M).sum()
        mu, k, _ = tab.transport(Ti, one(cfg["p_inf"]), X, cvs)
        self.mu0, self.k0, self.Re = float(mu), float(k), cfg["reynolds"]
        self.Pr = self.mu0 * cp / self.k0
        self.Tref = (self.gam - 1.0) * cfg["T_inf"]
        self.L = self.Re * self.mu0 / (self.rho0 * self.a0)
        nx, ny = self.nx, self.ny
        dx = (cfg["x1"] - cfg["x0"]) / nx
        self.xi = 1.0 / dx
        xc = cfg["x0"] + dx * (torch.arange(nx, dtype=F64, device=DEV) + 0.5)
        xf = cfg["x0"] + dx * torch.arange(nx + 1, dtype=F64, device=DEV)
        self.yf, dyf = self._ymap(torch.arange(ny + 1, dtype=F64, device=DEV))
        yc, dyc = self._ymap(torch.arange(ny, dtype=F64, device=DEV) + 0.5)
        self.eta_c, self.eta_f = 1.0 / dyc[:, None], 1.0 / dyf[:, None]
        self.ox, self.oy = Operators(nx), Operators(ny)
        ref, sig = {}, {}
        for where, x, y in (("c", xc, yc), ("u", xf, yc), ("v", xc, self.yf)):
            x, y = x[None, :].expand(len(y), len(x)), y[:, None].expand(len(y), len(x))
            T, p, u, v, Y = self._profile(x, y)
            rho = p / (RU * (Y / M[:, :, None]).sum(0) * T) / self.rho0
            if where == "c":
                e = (Y * tab.energy(T.reshape(-1)).reshape(Y.shape)).sum(0) / self.a0 ** 2
                ref["c"] = torch.cat([rho[None], rho * Y[1:], (rho * (e + 0.5 * (u * u + v * v)))[None]])
            else:
                ref[where] = rho * (u if where == "u" else v)
            sig[where] = self._sponge(x, y)
        self.ref, self.sig = ref, sig

    def _ymap(self, eta):
        c, s = self.c, eta / self.ny
        L, q = c["y1"] - c["y0"], c["y_param"]
        if c["y_stretch"] == "tanh":
            return (c["y0"] + L * (1 - torch.tanh(q * (1 - s)) / math.tanh(q)),
                    L * q / torch.cosh(q * (1 - s)) ** 2 / math.tanh(q) / self.ny)
        return c["y0"] + L * ((1 - q) * s ** 3 + q * s), L * (3 * (1 - q) * s ** 2 + q) / self.ny

    def _shock(self, M1, th):
        g = self.gam
        d = lambda b: math.atan(2 / math.tan(b) * (M1 ** 2 * math.sin(b) ** 2 - 1)  # noqa: E731
                                / (M1 ** 2 * (g + math.cos(2 * b)) + 2))
        lo = hi = math.asin(1 / M1) + 1e-12
        while d(hi + 1e-3) > d(hi):
            hi += 1e-3
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if d(mid) < th else (lo, mid)
        b = 0.5 * (lo + hi)
        m2 = (M1 * math.sin(b)) ** 2
        p21, r21 = 1 + 2 * g / (g + 1) * (m2 - 1), (g + 1) * m2 / ((g - 1) * m2 + 2)
        M2 = math.sqrt((1 + 0.5 * (g - 1) * m2) / (g * m2 - 0.5 * (g - 1))) / math.sin(b - th)
        return b, p21, p21 / r21, M2

    def _profile(self, x, y):
        c, g = self.c, self.gam

        def edge(Te, pe, ue, ve, Me):
            f = torch.erf(2.0 * (y - c["y0"]) / (c["delta_coef"] * torch.sqrt(x / (self.Re * c["mach"]))))
            Tr = Te * (1.0 + 0.85 * 0.5 * (g - 1.0) * Me ** 2)
            return torch.stack([c["T_wall"] + (Tr - c["T_wall"]) * f - (Tr - Te) * f * f,
                                torch.full_like(f, pe), ue * f, ve * f]), f

        q, f = edge(c["T_inf"], c["p_inf"], c["mach"], 0.0, c["mach"])
        if c["flow"] == "sbli":
            th = math.radians(c["shock_deflection_deg"])
            b, p21, T21, M2 = self._shock(c["mach"], th)
            V2 = M2 * math.sqrt(T21)
            q2, _ = edge(c["T_inf"] * T21, c["p_inf"] * p21, V2 * math.cos(th), -V2 * math.sin(th), M2)
            H = 0.5 * (1.0 + torch.tanh((y - (c["shock_x"] - x) * math.tan(b)) / c["shock_width"]))
            q = (1.0 - H) * q + H * q2
        m = c["minor_species"] * 4.0 * f * (1.0 - f)
        seeds = {"N2": lambda v: v * (1.0 - m), "O2": lambda v: v * (1.0 - m), "NO": lambda v: 0.5 * m,
                 "N": lambda v: 0.2 * m, "O": lambda v: 0.3 * m}
        Y = torch.stack([seeds.get(n, lambda v: v + 0.0 * m)(v) for n, v in zip(self.t.names, c["Y_inf"])])
        return (*q, Y)

    def _sponge(self, x, y):
        c = self.c
        r = torch.zeros_like(x)
        if c["sponge_in"] > 0:
            r = r + ((c["x0"] + c["sponge_in"] - x) / c["sponge_in"]).clamp(0, 1) ** 3
        if c["sponge_out"] > 0:
            r = r + ((x - (c["x1"] - c["sponge_out"])) / c["sponge_out"]).clamp(0, 1) ** 3
        if c["sponge_top_cells"] > 0:
            yt = self.yf[self.ny - c["sponge_top_cells"]]
            r = r + ((y - yt) / (c["y1"] - yt)).clamp(0, 1) ** 3
        return c["sponge_sigma"] * r

    def unpack(self, U):
        nx, ny, k = self.nx, self.ny, (self.t.ns + 1) * self.nx * self.ny
        return {"c": U[:k].view(-1, ny, nx), "u": U[k:k + (nx + 1) * ny].view(ny, nx + 1),
                "v": U[k + (nx + 1) * ny:].view(ny + 1, nx)}

    @staticmethod
    def pack(q):
        return torch.cat([q[k].reshape(-1) for k in ("c", "u", "v")])

    def initial(self, noise):
        ref = self.pack(self.ref)
        q, r = self.unpack(ref * (1.0 + self.c["noise_amp"] * torch.as_tensor(noise, device=DEV))), self.ref
        q["u"][:, [0, -1]], q["v"][[0, -1]] = r["u"][:, [0, -1]], r["v"][[0, -1]]
        return self.pack(q)

    def _artificial(self, rho, th, T, e, Y, ux, vy, uy, vx):
        c, dx, dy = self.c, 1.0 / self.xi, 1.0 / self.eta_c

        def d4(f, ax):
            f = f.movedim(ax, -1)
            d = f[..., :-4] - 4 * f[..., 1:-3] + 6 * f[..., 2:-2] - 4 * f[..., 3:-1] + f[..., 4:]
            d = torch.cat([d[..., :1], d[..., :1], d, d[..., -1:], d[..., -1:]], -1)
            return d.movedim(-1, ax)

        def smooth(f):
            w = (3565 / 10368, 3091 / 12960, 1997 / 25920, 149 / 12960, 107 / 103680)
            for ax in (-1, -2):
                f = f.movedim(ax, -1)
                n = f.shape[-1]
                g = torch.cat([f[..., :1].expand(*f.shape[:-1], 4), f, f[..., -1:].expand(*f.shape[:-1], 4)], -1)
                f = w[0] * f + sum(w[k] * (g[..., 4 - k:4 - k + n] + g[..., 4 + k:4 + k + n]) for k in range(1, 5))
                f = f.movedim(-1, ax)
            return f

        div, om = ux + vy, vx - uy
        S = torch.sqrt(ux * ux + vy * vy + 0.5 * (uy + vx) ** 2)
        fsw = torch.where(div < 0, div * div / (div * div + om * om + 1e-32), torch.zeros_like(div))
        mu = smooth(c["C_mu"] * rho * (d4(S, -1) * dx * dx + d4(S, -2) * dy * dy).abs())
        be = smooth(c["C_beta"] * rho * fsw * (d4(div, -1) * dx * dx + d4(div, -2) * dy * dy).abs())
        ka = smooth(c["C_kappa"] * rho * th["a"] / T * (d4(e, -1) * dx + d4(e, -2) * dy).abs())
        D = smooth(c["C_D"] * th["a"] * (d4(Y, -1) * dx + d4(Y, -2) * dy).abs())
        if self.t.ie is not None:
            D[self.t.ie] = 0.0
        return mu, be, ka, D

    def _current(self, J):
        t = self.t
        if t.ie is not None:
            J[t.ie] = t.M[t.ie] * sum(J[i] / t.M[i] for i in range(t.ns) if t.q[i] > 0)
            J[0] = -J[1:].sum(0)
        return J

    def rhs(self, U):
        t, X, Y_, xi, ec, ef = self.t, self.ox.x, self.oy.y, self.xi, self.eta_c, self.eta_f
        q = self.unpack(U)
        rho, rE, ru, rv = q["c"][0], q["c"][-1], q["u"], q["v"]
        Y = torch.cat([(rho - q["c"][1:-1].sum(0))[None], q["c"][1:-1]]) / rho
        uc, vc = X("Ifc", ru) / rho, Y_("Ifc", rv) / rho
        e = rE / rho - 0.5 * (uc * uc + vc * vc)
        f = t.closure(rho.reshape(-1) * self.rho0, e.reshape(-1) * self.a0 ** 2, Y.reshape(t.ns, -1))
        th = {k: v.reshape(*v.shape[:-1], self.ny, self.nx) for k, v in f.items()}
        T, p, h = th["T"] / self.Tref, th["p"] / (self.rho0 * self.a0 ** 2), th["h"] / self.a0 ** 2
        th["a"] = th["a"] / self.a0
        H = (rE + p) / rho
        rxf, ryf = X("Icf", rho), Y_("Icf", rho)
        uf, vf = ru / rxf, rv / ryf
        ux, vy = xi * X("Dfc", uf), ec * Y_("Dfc", vf)
        uy, vx = ef * Y_("Dcf", uf, 0.0), xi * X("Dcf", vf)
        ucn, vcn = Y_("Icf", uf, 0.0), X("Icf", vf)
        mu, K = th["mu"] / self.mu0 / self.Re, th["k"] / self.k0 / (self.Re * self.Pr)
        D, be = th["D"] * self.rho0 / self.mu0 / self.Re, torch.zeros_like(rho)
        if self.c["artificial_diffusivity"]:
            m, be, ka, Ds = self._artificial(rho, th, T, e, Y, ux, vy, X("Ifc", Y_("Ifc", uy)),
                                             X("Ifc", Y_("Ifc", vx)))
            mu, K, D = mu + m, K + ka, D + Ds
        M = torch.tensor(t.M, dtype=F64, device=DEV)[:, None, None]
        Gd = rho * M / th["Mmix"] * D
        div = ux + vy
        txx, tyy = (mu * (2.0 * g - 2.0 / 3.0 * div) + be * div for g in (ux, vy))
        txy = Y_("Icf", X("Icf", mu)) * (uy + vx)
        G = X("Icf", Gd) * (xi * X("Dcf", th["X"]))
        Yf = X("Icf", Y)
        J = self._current(Yf * G.sum(0) - G)
        Fx = ru * Yf + J
        FEx = (ru * X("Icf", H) - X("Icf", K) * (xi * X("Dcf", T)) + (X("Icf", h) * J).sum(0)
               - X("Icf", txx) * uf - Y_("Ifc", txy) * X("Icf", vc))
        G = Y_("Icf", Gd) * (ef * Y_("Dcf", th["X"]))
        Yf = Y_("Icf", Y)
        J = self._current(Yf * G.sum(0) - G)
        J[:, 0] = 0.0
        Fy = rv * Yf + J
        FEy = (rv * Y_("Icf", H) - Y_("Icf", K) * (ef * Y_("Dcf", T, self.c["T_wall"] / self.Tref))
               + (Y_("Icf", h) * J).sum(0) - Y_("Icf", tyy) * vf - X("Ifc", txy) * Y_("Icf", uc, 0.0))
        Gxx = X("Ifc", ru * uf) + p - txx
        Gyy = Y_("Ifc", rv * vf) + p - tyy
        Gxy = Y_("Icf", rxf) * ucn * vcn - txy
        d = lambda a, b: -(xi * X("Dfc", a) + ec * Y_("Dfc", b))  # noqa: E731
        w = th["wdot"] * self.L / (self.rho0 * self.a0)
        R = {"c": torch.cat([d(ru, rv)[None], d(Fx, Fy)[1:] + w[1:], d(FEx, FEy)[None]]),
             "u": -(xi * X("Dcf", Gxx) + ec * Y_("Dfc", Gxy)),
             "v": -(xi * X("Dfc", Gxy) + ef * Y_("Dcf", Gyy))}
        R = {k: R[k] - self.sig[k] * (q[k] - self.ref[k]) for k in R}
        R["u"][:, [0, -1]], R["v"][[0, -1]] = 0.0, 0.0
        return self.pack(R)

    def _filtered(self, U):
        q = self.unpack(U)
        for ax in (-1, -2):
            for k in q:
                f = q[k].movedim(ax, -1)
                n, g = f.shape[-1], f.movedim(ax, -1).movedim(-1, ax).clone()
                for i in range(1, n - 1):
                    m = min(i, n - 1 - i, 5)
                    if m == 5 and i > 5:
                        continue
                    stop = n - 5 if m == 5 else i + 1
                    g[..., i:stop] = f[..., i:stop] - self.c["filter_sigma"] / 4.0 ** m * sum(
                        (-1) ** j * math.comb(2 * m, m + j) * f[..., i + j:stop + j] for j in range(-m, m + 1))
                q[k] = g.movedim(-1, ax)
        return self.pack(q)

    def step(self, U):
        Q = torch.zeros_like(U)
        for a, b in ((0.0, 1 / 3), (-5 / 9, 15 / 16), (-153 / 128, 8 / 15)):
            Q = a * Q + self.c["dt"] * self.rhs(U)
            U = U + b * Q
        return self._filtered(U) if self.c["filter_sigma"] > 0 else U


def exact(case, seed):
    if case["op"] == "thermo":
        cfg = I.with_species(I.bl_case()) if case["gas"] == "air11" else I.bl_case()
        tab = Table(A.table_path(cfg))
        _, rho, e, Y = _thermo_inputs(case, seed, tab)
        parts = [tab.closure(rho[k:k + 500000], e[k:k + 500000], Y[:, k:k + 500000])
                 for k in range(0, case["n"], 500000)]
        return {k: torch.cat([q[k] for q in parts], -1) for k in ("T", "p", "wdot", "mu", "k", "D")}
    if case["op"] == "batch":
        tab, out = None, []
        for k, cfg in enumerate(_batch_configs(case)):
            tab = tab or Table(A.table_path(cfg))
            flow = Flow(cfg, tab)
            n = flow.pack(flow.ref).numel()
            out.append(flow.step(flow.initial(_noise(n, seed + 1000003 * k))))
        return out
    if case["kind"] != "cneq" or case["nz"] > 1:
        return None             # equilibrium compositions and three dimensions: no plain form here
    cfg = _config(case)
    flow = Flow(cfg, Table(A.table_path(cfg)))
    U = flow.initial(_noise(flow.pack(flow.ref).numel(), seed))
    return {"dUdt": flow.rhs(U)} if case["op"] == "rhs" else {"U": flow.step(U)}
