"""Binary64 precision of the integer kernels entry by entry, on fields whose entries differ in size:
normwise comparisons do not see what a small entry loses beside a large one.

State filter: out = f - sigma d with the tenth difference d over 1024. d is within one rounding of
itself and 2^-54 of the largest entry of its own window (tests/test_fix_runs_method.py), the final
operation rounds once.

Line operators: the density of a passive species carried at unit mass flux along one direction has the
right-hand side -metric D(I(Y)) (interpolation to faces, derivative back), here against the same two
solves in extended precision. A line solve is within thirty units of 2^-60 (truncated inputs, products
and shifts along two recurrences with factors 1/3 and 0.148) of the largest value near the row: within
sixteen rows, farther values weighted by 2^(-11/8) or 2^(-20/8) a row; closure rows are five binary64
products each; values more than 64 rows away are left out (rho^64 < 2^-101), lines cut into chunks
or extended by margins start 40 rows early (rho^40 < 2^-63, of the recurrence's values, up to four
times the largest input).
Interpolation's error and rounding go through the derivative's matrix; its result rounds, and the
metric's product and rounding add a few units in the last place."""
from fractions import Fraction as Fr

import numpy as np
import pytest

from gpu_util import gpu_state, oracle_case
from oracle import flow as F
from oracle import flow3d as F3
from oracle.compact import lagrange_weights
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TENTH = [-1, 10, -45, 120, -210, 252, -210, 120, -45, 10, -1]
EPS = Fr(2) ** -53


def test_state_filter_entry_by_entry(table):
    import torch
    from paper_2210_05547_gb300 import abi as A
    nx, ny, sigma = 131, 24, 0.75
    cfg = I.sbli_case(nx, ny)
    cfg["filter_sigma"] = sigma
    q = F.unpack(5, nx, ny, oracle_case(table, cfg).U0)
    q = {k: np.repeat(v[ny // 2][None], v.shape[0], axis=0) for k, v in q.items()}   # rows all alike
    x = np.arange(nx)
    f = {"rhou": 0.4 * np.sin((np.arange(nx + 1) - 60.3) / 9),
         "rs1": 0.05 * (1 + 0.02 * np.sin(x / 9)),
         "rs2": 1e-9 + 1e-3 * (1 + np.tanh((x - 70) / 2)),
         "rs3": 1e-3 * 10.0 ** (-0.1 * x)}
    for k, v in f.items():
        q[k][:] = v
    gas, st = gpu_state(cfg)
    st.U.copy_(torch.as_tensor(F.pack(5, nx, ny, q)))
    A.rk_stage(st, 2, 0.0)                           # a step of zero length: the filter alone
    got = F.unpack(5, nx, ny, st.U.cpu().numpy())
    s = Fr(sigma)
    for k, a in f.items():
        for i in range(5, a.size - 5):
            w = a[i - 5:i + 6]
            d = sum(Fr(float(v)) * c for v, c in zip(w, TENTH)) / 1024
            out = Fr(float(got[k][ny // 2, i]))
            bound = EPS * abs(out) + s * (EPS * abs(d) + EPS / 2 * Fr(float(np.abs(w).max())))
            assert abs(out - (Fr(float(a[i])) - s * d)) <= bound, (k, i)


L = np.longdouble
U53, U55 = 2.0 ** -53, 2.0 ** -55


class Line:
    """One operator (kind 0 interpolation to faces, 1 derivative to centres) on a line of n cells."""

    def __init__(self, kind, n, periodic):
        self.kind, self.per, self.n = kind, periodic, n
        self.m = n if periodic or kind else n + 1
        self.al, self.wa, self.wb = ((L(3) / 10, L(3) / 4, L(1) / 20), (L(9) / 62, L(63) / 62, L(17) / 186))[kind]
        self.rows = []
        if not periodic:
            src = [Fr(2 * k + 1, 2) for k in range(n)] if kind == 0 else [Fr(k) for k in range(n + 1)]
            first = 1 if kind else 2
            for r in list(range(first)) + list(range(n - 1, self.m)):
                at, c = (Fr(2 * r + 1, 2) if kind else Fr(r)), (0 if r < first else len(src) - 5)
                self.rows.append((r, c, [L(float(w)) for w in lagrange_weights(src[c:c + 5], at, bool(kind))]))

    def rhs(self, x):
        s = -1 if self.kind else 1
        o = 1 if self.kind else 2
        i = np.arange(self.m)
        g = lambda k: x[(i - o + k) % len(x)]  # noqa: E731
        return self.wa * (g(2) + s * g(1)) + self.wb * (g(3) + s * g(0))

    def __call__(self, x):
        x = x.astype(L)
        b = self.rhs(x)
        ext = 120 if self.per else 0                     # periods beyond decay below 2^-190
        if self.per:
            b = b[np.arange(-ext, self.m + ext) % self.m]
        off = np.full(b.size, self.al)
        for r, c, w in self.rows:
            off[r], b[r] = 0, sum(v * x[c + k] for k, v in enumerate(w))
        up = np.zeros(b.size, dtype=L)
        for r in range(b.size):
            p = 1 - (off[r] * up[r - 1] if r else 0)
            up[r], b[r] = off[r] / p, (b[r] - (off[r] * b[r - 1] if r else 0)) / p
        for r in range(b.size - 2, -1, -1):
            b[r] -= up[r] * b[r + 1]
        return b[ext:ext + self.m]

    def error(self, x):
        """Bound on the solve's own error, without the result's rounding."""
        a, i = np.abs(x).astype(float), np.arange(self.m)
        near = np.zeros(self.m)
        for j in range(a.size):
            d = np.abs(i - j)
            if self.per:
                d = np.minimum(d, a.size - d)
            near = np.maximum(near, a[j] * 2.0 ** (-(20 if self.kind else 11) / 8 * np.maximum(0, d - 16)))
        e = U55 * near
        rho = 0.1484 if self.kind else 1 / 3
        for r, c, w in self.rows:
            e = e + 5 * U53 * sum(abs(float(v)) * a[c + k] for k, v in enumerate(w)) * rho ** np.abs(i - r)
        cut = self.m % 8 or self.m > 2304 if self.per else self.m > 2301
        return e + (2.0 ** -61 if cut else 2.0 ** -99) * a.max()


@pytest.mark.parametrize("axis,n", [("x", 21), ("x", 131), ("y", 131), ("z", 40), ("z", 37),
                                    ("x", 2400), ("y", 2400), ("z", 2400)])
def test_lines_entry_by_entry(axis, n):
    import torch
    from paper_2210_05547_gb300 import abi as A
    nx, ny, nz = (n if axis == a else 9 for a in "xyz")
    cfg = dict(I.box_case(nx, ny, kind="cpg"), sponge_sigma=0.0)
    if axis == "z":
        cfg.update(nz=nz, z0=0.0, z1=2.0, jet=0)
    x = np.arange(n) / n
    fall = min(12.0, 0.2 * n)                            # decades
    if axis == "z":
        Y = [10.0 ** (-0.5 * fall * (1 - np.cos(2 * np.pi * x))), 0.01 * (2 + np.sin(2 * np.pi * x)),
             1e-14 + 0.01 * np.exp(-200 * (x - 0.5) ** 2), np.sin(4 * np.pi * x)]
    else:
        Y = [10.0 ** (-fall * x), 10.0 ** (1.5 * fall * (x - 1)),
             1e-12 + 0.01 * (1 + np.tanh((np.arange(n) - n / 2) / 2.0)), np.sin(9 * x)]
    Y = [0.05 * v for v in Y]
    mod = F3 if axis == "z" else F
    shape = (nx, ny, nz) if axis == "z" else (nx, ny)
    q = {k: np.zeros(s) for k, s in mod.state_layout(5, *shape)}
    ones = {"x": (1, -1), "y": (-1, 1), "z": (-1, 1, 1)}[axis]
    q["rho"][:] = 1.0
    q["rhoE"][:] = 0.5 + 1.0 / (1.4 * 0.4)
    q["rhou" if axis == "x" else ("rhov" if axis == "y" else "rhow")][:] = 1.0
    for s, v in enumerate(Y):
        q[f"rs{s + 1}"][:] = v.reshape(ones)
    gas = A.gas_model_load(cfg)
    U = torch.as_tensor(mod.pack(5, *shape, q)).cuda()
    own, dQ = torch.empty_like(U), torch.empty_like(U)
    st = A.state_init(gas, cfg, own, dQ, None)
    R = torch.empty_like(U)
    A.rhs(gas, st.grid, U, R)
    got = mod.unpack(5, *shape, R.cpu().numpy())
    grid = F.make_grid(cfg)
    met = {"x": lambda: grid.xi_c, "y": lambda: grid.eta_c, "z": lambda: np.full(n, n / 2.0)}[axis]()
    ic, dc = Line(0, n, axis == "z"), Line(1, n, axis == "z")
    D = np.abs(np.array([dc(e) for e in np.eye(ic.m)]).astype(float)).T if n < 200 else None
    for s, v in enumerate(Y):
        f = ic(v)
        exact = -met * dc(f)
        ef = ic.error(v) + U53 * np.abs(f).astype(float)
        if D is not None:
            through = D @ ef
        else:                                            # |D| by its decay: 8.2 x 0.1484^distance
            i = np.arange(dc.m)[:, None]
            through = sum(8.2 * 0.1484 ** abs(k) * ef[np.clip(i[:, 0] + k, 0, ic.m - 1)] for k in range(-40, 41))
        bound = met * (through + dc.error(f)) + 8 * U53 * np.abs(exact).astype(float)
        a = got[f"rs{s + 1}"]
        a = a[4, 4] if axis == "z" and a.ndim == 4 else (a[:, 4, 4] if axis == "z" else (a[4] if axis == "x" else a[:, 4]))
        ratio = np.abs(a.astype(L) - exact).astype(float) / bound
        assert ratio.max() <= 1.0, (s, int(ratio.argmax()), float(ratio.max()))
