"""The integer closure (closure_fix.cuh) at the ends of its ranges and the states it hands to the
binary64 closure, through hyp_thermo_eval against the oracle, five- and eleven-species air.

Tolerances: T from converged inversions, 1e-13 as in test_gpu_thermo; the other outputs are smooth
in T and X with condition numbers of order ten (the collision integrals, T^(3/2), ln T): 1e-12.
D_s = (1 - X_s) / den_s carries the rounding of X_s: (ns / 2 + 2) eps / (1 - X_s) on top (the
product Y / M, half of the ns - 1 additions of the sum, the reciprocal and the product with it), so
its reference takes X_s in extended precision (the oracle's own X_s is off by as much). The production rates
are differences of forward and backward rates whose exponents T_a / T reach 2000 at 60 K: a few
eps T_a / T of the larger of the two."""
import numpy as np
import pytest

from oracle import gas as G
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _eval(cfg, rho, e, Y):
    import torch
    from paper_2210_05547_gb300 import abi as A
    gas = A.gas_model_load(cfg)
    n = rho.size
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).cuda()  # noqa: E731
    out = {k: torch.empty(n, dtype=torch.float64, device="cuda") for k in ("T", "p", "mu", "k")}
    out["wdot"] = torch.empty((gas.ns, n), dtype=torch.float64, device="cuda")
    out["D"] = torch.empty((gas.ns, n), dtype=torch.float64, device="cuda")
    out["status"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    A.thermo_eval(gas, dev(rho), dev(e), dev(Y), **out)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


def _compositions(tab, rng, m):
    """Mass fractions (ns, n): mixed, nearly pure, pure, with small negative traces, and far
    outside [0, 1] (mole fractions beyond the fixed-point range)."""
    ns = tab.ns
    heavy = np.nonzero(tab.heavy())[0]
    mixed = np.zeros((ns, m))
    mixed[heavy] = rng.dirichlet(np.ones(heavy.size), m).T
    near = np.zeros((ns, m))
    trace = rng.dirichlet(np.ones(heavy.size), m).T * 10.0 ** -rng.uniform(1, 12, m)
    near[heavy] = trace
    lead = heavy[rng.integers(0, heavy.size, m)]
    near[lead, np.arange(m)] = 0.0
    near[lead, np.arange(m)] = 1.0 - near.sum(axis=0)
    pure = np.zeros((ns, heavy.size))
    pure[heavy, np.arange(heavy.size)] = 1.0
    neg = mixed.copy()
    neg[heavy[-1]] = -1e-9 * rng.uniform(0, 1, m)
    neg[heavy[0]] += 1.0 - neg.sum(axis=0)
    far = np.zeros((ns, 16))
    far[0], far[1] = 4.0, -3.0
    return np.concatenate([mixed, near, pure, neg, far], axis=1)


@pytest.mark.parametrize("gas", ["air5", "air11"])
def test_ranges_against_the_oracle(gas, table, table11):
    rng = np.random.default_rng(17)
    tab = table if gas == "air5" else table11
    cfg = I.bl_case() if gas == "air5" else I.with_species(I.bl_case())
    Y = _compositions(tab, rng, 3001)
    n = Y.shape[1]
    T = np.exp(rng.uniform(np.log(55.0), np.log(9.5e4), n))
    T[:8] = [50.0 * (1 + 1e-12), 64.0, 1024.0, np.nextafter(1024.0, 0), 65536.0, 99999.0, 72.0, 2.0e4]
    rho = np.exp(rng.uniform(np.log(1e-8), np.log(1e2), n))
    e = G.mixture_energy(tab, T, Y)
    g, o = _eval(cfg, rho, e, Y), G.thermo_eval(tab, rho, e, Y)
    # where the energy determines T: the cancellation of formation against thermal energy sets
    # how far two inversions sit apart
    cond = 8 * EPS * np.sum(np.abs(Y) * np.abs(G.energy_species(tab, T)), axis=0) / (o["cv"] * T)
    assert np.all(g["status"] == o["status"])
    ok = (o["cv"] > 0) & (np.abs(o["T"] / T - 1) < 1e-9)
    assert ok.sum() > 0.98 * n
    dT = 1e-13 + cond
    assert np.all(np.abs(g["T"] / o["T"] - 1)[ok] <= dT[ok])
    for k in ("p", "mu", "k"):
        assert np.all((np.abs(g[k] - o[k]) <= (1e-12 + 30 * dT) * np.abs(o[k]))[ok]), k
    L = np.longdouble
    X = Y.astype(L) / tab.M()[:, None].astype(L)
    X = X / X.sum(axis=0)
    Db = G.binary_diffusion(tab, o["T"], o["p"])
    heavy = np.nonzero(tab.heavy())[0]
    for s in heavy:
        den = sum(X[r] / Db[s, r] for r in heavy if r != s)
        some = ok & (np.abs(1 - X[s]) > 64 * EPS) & (den != 0)   # a pure species: rounding over rounding
        D = (1 - X[s, some]) / den[some] * (2 if tab.species[s].charge > 0 else 1)
        tol = 1e-12 + 30 * dT[some] + (tab.ns / 2 + 2) * EPS / np.abs(1 - X[s, some])
        assert np.all(np.abs(g["D"][s, some] - D) <= tol * np.abs(D)), s
    conc = rho * Y / tab.M()[:, None]
    kf, kb, R = G.reaction_rates(tab, o["T"], conc)
    gross = np.zeros_like(Y)
    for ir, r in enumerate(tab.reactions):
        f, b = kf[ir].copy(), kb[ir].copy()
        for s in range(tab.ns):
            f *= conc[s] ** int(r.nu_f[s])
            b *= conc[s] ** int(r.nu_b[s])
        nu = np.abs(r.nu_b - r.nu_f) * tab.M()
        gross += nu[:, None] * (np.abs(f) + np.abs(b))
    tol = (1e-12 + (50 + 3.4e5 / T) * (dT + 16 * EPS)) * gross + 1e-290
    assert np.all((np.abs(g["wdot"] - o["wdot"]) <= tol)[:, ok])


def test_invalid_states_are_flagged_as_before():
    cfg = I.bl_case()
    Y = np.zeros((5, 6))
    Y[0], Y[1] = 0.767, 0.233
    e = np.full(6, 4.0e5)
    rho = np.array([0.1, 0.0, -0.2, np.nan, 0.1, 0.1])
    e[4] = np.nan
    Y[0, 5] = np.nan
    g = _eval(cfg, rho, e, Y)
    assert list(g["status"][:4]) == [0, 4, 4, 4]
    assert g["status"][4] == 1 and g["status"][5] == 1
    assert np.isfinite(g["T"]).all() and np.isnan(g["mu"][5])
