"""D_s of a species among traces, D = (1 - X_s) / sum_r X_r / D_sr, through hyp_thermo_eval.

1 - X_s carries the rounding of X_s, which hides the sum's own error in a comparison of D. But X_s in
[1/2, 1) is a multiple of 2^-53, so D times the exact sum is one too, up to the relative error of the
sum, the collision integrals and the quotient: a few units in the last place each, 64 x 2^-53 in all.
The multiple itself is that of X_s to the rounding of X_s (ns / 2 + 2 units, as in
test_gpu_closure_fix)."""
import numpy as np
import pytest

from oracle import gas as G
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("gas", ["air5", "air11"])
def test_sum_of_traces_keeps_binary64_precision(gas, table, table11):
    import torch
    from paper_2210_05547_gb300 import abi as A
    tab = table if gas == "air5" else table11
    cfg = I.bl_case() if gas == "air5" else I.with_species(I.bl_case())
    rng = np.random.default_rng(23)
    n = 3001
    heavy = np.nonzero(tab.heavy())[0]
    Y = np.zeros((tab.ns, n))
    Y[heavy] = rng.dirichlet(np.ones(heavy.size), n).T * 10.0 ** -rng.uniform(4.5, 12, n)
    lead = heavy[rng.integers(0, heavy.size, n)]
    at = np.arange(n)
    Y[lead, at] = 0.0
    Y[lead, at] = 1.0 - Y.sum(axis=0)
    T = np.exp(rng.uniform(np.log(300.0), np.log(15000.0), n))
    rho = np.exp(rng.uniform(np.log(1e-4), 0.0, n))
    e = G.mixture_energy(tab, T, Y)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).cuda()  # noqa: E731
    Tg, pg = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    Dg = torch.empty((tab.ns, n), dtype=torch.float64, device="cuda")
    A.thermo_eval(A.gas_model_load(cfg), dev(rho), dev(e), dev(Y), T=Tg, p=pg, D=Dg)
    Tg, pg, Dg = (v.cpu().numpy() for v in (Tg, pg, Dg))
    L = np.longdouble
    X = Y.astype(L) / tab.M()[:, None].astype(L)
    X = X / X.sum(axis=0)
    Db = G.binary_diffusion(tab, Tg, pg)
    for s in heavy:
        own = lead == s
        den = sum(X[r, own] / Db[s, r, own] for r in heavy if r != s)
        D = Dg[s, own] / (2 if tab.species[s].charge > 0 else 1)
        v = D * den / U
        k = np.round(v)
        assert np.all(np.abs(v - k) <= 64 * U * np.abs(v)), (s, float(np.max(np.abs(v - k) / np.abs(v)) / U))
        rest = sum(X[r, own] for r in heavy if r != s)
        assert np.all(np.abs(k - rest / U) <= tab.ns / 2 + 2.5), s
