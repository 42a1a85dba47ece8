"""HYP_MIXED evaluates the forward-rate exponentials (Eq. 13) in binary32, the backward rates and
all else of the production rates as HYP_FP64: hyp_thermo_eval against the oracle's rates with each
forward exponent n ln T - T_a / T rounded to binary32, on the integer closure and on compositions
that take the binary64 one.

Bound per state and species: expf is within 1 unit in the last place (2^-23 relative) of the
forward terms; the rest is test_gpu_closure_fix's bound of the FP64 rates. States with an exponent
within 1e-9 of a binary32 rounding boundary (where T's own rounding decides) are left out."""
import numpy as np
import pytest

from oracle import gas as G
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _rates(tab, T, conc):
    """Production rates with binary32 forward exponents, the forward and the gross terms, and which
    states' exponents round the same after a change of 1e-9."""
    kf, kb, _ = G.reaction_rates(tab, T, conc)
    w, fwd, gross = (np.zeros((tab.ns, T.size)) for _ in range(3))
    safe = np.ones(T.size, dtype=bool)
    for ir, r in enumerate(tab.reactions):
        x = r.n * np.log(T) - r.Ta / T
        safe &= np.float32(x - 1e-9) == np.float32(x + 1e-9)
        f = r.C * np.exp(np.float32(x).astype(np.float64))
        b = kb[ir].copy()
        for s in range(tab.ns):
            f = f * conc[s] ** int(r.nu_f[s])
            b = b * conc[s] ** int(r.nu_b[s])
        nu = (r.nu_b - r.nu_f) * tab.M()
        w += nu[:, None] * (f - b)
        fwd += np.abs(nu)[:, None] * np.abs(f)
        gross += np.abs(nu)[:, None] * (np.abs(f) + np.abs(b))
    return w, fwd, gross, safe


@pytest.mark.parametrize("far", [False, True], ids=["integer closure", "binary64 closure"])
def test_forward_rate_exponentials_in_binary32(table, far):
    import torch
    from paper_2210_05547_gb300 import abi as A
    rng = np.random.default_rng(5)
    n = 4001
    T = np.exp(rng.uniform(np.log(1500.0), np.log(15000.0), n))
    rho = np.exp(rng.uniform(np.log(1e-4), 0.0, n))
    Y = rng.dirichlet(np.ones(5), n).T
    if far:                                          # |X| beyond the fixed-point range
        Y[0], Y[1] = 4.0 + Y[0], -3.0 - Y[2:].sum(axis=0) - Y[0]
    e = G.mixture_energy(table, T, Y)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64).cuda()  # noqa: E731
    w = torch.empty((5, n), dtype=torch.float64, device="cuda")
    A.thermo_eval(A.gas_model_load(I.bl_case()), dev(rho), dev(e), dev(Y), wdot=w, precision=A.MIXED)
    got = w.cpu().numpy()
    o = G.thermo_eval(table, rho, e, Y)
    ref, fwd, gross, safe = _rates(table, o["T"], rho * Y / table.M()[:, None])
    ok = safe & (o["cv"] > 0) & (np.abs(o["T"] / T - 1) < 1e-9)
    assert ok.sum() > 0.9 * n
    dT = 1e-13 + 8 * 2.0 ** -53 * np.sum(np.abs(Y) * np.abs(G.energy_species(table, T)), axis=0) / (o["cv"] * T)
    tol = 2.0 ** -23 * fwd + (1e-12 + (50 + 3.4e5 / T) * (dT + 16 * 2.0 ** -53)) * gross + 1e-290
    assert np.all((np.abs(got - ref) <= tol)[:, ok])
