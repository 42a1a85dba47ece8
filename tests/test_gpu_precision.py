"""Binary64 precision of the integer kernels entry by entry, on fields whose entries differ in size:
normwise comparisons do not see what a small entry loses beside a large one.

State filter: out = f - sigma d with the tenth difference d over 1024. d is within one rounding of
itself and 2^-54 of the largest entry of its own window (tests/test_fix_runs_method.py), the final
operation rounds once."""
from fractions import Fraction as Fr

import numpy as np
import pytest

from gpu_util import gpu_state, oracle_case
from oracle import flow as F
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
