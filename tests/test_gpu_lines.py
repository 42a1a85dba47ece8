"""The compact line solver where its plan changes: lines cut into chunks (more than 288 segments of
eight rows), one-segment remainders, lines that hold NaN or infinities.

The reference is the plain 64-bit right-hand side of perf/cases.py (every operator a dense matrix).
Bound per entry kind, as in gpu_util: 1e-12 of the largest value plus 32 times the change of the
reference when every state entry moves by one unit in the last place."""
import importlib.util
import os

import numpy as np
import pytest

from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def cases():
    spec = importlib.util.spec_from_file_location("cases", os.path.join(ROOT, "perf", "cases.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def _rhs(cfg, U):
    import torch
    from paper_2210_05547_gb300 import abi as A
    gas = A.gas_model_load(cfg)
    own, dQ = torch.empty_like(U), torch.empty_like(U)
    st = A.state_init(gas, cfg, own, dQ, None)
    R = torch.empty_like(U)
    A.rhs(gas, st.grid, U, R)
    torch.cuda.synchronize()
    return R


@pytest.mark.parametrize("nx,ny", [(2298, 9), (2299, 11), (2302, 10), (4600, 8), (10, 2301), (21, 22),
                                   (22, 21), (13, 14)])
def test_long_and_remainder_lines(cases, nx, ny):
    import torch
    from paper_2210_05547_gb300 import abi as A
    cfg = I.bl_case(nx, ny)
    flow = cases.Flow(cfg, cases.Table(A.table_path(cfg)))
    U = flow.initial(cases._noise(flow.pack(flow.ref).numel(), 3))
    ref, R = flow.rhs(U), _rhs(cfg, U)
    g = torch.Generator(device="cuda").manual_seed(7)
    up = torch.rand(U.numel(), generator=g, device="cuda") < 0.5
    inf = torch.tensor(float("inf"), dtype=U.dtype, device="cuda")
    moved = flow.rhs(torch.where(up, torch.nextafter(U, inf), torch.nextafter(U, -inf)))
    q, r, m = flow.unpack(R), flow.unpack(ref), flow.unpack(moved)
    for k in q:
        fields = zip(q[k], r[k], m[k]) if k == "c" else [(q[k], r[k], m[k])]
        for i, (a, b, c) in enumerate(fields):
            bound = 1e-12 * b.abs().max() + 32 * (c - b).abs().max()
            assert (a - b).abs().max() <= bound, (k, i, float((a - b).abs().max()), float(bound))


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e290])
def test_wild_values_stay_near_their_lines(cases, bad):
    import torch
    from paper_2210_05547_gb300 import abi as A
    cfg = I.bl_case(600, 200)
    flow = cases.Flow(cfg, cases.Table(A.table_path(cfg)))
    U = flow.initial(np.zeros(flow.pack(flow.ref).numel()))
    clean = flow.unpack(_rhs(cfg, U))
    U[30 * 600 + 60] = bad                           # rho at column 60 of row 30
    R = flow.unpack(_rhs(cfg, U))
    assert not torch.isfinite(R["c"][:, 30, 60]).all() or bad == 1e290
    # four operators in a row, each reaching at most 56 columns
    far = (clean["c"][:, :, 400:], R["c"][:, :, 400:])
    assert torch.isfinite(far[1]).all()
    assert (far[0] - far[1]).abs().max() <= 1e-9 * far[0].abs().max()
