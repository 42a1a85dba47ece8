"""The Gaussian filter of the artificial diffusivities and the state filter, whose threads take four
entries of a line at a time: grids whose sides leave every remainder, and lines shorter than one
stencil. The right-hand side to gpu_util's criterion. The state filter against the oracle's to
16 units in the last place of each field's largest value (eleven terms of weights summing to 1/2 in
magnitude, twice, and the final sum)."""
import numpy as np
import pytest

from gpu_util import check_rhs, gpu_rhs, gpu_state, oracle_case
from oracle import flow as F
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(24, 29), (25, 30), (26, 31), (27, 28)])
def test_rhs_with_artificial_diffusivity(table, nx, ny):
    cfg = I.sbli_case(nx, ny)
    case = oracle_case(table, cfg)
    gas, st = gpu_state(cfg)
    bad, _ = check_rhs(case, case.U0, gpu_rhs(gas, st, case.U0))
    assert not bad, bad


@pytest.mark.parametrize("nx,ny", [(8, 9), (9, 10), (10, 11), (11, 8), (13, 15), (64, 33)])
def test_state_filter(table, nx, ny):
    import torch
    from paper_2210_05547_gb300 import abi as A
    cfg = I.sbli_case(nx, ny)
    case = oracle_case(table, cfg)
    gas, st = gpu_state(cfg)
    st.U.copy_(torch.as_tensor(case.U0))
    A.rk_stage(st, 2, 0.0)                           # a step of zero length: the filter alone
    got = F.unpack(5, nx, ny, st.U.cpu().numpy())
    want = F.unpack(5, nx, ny, F.filter_state(case, case.U0))
    for k in want:
        assert np.abs(got[k] - want[k]).max() <= 16 * 2.0 ** -53 * np.abs(want[k]).max(), k
