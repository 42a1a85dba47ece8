"""hyp_rhs_noalloc's size limit does not depend on the size of an internal record: 33 x 184 and
596 x 10 cells lie just inside it (1,572,835 and 1,572,816 of 1,572,864 doubles: 111 per cell, 70 and
67 per x- and y-face, 8 per corner, and 87 line jobs of 144 bytes), 34 x 184 and 597 x 10 outside."""
import numpy as np
import pytest

from gpu_util import gpu_state, oracle_case
from oracle import flow as F
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(33, 184), (596, 10)])
def test_grids_just_inside_are_accepted(table, nx, ny):
    import torch
    from paper_2210_05547_gb300 import abi as A
    cfg = I.bl_case(nx, ny)
    gas, st = gpu_state(cfg)
    case = oracle_case(table, cfg)
    tol, _ = F.parity_tolerance(case, case.U0)
    U = torch.as_tensor(case.U0).cuda()
    R, Rn = torch.empty_like(U), torch.full_like(U, float("nan"))
    A.rhs(gas, st.grid, U, R)
    A.rhs_noalloc(gas, st.grid, U, Rn)
    a, b = (F.unpack(5, nx, ny, v.cpu().numpy()) for v in (R, Rn))
    for k in a:
        assert np.abs(a[k] - b[k]).max() <= tol[k], k


@pytest.mark.parametrize("nx,ny", [(34, 184), (597, 10)])
def test_grids_just_outside_are_refused(nx, ny):
    import torch
    from paper_2210_05547_gb300 import abi as A
    gas, st = gpu_state(I.bl_case(nx, ny))
    with pytest.raises(A.HypError, match="too large for hyp_rhs_noalloc"):
        A.rhs_noalloc(gas, st.grid, st.U, torch.empty_like(st.U))
