"""The event profile names the kernels that ran: one launch of k_stress_c per right-hand side, with
and without the artificial diffusivities that it adds, and no entry for kernels that are gone."""
import pytest

from gpu_util import gpu_state
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [I.sbli_case(64, 48), I.bl_case(64, 48)], ids=["with", "without"])
def test_names_and_counts(cfg):
    import torch
    from paper_2210_05547_gb300 import abi as A
    gas, st = gpu_state(cfg)
    R = torch.empty_like(st.U)
    A.grid_profile(st.grid, True)
    for _ in range(3):
        A.rhs(gas, st.grid, st.U, R)
    A.grid_profile(st.grid, False)
    prof = A.grid_profile_read(st.grid)
    assert "k_ad_combine" not in prof
    assert prof["k_stress_c"][1] == 3 and prof["k_closure"][1] == 3
    assert ("k_gauss" in prof and prof["k_gauss"][1] == 6) == bool(cfg["artificial_diffusivity"])
