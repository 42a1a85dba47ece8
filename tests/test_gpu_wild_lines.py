"""NaN and infinities on lines along y and z: the block's lines take the binary64 form of the solver,
whose exchanges reach eight segments of eight rows (and the rows of the ends), so four operators in a
row reach at most 4 x 80 rows; values beyond agree with the clean field's to rounding."""
import numpy as np
import pytest

from oracle import flow as F
from oracle import flow3d as F3
from paper_2210_05547_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("axis,n", [("y", 480), ("z", 720), ("z", 723)])
def test_wild_values_stay_near(axis, n, bad):
    import torch
    from paper_2210_05547_gb300 import abi as A
    nx, ny, nz = (n if axis == a else 9 for a in "xyz")
    cfg = dict(I.box_case(nx, ny, kind="cpg"), sponge_sigma=0.0)
    if axis == "z":
        cfg.update(nz=nz, z0=0.0, z1=2.0, jet=0)
    mod, shape = (F3, (nx, ny, nz)) if axis == "z" else (F, (nx, ny))
    gas = A.gas_model_load(cfg)
    size = A.state_size(gas, cfg)
    U = torch.empty(size, dtype=torch.float64, device="cuda")
    st = A.state_init(gas, cfg, U, torch.empty_like(U), I.state_noise(size, 5))
    U.mul_(1.0 + 1e-3 * torch.as_tensor(I.state_noise(size, 6)).cuda())
    R, W = torch.empty_like(U), U.clone()
    A.rhs(gas, st.grid, U, R)
    W[(60 * ny + 4) * nx + 4 if axis == "z" else 60 * nx + 4] = bad      # rho at row or plane 60
    Rw = torch.empty_like(U)
    A.rhs(gas, st.grid, W, Rw)
    clean, wild = (mod.unpack(5, *shape, v.cpu().numpy()) for v in (R, Rw))
    assert not np.isfinite(wild["rho"][60]).all()
    for k in clean:
        far = slice(60 + 328, None if axis == "y" else n + 60 - 328)
        a, b = clean[k][far], wild[k][far]
        assert a.shape[0] > 0 and np.isfinite(b).all(), k
        assert np.abs(a - b).max() <= 1e-9 * np.abs(clean[k]).max(), k
