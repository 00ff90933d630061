"""The four-cells-per-thread RK4 stage, which meshes of 400 k cells and more with
nx a multiple of four take, against the one-cell stage of the FP64 plan."""
import numpy as np
import pytest

from paper_2008_02478_gb300 import inputs
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("images", [None, (1, 1, 0), (1, 0, 0)])
@pytest.mark.parametrize("n", [(400, 334, 3), (64, 400, 16), (1000, 401, 1), (404, 1000, 1)])
def test_quad_stage_matches_one_cell_stage(n, images):
    """max |m - m_64| <= 1e-6: four stages each add the rounding of m (6e-8) and
    dt gamma times that of the field (2.2e-8 m/A s^2 x 1e-6 of 1e6 A/m); a wrong
    neighbour would show at 3e-2."""
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import LLGParams, Plan
    m0 = inputs.random_unit(*n, seed=3).astype(np.float32)
    out = []
    for fp64 in (False, True):
        plan = Plan(*n, 4e-9, 4e-9, 4e-9, fp64=fp64, images=images)
        m = torch.tensor(m0, dtype=plan.dtype, device="cuda")
        plan.llg_step(m, LLGParams(Ms=8e5, A=1.3e-11, alpha=0.1, Hext=(1e4, 0.0, 3e4), Ku=5e4), 1e-13)
        out.append(m.double().cpu().numpy())
        plan.close()
    assert np.abs(out[0] - out[1]).max() <= 1e-6
