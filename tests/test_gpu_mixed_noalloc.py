"""boris_demag_apply_noalloc on plans with mixed-radix lengths: it takes a mesh where the buffers that
the plan's own schedule uses fit its array, and gives boris_demag_apply's field bit by bit."""
import ctypes

import pytest

from paper_2008_02478_gb300 import inputs
from tests.gpu_util import to_dev, torch_cuda

pytestmark = pytest.mark.gpu

ARRAY = 32 << 20


# (mesh, schedule kind): the plane kernel keeps the half spectrum X alone, the passes also the padded one
@pytest.mark.parametrize("n,kind", [((32, 32, 4), 3), ((256, 256, 8), 3), ((512, 512, 2), 3), ((600, 700, 4), 3),
                                    ((39, 210, 24), 4), ((62, 894, 6), 4), ((160, 640, 12), 4)])
def test_array_holds_what_the_schedule_uses(n, kind):
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import Plan, lib
    nx, ny, nz = n
    plan = Plan(*n, 3e-9, 3e-9, 3e-9)
    assert plan.schedule()[0] == kind
    px, py, _ = plan.padded()
    rows = (px // 2 + 1) * 3 * nz * 8
    need = (rows * ny + 255) // 256 * 256 + (rows * py if kind == 4 else 0)
    M = to_dev(torch, 8e5 * inputs.random_unit(*n, seed=4))
    ref, H = plan.apply(M), torch.full_like(M, 7.0)
    L = lib()
    for _ in range(2):
        rc = L.boris_demag_apply_noalloc(plan._h, ctypes.c_void_p(M.data_ptr()), ctypes.c_void_p(H.data_ptr()))
        assert rc == (0 if need <= ARRAY else -4), L.boris_last_error()
    torch.cuda.synchronize()
    assert torch.equal(H, ref if need <= ARRAY else torch.full_like(M, 7.0))
