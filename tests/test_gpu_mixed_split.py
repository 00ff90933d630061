"""GPU parity of the y, z and y passes on mixed-radix lengths (mixed_split.cu): every z length, edges of
the 32-bin tiles and of the length classes, against the oracle (1e-5 relative L2, as the demag tests)."""
import pytest

import oracle
from gpu_util import assert_close, to_dev, torch_cuda
from paper_2008_02478_gb300 import inputs

pytestmark = pytest.mark.gpu

MESHES = [(5, 6, 2), (2, 2, 3), (13, 16, 4), (9, 31, 5), (8, 32, 6), (33, 33, 7), (9, 64, 8), (12, 65, 9), (24, 20, 12),
          (10, 97, 13), (11, 30, 16), (12, 128, 17), (7, 12, 20), (16, 40, 21), (9, 161, 24), (18, 12, 25), (6, 300, 32),
          (4, 512, 3), (3, 500, 11), (2, 1030, 4), (520, 9, 3), (700, 5, 10)]


@pytest.mark.parametrize("n", MESHES)
def test_passes_match_oracle(n, monkeypatch):
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import Plan
    h = (3e-9, 2e-9, 2.5e-9)
    M = 8e5 * inputs.random_unit(*n, seed=sum(n))
    monkeypatch.setenv("BORIS_YZ_KIND", "4")
    plan = Plan(*n, *h)
    assert plan.schedule()[0] == 4
    ref = oracle.DemagPlan(*n, *h).apply(M)
    H = plan.apply(to_dev(torch, M, False)).cpu().numpy()
    assert_close(H, ref, 1e-5)


@pytest.mark.parametrize("n", [(39, 210, 24), (62, 894, 6), (160, 640, 12)])
def test_meshes_that_take_the_passes(n):
    """Chosen without a switch; steps of the plan and its allocation-free form agree with it."""
    torch = torch_cuda()
    import ctypes
    from paper_2008_02478_gb300.binding import Plan, lib
    h = (3e-9, 3e-9, 3e-9)
    M = 8e5 * inputs.random_unit(*n, seed=3)
    plan = Plan(*n, *h)
    assert plan.schedule()[0] == 4
    Md = to_dev(torch, M, False)
    H = plan.apply(Md)
    assert_close(H.cpu().numpy(), oracle.DemagPlan(*n, *h).apply(M), 1e-5)
    H2 = torch.empty_like(H)
    rc = lib().boris_demag_apply_noalloc(plan._h, ctypes.c_void_p(Md.data_ptr()), ctypes.c_void_p(H2.data_ptr()))
    if rc == 0:  # the mesh's spectrum fits the fixed workspace
        torch.cuda.synchronize()
        assert torch.equal(H, H2)


@pytest.mark.parametrize("n,fp64", [((16, 16, 1), False), ((16, 16, 4), True)])
def test_the_passes_refuse_what_they_cannot(n, fp64, monkeypatch):
    """One plane has no z stage, and FP64 plans have no passes."""
    torch_cuda()
    from paper_2008_02478_gb300.binding import BorisError, Plan
    monkeypatch.setenv("BORIS_YZ_KIND", "4")
    with pytest.raises(BorisError) as e:
        Plan(*n, 1e-9, 1e-9, 1e-9, fp64=fp64)
    assert e.value.code == -4
