"""GPU parity of the plane schedule on mixed-radix lengths (plane_conv.cuh, mixed_x.cuh): the edges of
its length classes, z sizes and kernel classes against the oracle."""
import pytest

import oracle
from gpu_util import assert_close, to_dev, torch_cuda
from paper_2008_02478_gb300 import inputs

pytestmark = pytest.mark.gpu

# (nx, ny, nz): each axis at the largest cell count of a length or one above the previous one
MESHES = [(2, 3, 1), (5, 6, 2), (8, 10, 1), (9, 12, 3), (13, 16, 4), (17, 20, 1), (25, 32, 5), (33, 40, 6),
          (49, 64, 2), (65, 80, 1), (81, 96, 4), (97, 120, 1), (12, 121, 7), (128, 9, 8), (160, 161, 1), (11, 192, 9),
          (193, 12, 12), (241, 14, 2), (10, 256, 13), (257, 12, 16), (12, 320, 5), (384, 10, 1), (10, 385, 4),
          (480, 9, 2), (9, 481, 8), (512, 16, 16), (513, 8, 3), (8, 640, 6), (641, 6, 1), (6, 768, 5), (769, 5, 1),
          (5, 960, 2), (961, 4, 1), (4, 1024, 4), (1025, 4, 2), (4, 1280, 1), (3, 1536, 2), (1537, 3, 1), (2, 2048, 1),
          (2048, 2, 1), (14, 12, 17), (12, 14, 20), (16, 20, 21), (20, 16, 24), (18, 12, 25), (12, 18, 32)]


@pytest.mark.parametrize("n", MESHES)
@pytest.mark.parametrize("fp64", [False, True])
def test_plane_schedule_matches_oracle(n, fp64, monkeypatch):
    """Tolerances are those of the demag parity tests: 1e-5 in FP32, 1e-9 in FP64."""
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import BorisError, Plan
    h = (3e-9, 2e-9, 2.5e-9)
    M = 8e5 * inputs.random_unit(*n, seed=sum(n))
    monkeypatch.setenv("BORIS_YZ_KIND", "3")
    try:
        plan = Plan(*n, *h, fp64=fp64)
    except BorisError as e:
        assert fp64 and e.code == -4  # in FP64 the longest lines of several planes exceed shared memory
        pytest.skip("the plane does not fit shared memory")
    px, py, pz = plan.padded()
    assert plan.schedule()[0] == 3
    assert px >= 2 * n[0] - 1 and py >= 2 * n[1] - 1 and pz >= 2 * n[2] - 1
    H = plan.apply(to_dev(torch, M, fp64)).cpu().numpy()
    assert_close(H, oracle.DemagPlan(*n, *h).apply(M), 1e-9 if fp64 else 1e-5)
