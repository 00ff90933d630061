"""Meshes on which the mixed-radix schedules measured slower than the power-of-two ones are not given
to them, and the ones they were made for are."""
import pytest

from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def kind(n, fp64):
    torch_cuda()
    from paper_2008_02478_gb300.binding import Plan
    plan = Plan(*n, 3e-9, 3e-9, 3e-9, fp64=fp64)
    k = plan.schedule()[0]
    plan.close()
    return k


@pytest.mark.parametrize("n", [(387, 51, 32), (457, 463, 4), (393, 479, 2), (389, 28, 15), (420, 30, 14), (415, 25, 29),
                               (919, 8, 32),
                               (214, 56, 25), (49, 3, 18), (34, 3, 20), (51, 7, 6), (64, 4, 11)])
def test_fp64_meshes_left_to_powers_of_two(n):
    assert kind(n, True) < 3


@pytest.mark.parametrize("n", [(128, 128, 16), (32, 70, 1), (59, 21, 3), (407, 111, 18), (428, 4, 13), (186, 32, 29)])
def test_fp64_meshes_on_mixed_lengths(n):
    assert kind(n, True) == 3


@pytest.mark.parametrize("n", [(3, 395, 4), (4, 720, 2), (2, 54, 31), (4, 42, 28), (4, 52, 16), (2, 931, 4), (6, 815, 2), (5, 404, 3),
                               (3, 16, 27), (2, 59, 15)])
def test_few_lines_left_to_powers_of_two(n):
    assert kind(n, False) < 3


@pytest.mark.parametrize("n,k", [((32, 32, 4), 3), ((16, 16, 27), 3), ((4, 39, 13), 3), ((4, 1394, 3), 4), ((3, 1500, 16), 4), ((5, 500, 30), 4),
                                 ((12, 300, 20), 4), ((160, 640, 12), 4)])
def test_fp32_meshes_on_mixed_lengths(n, k):
    assert kind(n, False) == k


# long z stages with one CTA per SM and several planes for each, where the estimates are close and
# both schedules are timed (10 to 25 % apart)
@pytest.mark.parametrize("n", [(431, 189, 21), (432, 172, 21), (855, 190, 22), (350, 126, 26), (8, 394, 26)])
def test_close_estimates_are_timed(n):
    """The plan takes the power-of-two schedules, and its field is that of a plan made for them (FP32
    rounding of the transforms, 1e-6, where the two chose different ones)."""
    torch = torch_cuda()
    from paper_2008_02478_gb300 import inputs
    from paper_2008_02478_gb300.binding import Plan
    M = torch.tensor(8e5 * inputs.random_unit(*n, seed=6), dtype=torch.float32, device="cuda")
    with pytest.MonkeyPatch.context() as mp:
        mp.setenv("BORIS_YZ_KIND", "2")
        ref = Plan(*n, 3e-9, 3e-9, 4e-9, images=(1, 0, 0))
    plan = Plan(*n, 3e-9, 3e-9, 4e-9, images=(1, 0, 0))
    assert plan.schedule()[0] == 2 and plan.padded() == ref.padded()
    H, H0 = plan.apply(M), ref.apply(M)
    assert (H - H0).norm() <= 1e-6 * H0.norm()
    plan.sync_status()


# (0.7 and less of the power-of-two time)
@pytest.mark.parametrize("n,k", [((283, 269, 24), 4), ((55, 767, 26), 4), ((56, 1711, 3), 4), ((34, 466, 13), 4), ((72, 410, 9), 4)])
def test_close_estimates_that_stay(n, k):
    assert kind(n, False) == k
