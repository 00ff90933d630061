"""The power-of-two passes on the meshes whose plans take mixed-radix lengths by default: parity with the
oracle under the tolerances of the demag, adjoint and multi-mesh tests (1e-5 in FP32, 1e-9 in FP64), and
the mixed-radix passes together with the 1024- and 2048-point transforms."""
import numpy as np
import pytest

import oracle
from oracle import llg
from oracle import multilayer as ml
from paper_2008_02478_gb300 import inputs
from tests.gpu_util import assert_close, to_dev, torch_cuda
from tests.test_gpu_adjoint import BIG
from tests.test_gpu_demag import CASES
from tests.test_gpu_ml_frames import make_case, sampled

pytestmark = pytest.mark.gpu


def padded(n):
    return 1 if n == 1 else 1 << (2 * n - 2).bit_length()


def pow2_plan(monkeypatch, n, h, fp64):
    """A plan on powers of two: the split schedule, else a fused one."""
    from paper_2008_02478_gb300.binding import BorisError, Plan
    for kind in (2, 1, 0):
        monkeypatch.setenv("BORIS_YZ_KIND", str(kind))
        try:
            plan = Plan(*n, *h, fp64=fp64)
        except BorisError as e:
            assert e.code == -4
            continue
        assert plan.schedule()[0] == kind and plan.padded() == tuple(padded(v) for v in n)
        return plan
    raise AssertionError("no power-of-two schedule")


@pytest.mark.parametrize("n,h", CASES)
@pytest.mark.parametrize("fp64", [False, True])
def test_demag_matches_oracle(n, h, fp64, monkeypatch):
    torch = torch_cuda()
    M = 8e5 * inputs.random_unit(*n, seed=1)
    plan = pow2_plan(monkeypatch, n, h, fp64)
    H = plan.apply(to_dev(torch, M, fp64)).cpu().numpy()
    plan.sync_status()
    assert_close(H, oracle.DemagPlan(*n, *h).apply(M), 1e-9 if fp64 else 1e-5)


@pytest.mark.parametrize("n,h", BIG)
@pytest.mark.parametrize("fp64", [False, True])
def test_step_backward_matches_oracle(n, h, fp64, monkeypatch):
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import LLGParams
    Ms = inputs.smooth_noise(*n, 2.0, 6e5, 1e6, 15)
    Ku = inputs.smooth_noise(*n, 2.0, 0.0, 5e5, 16)
    prm = llg.Params(cell=h, Ms=Ms, A=1.3e-11, alpha=0.02, Ku=Ku, easy=(0.0, 0.0, 1.0), Hext=(0.0, 0.0, 2e4))
    m0, gout, dt = inputs.smooth_texture(*n, 1.5, 17), inputs.random_unit(*n, seed=18), 1e-13
    ref = llg.rk4_step_vjp(m0, dt, prm, oracle.DemagPlan(*n, *h).apply, gout)
    plan = pow2_plan(monkeypatch, n, h, fp64)
    p = LLGParams(A=prm.A, alpha=prm.alpha, gamma=prm.gamma, easy=prm.easy, Hext=prm.Hext,
                  Ms_map=to_dev(torch, Ms, fp64), Ku_map=to_dev(torch, Ku, fp64))
    gMs = torch.zeros(n[::-1], dtype=plan.dtype, device="cuda")
    gKu = torch.zeros_like(gMs)
    gm = plan.llg_step_backward(to_dev(torch, m0, fp64), p, dt, to_dev(torch, gout, fp64), None, gMs, gKu)
    for got, want in zip((gm, gMs, gKu), ref):
        assert_close(got.cpu().numpy(), want, 1e-9 if fp64 else 1e-3)


# (px, py): x passes of 1024 and 2048 points with mixed-radix y passes, and with the 1024-point ones
@pytest.mark.parametrize("n,p", [((500, 130, 3), (1024, 320)), ((490, 490, 2), (1024, 1024)), ((1000, 130, 3), (2048, 320)),
                                 ((1000, 490, 2), (2048, 1024)), ((30, 500, 9), (64, 1024))])
def test_passes_with_power_of_two_axes(n, p, monkeypatch):
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import Plan
    h = (3e-9, 2e-9, 2.5e-9)
    M = 8e5 * inputs.random_unit(*n, seed=sum(n))
    monkeypatch.setenv("BORIS_YZ_KIND", "4")
    plan = Plan(*n, *h)
    assert plan.schedule()[0] == 4 and plan.padded()[:2] == p
    H = plan.apply(to_dev(torch, M)).cpu().numpy()
    assert_close(H, oracle.DemagPlan(*n, *h).apply(M), 1e-5)


@pytest.mark.parametrize("n", [(39, 210, 24), (62, 894, 6)])
def test_steps_agree_between_schedules(n, monkeypatch):
    """max |m - m'| <= 1e-6 after an RK4 step on the passes and on powers of two: four stages each add
    the rounding of m (6e-8) and dt gamma times that of the field (2.2e-8 m/A s^2 x 1e-6 of 1e6 A/m)."""
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import LLGParams, Plan
    h, prm = (3e-9, 3e-9, 3e-9), LLGParams(Ms=8e5, A=1.3e-11, alpha=0.1, Hext=(1e4, 0.0, 3e4), Ku=5e4)
    out = []
    for plan in (Plan(*n, *h), pow2_plan(monkeypatch, n, h, False)):
        m = to_dev(torch, inputs.random_unit(*n, seed=3))
        plan.llg_step(m, prm, 1e-13)
        out.append((plan.schedule()[0], m.cpu().numpy()))
    assert out[0][0] == 4 and out[1][0] == 2
    assert np.abs(out[0][1] - out[1][1]).max() <= 1e-6


# frames one cell wide keep the power-of-two passes with copies into and out of the frame
@pytest.mark.parametrize("layers", [[(1, 20, 2), (1, 12, 1)], [(30, 1, 2), (12, 1, 1)], [(1, 1, 3), (1, 1, 2)]])
def test_frames_one_cell_wide(layers):
    torch = torch_cuda()
    st, m, M, plan = make_case(layers)
    H = plan.apply(torch.tensor(M, dtype=torch.float32, device="cuda")).cpu().numpy()
    cells, got = sampled(st, H)
    assert_close(got, ml.direct_at(st, M, cells), 1e-5)
