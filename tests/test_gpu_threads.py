"""Two host threads, each with a plan and a stream of its own: calls of one plan neither fail nor
change the results of the other's.  The pairs run the same kernels with different amounts of shared
memory per CTA: the limit that a launch is checked against belongs to the kernel, not to the plan."""
import threading

import pytest

from paper_2008_02478_gb300 import inputs
from tests.gpu_util import torch_cuda
from tests.test_gpu_multilayer import make_plan, stack_case

pytestmark = pytest.mark.gpu


def run_in_two_threads(torch, make, calls):
    """make(k): (plan, field) of thread k, made on that thread's stream."""
    streams = [torch.cuda.Stream() for _ in range(2)]
    plans, errors = [], []
    for k in range(2):
        with torch.cuda.stream(streams[k]):
            plan, M = make(k)
            plans.append((plan, M, torch.empty_like(M), plan.apply(M).clone()))
    torch.cuda.synchronize()
    start = threading.Barrier(2)

    def work(k):
        plan, M, H, _ = plans[k]
        try:
            with torch.cuda.stream(streams[k]):
                start.wait()
                for _ in range(calls):
                    plan.apply(M, H)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for plan, _, H, ref in plans:
        assert torch.equal(H, ref)
        plan.close()


# the passes on mixed-radix lengths: the z kernel of half length 24 with 21 and 24 planes, of 32 with 25 and 32
@pytest.mark.parametrize("planes", [(21, 24), (25, 32)])
def test_passes_with_different_numbers_of_planes(planes, monkeypatch):
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import Plan
    monkeypatch.setenv("BORIS_YZ_KIND", "4")

    def make(k):
        plan = Plan(16, 40, planes[k], 3e-9, 3e-9, 3e-9)
        assert plan.schedule()[0] == 4
        return plan, torch.tensor(8e5 * inputs.random_unit(16, 40, planes[k], seed=k), dtype=torch.float32, device="cuda")

    run_in_two_threads(torch, make, 6000)


# (environment, meshes of the two plans): the power-of-two schedules, on x lengths below 256
@pytest.mark.parametrize("env,meshes", [
    ({"BORIS_YZ_KIND": "0", "BORIS_YZ_CLUSTER": "4"}, [(16, 60, 20), (100, 40, 32)]),
    ({"BORIS_YZ_KIND": "0", "BORIS_YZ_CLUSTER": "8"}, [(20, 100, 25), (60, 120, 32)]),
    ({"BORIS_YZ_KIND": "1", "BORIS_YZ_CLUSTER": "8"}, [(30, 60, 30), (30, 120, 20)]),
    ({"BORIS_YZ_KIND": "2"}, [(30, 30, 3), (60, 60, 3)]),
])
def test_power_of_two_schedules_of_different_sizes(env, meshes, monkeypatch):
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import BorisError, Plan
    for k, v in env.items():
        monkeypatch.setenv(k, v)

    def make(k):
        n = meshes[k]
        plan = Plan(*n, 3e-9, 3e-9, 3e-9)
        assert plan.schedule()[0] == int(env["BORIS_YZ_KIND"])
        return plan, torch.tensor(8e5 * inputs.random_unit(*n, seed=k), dtype=torch.float32, device="cuda")

    try:
        run_in_two_threads(torch, make, 2000)
    except BorisError as e:
        assert e.code == -4
        pytest.skip("schedule does not fit")


# the inter-plane sum: numbers of planes that share a kernel (its targets per warp)
@pytest.mark.parametrize("variant,planes", [(0, (33, 40)), (1, (17, 24)), (2, (17, 24)), (2, (25, 32)), (3, (25, 32))])
def test_multi_mesh_sums_of_different_numbers_of_planes(variant, planes, monkeypatch):
    torch = torch_cuda()
    monkeypatch.setenv("BORIS_ML_MIX", str(variant))

    def make(k):
        st, _, M, _ = stack_case([(12, 10, planes[k])], [2e-9], [], 4e-9, seed=k)
        plan = make_plan(st)
        assert plan.schedule()[2] == variant
        return plan, torch.tensor(M, dtype=torch.float32, device="cuda")

    run_in_two_threads(torch, make, 4000)


def test_plans_made_in_two_threads(monkeypatch):
    """Kernel spectra built side by side: transforms of different lengths."""
    torch = torch_cuda()
    monkeypatch.setenv("BORIS_YZ_KIND", "0")
    from paper_2008_02478_gb300.binding import Plan
    meshes = [(200, 3, 2), (30, 5, 10)]
    ref, errors = [], []
    for n in meshes:
        M = torch.tensor(8e5 * inputs.random_unit(*n, seed=5), dtype=torch.float32, device="cuda")
        ref.append((M, Plan(*n, 3e-9, 3e-9, 3e-9, images=(1, 0, 0)).apply(M)))
    torch.cuda.synchronize()

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(20):
                    plan = Plan(*meshes[k], 3e-9, 3e-9, 3e-9, images=(1, 0, 0))
                    H = plan.apply(ref[k][0])
                    torch.cuda.current_stream().synchronize()
                    # (the schedule is chosen by timing, so not bit by bit)
                    assert (H - ref[k][1]).norm() <= 1e-5 * ref[k][1].norm()
                    plan.close()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
