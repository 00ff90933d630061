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
