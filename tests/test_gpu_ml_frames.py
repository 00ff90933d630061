"""GPU parity of the multi-mesh field over frame lengths: the mixed-radix and
the 1024-point x and y passes, whose rows are windows of the frame, against
Eq. 4's direct sum at sampled cells, each layer's corners among them (1e-5
relative L2, the FP32 bound of the other multi-mesh tests)."""
import numpy as np
import pytest

from oracle import llg
from oracle import multilayer as ml
from paper_2008_02478_gb300 import inputs
from tests.gpu_util import assert_close, rel_l2, torch_cuda
from tests.test_gpu_multilayer import make_plan, stack_case

pytestmark = pytest.mark.gpu

FRAMES = [
    [(2, 2, 1), (1, 1, 2)],                 # the shortest lines; one-cell windows
    [(37, 23, 2), (12, 22, 1), (5, 3, 3)],  # odd offsets, remainders of every tile
    [(100, 75, 1), (99, 16, 2), (1, 75, 1)],
    [(511, 6, 1), (300, 3, 2)],             # 1024-point x, odd and even rows
    [(505, 7, 2), (120, 2, 1)],             # the same on a frame of odd height
    [(6, 512, 1), (3, 333, 2), (1, 7, 1)],  # 1024-point y
    [(509, 490, 1), (48, 51, 1), (510, 17, 1)],  # both, windows at odd rows
    [(701, 20, 1), (20, 9, 2)],             # three-pass lengths
]


def sampled(st, H):
    """(cells, the rows of the concatenated field H at them): each layer's corners and four more."""
    offs = np.cumsum([0] + st.counts)
    cells = []
    for l, (nx, ny, nz) in enumerate(st.n):
        n = st.counts[l]
        cells += [offs[l], offs[l] + nx - 1, offs[l] + n - nx, offs[l + 1] - 1]
        cells += list(offs[l] + inputs.rng(7 + l).integers(0, n, 4))
    cells = np.unique(cells)
    rows = []
    for gi in cells:
        l = int(np.searchsorted(offs, gi, side="right") - 1)
        rows.append([H[3 * offs[l] + c * st.counts[l] + gi - offs[l]] for c in range(3)])
    return cells, np.array(rows, dtype=np.float64)


def make_case(layers):
    hz = [2e-9, 3e-9, 1e-9][:len(layers)]
    st, m, M, _ = stack_case(layers, hz, [1e-9] * (len(layers) - 1), 4e-9, seed=21)
    return st, m, M, make_plan(st)


@pytest.mark.parametrize("layers", FRAMES)
def test_frames_match_direct_sum(layers):
    torch = torch_cuda()
    st, m, M, plan = make_case(layers)
    H = plan.apply(torch.tensor(M, dtype=torch.float32, device="cuda")).cpu().numpy()
    cells, got = sampled(st, H)
    assert_close(got, ml.direct_at(st, M, cells), 1e-5)


@pytest.mark.parametrize("layers", FRAMES)
def test_frames_with_a_magnetisation_map(layers):
    """M_s differs in every cell.  One step with rotations of at most 2e-3: the
    increment is dt times the right-hand side of the direct sum's field to first
    order, so within 2e-3 (half the largest rotation squared, plus FP32
    rounding of m: 1e-7 of 1e-3)."""
    torch = torch_cuda()
    from paper_2008_02478_gb300.binding import LLGParams
    st, m, _, plan = make_case(layers)
    ms = inputs.rng(5).uniform(4e5, 1.2e6, st.total()).astype(np.float32)
    m = m.astype(np.float32)
    offs = np.cumsum([0] + st.counts)
    M = m.astype(np.float64)
    for l, n in enumerate(st.counts):
        M[3 * offs[l]:3 * offs[l + 1]] *= np.tile(ms[offs[l]:offs[l + 1]].astype(np.float64), 3)
    dt = 6e-15
    mg = torch.tensor(m, device="cuda")
    plan.llg_step(mg, LLGParams(A=1e-20, alpha=0.1, Ms_map=torch.tensor(ms, device="cuda")), dt)
    cells, m1 = sampled(st, mg.cpu().numpy())
    _, m0 = sampled(st, m)
    H = ml.direct_at(st, M, cells)
    assert dt * 2.22e5 * np.abs(H).max() < 2e-3
    ref = dt * llg.llg_rhs(m0.T, H.T, llg.Params(cell=(1, 1, 1), alpha=0.1)).T
    assert rel_l2(m1 - m0, ref) < 2e-3


PLANES = [[1], [1, 2], [3, 4], [8], [4, 4, 1], [6, 6, 4], [10, 7], [16, 8, 1], [14, 20], [24, 16], [20, 1, 20], [16, 16, 16], [49]]


@pytest.mark.parametrize("planes", PLANES)
@pytest.mark.parametrize("ny,variant", [(5, 2), (5, 3), (35, 2)])
def test_persistent_sum_over_plane_counts(planes, ny, variant, monkeypatch):
    """The persistent inter-plane sum over its plane counts: one plane, fewer
    than the eight warps, equal and unequal counts of consecutive targets, and
    sources below, above and between a warp's targets; one and several column
    tiles.  Sampled cells of the direct sum."""
    torch = torch_cuda()
    if variant == 3 and sum(planes) > 35:
        pytest.skip("two blocks per SM hold 35 planes")
    monkeypatch.setenv("BORIS_ML_MIX", str(variant))
    st, m, M, plan = make_case([(5 - l, ny - l, nz) for l, nz in enumerate(planes)])
    assert plan.schedule()[2] == variant
    H = plan.apply(torch.tensor(M, dtype=torch.float32, device="cuda")).cpu().numpy()
    cells, got = sampled(st, H)
    assert_close(got, ml.direct_at(st, M, cells), 1e-5)
