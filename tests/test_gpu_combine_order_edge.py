"""Plans whose combine-order rows end on either side of what k_combine_order stages in
shared memory (12 K entries less its own static share): every trace length there
makes a plan, and the forward matches the FP64 oracle."""
import pytest

from oracle import oracle as orc
from paper_2404_10928_gb300 import phantoms as ph

from helpers import OP_TOL, f32, rel_l2

pytestmark = pytest.mark.gpu

# K + L of the rows: the staged limit and its neighbours, and the last lengths below
# 48 KB, where the row alone fits
ROWS = [12 * 1024 + d for d in (-65, -64, -63, -32, -31, -8, -7, -1, 0, 1)]


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10928_gb300 import build
    build.build()
    return torch


def _problem(K):
    return ph.custom(2, (40, 33), (1e-4, 1e-4), ph.ring_sensors(5, 14e-3), K, seed=73)


@pytest.mark.parametrize("row", ROWS)
def test_rows_at_the_edge_of_staging(torch_cuda, row):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    with Plan.from_problem(_problem(700)) as plan:
        L = plan.info()["window"]  # depends on the tile, c and fs only
    prob = _problem(row - L)
    x = f32(prob.x_true)
    with Plan.from_problem(prob) as plan:
        assert prob.n_samples + plan.info()["window"] == row
        xt = torch.tensor(x, dtype=torch.float32, device="cuda")
        p = plan.forward(xt).cpu().numpy()
        plan.set_sound_speed(1510.0)
        plan.set_sound_speed(prob.c)
        assert torch.equal(plan.forward(xt).cpu(), torch.tensor(p))
        plan.sync_status()
    assert rel_l2(p, orc.forward(orc.Geometry.of(prob), x)) <= OP_TOL
