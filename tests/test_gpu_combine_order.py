"""The combine order built on the device (k_combine_order): plans whose tables
come from one warp's share, several 32-tile chunks, rows longer than the staged
limit and tiles skipped at both ends, through the forward operator against the
FP64 oracle, and the speed-of-sound change against a fresh plan."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2404_10928_gb300 import phantoms as ph

from helpers import OP_TOL, f32, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10928_gb300 import build
    build.build()
    return torch


RING = ph.ring_sensors(5, 14e-3)
CASES = {
    "one-tile": ph.custom(2, (20, 9), (1e-4, 1e-4), RING, 700, seed=71),
    "33-tiles": ph.custom(2, (33 * 32 - 5, 7), (2e-5, 1e-4), RING, 700, seed=72),
    # rows of K + L samples too long for shared memory
    "long-rows": ph.custom(2, (70, 70), (1e-4, 1e-4), RING, 12300, seed=73),
    # traces that start late and end early: tiles skipped on both sides
    "skipped-tiles": ph.custom(2, (150, 130), (1e-4, 1e-4), RING, 40, seed=74, t0=350 / 40e6),
    "3d-equal-starts": ph.custom(3, (40, 24, 20), (2e-4, 2e-4, 2e-4),
                                 ph.planar_array(2, 2, 1e-3, 6e-3), 300, seed=75),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_forward_with_device_built_order(torch_cuda, name):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = CASES[name]
    x = f32(prob.x_true)
    xt = torch.tensor(x, dtype=torch.float32, device="cuda")
    with Plan.from_problem(prob) as plan, Plan.from_problem(prob, c=1520.0) as fresh:
        p = plan.forward(xt).cpu().numpy()
        plan.set_sound_speed(1520.0)  # rebuilds the tables in place
        assert torch.equal(plan.forward(xt), fresh.forward(xt))
        plan.sync_status()
    ref = orc.forward(orc.Geometry.of(prob), x)
    assert rel_l2(p, ref) <= OP_TOL, rel_l2(p, ref)
