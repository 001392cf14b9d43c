"""The tensor-core kernels of the frequency-domain model at the edges of their
frequency blocks (64 per adjoint n-tile, 128 and 256 per forward block, a ragged
last block), on ragged tiles, for a sensor inside the grid, zero tiles, scales
far from 1 and non-finite inputs, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2404_10928_gb300 import phantoms as ph

from helpers import f32, rel_l2

pytestmark = pytest.mark.gpu

# the FP32 phase error bound of tests/test_gpu_freq.py (1.1e-5 rad at 20 MHz), times ten
FREQ_TOL = 1e-4


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10928_gb300 import build
    build.build()
    return torch


def _problem(dim):
    if dim == 2:  # three tiles wide, the last one 6 pixels; one sensor inside the grid
        sens = np.concatenate([ph.ring_sensors(8, 6e-3), [[0.213e-3, -0.547e-3]]])
        return ph.custom(2, (70, 33), (1e-4, 1e-4), sens, 64, seed=61)
    return ph.custom(3, (20, 9, 17), (2e-4, 2e-4, 2e-4), ph.planar_array(3, 3, 0.8e-3, 3.5e-3), 64,
                     seed=62)


@pytest.mark.parametrize("dim,q,scale", [(2, 44, 1.0), (2, 64, 1e-20), (2, 65, 1.0), (2, 72, 1e12),
                                         (2, 128, 1.0), (2, 129, 1.0), (2, 256, 1.0),
                                         (2, 257, 1.0), (2, 385, 1.0), (3, 72, 1.0), (3, 130, 1.0)])
def test_freq_blocks_match_oracle(torch_cuda, dim, q, scale):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = _problem(dim)
    geo = orc.Geometry.of(prob)
    df = 20e6 / q
    rng = np.random.default_rng(q)
    x = f32(prob.x_true * scale)
    if dim == 2:
        x.reshape(33, 70)[:32, :32] = 0.0  # a tile of zeros
    pq = (rng.standard_normal((prob.n_sensors, q)) + 1j * rng.standard_normal((prob.n_sensors, q)))
    pq[1] = 0.0  # a silent sensor
    pq = (scale * pq).astype(np.complex64).astype(np.complex128)
    with Plan.from_problem(prob) as plan:
        xt = torch.tensor(x, dtype=torch.float32, device="cuda")
        pt = torch.tensor(pq, dtype=torch.complex64, device="cuda")
        p = plan.freq_forward(xt, q, 0.0, df).cpu().numpy()
        g = plan.freq_adjoint(pt, q, 0.0, df).cpu().numpy()
        # a NaN pixel reaches every spectrum, a NaN sample every pixel
        xt[5] = float("nan")
        pt[2, 3] = complex(float("inf"), 0.0)
        p_bad = plan.freq_forward(xt, q, 0.0, df)[:, 1:]
        g_bad = plan.freq_adjoint(pt, q, 0.0, df)
        assert not torch.isfinite(torch.view_as_real(p_bad)).any()
        assert not torch.isfinite(g_bad).any()
        plan.sync_status()
    assert rel_l2(p, orc.freq_forward(geo, x, q, 0.0, df)) <= FREQ_TOL
    assert rel_l2(g, orc.freq_adjoint(geo, pq, q, 0.0, df)) <= FREQ_TOL
