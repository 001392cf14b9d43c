"""The gathers that share a pair's arrival over several frames (k_adjoint_frames)
and the TV launch over all frames: bit for bit the single-frame results for every
frame count, work split and dimension, and frames that do not leak into one
another."""
import numpy as np
import pytest

from paper_2404_10928_gb300 import phantoms as ph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_10928_gb300 import build
    build.build()
    return torch


def _problem(dim):
    if dim == 2:  # ragged tiles, a sensor inside the grid, more sensors than a stage
        sens = np.concatenate([ph.ring_sensors(20, 6e-3), [[0.213e-3, -0.547e-3]]])
        return ph.custom(2, (70, 37), (1e-4, 1e-4), sens, 300, seed=81)
    return ph.custom(3, (20, 9, 17), (2e-4, 2e-4, 2e-4), ph.planar_array(3, 3, 0.8e-3, 3.5e-3), 250,
                     seed=82)


@pytest.mark.parametrize("dim,cluster,warps", [(2, 0, 0), (2, 1, 8), (2, 2, 4), (2, 8, 4), (3, 0, 0),
                                               (3, 4, 4)])
def test_frames_equal_single_frames(torch_cuda, dim, cluster, warps):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Plan
    prob = _problem(dim)
    gen = torch.Generator(device="cuda").manual_seed(3)
    S, K, N = prob.n_sensors, prob.n_samples, prob.n_pixels
    with Plan.from_problem(prob, adj_cluster=cluster, adj_warps=warps) as plan:
        for n in (6, 1, 2, 3, 5, 4):  # fewer frames after more: stale partners
            p = torch.randn((n, S, K), generator=gen, device="cuda")
            x = torch.randn((n, N), generator=gen, device="cuda")
            one = torch.stack([plan.adjoint(q) for q in p])
            assert torch.equal(plan.adjoint_frames(p), one)
            # image and slopes in one gather against each alone
            gx, gc = plan.data_tv_loss_vjp_frames(x, p, None, 0.0, 1.0, need_c=True)
            gx1, _ = plan.data_tv_loss_vjp_frames(x, p, None, 0.0, 1.0)
            _, gc1 = plan.data_tv_loss_vjp_frames(x, p, None, 0.0, 1.0, need_x=False, need_c=True)
            assert torch.equal(gx, gx1) and torch.equal(gc, gc1)
            assert torch.equal(gx, -2.0 * one)
            # the sum over frames: each frame's own derivative, to the rounding of the sum
            each = sum(float(plan.dc(a, b)) for a, b in zip(x, p))
            mags = sum(abs(float(plan.dc(a, b))) for a, b in zip(x, p))
            assert abs(float(gc) + 2.0 * each) <= 1e-9 * mags
            assert float(plan.dc_frames(x, p)) == pytest.approx(each, abs=1e-9 * mags)
            if n > 1:  # a NaN frame leaves the others alone
                bad = p.clone()
                bad[1] = float("nan")
                out = plan.adjoint_frames(bad)
                keep = [f for f in range(n) if f != 1]
                assert torch.equal(out[keep], one[keep]) and torch.isnan(out[1]).all()
            vals, grads = plan.tv_frames(x, 1e-3)
            for f in range(n):
                v, g = plan.tv(x[f], 1e-3)
                assert torch.equal(g, grads[f])
                assert abs(float(v) - float(vals[f])) <= 1e-12 * float(v)
        plan.sync_status()
