"""Residuals packed by the combine (its warps overlap by one group of samples) and
the TV gradient in the FISTA epilogue: one step of each method against the same
step composed from the single operators, at row lengths around the warp, group
and block edges, with FP16 traces, in 2D and with many windows per sample."""
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


def _problem(dim, K):
    if dim == 2:
        return ph.custom(2, (45, 37), (1e-4, 1e-4), ph.ring_sensors(7, 5e-3), K, seed=91,
                         t0=60 / 40e6 if K < 150 else 0.0)
    # window starts every few samples: the one-sample-per-thread combine
    return ph.custom(3, (64, 40, 40), (2e-4, 2e-4, 2e-4), ph.planar_array(3, 2, 2e-3, 6e-3), K,
                     seed=92, t0=60 / 40e6)


@pytest.mark.parametrize("dim,K,f16", [(2, 2, False), (2, 3, False), (2, 123, False),
                                       (2, 124, True), (2, 125, False), (2, 991, False),
                                       (2, 992, False), (2, 993, True), (2, 1117, False),
                                       (3, 31, False), (3, 60, False), (3, 249, True)])
def test_steps_equal_their_operators(torch_cuda, dim, K, f16):
    torch = torch_cuda
    from paper_2404_10928_gb300.api import Batch, Plan
    prob = _problem(dim, K)
    gen = torch.Generator(device="cuda").manual_seed(K)
    with Plan.from_problem(prob, y_dtype="f16" if f16 else "f32") as plan:
        y = torch.randn((prob.n_sensors, K), generator=gen, device="cuda")
        y = y.half() if f16 else y
        x0 = torch.rand(prob.n_pixels, generator=gen, device="cuda")
        r = y.float() - plan.forward(x0)
        g = plan.adjoint(r)
        om = 0.3 * float(x0.norm() / g.norm()) if float(g.norm()) > 0 else 1.0
        want = torch.clamp_min(x0.double() + om * g.double(), 0.0)

        def close(a, b):
            assert float((a.double() - b).norm()) <= 1e-6 * float(b.norm())

        x, hist = plan.reconstruct(y, "landweber", 1, x0=x0, omega=om, history=True)
        close(x, want)
        assert hist[0] == pytest.approx(float((r.double() ** 2).sum()), rel=1e-6)
        xs = [x0.clone()]
        with Batch([plan]) as batch:
            bh = batch.landweber([y], xs, [om], 1, history=True)
        close(xs[0], want)
        assert bh[0][0] == pytest.approx(hist[0], rel=1e-12)
        # FISTA's first step from z = x0: the gradient of the data and TV terms
        _, tg = plan.tv(x0, 1e-2)
        tvw = 0.1 * float(g.norm() / tg.norm()) if float(g.norm()) > 0 else 1e-3
        z = x0.double() + om * (2.0 * g.double() - tvw * tg.double())
        xf = plan.reconstruct(y, "fista", 1, x0=x0, omega=om, l1=1e-3, tv=tvw, tv_eps=1e-2)
        close(xf, torch.clamp_min(z - om * 1e-3, 0.0))
        # CGLS's first step: alpha = ||s||^2 / ||A s||^2 from the packed residual
        s, q = g.double(), plan.forward(g).double()
        if float(q.norm()) > 0:
            alpha = float((s * s).sum() / (q * q).sum())
            xc = plan.reconstruct(y, "cgls", 1, x0=x0, nonneg=False)
            close(xc, x0.double() + alpha * s)
        plan.sync_status()
